// Tiled tensor-core GEMM for the global (single-domain) analysis at large ensemble sizes.
//
// Operand formats.  An R x K matrix is stored in BF16 with R and K padded by zeros to multiples of 128 and
// 64.  "Tiled": tiles of 128 rows x 64 columns (16 KB), tile (rb, kb) at byte offset (rb * nkb + kb) * 16384,
// each in the canonical no-swizzle K-major layout of umma.cuh; a tile can be A or, read MN-major, the second
// factor itself, which the matrix iteration needs (its iterates are both).  "Sliced": the 16 KB are four
// slices of 128 rows x 16 columns (4 KB), each in that layout, so that a product can take any multiple of 16
// columns as one contiguous copy; used where both operands are K-major.  A split operand has a second, "lo",
// set holding bf16(x - float(hi)): hi * hi + hi * lo + lo * hi reproduces an FP32 product to ~2^-16.
//
// C (M x N) = A (M x K) B (N x K)^T in pieces of 128 rows x up to 256 columns, dealt to the CTAs by
// gemm_plan.  A producer warp fills a ring of shared-memory stages with bulk copies, an MMA warp issues
// tcgen05.mma into one of two accumulators in tensor memory, and four warps read the other back for the
// epilogue, so that a piece's read-out runs under the next one's products (one CTA per piece, 128 threads
// doing all three in turn and 8-byte row-strided stores, took 103 / 90 / 43 us for the noise draw, the
// transform and the Gram at n_act = 4833, m = 1024; this takes 53 / 39 / 36 us).
//
// What bounds a split product is the time from a stage's refill to its use, about 2500 cycles: a ring of S
// stages, each M cycles of products, takes (2500 + M) / S per stage.  Per 64 columns of K a 128 x 256 piece
// has 1548 cycles of products; two whole-tile stages of 96 KB took 2050, four of two slices take 1674.  (One
// slice per stage costs more again, 2500: the producer's waits and copies come to 600 cycles per stage.)
// Narrower pieces take 1410 (128 columns) and 1395 (64).  Every CTA copies its own operands:
// pairs of CTAs that shared the columns of B took 55 / 37 us for the noise draw and the Gram, this 53 / 36 (row
// tiles dealt one by one come out more even).

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstring>
#include <vector>

#include "../../include/letkf.h"
#include "gemm_ring.cuh"
#include "internal.hpp"
#include "umma.cuh"

namespace letkf {

using namespace umma;

namespace {

constexpr int GT = 192;                   // threads per CTA: producer warp, MMA warp, four epilogue warps
constexpr int GEMM_EPI = 4 * 32 * 36 * 4;  // 32 rows x 32 columns per epilogue warp, padded rows
constexpr int GEMM_SMEM = 1024 + 192 * 1024 + GEMM_EPI;

template <bool MN>
__global__ void __launch_bounds__(GT, 1) gemm_kernel(const __grid_constant__ GemmArgs g) {
    using L = GemmStage<MN>;
    constexpr int BN = MN ? 64 : 256;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    __shared__ __align__(8) uint64_t full[L::MOST], empty[L::MOST], tfull[2], tempty[2];
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag, filled;
    const Ring ring = make_ring<MN>(smem, full, empty, g.bn);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, uwarp = uniform_warp();
    if (tid == 0) {
        for (int s = 0; s < L::MOST; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(&tfull[a], 1);
            mbar_init(&tempty[a], 128);
        }
        abort_flag = filled = 0;
        fence_mbar_init();
    }
    if (warp == 0) {
        tmem_alloc(&tmem_slot, 2 * BN);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;
    const bool split = g.split != 0;
    const int i0 = g.start[blockIdx.x], i1 = g.start[blockIdx.x + 1];
    struct Work {
        int ty, col0, kb0, kb1, width, share;
    };
    auto work = [&](int i) {
        const int4 it = g.items[i];
        Work w;
        w.ty = it.x;
        w.width = it.w & 0x3FF;
        w.col0 = it.y;
        w.kb0 = it.z & 0xFFFF;
        w.kb1 = it.z >> 16;
        w.share = it.w >> 10;
        return w;
    };
    if (uwarp == 0 && elect_one()) {
        RingPos pos;
        bool ok = true;
        for (int i = i0; i < i1 && ok; ++i) {
            const Work w = work(i);
            const RingOperands o = ring_operands<MN>(g.a_hi, split ? g.a_lo : nullptr, g.a_nkb, w.ty, g.b_hi, g.b_lo,
                                                     g.b_nkb, w.col0, w.width);
            ok = ring_fill<MN>(ring, pos, o, w.kb0 * 64 / L::KC, w.kb1 * 64 / L::KC);
        }
        filled = pos.c;
        if (!ok) {
            atomicOr(g.status, ST_TIMEOUT);
            abort_flag = 1;
        }
    } else if (uwarp == 1 && elect_one()) {
        RingPos pos;
        int n = 0;
        bool ok = true;
        for (int i = i0; i < i1 && ok; ++i, ++n) {
            const Work w = work(i);
            const int acc_i = n & 1;
            ok = n < 2 || mbar_wait_bounded(&tempty[acc_i], ((n >> 1) - 1) & 1, GEMM_WAIT);
            tc_fence_after();
            ok = ok && ring_issue<MN>(ring, pos, tmem + acc_i * BN, w.width, split, (w.kb1 - w.kb0) * 64 / L::KC);
            if (ok) mma_commit(&tfull[acc_i]);
        }
        if (!ok) {
            atomicOr(g.status, ST_TIMEOUT);
            abort_flag = 1;
        }
    } else if (warp >= 2) {
        const int quad = warp & 3, trow = 32 * quad + lane;      // TMEM lane = tile row of this thread
        float* stg = reinterpret_cast<float*>(smem + 192 * 1024) + quad * 32 * 36;
        const bool vec = ((g.ldc | g.c_split_stride) & 3) == 0 && (reinterpret_cast<uintptr_t>(g.c) & 15) == 0;
        int n = 0;
        for (int i = i0; i < i1; ++i) {
            const Work w = work(i);
            const int acc_i = n & 1;
            const bool ok = mbar_wait_bounded(&tfull[acc_i], (n >> 1) & 1, GEMM_WAIT);
            if (__any_sync(0xffffffffu, !ok || *reinterpret_cast<volatile int*>(&abort_flag))) {
                if (lane == 0) {
                    atomicOr(g.status, ST_TIMEOUT);
                    abort_flag = 1;
                }
                break;
            }
            tc_fence_after();
            const int row0 = w.ty * 128, col0 = w.col0, row = row0 + trow;
#pragma unroll 1
            for (int c0 = 0; c0 < w.width; c0 += 64) {
                float v[64];
                tmem_ld64(tmem + acc_i * BN + ((uint32_t)(quad * 32) << 16) + c0, v);
                // ADD_ROW: add[row] + acc; F32: acc; valid rows and columns only.  32 columns at a time
                // through shared memory, so that a warp writes whole 128-byte row pieces
                float* cz = g.c + (size_t)w.share * g.c_split_stride;
                const float base = g.mode == GEMM_EPI_ADD_ROW && row < g.M ? g.add[row] : 0.f;
#pragma unroll
                for (int hf = 0; hf < 64; hf += 32) {
                    __syncwarp();
#pragma unroll
                    for (int j = 0; j < 32; j += 4)
                        *reinterpret_cast<float4*>(stg + lane * 36 + j) = make_float4(
                            base + v[hf + j], base + v[hf + j + 1], base + v[hf + j + 2], base + v[hf + j + 3]);
                    __syncwarp();
#pragma unroll 2
                    for (int q = 0; q < 8; ++q) {
                        const int rr = 4 * q + (lane >> 3), cc = 4 * (lane & 7);
                        const int gr = row0 + 32 * quad + rr, gc = col0 + c0 + hf + cc;
                        const float4 o = *reinterpret_cast<const float4*>(stg + rr * 36 + cc);
                        if (gr >= g.M) continue;
                        float* dst = cz + (size_t)gr * g.ldc + gc;
                        if (vec && gc + 4 <= g.N) {
                            *reinterpret_cast<float4*>(dst) = o;
                        } else {
                            if (gc + 0 < g.N) dst[0] = o.x;
                            if (gc + 1 < g.N) dst[1] = o.y;
                            if (gc + 2 < g.N) dst[2] = o.z;
                            if (gc + 3 < g.N) dst[3] = o.w;
                        }
                    }
                }
            }
            tc_fence_before();
            mbar_arrive(&tempty[acc_i]);
            ++n;
        }
    }
    __syncwarp();
    __syncthreads();
    // copies still in flight after a wait gave up land in shared memory before the CTA leaves
    if (abort_flag && tid == 0) ring_drain(ring, filled);
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, 2 * BN);
}

// FP32 R x K (leading dimension ld) -> tiled BF16 hi (and lo) with zero padding to
// rows_pad x cols_pad.  One thread per 8 consecutive columns of one row (one 16-byte store).
__global__ void to_tiles_kernel(const float* __restrict__ src, int R, int K, int ld, int rows_pad, int cols_pad,
                                int sliced, uint8_t* __restrict__ hi, uint8_t* __restrict__ lo) {
    const int g8 = cols_pad >> 3;
    const size_t total = (size_t)rows_pad * g8;
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < total; t += (size_t)gridDim.x * blockDim.x) {
        const int r = (int)(t / g8), c = (int)(t - (size_t)r * g8) * 8;
        __align__(16) __nv_bfloat16 h[8], l[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const float x = (r < R && c + q < K) ? src[(size_t)r * ld + c + q] : 0.f;
            split_bf16(x, h[q], l[q]);
        }
        const size_t off = sliced ? slice_offset(r, c, cols_pad >> 6) : tiled_offset(r, c, cols_pad >> 6);
        *reinterpret_cast<uint4*>(hi + off) = *reinterpret_cast<const uint4*>(h);
        if (lo) *reinterpret_cast<uint4*>(lo + off) = *reinterpret_cast<const uint4*>(l);
    }
}

}  // namespace

size_t tiled_bytes(int rows, int cols) {
    return (size_t)((rows + 127) / 128) * ((cols + 63) / 64) * GEMM_TILE_B;
}

// The pieces are dealt longest first, each to the CTA with the least work so far.  A piece costs the
// measured cycles per K step at its width, and its read-out.  Narrow pieces cost more per column but come
// out more even: every width is tried, also with only the last, uneven round cut up, and the plan whose
// busiest CTA is done first is taken.  (Noise draw at n_act = 4833, m = 1024, a triangular factor whose
// row tiles take 2 to 76 steps: 128 columns, 53 us; with 256 the longest piece alone is 68 us.)
GemmPlan gemm_plan(const GemmShape& s, int sms) {
    GemmPlan best;
    best.cycles = -1;
    const int fit = std::max(1, sms);
    auto cost = [&](const int4& p) -> long long {
        const int w = p.w & 0x3FF, steps = (p.z >> 16) - (p.z & 0xFFFF);
        const int c = s.mn ? 768 : w == 64 ? 1395 : w == 128 ? 1410 : 1674;
        return (long long)steps * c + 1000 + 8 * w;
    };
    auto pieces = [&](int row, int col, int width, std::vector<int4>& out) {   // one column group of one row tile
        const int kend = s.lower ? std::min(s.nkb, 2 * (row + 1)) : s.nkb;
        for (int k = 0; k < s.ksplit; ++k) {
            const int k0 = (int)((long long)kend * k / s.ksplit), k1 = (int)((long long)kend * (k + 1) / s.ksplit);
            out.push_back(make_int4(row, col, k0 | (k1 << 16), width | (k << 10)));
        }
    };
    for (int base = s.bn; base >= 64; base /= 2)
        for (int tail = base; tail >= 64; tail /= 2) {
            std::vector<int4> all;
            for (int r = 0; r < s.m_tiles; ++r)
                for (int c = 0; c < s.N;) {
                    int w = base;
                    while (w > 64 && (c % w || c + w > (s.N + 63) / 64 * 64)) w /= 2;
                    if (!s.upper || c + w > r * 128) pieces(r, c, w, all);
                    c += w;
                }
            auto longer = [&](const int4& a, const int4& b) { return cost(a) > cost(b); };
            std::stable_sort(all.begin(), all.end(), longer);
            if (tail < base) {      // the pieces of an uneven last round, cut up
                const size_t even = all.size() / fit * fit;
                std::vector<int4> cut(all.begin(), all.begin() + even);
                for (size_t i = even; i < all.size(); ++i) {
                    const int w = all[i].w & 0x3FF, t = std::min(w, tail);
                    for (int c = 0; c < w; c += t)
                        cut.push_back(make_int4(all[i].x, all[i].y + c, all[i].z, (all[i].w & ~0x3FF) | t));
                }
                all.swap(cut);
                std::stable_sort(all.begin(), all.end(), longer);
            }
            GemmPlan p;
            p.bn = base;
            p.ncta = (int)std::min<size_t>(fit, all.size());
            std::vector<std::vector<int4>> mine(p.ncta);
            std::vector<long long> load(p.ncta, 0);
            for (const int4& it : all) {
                const int q = (int)(std::min_element(load.begin(), load.end()) - load.begin());
                mine[q].push_back(it);
                load[q] += cost(it);
            }
            for (const auto& v : mine) {
                p.start.push_back((int)p.items.size());
                p.items.insert(p.items.end(), v.begin(), v.end());
            }
            p.start.push_back((int)p.items.size());
            p.cycles = *std::max_element(load.begin(), load.end());
            if (best.cycles < 0 || p.cycles < best.cycles) best = p;
        }
    return best;
}

int gemm_prepare() {
    for (auto* fn : {gemm_kernel<false>, gemm_kernel<true>})
        if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, GEMM_SMEM) != cudaSuccess)
            return LETKF_ECUDA;
    return LETKF_OK;
}

int gemm_launch(const GemmArgs& g, const GemmPlan& p, cudaStream_t stream) {
    if ((g.b_mn && p.bn != 64) || p.ncta < 1 || !p.d_start || !p.d_items) return LETKF_EINVAL;
    GemmArgs a = g;
    a.start = p.d_start;
    a.items = p.d_items;
    a.bn = p.bn;
    if (g.b_mn)
        gemm_kernel<true><<<p.ncta, GT, GEMM_SMEM, stream>>>(a);
    else
        gemm_kernel<false><<<p.ncta, GT, GEMM_SMEM, stream>>>(a);
    return cudaGetLastError() == cudaSuccess ? LETKF_OK : LETKF_ECUDA;
}

int to_tiles(const float* src, int R, int K, int ld, void* hi, void* lo, int sliced, cudaStream_t stream) {
    const int rp = (R + 127) / 128 * 128, kp = (K + 63) / 64 * 64;
    const size_t total = (size_t)rp * (kp / 8);
    const int grid = (int)std::min<size_t>((total + 255) / 256, 65535);
    to_tiles_kernel<<<grid, 256, 0, stream>>>(src, R, K, ld, rp, kp, sliced, static_cast<uint8_t*>(hi),
                                              static_cast<uint8_t*>(lo));
    return cudaGetLastError() == cudaSuccess ? LETKF_OK : LETKF_ECUDA;
}

}  // namespace letkf

// C (M x N, leading dimension N) = A (M x K) B (N x K)^T through the tiled tensor-core GEMM, for
// tests: A and B are FP32 row-major device arrays, converted to tiled BF16 (split when split = 1).
extern "C" int letkf_gemm_selftest(const float* A, const float* B, float* C, int M, int N, int K, int split, int bn,
                                   int b_mn, void* stream) {
    using namespace letkf;
    if (!A || !B || !C || M < 1 || N < 1 || K < 1 || M > 16384 || N > 16384 || K > 65536 ||
        (split != 0 && split != 1) || (bn != 64 && bn != 128 && bn != 256) || (b_mn != 0 && b_mn != 1) ||
        (b_mn && bn != 64))
        return LETKF_EINVAL;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int mp = (M + 127) / 128 * 128, kp = (K + 63) / 64 * 64;
    const int np = (N + bn - 1) / bn * bn > (N + 127) / 128 * 128 ? (N + bn - 1) / bn * bn : (N + 127) / 128 * 128;
    uint8_t *ah = nullptr, *al = nullptr, *bh = nullptr, *bl = nullptr;
    int* st = nullptr;
    int rc = gemm_prepare();
    GemmShape shape;
    shape.m_tiles = mp / 128;
    shape.N = N;
    shape.nkb = kp / 64;
    shape.bn = bn;
    shape.mn = b_mn;
    GemmPlan plan = gemm_plan(shape, 152);
    // B as tiles of B (N x K) itself, or (b_mn) of B given as K x N, rows padded to 128
    const size_t ab = tiled_bytes(mp, kp), bb = b_mn ? tiled_bytes((K + 127) / 128 * 128, (N + 63) / 64 * 64)
                                                     : tiled_bytes(np, kp);
    if (!rc && (cudaMalloc(&ah, ab) != cudaSuccess || cudaMalloc(&al, ab) != cudaSuccess ||
                cudaMalloc(&bh, bb) != cudaSuccess || cudaMalloc(&bl, bb) != cudaSuccess ||
                cudaMalloc(&st, sizeof(int)) != cudaSuccess ||
                cudaMalloc(&plan.d_items, plan.items.size() * sizeof(int4)) != cudaSuccess ||
                cudaMalloc(&plan.d_start, plan.start.size() * sizeof(int)) != cudaSuccess))
        rc = LETKF_ENOMEM;
    if (!rc) {
        cudaMemsetAsync(st, 0, sizeof(int), s);
        cudaMemcpyAsync(plan.d_items, plan.items.data(), plan.items.size() * sizeof(int4), cudaMemcpyHostToDevice, s);
        cudaMemcpyAsync(plan.d_start, plan.start.data(), plan.start.size() * sizeof(int), cudaMemcpyHostToDevice, s);
        rc = to_tiles(A, M, K, K, ah, al, !b_mn, s);
        if (!rc) rc = b_mn ? to_tiles(B, K, N, N, bh, bl, 0, s) : to_tiles(B, N, K, K, bh, bl, 1, s);
    }
    if (!rc) {
        GemmArgs g{};
        g.a_hi = ah;
        g.a_lo = split ? al : nullptr;
        g.b_hi = bh;
        g.b_lo = split ? bl : nullptr;
        g.a_nkb = kp / 64;
        g.b_nkb = b_mn ? (N + 63) / 64 : kp / 64;
        g.b_mn = b_mn;
        g.split = split;
        g.M = M;
        g.N = N;
        g.mode = GEMM_EPI_F32;
        g.c = C;
        g.ldc = N;
        g.status = st;
        rc = gemm_launch(g, plan, s);
    }
    int h = 0;
    if (!rc && (cudaMemcpyAsync(&h, st, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
                cudaStreamSynchronize(s) != cudaSuccess))
        rc = LETKF_ECUDA;
    cudaStreamSynchronize(s);
    cudaFree(ah);
    cudaFree(al);
    cudaFree(bh);
    cudaFree(bl);
    cudaFree(st);
    cudaFree(plan.d_items);
    cudaFree(plan.d_start);
    if (rc) return rc;
    return h ? LETKF_ETIMEOUT : LETKF_OK;
}
