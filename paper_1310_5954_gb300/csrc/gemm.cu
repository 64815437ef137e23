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
// transform and the Gram at n_act = 4833, m = 1024; this takes 53 / 39 / 35 us).
//
// What bounds a split product is the time from a stage's refill to its use, about 2500 cycles: a ring of S
// stages, each M cycles of products, takes (2500 + M) / S per stage.  Per 64 columns of K a 128 x 256 piece
// has 1548 cycles of products; two whole-tile stages of 96 KB took 2050, four of two slices take 1645.  (One
// slice per stage costs more again, 2500: the producer's waits and copies come to 600 cycles per stage.)
// Narrower pieces take 1410 (128 columns) and 1395 (64).  Two CTAs of a cluster take the two row tiles of a
// piece and copy half of the B chunk each to both (multicast): 64 KB instead of 96 KB per step from L2, 1645
// against 1674 cycles alone, and less when all SMs read at once; clusters of four (2 x 2 CTAs, 1555 cycles)
// leave 8 of 152 SMs idle and lose that again (transform 44 us, noise draw 56 us).

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstring>
#include <vector>

#include "../../include/letkf.h"
#include "internal.hpp"
#include "umma.cuh"

namespace letkf {

using namespace umma;

namespace {

constexpr int GT = 192;                   // threads per CTA: producer warp, MMA warp, four epilogue warps
constexpr int TILE_B = 128 * 64 * 2;      // bytes of one operand tile
constexpr long long GEMM_WAIT = 4000000000LL;

__device__ __forceinline__ void split_bf16(float x, __nv_bfloat16& h, __nv_bfloat16& l) {
    h = __float2bfloat16_rn(x);
    l = __float2bfloat16_rn(x - __bfloat162float(h));
}

// Byte offset of element (row, col) in a tiled operand with nkb column tiles.
__device__ __forceinline__ size_t tiled_offset(int row, int col, int nkb) {
    return ((size_t)(row >> 7) * nkb + (col >> 6)) * TILE_B + op_offset(row & 127, col & 63, 64);
}

// One stage: KC columns of A (128 rows, hi and lo) and of B (bn rows or columns).  MN: a whole tile, B read
// MN-major; else SL slices of 16 columns.  A unit (tile or slice) is [A hi, A lo, B hi, B lo].
template <bool MN>
struct GemmStage {
    static constexpr int UC = MN ? 64 : 16, SL = MN ? 1 : 2, KC = UC * SL;    // columns of a unit, units, columns
    static constexpr int A_BYTES = 128 * 2 * UC;
    static constexpr int RING = 192 * 1024, MOST = MN ? 4 : 8;
    static constexpr int EPI = 4 * 32 * 36 * 4;        // 32 rows x 32 columns per epilogue warp, padded rows
    static constexpr int BYTES = 1024 + RING + EPI;
};

// CM CTAs per cluster, along the rows: they share the columns of B.
template <int CM, bool MN>
__global__ void __launch_bounds__(GT, 1) gemm_kernel(const __grid_constant__ GemmArgs g) {
    using L = GemmStage<MN>;
    constexpr int BN = MN ? 64 : 256;
    const uint32_t b_slot = (uint32_t)g.bn * 2 * L::UC, unit = 2 * L::A_BYTES + 2 * b_slot, stage_b = L::SL * unit;
    const int stages = min(L::MOST, L::RING / (int)stage_b);
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    __shared__ __align__(8) uint64_t full[L::MOST], empty[L::MOST], tfull[2], tempty[2];
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag, issued;        // issued: stages the producer filled (for the drain on abort)
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, uwarp = uniform_warp();
    const uint32_t rank = CM > 1 ? cluster_rank() : 0u;
    if (tid == 0) {
        for (int s = 0; s < L::MOST; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], CM);              // every CTA this one's copies reach
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(&tfull[a], 1);
            mbar_init(&tempty[a], 128);
        }
        abort_flag = issued = 0;
        fence_mbar_init();
    }
    if (warp == 0) {
        tmem_alloc(&tmem_slot, 2 * BN);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (CM > 1) cluster_sync();                    // every barrier is initialised before a peer's copy arrives
    const uint32_t tmem = tmem_slot;
    const bool on = g.run == nullptr || *g.run != 0;
    if (g.next_flag && blockIdx.x == 0 && tid == 0) {
        // this launch decides whether the next step runs (see GemmArgs), also when it does
        // nothing itself, so that a finished iteration stays finished
        *g.next_flag = (on && __uint_as_float(*g.dev_in) >= g.run_tol) ? 1 : 0;
        if (on) {
            *g.dev_in = 0u;
            if (g.z_final) *g.z_final = g.z_index;
            if (g.steps) *g.steps += 1;
        }
    }
    const bool split = g.split != 0;
    const int cid = blockIdx.x / CM;
    const int i0 = on ? g.start[cid] : 0, i1 = on ? g.start[cid + 1] : 0;
    struct Work {
        int ty, col0, kb0, kb1, width, share, z;
    };
    auto work = [&](int i) {
        const int4 it = g.items[i];
        Work w;
        w.ty = it.x * CM + rank;
        w.width = it.w & 0x3FF;
        w.col0 = it.y;
        w.kb0 = it.z & 0xFFFF;
        w.kb1 = it.z >> 16;
        w.share = (it.w >> 10) & 0xFFFF;
        w.z = it.w >> 28;
        return w;
    };
    if (uwarp == 0 && elect_one()) {
        constexpr uint16_t all = (uint16_t)((1u << CM) - 1u);
        // Each CTA copies its part of a chunk of B to all of them.
        // 256 columns are two consecutive 128-row tiles, copied next to each other so that one descriptor
        // with the same row-group stride spans all 256 rows
        auto copy_b = [&](uint8_t* dst, const uint8_t* src, uint32_t bytes, size_t next, uint64_t* bar) {
            if (CM > 1) {
                const uint32_t part = bytes / CM, off = rank * part;
                bulk_g2s_multicast(dst + off, src + (off / L::A_BYTES) * next + off % L::A_BYTES, part, bar, all);
            } else {
                bulk_g2s(dst, src, min(bytes, (uint32_t)L::A_BYTES), bar);
                if (bytes > L::A_BYTES) bulk_g2s(dst + L::A_BYTES, src + next, L::A_BYTES, bar);
            }
        };
        int c = 0, s = 0, par = 0;                 // stages filled so far, the next one and its parity
        bool ok = true;
        for (int i = i0; i < i1 && ok; ++i) {
            const Work w = work(i);
            // a CTA past the last row tile reads that one's operands (its results are dropped)
            const int ty = min(w.ty, g.m_tiles - 1), col0 = w.col0;
            const uint32_t b_bytes = (uint32_t)w.width * (MN ? 128u : 32u);
            const uint32_t stage_bytes = (split ? 2u : 1u) * L::SL * (L::A_BYTES + b_bytes);
            const size_t a_row = (size_t)ty * g.a_nkb * TILE_B;
            // K-major B (rows = N): the 128-row tile holding this CTA's columns, from the slice's second half
            // for odd blocks of 64.  MN-major B (the second factor itself, rows = K; width 64): step kb takes
            // rows 64 kb .. 64 kb + 63 of column tile col0 / 64, the first or second half of that tile.
            const size_t b_row = MN ? (size_t)(col0 >> 6) * TILE_B
                                    : (size_t)(col0 >> 7) * g.b_nkb * TILE_B + ((col0 & 64) ? L::A_BYTES / 2 : 0);
            const size_t b_next = (size_t)g.b_nkb * TILE_B;
            const uint8_t *a_hi = g.a_hi[w.z] + a_row, *b_hi = g.b_hi[w.z] + b_row;
            const uint8_t *a_lo = split ? g.a_lo[w.z] + a_row : nullptr, *b_lo = split ? g.b_lo[w.z] + b_row : nullptr;
            const int k_end = w.kb1 * 64 / L::KC;
            for (int k = w.kb0 * 64 / L::KC; k < k_end; ++k, ++c) {
                if (c >= stages && !mbar_wait_bounded(&empty[s], par ^ 1, GEMM_WAIT)) {
                    atomicOr(g.status, ST_TIMEOUT);
                    abort_flag = 1;
                    ok = false;
                    break;
                }
                mbar_arrive_expect_tx(&full[s], stage_bytes);
#pragma unroll
                for (int u = 0; u < L::SL; ++u) {
                    uint8_t* st = smem + s * stage_b + u * unit;
                    const size_t ao = (size_t)(k * L::SL + u) * L::A_BYTES;
                    const size_t bo = MN ? (size_t)(k >> 1) * g.b_nkb * TILE_B + (size_t)(k & 1) * (TILE_B / 2) : ao;
                    bulk_g2s(st, a_hi + ao, L::A_BYTES, &full[s]);
                    copy_b(st + 2 * L::A_BYTES, b_hi + bo, b_bytes, b_next, &full[s]);
                    if (split) {
                        bulk_g2s(st + L::A_BYTES, a_lo + ao, L::A_BYTES, &full[s]);
                        copy_b(st + 2 * L::A_BYTES + b_slot, b_lo + bo, b_bytes, b_next, &full[s]);
                    }
                }
                if (++s == stages) s = 0, par ^= 1;
            }
        }
        issued = c;
    } else if (uwarp == 1 && elect_one()) {
        // A: K-adjacent core matrices 128 B apart, row-adjacent 1024 B in a tile, 256 B in a slice; K-major B
        // alike.  MN-major B: N-adjacent core matrices 128 B apart, K-adjacent 1024 B, a K step 2048 B
        constexpr uint32_t a_sbo = MN ? 1024u : 256u, b_lbo = MN ? 1024u : 128u, b_sbo = MN ? 128u : 256u;
        constexpr uint32_t a_step = 256u, b_step = 2048u;   // within a tile; slices lie a unit apart
        constexpr uint16_t all = (uint16_t)((1u << CM) - 1u);       // their copies fill this CTA's stages
        int n = 0, s = 0, par = 0;
        bool ok = true;
        for (int i = i0; i < i1 && ok; ++i) {
            const Work w = work(i);
            const uint32_t idesc = idesc_bf16(128, w.width, MN);
            const int acc_i = n & 1;
            if (n >= 2 && !mbar_wait_bounded(&tempty[acc_i], ((n >> 1) - 1) & 1, GEMM_WAIT)) ok = false;
            tc_fence_after();
            const uint32_t dt = tmem + acc_i * BN;
            const int k_begin = w.kb0 * 64 / L::KC, k_end = w.kb1 * 64 / L::KC;
            for (int kc = k_begin; kc < k_end && ok; ++kc) {
                if (!mbar_wait_bounded(&full[s], par, GEMM_WAIT)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t st = smem_u32(smem + s * stage_b);
                const uint32_t sa_lo = st + L::A_BYTES, sb_hi = st + 2 * L::A_BYTES, sb_lo = sb_hi + b_slot;
#pragma unroll
                for (int k = 0; k < L::KC / 16; ++k) {
                    const uint32_t acc = (kc > k_begin || k > 0) ? 1u : 0u;
                    const uint32_t da = MN ? a_step * k : unit * k, db = MN ? b_step * k : unit * k;
                    const uint64_t ah = sdesc(st + da, 128, a_sbo), bh = sdesc(sb_hi + db, b_lbo, b_sbo);
                    mma_bf16(dt, ah, bh, idesc, acc);
                    if (split) {
                        mma_bf16(dt, ah, sdesc(sb_lo + db, b_lbo, b_sbo), idesc, 1u);
                        mma_bf16(dt, sdesc(sa_lo + da, 128, a_sbo), bh, idesc, 1u);
                    }
                }
                if (CM > 1)
                    mma_commit_multicast(&empty[s], all);
                else
                    mma_commit(&empty[s]);
                if (++s == stages) s = 0, par ^= 1;
            }
            if (ok) mma_commit(&tfull[acc_i]);
            ++n;
        }
        if (!ok) {
            atomicOr(g.status, ST_TIMEOUT);
            abort_flag = 1;
        }
    } else if (warp >= 2) {
        const int quad = warp & 3, trow = 32 * quad + lane;      // TMEM lane = tile row of this thread
        float* stg = reinterpret_cast<float*>(smem + L::RING) + quad * 32 * 36;
        const bool vec = ((g.ldc | g.c_split_stride) & 3) == 0 && (reinterpret_cast<uintptr_t>(g.c) & 15) == 0;
        float dev = 0.f;
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
            const bool mine = w.ty < g.m_tiles;
#pragma unroll 1
            for (int c0 = 0; c0 < w.width; c0 += 64) {
                float v[64];
                tmem_ld64(tmem + acc_i * BN + ((uint32_t)(quad * 32) << 16) + c0, v);
                if (!mine) continue;
                if (g.mode == GEMM_EPI_TILES) {
                    // out = alpha * acc + beta * I, as a tiled operand (all padded positions written:
                    // rows and columns beyond M, N get zeros)
#pragma unroll
                    for (int j = 0; j < 64; j += 8) {
                        __align__(16) __nv_bfloat16 h[8], l[8];
#pragma unroll
                        for (int q = 0; q < 8; ++q) {
                            const int col = col0 + c0 + j + q;
                            const bool in = row < g.M && col < g.N;
                            const float x = in ? g.alpha * v[j + q] + (row == col ? g.beta : 0.f) : 0.f;
                            if (g.dev && in) dev = fmaxf(dev, fabsf(v[j + q] - (row == col ? 1.f : 0.f)));
                            split_bf16(x, h[q], l[q]);
                        }
                        const size_t off = tiled_offset(row, col0 + c0 + j, g.o_nkb);
                        *reinterpret_cast<uint4*>(g.o_hi[w.z] + off) = *reinterpret_cast<const uint4*>(h);
                        if (g.o_lo[w.z]) *reinterpret_cast<uint4*>(g.o_lo[w.z] + off) = *reinterpret_cast<const uint4*>(l);
                    }
                } else {
                    // F32: alpha acc; ADD_ROW: add[row] + acc; valid rows and columns only.  32 columns
                    // at a time through shared memory, so that a warp writes whole 128-byte row pieces
                    float* cz = g.c + (size_t)w.share * g.c_split_stride;
                    const bool add = g.mode == GEMM_EPI_ADD_ROW;
                    const float base = add && row < g.M ? g.add[row] : 0.f;
#pragma unroll
                    for (int hf = 0; hf < 64; hf += 32) {
                        __syncwarp();
#pragma unroll
                        for (int j = 0; j < 32; j += 4) {
                            float4 o;
                            o.x = add ? base + v[hf + j] : g.alpha * v[hf + j];
                            o.y = add ? base + v[hf + j + 1] : g.alpha * v[hf + j + 1];
                            o.z = add ? base + v[hf + j + 2] : g.alpha * v[hf + j + 2];
                            o.w = add ? base + v[hf + j + 3] : g.alpha * v[hf + j + 3];
                            *reinterpret_cast<float4*>(stg + lane * 36 + j) = o;
                        }
                        __syncwarp();
#pragma unroll 2
                        for (int q = 0; q < 8; ++q) {
                            const int rr = 4 * q + (lane >> 3), cc = 4 * (lane & 7);
                            const int gr = row0 + 32 * quad + rr, gc = col0 + c0 + hf + cc;
                            const float4 o = *reinterpret_cast<const float4*>(stg + rr * 36 + cc);
                            if (gr < g.M) {
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
                }
            }
            tc_fence_before();
            mbar_arrive(&tempty[acc_i]);
            ++n;
        }
        if (g.dev) {
            for (int o = 16; o > 0; o >>= 1) dev = fmaxf(dev, __shfl_xor_sync(0xffffffffu, dev, o));
            if (lane == 0) atomicMax(g.dev, __float_as_uint(dev));
        }
    }
    __syncwarp();
    __syncthreads();
    // copies still in flight after a wait gave up land in shared memory before the CTA leaves
    if (abort_flag && tid == 0)
        for (int c = max(0, issued - stages); c < issued; ++c)
            mbar_wait_bounded(&full[c % stages], (c / stages) & 1, GEMM_WAIT);
    tc_fence_before();
    __syncthreads();
    if (CM > 1) cluster_sync();                    // no peer's copy or arrival comes after a CTA has left
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
    return (size_t)((rows + 127) / 128) * ((cols + 63) / 64) * TILE_B;
}

// The pieces are dealt longest first, each to the cluster with the least work so far.  A piece costs the
// measured cycles per K step at its width, and its read-out.  Narrow pieces cost more per column but come
// out more even: every width is tried, also with only the last, uneven round cut up, and the plan whose
// busiest cluster is done first is taken.  (Noise draw at n_act = 4833, m = 1024, a triangular factor whose
// row tiles take 2 to 76 steps: 128 columns, 53 us; with 256 the longest piece alone is 68 us.)
GemmPlan gemm_plan(const GemmShape& s, int sms) {
    GemmPlan best;
    best.cycles = -1;
    const int fit = std::max(1, sms / s.cm);
    auto cost = [&](const int4& p) -> long long {
        const int w = p.w & 0x3FF, steps = (p.z >> 16) - (p.z & 0xFFFF);
        const int c = s.mn ? 768 : w == 64 ? 1395 : w == 128 ? 1410 : 1645;
        return (long long)steps * c + 1000 + 8 * w;
    };
    auto pieces = [&](int row, int col, int width, std::vector<int4>& out) {   // one column group of one row group
        const int last = std::min(s.m_tiles, (row + 1) * s.cm);      // row tiles [row * cm, last)
        const int kend = s.lower ? std::min(s.nkb, 2 * last) : s.nkb;
        for (int z = 0; z < s.batch; ++z)
            for (int k = 0; k < s.ksplit; ++k) {
                const int k0 = (int)((long long)kend * k / s.ksplit), k1 = (int)((long long)kend * (k + 1) / s.ksplit);
                out.push_back(make_int4(row, col, k0 | (k1 << 16), width | (k << 10) | (z << 28)));
            }
    };
    for (int base = s.bn; base >= 64; base /= 2)
        for (int tail = base; tail >= 64; tail /= 2) {
            std::vector<int4> all;
            for (int r = 0; r * s.cm < s.m_tiles; ++r)
                for (int c = 0; c < s.N;) {
                    int w = base;
                    while (w > 64 && (c % w || c + w > (s.N + 63) / 64 * 64)) w /= 2;
                    if (!s.upper || c + w > r * s.cm * 128) pieces(r, c, w, all);
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
            p.cm = s.cm;
            p.ncl = (int)std::min<size_t>(fit, all.size());
            std::vector<std::vector<int4>> mine(p.ncl);
            std::vector<long long> load(p.ncl, 0);
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

namespace {
template <typename F>
int gemm_with(bool mn, int cm, F&& f) {
    if (mn) return cm == 1 ? f(gemm_kernel<1, true>, GemmStage<true>::BYTES) : LETKF_EINVAL;
    if (cm == 1) return f(gemm_kernel<1, false>, GemmStage<false>::BYTES);
    return cm == 2 ? f(gemm_kernel<2, false>, GemmStage<false>::BYTES) : LETKF_EINVAL;
}
}  // namespace

int gemm_prepare() {
    for (int k = 0; k < 3; ++k) {
        const int rc = gemm_with(k == 2, k == 1 ? 2 : 1, [](auto* fn, int smem) -> int {
            return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) == cudaSuccess
                       ? LETKF_OK
                       : LETKF_ECUDA;
        });
        if (rc) return rc;
    }
    return LETKF_OK;
}

int gemm_launch(const GemmArgs& g, const GemmPlan& p, cudaStream_t stream) {
    if ((g.b_mn && p.bn != 64) ||  p.ncl < 1 || !p.d_start || !p.d_items) return LETKF_EINVAL;
    GemmArgs a = g;
    a.start = p.d_start;
    a.items = p.d_items;
    a.bn = p.bn;
    return gemm_with(g.b_mn != 0, p.cm, [&](auto* fn, int smem) -> int {
        cudaLaunchAttribute at;
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = p.cm;
        at.val.clusterDim.y = at.val.clusterDim.z = 1;
        cudaLaunchConfig_t cfg;
        std::memset(&cfg, 0, sizeof(cfg));
        cfg.gridDim = dim3(p.cm * p.ncl);
        cfg.blockDim = dim3(GT);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = stream;
        cfg.attrs = &at;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, fn, a) == cudaSuccess ? LETKF_OK : LETKF_ECUDA;
    });
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
    shape.cm = !b_mn && mp > 128 ? 2 : 1;       // as the analysis has it
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
        g.a_hi[0] = ah;
        g.a_lo[0] = split ? al : nullptr;
        g.b_hi[0] = bh;
        g.b_lo[0] = split ? bl : nullptr;
        g.m_tiles = mp / 128;
        g.a_nkb = kp / 64;
        g.b_nkb = b_mn ? (N + 63) / 64 : kp / 64;
        g.b_mn = b_mn;
        g.split = split;
        g.M = M;
        g.N = N;
        g.mode = GEMM_EPI_F32;
        g.c = C;
        g.ldc = N;
        g.alpha = 1.f;
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
