// From the Gram's partial products to the weights of a global analysis, in one cooperative kernel: the Gram
// G and the bound s, A_s = (I + G/c)/s_ns, the Newton-Schulz iteration Z -> A_s^{-1/2}, the mean weights
// (refined once) and the operand W^T = (w_bar 1^T + Z / sqrt(s_ns))^T of the transform.
//
// The iteration is a chain of m x m products (P = Z Y; Y T and T Z, T = a I - b P), each a few
// microseconds of work even at m = 1024.  As a graph of launches per product, with the passes before and
// behind it as kernels of their own, most of the time went into starting them, 12 steps' worth of which
// found the iteration already finished.  Here the CTAs, one per SM, go from phase to phase through a grid
// barrier (1.6 us), the ring of operand stages and the tensor-memory accumulators stay set up, the decision
// to stop needs no launch, and the last step leaves out Y, which only a next one would read.  With what
// is before and behind it: 160 -> 80 us at m = 197, 298 -> 168 us at m = 1024 (86 and 173 us with a slower
// barrier, before that 107 and 219 with seven plain steps; five are taken, see NsStep).
//
// A product is dealt in tiles of 128 x 64, B read MN-major (see gemm.cu): at m = 1024 that is 128 tiles for
// P (9 us: 1.4 until the first operands are there, 6.2 of products at 60 cycles each, 1.2 to read out) and
// 256 for the pair (16 us, two tiles per CTA).  At m = 197 a product takes 4 us and the barriers as much as
// the products: latency bounds it.

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstring>

#include "../../include/letkf.h"
#include "common.cuh"
#include "gemm_ring.cuh"
#include "internal.hpp"
#include "umma.cuh"

namespace letkf {

using namespace umma;

namespace {

constexpr int NS_MAX = ROOT_STEPS;
constexpr float NS_TOL = 1e-2f;   // of max |P - I| at the last step (see NsStep)
constexpr int RT = 320;           // eight epilogue warps, a producer warp, an MMA warp
constexpr int RW = RT / 32;
constexpr int ROOT_SMEM = 1024 + GemmStage<true>::RING;

// The coefficients of an iteration step, P = Z Y, T = a I - b P, Y <- Y T, Z <- T Z.  With eigenvalues x^2 of
// P a step maps x -> x (a - b x^2).  The plain step (a = 3/2, b = 1/2) raises small x by 1.5 only;
// a = 3 rho / 2, b = rho^3 / 2 raises them by 1.5 rho and keeps [l, 1] in [l', 1], best with
// rho^2 = 3 / (1 + l + l^2), where l and 1 land on the same l' (J. Chen and E. Chow, "A stable scaling of
// Newton-Schulz for improving the sign function computation of a Hermitian matrix", 2014).  l is known:
// (I + G/c)/s has no eigenvalue below 1/s, and has that one (the anomalies of a row add up to zero).  rho^2
// stays below NS_SCALE, so that what is 1 up to rounding lands at NS_EDGE or above.  The first step is a plain
// one, from s = NS_WIDE_FROM on A_s scaled up by NS_SCALE, which is the same as that rho (below, l is the
// larger without: s = 14 0.395 and 0.387, 6 0.395 and 0.578).  From l = NS_PLAIN on the steps are plain.
//
// When to stop is known from l as well: the update from l >= NS_DONE is the last, and leaves every x within
// 1.5 (1 - NS_DONE)^2 = 3e-5 of 1.  max |P - I| < NS_TOL must hold as well, which rounding can break; alone it
// does not do, since an element of v v^T shows 1/m of what is left along a direction v (with it alone, and plain
// steps up to s = 16: anomalies off by 7e-3 at s = 2.5, m = 300, by 6e-4 at s = 25; now 1e-5 and 2e-5).
//
// Unscaled plain steps, stopped by max |P - I| alone, needed 7 steps at s = 25 (m = 197) and s = 39 (m = 1024),
// this 5; at s = 1 / 2 / 4 / 10 they need 2 / 4 / 5 / 6, this 2 / 3 / 4 / 5.  The error against 64 bits, dominated
// by the rounding of the iterates, is no larger (geometric means, s = 1 .. 60, m = 64 .. 240: 7.1e-6 to 1.1e-5
// against 7.6e-6 to 1.8e-5; 16 sizes m = 100 .. 700 on 32 x 32 and 40 x 40, frames 1 to 3 of a cold start:
// anomalies 1.1e-4 against 1.5e-4, mean 4.8e-5 against 4.8e-5).
//
// Above s = NS_SCALED_TO the scaled steps are wrong: they raise the rounding along the smallest eigenvalues
// by up to 2.4 a step, and an ensemble of fewer members than slopes has none there but the constant one.
// m = 197, 1400 slopes, mean's error against 64 bits, scaled / plain: s = 2e3 7e-5 / 7e-5, 2e4 1.2e-4 /
// 1.1e-4, 2e6 2.1e-4 / 9e-5, from 2e7 NaN / 7e-5.  Unscaled plain steps take over (l = 1), stopped by
// max |P - I| alone: the bulk of the spectrum, at its low end there, comes last, and is on the diagonal.
constexpr float NS_SCALE = 2.5f, NS_EDGE = 0.395f;   // NS_EDGE: sqrt(2.5) (3 - 2.5) / 2
constexpr float NS_PLAIN = 0.94f, NS_DONE = 0.9955f;
constexpr float NS_WIDE_FROM = 14.f, NS_SCALED_TO = 1e4f;
struct NsStep {
    float a, b;
    bool last;          // as far as l tells
};
// The scale of A_s, and the bound l after the first step.
__device__ __forceinline__ float ns_scale(float s) { return s >= NS_WIDE_FROM && s <= NS_SCALED_TO ? s / NS_SCALE : s; }
__device__ __forceinline__ float ns_first(float s) {
    if (!(s <= NS_SCALED_TO)) return 1.f;
    const float l2 = 1.f / ns_scale(s), l = 0.5f * sqrtf(l2) * (3.f - l2);
    return s >= NS_WIDE_FROM ? fminf(l, NS_EDGE) : l;
}
// The next step, and the bound behind it.
__device__ __forceinline__ NsStep ns_next(float& l) {
    NsStep t = {1.5f, 0.5f, l >= NS_DONE};
    if (l < NS_PLAIN) {
        const float r2 = fminf(NS_SCALE, 3.f / (1.f + l + l * l)), r = sqrtf(r2);
        t.a = 1.5f * r;
        t.b = 0.5f * r * r2;
        l = fminf(l * (t.a - t.b * l * l), t.a - t.b);
    } else {
        l *= t.a - t.b * l * l;
    }
    return t;
}

struct Tiles {
    uint8_t *hi, *lo;
};

struct Cta {
    uint64_t full[4], empty[4], tfull[2], tempty[2];
    uint32_t tmem;
    int abort, filled;
    float red[RW];
};

// Every thread's writes before, by any CTA, are seen behind it, by loads and by bulk copies.
// False: a wait ran out, here or in another CTA.
__device__ __forceinline__ bool grid_sync(unsigned* bar, unsigned& target, Cta* cta, int* status) {
    asm volatile("fence.proxy.async;" ::: "memory");
    __syncthreads();
    target += gridDim.x;
    if (threadIdx.x == 0) {
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
        const long long t0 = clock64();
        // the load acquires, so that no fence follows the last one; the flag and the clock are looked at now
        // and then (a second load per turn would delay the first)
        for (unsigned polls = 1; !cta->abort; ++polls) {
            unsigned seen, gave_up;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(bar) : "memory");
            if (seen >= target) break;
            if (polls & 63) continue;
            asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(gave_up) : "l"(bar + 1) : "memory");
            if (gave_up || clock64() - t0 > GEMM_WAIT) cta->abort = 1;
        }
        if (cta->abort) {
            asm volatile("st.relaxed.gpu.global.u32 [%0], 1;" ::"l"(bar + 1) : "memory");
            atomicOr(status, ST_TIMEOUT);
        }
    }
    __syncthreads();
    return cta->abort == 0;
}

__device__ __forceinline__ float warp_max(float v) {
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// Eight consecutive columns of a row as hi and lo, one 16-byte store each.
__device__ __forceinline__ void store_split(uint8_t* hi, uint8_t* lo, const float (&x)[8]) {
    uint32_t h[4], l[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const __nv_bfloat162 a = __floats2bfloat162_rn(x[2 * q], x[2 * q + 1]);
        h[q] = *reinterpret_cast<const uint32_t*>(&a);
        const __nv_bfloat162 b = __floats2bfloat162_rn(x[2 * q] - __uint_as_float(h[q] << 16),
                                                       x[2 * q + 1] - __uint_as_float(h[q] & 0xFFFF0000u));
        l[q] = *reinterpret_cast<const uint32_t*>(&b);
    }
    *reinterpret_cast<uint4*>(hi) = make_uint4(h[0], h[1], h[2], h[3]);
    *reinterpret_cast<uint4*>(lo) = make_uint4(l[0], l[1], l[2], l[3]);
}

struct Product {
    Tiles a, b, out;
};

// out = alpha A B + beta I for `count` products of m x m operands in tiles, this CTA's pieces of them; with
// dev, max |A B - I| over valid entries as well (infinite when one is not finite).  Positions beyond m get zeros.  Threads keep the ring's
// position (chunks) and the number of accumulators used (acc) in step.
__device__ __forceinline__ void products(const Ring& ring, Cta* cta, int& chunks, int& acc, const Product* p, int count,
                                         int m, int mp, float alpha, float beta, unsigned* dev, int* status) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, uwarp = uniform_warp();
    const int nkb = mp >> 6, rt = mp >> 7, ct = (m + 63) >> 6, steps = ct, per = rt * ct, total = per * count;
    const int mine = (total - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;   // <= 0: none
    if (uwarp == 8 && elect_one()) {
        RingPos pos;
        pos.c = chunks;
        pos.s = chunks % ring.stages;
        pos.par = (chunks / ring.stages) & 1;
        bool ok = true;
        for (int t = blockIdx.x; t < total && ok; t += gridDim.x) {
            const Product& q = p[t / per];
            const int u = t % per;
            ok = ring_fill<true>(ring, pos, ring_operands<true>(q.a.hi, q.a.lo, nkb, u / ct, q.b.hi, q.b.lo, nkb,
                                                                (u % ct) * 64, 64), 0, steps);
        }
        cta->filled = pos.c;
        if (!ok) cta->abort = 1;
    } else if (uwarp == 9 && elect_one()) {
        RingPos pos;
        pos.c = chunks;
        pos.s = chunks % ring.stages;
        pos.par = (chunks / ring.stages) & 1;
        bool ok = true;
        for (int t = blockIdx.x, n = acc; t < total && ok; t += gridDim.x, ++n) {
            ok = n < 2 || mbar_wait_bounded(&cta->tempty[n & 1], ((n >> 1) - 1) & 1, GEMM_WAIT);
            tc_fence_after();
            ok = ok && ring_issue<true>(ring, pos, cta->tmem + (n & 1) * 64, 64, true, steps);
            if (ok) mma_commit(&cta->tfull[n & 1]);
        }
        if (!ok) cta->abort = 1;
    } else if (warp < 8) {
        const int quad = warp & 3, half = warp >> 2;      // TMEM lanes and columns of this warp
        float worst = 0.f, finite = 0.f;     // (fmaxf drops a NaN; 0 x keeps it)
        for (int t = blockIdx.x, n = acc; t < total; t += gridDim.x, ++n) {
            const bool ok = mbar_wait_bounded(&cta->tfull[n & 1], (n >> 1) & 1, GEMM_WAIT);
            if (__any_sync(0xffffffffu, !ok)) {
                cta->abort = 1;
                break;
            }
            tc_fence_after();
            const int u = t % per, row = (u / ct) * 128 + 32 * quad + lane, c0 = (u % ct) * 64 + 32 * half;
            const Tiles out = p[t / per].out;
            uint32_t v[4][8];
            const uint32_t at = cta->tmem + (n & 1) * 64 + 32 * half + ((uint32_t)(32 * quad) << 16);
#pragma unroll
            for (int j = 0; j < 4; ++j) tmem_ld8_async(at + 8 * j, v[j]);
            tmem_wait_ld();
            tc_fence_before();
            mbar_arrive(&cta->tempty[n & 1]);
            const int r0 = row - lane;
            uint8_t *hi = out.hi + tiled_offset(row, c0, nkb), *lo = out.lo + tiled_offset(row, c0, nkb);
            if (r0 + 32 <= m && c0 + 32 <= m && r0 != c0) {         // neither the edge nor the diagonal
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    float x[8];
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        x[q] = __uint_as_float(v[j][q]);
                        worst = fmaxf(worst, fabsf(x[q]));
                        finite = fmaf(x[q], 0.f, finite);
                        x[q] *= alpha;
                    }
                    store_split(hi + 128 * j, lo + 128 * j, x);
                }
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    float x[8];
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        const int col = c0 + 8 * j + q;
                        const bool in = row < m && col < m;
                        x[q] = __uint_as_float(v[j][q]);
                        if (in) {
                            worst = fmaxf(worst, fabsf(x[q] - (row == col ? 1.f : 0.f)));
                            finite = fmaf(x[q], 0.f, finite);
                        }
                        x[q] = in ? alpha * x[q] + (row == col ? beta : 0.f) : 0.f;
                    }
                    store_split(hi + 128 * j, lo + 128 * j, x);
                }
            }
        }
        if (dev) {
            worst = warp_max(finite == 0.f ? worst : INFINITY);
            if (lane == 0) cta->red[warp] = worst;
            asm volatile("bar.sync 1, 256;" ::: "memory");
            if (threadIdx.x == 0) {
                for (int w = 1; w < 8; ++w) worst = fmaxf(worst, cta->red[w]);
                atomicMax(dev, __float_as_uint(worst));
            }
        }
    }
    __syncwarp();
    if (mine > 0) {
        chunks += mine * steps;
        acc += mine;
    }
}

__device__ __forceinline__ void unpack8(uint4 h, uint4 l, float (&v)[8]) {
    const __nv_bfloat16* hb = reinterpret_cast<const __nv_bfloat16*>(&h);
    const __nv_bfloat16* lb = reinterpret_cast<const __nv_bfloat16*>(&l);
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = __bfloat162float(hb[q]) + __bfloat162float(lb[q]);
}

// Copies a vector that other CTAs wrote into shared memory.
__device__ __forceinline__ void take(const float* v, int m, float* sv) {
    __syncthreads();
    for (int i = threadIdx.x; i < m; i += RT) sv[i] = __ldcg(v + i);
    __syncthreads();
}

// out[i] = (add ? out[i] : 0) + scale * sum_j Z[i][j] v[j], one warp per row
__device__ __forceinline__ void root_gemv(Tiles z, int nkb, int m, const float* sv, float scale, bool add, float* out) {
    const int lane = threadIdx.x & 31;
    for (int i = blockIdx.x * RW + (threadIdx.x >> 5); i < m; i += gridDim.x * RW) {
        float s = 0.f;
        for (int j0 = 8 * lane; j0 < m; j0 += 1024) {
            uint4 h[4], l[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                h[k] = l[k] = make_uint4(0, 0, 0, 0);
                if (j0 + 256 * k < m) {
                    const size_t off = tiled_offset(i, j0 + 256 * k, nkb);
                    h[k] = __ldcg(reinterpret_cast<const uint4*>(z.hi + off));
                    l[k] = __ldcg(reinterpret_cast<const uint4*>(z.lo + off));
                }
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                float a[8];
                unpack8(h[k], l[k], a);
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    if (j0 + 256 * k + q < m) s += a[q] * sv[j0 + 256 * k + q];
            }
        }
        s = warp_sum(s);
        if (lane == 0) out[i] = (add ? __ldcg(out + i) : 0.f) + scale * s;
    }
}

// Row and first column of 16-byte unit u of a tiled operand: neighbouring threads take neighbouring units.
__device__ __forceinline__ void unit_at(int u, int nkb, int& row, int& col) {
    const int t = u >> 10, rb = t / nkb;
    row = rb * 128 + ((u >> 6) & 15) * 8 + (u & 7);
    col = (t - rb * nkb) * 64 + ((u >> 3) & 7) * 8;
}

__global__ void __launch_bounds__(RT, 1) root_kernel(const __grid_constant__ RootArgs a) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    __shared__ __align__(8) Cta cta;
    const Ring ring = make_ring<true>(smem, cta.full, cta.empty, 64);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        for (int s = 0; s < 4; ++s) {
            mbar_init(&cta.full[s], 1);
            mbar_init(&cta.empty[s], 1);
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(&cta.tfull[s], 1);
            mbar_init(&cta.tempty[s], 256);
        }
        cta.abort = cta.filled = 0;
        fence_mbar_init();
    }
    if (warp == 0) {
        tmem_alloc(&cta.tmem, 128);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();

    const int m = a.m, mp = a.mp, ld = a.ldg, nkb = mp >> 6;
    const Tiles as{a.as_hi, a.as_lo}, tt{a.t_hi, a.t_lo};
    const Tiles y[2] = {{a.y_hi[0], a.y_lo[0]}, {a.y_hi[1], a.y_lo[1]}};
    const Tiles z[2] = {{a.z_hi[0], a.z_lo[0]}, {a.z_hi[1], a.z_lo[1]}};
    const int units = mp * (mp >> 3);          // 16-byte units of a tiled m x m operand
    unsigned target = 0;
    int chunks = 0, acc = 0, steps = 1, zf = 1;
    bool run = *a.frame_bad == 0, ok = true;
    float s = 1.f, sn = 1.f;                   // the bound, and the scale of A_s

    // G = sum of the shares, in order: the blocks of 64 x 64 on and above the diagonal, and their mirror;
    // sq = a block's part of the squared Frobenius norm; b = column m
    {
        float(*blk)[65] = reinterpret_cast<float(*)[65]>(smem);
        const int nb = (m + 63) >> 6, blocks = nb * (nb + 1) / 2, ty = tid >> 4, tx = tid & 15;
        for (int t = blockIdx.x; t < blocks; t += gridDim.x) {
            int bi = 0, first = 0;
            while (first + nb - bi <= t) first += nb - bi++;
            const int bj = bi + t - first;
            float sum = 0.f;
            if (tid < 256) {
                const int i0 = 64 * bi + ty, j = 64 * bj + 4 * tx;
                const float* src = a.part + (size_t)i0 * ld + j;
                float4 v[4];
#pragma unroll
                for (int r = 0; r < 4; ++r) v[r] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
                for (int k = 0; k < a.splits; ++k) {
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (i0 + 16 * r < m && j < ld)
                            x = *reinterpret_cast<const float4*>(src + k * a.stride + (size_t)16 * r * ld);
                        v[r].x += x.x;
                        v[r].y += x.y;
                        v[r].z += x.z;
                        v[r].w += x.w;
                    }
                }
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    if (i0 + 16 * r < m && j < ld) {
                        *reinterpret_cast<float4*>(a.G + (size_t)(i0 + 16 * r) * ld + j) = v[r];
                        sum += (j < m ? v[r].x * v[r].x : 0.f) + (j + 1 < m ? v[r].y * v[r].y : 0.f) +
                               (j + 2 < m ? v[r].z * v[r].z : 0.f) + (j + 3 < m ? v[r].w * v[r].w : 0.f);
                    }
                    float* d = &blk[ty + 16 * r][4 * tx];
                    d[0] = v[r].x;
                    d[1] = v[r].y;
                    d[2] = v[r].z;
                    d[3] = v[r].w;
                }
            }
            sum = warp_sum(sum);
            if (lane == 0) cta.red[warp] = sum;
            __syncthreads();
            if (bj > bi && tid < 256) {
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const int jj = ty + 16 * r, j = 64 * bj + jj;
                    if (j < m)
                        *reinterpret_cast<float4*>(a.G + (size_t)j * ld + 64 * bi + 4 * tx) =
                            make_float4(blk[4 * tx][jj], blk[4 * tx + 1][jj], blk[4 * tx + 2][jj], blk[4 * tx + 3][jj]);
                }
            }
            if (tid == 0) {
                float v = 0.f;
                for (int w = 0; w < 8; ++w) v += cta.red[w];
                a.sq[t] = bj > bi ? 2.f * v : v;
            }
            __syncthreads();
        }
        for (int i = blockIdx.x * RT + tid; i < m; i += gridDim.x * RT) {
            float v = 0.f;
#pragma unroll 8
            for (int k = 0; k < a.splits; ++k) v += a.part[k * a.stride + (size_t)i * ld + m];
            a.b[i] = v;
        }
        if (blockIdx.x == 0 && tid < NS_MAX) a.dev[tid] = 0u;
        ok = grid_sync(a.bar, target, &cta, a.status);
        // s = 1 + |G|_F / c
        float sum = 0.f;
        for (int t = tid; t < blocks; t += RT) sum += __ldcg(a.sq + t);
        sum = warp_sum(sum);
        if (lane == 0) cta.red[warp] = sum;
        __syncthreads();
        sum = 0.f;
        for (int w = 0; w < RW; ++w) sum += cta.red[w];
        s = 1.f + sqrtf(sum) / a.c;
        sn = ns_scale(s);
    }

    // A_s = (I + G/c)/s_ns and the first step's Z_1 = T_0 = (3I - A_s)/2
    if (ok) {
        const float inv = 1.f / sn, invc = 1.f / (a.c * sn);
        for (int u = blockIdx.x * RT + tid; u < units; u += gridDim.x * RT) {
            int i, j0;
            unit_at(u, nkb, i, j0);
            __align__(16) float g[8];
#pragma unroll
            for (int q = 0; q < 8; q += 4)
                *reinterpret_cast<float4*>(g + q) = i < m && j0 + q < ld
                                                        ? __ldcg(reinterpret_cast<const float4*>(a.G + (size_t)i * ld + j0 + q))
                                                        : make_float4(0.f, 0.f, 0.f, 0.f);
            float av[8], tv[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int j = j0 + q;
                av[q] = tv[q] = 0.f;
                if (i < m && j < m) {
                    av[q] = g[q] * invc + (i == j ? inv : 0.f);
                    tv[q] = (i == j ? 1.5f : 0.f) - 0.5f * av[q];
                }
            }
            const size_t off = (size_t)u * 16;
            store_split(as.hi + off, as.lo + off, av);
            store_split(z[1].hi + off, z[1].lo + off, tv);
        }
        ok = grid_sync(a.bar, target, &cta, a.status);
    }

    // the iteration; a rejected frame takes none of it (its result is not used)
    if (ok && run) {
        const Product p{as, z[1], y[1]};
        products(ring, &cta, chunks, acc, &p, 1, m, mp, 1.f, 0.f, nullptr, a.status);
        ok = grid_sync(a.bar, target, &cta, a.status);
    }
    float l = ns_first(s);
    for (int k = 1; ok && run && k < NS_MAX; ++k) {
        const NsStep ns = ns_next(l);
        const int from = k & 1, to = from ^ 1;
        const Product p{z[from], y[from], tt};
        products(ring, &cta, chunks, acc, &p, 1, m, mp, -ns.b, ns.a, a.dev + k, a.status);
        ok = grid_sync(a.bar, target, &cta, a.status);
        if (!ok) break;
        run = !ns.last || __uint_as_float(__ldcg(a.dev + k)) >= NS_TOL;      // whether a step follows, which needs Y
        const Product two[2] = {{tt, z[from], z[to]}, {y[from], tt, y[to]}};
        products(ring, &cta, chunks, acc, two, run ? 2 : 1, m, mp, 1.f, 0.f, nullptr, a.status);
        ok = grid_sync(a.bar, target, &cta, a.status);
        zf = to;
        ++steps;
    }

    // mean weights, refined once: w = Z^2 b / (c s_ns); w += Z^2 (b - (c I + G) w) / (c s_ns)
    const float scale = 1.f / (a.c * sn);
    float* sv = reinterpret_cast<float*>(smem);
    for (int pass = 0; ok && pass < 2; ++pass) {
        take(pass ? a.r : a.b, m, sv);
        root_gemv(z[zf], nkb, m, sv, 1.f, false, a.u);
        if (!(ok = grid_sync(a.bar, target, &cta, a.status))) break;
        take(a.u, m, sv);
        root_gemv(z[zf], nkb, m, sv, scale, pass != 0, a.wbar);
        if (!(ok = grid_sync(a.bar, target, &cta, a.status))) break;
        if (pass) break;
        take(a.wbar, m, sv);
        for (int i = blockIdx.x * RW + warp; i < m; i += gridDim.x * RW) {
            float v = 0.f;
            for (int j0 = 4 * lane; j0 < m; j0 += 1024) {
                float4 g[8];
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    g[k] = j0 + 128 * k < m ? __ldcg(reinterpret_cast<const float4*>(a.G + (size_t)i * ld + j0 + 128 * k))
                                            : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const int j = j0 + 128 * k;
                    if (j < m) v += g[k].x * sv[j];
                    if (j + 1 < m) v += g[k].y * sv[j + 1];
                    if (j + 2 < m) v += g[k].z * sv[j + 2];
                    if (j + 3 < m) v += g[k].w * sv[j + 3];
                }
            }
            v = warp_sum(v);
            if (lane == 0) a.r[i] = __ldcg(a.b + i) - (a.c * sv[i] + v);
        }
        ok = grid_sync(a.bar, target, &cta, a.status);
    }

    // W^T: element (j, k) = w_bar[k] + Z[j][k] / sqrt(s_ns) (W = w_bar 1^T + T_a; T_a symmetric)
    if (ok) {
        const float rs = rsqrtf(sn);
        take(a.wbar, m, sv);
        for (int u = blockIdx.x * RT + tid; u < units; u += gridDim.x * RT) {
            int j, k0;
            unit_at(u, nkb, j, k0);
            float v[8];
            unpack8(__ldcg(reinterpret_cast<const uint4*>(z[zf].hi + (size_t)u * 16)),
                    __ldcg(reinterpret_cast<const uint4*>(z[zf].lo + (size_t)u * 16)), v);
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = j < m && k0 + q < m ? sv[k0 + q] + rs * v[q] : 0.f;
            const size_t to = slice_offset(j, k0, nkb);
            store_split(a.wt_hi + to, a.wt_lo + to, v);
        }
    }
    if (blockIdx.x == 0 && tid == 0) {
        a.stats->s = s;
        a.stats->steps = steps;
        if (ok && run) atomicOr(a.status, ST_NOCONV);     // the step limit stopped the iteration
    }
    __syncthreads();
    if (cta.abort && tid == 0) ring_drain(ring, cta.filled);
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(cta.tmem, 128);
}

}  // namespace

int root_prepare() {
    return cudaFuncSetAttribute(root_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, ROOT_SMEM) == cudaSuccess
               ? LETKF_OK
               : LETKF_ECUDA;
}

int root_launch(const RootArgs& a, int sms, cudaStream_t stream) {
    // as many CTAs as the pair of products has tiles (more would only wait at the barriers), at least as
    // many as the passes over m x m entries can use, one per SM at most
    const int tiles = 2 * (a.mp / 128) * ((a.m + 63) / 64);
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeCooperative;
    at.val.cooperative = 1;
    cudaLaunchConfig_t cfg;
    std::memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3(std::min(sms, std::max(32, tiles)));
    cfg.blockDim = dim3(RT);
    cfg.dynamicSmemBytes = ROOT_SMEM;
    cfg.stream = stream;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, root_kernel, a) == cudaSuccess ? LETKF_OK : LETKF_ECUDA;
}

}  // namespace letkf
