// Global ETKF (Sect. 2.2: one domain, the whole pupil) at large ensemble sizes, on the tiled
// tensor-core GEMM of gemm.cu.  With S = Y'/sigma (p x m) and d = (y - y_bar)/sigma:
//
//   [S d]^T [S d]      one product (K = p) gives G = S^T S, b = S^T d                 (Gram)
//   A_s = (I + G/c)/s  c = m - 1, s = 1 + ||G||_F / c, or less by up to 2.5 (root.cu); eigenvalues in (0, 2.5]
//   Z = A_s^(-1/2)     coupled Newton-Schulz: P = Z Y, T = a I - b P, Y <- Y T, Z <- T Z,
//                      from Y = A_s, Z = I (first step without products: P = A_s, Z = T)
//   T_a = Z / sqrt(s) = (I + G/c)^(-1/2),   w_bar = Z^2 b / (c s), refined once against the
//                      FP32 operator (c I + G)
//   X_a = x_bar 1^T + X' (w_bar 1^T + T_a)  one product (K = m), the mean added per row
//
// then the AR forecast of the plain path (forecast_kernel), with the dense process noise
// V = L xi drawn as one more product.  Every product is a three-term split-BF16 product
// (FP32-level, ~2^-16 per element).  The iteration's products are true products (the second
// factor's tiles read MN-major): the matrices are symmetric in exact arithmetic, but taking
// A B^T for A B lets the rounding's antisymmetric part grow until the iteration diverges at the
// conditioning of the first frames (s ~ 1e4).  From the Gram's shares to W^T everything is one
// cooperative kernel (root.cu); the iteration runs at most ROOT_STEPS steps and stops by the spectrum's known
// bound and max |P - I| < 1e-2 (ST_NOCONV when the limit stops it).

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "../../include/letkf.h"
#include "common.cuh"
#include "gemm_ring.cuh"
#include "internal.hpp"
#include "umma.cuh"

namespace letkf {

struct GlobalState {
    int mr = 0, pk = 0, mp = 0, nr = 0, ka = 0;   // padded sizes: S' rows, slopes, m, state rows, actuators
    uint8_t *st_hi = nullptr, *st_lo = nullptr;   // [S d]^T slices (mr x pk)
    float* G = nullptr;                            // m x (m+1) Gram, row-major
    float* Gpart = nullptr;                        // partial Grams of the upper tiles, one per share
    int ldg = 0, gram_split = 1;                   // leading dimension of the Gram, shares of its K steps
    GemmPlan pl_gram, pl_tr, pl_tr1, pl_noise;     // Gram, transform (both instants / the first), noise draw
    uint8_t *as_hi = nullptr, *as_lo = nullptr, *t_hi = nullptr, *t_lo = nullptr;
    uint8_t *y_hi[2] = {}, *y_lo[2] = {}, *z_hi[2] = {}, *z_lo[2] = {};
    uint8_t *xp_hi = nullptr, *xp_lo = nullptr;    // X' slices (nr x mp)
    uint8_t *wt_hi = nullptr, *wt_lo = nullptr;    // W^T slices (mp x mp)
    uint8_t *l_hi = nullptr, *l_lo = nullptr;      // L slices (rup(n_act) x ka)
    uint8_t *xi_hi = nullptr, *xi_lo = nullptr;    // xi^T slices (mp x ka)
    float *xbar = nullptr, *sq = nullptr, *wbar = nullptr, *u = nullptr, *r = nullptr, *b = nullptr;
    RootStats* stats = nullptr;
    unsigned *dev = nullptr, *bar = nullptr;       // max |P - I| of each step; the grid barrier of the iteration
    int4* corner = nullptr;                        // per valid subaperture: its four corner actuators
    cudaStream_t side = nullptr;                   // a step's normals, beside its analysis
    cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
    bool forked = false;                           // normals on the side stream that no product has waited for
    std::vector<void*> allocs;
};

namespace {

int rup(int v, int a) { return (v + a - 1) / a * a; }

// Columns of the slopes' operand: the x and y slopes of eight subapertures to a slice (see gl_slopes_kernel).
int slope_cols(int n_subv) { return rup(2 * rup(n_subv, 8), 64); }

// The plans of the analysis's products, and the Gram's shares: as many as make its pieces fill the SMs,
// against the partial Grams that every share writes and the reduction reads (at 2 KB per cycle).
struct Plans {
    GemmPlan gram, tr, tr1, noise;
    int split = 1;
};
Plans plans_for(int n_act, int n_subv, int m, bool dense, bool lower, int sms) {
    Plans P;
    const int mt = rup(m, 128) / 128, rows = rup(2 * n_act, 128) / 128, acts = rup(n_act, 128) / 128;
    GemmShape g;
    g.m_tiles = mt;             // row m of the Gram is its column m
    g.N = m + 1;
    g.nkb = slope_cols(n_subv) / 64;
    g.bn = 256;
    g.upper = 1;
    long long best = -1;
    for (g.ksplit = 1; g.ksplit <= std::max(1, std::min(g.nkb / 2, 16)); ++g.ksplit) {
        GemmPlan p = gemm_plan(g, sms);
        const long long t = p.cycles + (long long)g.ksplit * m * m * 4 / 2048;
        if (best >= 0 && t >= best) continue;
        best = t;
        P.gram = p;
        P.split = g.ksplit;
    }
    GemmShape t;
    t.m_tiles = rows;
    t.N = m;
    t.nkb = rup(m, 128) / 64;
    t.bn = 256;
    P.tr = gemm_plan(t, sms);
    t.m_tiles = acts;
    P.tr1 = gemm_plan(t, sms);
    if (dense) {
        t.nkb = rup(n_act, 64) / 64;
        t.lower = lower;
        P.noise = gemm_plan(t, sms);
    }
    return P;
}

// Eight consecutive columns of a row as hi and lo, one 16-byte store each.
__device__ __forceinline__ void store8(uint8_t* hi, uint8_t* lo, size_t off, const float (&v)[8]) {
    __align__(16) __nv_bfloat16 h[8], l[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) split_bf16(v[q], h[q], l[q]);
    *reinterpret_cast<uint4*>(hi + off) = *reinterpret_cast<const uint4*>(h);
    *reinterpret_cast<uint4*>(lo + off) = *reinterpret_cast<const uint4*>(l);
}

// Member means of the state rows and the X' slices, element (r, i) = X[r][i] - x_bar[r] for r < n, i < m
// and zero beyond (for the rows below n_x rounded up to eight); resets the iteration's grid barrier.  Bound by HBM: X is read once, from HBM for the
// means, one warp per row, and again, now from L1, by threads that take the eight rows of a core matrix side
// by side, so that the slices are written in pieces of 256 bytes.  (Two kernels, the second with one thread
// per row piece and 16-byte stores 2 KB apart, took 11 + 26 us at n = 9666, m = 1024; this 19 us.)
__global__ void __launch_bounds__(256) gl_center_kernel(const float* __restrict__ X, int n, int n_x, int m, int m_pad, int mp,
                                                        float* __restrict__ xbar, uint8_t* __restrict__ hi,
                                                        uint8_t* __restrict__ lo, unsigned* __restrict__ bar) {
    __shared__ float mu_sh[8];
    if (blockIdx.x == 0 && threadIdx.x < 2) bar[threadIdx.x] = 0u;
    const int r0 = blockIdx.x * 8, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    {
        const int r = r0 + warp;
        float s = 0.f;
        if (r < n) {
            const float* x = X + (size_t)r * m_pad;
            const int m4 = m & ~3;
#pragma unroll 8
            for (int i = 4 * lane; i < m4; i += 128) {
                const float4 v = *reinterpret_cast<const float4*>(x + i);
                s += (v.x + v.y) + (v.z + v.w);
            }
            if (lane < m - m4) s += x[m4 + lane];
        }
        s = warp_sum(s);
        if (lane == 0) {
            mu_sh[warp] = s / (float)m;
            if (r < n) xbar[r] = s / (float)m;
        }
    }
    __syncthreads();
    if (r0 >= n_x) return;
    const int r = r0 + (threadIdx.x & 7);
    const float mu = mu_sh[threadIdx.x & 7];
    const float* x = X + (size_t)r * m_pad;
    for (int i0 = 8 * (threadIdx.x >> 3); i0 < mp; i0 += 256) {
        float v[8];
        if (r < n && i0 + 8 <= m) {
            const float4 a = *reinterpret_cast<const float4*>(x + i0), b = *reinterpret_cast<const float4*>(x + i0 + 4);
            v[0] = a.x - mu;
            v[1] = a.y - mu;
            v[2] = a.z - mu;
            v[3] = a.w - mu;
            v[4] = b.x - mu;
            v[5] = b.y - mu;
            v[6] = b.z - mu;
            v[7] = b.w - mu;
        } else {
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = (r < n && i0 + q < m) ? x[i0 + q] - mu : 0.f;
        }
        store8(hi, lo, umma::slice_offset(r, i0, mp >> 6), v);
    }
}

// [S d]^T as slices: row i < m is member i's observed-anomaly slopes / sigma, row m the innovation
// (y - D x_bar) / sigma, the rest zero.  The order of the slopes is free (the Gram sums over them): columns
// 16 g .. 16 g + 7 are the x slopes of subapertures 8 g .. 8 g + 7, the next eight their y slopes, padded
// with zeros, so that a thread (one row, one group) takes both from the same corners, and a corner that two
// neighbouring subapertures share once: 16 to 18 loads for 16 slopes, where one thread per 8 slopes of one
// kind loaded 32 (34 us at n_subv = 4632, m = 1024; this 22).
__global__ void __launch_bounds__(256) gl_slopes_kernel(const float* __restrict__ X, const float* __restrict__ xbar,
                                                        const float* __restrict__ y, const int4* __restrict__ corner,
                                                        int n_subv, int row_obs, int m, int m_pad, int mr, int pk,
                                                        float inv_sigma, uint8_t* __restrict__ hi,
                                                        uint8_t* __restrict__ lo) {
    const size_t total = (size_t)mr * (pk >> 4);
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < total; t += (size_t)gridDim.x * blockDim.x) {
        const int i = (int)(t % mr), g = (int)(t / mr), k0 = 8 * g;
        float sx[8], sy[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) sx[q] = sy[q] = 0.f;
        if (i <= m && k0 < n_subv) {
            const float* x = i < m ? X + (size_t)row_obs * m_pad + i : nullptr;
            auto at = [&](int act) {
                const float b = xbar[row_obs + act];
                return i < m ? x[(size_t)act * m_pad] - b : b;
            };
            int4 c[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) c[q] = corner[min(k0 + q, n_subv - 1)];
            float r0[8], r1[8];               // the right-hand corners
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                r0[q] = at(c[q].y);
                r1[q] = at(c[q].w);
            }
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                float l0, l1;                 // the left-hand ones: usually the neighbour's right
                if (q > 0 && c[q].x == c[q > 0 ? q - 1 : 0].y && c[q].z == c[q > 0 ? q - 1 : 0].w) {
                    l0 = r0[q > 0 ? q - 1 : 0];
                    l1 = r1[q > 0 ? q - 1 : 0];
                } else {
                    l0 = at(c[q].x);
                    l1 = at(c[q].z);
                }
                const float dx = 0.5f * ((r0[q] + r1[q]) - (l0 + l1)), dy = 0.5f * ((l1 + r1[q]) - (l0 + r0[q]));
                if (k0 + q < n_subv) {
                    sx[q] = (i < m ? dx : y[k0 + q] - dx) * inv_sigma;
                    sy[q] = (i < m ? dy : y[n_subv + k0 + q] - dy) * inv_sigma;
                }
            }
        }
        const size_t off = umma::slice_offset(i, 16 * g, pk >> 6);
        store8(hi, lo, off, sx);
        store8(hi, lo, off + 128, sy);
    }
}

// a rejected frame (non-finite slopes) leaves the ensemble as it was
__global__ void gl_reject_kernel(const float* __restrict__ X, float* __restrict__ Xo, size_t count,
                                 const int* __restrict__ frame_bad) {
    if (!*frame_bad) return;
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < count; t += (size_t)gridDim.x * blockDim.x)
        Xo[t] = X[t];
}

// xi^T slices for the noise product: element (member i, actuator j) = Philox normal (stream 1,
// frame, counter (j / 4, i)), the same draws as the plain forecast's white-noise path.  One thread per
// member and eight actuators: a warp writes pieces of 128 bytes.
__global__ void __launch_bounds__(256) gl_normals_kernel(unsigned long long seed, uint32_t frame, int n_act, int m, int mp,
                                                         int ka, uint8_t* __restrict__ hi, uint8_t* __restrict__ lo) {
    const size_t total = (size_t)mp * (ka >> 3);
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < total; t += (size_t)gridDim.x * blockDim.x) {
        const int g = (int)(t / mp), i = (int)(t - (size_t)g * mp);
        float z[8];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float w[4] = {0.f, 0.f, 0.f, 0.f};
            if (i < m && 8 * g + 4 * h < n_act) normals4<float>(seed, 1u, frame, (uint32_t)i, (uint32_t)(2 * g + h), w);
#pragma unroll
            for (int r = 0; r < 4; ++r) z[4 * h + r] = 8 * g + 4 * h + r < n_act ? w[r] : 0.f;
        }
        store8(hi, lo, umma::slice_offset(i, 8 * g, ka >> 6), z);
    }
}

int grid_for(size_t work, int block) {
    return (int)std::max<size_t>(1, std::min<size_t>((work + block - 1) / block, 152 * 16));
}

GemmArgs gemm_args(const uint8_t* ah, const uint8_t* al, const uint8_t* bh, const uint8_t* bl, int nkb, int M,
                   int N, int* status) {
    GemmArgs g{};
    g.a_hi = ah;
    g.a_lo = al;
    g.b_hi = bh;
    g.b_lo = bl;
    g.a_nkb = g.b_nkb = nkb;
    g.split = 1;
    g.M = M;
    g.N = N;
    g.status = status;
    return g;
}

}  // namespace

size_t global_bytes(int n_act, int n_subv, int m, bool dense, bool lower, int sms) {
    const int mr = rup(m + 1, 128), pk = slope_cols(n_subv), mp = rup(m, 128), nr = rup(2 * n_act, 128);
    const int ka = rup(n_act, 64);
    const size_t gram = (size_t)m * rup(m + 1, 4) * 4;
    const Plans P = plans_for(n_act, n_subv, m, dense, lower, sms);
    // [S d]^T, the Gram and its shares, A_s, T, Y (2), Z (2), X', W^T (hi and lo each)
    size_t b = 2 * tiled_bytes(mr, pk) + gram * (1 + P.split) + 12 * tiled_bytes(mp, mp) + 2 * tiled_bytes(nr, mp) +
               2 * tiled_bytes(mp, mp);
    if (dense) b += 2 * tiled_bytes(rup(n_act, 128), ka) + 2 * tiled_bytes(mp, ka);
    for (const GemmPlan* p : {&P.gram, &P.tr, &P.tr1, &P.noise}) b += p->bytes();
    b += (size_t)2 * n_act * 4 + (size_t)4 * m * 4 + (size_t)root_parts(m) * 4 + sizeof(RootStats) + ROOT_STEPS * 4 + 8 +
         (size_t)n_subv * 16;
    return b;
}

int global_prepare(letkf_ctx* c) {
    GlobalState* S = new GlobalState;
    c->gstate = S;
    const int m = c->m;
    S->mr = rup(m + 1, 128);
    S->pk = slope_cols(c->n_subv);
    S->mp = rup(m, 128);
    S->nr = rup(c->n, 128);
    S->ka = rup(c->n_act, 64);
    const bool dense = c->Lq != nullptr;
    auto get = [&](size_t bytes, void** p) {
        if (cudaMalloc(p, bytes) != cudaSuccess) return false;
        S->allocs.push_back(*p);
        c->device_bytes += bytes;
        return true;
    };
    bool ok = true;
    const size_t tst = tiled_bytes(S->mr, S->pk), tsq = tiled_bytes(S->mp, S->mp);
    ok = ok && get(tst, (void**)&S->st_hi) && get(tst, (void**)&S->st_lo);
    Plans P = plans_for(c->n_act, c->n_subv, m, dense, c->lq_lower != 0, c->sms);
    S->ldg = rup(m + 1, 4);
    S->gram_split = P.split;
    ok = ok && get((size_t)m * S->ldg * 4, (void**)&S->G) &&
         get((size_t)P.split * m * S->ldg * 4, (void**)&S->Gpart);
    for (auto& q : {std::make_pair(&P.gram, &S->pl_gram), std::make_pair(&P.tr, &S->pl_tr),
                    std::make_pair(&P.tr1, &S->pl_tr1),
                    std::make_pair(&P.noise, &S->pl_noise)}) {
        GemmPlan& p = *q.first;
        if (!p.ncta) continue;
        const size_t bi = p.items.size() * sizeof(int4), bs = p.start.size() * sizeof(int);
        ok = ok && get(bi, (void**)&p.d_items) && get(bs, (void**)&p.d_start);
        if (ok && (cudaMemcpy(p.d_items, p.items.data(), bi, cudaMemcpyHostToDevice) != cudaSuccess ||
                   cudaMemcpy(p.d_start, p.start.data(), bs, cudaMemcpyHostToDevice) != cudaSuccess))
            return LETKF_ECUDA;
        *q.second = std::move(p);
    }
    ok = ok && get(tsq, (void**)&S->as_hi) && get(tsq, (void**)&S->as_lo) && get(tsq, (void**)&S->t_hi) &&
         get(tsq, (void**)&S->t_lo);
    for (int q = 0; q < 2; ++q)
        ok = ok && get(tsq, (void**)&S->y_hi[q]) && get(tsq, (void**)&S->y_lo[q]) && get(tsq, (void**)&S->z_hi[q]) &&
             get(tsq, (void**)&S->z_lo[q]);
    const size_t txp = tiled_bytes(S->nr, S->mp);
    ok = ok && get(txp, (void**)&S->xp_hi) && get(txp, (void**)&S->xp_lo);
    ok = ok && get(tsq, (void**)&S->wt_hi) && get(tsq, (void**)&S->wt_lo);
    if (dense) {
        const size_t tl = tiled_bytes(rup(c->n_act, 128), S->ka), tx = tiled_bytes(S->mp, S->ka);
        ok = ok && get(tl, (void**)&S->l_hi) && get(tl, (void**)&S->l_lo) && get(tx, (void**)&S->xi_hi) &&
             get(tx, (void**)&S->xi_lo);
    }
    ok = ok && get((size_t)c->n * 4, (void**)&S->xbar) && get((size_t)root_parts(m) * 4, (void**)&S->sq) &&
         get((size_t)m * 4, (void**)&S->wbar) && get((size_t)m * 4, (void**)&S->u) && get((size_t)m * 4, (void**)&S->r) &&
         get((size_t)m * 4, (void**)&S->b) && get(sizeof(RootStats), (void**)&S->stats) &&
         get(ROOT_STEPS * 4, (void**)&S->dev) && get(8, (void**)&S->bar) && get((size_t)c->n_subv * 16, (void**)&S->corner);
    if (!ok) return LETKF_ENOMEM;
    // corner actuators of every valid subaperture: (r,c) (r,c+1) (r+1,c) (r+1,c+1)
    const HostModel& h = c->host;
    const int na = h.n_sub + 1;
    std::vector<int4> cor(c->n_subv);
    for (int k = 0; k < c->n_subv; ++k) {
        const int r = h.sub_rc[2 * k], cc = h.sub_rc[2 * k + 1];
        cor[k] = make_int4(h.act_index[(size_t)r * na + cc], h.act_index[(size_t)r * na + cc + 1],
                           h.act_index[(size_t)(r + 1) * na + cc], h.act_index[(size_t)(r + 1) * na + cc + 1]);
    }
    if (cudaMemcpy(S->corner, cor.data(), cor.size() * sizeof(int4), cudaMemcpyHostToDevice) != cudaSuccess)
        return LETKF_ECUDA;
    int rc = gemm_prepare();
    if (rc || (rc = root_prepare())) return rc;
    // slices of the process-noise factor, once
    if (dense && (rc = to_tiles(static_cast<const float*>(c->Lq), c->n_act, c->n_act, c->n_act, S->l_hi, S->l_lo, 1,
                                c->stream)))
        return rc;
    // zero the square buffers: products write columns up to m rounded to the CTA tile width only,
    // and the columns beyond (up to m rounded to 128) must read as zeros
    for (void* p : {(void*)S->as_hi, (void*)S->as_lo, (void*)S->t_hi, (void*)S->t_lo, (void*)S->y_hi[0],
                    (void*)S->y_lo[0], (void*)S->y_hi[1], (void*)S->y_lo[1], (void*)S->z_hi[0], (void*)S->z_lo[0],
                    (void*)S->z_hi[1], (void*)S->z_lo[1], (void*)S->wt_hi, (void*)S->wt_lo})
        if (cudaMemsetAsync(p, 0, tsq, c->stream) != cudaSuccess) return LETKF_ECUDA;
    if (dense && (cudaStreamCreateWithFlags(&S->side, cudaStreamNonBlocking) != cudaSuccess ||
                  cudaEventCreateWithFlags(&S->ev_fork, cudaEventDisableTiming) != cudaSuccess ||
                  cudaEventCreateWithFlags(&S->ev_join, cudaEventDisableTiming) != cudaSuccess))
        return LETKF_ECUDA;
    return LETKF_OK;
}

void global_free(letkf_ctx* c) {
    GlobalState* S = c->gstate;
    if (!S) return;
    if (S->side) {
        cudaStreamSynchronize(S->side);
        cudaStreamDestroy(S->side);
    }
    if (S->ev_fork) cudaEventDestroy(S->ev_fork);
    if (S->ev_join) cudaEventDestroy(S->ev_join);
    for (void* p : S->allocs) cudaFree(p);
    delete S;
    c->gstate = nullptr;
}

namespace {
int draw_normals(letkf_ctx* c, GlobalState* S, cudaStream_t stream) {
    gl_normals_kernel<<<grid_for((size_t)S->mp * (S->ka >> 3), 256), 256, 0, stream>>>(
        c->seed, (uint32_t)c->frame, c->n_act, c->m, S->mp, S->ka, S->xi_hi, S->xi_lo);
    return cudaGetLastError() == cudaSuccess ? LETKF_OK : LETKF_ECUDA;
}
}  // namespace

int global_analyze(letkf_ctx* c, const void* yv, double sigma, bool step) {
    GlobalState* S = c->gstate;
    if (!S) return LETKF_ESTATE;
    if (sigma > 0) c->sigma = sigma;
    cudaStream_t st = c->stream;
    const bool first_only = step && c->a2 == 0.0;
    // a step's normals (18 us at n_act = 4833, m = 1024) beside its analysis, most of which waits for memory
    // or at barriers; the product that reads them comes after it
    if (step && S->side) {
        if (cudaEventRecord(S->ev_fork, st) != cudaSuccess || cudaStreamWaitEvent(S->side, S->ev_fork, 0) != cudaSuccess ||
            draw_normals(c, S, S->side) != LETKF_OK || cudaEventRecord(S->ev_join, S->side) != cudaSuccess)
            return LETKF_ECUDA;
        S->forked = true;
    }
    int rc = launch_precheck(c, yv);
    if (rc) return rc;
    const float* X = static_cast<const float*>(c->X[c->cur]);
    float* Xo = static_cast<float*>(c->X[c->cur ^ 1]);
    const int m = c->m, n = c->n;
    const float cm = (float)(m - 1);
    prof_begin(c, STAGE_OBS);
    // rows of the analysis: both instants, or the first, which the AR(1) forecast makes both from
    const int rows = first_only ? c->n_act : n;
    gl_center_kernel<<<S->nr / 8, 256, 0, st>>>(X, n, rup(rows, 128), m, c->m_pad, S->mp, S->xbar, S->xp_hi, S->xp_lo, S->bar);
    gl_slopes_kernel<<<grid_for((size_t)S->mr * (S->pk >> 4), 256), 256, 0, st>>>(
        X, S->xbar, static_cast<const float*>(yv), S->corner, c->n_subv, c->obs_block == 1 ? c->n_act : 0, m, c->m_pad,
        S->mr, S->pk, (float)(1.0 / c->sigma), S->st_hi, S->st_lo);
    prof_end(c);
    if (cudaGetLastError() != cudaSuccess) return LETKF_ECUDA;
    // Gram [S d]^T [S d]
    prof_begin(c, STAGE_GRAM);
    // the upper tiles only (the Gram is symmetric), K split so that they fill the SMs
    GemmArgs g = gemm_args(S->st_hi, S->st_lo, S->st_hi, S->st_lo, S->pk >> 6, m, m + 1, c->d_status);
    g.mode = GEMM_EPI_F32;
    g.c = S->Gpart;
    g.ldc = S->ldg;
    g.c_split_stride = (size_t)m * S->ldg;
    if ((rc = gemm_launch(g, S->pl_gram, st))) return rc;
    prof_end(c);
    // Gram, inverse square root, weights
    prof_begin(c, STAGE_EIG);
    RootArgs ra;
    std::memset(&ra, 0, sizeof(ra));
    ra.part = S->Gpart;
    ra.stride = (size_t)m * S->ldg;
    ra.splits = S->gram_split;
    ra.m = m;
    ra.mp = S->mp;
    ra.ldg = S->ldg;
    ra.c = cm;
    ra.G = S->G;
    ra.as_hi = S->as_hi;
    ra.as_lo = S->as_lo;
    ra.t_hi = S->t_hi;
    ra.t_lo = S->t_lo;
    for (int q = 0; q < 2; ++q) {
        ra.y_hi[q] = S->y_hi[q];
        ra.y_lo[q] = S->y_lo[q];
        ra.z_hi[q] = S->z_hi[q];
        ra.z_lo[q] = S->z_lo[q];
    }
    ra.wt_hi = S->wt_hi;
    ra.wt_lo = S->wt_lo;
    ra.sq = S->sq;
    ra.b = S->b;
    ra.r = S->r;
    ra.u = S->u;
    ra.wbar = S->wbar;
    ra.dev = S->dev;
    ra.bar = S->bar;
    ra.stats = S->stats;
    ra.frame_bad = c->d_frame_bad;
    ra.status = c->d_status;
    if ((rc = root_launch(ra, c->sms, st))) return rc;
    prof_end(c);
    // transform X_a = x_bar + X' W
    prof_begin(c, STAGE_TRANSFORM);
    g = gemm_args(S->xp_hi, S->xp_lo, S->wt_hi, S->wt_lo, S->mp >> 6, rows, m, c->d_status);
    g.mode = GEMM_EPI_ADD_ROW;
    g.c = Xo;
    g.ldc = c->m_pad;
    g.add = S->xbar;
    if ((rc = gemm_launch(g, first_only ? S->pl_tr1 : S->pl_tr, st))) return rc;
    gl_reject_kernel<<<152, 256, 0, st>>>(X, Xo, (size_t)n * c->m_pad, c->d_frame_bad);
    prof_end(c);
    return cudaGetLastError() == cudaSuccess ? LETKF_OK : LETKF_ECUDA;
}

int global_forecast(letkf_ctx* c, const void* v_user, void* xpred, int in_analysis, bool step) {
    GlobalState* S = c->gstate;
    const bool first_only = step && c->a2 == 0.0;
    if (v_user || !c->Lq || !S) return launch_forecast(c, v_user, xpred, in_analysis, first_only);
    // V = L xi on the tensor cores (FP32-level), into c->V with leading dimension m
    prof_begin(c, STAGE_NOISE);
    // (outside a step there is only something to wait for when one failed between its halves)
    if (S->forked) {
        if (cudaStreamWaitEvent(c->stream, S->ev_join, 0) != cudaSuccess) return LETKF_ECUDA;
        S->forked = false;
    }
    if (!step) {
        const int rd = draw_normals(c, S, c->stream);
        if (rd) return rd;
    }
    GemmArgs g = gemm_args(S->l_hi, S->l_lo, S->xi_hi, S->xi_lo, S->ka >> 6, c->n_act, c->m, c->d_status);
    g.mode = GEMM_EPI_F32;
    g.c = static_cast<float*>(c->V);
    g.ldc = c->m;
    const int rc = gemm_launch(g, S->pl_noise, c->stream);
    prof_end(c);
    if (rc) return rc;
    return launch_forecast(c, c->V, xpred, in_analysis, first_only);
}

}  // namespace letkf

// Newton-Schulz steps of the last global analysis (the first, product-free step included) and the
// bound s it scaled by; synchronises the context's stream.
extern "C" int letkf_global_stats(letkf_ctx* c, int* ns_steps, double* s_bound) {
    using namespace letkf;
    if (!c || !ns_steps || !s_bound) return LETKF_EINVAL;
    GlobalState* S = c->gstate;
    if (!S) return LETKF_ESTATE;
    RootStats st;
    if (cudaSetDevice(c->device) != cudaSuccess || cudaStreamSynchronize(c->stream) != cudaSuccess ||
        cudaMemcpy(&st, S->stats, sizeof(st), cudaMemcpyDeviceToHost) != cudaSuccess)
        return LETKF_ECUDA;
    *ns_steps = st.steps;
    *s_bound = st.s;
    return LETKF_OK;
}
