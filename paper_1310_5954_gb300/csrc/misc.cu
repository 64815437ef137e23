// Frame ingest check, process-noise draws, AR(1) forecast and initial ensemble.
//
// Forecast (Sect. 2.1): A1 = [[a I, 0], [I, 0]] on the two-instant state, so per
// member: second instant <- first, first <- a * first + v.  The perturbation is
// v = L xi with xi counter-based Philox4x32-10 normals (stream 1, frame k); with
// a dense L the product is one GEMM per frame (FP64 / FP32: row_gemm_kernel below on the
// CUDA cores; mixed precision: the BF16 tensor-core kernel of noise.cu), with white noise it is
// drawn inline.

#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "common.cuh"
#include "internal.hpp"
#include "umma.cuh"

namespace letkf {
namespace {

// Slope check of a frame: any NaN/Inf rejects the frame.  Also resets the work-queue counter
// of the fused kernel that follows in stream order.
template <typename T>
__global__ void precheck_kernel(const T* __restrict__ y, int p, int* frame_bad, int* status, int* queue) {
    __shared__ int bad;
    if (threadIdx.x == 0) {
        bad = 0;
        queue[0] = 0;
    }
    __syncthreads();
    int mine = 0;
    for (int i = threadIdx.x; i < p; i += blockDim.x)
        if (!finite_val(y[i])) mine = 1;
    if (mine) atomicOr(&bad, 1);
    __syncthreads();
    if (threadIdx.x == 0) {
        *frame_bad = bad;
        if (bad) atomicOr(status, ST_NONFINITE);
    }
}

// xi[j, i] for j < n_act, i < m: one Philox call gives four consecutive j.
template <typename O>
__global__ void normals_kernel(O* __restrict__ out, int ld, int n_act, int m, unsigned long long seed,
                               uint32_t stream, uint32_t frame) {
    const int nq = (n_act + 3) / 4;
    const int total = nq * m;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += gridDim.x * blockDim.x) {
        const int q = t / m, i = t - q * m;
        float zf[4];
        double zd[4];
        if (sizeof(O) == 8) {
            normals4<double>(seed, stream, frame, (uint32_t)i, (uint32_t)q, zd);
        } else {
            normals4<float>(seed, stream, frame, (uint32_t)i, (uint32_t)q, zf);
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int j = 4 * q + r;
            if (j < n_act) {
                if (sizeof(O) == 8)
                    out[(size_t)j * ld + i] = (O)zd[r];
                else
                    out[(size_t)j * ld + i] = (O)zf[r];
            }
        }
    }
}

// In-place forecast of the ensemble X (n x m_pad) and the mean of the new first instant.
// first_only: the second instant takes no part (AR(1)) and need not hold an analysis.
// vmode 0: v from V (ld vld); 1: white noise q * xi drawn inline; 2: no perturbation.
template <typename T>
__global__ void forecast_kernel(T* __restrict__ X, const T* __restrict__ V, int vld, int vmode, T q_white,
                                T a, T a2, int n_act, int m, int m_pad, T* __restrict__ xpred,
                                const int* __restrict__ frame_bad, int check_bad, unsigned long long seed,
                                uint32_t frame, int first_only) {
    const bool skip = check_bad && *frame_bad;
    const int lane = threadIdx.x & 31;
    const int warps = (gridDim.x * blockDim.x) >> 5;
    for (int j = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; j < n_act; j += warps) {
        T* x1 = X + (size_t)j * m_pad;
        T* x2 = X + (size_t)(n_act + j) * m_pad;
        T s = 0;
        // four members per lane per pass, their loads issued before any store (large ensembles)
        for (int i0 = lane; i0 < m; i0 += 128) {
            T v1[4], v2[4], v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int i = i0 + 32 * u;
                v1[u] = i < m ? x1[i] : (T)0;
                v2[u] = (i < m && !skip && !first_only) ? x2[i] : (T)0;
                v[u] = (i < m && !skip && vmode == 0) ? V[(size_t)j * vld + i] : (T)0;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int i = i0 + 32 * u;
                if (i >= m) continue;
                if (!skip) {
                    if (vmode == 1) {
                        T z[4];
                        normals4<T>(seed, 1u, frame, (uint32_t)i, (uint32_t)(j >> 2), z);
                        v[u] = q_white * z[j & 3];
                    }
                    x2[i] = v1[u];
                    v1[u] = a * v1[u] + a2 * v2[u] + v[u];
                    x1[i] = v1[u];
                }
                s += v1[u];
            }
        }
        s = warp_sum(s);
        if (xpred && lane == 0) xpred[j] = s / (T)m;
    }
}

template <typename T>
__global__ void axpy_rows_kernel(T* __restrict__ dst, const T* __restrict__ src, T alpha, T beta, int rows,
                                 int cols, int ld) {
    // dst = alpha * dst + beta * src (rows x cols, leading dimension ld)
    const size_t total = (size_t)rows * cols;
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < total; t += (size_t)gridDim.x * blockDim.x) {
        const size_t r = t / cols, cidx = t - r * cols;
        dst[r * ld + cidx] = alpha * dst[r * ld + cidx] + beta * src[r * ld + cidx];
    }
}

__global__ void f64_to_f32(const double* __restrict__ in, float* __restrict__ out, size_t n) {
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < n; t += (size_t)gridDim.x * blockDim.x)
        out[t] = (float)in[t];
}

int grid_for(size_t work, int block) {
    size_t g = (work + block - 1) / block;
    if (g > 8192) g = 8192;
    if (g < 1) g = 1;
    return (int)g;
}

// V (n x m, row stride ldv) = L (n x n, row-major) * Xi (n x m, row stride ldx), in the state type
// on the CUDA cores.  A CTA computes a 64 x 64 tile of V: 256 threads, each a 4 x 4 register block
// (rows ty + 16 i, columns tx + 16 j, so that a warp's shared-memory reads hit distinct banks),
// over K steps of 16 staged in shared memory, the next step's tile prefetched into registers while
// the current one is multiplied.  With a lower-triangular L the K loop of a row block stops at its
// last row (the zero upper triangle is never read).  Every sum runs over k in increasing order.
constexpr int RG_BM = 64, RG_BN = 64, RG_BK = 16, RG_THREADS = 256;

template <typename T>
__global__ void __launch_bounds__(RG_THREADS) row_gemm_kernel(const T* __restrict__ L, const T* __restrict__ Xi,
                                                              T* __restrict__ V, int n, int m, int ldx, int ldv,
                                                              int lower) {
    __shared__ T As[RG_BK][RG_BM + 1];   // As[k][row]: L tile, transposed
    __shared__ T Bs[RG_BK][RG_BN];       // Bs[k][col]: Xi tile
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int r0 = blockIdx.x * RG_BM, c0 = blockIdx.y * RG_BN;
    const int kend = lower ? min(n, r0 + RG_BM) : n;
    // loads: A, 64 rows x 16 k, thread -> row tid / 4, k 4 (tid % 4) .. + 3;
    //        B, 16 k x 64 columns, thread -> k tid / 16, columns 4 (tid % 16) .. + 3
    const int ar = tid >> 2, ak = 4 * (tid & 3);
    const int bk = tid >> 4, bc = 4 * (tid & 15);
    T ra[4], rb[4];
    auto fetch = [&](int k0) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int r = r0 + ar, k = k0 + ak + u;
            ra[u] = (r < n && k < kend) ? L[(size_t)r * n + k] : T(0);
            const int kk = k0 + bk, cc = c0 + bc + u;
            rb[u] = (kk < kend && cc < m) ? Xi[(size_t)kk * ldx + cc] : T(0);
        }
    };
    T acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = T(0);
    if (kend > 0) fetch(0);
    for (int k0 = 0; k0 < kend; k0 += RG_BK) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            As[ak + u][ar] = ra[u];
            Bs[bk][bc + u] = rb[u];
        }
        __syncthreads();
        if (k0 + RG_BK < kend) fetch(k0 + RG_BK);
#pragma unroll
        for (int k = 0; k < RG_BK; ++k) {
            T a[4], b[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) a[i] = As[k][ty + 16 * i];
#pragma unroll
            for (int j = 0; j < 4; ++j) b[j] = Bs[k][tx + 16 * j];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int r = r0 + ty + 16 * i;
        if (r >= n) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int cc = c0 + tx + 16 * j;
            if (cc < m) V[(size_t)r * ldv + cc] = acc[i][j];
        }
    }
}

// The per-frame draw V = L Xi in the state type on the CUDA cores.  Both operands are laid out for
// bulk copies: L once, at creation, as chunks of 16 values of k by BM rows (k-major, so that a
// thread's rows are adjacent; a lower-triangular factor keeps the chunks up to each row block's last
// row only), Xi by its generator as 16 rows of BN columns.  A work item is a BM x BN tile of V over a
// run of chunks: one thread refills a ring of four chunk pairs, 256 threads compute TM x TN register
// blocks (TM adjacent rows, columns tx + CX j).  A row block's chunks are split into runs of equal
// length so that all items together fill two CTAs per SM once; a split tile's runs go to the scratch
// and rg_reduce_kernel adds them in order, so the result does not depend on scheduling.
//
// What bounds it: the FMA pipe (an 8 x 7 block does 56 multiply-adds per 9 shared-memory reads), in
// FP64 the two FP64 lanes of an SM: there the tiles are 32 rows by 8 TN columns, so that few of the
// multiply-adds are padding.  Measured, normals and product (before: 64 x 128 tiles of K pieces of
// 512, scalar loads, the last CTA of a tile summing its pieces): 69 actuators, m = 20, FP64 180 -> 21 us;
// 1 353, m = 50, FP32 93 -> 22 us; 4 836, m = 100, FP32 frame 242 -> 192 us (the draw runs beside it).
constexpr int RK_KC = 16, RK_STAGES = 4, RK_THREADS = 256, RK_ITEMS = 2 * 152;
constexpr long long RK_WAIT = 4000000000LL;

// Chunks before row block rb (nk: chunks of a full row).
__host__ __device__ inline size_t rk_prefix(int rb, int bm, int nk, int lower) {
    return lower ? (size_t)(bm / RK_KC) * rb * (rb + 1) / 2 : (size_t)rb * nk;
}

template <typename T, int CX, int TM, int TN>
__global__ void __launch_bounds__(RK_THREADS, 2) rg_kernel(const T* __restrict__ Lt, const T* __restrict__ Xi,
                                                           T* __restrict__ V, int n, int m, int ldv, int lower,
                                                           const int4* __restrict__ items,
                                                           const int4* __restrict__ tiles, T* __restrict__ part,
                                                           int* __restrict__ status) {
    constexpr int RX = RK_THREADS / CX, BM = RX * TM, BN = CX * TN;
    constexpr uint32_t A_B = RK_KC * BM * sizeof(T), B_B = RK_KC * BN * sizeof(T);
    extern __shared__ __align__(128) unsigned char rk_smem[];
    __shared__ __align__(8) uint64_t full[RK_STAGES];
    const int tid = threadIdx.x, tx = tid % CX, ty = tid / CX;
    const int4 it = items[blockIdx.x];   // tile, first chunk, end chunk, run
    const int4 tl = tiles[it.x];         // row block, column block, runs, first scratch slot
    const int nk = (n + RK_KC - 1) / RK_KC, nc = it.z - it.y;
    const unsigned char* ga = reinterpret_cast<const unsigned char*>(Lt) + (rk_prefix(tl.x, BM, nk, lower) + it.y) * A_B;
    const unsigned char* gb = reinterpret_cast<const unsigned char*>(Xi) + ((size_t)tl.y * nk + it.y) * B_B;
    auto load = [&](int c) {
        const int s = c % RK_STAGES;
        unsigned char* st = rk_smem + s * (A_B + B_B);
        umma::mbar_arrive_expect_tx(&full[s], A_B + B_B);
        umma::bulk_g2s(st, ga + (size_t)c * A_B, A_B, &full[s]);
        umma::bulk_g2s(st + A_B, gb + (size_t)c * B_B, B_B, &full[s]);
    };
    if (tid == 0) {
        for (int s = 0; s < RK_STAGES; ++s) umma::mbar_init(&full[s], 1);
        umma::fence_mbar_init();
    }
    __syncthreads();
    const int uwarp = umma::uniform_warp();
    if (uwarp == 0 && umma::elect_one())
        for (int c = 0; c < nc && c < RK_STAGES; ++c) load(c);
    T acc[TM][TN];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = T(0);
    int issued = min(nc, RK_STAGES), done = 0;
    bool ok = true;
    for (int c = 0; c < nc; ++c) {
        const int s = c % RK_STAGES;
        ok = umma::mbar_wait_bounded(&full[s], (uint32_t)((c / RK_STAGES) & 1), RK_WAIT);
        if (ok) {
            const T* As = reinterpret_cast<const T*>(rk_smem + s * (A_B + B_B));
            const T* Bs = As + RK_KC * BM;
#pragma unroll
            for (int k = 0; k < RK_KC; ++k) {
                T a[TM], b[TN];
                if constexpr (TM % 4 == 0 && sizeof(T) == 4) {
#pragma unroll
                    for (int i = 0; i < TM; i += 4) {
                        const float4 v = *reinterpret_cast<const float4*>(As + k * BM + ty * TM + i);
                        a[i] = v.x; a[i + 1] = v.y; a[i + 2] = v.z; a[i + 3] = v.w;
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < TM; ++i) a[i] = As[k * BM + ty * TM + i];
                }
#pragma unroll
                for (int j = 0; j < TN; ++j) b[j] = Bs[k * BN + tx + CX * j];
#pragma unroll
                for (int i = 0; i < TM; ++i)
#pragma unroll
                    for (int j = 0; j < TN; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
            }
        }
        done = c + 1;
        if (__syncthreads_or(!ok)) break;          // the stage is read by every warp: it can be refilled
        if (c + RK_STAGES < nc) {
            if (uwarp == 0 && umma::elect_one()) load(c + RK_STAGES);
            issued = c + RK_STAGES + 1;
        }
    }
    if (done < nc || !ok) {
        // a copy did not land in time: the ones in flight get a bounded time before the CTA leaves
        if (tid == 0) {
            atomicOr(status, ST_TIMEOUT);
            for (int c = done; c < issued; ++c)
                umma::mbar_wait_bounded(&full[c % RK_STAGES], (uint32_t)((c / RK_STAGES) & 1), RK_WAIT / 8);
        }
        return;
    }
    const int r0 = tl.x * BM + ty * TM, c0 = tl.y * BN + tx;
    if (tl.z == 1) {
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int j = 0; j < TN; ++j)
                if (r0 + i < n && c0 + CX * j < m) V[(size_t)(r0 + i) * ldv + c0 + CX * j] = acc[i][j];
        return;
    }
    T* mine = part + (size_t)(tl.w + it.w) * BM * BN + (size_t)ty * TM * BN + tx;
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) mine[i * BN + CX * j] = acc[i][j];
}

// Tiles split into runs: V = the sum of the runs' partial tiles, in order.  blockIdx.y: the tile;
// four columns per thread.
template <typename T>
__global__ void rg_reduce_kernel(const T* __restrict__ part, const int4* __restrict__ tiles, int bm, int bn,
                                 T* __restrict__ V, int n, int m, int ldv) {
    const int4 tl = tiles[blockIdx.y];
    const int e = blockIdx.x * blockDim.x + threadIdx.x, c4 = bn >> 2;
    if (tl.z == 1 || e >= bm * c4) return;
    const int r = e / c4, c = 4 * (e - r * c4), row = tl.x * bm + r, col = tl.y * bn + c;
    if (row >= n || col >= m) return;
    const T* p = part + (size_t)tl.w * bm * bn + (size_t)r * bn + c;
    T s[4] = {T(0), T(0), T(0), T(0)};
    for (int q = 0; q < tl.z; ++q, p += (size_t)bm * bn) {
        if constexpr (sizeof(T) == 4) {
            const float4 v = *reinterpret_cast<const float4*>(p);
            s[0] += v.x; s[1] += v.y; s[2] += v.z; s[3] += v.w;
        } else {
            const double2 v = *reinterpret_cast<const double2*>(p), w = *reinterpret_cast<const double2*>(p + 2);
            s[0] += v.x; s[1] += v.y; s[2] += w.x; s[3] += w.y;
        }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
        if (col + u < m) V[(size_t)row * ldv + col + u] = s[u];
}

// The normals of a draw in rg_kernel's layout: column block i / bn, then 16-row chunks of bn columns,
// which is row k of bn columns throughout.  Rows and columns past n_act and m keep the zeros the
// buffer was made with.
template <typename O>
__global__ void rg_normals_kernel(O* __restrict__ out, int bn, int n_act, int m, unsigned long long seed,
                                  uint32_t stream, uint32_t frame) {
    const int nq = (n_act + 3) / 4, total = nq * m;
    const size_t krows = (size_t)(n_act + RK_KC - 1) / RK_KC * RK_KC;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += gridDim.x * blockDim.x) {
        const int q = t / m, i = t - q * m;
        O z[4];
        normals4<O>(seed, stream, frame, (uint32_t)i, (uint32_t)q, z);
        O* o = out + ((size_t)(i / bn) * krows + 4 * q) * bn + i % bn;
#pragma unroll
        for (int r = 0; r < 4; ++r)
            if (4 * q + r < n_act) o[(size_t)r * bn] = z[r];
    }
}

// L (FP64, row-major) into rg_kernel's chunks: element (row block, chunk, k, row).
template <typename T>
__global__ void rg_pack_kernel(const double* __restrict__ L, T* __restrict__ Lt, int n, int bm, int lower) {
    const int rb = blockIdx.y, nk = (n + RK_KC - 1) / RK_KC;
    const int kend = lower ? min(n, (rb + 1) * bm) : n, chunks = (kend + RK_KC - 1) / RK_KC;
    T* out = Lt + rk_prefix(rb, bm, nk, lower) * RK_KC * bm;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < chunks * RK_KC * bm; e += gridDim.x * blockDim.x) {
        const int k = e / bm, row = rb * bm + e - k * bm;
        out[e] = (row < n && k < kend) ? (T)L[(size_t)row * n + k] : T(0);
    }
}

// Tile shape of a draw: FP32 rows by the size of the system (large tiles where there are enough of
// them to fill the SMs), FP64 always 32; the columns split evenly into blocks of at most 128 (FP64:
// 64), each rounded up to a width rg_launch has.
struct RkShape {
    int cx, tm, tn, bm, bn, ncb, nrb, nk;
};
RkShape rk_shape(int n, int m, size_t eb) {
    RkShape s;
    const int most = eb == 8 ? 64 : 128;
    s.cx = eb == 8 ? 8 : 16;
    s.tm = eb == 8 ? 1 : (n >= 2048 ? 8 : n >= 512 ? 4 : 2);
    s.ncb = (m + most - 1) / most;
    const int w = (m + s.ncb - 1) / s.ncb;
    static const int w4[] = {2, 4, 6, 7, 8}, w8[] = {3, 5, 8};
    const int* ws = eb == 8 ? w8 : w4;
    while (*ws * s.cx < w) ++ws;
    s.tn = *ws;
    s.bm = RK_THREADS / s.cx * s.tm;
    s.bn = s.cx * s.tn;
    s.nrb = (n + s.bm - 1) / s.bm;
    s.nk = (n + RK_KC - 1) / RK_KC;
    return s;
}

template <typename T, typename F>
int rk_with(const RkShape& s, F&& f) {     // f(kernel of this shape)
#define RK_CASE(CX, TM, TN) \
    if (s.cx == CX && s.tm == TM && s.tn == TN) return f(rg_kernel<T, CX, TM, TN>)
    if constexpr (sizeof(T) == 8) {
        RK_CASE(8, 1, 3);
        RK_CASE(8, 1, 5);
        RK_CASE(8, 1, 8);
    } else {
        RK_CASE(16, 2, 2); RK_CASE(16, 2, 4); RK_CASE(16, 2, 6); RK_CASE(16, 2, 7); RK_CASE(16, 2, 8);
        RK_CASE(16, 4, 2); RK_CASE(16, 4, 4); RK_CASE(16, 4, 6); RK_CASE(16, 4, 7); RK_CASE(16, 4, 8);
        RK_CASE(16, 8, 2); RK_CASE(16, 8, 4); RK_CASE(16, 8, 6); RK_CASE(16, 8, 7); RK_CASE(16, 8, 8);
    }
#undef RK_CASE
    return LETKF_EINVAL;
}

int rk_smem_bytes(const RkShape& s, size_t eb) { return RK_STAGES * RK_KC * (s.bm + s.bn) * (int)eb; }

template <typename T>
int rg_product(letkf_ctx* c, const void* xi, void* V, cudaStream_t stream) {
    const int n = c->n_act, m = c->m;
    const RkShape s = rk_shape(n, m, sizeof(T));
    const int rc = rk_with<T>(s, [&](auto* k) -> int {
        k<<<c->rg_n_items, RK_THREADS, rk_smem_bytes(s, sizeof(T)), stream>>>(
            (const T*)c->Lq, (const T*)xi, (T*)V, n, m, c->m_pad, c->lq_lower, (const int4*)c->rg_items,
            (const int4*)c->rg_tiles, (T*)c->rg_part, c->d_status);
        return cudaGetLastError() == cudaSuccess ? LETKF_OK : LETKF_ECUDA;
    });
    if (rc || !c->rg_part) return rc;
    rg_reduce_kernel<T><<<dim3((s.bm * (s.bn >> 2) + 255) / 256, s.nrb * s.ncb), 256, 0, stream>>>(
        (const T*)c->rg_part, (const int4*)c->rg_tiles, s.bm, s.bn, (T*)V, n, m, c->m_pad);
    return cudaGetLastError() == cudaSuccess ? LETKF_OK : LETKF_ECUDA;
}

// FP64 / FP32: V (n_act x m, ld m_pad) = L (n_act x n_act, row-major) * Xi (n_act x m, ld xld) on
// `stream`.  (Mixed precision uses noise.cu.)  The per-frame draw uses the split-K kernel and the
// context's work tables; the initial ensemble's products (once) the plain row_gemm_kernel.
int noise_gemm(letkf_ctx* c, const void* L, const void* Xi, int xld, int gemm_type, void* V, cudaStream_t stream,
               bool lower) {
    const int m = c->m, na = c->n_act;
    const dim3 grid((na + RG_BM - 1) / RG_BM, (m + RG_BN - 1) / RG_BN);
    if (gemm_type == 0)
        row_gemm_kernel<double><<<grid, RG_THREADS, 0, stream>>>((const double*)L, (const double*)Xi, (double*)V, na,
                                                                 m, xld, c->m_pad, lower ? 1 : 0);
    else if (gemm_type == 1)
        row_gemm_kernel<float><<<grid, RG_THREADS, 0, stream>>>((const float*)L, (const float*)Xi, (float*)V, na, m,
                                                                xld, c->m_pad, lower ? 1 : 0);
    else
        return LETKF_EINVAL;
    return cudaGetLastError() == cudaSuccess ? LETKF_OK : LETKF_ECUDA;
}

int gemm_type_of(const letkf_ctx* c) {
    return c->precision == LETKF_PREC_FP64 ? 0 : (c->precision == LETKF_PREC_FP32 ? 1 : 2);
}

}  // namespace

int draw_perturbations_impl(letkf_ctx* c, unsigned long long frame);

int launch_precheck(letkf_ctx* c, const void* y) {
    prof_begin(c, STAGE_CHECK);
    if (c->precision == LETKF_PREC_FP64)
        precheck_kernel<double><<<1, 1024, 0, c->stream>>>((const double*)y, c->p, c->d_frame_bad, c->d_status,
                                                            c->d_queue);
    else
        precheck_kernel<float><<<1, 1024, 0, c->stream>>>((const float*)y, c->p, c->d_frame_bad, c->d_status,
                                                           c->d_queue);
    prof_end(c);
    return cudaGetLastError() == cudaSuccess ? LETKF_OK : LETKF_ECUDA;
}

int draw_perturbations(letkf_ctx* c, unsigned long long frame) {
    prof_begin(c, STAGE_NOISE);
    const int rc = draw_perturbations_impl(c, frame);
    prof_end(c);
    return rc;
}

int draw_perturbations_impl(letkf_ctx* c, unsigned long long frame) {
    return draw_perturbations_on(c, frame, c->Xi, c->V, c->stream);
}

// The per-frame product (factor and work tables made by rg_prepare).
int rg_draw_product(letkf_ctx* c, const void* Xi, void* V, cudaStream_t stream) {
    if (c->rg_n_items < 1) return LETKF_EINVAL;
    return c->precision == LETKF_PREC_FP64 ? rg_product<double>(c, Xi, V, stream) : rg_product<float>(c, Xi, V, stream);
}

int draw_perturbations_on(letkf_ctx* c, unsigned long long frame, void* xi, void* v_out, cudaStream_t stream) {
    if (c->Lt) return noise_draw(c, frame, xi, v_out, stream);
    NormalsNode nn;
    normals_node_params(c, frame, xi, &nn);
    if (cudaLaunchKernel(nn.params.func, nn.params.gridDim, nn.params.blockDim, nn.args, 0, stream) != cudaSuccess)
        return LETKF_ECUDA;
    return rg_draw_product(c, xi, v_out, stream);
}

int draw_product_on(letkf_ctx* c, const void* xi, void* v_out, cudaStream_t stream) {
    if (c->Lt) return noise_product(c, xi, v_out, stream);
    return rg_draw_product(c, xi, v_out, stream);
}

// Kernel-node parameters of the normals launch draw_perturbations_on makes for `frame` into xi
// (same function, grid and arguments), for updating that node of a captured graph.
int normals_node_params(letkf_ctx* c, unsigned long long frame, void* xi, NormalsNode* nn) {
    if (c->Lt) return noise_normals_params(c, frame, xi, nn);
    const int gt = gemm_type_of(c);
    const int nq = (c->n_act + 3) / 4;
    nn->out = xi;
    nn->ld = rk_shape(c->n_act, c->m, gt == 0 ? 8 : 4).bn;
    nn->n_act = c->n_act;
    nn->m = c->m;
    nn->seed = c->seed;
    nn->stream_id = 1u;
    nn->frame = (uint32_t)frame;
    nn->args[0] = &nn->out;
    nn->args[1] = &nn->ld;
    nn->args[2] = &nn->n_act;
    nn->args[3] = &nn->m;
    nn->args[4] = &nn->seed;
    nn->args[5] = &nn->stream_id;
    nn->args[6] = &nn->frame;
    cudaKernelNodeParams& kp = nn->params;
    kp.func = gt == 0 ? (void*)rg_normals_kernel<double> : (void*)rg_normals_kernel<float>;
    kp.gridDim = dim3(grid_for((size_t)nq * c->m, 128));
    kp.blockDim = dim3(128);
    kp.sharedMemBytes = 0;
    kp.kernelParams = nn->args;
    kp.extra = nullptr;
    return LETKF_OK;
}

namespace {

// Around a draw on the context's stream where there is a side stream that draws as well: the draws made there
// so far are done before it, and noise_side (fused.cu) has the later ones wait for it.  In a stream capture of the
// caller's the events are external ones: they count as they stand when the caller's graph runs.
bool capturing(letkf_ctx* c) {
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(c->stream, &st) == cudaSuccess) return st == cudaStreamCaptureStatusActive;
    cudaGetLastError();    // the legacy stream while another one is captured
    return false;
}

int draws_join(letkf_ctx* c) {
    if (!c->side) return LETKF_OK;
    const unsigned flag = capturing(c) ? cudaEventWaitExternal : cudaEventWaitDefault;
    for (cudaEvent_t ev : c->ev_v_ready)
        if (cudaStreamWaitEvent(c->stream, ev, flag) != cudaSuccess) return LETKF_ECUDA;
    return LETKF_OK;
}

int draws_fork(letkf_ctx* c) {
    if (!c->side) return LETKF_OK;
    const bool cap = capturing(c);
    if (cudaEventRecordWithFlags(c->ev_draw, c->stream, cap ? cudaEventRecordExternal : cudaEventRecordDefault) != cudaSuccess)
        return LETKF_ECUDA;
    c->draw_wait = cap ? 2 : std::max(c->draw_wait, 1);
    return LETKF_OK;
}

}  // namespace

int launch_forecast(letkf_ctx* c, const void* v_user, void* xpred, int in_analysis, bool first_only) {
    int vmode, vld;
    const void* Vp;
    if (v_user) {
        vmode = 0;
        Vp = v_user;
        vld = c->m;
    } else if (c->Lq || c->Lt) {
        int rc = draws_join(c);
        if (rc || (rc = draw_perturbations(c, c->frame)) || (rc = draws_fork(c))) return rc;
        vmode = 0;
        Vp = c->V;
        vld = c->m_pad;
    } else {
        vmode = c->q_white > 0 ? 1 : 2;
        Vp = nullptr;
        vld = 0;
    }
    const int g = grid_for((size_t)c->n_act * 32, 256);
    prof_begin(c, STAGE_FORECAST);
    if (c->precision == LETKF_PREC_FP64)
        forecast_kernel<double><<<g, 256, 0, c->stream>>>((double*)c->X[c->cur], (const double*)Vp, vld, vmode,
                                                          c->q_white, c->a, c->a2, c->n_act, c->m, c->m_pad,
                                                          (double*)xpred, c->d_frame_bad, in_analysis, c->seed,
                                                          (uint32_t)c->frame, first_only ? 1 : 0);
    else
        forecast_kernel<float><<<g, 256, 0, c->stream>>>((float*)c->X[c->cur], (const float*)Vp, vld, vmode,
                                                         (float)c->q_white, (float)c->a, (float)c->a2, c->n_act, c->m,
                                                         c->m_pad,
                                                         (float*)xpred, c->d_frame_bad, in_analysis, c->seed,
                                                         (uint32_t)c->frame, first_only ? 1 : 0);
    prof_end(c);
    return cudaGetLastError() == cudaSuccess ? LETKF_OK : LETKF_ECUDA;
}

RowGemmPlan rg_plan(int n, int m, bool lower, size_t eb, int* items, int* tiles) {
    const RkShape s = rk_shape(n, m, eb);
    auto chunks = [&](int rb) { return ((lower ? std::min(n, (rb + 1) * s.bm) : n) + RK_KC - 1) / RK_KC; };
    // the shortest run with which all items fit on the chip at once
    int run = 1;
    for (;; ++run) {
        long long n_items = 0;
        for (int rb = 0; rb < s.nrb; ++rb) n_items += (chunks(rb) + run - 1) / run;
        if (n_items * s.ncb <= RK_ITEMS || run >= s.nk) break;
    }
    RowGemmPlan P;
    P.l_elems = (rk_prefix(s.nrb - 1, s.bm, s.nk, lower) + chunks(s.nrb - 1)) * RK_KC * s.bm;
    P.xi_elems = (size_t)s.ncb * s.nk * RK_KC * s.bn;
    // the longest row blocks first
    for (int rb = s.nrb - 1; rb >= 0; --rb)
        for (int cb = 0; cb < s.ncb; ++cb) {
            const int ch = chunks(rb), np = (ch + run - 1) / run;
            if (tiles) {
                int* t = tiles + 4 * P.n_tiles;
                t[0] = rb; t[1] = cb; t[2] = np; t[3] = np > 1 ? P.n_slots : 0;
            }
            for (int p = 0; p < np; ++p) {
                if (items) {
                    int* it = items + 4 * P.n_items;
                    it[0] = P.n_tiles; it[1] = (int)((long long)p * ch / np); it[2] = (int)((long long)(p + 1) * ch / np);
                    it[3] = p;
                }
                ++P.n_items;
            }
            if (np > 1) P.n_slots += np;
            ++P.n_tiles;
        }
    P.part_elems = (size_t)P.n_slots * s.bm * s.bn;
    return P;
}

size_t rg_bytes(int n, int m, bool lower, size_t eb) {
    const RowGemmPlan P = rg_plan(n, m, lower, eb, nullptr, nullptr);
    return 16 * (size_t)P.n_items + 16 * (size_t)P.n_tiles + eb * (P.part_elems + P.l_elems + P.xi_elems);
}

size_t rg_xi_bytes(int n, int m, size_t eb) {
    const RkShape s = rk_shape(n, m, eb);
    return eb * (size_t)s.ncb * s.nk * RK_KC * s.bn;
}

// The factor in rg_kernel's layout (L64: FP64 row-major, on the device), normals buffer, work tables
// and scratch of the per-frame draw.
template <typename T>
int rg_prepare(letkf_ctx* c, const double* L64) {
    const int n = c->n_act, m = c->m;
    const bool lower = c->lq_lower != 0;
    const RkShape s = rk_shape(n, m, sizeof(T));
    const RowGemmPlan P = rg_plan(n, m, lower, sizeof(T), nullptr, nullptr);
    std::vector<int> items(4 * (size_t)P.n_items), tiles(4 * (size_t)P.n_tiles);
    rg_plan(n, m, lower, sizeof(T), items.data(), tiles.data());
    if (cudaMalloc(&c->Lq, P.l_elems * sizeof(T)) != cudaSuccess ||
        cudaMalloc(&c->Xi, P.xi_elems * sizeof(T)) != cudaSuccess ||
        cudaMalloc(&c->rg_items, items.size() * 4) != cudaSuccess ||
        cudaMalloc(&c->rg_tiles, tiles.size() * 4) != cudaSuccess)
        return LETKF_ENOMEM;
    if (P.part_elems && cudaMalloc(&c->rg_part, P.part_elems * sizeof(T)) != cudaSuccess) return LETKF_ENOMEM;
    if (cudaMemset(c->Xi, 0, P.xi_elems * sizeof(T)) != cudaSuccess ||
        cudaMemcpy(c->rg_items, items.data(), items.size() * 4, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(c->rg_tiles, tiles.data(), tiles.size() * 4, cudaMemcpyHostToDevice) != cudaSuccess)
        return LETKF_ECUDA;
    rg_pack_kernel<T><<<dim3(64, s.nrb), 256, 0, c->stream>>>(L64, (T*)c->Lq, n, s.bm, lower ? 1 : 0);
    if (cudaGetLastError() != cudaSuccess) return LETKF_ECUDA;
    c->rg_n_items = P.n_items;
    c->device_bytes += rg_bytes(n, m, lower, sizeof(T));
    // (the attribute belongs to the kernel: every context with this shape sets the same value)
    return rk_with<T>(s, [&](auto* k) -> int {
        return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, rk_smem_bytes(s, sizeof(T))) == cudaSuccess
                   ? LETKF_OK
                   : LETKF_ECUDA;
    });
}

// Initial ensemble (Sect. 2.2): second instant = P0 xi0, first = a * second + L xi1, with
// xi0, xi1 the Philox draws (stream 0, frames 0 and 1).  P0 defaults to L times the stationary
// standard deviation of the AR model (1 / sqrt(1 - a^2) for AR(1)).
int init_ensemble(letkf_ctx* c, const double* L_host, const double* P0_host) {
    const int na = c->n_act, m = c->m;
    const bool f64 = c->precision == LETKF_PREC_FP64;
    const size_t eb = f64 ? 8 : 4;
    const size_t nn = (size_t)na * na;
    const size_t row = (size_t)c->m_pad * eb;
    // buffers for the process-noise draws of later frames
    if (L_host && c->precision == LETKF_PREC_MIXED) {
        const int rc = noise_prepare(c, L_host);
        if (rc) return rc;
        const size_t xib = noise_xi_bytes(na, m);
        if (cudaMalloc(&c->Xi, xib) != cudaSuccess) return LETKF_ENOMEM;
        cudaMemset(c->Xi, 0, xib);
        c->device_bytes += xib;
    } else if (L_host) {
        void* tmp = nullptr;
        if (cudaMalloc(&tmp, nn * 8) != cudaSuccess) return LETKF_ENOMEM;
        cudaMemcpy(tmp, L_host, nn * 8, cudaMemcpyHostToDevice);
        int rc = LETKF_OK;
        if (c->path == LETKF_PATH_GLOBAL) {   // draws with its tiled GEMM, from tiles of the FP32 factor
            if (cudaMalloc(&c->Lq, nn * eb) != cudaSuccess) {
                rc = LETKF_ENOMEM;
            } else {
                c->device_bytes += nn * eb;
                f64_to_f32<<<grid_for(nn, 256), 256, 0, c->stream>>>((const double*)tmp, (float*)c->Lq, nn);
            }
        } else {
            rc = f64 ? rg_prepare<double>(c, (const double*)tmp) : rg_prepare<float>(c, (const double*)tmp);
        }
        cudaStreamSynchronize(c->stream);
        cudaFree(tmp);
        if (rc) return rc;
    }
    // the initial ensemble itself is formed at full state precision (FP64 or FP32 GEMMs)
    const int gt = f64 ? 0 : 1;
    void *Lf = nullptr, *Pf = nullptr, *xi = nullptr;
    const size_t fb = f64 ? 8 : 4;
    auto upload_conv = [&](const double* src, double scale, void** dst) -> int {
        void* tmp = nullptr;
        if (cudaMalloc(&tmp, nn * 8) != cudaSuccess) return LETKF_ENOMEM;
        std::vector<double> h(src, src + nn);
        if (scale != 1.0)
            for (auto& v : h) v *= scale;
        cudaMemcpy(tmp, h.data(), nn * 8, cudaMemcpyHostToDevice);
        if (cudaMalloc(dst, nn * fb) != cudaSuccess) { cudaFree(tmp); return LETKF_ENOMEM; }
        if (f64)
            cudaMemcpy(*dst, tmp, nn * 8, cudaMemcpyDeviceToDevice);
        else
            f64_to_f32<<<grid_for(nn, 256), 256, 0, c->stream>>>((const double*)tmp, (float*)*dst, nn);
        cudaStreamSynchronize(c->stream);
        cudaFree(tmp);
        return LETKF_OK;
    };
    int rc = LETKF_OK;
    // the stationary factor is lower triangular when given as a Cholesky factor, or when it is L scaled
    const bool p0_lower = P0_host ? lower_triangular(P0_host, na) : c->lq_lower != 0;
    if (cudaMalloc(&xi, (size_t)na * row) != cudaSuccess) return LETKF_ENOMEM;
    cudaMemset(xi, 0, (size_t)na * row);
    // stationary standard deviation of the AR model with unit innovations (the default P0 scale):
    // AR(2) gamma_0 = (1 - a2) / ((1 + a2) ((1 - a2)^2 - a^2)), which is 1 / (1 - a^2) for a2 = 0
    const double a2 = c->a2;
    const double sa = std::sqrt((1.0 - a2) / ((1.0 + a2) * ((1.0 - a2) * (1.0 - a2) - c->a * c->a)));
    void* X = c->X[0];
    void* X2 = static_cast<char*>(X) + (size_t)na * row;  // second instant rows
    const int nq = (na + 3) / 4;
    const int g = grid_for((size_t)nq * m, 256);
    auto draw = [&](uint32_t frame) {
        if (f64)
            normals_kernel<double><<<g, 256, 0, c->stream>>>((double*)xi, c->m_pad, na, m, c->seed, 0u, frame);
        else
            normals_kernel<float><<<g, 256, 0, c->stream>>>((float*)xi, c->m_pad, na, m, c->seed, 0u, frame);
    };
    if (L_host) {
        if ((rc = upload_conv(L_host, 1.0, &Lf))) goto done;
        if (P0_host) {
            if ((rc = upload_conv(P0_host, 1.0, &Pf))) goto done;
        } else {
            if ((rc = upload_conv(L_host, sa, &Pf))) goto done;
        }
        draw(0);
        if ((rc = noise_gemm(c, Pf, xi, c->m_pad, gt, X2, c->stream, p0_lower))) goto done;
        draw(1);
        if ((rc = noise_gemm(c, Lf, xi, c->m_pad, gt, X, c->stream, c->lq_lower != 0))) goto done;  // first rows <- L xi1
    } else {
        // white noise: second = (q / sqrt(1 - a^2)) xi0 (or P0 xi0), first = a second + q xi1
        if (P0_host) {
            if ((rc = upload_conv(P0_host, 1.0, &Pf))) goto done;
            draw(0);
            if ((rc = noise_gemm(c, Pf, xi, c->m_pad, gt, X2, c->stream, p0_lower))) goto done;
        } else {
            draw(0);
            cudaMemcpyAsync(X2, xi, (size_t)na * row, cudaMemcpyDeviceToDevice, c->stream);
            if (f64)
                axpy_rows_kernel<double><<<grid_for((size_t)na * m, 256), 256, 0, c->stream>>>(
                    (double*)X2, (const double*)xi, 0.0, c->q_white * sa, na, m, c->m_pad);
            else
                axpy_rows_kernel<float><<<grid_for((size_t)na * m, 256), 256, 0, c->stream>>>(
                    (float*)X2, (const float*)xi, 0.f, (float)(c->q_white * sa), na, m, c->m_pad);
        }
        draw(1);
        if (f64)
            axpy_rows_kernel<double><<<grid_for((size_t)na * m, 256), 256, 0, c->stream>>>(
                (double*)X, (const double*)xi, 0.0, c->q_white, na, m, c->m_pad);
        else
            axpy_rows_kernel<float><<<grid_for((size_t)na * m, 256), 256, 0, c->stream>>>(
                (float*)X, (const float*)xi, 0.f, (float)c->q_white, na, m, c->m_pad);
    }
    // first += a * second
    if (f64)
        axpy_rows_kernel<double><<<grid_for((size_t)na * m, 256), 256, 0, c->stream>>>(
            (double*)X, (const double*)X2, 1.0, c->a, na, m, c->m_pad);
    else
        axpy_rows_kernel<float><<<grid_for((size_t)na * m, 256), 256, 0, c->stream>>>(
            (float*)X, (const float*)X2, 1.f, (float)c->a, na, m, c->m_pad);
    if (cudaStreamSynchronize(c->stream) != cudaSuccess || cudaGetLastError() != cudaSuccess) rc = LETKF_ECUDA;
done:
    cudaStreamSynchronize(c->stream);
    if (Lf) cudaFree(Lf);
    if (Pf) cudaFree(Pf);
    if (xi) cudaFree(xi);
    return rc;
}

}  // namespace letkf
