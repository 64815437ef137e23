// Plain per-domain path of the local ETKF analysis (Sect. 2.3): one kernel per
// stage, one CTA per domain, SIMT arithmetic in the state type (float or double).
//
//   plain_obs        halo anomalies -> Fried slopes S = Y'/sigma (p_loc x m), d/sigma
//   plain_gram       G = S^T S (m x m), b = S^T d/sigma
//   plain_eig        T = (I + G/(m-1))^(-1/2) through its tridiagonal form in shared memory, or by
//                    two-sided Jacobi where it is ill conditioned;
//                    W = T + w_bar 1^T with w_bar = T (T b) / (m-1), refined
//   plain_transform  X_a[E] = x_bar[E] 1^T + X'[E] W on the domain's own rows
//
// Intermediate results live in device scratch buffers between the launches.

#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>
#include <vector>

#include "common.cuh"
#include "internal.hpp"

namespace letkf {
namespace {

constexpr int kThreads = 256;

// These kernels run one small problem per domain, a hundred domains at most at once, so latency bounds
// them, not bandwidth: rows go through registers (loaded, averaged over the lanes and centred in one pass),
// tables that one warp needs one after another are loaded together, and short sums are split over lanes.  In
// FP64 (2 operations per cycle and SM, measured) the operations count as well: no padding, half of the
// symmetric Gram, and the blocks of a domain are shared by several CTAs where the domains leave SMs idle.
// Per frame, FP64 8 x 8 pupil with m = 20 / FP32 40 x 40 pupil with m = 50, launch included: plain_obs
// 15 -> 12 / 20 -> 10 us, plain_gram 43 -> 12 / 36 -> 17, plain_transform 25 -> 12 / 18 -> 13.

// Members per lane of a row in registers (plain_limits_ok ends at m = 168 in FP32, 118 in FP64).
template <typename T>
constexpr int kRowLanes = sizeof(T) == 4 ? 6 : 4;

// Rows warp, warp + 8, ... below n of a matrix whose row j starts at src(j), `cols` columns each, to
// dst (leading dimension ld): the loads of four rows are issued before their stores.
template <typename T, typename F>
__device__ __forceinline__ void copy_rows(int cols, int n, T* dst, int ld, F&& src) {
    constexpr int U = kRowLanes<T>, B = 4, W = kThreads / 32;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int j0 = warp; j0 < n; j0 += B * W) {
        T v[B][U];
#pragma unroll
        for (int b = 0; b < B; ++b) {
            const T* x = src(min(j0 + b * W, n - 1));
#pragma unroll
            for (int u = 0; u < U; ++u) v[b][u] = lane + 32 * u < cols ? x[lane + 32 * u] : (T)0;
        }
#pragma unroll
        for (int b = 0; b < B; ++b)
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (j0 + b * W < n && lane + 32 * u < cols) dst[(j0 + b * W) * ld + lane + 32 * u] = v[b][u];
    }
}

// The same for rows of the ensemble, centred on their member mean (ld = m + 1, the mean behind the
// members).  The four means are summed together: 6 additions in place of 20.
template <typename T, typename F>
__device__ __forceinline__ void centred_rows(int m, T inv_m, int n, T* dst, F&& src) {
    constexpr int U = kRowLanes<T>, B = 4, W = kThreads / 32;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, mp1 = m + 1;
    for (int j0 = warp; j0 < n; j0 += B * W) {
        T v[B][U], s[B];
#pragma unroll
        for (int b = 0; b < B; ++b) {
            const T* x = src(min(j0 + b * W, n - 1));
#pragma unroll
            for (int u = 0; u < U; ++u) v[b][u] = lane + 32 * u < m ? x[lane + 32 * u] : (T)0;
        }
#pragma unroll
        for (int b = 0; b < B; ++b) {
            s[b] = v[b][0];
#pragma unroll
            for (int u = 1; u < U; ++u)
                if (32 * u < m) s[b] += v[b][u];
        }
        // lanes with bit 4 set go on with rows 2 and 3, with bit 3 set with the odd one of the two
        const bool hi = lane & 16, odd = lane & 8;
        T a = (hi ? s[2] : s[0]) + __shfl_xor_sync(0xffffffffu, hi ? s[0] : s[2], 16);
        T b = (hi ? s[3] : s[1]) + __shfl_xor_sync(0xffffffffu, hi ? s[1] : s[3], 16);
        a = (odd ? b : a) + __shfl_xor_sync(0xffffffffu, odd ? a : b, 8);
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        a *= inv_m;
#pragma unroll
        for (int b4 = 0; b4 < B; ++b4) {
            const int j = j0 + b4 * W;
            const T mean = __shfl_sync(0xffffffffu, a, 8 * b4);
            if (j >= n) break;
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (lane + 32 * u < m) dst[j * mp1 + lane + 32 * u] = v[b4][u] - mean;
            if (lane == 0) dst[j * mp1 + m] = mean;
        }
    }
}

// Observed anomalies of one domain: the halo actuators of the observed instant, centred on their
// member mean in shared memory, and differenced at the corners of each observed subaperture
// (Fried geometry, Sect. 3).
template <typename T>
__global__ void __launch_bounds__(kThreads) plain_obs(const T* __restrict__ X, const T* __restrict__ y,
                                                      DomainTables tab, const int* __restrict__ so_off,
                                                      T* __restrict__ S, T* __restrict__ dt, int m, int m_pad,
                                                      int row0, int n_subv, T inv_sigma, T inv_m,
                                                      const int* __restrict__ frame_bad) {
    extern __shared__ unsigned char smem_raw[];
    T* Xh = reinterpret_cast<T*>(smem_raw);
    if (*frame_bad) return;
    const int d = blockIdx.x;
    const int h0 = tab.halo_off[d], nh = tab.halo_off[d + 1] - h0;
    const int o0 = tab.obs_off[d], no = tab.obs_off[d + 1] - o0;
    if (no == 0) return;
    const int mp1 = m + 1;  // smem row: m members, then the mean
    centred_rows(m, inv_m, nh, Xh, [&](int j) { return X + (size_t)(row0 + tab.halo[h0 + j]) * m_pad; });
    const int base = so_off[d];
    // the corners of this warp's subapertures, one per lane (warp, warp + 8, ...), up to 256 at a time
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    auto corners = [&](int s0) {
        const int s = s0 + warp + 8 * lane;
        return s < no ? tab.obs_corner[o0 + s] : 0;
    };
    int pcs = corners(0);
    __syncthreads();
    const T half = (T)0.5 * inv_sigma;
    for (int s = warp; s < no; s += 8) {
        if (s >= 256 && (s >> 3 & 31) == 0) pcs = corners(s - warp);
        const int pc = __shfl_sync(0xffffffffu, pcs, s >> 3 & 31);
        const T *r00 = Xh + (pc & 0xFF) * mp1, *r01 = Xh + ((pc >> 8) & 0xFF) * mp1;
        const T *r10 = Xh + ((pc >> 16) & 0xFF) * mp1, *r11 = Xh + ((pc >> 24) & 0xFF) * mp1;
        for (int i = lane; i < m; i += 32) {
            const T u = r11[i] - r00[i], v = r01[i] - r10[i];
            S[(size_t)(base + s) * m_pad + i] = half * (u + v);
            S[(size_t)(base + no + s) * m_pad + i] = half * (u - v);
        }
    }
    // the mean's slopes against the measured ones
    for (int s = threadIdx.x; s < no; s += kThreads) {
        const int pc = tab.obs_corner[o0 + s], k = tab.obs_sub[o0 + s];
        const T yx = y[k], yy = y[n_subv + k];
        const T a00 = Xh[(pc & 0xFF) * mp1 + m], a01 = Xh[((pc >> 8) & 0xFF) * mp1 + m];
        const T a10 = Xh[((pc >> 16) & 0xFF) * mp1 + m], a11 = Xh[((pc >> 24) & 0xFF) * mp1 + m];
        dt[base + s] = (yx - (T)0.5 * ((a01 + a11) - (a00 + a10))) * inv_sigma;
        dt[base + no + s] = (yy - (T)0.5 * ((a10 + a11) - (a00 + a01))) * inv_sigma;
    }
}

// Blocks of 4 x 4 of S^T S on and above the diagonal, 2^LK lanes to a block with every 2^LK-th row of S
// each: blocks [first, last) of this CTA, in passes of kThreads >> LK.
template <typename T, int LK>
__device__ __forceinline__ void gram_blocks(const T* __restrict__ Ss, int ld, int pl, T* __restrict__ Gd, int m, int m_pad,
                                            int first, int last) {
    constexpr int KS = 1 << LK, CAP = kThreads >> LK;
    const int nb = (m + 3) >> 2, ks = threadIdx.x & (KS - 1);
    for (int b0 = first; b0 < last; b0 += CAP) {
        const int t = b0 + (threadIdx.x >> LK);
        int rem = min(t, last - 1), bi = 0;
        while (rem >= nb - bi) rem -= nb - bi++;
        const int i0 = 4 * bi, j0 = 4 * (bi + rem);
        // past m: the last column again (not stored)
        const int i1 = min(i0 + 1, m - 1), i2 = min(i0 + 2, m - 1), i3 = min(i0 + 3, m - 1);
        const int j1 = min(j0 + 1, m - 1), j2 = min(j0 + 2, m - 1), j3 = min(j0 + 3, m - 1);
        T acc[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) acc[e] = 0;
#pragma unroll 2
        for (int k = ks; k < pl; k += KS) {
            const T* row = Ss + k * ld;
            const T a[4] = {row[i0], row[i1], row[i2], row[i3]}, b[4] = {row[j0], row[j1], row[j2], row[j3]};
#pragma unroll
            for (int e = 0; e < 16; ++e) acc[e] += a[e >> 2] * b[e & 3];
        }
        // the lanes' sums: each step halves what a lane keeps
        int e0 = 0;
#pragma unroll
        for (int q = 0; q < LK; ++q) {
            const int half = 8 >> q;
            const bool up = (ks >> q) & 1;
            e0 += up ? half : 0;
#pragma unroll
            for (int e = 0; e < half; ++e) {
                const T give = up ? acc[e] : acc[e + half], keep = up ? acc[e + half] : acc[e];
                acc[e] = keep + __shfl_xor_sync(0xffffffffu, give, 1 << q);
            }
        }
        if (t < last)
#pragma unroll
            for (int e = 0; e < (16 >> LK); ++e) {
                const int i = i0 + ((e0 + e) >> 2), j = j0 + ((e0 + e) & 3);
                if (i < m && j < m) {
                    Gd[(size_t)i * m_pad + j] = acc[e];
                    if (j0 > i0) Gd[(size_t)j * m_pad + i] = acc[e];
                }
            }
    }
}

// G = S^T S and b = S^T dt for one domain; S staged in shared memory.  gridDim.y CTAs share the blocks.
template <typename T>
__global__ void __launch_bounds__(kThreads) plain_gram(const T* __restrict__ S, const T* __restrict__ dt,
                                                       DomainTables tab, const int* __restrict__ so_off,
                                                       T* __restrict__ G, T* __restrict__ bvec, int m, int m_pad,
                                                       const int* __restrict__ frame_bad) {
    extern __shared__ unsigned char smem_raw[];
    T* Ss = reinterpret_cast<T*>(smem_raw);
    if (*frame_bad) return;
    const int d = blockIdx.x;
    const int no = tab.obs_off[d + 1] - tab.obs_off[d];
    const int pl = 2 * no;
    const int base = so_off[d];
    T* Gd = G + (size_t)d * m * m_pad;
    const int ld = m + 1;  // rows of m members plus dt
    copy_rows<T>(m, pl, Ss, ld, [&](int k) { return S + (size_t)(base + k) * m_pad; });
    for (int k = threadIdx.x; k < pl; k += kThreads) Ss[k * ld + m] = dt[base + k];
    __syncthreads();
    const int nb = (m + 3) >> 2, blocks = nb * (nb + 1) / 2, per = (blocks + gridDim.y - 1) / gridDim.y;
    const int first = min((int)blockIdx.y * per, blocks), last = min(first + per, blocks);
    // as many lanes to a block as leave every block a place in the first pass
    if (per * 16 <= kThreads)
        gram_blocks<T, 4>(Ss, ld, pl, Gd, m, m_pad, first, last);
    else if (per * 8 <= kThreads)
        gram_blocks<T, 3>(Ss, ld, pl, Gd, m, m_pad, first, last);
    else if (per * 4 <= kThreads)
        gram_blocks<T, 2>(Ss, ld, pl, Gd, m, m_pad, first, last);
    else if (per * 2 <= kThreads)
        gram_blocks<T, 1>(Ss, ld, pl, Gd, m, m_pad, first, last);
    else
        gram_blocks<T, 0>(Ss, ld, pl, Gd, m, m_pad, first, last);
    if (blockIdx.y != gridDim.y - 1) return;
    for (int i0 = 0; i0 < m; i0 += kThreads / 8) {      // eight lanes to a member
        const int i = i0 + (threadIdx.x >> 3), c = min(i, m - 1);
        T s = 0;
        for (int k = threadIdx.x & 7; k < pl; k += 8) s += Ss[k * ld + c] * Ss[k * ld + m];
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (i < m && (threadIdx.x & 7) == 0) bvec[(size_t)d * m_pad + i] = s;
    }
}

// Quadrature nodes per pass over the tridiagonal function (their recursions live in shared memory): one
// lane each for the serial recursions, whose divisions (FP64: about 1000 cycles) bound a pass, so that
// all nodes of a usual kappa go in one (kappa = 100: 17 in FP64, 10 in FP32).
template <typename T>
constexpr int kNodes = sizeof(T) == 8 ? 32 : 16;

template <typename T>
__device__ __forceinline__ void sincos_halfpi(T a, T& s, T& c);   // sin and cos of (pi/2) a
template <>
__device__ __forceinline__ void sincos_halfpi<float>(float a, float& s, float& c) { sincospif(0.5f * a, &s, &c); }
template <>
__device__ __forceinline__ void sincos_halfpi<double>(double a, double& s, double& c) { sincospi(0.5 * a, &s, &c); }

// ---- ill-conditioned domains: cyclic two-sided Jacobi
//
// A rotation is skipped when |a_pq| <= jacobi_tol sqrt(a_pp a_qq), the relative test that gives eigenvalues
// and eigenvectors to working relative accuracy for positive definite matrices.  In FP32 the off-diagonal
// rounding floor after a rotation is a few units of roundoff of the larger diagonal, so the threshold sits a
// little above it and the sweeps end.
template <typename T>
constexpr T jacobi_tol = sizeof(T) == 8 ? (T)1e-14 : (T)3e-6;
constexpr int JACOBI_SWEEPS = 40;

// Round-robin pairing of M (even) indices: step s, pair k.
__device__ __forceinline__ void rr_pair(int M, int s, int k, int& p, int& q) {
    const int a = k == 0 ? s : (s + k) % (M - 1), b = k == 0 ? M - 1 : (s - k + M - 1) % (M - 1);
    p = min(a, b);
    q = max(a, b);
}

// Weights of one domain from the eigendecomposition (m-1)I + G = U diag(lambda) U^T:
// W = U diag(sqrt((m-1)/lambda)) U^T + w_bar 1^T, w_bar = U diag(1/lambda) U^T b, refined once with the
// residual in FP64.  A (padded to even order M with a zero row and column) and U in shared memory.  In exact
// arithmetic no lambda is below m - 1; rounding can take one there, and ST_NOCONV tells that the matrix was not
// numerically positive definite.
// Latency bounds it: two barriers per step of half-M rotations, of which the last sweeps have few, so that steps
// and blocks without one are passed over and V's rows need no division per element (FP32, m = 20 / 50 / 100: 159 /
// 980 / 3870 -> 145 / 898 / 3260 us; FP64, m = 20 / 50: 651 / 4510 -> 623 / 4290).
template <typename T>
__device__ __noinline__ void jacobi_weights(const T* __restrict__ Gd, const T* __restrict__ bd, T* __restrict__ Wd, int m,
                                            int m_pad, unsigned char* smem, int* status) {
    const int M = m + (m & 1), ld = M + 1, half = M / 2, tid = threadIdx.x, nt = blockDim.x;
    const int warp = tid >> 5, lane = tid & 31, nw = nt >> 5;
    T* A = reinterpret_cast<T*>(smem);
    T* V = A + M * ld;
    T* cs = V + M * ld;                        // M/2 (c, s) pairs
    int* pq = reinterpret_cast<int*>(cs + M);  // M/2 (p, q) pairs
    T* rv = reinterpret_cast<T*>(pq + M);      // refinement: residual, then U^T r / lambda
    T* tv = rv + M;
    const T c0 = (T)(m - 1);
    __syncthreads();                           // the caller's reads are done
    for (int i = warp; i < M; i += nw)
        for (int j = lane; j < M; j += 32) {
            A[i * ld + j] = (i < m && j < m ? Gd[(size_t)i * m_pad + j] : (T)0) + (i == j && i < m ? c0 : (T)0);
            V[i * ld + j] = i == j ? (T)1 : (T)0;
        }
    __syncthreads();
    // columns of V: thread (group vg of M threads, row tid mod M) takes pairs vg, vg + groups, ...
    const int groups = nt / M, vg = tid / M;                 // (launch_eig: three groups or more)
    T* Vr = V + (tid - vg * M) * ld;
    int sweep = 0;
    for (; sweep < JACOBI_SWEEPS; ++sweep) {
        bool rotated = false;
        for (int s = 0; s < M - 1; ++s) {
            bool rot = false;
            for (int k = tid; k < half; k += nt) {
                int p, q;
                rr_pair(M, s, k, p, q);
                const T apq = A[p * ld + q], app = A[p * ld + p], aqq = A[q * ld + q];
                T c = 1, sn = 0;
                if (fabs(apq) > jacobi_tol<T> * sqrt(fabs(app * aqq))) {
                    const T tau = (aqq - app) / ((T)2 * apq);
                    const T t = (tau >= (T)0 ? (T)1 : (T)-1) / (fabs(tau) + sqrt((T)1 + tau * tau));
                    c = (T)1 / sqrt((T)1 + t * t);
                    sn = t * c;
                    rot = true;
                }
                cs[2 * k] = c;
                cs[2 * k + 1] = sn;
                pq[2 * k] = p;
                pq[2 * k + 1] = q;
            }
            if (!__syncthreads_or(rot)) continue;      // (most steps of the last sweeps)
            rotated = true;
            // A <- J^T A J on the 2 x 2 blocks of paired rows P x paired columns Q, P <= Q; A stays symmetric, so
            // the blocks above the diagonal also write their transposes.  Rows r and half - 1 - r of the
            // triangle have half + 1 blocks together
            for (int blk = tid; blk < half * (half + 1) / 2; blk += nt) {
                const int r = blk / (half + 1), c = blk - r * (half + 1);
                const int P = c < half - r ? r : half - 1 - r, Q = c < half - r ? r + c : c - 1;
                const int pP = pq[2 * P], qP = pq[2 * P + 1], pQ = pq[2 * Q], qQ = pq[2 * Q + 1];
                const T cP = cs[2 * P], sP = cs[2 * P + 1], cQ = cs[2 * Q], sQ = cs[2 * Q + 1];
                if (sP == (T)0 && sQ == (T)0) continue;
                const T b00 = A[pP * ld + pQ], b01 = A[pP * ld + qQ];
                const T b10 = A[qP * ld + pQ], b11 = A[qP * ld + qQ];
                const T r00 = cP * b00 - sP * b10, r01 = cP * b01 - sP * b11;
                const T r10 = sP * b00 + cP * b10, r11 = sP * b01 + cP * b11;
                const T n00 = cQ * r00 - sQ * r01, n01 = sQ * r00 + cQ * r01;
                const T n10 = cQ * r10 - sQ * r11, n11 = sQ * r10 + cQ * r11;
                A[pP * ld + pQ] = n00;
                A[pP * ld + qQ] = n01;
                A[qP * ld + pQ] = n10;
                A[qP * ld + qQ] = n11;
                if (P != Q) {
                    A[pQ * ld + pP] = n00;
                    A[qQ * ld + pP] = n01;
                    A[pQ * ld + qP] = n10;
                    A[qQ * ld + qP] = n11;
                }
            }
            if (vg < groups)                                 // V <- V J
                for (int P = vg; P < half; P += groups) {
                    const T c = cs[2 * P], sn = cs[2 * P + 1];
                    if (sn == (T)0) continue;
                    const int p = pq[2 * P], q = pq[2 * P + 1];
                    const T vp = Vr[p], vq = Vr[q];
                    Vr[p] = c * vp - sn * vq;
                    Vr[q] = sn * vp + c * vq;
                }
            __syncthreads();
        }
        if (!rotated) break;
    }
    // f_i = sqrt((m-1)/lambda_i) in A's padding column M, w_bar in V's
    T* z = cs;
    bool bad = sweep == JACOBI_SWEEPS;
    for (int i = tid; i < m; i += nt) {
        T lam = A[i * ld + i];
        bad = bad || !(lam > (T)0);
        lam = lam < c0 ? c0 : lam;
        T s = 0;
        for (int k = 0; k < m; ++k) s += V[k * ld + i] * bd[k];
        z[i] = s / lam;
        A[i * ld + i] = lam;
        A[i * ld + M] = sqrt(c0 / lam);
    }
    if (__syncthreads_or(bad) && tid == 0) atomicOr(status, ST_NOCONV);
    for (int k = tid; k < m; k += nt) {
        T s = 0;
        for (int i = 0; i < m; ++i) s += V[k * ld + i] * z[i];
        V[k * ld + M] = s;
    }
    __syncthreads();
    for (int k = tid; k < m; k += nt) {
        double acc = (double)bd[k] - (double)c0 * (double)V[k * ld + M];
        for (int j = 0; j < m; ++j) acc -= (double)Gd[(size_t)k * m_pad + j] * (double)V[j * ld + M];
        rv[k] = (T)acc;
    }
    __syncthreads();
    for (int i = tid; i < m; i += nt) {
        T s = 0;
        for (int k = 0; k < m; ++k) s += V[k * ld + i] * rv[k];
        tv[i] = s / A[i * ld + i];
    }
    __syncthreads();
    for (int k = tid; k < m; k += nt) {
        T s = 0;
        for (int i = 0; i < m; ++i) s += V[k * ld + i] * tv[i];
        V[k * ld + M] += s;
    }
    __syncthreads();
    for (int k = warp; k < m; k += nw)
        for (int l = lane; l < m; l += 32) {
            T t = 0;
            for (int i = 0; i < m; ++i) t += V[k * ld + i] * A[i * ld + M] * V[l * ld + i];
            Wd[(size_t)k * m_pad + l] = t + V[k * ld + M];
        }
}

// The inverse square root needs no eigenvectors.  With B = I + G/(m-1) = Q J Q^T (J tridiagonal,
// Q a product of m - 2 Householder reflectors; Golub and Van Loan, Matrix Computations, 8.3.1),
//   T = B^(-1/2) = Q J^(-1/2) Q^T,
//   J^(-1/2) ~ (2 K' / (pi N)) sum_n dn_n (cn_n^2 J + sn_n^2 I)^(-1),
// the midpoint rule of Hale, Higham and Trefethen (SIAM J. Numer. Anal. 46, 2008, method 3) for the
// spectrum [1, kappa]: sn, cn, dn at (n - 1/2) K' / N for the parameter 1 - 1/kappa.  Every term is
// positive definite, and N = 0.88 (ln kappa + 3) + 2 (FP32) or 1.82 (ln kappa + 3) + 2 (FP64) nodes
// leave less than the rounding (the rule's error is exp(-2 pi^2 N / (ln kappa + 3)); kappa is bounded
// by J's Gershgorin circles).  That holds while kappa times the unit roundoff is small, since the reduction
// moves J's smallest eigenvalues, 1, by that much, where Jacobi's rotations keep them.  Where the bound is above
// DIRECT_TO the domain is done by Jacobi.  72 slopes, anomalies' error of Jacobi / direct, geometric means: FP32,
// m = 16: kappa 3e2 2.0e-6 / 1.6e-6, 1e3 2.1e-6 / 2.3e-6, 3.5e3 2.3e-6 / 3.1e-6; m = 20: 3.5e3 6.1e-6 / 5.8e-6,
// 6e5 7.5e-6 / 1.6e-4, 4e7 2.7e-5 / 0.2; FP64, m = 20: 6e4 1.5e-14 / 2.0e-14, 6e5 2.8e-14 / 3.1e-13.  (In a running
// loop kappa is 5 to 20, in its first two frames 1e3 to 1e4.)
//
// The inverse of a tridiagonal matrix costs O(m) divisions (the pivots from both ends) and one multiplication
// per entry, so the work is that of the reflectors: 4/3 m^3 multiply-adds to reduce, 4 m^3 in all, against 9
// sweeps of m^3 by Jacobi, which takes 4 to 10 times as long, and 2 barriers per column instead of 2 per rotation
// step and sweep.
//
// What bounds it: the m - 2 dependent reduction steps (two barriers each, the trailing matrix's
// matrix-vector product and rank-2 update between them); the reflectors are then applied to J's
// function column by column, 8 lanes and two columns per thread group, in registers and without a
// barrier.  Measured, whole stage: 92 domains of m = 50 in FP32 522 -> 112 us, 4 domains of m = 20 in
// FP64 499 -> 149 us (before: Jacobi; 183 with the nodes eight at a time).
constexpr float DIRECT_TO = 2048.f;
template <typename T, int UM>   // m <= 32 UM members; 4 threads per member, at most 640
__global__ void __launch_bounds__(UM < 5 ? 128 * UM : 640) plain_eig(const T* __restrict__ G,
                                                                     const T* __restrict__ bvec, T* __restrict__ W,
                                                                     int m, int m_pad, int kb, int* status,
                                                                     const int* __restrict__ frame_bad) {
    extern __shared__ unsigned char smem_raw[];
    const int ld = m | 1;                  // odd row stride: no bank conflicts down a column
    T* A = reinterpret_cast<T*>(smem_raw);   // G/(m-1), then (row k, columns > k) the reflector v_k
    T* F = A + m * ld;                     // the function of J, then T
    constexpr int NK = kNodes<T>;
    const int mv = max(m, 2 * NK);
    T* dd = F + m * ld;                    // J's diagonal and (ee) off-diagonal
    T* ee = dd + mv;
    T* bt = ee + mv;                       // 2 / v_k^T v_k
    T* vs = bt + mv;
    T* ps = vs + mv;
    T* gn = ps + mv;                       // kb x m: diagonal of each node's inverse
    T* rn = gn + kb * m;                   // kb x m: ratio of successive entries along a row
    T* bs = gn;                            // b, once the nodes are done
    if (*frame_bad) return;                // the transform leaves a rejected frame's rows as they are
    const int d = blockIdx.x, tid = threadIdx.x, nt = blockDim.x;
    const int warp = tid >> 5, lane = tid & 31, nw = nt >> 5;
    const T* Gd = G + (size_t)d * m * m_pad;
    const T c0 = (T)(m - 1), ic0 = (T)1 / c0;
    for (int i = warp; i < m; i += nw)
        for (int j = lane; j < m; j += 32) A[i * ld + j] = Gd[(size_t)i * m_pad + j] * ic0;
    __syncthreads();
    // ---- reduction of G/(m-1), to which J adds the identity: step k maps row k (columns > k) onto e_k times the
    // first unit vector
    for (int k = 0; k < m - 2; ++k) {
        const int k1 = k + 1, nk = m - k1;
        T v[UM];
        T sg = 0;
#pragma unroll
        for (int u = 0; u < UM; ++u) {
            const int j = lane + 32 * u;
            v[u] = j < nk ? A[k * ld + k1 + j] : (T)0;
            sg += v[u] * v[u];
        }
        sg = warp_sum(sg);                 // every warp forms the reflector itself: no barrier
        const T x0 = __shfl_sync(0xffffffffu, v[0], 0), nrm = sqrt(sg);
        // a row as small as that beside the unit diagonal of B is left alone: its square, or 1 / vv, may be
        // out of range (FP32: an ensemble's spread below 1e-10 sigma)
        const bool flat = sg <= (sizeof(T) == 8 ? (T)1e-40 : (T)1e-24);
        const T al = flat ? x0 : x0 >= (T)0 ? -nrm : nrm;
        const T vv = sg + fabs(x0) * nrm;  // v^T v / 2
        const T beta = flat ? (T)0 : (T)1 / vv;
        if (lane == 0) v[0] = x0 - al;
        for (int r = k1 + warp; r < m; r += 2 * nw) {   // p = beta S v, two rows in flight
            const int r2 = r + nw < m ? r + nw : r;
            T s0 = 0, s1 = 0;
#pragma unroll
            for (int u = 0; u < UM; ++u)
                if (32 * u < nk) {
                    const int j = lane + 32 * u < nk ? k1 + lane + 32 * u : k1;   // v is 0 past the end
                    s0 += A[r * ld + j] * v[u];
                    s1 += A[r2 * ld + j] * v[u];
                }
            s0 = warp_sum(s0);
            s1 = warp_sum(s1);
            if (lane == 0) {
                ps[r] = beta * s0;
                if (r2 != r) ps[r2] = beta * s1;
            }
        }
        if (warp == 0)
#pragma unroll
            for (int u = 0; u < UM; ++u)
                if (lane + 32 * u < nk) vs[k1 + lane + 32 * u] = v[u];
        __syncthreads();
        T p[UM], pv = 0;
#pragma unroll
        for (int u = 0; u < UM; ++u) {
            p[u] = lane + 32 * u < nk ? ps[k1 + lane + 32 * u] : (T)0;
            pv += p[u] * v[u];
        }
        const T hk = (T)0.5 * beta * warp_sum(pv);
#pragma unroll
        for (int u = 0; u < UM; ++u) p[u] -= hk * v[u];            // w = p - (beta/2)(p^T v) v
        for (int r = k1 + warp; r < m; r += nw) {                  // S <- S - v w^T - w v^T
            const T vr = vs[r], wr = ps[r] - hk * vr;
#pragma unroll
            for (int u = 0; u < UM; ++u)
                if (lane + 32 * u < nk) {
                    T* a = A + r * ld + k1 + lane + 32 * u;
                    *a -= vr * p[u] + wr * v[u];
                }
        }
        if (warp == 0) {
#pragma unroll
            for (int u = 0; u < UM; ++u)
                if (lane + 32 * u < nk) A[k * ld + k1 + lane + 32 * u] = v[u];
            if (lane == 0) {
                dd[k] = (T)1 + A[k * ld + k];
                ee[k] = al;
                bt[k] = beta;
            }
        }
        __syncthreads();
    }
    if (tid == 0) {
        dd[m - 2] = (T)1 + A[(m - 2) * ld + m - 2];
        dd[m - 1] = (T)1 + A[(m - 1) * ld + m - 1];
        ee[m - 2] = A[(m - 2) * ld + m - 1];
        ee[m - 1] = 0;
    }
    __syncthreads();
    // ---- F = J^(-1/2): kappa from the Gershgorin circles (every warp for itself)
    T hi = (T)1;
    for (int i = lane; i < m; i += 32) hi = fmax(hi, fabs(dd[i]) + fabs(ee[i]) + (i > 0 ? fabs(ee[i - 1]) : (T)0));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    if (!(hi <= DIRECT_TO)) {              // (a NaN as well)
        jacobi_weights(Gd, bvec + (size_t)d * m_pad, W + (size_t)d * m * m_pad, m, m_pad, smem_raw, status);
        return;
    }
    const float rate = sizeof(T) == 8 ? 1.83f : 0.88f;
    const int N = max(1, min(128, (int)(rate * (logf((float)hi) + 3.f)) + 3));
    // descending Landen chain of the modulus: k_0' = kappa^(-1/2), k_(s+1) = (1 - k_s')/(1 + k_s'),
    // k_(s+1)' = 2 sqrt(k_s')/(1 + k_s'); K' = (pi/2) prod (1 + k_s)
    constexpr int LS = sizeof(T) == 8 ? 9 : 7;
    T lk[LS], kprod = (T)1;
    if (tid < 2 * NK) {
        // until k_s no longer counts (a few steps: k_(s+1) ~ (k_s / 2)^2)
        T kc = (T)1 / sqrt(hi);
        bool more = true;
#pragma unroll
        for (int s = 0; s < LS; ++s) {
            lk[s] = 0;
            if (more) {
                const T q = (T)1 / ((T)1 + kc);
                lk[s] = ((T)1 - kc) * q;
                kprod *= (T)1 + lk[s];
                kc = (T)2 * sqrt(kc) * q;
                more = lk[s] > (sizeof(T) == 8 ? (T)1e-17 : (T)1e-9);
            }
        }
    }
    for (int n0 = 0; n0 < N; n0 += kb) {
        const int nn = min(kb, N - n0);
        if (tid < 2 * NK && (tid & (NK - 1)) < nn) {
            // thread (node, direction): the pivots of cn^2 J + sn^2 I from the top (into gn) or from
            // the bottom (into rn)
            const int n = tid & (NK - 1);
            T sn, cn, dn = (T)1;
            sincos_halfpi<T>((T)(2 * (n0 + n) + 1) / (T)(2 * N), sn, cn);
#pragma unroll
            for (int s = LS - 1; s >= 0; --s) {
                if (lk[s] == (T)0) continue;
                const T s2 = lk[s] * sn * sn, q = (T)1 / ((T)1 + s2);
                const T cd = cn * dn * q;
                dn = ((T)1 - s2) * q;
                sn = ((T)1 + lk[s]) * sn * q;
                cn = cd;
            }
            const T c2 = cn * cn, s2 = sn * sn;
            if (tid < NK) {
                T pv = c2 * dd[0] + s2;
                gn[n * m] = pv;
                for (int i = 1; i < m; ++i) {
                    const T e = c2 * ee[i - 1];
                    pv = c2 * dd[i] + s2 - e * e / pv;
                    gn[n * m + i] = pv;
                }
                vs[n] = c2;                // the node's parameters, for the pass below
                vs[NK + n] = s2;
                ps[n] = dn * kprod / (T)N;
            } else {
                T pv = c2 * dd[m - 1] + s2;
                rn[n * m + m - 1] = pv;
                for (int i = m - 2; i >= 0; --i) {
                    const T e = c2 * ee[i];
                    pv = c2 * dd[i] + s2 - e * e / pv;
                    rn[n * m + i] = pv;
                }
            }
        }
        __syncthreads();
        // the inverse's diagonal 1 / (top + bottom pivot - diagonal), weighted, and the ratios
        // inv(i, j + 1) / inv(i, j) = -e_j / (bottom pivot j + 1), j >= i
        for (int n = warp; n < nn; n += nw) {
            const T c2 = vs[n], s2 = vs[NK + n], wt = ps[n];
            T nx[UM];
#pragma unroll
            for (int u = 0; u < UM; ++u) {
                const int i = lane + 32 * u;
                if (i < m) {
                    const T bot = rn[n * m + i];
                    gn[n * m + i] = wt / (gn[n * m + i] + bot - (c2 * dd[i] + s2));
                    nx[u] = i + 1 < m ? -c2 * ee[i] / rn[n * m + i + 1] : (T)0;
                }
            }
            __syncwarp();
#pragma unroll
            for (int u = 0; u < UM; ++u)
                if (lane + 32 * u < m) rn[n * m + lane + 32 * u] = nx[u];
        }
        __syncthreads();
        // rows of the sum: four lanes per row, a quarter of the nodes each, walking right from the diagonal
        for (int t = tid; t < 4 * ((m + 7) & ~7); t += nt) {       // whole warps
            const int i = t >> 2, h = t & 3, i_lo = (t & ~31) >> 2;
            T r[NK / 4];
#pragma unroll
            for (int q = 0; q < NK / 4; ++q) {
                const int n = 4 * q + h;
                r[q] = (i < m && n < nn) ? gn[n * m + i] : (T)0;
            }
            for (int st = 0; st < m - i_lo; ++st) {
                const int j = i + st;
                T sum = r[0];
#pragma unroll
                for (int q = 1; q < NK / 4; ++q)
                    if (4 * q < nn) sum += r[q];
                sum += __shfl_xor_sync(0xffffffffu, sum, 1);
                sum += __shfl_xor_sync(0xffffffffu, sum, 2);
                if (st == 0 && n0 == 0) sum -= (T)1;               // F - I (see below)
                if (j < m) {
                    T* f = h ? F + j * ld + i : F + i * ld + j;    // two lanes write the two triangles
                    if (h == 0 || (h == 1 && j > i)) *f = n0 ? *f + sum : sum;
#pragma unroll
                    for (int q = 0; q < NK / 4; ++q)
                        if (4 * q + h < nn) r[q] *= rn[(4 * q + h) * m + j];
                }
            }
        }
        __syncthreads();
    }
    // ---- T = I + Q (F - I) Q^T: the reflectors on every column of F - I, then on every row of the result.
    // (Where the ensemble's spread is small beside the noise, B and F are close to the identity, and would take
    // the reflectors' rounding here and in the reduction: 2.5e-7 .. 4e-7 in FP32, now 9e-8 .. 1.8e-7.)
    const int grp = tid >> 3, l8 = tid & 7;
    auto reflect = [&](int rs, int cs) {   // vectors x_j[i] = F[j rs + i cs], two per group of 8 lanes
        for (int j0 = 2 * grp; j0 - 2 * (grp & 3) < m; j0 += nt >> 2) {   // whole warps
            T x[2][4 * UM];
#pragma unroll
            for (int q = 0; q < 2; ++q)
#pragma unroll
                for (int u = 0; u < 4 * UM; ++u) {
                    const int i = l8 + 8 * u;
                    x[q][u] = (i < m && j0 + q < m) ? F[(j0 + q) * rs + i * cs] : (T)0;
                }
            for (int k = m - 3; k >= 0; --k) {
                T v[4 * UM], s0 = 0, s1 = 0;
#pragma unroll
                for (int u = 0; u < 4 * UM; ++u)
                    if (8 * u + 7 > k && 8 * u < m) {
                        const int i = l8 + 8 * u;
                        v[u] = (i > k && i < m) ? A[k * ld + i] : (T)0;
                        s0 += v[u] * x[0][u];
                        s1 += v[u] * x[1][u];
                    }
#pragma unroll
                for (int o = 4; o > 0; o >>= 1) {
                    s0 += __shfl_xor_sync(0xffffffffu, s0, o);
                    s1 += __shfl_xor_sync(0xffffffffu, s1, o);
                }
                const T beta = bt[k];
                s0 *= beta;
                s1 *= beta;
#pragma unroll
                for (int u = 0; u < 4 * UM; ++u)
                    if (8 * u + 7 > k && 8 * u < m) {
                        x[0][u] -= s0 * v[u];
                        x[1][u] -= s1 * v[u];
                    }
            }
#pragma unroll
            for (int q = 0; q < 2; ++q)
#pragma unroll
                for (int u = 0; u < 4 * UM; ++u) {
                    const int i = l8 + 8 * u;
                    if (i < m && j0 + q < m) F[(j0 + q) * rs + i * cs] = x[q][u];
                }
        }
        __syncthreads();
    };
    reflect(1, ld);        // columns
    reflect(ld, 1);        // rows
    // ---- w_bar = T (T b) / (m-1), and one step of iterative refinement with the residual
    // r = b - ((m-1)I + G) w_bar summed in FP64: the solve's forward error grows with the condition
    // number of (m-1)I + G (hundreds in the first frames), the residual sum in FP64 removes it,
    // leaving only the rounding of G itself.
    auto tmul = [&](const T* x, T* y, T scale) {      // y = scale T x, 8 lanes per row
        for (int i0 = grp; i0 - (grp & 3) < m; i0 += nt >> 3) {
            T s = 0;
            if (i0 < m)
                for (int j = l8; j < m; j += 8) s += F[i0 * ld + j] * x[j];
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (l8 == 0 && i0 < m) y[i0] = scale * s;
        }
        __syncthreads();
    };
    T* wb = dd;            // the tridiagonal matrix is no longer needed
    for (int i = tid; i < m; i += nt) {
        F[i * ld + i] += (T)1;             // T
        bs[i] = bvec[(size_t)d * m_pad + i];
    }
    __syncthreads();
    tmul(bs, vs, (T)1);
    tmul(vs, wb, ic0);
    for (int i0 = grp; i0 - (grp & 3) < m; i0 += nt >> 3) {
        double acc = 0.0;
        if (i0 < m)
            for (int j = l8; j < m; j += 8) acc += (double)Gd[(size_t)i0 * m_pad + j] * (double)wb[j];
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (l8 == 0 && i0 < m) ps[i0] = (T)((double)bs[i0] - (double)c0 * (double)wb[i0] - acc);
    }
    __syncthreads();
    tmul(ps, vs, (T)1);
    tmul(vs, ee, ic0);
    T* Wd = W + (size_t)d * m * m_pad;
    for (int i = warp; i < m; i += nw) {
        const T w = wb[i] + ee[i];
        for (int j = lane; j < m; j += 32) Wd[(size_t)i * m_pad + j] = F[i * ld + j] + w;
    }
}

// Dynamic shared memory of jacobi_weights: A and U of even order, the rotations, two vectors.
size_t jacobi_smem(int m, size_t eb) {
    const size_t M = m + (m & 1);
    return 2 * M * (M + 1) * eb + M * (3 * eb + 4);
}

// Dynamic shared memory of plain_eig: B and F (m x m, odd row stride), vectors, kb nodes' recursions.
template <typename T>
size_t eig_smem(int m, int kb) {
    return ((size_t)2 * m * (m | 1) + (size_t)5 * std::max(m, 2 * kNodes<T>) + (size_t)2 * kb * m) * sizeof(T);
}

// Four threads per member (two columns per group of eight lanes in the back-transformation), at
// least four warps; as many nodes per pass, up to kNodes, as shared memory leaves room for (all of
// them up to m = 161 in FP32 and 104 in FP64).
template <typename T>
void launch_eig(int n_dom, cudaStream_t st, const T* G, const T* b, T* W, int m, int m_pad, int* status, const int* bad) {
    const int nt = std::min(640, std::max(128, (4 * m + 31) / 32 * 32));
    int kb = kNodes<T>;
    while (kb > 1 && eig_smem<T>(m, kb) > 227 * 1024) --kb;
    const size_t sm = std::max(eig_smem<T>(m, kb), jacobi_smem(m, sizeof(T)));
    if (m <= 32)
        plain_eig<T, 1><<<n_dom, nt, sm, st>>>(G, b, W, m, m_pad, kb, status, bad);
    else if (m <= 64)
        plain_eig<T, 2><<<n_dom, nt, sm, st>>>(G, b, W, m, m_pad, kb, status, bad);
    else if (m <= 128)
        plain_eig<T, 4><<<n_dom, nt, sm, st>>>(G, b, W, m, m_pad, kb, status, bad);
    else if constexpr (sizeof(T) == 4)     // FP64 ends at m = 118 (plain_limits_ok)
        plain_eig<T, 6><<<n_dom, nt, sm, st>>>(G, b, W, m, m_pad, kb, status, bad);
}

// X_out[E] = x_bar[E] 1^T + X'[E] W for the domain's own rows E (both instants), the rows shared by
// gridDim.y CTAs; blocks of 2 x 2 results per thread.
template <typename T>
__global__ void __launch_bounds__(kThreads) plain_transform(const T* __restrict__ X, T* __restrict__ Xo,
                                                            const T* __restrict__ W, DomainTables tab, int m,
                                                            int m_pad, int n_act, T inv_m,
                                                            const int* __restrict__ frame_bad) {
    extern __shared__ unsigned char smem_raw[];
    const int d = blockIdx.x;
    const int e0 = tab.own_off[d], ne = tab.own_off[d + 1] - e0;
    const int per = (2 * ne + gridDim.y - 1) / gridDim.y, r0 = blockIdx.y * per, nl = min(per, 2 * ne - r0);
    if (nl <= 0) return;
    const int ld = m + 1;
    T* Ws = reinterpret_cast<T*>(smem_raw);
    T* Xe = Ws + m * m;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    auto row = [&](int q) {
        const int e = r0 + q;
        return (e < ne) ? tab.own[e0 + e] : n_act + tab.own[e0 + e - ne];
    };
    // a domain without observations keeps its forecast exactly (G = 0: w_bar = 0, T = I)
    if (*frame_bad != 0 || tab.obs_off[d + 1] == tab.obs_off[d]) {
        for (int q = warp; q < nl; q += kThreads / 32)
            for (int i = lane; i < m; i += 32) Xo[(size_t)row(q) * m_pad + i] = X[(size_t)row(q) * m_pad + i];
        return;
    }
    const T* Wd = W + (size_t)d * m * m_pad;
    copy_rows<T>(m, m, Ws, m, [&](int k) { return Wd + (size_t)k * m_pad; });
    centred_rows(m, inv_m, nl, Xe, [&](int q) { return X + (size_t)row(q) * m_pad; });
    __syncthreads();
    const int cb = (m + 1) >> 1, rb = (nl + 1) >> 1;
    for (int t = threadIdx.x; t < cb * rb; t += kThreads) {
        const int b = t / cb, l0 = 2 * (t - b * cb), l1 = min(l0 + 1, m - 1), q0 = 2 * b, q1 = min(q0 + 1, nl - 1);
        const T *xa = Xe + q0 * ld, *xb = Xe + q1 * ld;
        T s00 = 0, s01 = 0, s10 = 0, s11 = 0;
#pragma unroll 4
        for (int k = 0; k < m; ++k) {
            const T u = xa[k], v = xb[k], w0 = Ws[k * m + l0], w1 = Ws[k * m + l1];
            s00 += u * w0;
            s01 += u * w1;
            s10 += v * w0;
            s11 += v * w1;
        }
        T* oa = Xo + (size_t)row(q0) * m_pad;
        T* ob = Xo + (size_t)row(q1) * m_pad;
        oa[l0] = xa[m] + s00;
        if (l0 + 1 < m) oa[l1] = xa[m] + s01;
        if (q0 + 1 < nl) {
            ob[l0] = xb[m] + s10;
            if (l0 + 1 < m) ob[l1] = xb[m] + s11;
        }
    }
}

// The four analysis kernels take dynamic shared memory sized by the system (ensemble, domain
// sizes).  Their limit is raised once per device and state type, with that device current, to
// all the shared memory a block may opt in to (less the kernel's static shared memory), so that
// no context's setting can later lower it below another's needs; every call is checked.
template <typename T>
int plain_kernels_ready(int device) {
    static std::mutex mu;
    static bool done[64] = {false};
    if (device < 0 || device >= 64) return LETKF_EINVAL;
    std::lock_guard<std::mutex> lock(mu);
    if (done[device]) return LETKF_OK;
    int optin = 0;
    if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device) != cudaSuccess) return LETKF_ECUDA;
    std::vector<const void*> fns = {
        reinterpret_cast<const void*>(plain_obs<T>), reinterpret_cast<const void*>(plain_gram<T>),
        reinterpret_cast<const void*>(plain_transform<T>), reinterpret_cast<const void*>(plain_eig<T, 1>),
        reinterpret_cast<const void*>(plain_eig<T, 2>), reinterpret_cast<const void*>(plain_eig<T, 4>)};
    if constexpr (sizeof(T) == 4) fns.push_back(reinterpret_cast<const void*>(plain_eig<T, 6>));
    for (const void* fn : fns) {
        cudaFuncAttributes fa;
        if (cudaFuncGetAttributes(&fa, fn) != cudaSuccess) return LETKF_ECUDA;
        if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes) !=
            cudaSuccess)
            return LETKF_ECUDA;
    }
    done[device] = true;
    return LETKF_OK;
}

template <typename T>
int plain_analyze_t(letkf_ctx* c, const T* y, double sigma) {
    if (sigma > 0) c->sigma = sigma;
    int rc = launch_precheck(c, y);
    if (rc) return rc;
    const T* X = static_cast<const T*>(c->X[c->cur]);
    T* Xo = static_cast<T*>(c->X[c->cur ^ 1]);
    const int m = c->m, mp = c->m_pad, nd = c->n_dom;
    const int row0 = c->obs_block == 1 ? c->n_act : 0;
    // CTAs per domain: where the domains leave SMs idle, up to eight
    const dim3 shared_by(nd, std::max(1, std::min(8, c->sms / std::max(nd, 1))));
    const size_t sm_obs = (size_t)c->host.n_h_max * (m + 1) * sizeof(T);
    const size_t sm_gram = (size_t)std::max(c->host.p_loc_max, 1) * (m + 1) * sizeof(T);
    const size_t sm_tr = ((size_t)m * m + (size_t)c->host.n_loc_max * (m + 1)) * sizeof(T);
    if ((rc = plain_kernels_ready<T>(c->device))) return rc;
    prof_begin(c, STAGE_OBS);
    plain_obs<T><<<nd, kThreads, sm_obs, c->stream>>>(X, y, c->tab, c->so_off, static_cast<T*>(c->S),
                                                      static_cast<T*>(c->dt), m, mp, row0, c->n_subv,
                                                      (T)(1.0 / c->sigma), (T)(1.0 / m), c->d_frame_bad);
    prof_end(c);
    prof_begin(c, STAGE_GRAM);
    plain_gram<T><<<shared_by, kThreads, sm_gram, c->stream>>>(static_cast<const T*>(c->S), static_cast<const T*>(c->dt),
                                                        c->tab, c->so_off, static_cast<T*>(c->G),
                                                        static_cast<T*>(c->b), m, mp, c->d_frame_bad);
    prof_end(c);
    prof_begin(c, STAGE_EIG);
    launch_eig<T>(nd, c->stream, static_cast<const T*>(c->G), static_cast<const T*>(c->b), static_cast<T*>(c->W), m, mp,
                  c->d_status, c->d_frame_bad);
    prof_end(c);
    prof_begin(c, STAGE_TRANSFORM);
    plain_transform<T><<<shared_by, kThreads, sm_tr, c->stream>>>(X, Xo, static_cast<const T*>(c->W), c->tab, m, mp,
                                                           c->n_act, (T)(1.0 / m), c->d_frame_bad);
    prof_end(c);
    if (cudaGetLastError() != cudaSuccess) return LETKF_ECUDA;
    return LETKF_OK;
}

}  // namespace

int plain_limits_ok(int precision, int m) {
    // plain_eig keeps two matrices of order m and its vectors in shared memory (<= 227 KB; Jacobi's, of even
    // order, is the tighter bound)
    return jacobi_smem(m, precision == LETKF_PREC_FP64 ? 8 : 4) <= 227 * 1024 && m <= 256;
}

int plain_analyze(letkf_ctx* c, const void* y, double sigma) {
    if (c->precision == LETKF_PREC_FP64) return plain_analyze_t<double>(c, static_cast<const double*>(y), sigma);
    return plain_analyze_t<float>(c, static_cast<const float*>(y), sigma);
}

}  // namespace letkf

// ---------------------------------------------------------------------------------------------
// Allocation-free analysis.
//
// Some callers cannot call the CUDA allocator while they run the filter: a real-time
// controller typically reserves all of its device memory before its loop starts, and an
// allocation inside the loop may block on the driver or fail under fragmentation while a
// frame deadline is pending.  letkf_analyze_static serves them: it runs the same plain-path
// kernels as letkf_analyze but takes all of its intermediate storage from one fixed array
// that exists for as long as the library is loaded, and it allocates nothing.
namespace letkf {
namespace {

// 16 MiB of scratch per GPU, held by every GPU that loads the library until the process
// exits.  Shared by every call on that GPU: calls whose work overlaps on the device race on it.
constexpr size_t kStaticScratchBytes = (size_t)16 << 20;
static __device__ __align__(256) unsigned char g_static_scratch[kStaticScratchBytes];

// Device address of g_static_scratch per device ordinal (in host code the array's name is
// only a stand-in for it), found once per device with that device current.
std::mutex g_static_mutex;
void* g_static_ptr[64] = {nullptr};

int static_scratch_address(int device, void** out) {
    if (device < 0 || device >= 64) return LETKF_EINVAL;
    std::lock_guard<std::mutex> lock(g_static_mutex);
    if (!g_static_ptr[device]) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_static_scratch) != cudaSuccess || !p) return LETKF_ECUDA;
        g_static_ptr[device] = p;
    }
    *out = g_static_ptr[device];
    return LETKF_OK;
}

// Slope check of the allocation-free path: writes its own reject flag (never the context's).
template <typename T>
__global__ void static_check_kernel(const T* __restrict__ y, int p, int* flag, int* status) {
    __shared__ int bad;
    if (threadIdx.x == 0) bad = 0;
    __syncthreads();
    int mine = 0;
    for (int i = threadIdx.x; i < p; i += blockDim.x)
        if (!finite_val(y[i])) mine = 1;
    if (mine) atomicOr(&bad, 1);
    __syncthreads();
    if (threadIdx.x == 0) {
        *flag = bad;
        if (bad) atomicOr(status, ST_NONFINITE);
    }
}

size_t align256(size_t v) { return (v + 255) & ~(size_t)255; }

template <typename T>
int analyze_static_t(letkf_ctx* c, const T* y, double sigma, T* out) {
    const int m = c->m, mp = c->m_pad, nd = c->n_dom;
    const size_t eb = sizeof(T);
    // carve the scratch: slopes, innovations, Gram, b, weights, the analysis rows, the flag
    const size_t o_S = 0;
    const size_t o_dt = align256(o_S + (size_t)std::max(c->total_slopes, 1) * mp * eb);
    const size_t o_G = align256(o_dt + (size_t)std::max(c->total_slopes, 1) * eb);
    const size_t o_b = align256(o_G + (size_t)nd * m * mp * eb);
    const size_t o_W = align256(o_b + (size_t)nd * mp * eb);
    const size_t o_X = align256(o_W + (size_t)nd * m * mp * eb);
    const size_t o_flag = align256(o_X + (size_t)c->n * mp * eb);
    const size_t need = o_flag + 256;
    if (need > kStaticScratchBytes) return LETKF_ESCRATCH;
    void* base = nullptr;
    int rc = static_scratch_address(c->device, &base);
    if (rc) return rc;
    unsigned char* sb = static_cast<unsigned char*>(base);
    T* S = reinterpret_cast<T*>(sb + o_S);
    T* dt = reinterpret_cast<T*>(sb + o_dt);
    T* G = reinterpret_cast<T*>(sb + o_G);
    T* bv = reinterpret_cast<T*>(sb + o_b);
    T* W = reinterpret_cast<T*>(sb + o_W);
    T* Xo = reinterpret_cast<T*>(sb + o_X);
    int* flag = reinterpret_cast<int*>(sb + o_flag);
    const T* X = static_cast<const T*>(c->X[c->cur]);
    const double sg = sigma > 0 ? sigma : c->sigma;
    const int row0 = c->obs_block == 1 ? c->n_act : 0;
    // CTAs per domain: where the domains leave SMs idle, up to eight
    const dim3 shared_by(nd, std::max(1, std::min(8, c->sms / std::max(nd, 1))));
    const size_t sm_obs = (size_t)c->host.n_h_max * (m + 1) * sizeof(T);
    const size_t sm_gram = (size_t)std::max(c->host.p_loc_max, 1) * (m + 1) * sizeof(T);
    const size_t sm_tr = ((size_t)m * m + (size_t)c->host.n_loc_max * (m + 1)) * sizeof(T);
    if ((rc = plain_kernels_ready<T>(c->device))) return rc;
    static_check_kernel<T><<<1, 1024, 0, c->stream>>>(y, c->p, flag, c->d_status);
    plain_obs<T><<<nd, kThreads, sm_obs, c->stream>>>(X, y, c->tab, c->so_off, S, dt, m, mp, row0, c->n_subv,
                                                      (T)(1.0 / sg), (T)(1.0 / m), flag);
    plain_gram<T><<<shared_by, kThreads, sm_gram, c->stream>>>(S, dt, c->tab, c->so_off, G, bv, m, mp, flag);
    launch_eig<T>(nd, c->stream, G, bv, W, m, mp, c->d_status, flag);
    plain_transform<T><<<shared_by, kThreads, sm_tr, c->stream>>>(X, Xo, W, c->tab, m, mp, c->n_act, (T)(1.0 / m), flag);
    if (cudaGetLastError() != cudaSuccess) return LETKF_ECUDA;
    if (cudaMemcpy2DAsync(out, (size_t)m * eb, Xo, (size_t)mp * eb, (size_t)m * eb, c->n, cudaMemcpyDeviceToDevice,
                          c->stream) != cudaSuccess)
        return LETKF_ECUDA;
    return LETKF_OK;
}

}  // namespace
}  // namespace letkf

extern "C" int letkf_analyze_static(letkf_ctx* c, const void* y_dev, double sigma, void* xa_dev) {
    if (!c || !y_dev || !xa_dev) return LETKF_EINVAL;
    if (c->path != LETKF_PATH_PLAIN) return LETKF_EINVAL;
    if (c->phase != 0) return LETKF_ESTATE;
    if (cudaSetDevice(c->device) != cudaSuccess) return LETKF_ECUDA;
    if (c->precision == LETKF_PREC_FP64)
        return letkf::analyze_static_t<double>(c, static_cast<const double*>(y_dev), sigma, static_cast<double*>(xa_dev));
    return letkf::analyze_static_t<float>(c, static_cast<const float*>(y_dev), sigma, static_cast<float*>(xa_dev));
}
