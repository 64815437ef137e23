// Operand ring of the tiled tensor-core products: one thread fills stages of shared memory with bulk copies,
// another issues the products of a stage and hands it back.  Used by the GEMM kernel (gemm.cu, where the
// operand formats are described) and by the matrix iteration of the global analysis (root.cu).
#pragma once

#include <cuda_bf16.h>

#include <cstdint>

#include "umma.cuh"

namespace letkf {

constexpr int GEMM_TILE_B = 128 * 64 * 2;           // bytes of one operand tile
constexpr long long GEMM_WAIT = 4000000000LL;       // cycles

// One stage: KC columns of A (128 rows, hi and lo) and of B (bn rows or columns).  MN: a whole tile, B read
// MN-major; else SL slices of 16 columns.  A unit (tile or slice) is [A hi, A lo, B hi, B lo].
template <bool MN>
struct GemmStage {
    static constexpr int UC = MN ? 64 : 16, SL = MN ? 1 : 2, KC = UC * SL;    // columns of a unit, units, columns
    static constexpr int A_BYTES = 128 * 2 * UC;
    static constexpr int RING = 192 * 1024, MOST = MN ? 4 : 8;
};

// Where a thread stands in the ring: stages passed, the next one and its parity.
struct RingPos {
    int c = 0, s = 0, par = 0;
    __device__ __forceinline__ void next(int stages) {
        ++c;
        if (++s == stages) s = 0, par ^= 1;
    }
};

struct Ring {
    uint8_t* smem;
    uint64_t *full, *empty;
    int stages;
    uint32_t b_slot, unit, stage_b;     // bytes of B hi or lo in a unit, of a unit, of a stage
};

template <bool MN>
__device__ __forceinline__ Ring make_ring(uint8_t* smem, uint64_t* full, uint64_t* empty, int bn) {
    using L = GemmStage<MN>;
    Ring r;
    r.smem = smem;
    r.full = full;
    r.empty = empty;
    r.b_slot = (uint32_t)bn * 2 * L::UC;
    r.unit = 2 * L::A_BYTES + 2 * r.b_slot;
    r.stage_b = L::SL * r.unit;
    r.stages = min(L::MOST, L::RING / (int)r.stage_b);
    return r;
}

// Operands of one piece: a_* at its row tile and b_* at its columns, each from K = 0; a_lo null: single BF16.
struct RingOperands {
    const uint8_t *a_hi, *a_lo, *b_hi, *b_lo;
    int b_nkb;          // column tiles per row tile of B
    int width;          // columns of the piece
};
// K-major B (rows = N): the 128-row tile holding column col0, from the slice's second half for odd blocks of
// 64.  MN-major B (the second factor itself, rows = K; width 64): step k takes rows 64 k .. 64 k + 63 of
// column tile col0 / 64, the first or second half of that tile.
template <bool MN>
__device__ __forceinline__ RingOperands ring_operands(const uint8_t* a_hi, const uint8_t* a_lo, int a_nkb, int row_tile,
                                                      const uint8_t* b_hi, const uint8_t* b_lo, int b_nkb, int col0,
                                                      int width) {
    const size_t a = (size_t)row_tile * a_nkb * GEMM_TILE_B;
    const size_t b = MN ? (size_t)(col0 >> 6) * GEMM_TILE_B
                        : (size_t)(col0 >> 7) * b_nkb * GEMM_TILE_B + ((col0 & 64) ? GemmStage<MN>::A_BYTES / 2 : 0);
    return {a_hi + a, a_lo ? a_lo + a : nullptr, b_hi + b, a_lo ? b_lo + b : nullptr, b_nkb, width};
}

// Copies steps [k0, k1) (of KC columns) of a piece into the ring; one thread.  False: a wait ran out.
template <bool MN>
__device__ __forceinline__ bool ring_fill(const Ring& r, RingPos& p, const RingOperands& o, int k0, int k1) {
    using namespace umma;
    using L = GemmStage<MN>;
    const bool split = o.a_lo != nullptr;
    const uint32_t b_bytes = (uint32_t)o.width * 2 * L::UC;
    const uint32_t stage_bytes = (split ? 2u : 1u) * L::SL * (L::A_BYTES + b_bytes);
    const size_t b_next = (size_t)o.b_nkb * GEMM_TILE_B;
    // 256 columns are two consecutive 128-row tiles, copied next to each other so that one descriptor
    // with the same row-group stride spans all 256 rows
    auto copy_b = [&](uint8_t* dst, const uint8_t* src, uint64_t* bar) {
        bulk_g2s(dst, src, min(b_bytes, (uint32_t)L::A_BYTES), bar);
        if (b_bytes > L::A_BYTES) bulk_g2s(dst + L::A_BYTES, src + b_next, L::A_BYTES, bar);
    };
    for (int k = k0; k < k1; ++k) {
        uint64_t* full = &r.full[p.s];
        if (p.c >= r.stages && !mbar_wait_bounded(&r.empty[p.s], p.par ^ 1, GEMM_WAIT)) return false;
        mbar_arrive_expect_tx(full, stage_bytes);
#pragma unroll
        for (int u = 0; u < L::SL; ++u) {
            uint8_t* st = r.smem + p.s * r.stage_b + u * r.unit;
            const size_t ao = (size_t)(k * L::SL + u) * L::A_BYTES;
            const size_t bo = MN ? (size_t)(k >> 1) * b_next + (size_t)(k & 1) * (GEMM_TILE_B / 2) : ao;
            bulk_g2s(st, o.a_hi + ao, L::A_BYTES, full);
            copy_b(st + 2 * L::A_BYTES, o.b_hi + bo, full);
            if (split) {
                bulk_g2s(st + L::A_BYTES, o.a_lo + ao, L::A_BYTES, full);
                copy_b(st + 2 * L::A_BYTES + r.b_slot, o.b_lo + bo, full);
            }
        }
        p.next(r.stages);
    }
    return true;
}

// Issues the products of `steps` stages into the accumulator at TMEM column address dt; one elected thread.
template <bool MN>
__device__ __forceinline__ bool ring_issue(const Ring& r, RingPos& p, uint32_t dt, int width, bool split, int steps) {
    using namespace umma;
    using L = GemmStage<MN>;
    // A: K-adjacent core matrices 128 B apart, row-adjacent 1024 B in a tile, 256 B in a slice; K-major B
    // alike.  MN-major B: N-adjacent core matrices 128 B apart, K-adjacent 1024 B, a K step 2048 B
    constexpr uint32_t a_sbo = MN ? 1024u : 256u, b_lbo = MN ? 1024u : 128u, b_sbo = MN ? 128u : 256u;
    const uint32_t idesc = idesc_bf16(128, width, MN);
    for (int kc = 0; kc < steps; ++kc) {
        if (!mbar_wait_bounded(&r.full[p.s], p.par, GEMM_WAIT)) return false;
        tc_fence_after();
        const uint32_t st = smem_u32(r.smem + p.s * r.stage_b);
        const uint32_t sa_lo = st + L::A_BYTES, sb_hi = st + 2 * L::A_BYTES, sb_lo = sb_hi + r.b_slot;
#pragma unroll
        for (int k = 0; k < L::KC / 16; ++k) {
            const uint32_t da = MN ? 256u * k : r.unit * k, db = MN ? 2048u * k : r.unit * k;
            const uint64_t ah = sdesc(st + da, 128, a_sbo), bh = sdesc(sb_hi + db, b_lbo, b_sbo);
            mma_bf16(dt, ah, bh, idesc, (kc > 0 || k > 0) ? 1u : 0u);
            if (split) {
                mma_bf16(dt, ah, sdesc(sb_lo + db, b_lbo, b_sbo), idesc, 1u);
                mma_bf16(dt, sdesc(sa_lo + da, 128, a_sbo), bh, idesc, 1u);
            }
        }
        mma_commit(&r.empty[p.s]);
        p.next(r.stages);
    }
    return true;
}

// After a wait gave up: the copies of the last stages filled (`filled` in all) land before the CTA leaves.
__device__ __forceinline__ void ring_drain(const Ring& r, int filled) {
    for (int c = max(0, filled - r.stages); c < filled; ++c)
        umma::mbar_wait_bounded(&r.full[c % r.stages], (c / r.stages) & 1, GEMM_WAIT);
}

__device__ __forceinline__ void split_bf16(float x, __nv_bfloat16& h, __nv_bfloat16& l) {
    h = __float2bfloat16_rn(x);
    l = __float2bfloat16_rn(x - __bfloat162float(h));
}

// Byte offset of element (row, col) in a tiled operand with nkb column tiles.
__device__ __forceinline__ size_t tiled_offset(int row, int col, int nkb) {
    return ((size_t)(row >> 7) * nkb + (col >> 6)) * GEMM_TILE_B + umma::op_offset(row & 127, col & 63, 64);
}

}  // namespace letkf
