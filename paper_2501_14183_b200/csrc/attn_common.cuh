// Shared pieces of the attention forward / backward: workspace layout, TMA tensor maps, tile geometry.
#pragma once

#include <cuda.h>

#include "common.cuh"
#include "kernels.h"

namespace vardrop {

constexpr int kTile = 128;          // tokens per query tile and per key tile
constexpr int kDP = 64;             // elements per tile row (heads of 32 leave the upper half zero)
constexpr int kRowBytes = kDP * 2;  // one (token, head) row of bf16: 128 bytes = one swizzle row
constexpr int kTileBytes = kTile * kRowBytes;   // 16 KiB

struct AttnWs {
    size_t staged[2];         // [B, Ncap, H, D] bf16 copies of the kept rows of Q and of dO (selections of many tiles)
    size_t delta;             // [B, H, Ncap] fp32; few tiles: [B, H] int32 counters instead
    size_t dq_acc;            // [B, Ncap, H, 64] fp32
    size_t total;
    int Ncap;
};

inline AttnWs attn_layout(const vardrop_attn_cfg& c) {
    AttnWs w;
    w.Ncap = (c.N + kTile - 1) / kTile * kTile;
    size_t o = kWsHeaderBytes;
    for (size_t& s : w.staged) { s = o; o += align_up(static_cast<size_t>(c.B) * w.Ncap * c.H * kRowBytes, 1024); }
    w.delta = o; o += align_up(sizeof(float) * c.B * c.H * w.Ncap, 1024);
    w.dq_acc = o; o += align_up(static_cast<size_t>(c.B) * w.Ncap * c.H * kDP * sizeof(float), 1024);
    w.total = o;
    return w;
}

// Tensor map over a [B, tokens, H, D] bf16 tensor with the given element strides: box = one (b, h) tile of 128 tokens x 64
// elements, 128-byte swizzle.  What lies outside the tensor reads as zero: tokens past the end, and the upper half of a 64-element
// row of a tensor with D = 32.
int make_tile_map(CUtensorMap* map, const void* base, int D, int B, int tokens, int H, long long sB, long long sN, long long sH);

// Tensor map over the fp32 dQ' accumulator [B, Ncap, H, 64]: box = 128 tokens x 32 floats (one 128-byte swizzled row
// per token) of one head, the unit of the backward kernel's bulk reduce-add.
int make_acc_map(CUtensorMap* map, const void* base, int B, int Ncap, int H);

// Number of SMs of the current device (cached per thread and device).
int sm_count();

// Element strides of q, k, v (the head dimension is contiguous).
struct QkvLayout {
    long long sB, sN, sH;
};
inline QkvLayout qkv_layout(const vardrop_attn_cfg& c) {
    QkvLayout L;
    const bool dflt = c.sB == 0 && c.sN == 0 && c.sH == 0;
    L.sH = dflt ? c.D : c.sH;
    L.sN = dflt ? static_cast<long long>(c.H) * c.D : c.sN;
    L.sB = dflt ? static_cast<long long>(c.N) * c.H * c.D : c.sB;
    return L;
}

// First 1024-byte boundary at or after p (swizzled tiles need it).
__device__ __forceinline__ unsigned char* align_tiles(unsigned char* p) {
    return reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(p) + 1023) & ~static_cast<uintptr_t>(1023));
}

// ---- how a 128-token operand tile reaches shared memory ------------------------------------------------------------
// Without a selection: one box of the caller's tensor by the copy engine.  With one: 16-byte asynchronous copies of the kept
// variates' rows straight from the caller's tensor, any strides (row j of the tile is variate idx[tok0 + j], zeros from n_valid
// on).  (Row gathers by the copy engine, four rows an instruction, take 18 ns each, 0.6 us a tile: the many-tile forward of 1423 kept
// tokens ran 134 us with them against 97 with copies.)
__device__ __forceinline__ void cp_async16(uint32_t dst_smem, const void* src, uint32_t src_bytes) {      // src_bytes 16, or 0: zeros
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst_smem), "l"(src), "r"(src_bytes) : "memory");
}
// This thread arrives on `bar` once all its copies so far have landed (the barrier's count includes the arrival).  The tensor core
// reads through the async proxy: the waiter puts a proxy fence between its wait and the product.
__device__ __forceinline__ void cp_async_arrive(uint64_t* bar) {
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// Two warps share a tile, 64 rows each; `part` is this warp's place.  Eight lanes copy a row, lane group g = lane / 8 the sixteen rows
// from 64 part + 16 g on, whose sources every lane holds (no exchange between lanes: the copies share their issue queue with the
// exponentials of the softmax warps).
struct RowPicks {
    int n[16];                      // source rows, -1: none
};
__device__ __forceinline__ RowPicks tile_picks(const int32_t* idx, int tok0, int n_valid, int part) {
    RowPicks p;
    const int slot = tok0 + part * 64 + ((threadIdx.x & 31) >> 3) * 16;
    if (slot + 16 <= n_valid && (reinterpret_cast<uintptr_t>(idx + slot) & 15) == 0) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int4 v = __ldg(reinterpret_cast<const int4*>(idx + slot) + e);
            p.n[4 * e] = v.x; p.n[4 * e + 1] = v.y; p.n[4 * e + 2] = v.z; p.n[4 * e + 3] = v.w;
        }
    } else {
#pragma unroll
        for (int e = 0; e < 16; ++e) p.n[e] = slot + e < n_valid ? __ldg(idx + slot + e) : -1;
    }
    return p;
}
// The picked rows of one tensor to a tile, or of two tensors (with kTwo) to two tiles in a row.
template <bool kTwo>
__device__ __forceinline__ void copy_tile_rows(unsigned char* tile, const __nv_bfloat16* base, const __nv_bfloat16* base2, long long sN, const RowPicks& picks, int D, int part) {
    const int lane = threadIdx.x & 31, chunk = lane & 7;
    const uint32_t live = chunk * 8 < D ? 16u : 0u;             // heads of 32: the upper half of the row is zeros
    const int c0 = live ? chunk * 8 : 0;
    const uint32_t dst = smem_u32(tile) + (part * 64 + (lane >> 3) * 16) * kRowBytes;
#pragma unroll
    for (int it = 0; it < 16; ++it) {
        const long long off = static_cast<long long>(max(picks.n[it], 0)) * sN + c0;
        const uint32_t to = dst + it * kRowBytes + (static_cast<uint32_t>(chunk ^ (it & 7)) << 4), bytes = picks.n[it] >= 0 ? live : 0u;
        cp_async16(to, base + off, bytes);
        if (kTwo) cp_async16(to + kTileBytes, base2 + off, bytes);
    }
}
// One warp's share of a tile when the whole CTA loads: 32 rows from tok0 on.  (Two loader warps need some 500 cycles a tile, bound by
// the latency of their address chains; a dozen warps bring the first tiles of a CTA in together.)
__device__ __forceinline__ void copy_32_picked(unsigned char* rows, const __nv_bfloat16* base, long long sN, int pick, int D) {      // pick: this lane's row, -1: none
    const int lane = threadIdx.x & 31, chunk = lane & 7;
    const uint32_t live = chunk * 8 < D ? 16u : 0u;
    const __nv_bfloat16* src = base + (live ? chunk * 8 : 0);
    const uint32_t dst = smem_u32(rows) + (lane >> 3) * kRowBytes + (static_cast<uint32_t>(chunk ^ (lane >> 3)) << 4);
#pragma unroll
    for (int it = 0; it < 8; ++it) {
        const int n = __shfl_sync(0xffffffffu, pick, 4 * it + (lane >> 3));
        cp_async16((dst ^ ((it & 1) * 64u)) + it * 4 * kRowBytes, src + static_cast<long long>(max(n, 0)) * sN, n >= 0 ? live : 0u);
    }
}
__device__ __forceinline__ void copy_32_rows(unsigned char* rows, const __nv_bfloat16* base, long long sN, const int32_t* idx, int tok0, int n_valid, int D) {
    const int slot = tok0 + (threadIdx.x & 31);
    copy_32_picked(rows, base, sN, slot < n_valid ? (idx ? __ldg(idx + slot) : slot) : -1, D);
}
// Quotient of 0 <= a by 1 <= d in a few instructions (an integer division is some forty dependent ones); the correction loops run
// more than once only for quotients beyond 2^22.
__device__ __forceinline__ int small_div(int a, int d) {
    int q = static_cast<int>(__fdividef(static_cast<float>(a), static_cast<float>(d)));
    int r = a - q * d;
#pragma unroll 1
    while (r < 0) { r += d; --q; }
#pragma unroll 1
    while (r >= d) { r -= d; ++q; }
    return q;
}

// Whether a call may meet many key tiles per head and instance, and so runs the kernels for that (and the backward takes its row statistics,
// operand tiles and the conversion of dQ' from launches of their own): the kept count is only known on the device, so the host goes by the
// largest it can be.  A selection keeps a fraction of the variates (a tenth to a third in the paper's settings); up to kManyTilesN variates that
// is a handful of tiles.  With few heads and instances a tile's latency counts for more than the launches, and the line lies lower.  Forward and
// backward, B = 8, H = 8, few | many: 200 of 2000 kept 29 | 34 us, 400 56 | 48, 1000 153 | 115; B = 1: 110 of 1100 14 | 20, 200 of 2000 23 | 24, 400 41 | 31, 1000 85 | 44.
constexpr int kManyTilesN = 2048, kManyTilesSmallN = 1024, kSmallHeads = 32;
inline bool attn_many_tiles(const vardrop_attn_cfg& c, const int32_t* sel_idx) {
    return sel_idx ? c.N > (c.B * c.H < kSmallHeads ? kManyTilesSmallN : kManyTilesN) : c.N > 2 * kTile;
}

// Whether the forward pass clears the dQ' accumulator, under its own work: for a selection (only training passes one), and where no
// prep launch follows; without a selection the forward pass may be inference, and the prep launch does it.
inline bool attn_fwd_clears(const vardrop_attn_cfg& c, const int32_t* sel_idx) { return sel_idx != nullptr || !attn_many_tiles(c, sel_idx); }

// Number of selection rows: one shared by the batch (or none at all), or one per instance.
inline int attn_sel_rows(const vardrop_attn_cfg& c, const int32_t* sel_idx) { return sel_idx && c.S > 1 ? c.S : 1; }

// Kept count that sizes the work: of the one selection, the largest of several (each warp looks on its own), or N.
__device__ __forceinline__ int largest_kept(const int32_t* n_sel, int S, int N) {
    if (!n_sel) return N;
    if (S <= 1) return __ldg(n_sel);
    int m = 0;
#pragma unroll 1
    for (int s = threadIdx.x & 31; s < S; s += 32) m = max(m, __ldg(n_sel + s));
    return __reduce_max_sync(0xffffffffu, m);
}

}  // namespace vardrop
