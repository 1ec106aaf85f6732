// Shared pieces of the attention backward kernels: parameters, the arithmetic between the products, the zero rows.
#pragma once

#include "attn_common.cuh"

namespace vardrop {

namespace {

__device__ __forceinline__ uint32_t pack2(float a, float b) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&v);
}
__device__ __forceinline__ float2 unpack2(uint32_t w) {
    return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w));
}
__device__ __forceinline__ float dot8(uint4 a, uint4 g) {
    const float2 a0 = unpack2(a.x), a1 = unpack2(a.y), a2 = unpack2(a.z), a3 = unpack2(a.w);
    const float2 g0 = unpack2(g.x), g1 = unpack2(g.y), g2 = unpack2(g.z), g3 = unpack2(g.w);
    return a0.x * g0.x + a0.y * g0.y + a1.x * g1.x + a1.y * g1.y + a2.x * g2.x + a2.y * g2.y + a3.x * g3.x + a3.y * g3.y;
}
__device__ __forceinline__ float sum8(float v) {       // over the eight lanes of a row
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    v += __shfl_xor_sync(0xffffffffu, v, 2);
    v += __shfl_xor_sync(0xffffffffu, v, 4);
    return v;
}

struct BwdParams {
    const __nv_bfloat16 *q, *k, *v;   // read by the row copies of a selection (boxes go through the tensor maps)
    const __nv_bfloat16* d_o;         // [B, N, H, D]
    const __nv_bfloat16* o;           // [B, N, H, D] forward output (rows 0 .. n_sel-1), for Delta
    const float* lse;       // [B, H, N]
    const float* delta;     // [B, H, Ncap] many tiles: Delta (few: computed here from o and dO)
    float* dq_acc;          // [B, Ncap, H, 64]
    __nv_bfloat16* dq;      // [B, N, H, D]
    __nv_bfloat16* dk;
    __nv_bfloat16* dv;
    const int32_t* sel_idx; // [S, N]; NULL: identity
    const int32_t* inv_idx; // [S, N]; NULL: identity (nothing dropped)
    int32_t* tile_done;     // few tiles: [B, H] items whose part of dQ' has landed; zeroed by the forward pass
    const int32_t* n_sel;   // [S]; NULL: N
    int* status;
    long long sB, sN, sH;   // element strides of q, k, v
    int B, N, Ncap, H, D, S;
    float scale, scale_log2;
    float half_inv_scale;   // many tiles: 0.5 / scale
};

inline BwdParams bwd_params(const void* q, const void* k, const void* v, const void* o, const float* lse, const void* d_o, const int32_t* sel_idx, const int32_t* n_sel,
                            const int32_t* inv_idx, const vardrop_attn_cfg& c, void* dq, void* dk, void* dv, void* ws) {
    const AttnWs w = attn_layout(c);
    const QkvLayout L = qkv_layout(c);
    char* base = static_cast<char*>(ws);
    BwdParams P{};
    P.q = static_cast<const __nv_bfloat16*>(q); P.k = static_cast<const __nv_bfloat16*>(k); P.v = static_cast<const __nv_bfloat16*>(v);
    P.d_o = static_cast<const __nv_bfloat16*>(d_o); P.o = static_cast<const __nv_bfloat16*>(o);
    P.lse = lse; P.delta = reinterpret_cast<const float*>(base + w.delta);
    P.dq_acc = reinterpret_cast<float*>(base + w.dq_acc);
    P.dq = static_cast<__nv_bfloat16*>(dq); P.dk = static_cast<__nv_bfloat16*>(dk); P.dv = static_cast<__nv_bfloat16*>(dv);
    P.sel_idx = sel_idx; P.n_sel = sel_idx ? n_sel : nullptr;
    P.inv_idx = sel_idx ? inv_idx : nullptr;
    P.tile_done = reinterpret_cast<int32_t*>(base + w.delta);
    P.status = reinterpret_cast<int*>(base);
    P.sB = L.sB; P.sN = L.sN; P.sH = L.sH;
    P.B = c.B; P.N = c.N; P.Ncap = w.Ncap; P.H = c.H; P.D = c.D; P.S = attn_sel_rows(c, sel_idx);
    P.scale = c.sm_scale > 0.f ? c.sm_scale : 1.f / sqrtf(static_cast<float>(c.D));
    P.scale_log2 = P.scale * 1.4426950408889634f;
    return P;
}

// The arithmetic between the products, as instructions that keep their order: left to itself the compiler puts the consumers of a pair
// of exponentials right behind it and a warp runs at the latency of the special-function unit instead of its rate.
__device__ __forceinline__ uint64_t pair_of(float lo, float hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void halves_of(uint64_t v, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }
__device__ __forceinline__ uint64_t fma_pair(uint64_t a, uint64_t b, uint64_t c) {      // two IEEE fp32 results per issue slot
    uint64_t d;
    asm volatile("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ uint64_t mul_pair(uint64_t a, uint64_t b) {
    uint64_t d;
    asm volatile("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ float fast_exp2(float x) {      // special-function unit; exp2(-inf) = 0
    float y;
    asm volatile("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    uint32_t d;
    asm volatile("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
    return d;
}

// A pair of floats from shared memory, issued here.  Read by all lanes alike, 8 bytes take 0.6 cycles of the shared-memory pipe, 16 bytes 2.1.
__device__ __forceinline__ uint64_t lds_pair(uint32_t addr) {
    uint64_t v;
    asm volatile("ld.shared.b64 %0, [%1];" : "=l"(v) : "r"(addr));
    return v;
}

// every lane of the warp waits; the result is the same in all of them
__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity) { return __all_sync(0xffffffffu, mbar_wait(bar, parity)); }
// the same with a sleep between polls
__device__ __forceinline__ bool warp_wait_relaxed(uint64_t* bar, uint32_t parity) { return __all_sync(0xffffffffu, mbar_wait_relaxed(bar, parity)); }

// Zero rows of dq, dk, dv for every dropped variate, by whichever warps of the CTA have nothing else to do: they take the CTA's rows eight at
// a time from a shared counter, look them up in inv_idx, and write one dropped row a call, 512 bytes a store instruction.  One row at a time,
// between other work: written in one go by every CTA at once they fill the memory's queues, and row loads behind them took 10000 cycles (200
// of 862 kept).
struct ZeroRows {
    int* taken;                         // groups of eight rows taken so far, by all warps of the CTA
    int base;
    unsigned mask;                      // dropped rows of the current group still to write
};
__device__ __forceinline__ bool write_zero_row(const BwdParams& P, ZeroRows& z) {      // false: none left
    const int lane = threadIdx.x & 31;
    if (!P.inv_idx) return false;
#pragma unroll 1
    while (z.mask == 0) {
        int g = 0;
        if (lane == 0) g = atomicAdd(z.taken, 1);
        z.base = (blockIdx.x + __shfl_sync(0xffffffffu, g, 0) * gridDim.x) * 8;
        if (z.base >= P.B * P.N) return false;
        const int r = z.base + lane;
        bool dropped = false;
        if (lane < 8 && r < P.B * P.N) {
            const int b = small_div(r, P.N), n = r - b * P.N;
            dropped = __ldg(P.inv_idx + static_cast<size_t>(P.S > 1 ? b : 0) * P.N + n) < 0;
        }
        z.mask = __ballot_sync(0xffffffffu, dropped);
    }
    const int chunks_row = P.H * (P.D / 8);                    // 16-byte chunks per (instance, variate) row
    const size_t row0 = static_cast<size_t>(z.base + __ffs(z.mask) - 1) * chunks_row;
    z.mask &= z.mask - 1;
    const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll 1
    for (int c = lane; c < chunks_row; c += 32) {
        reinterpret_cast<uint4*>(P.dq)[row0 + c] = zero;
        reinterpret_cast<uint4*>(P.dk)[row0 + c] = zero;
        reinterpret_cast<uint4*>(P.dv)[row0 + c] = zero;
    }
    return true;
}

// P^T = exp2(S^T scale - lse) of a thread's 32 queries, in place, and as bf16: batches of eight (exponents of g, exponentials of g - 1,
// rounding of g - 2) keep the special-function unit at its rate.
__device__ __forceinline__ void exp_step(float (&s)[32], uint32_t (&pk)[16], const uint64_t (&l)[16], uint64_t scale2) {
#pragma unroll
    for (int g = 0; g < 6; ++g) {
        if (g < 4) {
#pragma unroll
            for (int e = 8 * g; e < 8 * g + 8; e += 2) halves_of(fma_pair(pair_of(s[e], s[e + 1]), scale2, l[e >> 1]), s[e], s[e + 1]);
        }
        if (g >= 1 && g < 5) {
#pragma unroll
            for (int e = 8 * g - 8; e < 8 * g; ++e) s[e] = fast_exp2(s[e]);
        }
        if (g >= 2) {
#pragma unroll
            for (int e = 8 * g - 16; e < 8 * g - 8; e += 2) pk[e >> 1] = pack_bf16(s[e], s[e + 1]);
        }
    }
}
// dS^T = P^T o (dP^T - Delta) as bf16; Delta of eight queries is in registers, the next eight on their way.
__device__ __forceinline__ void ds_step(const float (&s)[32], float (&d)[32], uint32_t (&pk)[16], uint64_t (&dl)[2][4], uint32_t dlt) {
    const uint64_t minus1 = pair_of(-1.f, -1.f);
#pragma unroll
    for (int g = 0; g < 4; ++g) {
        if (g < 3) {
#pragma unroll
            for (int e = 0; e < 4; ++e) dl[(g + 1) & 1][e] = lds_pair(dlt + 32 * g + 32 + 8 * e);
        }
#pragma unroll
        for (int e = 8 * g; e < 8 * g + 8; e += 2) {
            halves_of(mul_pair(pair_of(s[e], s[e + 1]), fma_pair(dl[g & 1][(e >> 1) & 3], minus1, pair_of(d[e], d[e + 1]))), d[e], d[e + 1]);
            pk[e >> 1] = pack_bf16(d[e], d[e + 1]);
        }
    }
}
// Four 16-byte chunks (32 queries) of a row of a 64-query panel.
__device__ __forceinline__ void store_panel(unsigned char* panel, int row, int half, const uint32_t (&pk)[16]) {
#pragma unroll
    for (int q = 0; q < 4; ++q)
        *reinterpret_cast<uint4*>(panel + row * kRowBytes + (((half * 4 + q) ^ (row & 7)) << 4)) = make_uint4(pk[4 * q], pk[4 * q + 1], pk[4 * q + 2], pk[4 * q + 3]);
}

}  // namespace

}  // namespace vardrop
