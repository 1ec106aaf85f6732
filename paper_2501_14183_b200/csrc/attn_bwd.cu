// Attention backward over the kept variate tokens and the scatter of the gradients to the full layout.
//
// bwd_prep_kernel     many tiles: Delta_i = sum_d dO'_id O'_id, the kept rows laid out as tiles (selection), and the cleared dQ' accumulator
//                     (no selection: with one the forward pass clears it).
// attn_bwd_kernel     one CTA per SM.  Scores are formed transposed (S^T = K Q^T, dP^T = V dO^T) so that a thread owns (part of) a key row
//                     of tensor memory; P^T and dS^T feed dV += P^T dO, dK += dS^T Q and dQ_i = dS K.  Two shapes of the work:
//                       single   a kept set of one tile: two teams of 256 threads, each a whole (head, instance) on its own, no hand-offs
//                       pipeline several tiles: work items (128-key tile, head, instance), a warp role for each part of the work; dQ
//                                is added into an fp32 accumulator by bulk reduce-adds
//                     The same kernel writes the zero rows of every dropped variate.
// bwd_convert_kernel  many tiles: dQ' accumulator to bf16 rows of dq (fewer: by the CTA that finishes an (instance, head) pair).
//
// Each row of dq / dk / dv is written exactly once.
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

// ---------------------------------------------------------------------------------------------------------
// prep
// ---------------------------------------------------------------------------------------------------------
struct PrepParams {
    const uint4* o;         // [B, N, H, D] bf16
    const uint4* d_o;       // [B, N, H, D] bf16
    const __nv_bfloat16 *q, *k, *v;
    float* delta;           // [B, H, Ncap]
    float4* dq_acc;         // [B, Ncap, H, 64] fp32; NULL: cleared by the forward pass
    uint4* staged[4];       // [B, Ncap, H, D] bf16 copies of the kept rows of Q, K, V, and of dO: with a selection
    const int32_t* sel_idx; // [S, N]; NULL: identity, nothing is staged
    const int32_t* n_sel;   // [S] kept counts; NULL: N
    long long sB, sN, sH;
    int N, Ncap, H, D, S;
};

// One thread per 16-byte chunk of a (token, head) row of 64; the 8 threads of a row reduce Delta by shuffles.  With a selection the rows
// that the main kernel reads again for every key tile are laid out here once, zeros up to the tile's end (rows of dO past the kept ones
// may hold anything), so that it takes boxes: row copies by its two loader warps bound it at 1423 kept tokens (250 us against 170).
__global__ void __launch_bounds__(256) bwd_prep_kernel(const PrepParams P) {
    chain_wait();
    chain_release();
    const int b = blockIdx.y;
    const int n_sel = P.n_sel ? P.n_sel[P.S > 1 ? b : 0] : P.N;
    const int n_fill = min(P.Ncap, (n_sel + kTile - 1) / kTile * kTile);
    const int chunks_row = P.H * 8;
    const int src_chunks_head = P.D / 8;
    const int total = n_fill * chunks_row;            // a multiple of 8; blockDim is a multiple of 8
    const int32_t* sel = P.sel_idx ? P.sel_idx + static_cast<size_t>(P.S > 1 ? b : 0) * P.N : nullptr;
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += gridDim.x * blockDim.x) {
        const int i = small_div(idx, chunks_row);
        const int c = idx - i * chunks_row;
        const int h = c >> 3, dc = c & 7;
        uint4 vo = make_uint4(0u, 0u, 0u, 0u), vd = vo, vq = vo, vk = vo, vv = vo;
        if (i < n_sel && dc < src_chunks_head) {
            const size_t src = (static_cast<size_t>(b) * P.N + i) * (P.H * src_chunks_head) + h * src_chunks_head + dc;
            vo = __ldg(P.o + src);
            vd = __ldg(P.d_o + src);
            if (sel) {
                const long long from = b * P.sB + __ldg(sel + i) * P.sN + h * P.sH + dc * 8;
                vq = __ldg(reinterpret_cast<const uint4*>(P.q + from));
                vk = __ldg(reinterpret_cast<const uint4*>(P.k + from));
                vv = __ldg(reinterpret_cast<const uint4*>(P.v + from));
            }
        }
        if (sel && dc < src_chunks_head) {
            const size_t to = ((static_cast<size_t>(b) * P.Ncap + i) * P.H + h) * src_chunks_head + dc;
            P.staged[0][to] = vq; P.staged[1][to] = vk; P.staged[2][to] = vv; P.staged[3][to] = vd;
        }
        const float part = sum8(dot8(vo, vd));
        if (dc == 0) P.delta[(static_cast<size_t>(b) * P.H + h) * P.Ncap + i] = part;
        if (P.dq_acc) {
            const size_t dst = (static_cast<size_t>(b) * P.Ncap + i) * chunks_row + c;
            P.dq_acc[2 * dst] = make_float4(0.f, 0.f, 0.f, 0.f);
            P.dq_acc[2 * dst + 1] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
    }
}

// ---------------------------------------------------------------------------------------------------------
// main
// ---------------------------------------------------------------------------------------------------------
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
    int32_t* tile_done;     // [B, H] key tiles finished per (instance, head); zeroed by the forward pass
    const int32_t* n_sel;   // [S]; NULL: N
    int* status;
    long long sB, sN, sH;   // element strides of q, k, v
    int B, N, Ncap, H, D, S;
    float scale, scale_log2;
};

constexpr int kBwdGroup = 256;
// Few key tiles: the first warpgroup issues and loads, two worker groups follow, one of which also takes dQ out of tensor memory.  Many: a
// second warpgroup of its own takes dQ out (8192 variates: 3500 us against 3790 without it; one or two tiles: 23 us against 19).
// Register split (setmaxnreg works on whole warpgroups), within what the block was launched with: few, 640 x 96 = 128 x 64 + 512 x 104;
// many, 768 x 80 = 256 x 48 + 512 x 96.
template <bool kMany>
struct BwdShape {
    static constexpr int kFirst = kMany ? 8 : 4;                   // first worker warp
    static constexpr int kThreads = kFirst * 32 + 2 * kBwdGroup;
    static constexpr int kSmallRegs = kMany ? 48 : 64, kBigRegs = kMany ? 96 : 104;
};
constexpr uint32_t kBwdTmemCols = 512;
constexpr int kSlots = 3;              // ring of query-tile operands (Q tile, dO tile)
constexpr int kBwdHeader = 6144;       // barriers, item list, row statistics
constexpr int kBwdSmemBytes = kBwdHeader + 2 * kTileBytes /*K, V*/ + 2 * kSlots * kTileBytes /*Q, dO ring*/ + 2 * kTileBytes /*dS^T*/ +
                              2 * kTileBytes /*dQ tile, fp32, two 32-column halves*/;

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

// every lane of the warp waits; the result is the same in all of them
__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity) { return __all_sync(0xffffffffu, mbar_wait(bar, parity)); }
// the same with a sleep between polls
__device__ __forceinline__ bool warp_wait_relaxed(uint64_t* bar, uint32_t parity) { return __all_sync(0xffffffffu, mbar_wait_relaxed(bar, parity)); }

// named barrier among 256 threads (id 1 or 2), with an and-reduction of ok
__device__ __forceinline__ bool group_sync_and(int id, bool ok) {
    uint32_t r;
    asm volatile(
        "{\n.reg .pred p, q;\n"
        "setp.ne.b32 q, %1, 0;\n"
        "bar.red.and.pred p, %2, 256, q;\n"
        "selp.u32 %0, 1, 0, p;\n}"
        : "=r"(r)
        : "r"(static_cast<uint32_t>(ok)), "r"(id)
        : "memory");
    return r != 0;
}
__device__ __forceinline__ bool drain_sync_and(bool ok) {     // the same among the 128 threads that take dQ out
    uint32_t r;
    asm volatile(
        "{\n.reg .pred p, q;\n"
        "setp.ne.b32 q, %1, 0;\n"
        "bar.red.and.pred p, 3, 128, q;\n"
        "selp.u32 %0, 1, 0, p;\n}"
        : "=r"(r)
        : "r"(static_cast<uint32_t>(ok))
        : "memory");
    return r != 0;
}
__device__ __forceinline__ void group_sync(int id) { asm volatile("bar.sync %0, 256;" ::"r"(id) : "memory"); }

// Zero rows of dq, dk, dv for every dropped variate, by warps off the critical path.  The rows of all instances are dealt out in rounds
// of 32 per warp: `part` of `parts` warps of the grid looks rows (part + round parts) 32 .. + 31 up in inv_idx, one a lane, and
// writes the dropped ones, 512 bytes a store instruction.
__device__ __forceinline__ int zero_row_rounds(const BwdParams& P, int parts) { return P.inv_idx ? (P.B * P.N + parts * 32 - 1) / (parts * 32) : 0; }
__device__ __forceinline__ void zero_rows_round(const BwdParams& P, int part, int parts, int round) {
    const int lane = threadIdx.x & 31;
    const int chunks_row = P.H * (P.D / 8);                    // 16-byte chunks per (instance, variate) row
    const int base = (part + round * parts) * 32;
    const int r = base + lane;
    bool dropped = false;
    if (r < P.B * P.N) {
        const int b = small_div(r, P.N), n = r - b * P.N;
        dropped = __ldg(P.inv_idx + static_cast<size_t>(P.S > 1 ? b : 0) * P.N + n) < 0;
    }
    unsigned mask = __ballot_sync(0xffffffffu, dropped);
    const uint4 z = make_uint4(0u, 0u, 0u, 0u);
    uint4* dq4 = reinterpret_cast<uint4*>(P.dq);
    uint4* dk4 = reinterpret_cast<uint4*>(P.dk);
    uint4* dv4 = reinterpret_cast<uint4*>(P.dv);
#pragma unroll 1
    while (mask) {
        const int l = __ffs(mask) - 1;
        mask &= mask - 1;
        const size_t row0 = static_cast<size_t>(base + l) * chunks_row;
#pragma unroll 1
        for (int c = lane; c < chunks_row; c += 32) { dq4[row0 + c] = z; dk4[row0 + c] = z; dv4[row0 + c] = z; }
    }
}

// This thread's 32 columns (half `half`) of its row of a 64-column accumulator, scaled and rounded, to a bf16 staging tile.
__device__ __forceinline__ void stage_acc(unsigned char* tile, uint32_t tm, float mul, int row, int half) {
    unsigned char* rowp = tile + row * kRowBytes;
    float acc[32];
    tmem_ld32(tm + half * 32, acc);
    tmem_ld_wait();
#pragma unroll
    for (int q = 0; q < 4; ++q)
        *reinterpret_cast<uint4*>(rowp + (((half * 4 + q) ^ (row & 7)) << 4)) =
            make_uint4(pack2(acc[8 * q + 0] * mul, acc[8 * q + 1] * mul), pack2(acc[8 * q + 2] * mul, acc[8 * q + 3] * mul),
                       pack2(acc[8 * q + 4] * mul, acc[8 * q + 5] * mul), pack2(acc[8 * q + 6] * mul, acc[8 * q + 7] * mul));
}
// Rows of a staging tile to the full-layout gradient, 16 bytes a thread, eight threads a row, 256 threads: n[x] is the variate of row
// gt / 8 + 32 x, or -1.
__device__ __forceinline__ void store_rows(const unsigned char* tile, __nv_bfloat16* dst, const int (&n)[4], int gt, const BwdParams& P, int b, int h) {
    const int c = gt & 7, r0 = gt >> 3;
    if (c * 8 >= P.D) return;
    __nv_bfloat16* out = dst + (static_cast<size_t>(b) * P.N * P.H + h) * P.D + c * 8;
    const unsigned char* from = tile + r0 * kRowBytes + ((c ^ (r0 & 7)) << 4);
#pragma unroll
    for (int x = 0; x < 4; ++x)
        if (n[x] >= 0) *reinterpret_cast<uint4*>(out + static_cast<size_t>(n[x]) * P.H * P.D) = *reinterpret_cast<const uint4*>(from + x * 32 * kRowBytes);
}

// ---------------------------------------------------------------------------------------------------------
// single: a kept set of one tile
// ---------------------------------------------------------------------------------------------------------
// A team of 256 threads (two per key row, 64 queries each) does a (head, instance) by itself; the two teams of a CTA, and nothing else,
// fill each other's waits: with one tile the work is a chain of latencies (rows in, scores, exponentials, gradients, rows out) whose
// every path runs once or twice, so hand-offs between roles and unrolled code only lengthen it.
// Team memory: Q, K, V, dO, dS^T (two 64-query panels); tensor memory (256 columns): S^T [0,128), dP^T [128,256); P^T (bf16) goes over the
// first half of each 64-column half of S^T, dV and dK over dP^T, dQ over P^T once dV has read it.
__device__ __forceinline__ void bwd_single(const BwdParams& P, int kept, unsigned char* tiles, float* stats, uint64_t* bar, uint32_t tm0, int team, int gt, bool& ok) {
    unsigned char* sQ = tiles + team * 6 * kTileBytes;
    unsigned char* sdO = sQ + 3 * kTileBytes;           // Q, K, V, dO
    unsigned char* sdS = sQ + 4 * kTileBytes;
    float* s_lse = stats + team * 4 * kTile;            // minus the lse of a query, log2 domain
    float* s_none = s_lse + kTile;                      // the same for key rows that do not exist: -inf throughout
    float* s_delta = s_none + kTile;
    int* s_nout = reinterpret_cast<int*>(s_delta + kTile);
    const int warp = gt >> 5, row = gt & (kTile - 1), half = gt >> 7, id = team + 1;
    const uint32_t tm = tm0 + (static_cast<uint32_t>((warp & 3) * 32) << 16);
    const uint64_t d_q = umma_desc_sw128(smem_u32(sQ), 16, 1024), m_q = umma_desc_sw128(smem_u32(sQ), kTileBytes, 1024);
    const uint64_t scale2 = pair_of(P.scale_log2, P.scale_log2), minus1 = pair_of(-1.f, -1.f);
    if (half == 0) s_none[row] = -INFINITY;
    uint32_t t = 0;
#pragma unroll 1
    for (int item = blockIdx.x + team * gridDim.x; item < P.H * P.B && ok; item += 2 * gridDim.x, ++t) {
        const int b = small_div(item, P.H), h = item - b * P.H;
        const int n = P.S > 1 ? P.n_sel[b] : kept;
        const int32_t* idx = P.sel_idx ? P.sel_idx + static_cast<size_t>(P.S > 1 ? b : 0) * P.N : nullptr;
        if (n <= 0) { --t; continue; }
        // rows: every warp a quarter of Q or K, then of V or dO
#pragma unroll 1
        for (int x = warp >> 2; x < 4; x += 2) {
            const bool own = x < 3;                     // dO is compact and contiguous
            const __nv_bfloat16* from = own ? (x == 0 ? P.q : x == 1 ? P.k : P.v) + b * P.sB + h * P.sH : P.d_o + (static_cast<size_t>(b) * P.N * P.H + h) * P.D;
            copy_32_rows(sQ + x * kTileBytes + (warp & 3) * 32 * kRowBytes, from, own ? P.sN : static_cast<long long>(P.H) * P.D, own ? idx : nullptr,
                         (warp & 3) * 32, n, P.D);
            asm volatile("cp.async.commit_group;" ::: "memory");
        }
        if (half == 0) s_lse[row] = row < n ? P.lse[(static_cast<size_t>(b) * P.H + h) * P.N + row] * -1.4426950408889634f : -INFINITY;
        else s_nout[row] = row < n ? (idx ? __ldg(idx + row) : row) : -1;
        uint4 o[4];                                     // rows gt / 8 + 32 x of O, 16 bytes each, for Delta
        const int c8 = gt & 7, r8 = gt >> 3;
        {
            const __nv_bfloat16* from = P.o + (static_cast<size_t>(b) * P.N * P.H + h) * P.D + c8 * 8;
#pragma unroll
            for (int x = 0; x < 4; ++x)
                o[x] = r8 + 32 * x < n && c8 * 8 < P.D ? __ldg(reinterpret_cast<const uint4*>(from + static_cast<size_t>(r8 + 32 * x) * P.H * P.D)) : make_uint4(0u, 0u, 0u, 0u);
        }
        const uint32_t n16 = (n + 15) & ~15;
        asm volatile("cp.async.wait_group 1;" ::: "memory");             // Q, K
        fence_proxy_async_smem();
        tc_fence_before();
        group_sync(id);
        if (warp == 0) {
            tc_fence_after();
            if (elect_one()) {
#pragma unroll 1
                for (int ks = 0; ks < P.D / 16; ++ks)
                    tc_mma_bf16(tm0, umma_desc_advance(d_q, kTileBytes + ks * 32), umma_desc_advance(d_q, ks * 32), umma_idesc_bf16(128, n16, 0, 0), ks > 0);
            }
            __syncwarp();
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");             // V, dO
        fence_proxy_async_smem();
        tc_fence_before();
        group_sync(id);
        if (warp == 0) {
            tc_fence_after();
            if (elect_one()) {
#pragma unroll 1
                for (int ks = 0; ks < P.D / 16; ++ks)
                    tc_mma_bf16(tm0 + 128, umma_desc_advance(d_q, 2 * kTileBytes + ks * 32), umma_desc_advance(d_q, 3 * kTileBytes + ks * 32),
                                umma_idesc_bf16(128, n16, 0, 0), ks > 0);
                tc_commit(bar);
            }
            __syncwarp();
        }
#pragma unroll
        for (int x = 0; x < 4; ++x) {                   // Delta
            const int r = r8 + 32 * x;
            const float part = sum8(dot8(o[x], *reinterpret_cast<const uint4*>(sdO + r * kRowBytes + ((c8 ^ (r & 7)) << 4))));
            if (c8 == 0) s_delta[r] = part;
        }
        group_sync(id);
        ok = mbar_wait(bar, t & 1);
        tc_fence_after();
        // P^T = exp2(S^T scale - lse) and dS^T = P^T o (dP^T - Delta), 32 queries at a time
        const float* lse = row < n ? s_lse : s_none;
#pragma unroll 1
        for (int c = 0; c < 2; ++c) {
            const int q0 = half * 64 + c * 32;
            if (q0 >= n) break;
            float s[32], d[32];
            uint32_t pk[16];
            tmem_ld32(tm + q0, s);
            tmem_ld32(tm + 128 + q0, d);
            tmem_ld_wait();
#pragma unroll
            for (int g = 0; g < 6; ++g) {                // batches of eight: exponents of g, exponentials of g - 1, the rest of g - 2
                if (g < 4) {
#pragma unroll
                    for (int i = 8 * g; i < 8 * g + 8; i += 4) {
                        const float4 l4 = *reinterpret_cast<const float4*>(lse + q0 + i);
                        halves_of(fma_pair(pair_of(s[i], s[i + 1]), scale2, pair_of(l4.x, l4.y)), s[i], s[i + 1]);
                        halves_of(fma_pair(pair_of(s[i + 2], s[i + 3]), scale2, pair_of(l4.z, l4.w)), s[i + 2], s[i + 3]);
                    }
                }
                if (g >= 1 && g < 5) {
#pragma unroll
                    for (int i = 8 * g - 8; i < 8 * g; ++i) s[i] = fast_exp2(s[i]);
                }
                if (g >= 2) {
#pragma unroll
                    for (int i = 8 * g - 16; i < 8 * g - 8; i += 4) {
                        const float4 d4 = *reinterpret_cast<const float4*>(s_delta + q0 + i);
                        const uint64_t p01 = pair_of(s[i], s[i + 1]), p23 = pair_of(s[i + 2], s[i + 3]);
                        halves_of(mul_pair(p01, fma_pair(pair_of(d4.x, d4.y), minus1, pair_of(d[i], d[i + 1]))), d[i], d[i + 1]);
                        halves_of(mul_pair(p23, fma_pair(pair_of(d4.z, d4.w), minus1, pair_of(d[i + 2], d[i + 3]))), d[i + 2], d[i + 3]);
                        pk[i >> 1] = pack_bf16(s[i], s[i + 1]);
                        pk[(i >> 1) + 1] = pack_bf16(s[i + 2], s[i + 3]);
                    }
                }
            }
            tmem_st16(tm + half * 64 + c * 16, pk);
            unsigned char* to = sdS + half * kTileBytes + row * kRowBytes;
#pragma unroll
            for (int q = 0; q < 4; ++q)
                *reinterpret_cast<uint4*>(to + (((c * 4 + q) ^ (row & 7)) << 4)) =
                    make_uint4(pack_bf16(d[8 * q], d[8 * q + 1]), pack_bf16(d[8 * q + 2], d[8 * q + 3]), pack_bf16(d[8 * q + 4], d[8 * q + 5]), pack_bf16(d[8 * q + 6], d[8 * q + 7]));
        }
        tmem_st_wait();
        fence_proxy_async_smem();
        tc_fence_before();
        ok = group_sync_and(id, ok);
        if (!ok) break;
        if (warp == 0) {
            tc_fence_after();
            if (elect_one()) {
                const uint32_t idesc_kmn = umma_idesc_bf16(128, P.D, 0, 1), idesc_mnmn = umma_idesc_bf16(128, P.D, 1, 1);
                const int k_steps = n16 >> 4;
#pragma unroll 1
                for (int ks = 0; ks < k_steps; ++ks)     // dV = P^T dO
                    tc_mma_bf16_ta(tm0 + 128, tm0 + (ks >> 2) * 64 + (ks & 3) * 8, umma_desc_advance(m_q, 3 * kTileBytes + ks * 2048), idesc_kmn, ks > 0);
#pragma unroll 1
                for (int ks = 0; ks < k_steps; ++ks)     // dK = dS^T Q
                    tc_mma_bf16(tm0 + 192, umma_desc_advance(d_q, (4 + (ks >> 2)) * kTileBytes + (ks & 3) * 32), umma_desc_advance(m_q, ks * 2048), idesc_kmn, ks > 0);
#pragma unroll 1
                for (int ks = 0; ks < k_steps; ++ks)     // dQ = dS K (dS: the transposed view of the same tile)
                    tc_mma_bf16(tm0, umma_desc_advance(m_q, 4 * kTileBytes + ks * 2048), umma_desc_advance(m_q, kTileBytes + ks * 2048), idesc_mnmn, ks > 0);
                tc_commit(bar + 1);
            }
            __syncwarp();
        }
        ok = mbar_wait(bar + 1, t & 1);
        tc_fence_after();
        // every product is done: dV and dK are staged over dS^T, dQ over V
        int nout[4];
#pragma unroll
        for (int x = 0; x < 4; ++x) nout[x] = s_nout[r8 + 32 * x];
#pragma unroll 1
        for (int x = 0; x < 3; ++x) stage_acc(x < 2 ? sdS + x * kTileBytes : sQ + 2 * kTileBytes, tm + (x == 0 ? 128 : x == 1 ? 192 : 0), x == 0 ? 1.f : P.scale, row, half);
        tc_fence_before();
        ok = group_sync_and(id, ok);
        if (!ok) break;
#pragma unroll 1
        for (int x = 0; x < 3; ++x) store_rows(x < 2 ? sdS + x * kTileBytes : sQ + 2 * kTileBytes, x == 0 ? P.dv : x == 1 ? P.dk : P.dq, nout, gt, P, b, h);
        group_sync(id);                                  // the tiles are free
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
}

// ---------------------------------------------------------------------------------------------------------
// the kernel
// ---------------------------------------------------------------------------------------------------------
// Pipeline: the query loop of a key tile is two phases on 256 threads each, phase A of query tile i + 1 beside phase B of tile i (warp
// numbers of the few-tile form; in the many-tile form four warps that take dQ out come between the loaders and the phases).
//   warps 0, 1   issue the products (all lanes run the issue code, an elected lane executes a group of products): S^T and dV, the chain
//                through P^T, and dP^T, dK and dQ, the chain through dS^T
//   warps 2, 3   load K, V and a ring of (Q, dO) tiles with their row statistics; warp 3 decodes the items, warp 2 writes the zero rows
//   warps 4-11   phase A: P^T = exp2(S^T scale - lse), bf16, to tensor memory (the A operand of dV += P^T dO)
//   warps 12-19  phase B: dS^T = P^T o (dP^T - Delta) to shared memory (dK += dS^T Q, and dQ = dS K through the transposed view); dQ of the
//                tile before out of tensor memory for the bulk reduce-add; dV and dK of a finished key tile
// A phase frees what it has copied to registers at once: S^T and dP^T of the next tile are produced under the arithmetic of this one, and
// dS^T stays in registers until dK and dQ of the tile before have read the shared-memory tile.  (dS^T handed to dK through dP^T's own
// columns, as an earlier form did, makes phase B wait for dK and the next dP^T: 3900 cycles a tile pair.)
// What bounds it: shared-memory bandwidth and the hand-offs around it (a tile pair reads and writes some 270 KB of shared memory, 2200
// cycles, where its products need 1280) with many tiles; the chain of latencies with few.  Measured, B = 32, H = 8, D = 64: 119 kept 19 us
// (27 before), 200 kept 76 us without prep and convert launches (57 + 11 + 11); all of 862 215 us (229); all of 8192, B = 8, 3590 us (3640);
// 1423 kept of 8192, B = 8, 174 us.
// Tensor memory: S^T [0,128) dP^T [128,256) dV [256,320) dK [320,384) dQ [384,448) P^T [448,512).
template <bool kMany>
__global__ void __launch_bounds__(BwdShape<kMany>::kThreads, 1) attn_bwd_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                                                                   const __grid_constant__ CUtensorMap map_v, const __grid_constant__ CUtensorMap map_do,
                                                                   const __grid_constant__ CUtensorMap map_acc, const BwdParams P) {
    constexpr int kFirst = BwdShape<kMany>::kFirst;
    extern __shared__ unsigned char smem_dyn[];
    // Set-up first (shared-memory carve-up, barriers, tensor memory): it touches nothing another kernel produces, so it runs
    // while the previous kernel of the stream is still finishing.
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem_dyn);
    uint64_t* bar_kv_full = bars + 0;
    uint64_t* bar_kv_free = bars + 1;               // every product of the item is done (both issue warps)
    uint64_t* bar_q_full = bars + 2;                // [kSlots]
    uint64_t* bar_q_free = bar_q_full + kSlots;     // [kSlots] every product reading the slot is done (both issue warps)
    uint64_t* bar_s = bar_q_free + kSlots;          // S^T of a query tile complete
    uint64_t* bar_sfree = bar_s + 1;                // phase A holds S^T in registers (256)
    uint64_t* bar_p = bar_s + 2;                    // P^T in tensor memory (256)
    uint64_t* bar_pfree = bar_s + 3;                // phase B holds P^T in registers (256) and dV has read it (1)
    uint64_t* bar_dp = bar_s + 4;                   // dP^T of a query tile complete
    uint64_t* bar_dpfree = bar_s + 5;               // phase B holds dP^T in registers (256)
    uint64_t* bar_ds = bar_s + 6;                   // dS^T in shared memory (256)
    uint64_t* bar_dsfree = bar_s + 7;               // many: dK and dQ have read dS^T
    uint64_t* bar_g = bar_s + 8;                    // dQ of a query tile complete (few: and dK before it, dS^T has been read)
    uint64_t* bar_dqfree = bar_s + 9;               // dQ has left tensor memory (128 or 256)
    uint64_t* bar_acc = bar_s + 10;                 // dV, dK of the item final (both issue warps)
    uint64_t* bar_accfree = bar_s + 11;             // phase B holds them in registers (256)
    uint64_t* bar_first = bar_s + 13;               // the first item's row copies have landed (512)
    uint64_t* bar_item = bar_s + 14;                // [8] entry of the item list is written
    uint64_t* bar_team = bar_item + 8;              // [2][2] single: scores, gradients
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bar_team + 4);
    int* s_flag = reinterpret_cast<int*>(tmem_slot + 1);
    struct alignas(16) Item { int jt, h, b, n_sel; };               // n_sel < 0 ends the list
    Item* s_item = reinterpret_cast<Item*>(smem_dyn + 384);         // [8]
    float* s_lse = reinterpret_cast<float*>(smem_dyn + 512);        // [kSlots][128] minus the lse of the query tile in the slot, log2 domain
    float* s_delta = s_lse + kSlots * kTile;                        // [kSlots][128] its Delta
    static_assert(2 * kSlots <= 8, "the single teams keep eight arrays of 128 there");
    unsigned char* sK = align_tiles(reinterpret_cast<unsigned char*>(s_lse + 8 * kTile));
    unsigned char* sQ = sK + 2 * kTileBytes;            // kSlots slots of (Q tile, dO tile)
    unsigned char* sdSt = sQ + 2 * kSlots * kTileBytes; // dS^T : rows = keys, columns = queries (two 64-query panels); dV, dK staging at the end of an item
    unsigned char* sDQ = sdSt + 2 * kTileBytes;         // dQ_i as fp32: panel `half` = head dimensions 32 half .. 32 half + 31, 128-byte swizzled rows
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (sDQ + 2 * kTileBytes > smem_dyn + kBwdSmemBytes) {
        chain_wait();
        if (tid == 0) set_status(P.status, VARDROP_ERR_CUDA);
        return;
    }
    const bool boxes = kMany || P.sel_idx == nullptr;
    if (warp == 0) {
        tmem_alloc(tmem_slot, kBwdTmemCols);
        tmem_relinquish();
    }
    if (tid == 0) {
        // a box: one announcing arrival; row copies: one of every loader lane, and one of each loader for the row statistics
        mbar_init(bar_kv_full, boxes ? 1 : 64);
        mbar_init(bar_kv_free, 2);
        for (int st = 0; st < kSlots; ++st) {
            mbar_init(bar_q_full + st, boxes ? 1 : 66);
            mbar_init(bar_q_free + st, 2);
        }
        mbar_init(bar_s, 1);
        mbar_init(bar_sfree, kBwdGroup);
        mbar_init(bar_p, kBwdGroup);
        mbar_init(bar_pfree, kBwdGroup + 1);
        mbar_init(bar_dp, 1);
        mbar_init(bar_dpfree, kBwdGroup);
        mbar_init(bar_ds, kBwdGroup);
        mbar_init(bar_g, 1);
        mbar_init(bar_dsfree, 1);
        mbar_init(bar_dqfree, kMany ? kTile : kBwdGroup);
        mbar_init(bar_acc, 2);
        mbar_init(bar_accfree, kBwdGroup);
        mbar_init(bar_first, 2 * kBwdGroup);
        for (int i = 0; i < 8; ++i) mbar_init(bar_item + i, 1);
        for (int i = 0; i < 4; ++i) mbar_init(bar_team + i, 1);
        mbar_fence_init();
        if (boxes) {
            tma_prefetch_desc(&map_q);
            tma_prefetch_desc(&map_k);
            tma_prefetch_desc(&map_v);
            tma_prefetch_desc(&map_do);
        }
        tma_prefetch_desc(&map_acc);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    bool ok = true;
    int kept = 0, n_t = 0, n_items = 0;
    auto begin = [&]() {
        chain_wait();
        chain_release();
        kept = largest_kept(P.n_sel, P.S, P.N);
        n_t = (kept + kTile - 1) / kTile;                      // tiles of the longest selection
        n_items = n_t * P.H * P.B;                             // pipeline: (key tile, head, instance); short instances skip tiles
    };

    auto item_at = [&](uint32_t i) {
        Item it;
        ok &= warp_wait_relaxed(bar_item + (i & 7), (i >> 3) & 1);
        const int4 x = *reinterpret_cast<const int4*>(s_item + (i & 7));
        it.jt = x.x; it.h = x.y; it.b = x.z; it.n_sel = ok ? x.w : -1;
        return it;
    };

    if (warp < kFirst) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(BwdShape<kMany>::kSmallRegs));
    begin();
    // One backward pass per forward pass: the forward kernel left a mark (and cleared this workspace's counters); a backward pass that
    // does not find it (a second backward for the same forward, or two forwards sharing the workspace before their backwards) would
    // add into stale state, so it reports the call instead of returning wrong gradients.
    if (blockIdx.x == 0 && tid == 0 && atomicExch(P.status + kWsPairingWord, 0) != 1) set_status(P.status, VARDROP_ERR_INVALID_ARG);
    if (!kMany && n_t <= 1) {
        const int parts = 4 * gridDim.x, rounds = zero_row_rounds(P, parts);
#pragma unroll 1
        for (int round = 0; round < rounds; ++round) zero_rows_round(P, blockIdx.x * 4 + warp, parts, round);
    } else if (warp < 2) {
        // ------------------------------------------------------------ issue ---------------------------------------------
        const uint32_t idesc_kk = umma_idesc_bf16(128, 128, 0, 0);         // K-major x K-major, N = 128
        const uint32_t idesc_kmn = umma_idesc_bf16(128, P.D, 0, 1);        // A K-major, B MN-major
        const uint32_t idesc_mnmn = umma_idesc_bf16(128, P.D, 1, 1);       // A MN-major, B MN-major
        const uint64_t d_k = umma_desc_sw128(smem_u32(sK), 16, 1024), m_k = umma_desc_sw128(smem_u32(sK), kTileBytes, 1024);
        constexpr uint32_t kQOff = 2 * kTileBytes, kDsOff = (2 + 2 * kSlots) * kTileBytes;
        uint32_t t = 0;                                  // query tiles so far
#pragma unroll 1
        for (uint32_t i = 0; ok; ++i) {
            const Item it = item_at(i);
            if (it.n_sel < 0) break;
            const int n_q = (it.n_sel + kTile - 1) / kTile;
            ok &= warp_wait_relaxed(bar_kv_full, i & 1);
            auto wait_slot = [&](uint32_t tt) {
                ok &= warp_wait_relaxed(bar_q_full + tt % kSlots, (tt / kSlots) & 1);
                if (!boxes) fence_proxy_async_smem();    // rows written by asynchronous copies are read by the tensor core
                tc_fence_after();
            };
            auto scores = [&](uint32_t tt) {             // S^T = K Q^T (warp 0) or dP^T = V dO^T (warp 1) of query tile tt
                wait_slot(tt);
                const uint32_t q_off = kQOff + (tt % kSlots) * 2 * kTileBytes;
                if (elect_one()) {
                    const uint64_t a = umma_desc_advance(d_k, warp * kTileBytes), bd = umma_desc_advance(d_k, q_off + warp * kTileBytes);
                    const uint32_t d = tmem + warp * 128;
                    tc_mma_bf16(d, a, bd, idesc_kk, 0u);
                    tc_mma_bf16(d, umma_desc_advance(a, 32), umma_desc_advance(bd, 32), idesc_kk, 1u);
                    if (P.D > 32) {
                        tc_mma_bf16(d, umma_desc_advance(a, 64), umma_desc_advance(bd, 64), idesc_kk, 1u);
                        tc_mma_bf16(d, umma_desc_advance(a, 96), umma_desc_advance(bd, 96), idesc_kk, 1u);
                    }
                    tc_commit(warp == 0 ? bar_s : bar_dp);
                }
                __syncwarp();
            };
            scores(t);
#pragma unroll 1
            for (int x = 0; x < n_q && ok; ++x, ++t) {
                const uint32_t slot = t % kSlots, q_off = kQOff + slot * 2 * kTileBytes, acc = x > 0 ? 1u : 0u;
                if (x + 1 < n_q) {           // the next tile's scores, as soon as this one's are in registers
                    ok &= warp_wait_relaxed(warp == 0 ? bar_sfree : bar_dpfree, t & 1);
                    scores(t + 1);
                }
                if (warp == 0) {
                    ok &= warp_wait_relaxed(bar_p, t & 1);
                    if (x == 0 && i > 0) ok &= warp_wait_relaxed(bar_accfree, (i - 1) & 1);     // dV, dK of the previous item are out
                    tc_fence_after();
                    if (elect_one()) {                   // dV += P^T dO over the 128 queries
                        const uint64_t bd = umma_desc_advance(m_k, q_off + kTileBytes);
#pragma unroll
                        for (int ks = 0; ks < 8; ++ks) tc_mma_bf16_ta(tmem + 256, tmem + 448 + ks * 8, umma_desc_advance(bd, ks * 2048), idesc_kmn, ks > 0 ? 1u : acc);
                        tc_commit(bar_pfree);
                        tc_commit(bar_q_free + slot);
                    }
                } else {
                    ok &= warp_wait_relaxed(bar_ds, t & 1);
                    tc_fence_after();
                    const uint64_t ad = umma_desc_advance(d_k, kDsOff), bd = umma_desc_advance(m_k, q_off), am = umma_desc_advance(m_k, kDsOff);
                    auto issue_dk = [&]() {              // dK += dS^T Q (phase B has seen P^T of this tile: dV's wait for bar_accfree precedes)
#pragma unroll
                        for (int ks = 0; ks < 8; ++ks)
                            tc_mma_bf16(tmem + 320, umma_desc_advance(ad, (ks >> 2) * kTileBytes + (ks & 3) * 32), umma_desc_advance(bd, ks * 2048), idesc_kmn, ks > 0 ? 1u : acc);
                        tc_commit(bar_q_free + slot);
                    };
                    if (!kMany && elect_one()) issue_dk();
                    __syncwarp();
                    if (t > 0) ok &= warp_wait_relaxed(bar_dqfree, (t - 1) & 1);      // the previous dQ has left tensor memory
                    tc_fence_after();
                    if (elect_one()) {                   // dQ = dS K over the 128 keys, dS the transposed view of the tile
#pragma unroll
                        for (int ks = 0; ks < 8; ++ks)
                            tc_mma_bf16(tmem + 384, umma_desc_advance(am, ks * 2048), umma_desc_advance(m_k, ks * 2048), idesc_mnmn, ks > 0);
                        tc_commit(bar_g);
                        if (kMany) {                     // many: dQ first, it leaves tensor memory under dK
                            issue_dk();
                            tc_commit(bar_dsfree);
                        }
                    }
                }
                __syncwarp();
            }
            tc_commit_w(bar_acc);
            tc_commit_w(bar_kv_free);
        }
    } else if (warp < 4) {
        // ------------------------------------------------------------ loads ---------------------------------------------
        const int part = warp == 3 ? 0 : 1;
        int k = blockIdx.x;                              // next item to publish, in grid steps
        auto publish = [&](uint32_t i) {
            Item it{0, 0, 0, -1};
#pragma unroll 1
            for (; it.n_sel < 0 && k < n_items; k += gridDim.x) {
                const int hb = small_div(k, n_t);
                it.jt = k - hb * n_t;
                it.b = small_div(hb, P.H);
                it.h = hb - it.b * P.H;
                const int n = P.S > 1 ? P.n_sel[it.b] : kept;
                if (it.jt * kTile < n) it.n_sel = n;
            }
            if (lane == 0) {
                *reinterpret_cast<int4*>(s_item + (i & 7)) = make_int4(it.jt, it.h, it.b, it.n_sel);
                mbar_arrive(bar_item + (i & 7));
            }
            __syncwarp();
        };
        uint32_t t = 0;
        int z_round = 0;
        const int z_rounds = part == 1 ? zero_row_rounds(P, gridDim.x) : 0;
        if (kMany)                                       // nothing else to do for this warp
#pragma unroll 1
            for (; z_round < z_rounds; ++z_round) zero_rows_round(P, blockIdx.x, gridDim.x, z_round);
        const int z_slice = (z_rounds + n_t - 1) / n_t;  // rounds behind every query tile: done within the first item's
        if (part == 0) publish(0);
#pragma unroll 1
        for (uint32_t i = 0; ok; ++i) {
            if (part == 0) publish(i + 1);
            const Item it = item_at(i);
            if (it.n_sel < 0) break;
            const int n_q = (it.n_sel + kTile - 1) / kTile;
            int x = 0;
            // Row statistics of a query tile travel with it: asked for ahead of the wait for the slot, four rows a lane.
            const float* lse_row = P.lse + (static_cast<size_t>(it.b) * P.H + it.h) * P.N;
            const float* delta_row = P.delta ? P.delta + (static_cast<size_t>(it.b) * P.H + it.h) * P.Ncap : nullptr;
            const bool has_lse = part == 0, has_delta = delta_row && (boxes || part == 1);
            float st_lse[4], st_delta[4];
            auto stats_load = [&](int tile) {
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int r = tile * kTile + e * 32 + lane;
                    st_lse[e] = has_lse && r < it.n_sel ? __ldg(lse_row + r) : INFINITY;
                    st_delta[e] = has_delta && r < it.n_sel ? __ldg(delta_row + r) : 0.f;
                }
            };
            auto stats_store = [&](uint32_t slot) {      // minus the lse in the log2 domain: -inf switches a missing query off
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    if (has_lse) s_lse[slot * kTile + e * 32 + lane] = st_lse[e] * -1.4426950408889634f;
                    if (has_delta) s_delta[slot * kTile + e * 32 + lane] = st_delta[e];
                }
                __syncwarp();
            };
            if (boxes) {
                if (part == 0) {
                    ok = warp_wait_relaxed(bar_kv_free, (i & 1) ^ 1);
                    if (!ok) break;
                    if (lane == 0) {
                        mbar_expect_tx(bar_kv_full, 2 * kTileBytes);
                        tma_load_4d(sK, &map_k, bar_kv_full, 0, it.h, it.jt * kTile, it.b);
                        tma_load_4d(sK + kTileBytes, &map_v, bar_kv_full, 0, it.h, it.jt * kTile, it.b);
                    }
                    __syncwarp();
#pragma unroll 1
                    for (; x < n_q; ++x, ++t) {
                        const uint32_t slot = t % kSlots;
                        stats_load(x);
                        ok = warp_wait_relaxed(bar_q_free + slot, ((t / kSlots) & 1) ^ 1);
                        if (!ok) break;
                        stats_store(slot);
                        if (lane == 0) {
                            mbar_expect_tx(bar_q_full + slot, 2 * kTileBytes);
                            tma_load_4d(sQ + slot * 2 * kTileBytes, &map_q, bar_q_full + slot, 0, it.h, x * kTile, it.b);
                            tma_load_4d(sQ + slot * 2 * kTileBytes + kTileBytes, &map_do, bar_q_full + slot, 0, it.h, x * kTile, it.b);
                        }
                        __syncwarp();
                    }
                }
            } else {
                const int32_t* idx = P.sel_idx + static_cast<size_t>(P.S > 1 ? it.b : 0) * P.N;
                const long long base = it.b * P.sB + it.h * P.sH;
                const __nv_bfloat16* d_o = P.d_o + (static_cast<size_t>(it.b) * P.N * P.H + it.h) * P.D;
                if (i == 0) {                            // brought in by the other warps: pass it on
                    stats_load(0);
                    stats_store(0);
                    if (lane == 0) mbar_arrive(bar_q_full);
                    ok = warp_wait(bar_first, 0);
                    if (!ok) break;
                    mbar_arrive(bar_kv_full);
                    mbar_arrive(bar_q_full);
                    x = 1;
                    t = 1;
                } else {
                    ok = warp_wait_relaxed(bar_kv_free, (i & 1) ^ 1);
                    if (!ok) break;
                    copy_tile_rows<true>(sK, P.k + base, P.v + base, P.sN, tile_picks(idx, it.jt * kTile, it.n_sel, part), P.D, part);
                    cp_async_arrive(bar_kv_full);
                }
#pragma unroll 1
                for (; x < n_q; ++x, ++t) {
                    const uint32_t slot = t % kSlots;
                    RowPicks picks = tile_picks(idx, x * kTile, it.n_sel, part);
                    stats_load(x);
                    ok = warp_wait_relaxed(bar_q_free + slot, ((t / kSlots) & 1) ^ 1);
                    if (!ok) break;
                    stats_store(slot);
                    if (lane == 0) mbar_arrive(bar_q_full + slot);
                    unsigned char* to = sQ + slot * 2 * kTileBytes;
                    const __nv_bfloat16* from = P.q + base;
                    long long step = P.sN;
#pragma unroll 1
                    for (int e = 0; e < 2; ++e) {        // Q rows, then dO rows (compact and contiguous)
                        copy_tile_rows<false>(to, from, nullptr, step, picks, P.D, part);
                        if (e == 0) {
                            const int slot0 = x * kTile + part * 64 + (lane >> 3) * 16;
#pragma unroll
                            for (int r = 0; r < 16; ++r) picks.n[r] = slot0 + r < it.n_sel ? slot0 + r : -1;
                            to += kTileBytes;
                            from = d_o;
                            step = static_cast<long long>(P.H) * P.D;
                        }
                    }
                    cp_async_arrive(bar_q_full + slot);
#pragma unroll 1
                    for (int z = 0; z < z_slice && z_round < z_rounds; ++z, ++z_round) zero_rows_round(P, blockIdx.x, gridDim.x, z_round);
                }
            }
        }
#pragma unroll 1
        for (; z_round < z_rounds; ++z_round) zero_rows_round(P, blockIdx.x, gridDim.x, z_round);
        asm volatile("cp.async.wait_all;" ::: "memory");
    } else if (kMany) {
        // ------------------------------------------------------------ dQ out of tensor memory ---------------------------
        const int row = tid & (kTile - 1);
        const uint32_t tm = tmem + 384 + (static_cast<uint32_t>((warp & 3) * 32) << 16);
        const bool owner = row == 0;                     // the one thread that owns the bulk reductions
        uint32_t t = 0;
#pragma unroll 1
        for (uint32_t i = 0; ok; ++i) {
            const Item it = item_at(i);
            if (it.n_sel < 0) break;
            const int n_q = (it.n_sel + kTile - 1) / kTile;
#pragma unroll 1
            for (int x = 0; x < n_q; ++x, ++t) {
                if (owner) bulk_wait_group_read0();      // the previous reduction has read the staging tile
                ok &= warp_wait_relaxed(bar_g, t & 1);
                ok = drain_sync_and(ok);
                if (!ok) break;
                tc_fence_after();
#pragma unroll 1
                for (int c = 0; c < P.D; c += 32) {
                    float v[32];
                    tmem_ld32(tm + c, v);
                    tmem_ld_wait();
                    if (c + 32 >= P.D) {
                        tc_fence_before();
                        mbar_arrive(bar_dqfree);         // dQ is in registers: the next one may be produced
                    }
                    unsigned char* to = sDQ + (c >> 5) * kTileBytes + row * kRowBytes;      // fp32, 32-column panels of 128-byte swizzled rows
#pragma unroll
                    for (int e = 0; e < 8; ++e)
                        *reinterpret_cast<float4*>(to + (e ^ (row & 7)) * 16) = make_float4(v[4 * e], v[4 * e + 1], v[4 * e + 2], v[4 * e + 3]);
                }
                fence_proxy_async_smem();
                drain_sync_and(true);                    // the staging tile is complete
                if (owner) {
                    tma_reduce_add_4d(&map_acc, sDQ, 0, it.h, x * kTile, it.b);
                    if (P.D > 32) tma_reduce_add_4d(&map_acc, sDQ + kTileBytes, 32, it.h, x * kTile, it.b);
                    bulk_commit_group();
                }
            }
        }
        if (owner) bulk_wait_group0();                   // the last dQ reductions have landed
    }
    } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(BwdShape<kMany>::kBigRegs));
    begin();
    if (!kMany && n_t <= 1) {
        const int team = (warp - 4) >> 3;
        bwd_single(P, kept, sK, s_lse, bar_team + 2 * team, tmem + team * 256, team, (tid - 128) & (kBwdGroup - 1), ok);
    } else {
        // ------------------------------------------------------------ workers -------------------------------------------
        const int gt = (tid - kFirst * 32) & (kBwdGroup - 1), row = gt & (kTile - 1), half = gt >> 7;
        const uint32_t tm = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16);
        const int c8 = gt & 7, r8 = gt >> 3;
        if (!boxes) {                                    // the first item's K, V, Q, dO rows: one 32-row group a warp
            const Item it = item_at(0);
            if (it.n_sel >= 0) {
                const int x = (warp - kFirst) >> 2, g = (warp & 3) * 32;
                const bool own = x < 3;
                const __nv_bfloat16* from = own ? (x == 0 ? P.k : x == 1 ? P.v : P.q) + it.b * P.sB + it.h * P.sH : P.d_o + (static_cast<size_t>(it.b) * P.N * P.H + it.h) * P.D;
                copy_32_rows(sK + x * kTileBytes + g * kRowBytes, from, own ? P.sN : static_cast<long long>(P.H) * P.D,
                             own ? P.sel_idx + static_cast<size_t>(P.S > 1 ? it.b : 0) * P.N : nullptr, (x < 2 ? it.jt * kTile : 0) + g, it.n_sel, P.D);
                cp_async_arrive(bar_first);
            }
        }
        uint32_t t = 0;
        if (warp < kFirst + 8) {
            // -------------------------------------------------------- phase A: P^T ---------------------------------------
            const uint64_t scale2 = pair_of(P.scale_log2, P.scale_log2);
#pragma unroll 1
            for (uint32_t i = 0; ok; ++i) {
                const Item it = item_at(i);
                if (it.n_sel < 0) break;
                const int n_q = (it.n_sel + kTile - 1) / kTile;
                const bool key_valid = it.jt * kTile + row < it.n_sel;
#pragma unroll 1
                for (int x = 0; x < n_q; ++x, ++t) {
                    const bool have = mbar_test(bar_q_full + t % kSlots, (t / kSlots) & 1);     // the row statistics, with the tile
                    ok &= warp_wait(bar_s, t & 1);
                    if (!__all_sync(0xffffffffu, have)) ok &= warp_wait(bar_q_full + t % kSlots, (t / kSlots) & 1);
                    tc_fence_after();
                    float s[64];
                    tmem_ld32(tm + half * 64, s);
                    tmem_ld32(tm + half * 64 + 32, s + 32);
                    tmem_ld_wait();
                    tc_fence_before();
                    mbar_arrive(bar_sfree);              // S^T is in registers
                    uint32_t pw[32];
                    const float* lse2 = s_lse + (t % kSlots) * kTile + half * 64;
                    const bool p_free = t == 0 || mbar_test(bar_pfree, (t - 1) & 1);
#pragma unroll
                    for (int g = 0; g < 10; ++g) {       // batches of eight: exponents of g, exponentials of g - 1, rounding of g - 2
                        if (g < 8) {
#pragma unroll
                            for (int e = 8 * g; e < 8 * g + 8; e += 4) {
                                const float4 l4 = *reinterpret_cast<const float4*>(lse2 + e);
                                halves_of(fma_pair(pair_of(s[e], s[e + 1]), scale2, pair_of(l4.x, l4.y)), s[e], s[e + 1]);
                                halves_of(fma_pair(pair_of(s[e + 2], s[e + 3]), scale2, pair_of(l4.z, l4.w)), s[e + 2], s[e + 3]);
                            }
                        }
                        if (g >= 1 && g < 9) {
#pragma unroll
                            for (int e = 8 * g - 8; e < 8 * g; ++e) s[e] = fast_exp2(s[e]);
                        }
                        if (g >= 2) {
#pragma unroll
                            for (int e = 8 * g - 16; e < 8 * g - 8; e += 2) pw[e >> 1] = pack_bf16(s[e], s[e + 1]);
                        }
                    }
                    if (!key_valid) {                    // rows past n_sel hold zero keys: they must not count
#pragma unroll
                        for (int e = 0; e < 32; ++e) pw[e] = 0u;
                    }
                    if (!__all_sync(0xffffffffu, p_free)) ok &= warp_wait(bar_pfree, (t - 1) & 1);      // the previous P^T has been read by phase B and by dV
                    tc_fence_after();
                    tmem_st32(tm + 448 + half * 32, pw);
                    tmem_st_wait();
                    tc_fence_before();
                    mbar_arrive(bar_p);                  // dV may go, phase B may read P^T
                    if (!ok) break;
                }
            }
        } else {
            // -------------------------------------------------------- phase B: dS^T --------------------------------------
            const uint64_t minus1 = pair_of(-1.f, -1.f);
            const bool owner = gt == 0;                  // the one thread that owns the bulk reductions of dQ
            // dQ of query tile x of the item is in registers: to the fp32 staging tile, which one thread adds to the accumulator.
            auto reduce_dq = [&](const Item& it, int x, const float (&v)[32]) {
                if (owner) bulk_wait_group_read0();      // the reduction before, a tile ago, has read the staging tile
                group_sync(2);
                unsigned char* to = sDQ + half * kTileBytes + row * kRowBytes;
                if (half * 32 < P.D) {
#pragma unroll
                    for (int e = 0; e < 8; ++e) *reinterpret_cast<float4*>(to + (e ^ (row & 7)) * 16) = make_float4(v[4 * e], v[4 * e + 1], v[4 * e + 2], v[4 * e + 3]);
                }
                fence_proxy_async_smem();
                group_sync(2);
                if (owner) {
                    tma_reduce_add_4d(&map_acc, sDQ, 0, it.h, x * kTile, it.b);
                    if (P.D > 32) tma_reduce_add_4d(&map_acc, sDQ + kTileBytes, 32, it.h, x * kTile, it.b);
                    bulk_commit_group();
                }
            };
#pragma unroll 1
            for (uint32_t i = 0; ok; ++i) {
                const Item it = item_at(i);
                if (it.n_sel < 0) break;
                const int n_q = (it.n_sel + kTile - 1) / kTile;
                const __nv_bfloat16* o_row = P.o + (static_cast<size_t>(it.b) * P.N * P.H + it.h) * P.D + c8 * 8;
#pragma unroll 1
                for (int x = 0; x < n_q; ++x, ++t) {
                    float* dlt = s_delta + (t % kSlots) * kTile;
                    if (!kMany) {                        // Delta of this query tile: eight threads a row of O (from memory) and dO (from the slot)
                        uint4 o[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const int r = x * kTile + r8 + 32 * e;
                            o[e] = r < it.n_sel && c8 * 8 < P.D ? __ldg(reinterpret_cast<const uint4*>(o_row + static_cast<size_t>(r) * P.H * P.D)) : make_uint4(0u, 0u, 0u, 0u);
                        }
                        ok &= warp_wait(bar_q_full + t % kSlots, (t / kSlots) & 1);
                        const unsigned char* sdO = sQ + (t % kSlots) * 2 * kTileBytes + kTileBytes;
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const int r = r8 + 32 * e;
                            const float part = sum8(dot8(o[e], *reinterpret_cast<const uint4*>(sdO + r * kRowBytes + ((c8 ^ (r & 7)) << 4))));
                            if (c8 == 0) dlt[r] = part;
                        }
                        group_sync(2);
                    }
                    const bool have = mbar_test(bar_q_full + t % kSlots, (t / kSlots) & 1);
                    ok &= warp_wait(bar_p, t & 1);
                    if (!__all_sync(0xffffffffu, have)) ok &= warp_wait(bar_q_full + t % kSlots, (t / kSlots) & 1);
                    tc_fence_after();
                    uint32_t pw[32];                     // this thread's 64 probabilities, bf16 pairs; then its dS^T
                    tmem_ld32(tm + 448 + half * 32, reinterpret_cast<float*>(pw));
                    tmem_ld_wait();
                    tc_fence_before();
                    mbar_arrive(bar_pfree);
                    ok &= warp_wait(bar_dp, t & 1);
                    tc_fence_after();
                    uint64_t* bar_read = kMany ? bar_dsfree : bar_g;     // dK and dQ of a tile have read its dS^T
                    const bool ds_free = t == 0 || mbar_test(bar_read, (t - 1) & 1);
                    float dp[2][16];
                    tmem_ld16(tm + 128 + half * 64, dp[0]);
#pragma unroll
                    for (int c = 0; c < 4; ++c) {        // 16 queries at a time, the next ones on their way
                        float4 da[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) da[e] = *reinterpret_cast<const float4*>(dlt + half * 64 + c * 16 + 4 * e);
                        tmem_ld_wait();
                        if (c < 3) tmem_ld16(tm + 128 + half * 64 + (c + 1) * 16, dp[(c + 1) & 1]);
                        else { tc_fence_before(); mbar_arrive(bar_dpfree); }      // dP^T is in registers: the next one may be produced
                        const float* d = dp[c & 1];
#pragma unroll
                        for (int e = 0; e < 16; e += 4) {
                            const uint32_t w0 = pw[c * 8 + (e >> 1)], w1 = pw[c * 8 + (e >> 1) + 1];
                            const uint64_t p01 = pair_of(__uint_as_float(w0 << 16), __uint_as_float(w0 & 0xFFFF0000u));
                            const uint64_t p23 = pair_of(__uint_as_float(w1 << 16), __uint_as_float(w1 & 0xFFFF0000u));
                            float r0, r1, r2, r3;
                            halves_of(mul_pair(p01, fma_pair(pair_of(da[e >> 2].x, da[e >> 2].y), minus1, pair_of(d[e], d[e + 1]))), r0, r1);
                            halves_of(mul_pair(p23, fma_pair(pair_of(da[e >> 2].z, da[e >> 2].w), minus1, pair_of(d[e + 2], d[e + 3]))), r2, r3);
                            pw[c * 8 + (e >> 1)] = pack_bf16(r0, r1);
                            pw[c * 8 + (e >> 1) + 1] = pack_bf16(r2, r3);
                        }
                    }
                    if (!__all_sync(0xffffffffu, ds_free)) ok &= warp_wait(bar_read, (t - 1) & 1);
                    float dq[32];                        // few: dQ of the previous tile
                    if (!kMany && x > 0) {
                        tc_fence_after();
                        tmem_ld32(tm + 384 + half * 32, dq);
                        tmem_ld_wait();
                        tc_fence_before();
                        mbar_arrive(bar_dqfree);         // the next dQ may be produced
                    }
                    {
                        unsigned char* to = sdSt + half * kTileBytes + row * kRowBytes;
#pragma unroll
                        for (int q = 0; q < 8; ++q) *reinterpret_cast<uint4*>(to + ((q ^ (row & 7)) << 4)) = make_uint4(pw[4 * q], pw[4 * q + 1], pw[4 * q + 2], pw[4 * q + 3]);
                    }
                    fence_proxy_async_smem();
                    mbar_arrive(bar_ds);                 // dQ and dK may go
                    if (!kMany && x > 0) reduce_dq(it, x - 1, dq);
                    if (!ok) break;
                }
                ok = group_sync_and(2, ok);
                if (!ok) break;
                const int32_t* sel = P.sel_idx ? P.sel_idx + static_cast<size_t>(P.S > 1 ? it.b : 0) * P.N : nullptr;
                int nout[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int key = it.jt * kTile + r8 + 32 * e;
                    nout[e] = key < it.n_sel ? (sel ? __ldg(sel + key) : key) : -1;
                }
                // dQ of the last tile
                if (!kMany) {
                    ok = warp_wait(bar_g, (t - 1) & 1);
                    tc_fence_after();
                }
                if (kMany) {
                } else if (n_q > 1) {
                    float dq[32];
                    tmem_ld32(tm + 384 + half * 32, dq);
                    tmem_ld_wait();
                    tc_fence_before();
                    mbar_arrive(bar_dqfree);
                    reduce_dq(it, n_q - 1, dq);
                } else {                                 // nothing to accumulate: rounded and written here (key rows = query rows)
                    stage_acc(sDQ, tm + 384, P.scale, row, half);
                    tc_fence_before();
                    mbar_arrive(bar_dqfree);
                    group_sync(2);
                    store_rows(sDQ, P.dq, nout, gt, P, it.b, it.h);
                }
                // dV and dK of the key tile, staged over dS^T
                ok = warp_wait(bar_acc, i & 1);
                tc_fence_after();
#pragma unroll 1
                for (int e = 0; e < 2; ++e) stage_acc(sdSt + e * kTileBytes, tm + 256 + e * 64, e == 0 ? 1.f : P.scale, row, half);
                tc_fence_before();
                mbar_arrive(bar_accfree);
                ok = group_sync_and(2, ok);
                if (!ok) break;
#pragma unroll 1
                for (int e = 0; e < 2; ++e) store_rows(sdSt + e * kTileBytes, e == 0 ? P.dv : P.dk, nout, gt, P, it.b, it.h);
                group_sync(2);                           // the staging tiles are free
                if (!kMany && n_q > 1) {         // dQ' of this (instance, head) is complete once all its key tiles are: the last one converts it
                    if (owner) {
                        bulk_wait_group0();              // this item's reductions have landed
                        __threadfence();
                        *s_flag = atomicAdd(P.tile_done + it.b * P.H + it.h, 1) == n_q - 1;
                    }
                    group_sync(2);
                    if (*s_flag) {
                        __threadfence();
                        const int chunks_head = P.D / 8, sh = P.D > 32 ? 3 : 2;       // 16-byte output chunks per row
#pragma unroll 2
                        for (int e = gt; e < it.n_sel * chunks_head; e += kBwdGroup) {
                            const int j = e >> sh, dc = e & (chunks_head - 1);
                            const float4* acc = reinterpret_cast<const float4*>(P.dq_acc + ((static_cast<size_t>(it.b) * P.Ncap + j) * P.H + it.h) * kDP) + dc * 2;
                            const float4 a0 = __ldcg(acc), a1 = __ldcg(acc + 1);
                            const int n = sel ? __ldg(sel + j) : j;
                            *reinterpret_cast<uint4*>(P.dq + ((static_cast<size_t>(it.b) * P.N + n) * P.H + it.h) * P.D + dc * 8) =
                                make_uint4(pack2(a0.x * P.scale, a0.y * P.scale), pack2(a0.z * P.scale, a0.w * P.scale),
                                           pack2(a1.x * P.scale, a1.y * P.scale), pack2(a1.z * P.scale, a1.w * P.scale));
                        }
                    }
                    group_sync(2);                       // the flag is free
                }
            }
            if (!kMany && owner) bulk_wait_group0();     // the last dQ reductions have landed
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
    }
    }
    if (!ok) set_status(P.status, VARDROP_ERR_TIMEOUT);
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, kBwdTmemCols);
}

// ---------------------------------------------------------------------------------------------------------
// dq from the accumulator (paths with many key tiles)
// ---------------------------------------------------------------------------------------------------------
struct ConvertParams {
    const float4* dq_acc;    // [B, Ncap, H, 64] fp32
    uint4* dq;               // [B, N, H, D] bf16
    const int32_t* inv_idx;  // [S, N]; NULL: identity
    const int32_t* n_sel;    // [S]; NULL: N
    int N, Ncap, H, D, S;
    float scale;
};

__global__ void __launch_bounds__(256) bwd_convert_kernel(const ConvertParams P) {
    chain_wait();
    chain_release();
    const int b = blockIdx.y;
    const int srow = P.S > 1 ? b : 0;
    const int32_t* inv = P.inv_idx ? P.inv_idx + static_cast<size_t>(srow) * P.N : nullptr;
    const int chunks_head = P.D / 8;
    const int chunks_row = P.H * chunks_head;
    const int total = P.N * chunks_row;
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += gridDim.x * blockDim.x) {
        const int n = idx / chunks_row;
        const int c = idx - n * chunks_row;
        const int h = c / chunks_head, dc = c - h * chunks_head;
        const int j = inv ? inv[n] : n;
        if (j < 0) continue;                                     // dropped rows were zeroed by the main kernel
        const float4* src = P.dq_acc + ((static_cast<size_t>(b) * P.Ncap + j) * P.H + h) * (kDP / 4) + dc * 2;
        const float4 a = __ldcg(src), c2 = __ldcg(src + 1);
        P.dq[static_cast<size_t>(b) * total + idx] = make_uint4(pack2(a.x * P.scale, a.y * P.scale), pack2(a.z * P.scale, a.w * P.scale),
                                                                pack2(c2.x * P.scale, c2.y * P.scale), pack2(c2.z * P.scale, c2.w * P.scale));
    }
}

}  // namespace

int attn_bwd_launch(const void* q, const void* k, const void* v, const void* o, const float* lse, const void* d_o,
                    const int32_t* sel_idx, const int32_t* n_sel, const int32_t* inv_idx, const vardrop_attn_cfg& c, void* dq,
                    void* dk, void* dv, void* ws, cudaStream_t stream) {
    const AttnWs w = attn_layout(c);
    const QkvLayout L = qkv_layout(c);
    char* base = static_cast<char*>(ws);
    const float scale = c.sm_scale > 0.f ? c.sm_scale : 1.f / sqrtf(static_cast<float>(c.D));
    const long long HD = static_cast<long long>(c.H) * c.D;
    // With many key tiles Delta is precomputed by a small kernel (every key tile's CTA would otherwise recompute it from O).
    const bool many = attn_many_tiles(c, sel_idx);
    if (many) {
        PrepParams R{};
        R.o = static_cast<const uint4*>(o); R.d_o = static_cast<const uint4*>(d_o);
        R.delta = reinterpret_cast<float*>(base + w.delta);
        R.dq_acc = attn_fwd_clears(c, sel_idx) ? nullptr : reinterpret_cast<float4*>(base + w.dq_acc);
        R.q = static_cast<const __nv_bfloat16*>(q); R.k = static_cast<const __nv_bfloat16*>(k); R.v = static_cast<const __nv_bfloat16*>(v);
        for (int i = 0; i < 4; ++i) R.staged[i] = reinterpret_cast<uint4*>(base + w.staged[i]);
        R.sel_idx = sel_idx;
        R.sB = L.sB; R.sN = L.sN; R.sH = L.sH;
        R.n_sel = sel_idx ? n_sel : nullptr;
        R.N = c.N; R.Ncap = w.Ncap; R.H = c.H; R.D = c.D; R.S = attn_sel_rows(c);
        const long long work = static_cast<long long>(w.Ncap) * c.H * 8;
        int gx = static_cast<int>((work + 255) / 256);
        const int cap = max(1, 8 * sm_count() / c.B);              // about eight CTAs per SM in total
        if (gx > cap) gx = cap;
        cudaError_t perr;
        { LaunchScope ls_(K_BWD_PREP, stream); perr = launch_chained(bwd_prep_kernel, dim3(gx, c.B), dim3(256), 0, stream, R); }
        if (int st = check_cuda(perr, "attention: backward prep launch")) return st;
    }

    CUtensorMap mq{}, mk{}, mv{}, mdo{}, macc;
    if (many && sel_idx) {
        CUtensorMap* const maps[4] = {&mq, &mk, &mv, &mdo};
        for (int i = 0; i < 4; ++i)
            if (int st = make_tile_map(maps[i], base + w.staged[i], c.D, c.B, w.Ncap, c.H, w.Ncap * HD, HD, c.D)) return st;
    } else if (!sel_idx) {
        if (int st = make_tile_map(&mq, q, c.D, c.B, c.N, c.H, L.sB, L.sN, L.sH)) return st;
        if (int st = make_tile_map(&mk, k, c.D, c.B, c.N, c.H, L.sB, L.sN, L.sH)) return st;
        if (int st = make_tile_map(&mv, v, c.D, c.B, c.N, c.H, L.sB, L.sN, L.sH)) return st;
        if (int st = make_tile_map(&mdo, d_o, c.D, c.B, c.N, c.H, c.N * HD, HD, c.D)) return st;
    }
    if (int st = make_acc_map(&macc, base + w.dq_acc, c.B, w.Ncap, c.H)) return st;
    BwdParams P{};
    P.q = static_cast<const __nv_bfloat16*>(q); P.k = static_cast<const __nv_bfloat16*>(k); P.v = static_cast<const __nv_bfloat16*>(v);
    P.d_o = static_cast<const __nv_bfloat16*>(d_o); P.o = static_cast<const __nv_bfloat16*>(o);
    P.lse = lse; P.delta = many ? reinterpret_cast<const float*>(base + w.delta) : nullptr;
    P.dq_acc = reinterpret_cast<float*>(base + w.dq_acc);
    P.dq = static_cast<__nv_bfloat16*>(dq); P.dk = static_cast<__nv_bfloat16*>(dk); P.dv = static_cast<__nv_bfloat16*>(dv);
    P.sel_idx = sel_idx; P.n_sel = sel_idx ? n_sel : nullptr;
    P.inv_idx = sel_idx ? inv_idx : nullptr;
    P.tile_done = reinterpret_cast<int32_t*>(base + w.tile_done);
    P.status = reinterpret_cast<int*>(base);
    P.sB = L.sB; P.sN = L.sN; P.sH = L.sH;
    P.B = c.B; P.N = c.N; P.Ncap = w.Ncap; P.H = c.H; P.D = c.D; P.S = attn_sel_rows(c);
    P.scale = scale; P.scale_log2 = scale * 1.4426950408889634f;
    const long long worst = static_cast<long long>(w.Ncap / kTile) * c.H * c.B;
    const int grid = static_cast<int>(worst < sm_count() ? worst : sm_count());          // one CTA per SM (all of tensor memory)
    auto launch = [&](auto kernel, int threads, int& attr_dev) {
        int dev = 0;
        cudaGetDevice(&dev);
        if (attr_dev != dev) {
            if (int st = check_cuda(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kBwdSmemBytes), "attention: smem attribute")) return st;
            attr_dev = dev;
        }
        LaunchScope ls_(K_ATTN_BWD, stream);
        return check_cuda(launch_chained(kernel, dim3(grid), dim3(threads), kBwdSmemBytes, stream, mq, mk, mv, mdo, macc, P), "attention: backward launch");
    };
    static thread_local int attr_few = -1, attr_many = -1;
    if (int st = many ? launch(attn_bwd_kernel<true>, BwdShape<true>::kThreads, attr_many) : launch(attn_bwd_kernel<false>, BwdShape<false>::kThreads, attr_few)) return st;
    if (many) {
        ConvertParams F{};
        F.dq_acc = reinterpret_cast<const float4*>(base + w.dq_acc);
        F.dq = static_cast<uint4*>(dq);
        F.inv_idx = sel_idx ? inv_idx : nullptr;
        F.n_sel = sel_idx ? n_sel : nullptr;
        F.N = c.N; F.Ncap = w.Ncap; F.H = c.H; F.D = c.D; F.S = attn_sel_rows(c); F.scale = scale;
        const long long work = static_cast<long long>(c.N) * c.H * (c.D / 8);
        int gx = static_cast<int>((work + 255) / 256);
        const int cap = max(1, 8 * sm_count() / c.B);
        if (gx > cap) gx = cap;
        cudaError_t cerr;
        { LaunchScope ls_(K_BWD_CONVERT, stream); cerr = launch_chained(bwd_convert_kernel, dim3(gx, c.B), dim3(256), 0, stream, F); }
        if (int st = check_cuda(cerr, "attention: backward convert launch")) return st;
    }
    return VARDROP_OK;
}

}  // namespace vardrop
