// Attention backward over few key tiles of kept variate tokens (attn_bwd_many.cu: many) and the scatter of the gradients to the full layout.
//
// attn_bwd_kernel     one CTA per SM.  Scores are formed transposed (S^T = K Q^T, dP^T = V dO^T) so that a thread owns (part of) a key row
//                     of tensor memory; P^T and dS^T feed dV += P^T dO, dK += dS^T Q and dQ_i = dS K.  Two shapes of the work:
//                       single   a kept set of one tile: two teams of 256 threads, each a whole (head, instance) on its own, no hand-offs
//                       pipeline several tiles: work items (two neighbouring 128-key tiles, head, instance), a warp role for each part of
//                                the work; dQ is written by the item (two tiles or fewer) or added into an fp32 accumulator by bulk
//                                reduce-adds and converted by the CTA that finishes an (instance, head) pair
//                     The same kernel writes the zero rows of every dropped variate.
//
// Each row of dq / dk / dv is written exactly once.
#include "attn_bwd.cuh"

namespace vardrop {

namespace {

struct BwdParams {
    const __nv_bfloat16 *q, *k, *v;   // read by the row copies of a selection (boxes go through the tensor maps)
    const __nv_bfloat16* d_o;         // [B, N, H, D]
    const __nv_bfloat16* o;           // [B, N, H, D] forward output (rows 0 .. n_sel-1), for Delta
    const float* lse;       // [B, H, N]
    float* dq_acc;          // [B, Ncap, H, 64]
    __nv_bfloat16* dq;      // [B, N, H, D]
    __nv_bfloat16* dk;
    __nv_bfloat16* dv;
    const int32_t* sel_idx; // [S, N]; NULL: identity
    const int32_t* inv_idx; // [S, N]; NULL: identity (nothing dropped)
    int32_t* tile_done;     // [B, H] items whose part of dQ' has landed; zeroed by the forward pass
    const int32_t* n_sel;   // [S]; NULL: N
    int* status;
    long long sB, sN, sH;   // element strides of q, k, v
    int B, N, Ncap, H, D, S;
    float scale, scale_log2;
};

inline BwdParams bwd_params(const void* q, const void* k, const void* v, const void* o, const float* lse, const void* d_o, const int32_t* sel_idx, const int32_t* n_sel,
                            const int32_t* inv_idx, const vardrop_attn_cfg& c, void* dq, void* dk, void* dv, void* ws) {
    const AttnWs w = attn_layout(c);
    const QkvLayout L = qkv_layout(c);
    char* base = static_cast<char*>(ws);
    BwdParams P{};
    P.q = static_cast<const __nv_bfloat16*>(q); P.k = static_cast<const __nv_bfloat16*>(k); P.v = static_cast<const __nv_bfloat16*>(v);
    P.d_o = static_cast<const __nv_bfloat16*>(d_o); P.o = static_cast<const __nv_bfloat16*>(o);
    P.lse = lse;
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

__device__ __forceinline__ uint64_t fma_pair(uint64_t a, uint64_t b, uint64_t c) {      // two IEEE fp32 results per issue slot
    uint64_t d;
    asm volatile("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
// A pair of floats from shared memory, issued here.  Read by all lanes alike, 8 bytes take 0.6 cycles of the shared-memory pipe, 16 bytes 2.1.
__device__ __forceinline__ uint64_t lds_pair(uint32_t addr) {
    uint64_t v;
    asm volatile("ld.shared.b64 %0, [%1];" : "=l"(v) : "r"(addr));
    return v;
}

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
// ---------------------------------------------------------------------------------------------------------
// main
// ---------------------------------------------------------------------------------------------------------
constexpr int kBwdGroup = 256;
constexpr int kBwdThreads = 256 + 2 * kBwdGroup;
// Register split (setmaxnreg works on whole warpgroups): launched with 768 x 80 = 61440 registers; the first two warpgroups keep 56 a thread, the
// teams take 88: 256 x 56 + 512 x 88 = 59392.
constexpr int kBwdSmallRegs = 56;
constexpr int kBwdBigRegs = 88;
constexpr uint32_t kBwdTmemCols = 512;
constexpr int kBwdHeader = 3072;       // barriers, item list, row statistics
constexpr int kBwdSmemBytes = kBwdHeader + 4 * kTileBytes /*K, V of two key tiles*/ + 4 * kTileBytes /*two slots of Q, dO*/ +
                              4 * kTileBytes /*dS^T of two key tiles*/ + 2 * kTileBytes /*dQ tile, fp32, two 32-column halves*/;

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

// With a selection per instance, the i-th instance that keeps several tiles (`several`) or one; the whole warp looks.
__device__ __forceinline__ int nth_instance(const BwdParams& P, int i, bool several) {
#pragma unroll 1
    for (int base = 0; base < P.S; base += 32) {
        const int s = base + (threadIdx.x & 31), n = s < P.S ? __ldg(P.n_sel + s) : 0;
        const unsigned mask = __ballot_sync(0xffffffffu, several ? n > kTile : n > 0 && n <= kTile);
        if (i < __popc(mask)) return base + __fns(mask, 0, i + 1);
        i -= __popc(mask);
    }
    return 0;
}

// ---------------------------------------------------------------------------------------------------------
// single: a kept set of one tile
// ---------------------------------------------------------------------------------------------------------
// A team of 256 threads (two per key row, 64 queries each) does a (head, instance) by itself; the two teams of a CTA, and nothing else,
// fill each other's waits: with one tile the work is a chain of latencies (rows in, scores, exponentials, gradients, rows out) whose
// every path runs once or twice, so hand-offs between roles and unrolled code only lengthen it.
// Team memory: Q, K, V, dO, dS^T (two 64-query panels); tensor memory (256 columns): S^T [0,128), dP^T [128,256); P^T (bf16) goes over the
// first half of each 64-column half of S^T, dV and dK over dP^T, dQ over P^T once dV has read it.
template <bool kMixed>
__device__ __forceinline__ void bwd_single(const BwdParams& P, int kept, unsigned char* tiles, float* stats, uint64_t* bar, uint32_t tm0, int team, int gt, int first, int stride, int count, bool& ok) {
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
    const uint64_t scale2 = pair_of(P.scale_log2, P.scale_log2);
    if (half == 0) s_none[row] = -INFINITY;
    uint32_t t = 0;
#pragma unroll 1
    for (int item = first; item < count && ok; item += stride, ++t) {
        const int bi = small_div(item, P.H), h = item - bi * P.H, b = kMixed ? nth_instance(P, bi, false) : bi;
        const int n = kMixed ? P.n_sel[b] : kept;
        const int32_t* idx = P.sel_idx ? P.sel_idx + static_cast<size_t>(kMixed ? b : 0) * P.N : nullptr;
        if (n <= 0) { --t; continue; }                   // (nothing kept at all)
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
        // P^T and dS^T, 32 queries at a time (a thread's half of the tile is one panel)
        const float* lse = row < n ? s_lse : s_none;
#pragma unroll 1
        for (int c = 0; c < 2; ++c) {
            const int q0 = half * 64 + c * 32;
            if (q0 >= n) break;
            float s[32], d[32];
            uint32_t pk[16];
            uint64_t l[16], dl[2][4];
            tmem_ld32(tm + q0, s);
#pragma unroll
            for (int e = 0; e < 16; ++e) l[e] = lds_pair(smem_u32(lse + q0) + 8 * e);
            tmem_ld_wait();
            exp_step(s, pk, l, scale2);
            tmem_ld32(tm + 128 + q0, d);
            tmem_st16(tm + half * 64 + c * 16, pk);
#pragma unroll
            for (int e = 0; e < 4; ++e) dl[0][e] = lds_pair(smem_u32(s_delta + q0) + 8 * e);
            tmem_ld_wait();
            ds_step(s, d, pk, dl, smem_u32(s_delta + q0));
            store_panel(sdS + half * kTileBytes, row, c, pk);
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
// Pipeline: a work item is two neighbouring 128-key tiles of a (head, instance), one to a team of 256 threads, over all its query tiles in
// steps of 64 queries.  The two key tiles share the operands of a query tile, and dQ of a query tile leaves tensor memory once for both.
//   warps 0, 1    issue the products of team 0, 1 (all lanes run the issue code, an elected lane executes a group of products)
//   warps 2, 3    load a two-slot ring of (Q, dO) tiles with their row statistics, and K, V where boxes bring them; warp 3 decodes the items
//   warps 4-7     dQ of a query tile: issue it once both teams have handed over their dS^T, take it out of tensor memory, add it to the
//                 accumulator (or write it, with two key tiles or fewer); Delta and the zero rows (few tiles)
//   warps 8-15    team 0, warps 16-23  team 1: two threads a key row, 32 queries each.  A step: S^T to registers, P^T = exp2(S^T scale - lse)
//                 to tensor memory (the A operand of dV += P^T dO), dP^T to registers, dS^T = P^T o (dP^T - Delta) to shared memory (dK +=
//                 dS^T Q, and dQ = dS K through the transposed view); dV and dK of a finished key tile
// S^T and dP^T of a team share 64 columns: each is produced under the arithmetic on the other, and no product waits for P^T or dS^T to be
// read but by a whole step.  A warp arrives with one lane (256 arrivals on one barrier serialise).
// Tensor memory of team w, from 224 w: S^T / dP^T 64 | P^T 32 | dV 64 | dK 64; dQ from 448.
constexpr uint32_t kTeamCols = 224, kColP = 64, kColDv = 96, kColDk = 160, kColDq = 448;
constexpr int kTeamWarps = 8;

// kMixed: few tiles, a selection per instance, so that some instances may keep one tile and others several (its code costs the other calls 0.4 us
// of instruction fetch).
template <bool kMixed>
__global__ void __launch_bounds__(kBwdThreads, 1) attn_bwd_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                                                                  const __grid_constant__ CUtensorMap map_v, const __grid_constant__ CUtensorMap map_do,
                                                                  const __grid_constant__ CUtensorMap map_acc, const BwdParams P) {
    extern __shared__ unsigned char smem_dyn[];
    // Set-up first (shared-memory carve-up, barriers, tensor memory): it touches nothing another kernel produces, so it runs
    // while the previous kernel of the stream is still finishing.
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem_dyn);
    uint64_t* bar_kv_full = bars;                   // [2] K, V of team w
    uint64_t* bar_kv_free = bars + 2;               // every product of the item is done (both issue warps and the dQ warps)
    uint64_t* bar_q_full = bars + 3;                // [2] slot holds a query tile
    uint64_t* bar_q_free = bars + 5;                // [2] every product reading the slot is done (both issue warps)
    uint64_t* bar_x = bars + 7;                     // [2] S^T, then dP^T of a step complete
    uint64_t* bar_xfree = bars + 9;                 // [2] S^T is in registers, then dP^T (and P^T in tensor memory)
    uint64_t* bar_flag = bars + 11;                 // few: both teams have read whether the item was the last of its dQ' (16 warps)
    uint64_t* bar_ds = bars + 13;                   // [2] dS^T in shared memory
    uint64_t* bar_dk = bars + 15;                   // [2] dV and dK of a step done
    uint64_t* bar_tile = bars + 17;                 // [2] dS^T of the whole query tile in shared memory
    uint64_t* bar_accfree = bars + 19;              // [2] dV, dK of a key tile in registers
    uint64_t* bar_delta = bars + 21;                // [2] few: Delta of the slot's rows
    uint64_t* bar_g = bars + 23;                    // dQ of a query tile complete
    uint64_t* bar_first = bars + 24;                // the first query tile's row copies have landed (128)
    uint64_t* bar_item = bars + 25;                 // [8] entry of the item list is written
    uint64_t* bar_team = bars + 33;                 // [2][2] single: scores, gradients
    uint64_t* bar_conv = bars + 37;                 // few: whether this item was the last of its dQ' is known
    uint64_t* bar_skip = bars + 38;                 // [2] team w is in an item that it has no key tile in
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 40);
    int* s_flag = reinterpret_cast<int*>(tmem_slot + 1);
    ZeroRows zeros{s_flag + 1, 0, 0u};                              // (the word after that counts the flags written)
    struct alignas(16) Item { int jt, h, b, n_sel; };               // n_sel < 0 ends the list
    Item* s_item = reinterpret_cast<Item*>(smem_dyn + 336);         // [8]
    float* s_lse = reinterpret_cast<float*>(smem_dyn + 512);        // [2][128] minus the lse of the slot's rows, log2 domain
    float* s_delta = s_lse + 2 * kTile;                             // [2][128] their Delta
    float* s_none = s_delta + 2 * kTile;                            // [128] minus the lse for key rows that do not exist: -inf throughout
    static_assert(512 + 5 * kTile * sizeof(float) <= kBwdHeader, "header too small");
    unsigned char* sKV = align_tiles(smem_dyn + kBwdHeader);        // K, V of team 0, K, V of team 1
    unsigned char* sQ = sKV + 4 * kTileBytes;           // two slots of (Q tile, dO tile)
    unsigned char* sdS = sQ + 4 * kTileBytes;           // dS^T of team 0, 1: rows = keys, two 64-query panels; dV, dK staging at the end of an item
    unsigned char* sDQ = sdS + 4 * kTileBytes;          // dQ as fp32: two 32-column panels of 128-byte swizzled rows
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (sDQ + 2 * kTileBytes > smem_dyn + kBwdSmemBytes) {
        chain_wait();
        if (tid == 0) set_status(P.status, VARDROP_ERR_CUDA);
        return;
    }
    const bool boxes = P.sel_idx == nullptr;                   // operand tiles come as boxes, or as rows
    if (warp == 0) {
        tmem_alloc(tmem_slot, kBwdTmemCols);
        tmem_relinquish();
    }
    if (tid == 0) {
        for (int w = 0; w < 2; ++w) {
            mbar_init(bar_kv_full + w, boxes ? 1 : kBwdGroup);    // a box: one announcing arrival; row copies: every thread of the team
            mbar_init(bar_q_full + w, boxes ? 1 : 66);              // row copies: every loader lane, and one of each loader for the statistics
            mbar_init(bar_q_free + w, 2);
            mbar_init(bar_x + w, 1);
            mbar_init(bar_xfree + w, kTeamWarps);
            mbar_init(bar_ds + w, kTeamWarps);
            mbar_init(bar_dk + w, 1);
            mbar_init(bar_tile + w, kTeamWarps);
            mbar_init(bar_accfree + w, kTeamWarps);
            mbar_init(bar_delta + w, 4);
            mbar_init(bar_skip + w, 1);
        }
        mbar_init(bar_kv_free, 3);
        mbar_init(bar_flag, 2 * kTeamWarps);
        mbar_init(bar_g, 1);
        mbar_init(bar_conv, 1);
        mbar_init(bar_first, 128);
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
    if (tid < kTile) s_none[tid] = -INFINITY;
    if (tid == 0) s_flag[1] = s_flag[2] = 0;
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    bool ok = true;
    int kept = 0, n_t = 0, per_item = 1, n_slots = 0, n_items = 0;
    bool pipeline = true, singles = false;                     // this CTA has items of the pipeline; and, few, single-tile (head, instance) pairs
    int s_first = 0, s_stride = 1, s_count = 0;                // a team's first of those, the next one, and how many there are
    auto begin = [&]() {
        chain_wait();
        chain_release();
        kept = largest_kept(P.n_sel, P.S, P.N);
        n_t = (kept + kTile - 1) / kTile;                      // tiles of the longest selection
        // Instances with several tiles go through the pipeline, those with one by teams.
        int several = n_t > 1 ? P.B : 0, one = P.B - several;
        const int grid = static_cast<int>(gridDim.x), cta = static_cast<int>(blockIdx.x);
        int c = cta, takers = grid;                            // CTAs that take singles
        if (kMixed) {
            several = one = 0;
#pragma unroll 1
            for (int i = 0; i < P.S; i += 32) {
                const int n = i + lane < P.S ? __ldg(P.n_sel + i + lane) : 0;
                several += __popc(__ballot_sync(0xffffffffu, n > kTile));
                one += __popc(__ballot_sync(0xffffffffu, n > 0 && n <= kTile));
            }
        }
        // Key tiles of an item: two, except that where every key tile can have a CTA of its own it gets one (1000 of 2000 kept, B = 1, H = 8:
        // 64 tiles).  Two tiles are always one item, whose dQ is complete in place: the forward pass does not clear the accumulator then.
        per_item = n_t == 2 || n_t * P.H * several > grid ? 2 : 1;
        n_slots = (n_t + per_item - 1) / per_item;
        n_items = n_slots * P.H * several;                     // pipeline: (key tiles, head, instance); short instances skip some
        pipeline = kMixed ? cta < n_items : n_t > 1;
        s_count = one * P.H;
        if (kMixed && several && one) {
            // Both kinds: the CTAs without items take the singles if their teams can (32 instances of about 120 kept, a few of them above 128: forward
            // and backward 35 us with every instance in the pipeline, 29 so).
            const bool apart = n_items < grid && 2 * (grid - n_items) >= s_count;
            takers = apart ? grid - n_items : grid;
            c = apart ? cta - n_items : (cta + grid - n_items % grid) % grid;
        }
        singles = kMixed ? c >= 0 && c < s_count : n_t <= 1;
        s_first = c + (warp >= 16 ? takers : 0);
        s_stride = 2 * takers;
    };
    // A role of several warps shares a named barrier, which nothing bounds: a warp whose wait gives up leaves only behind such a barrier, where the
    // others learn of it.  The teams wait for their next item ahead of the last barrier of the current one; the dQ warps all pass a barrier at the end
    // of the list, so that one that only took it for the end meets the others.  (8192 variates, 1423 kept: with a barrier of their own at every item
    // 257 us instead of 252.)
    auto item_wait = [&](uint32_t i) { ok &= warp_wait_relaxed(bar_item + (i & 7), (i >> 3) & 1); };
    auto item_read = [&](uint32_t i) {
        const int4 x = *reinterpret_cast<const int4*>(s_item + (i & 7));
        return Item{x.x, x.y, x.z, x.w};
    };
    auto item_at = [&](uint32_t i) {                           // -1 for an item that did not come
        item_wait(i);
        Item it = item_read(i);
        if (!ok) it.n_sel = -1;
        return it;
    };
    auto warp_arrive = [&](uint64_t* bar) {                    // all lanes are done
        __syncwarp();
        if (lane == 0) mbar_arrive(bar);
    };
    auto phase_sync = [&]() {                                  // between the pipeline's use of shared and tensor memory and the teams'
        tc_fence_before();
        ok = __syncthreads_and(ok);
        tc_fence_after();
    };
    // first token of team w's key tile (n_sel: it has none)
    auto key0_of = [&](const Item& it, int w) { return w < per_item ? (it.jt + w) * kTile : it.n_sel; };
    // steps of query tile x: the second one only if it holds a query
    auto steps_of = [&](const Item& it, int x) { return it.n_sel - x * kTile > 64 ? 2 : 1; };

    if (warp < 8) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kBwdSmallRegs));
    begin();
    // One backward pass per forward pass: the forward kernel left a mark (and cleared this workspace's counters); a backward pass that
    // does not find it (a second backward for the same forward, or two forwards sharing the workspace before their backwards) would
    // add into stale state, so it reports the call instead of returning wrong gradients.
    if (blockIdx.x == 0 && tid == 0 && atomicExch(P.status + kWsPairingWord, 0) != 1) set_status(P.status, VARDROP_ERR_INVALID_ARG);
    if (!pipeline) {
        // nothing to issue, load or drain: the teams work by themselves
    } else if (warp < 2) {
        // ------------------------------------------------------------ issue ---------------------------------------------
        const int w = warp;
        const uint32_t idesc_kk = umma_idesc_bf16(128, 64, 0, 0);          // K-major x K-major, 64 queries
        const uint32_t idesc_kmn = umma_idesc_bf16(128, P.D, 0, 1);        // A K-major, B MN-major
        const uint64_t d_k = umma_desc_sw128(smem_u32(sKV), 16, 1024), m_k = umma_desc_sw128(smem_u32(sKV), kTileBytes, 1024);
        constexpr uint32_t kQOff = 4 * kTileBytes, kDsOff = 8 * kTileBytes;
        const uint32_t tm = tmem + w * kTeamCols;
        uint32_t t = 0, u = 0, ai = 0;                   // query tiles, steps of this team, items of this team so far
#pragma unroll 1
        for (uint32_t i = 0; ok; ++i) {
            const Item it = item_at(i);
            if (it.n_sel < 0) break;
            const int n_q = (it.n_sel + kTile - 1) / kTile;
            if (i > 0) ok &= warp_wait_relaxed(bar_kv_free, (i - 1) & 1);
            if (key0_of(it, w) >= it.n_sel) {            // no key tile for this team: pass the slots on
#pragma unroll 1
                for (int x = 0; x < n_q && ok; ++x, ++t) {
                    ok &= warp_wait_relaxed(bar_q_full + (t & 1), (t >> 1) & 1);
                    warp_arrive(bar_q_free + (t & 1));
                }
                ok &= warp_wait_relaxed(bar_skip + w, (i - ai) & 1);
                warp_arrive(bar_kv_free);
                continue;
            }
            ok &= warp_wait_relaxed(bar_kv_full + w, ai & 1);
            auto wait_slot = [&](uint32_t tt) {
                ok &= warp_wait_relaxed(bar_q_full + (tt & 1), (tt >> 1) & 1);
                if (!boxes) fence_proxy_async_smem();    // rows written by asynchronous copies are read by the tensor core
                tc_fence_after();
            };
            auto scores = [&](uint32_t tt, int hs, uint32_t which) {     // S^T = K Q^T (which 0) or dP^T = V dO^T (1) of 64 queries
                if (elect_one()) {
                    const uint64_t a = umma_desc_advance(d_k, (2 * w + which) * kTileBytes);
                    const uint64_t bd = umma_desc_advance(d_k, kQOff + (2 * (tt & 1) + which) * kTileBytes + hs * 64 * kRowBytes);
                    tc_mma_bf16(tm, a, bd, idesc_kk, 0u);
                    tc_mma_bf16(tm, umma_desc_advance(a, 32), umma_desc_advance(bd, 32), idesc_kk, 1u);
                    if (P.D > 32) {
                        tc_mma_bf16(tm, umma_desc_advance(a, 64), umma_desc_advance(bd, 64), idesc_kk, 1u);
                        tc_mma_bf16(tm, umma_desc_advance(a, 96), umma_desc_advance(bd, 96), idesc_kk, 1u);
                    }
                    tc_commit(bar_x + w);
                }
                __syncwarp();
            };
            wait_slot(t);
            scores(t, 0, 0);
#pragma unroll 1
            for (int x = 0; x < n_q && ok; ++x, ++t) {
                const int nh = steps_of(it, x);
                const uint32_t q_off = kQOff + 2 * (t & 1) * kTileBytes;
#pragma unroll 1
                for (int hs = 0; hs < nh && ok; ++hs, ++u) {
                    const uint32_t acc = x + hs > 0 ? 1u : 0u;
                    ok &= warp_wait(bar_xfree + w, 0);
                    tc_fence_after();
                    scores(t, hs, 1);
                    if (hs + 1 == nh && x + 1 < n_q) wait_slot(t + 1);
                    ok &= warp_wait(bar_xfree + w, 1);
                    if (acc == 0 && ai > 0) ok &= warp_wait(bar_accfree + w, (ai - 1) & 1);      // dV, dK of the previous item are out
                    tc_fence_after();
                    if (elect_one()) {                   // dV += P^T dO
                        const uint64_t bd = umma_desc_advance(m_k, q_off + kTileBytes + hs * 64 * kRowBytes);
#pragma unroll
                        for (int ks = 0; ks < 4; ++ks) tc_mma_bf16_ta(tm + kColDv, tm + kColP + ks * 8, umma_desc_advance(bd, ks * 2048), idesc_kmn, ks > 0 ? 1u : acc);
                    }
                    __syncwarp();
                    if (hs + 1 < nh) scores(t, 1, 0);
                    else if (x + 1 < n_q) scores(t + 1, 0, 0);
                    ok &= warp_wait(bar_ds + w, u & 1);
                    tc_fence_after();
                    if (elect_one()) {                   // dK += dS^T Q
                        const uint64_t ad = umma_desc_advance(d_k, kDsOff + (2 * w + hs) * kTileBytes), bd = umma_desc_advance(m_k, q_off + hs * 64 * kRowBytes);
#pragma unroll
                        for (int ks = 0; ks < 4; ++ks) tc_mma_bf16(tm + kColDk, umma_desc_advance(ad, ks * 32), umma_desc_advance(bd, ks * 2048), idesc_kmn, ks > 0 ? 1u : acc);
                        tc_commit(bar_dk + w);
                        if (hs + 1 == nh) tc_commit(bar_q_free + (t & 1));
                    }
                    __syncwarp();
                }
            }
            ++ai;
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
                const int hb = small_div(k, n_slots), bi = small_div(hb, P.H);
                it.jt = (k - hb * n_slots) * per_item;
                it.h = hb - bi * P.H;
                it.b = kMixed ? nth_instance(P, bi, true) : bi;
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
        if (part == 0) publish(0);
#pragma unroll 1
        for (uint32_t i = 0; ok && !(boxes && part == 1); ++i) {
            if (part == 0) publish(i + 1);
            const Item it = item_at(i);
            if (it.n_sel < 0) break;
            const int n_q = (it.n_sel + kTile - 1) / kTile;
            // Row statistics of a query tile travel with it: asked for ahead of the wait for the slot, four rows a lane.
            const float* lse_row = P.lse + (static_cast<size_t>(it.b) * P.H + it.h) * P.N;
            float st_lse[4];
            auto stats_load = [&](int tile) {
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int r = tile * kTile + e * 32 + lane;
                    st_lse[e] = part == 0 && r < it.n_sel ? __ldg(lse_row + r) : INFINITY;
                }
            };
            auto stats_store = [&](uint32_t slot) {      // minus the lse in the log2 domain: -inf switches a missing query off
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    if (part == 0) s_lse[slot * kTile + e * 32 + lane] = st_lse[e] * -1.4426950408889634f;
                }
                __syncwarp();
            };
            if (boxes) {
#pragma unroll 1
                for (int x = 0; x < n_q; ++x, ++t) {
                    const uint32_t slot = t & 1;
                    stats_load(x);
                    ok = warp_wait_relaxed(bar_q_free + slot, ((t >> 1) & 1) ^ 1);
                    if (!ok) break;
                    stats_store(slot);
                    if (lane == 0) {
                        mbar_expect_tx(bar_q_full + slot, 2 * kTileBytes);
                        tma_load_4d(sQ + slot * 2 * kTileBytes, &map_q, bar_q_full + slot, 0, it.h, x * kTile, it.b);
                        tma_load_4d(sQ + slot * 2 * kTileBytes + kTileBytes, &map_do, bar_q_full + slot, 0, it.h, x * kTile, it.b);
                    }
                    __syncwarp();
                    if (x == 0) {                        // the first query tile comes in under the item before; K and V replace that one's
                        ok = warp_wait_relaxed(bar_kv_free, (i & 1) ^ 1);
                        if (!ok) break;
                        if (lane == 0) {
#pragma unroll 1
                            for (int w = 0; w < 2; ++w) {
                                const int tok0 = key0_of(it, w);
                                if (tok0 >= it.n_sel) break;
                                mbar_expect_tx(bar_kv_full + w, 2 * kTileBytes);
                                tma_load_4d(sKV + 2 * w * kTileBytes, &map_k, bar_kv_full + w, 0, it.h, tok0, it.b);
                                tma_load_4d(sKV + (2 * w + 1) * kTileBytes, &map_v, bar_kv_full + w, 0, it.h, tok0, it.b);
                            }
                        }
                        __syncwarp();
                    }
                }
            } else {
                const int32_t* idx = P.sel_idx + static_cast<size_t>(P.S > 1 ? it.b : 0) * P.N;
                const __nv_bfloat16* q_base = P.q + it.b * P.sB + it.h * P.sH;
                const __nv_bfloat16* d_o = P.d_o + (static_cast<size_t>(it.b) * P.N * P.H + it.h) * P.D;
                int x = 0;
                if (i == 0) {                            // brought in by the dQ warps: pass it on
                    stats_load(0);
                    stats_store(0);
                    if (lane == 0) mbar_arrive(bar_q_full);
                    ok = warp_wait(bar_first, 0);
                    if (!ok) break;
                    mbar_arrive(bar_q_full);
                    x = 1;
                    t = 1;
                }
#pragma unroll 1
                for (; x < n_q; ++x, ++t) {
                    const uint32_t slot = t & 1;
                    RowPicks picks = tile_picks(idx, x * kTile, it.n_sel, part);
                    stats_load(x);
                    ok = warp_wait_relaxed(bar_q_free + slot, ((t >> 1) & 1) ^ 1);
                    if (!ok) break;
                    stats_store(slot);
                    if (lane == 0) mbar_arrive(bar_q_full + slot);
                    unsigned char* to = sQ + slot * 2 * kTileBytes;
                    const __nv_bfloat16* from = q_base;
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
                }
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
    } else {
        // ------------------------------------------------------------ dQ ------------------------------------------------
        const int row = tid & (kTile - 1);
        const uint32_t tm = tmem + kColDq + (static_cast<uint32_t>((warp & 3) * 32) << 16);
        const bool owner = row == 0;                     // the one thread that owns the bulk reductions
        const uint32_t idesc_mnmn = umma_idesc_bf16(128, P.D, 1, 1);       // A MN-major, B MN-major
        const uint64_t m_k = umma_desc_sw128(smem_u32(sKV), kTileBytes, 1024);
        // Columns taken out at a time: these warps also hold Delta's loads and the output rows (862 variates, 200 kept: 43.4 us with 32, 41.5 with 16).
        constexpr int kDrain = 16;
        bool zeros_left = true;
        uint32_t t = 0, t1 = 0;                          // query tiles so far, and those with a second key tile
#pragma unroll 1
        for (uint32_t i = 0;; ++i) {
            const Item it = item_at(i);
            if (it.n_sel < 0) { ok = drain_sync_and(ok); break; }
            const int n_q = (it.n_sel + kTile - 1) / kTile;
            const bool two = key0_of(it, 1) < it.n_sel;
            const bool direct = n_q <= per_item;              // dQ is complete here
            const int32_t* sel = P.sel_idx ? P.sel_idx + static_cast<size_t>(P.S > 1 ? it.b : 0) * P.N : nullptr;
            const int c8 = row & 7, r8 = row >> 3;
            const size_t compact = (static_cast<size_t>(it.b) * P.N * P.H + it.h) * P.D;
            if (!boxes && i == 0) {                      // the first query tile's rows, 32 a warp
                copy_32_rows(sQ + (warp & 3) * 32 * kRowBytes, P.q + it.b * P.sB + it.h * P.sH, P.sN, sel, (warp & 3) * 32, it.n_sel, P.D);
                copy_32_rows(sQ + kTileBytes + (warp & 3) * 32 * kRowBytes, P.d_o + compact, static_cast<long long>(P.H) * P.D, nullptr, (warp & 3) * 32, it.n_sel, P.D);
                cp_async_arrive(bar_first);
            }
            // Delta of a query tile: eight threads a row of O (from memory) and dO (from the slot)
            auto delta_of = [&](int x, uint32_t tt) {
                const __nv_bfloat16* from = P.o + compact + c8 * 8;
                const unsigned char* sdO = sQ + (2 * (tt & 1) + 1) * kTileBytes;
                float* dlt = s_delta + (tt & 1) * kTile;
                uint4 o[8];                              // asked for together, ahead of the wait for the slot
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const int r = x * kTile + r8 + 16 * e;
                    o[e] = r < it.n_sel && c8 * 8 < P.D ? __ldg(reinterpret_cast<const uint4*>(from + static_cast<size_t>(r) * P.H * P.D)) : make_uint4(0u, 0u, 0u, 0u);
                }
                ok &= warp_wait_relaxed(bar_q_full + (tt & 1), (tt >> 1) & 1);
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const int r = r8 + 16 * e;
                    const float part = sum8(dot8(o[e], *reinterpret_cast<const uint4*>(sdO + r * kRowBytes + ((c8 ^ (r & 7)) << 4))));
                    if (c8 == 0) dlt[r] = part;
                }
                warp_arrive(bar_delta + (tt & 1));
            };
            delta_of(0, t);
#pragma unroll 1
            for (int x = 0; x < n_q; ++x, ++t) {
                if (x + 1 < n_q) delta_of(x + 1, t + 1);
                while (zeros_left && warp != 4 && !__all_sync(0xffffffffu, mbar_test(bar_tile, t & 1))) {       // nothing else to do
                    zeros_left = write_zero_row(P, zeros);
                    __nanosleep(100);
                }
                ok &= warp_wait_relaxed(bar_tile, t & 1);
                if (two) ok &= warp_wait_relaxed(bar_tile + 1, t1 & 1);
                t1 += two ? 1 : 0;
                if (owner) bulk_wait_group_read0();      // the previous reduction has read the staging tile
                ok = drain_sync_and(ok);                 // and every thread has read the previous dQ
                if (!ok) break;
                if (warp == 4) {
                    fence_proxy_async_smem();
                    tc_fence_after();
                    if (elect_one()) {                   // dQ = dS K over the keys of both tiles, dS the transposed view of dS^T
#pragma unroll 1
                        for (int w = 0; w < (two ? 2 : 1); ++w) {
                            const uint64_t am = umma_desc_advance(m_k, (8 + 2 * w) * kTileBytes), bm = umma_desc_advance(m_k, 2 * w * kTileBytes);
#pragma unroll
                            for (int ks = 0; ks < 8; ++ks)
                                tc_mma_bf16(tmem + kColDq, umma_desc_advance(am, ks * 2048), umma_desc_advance(bm, ks * 2048), idesc_mnmn, w + ks > 0 ? 1u : 0u);
                        }
                        tc_commit(bar_g);
                    }
                    __syncwarp();
                }
                int nout[8];                             // where this thread's rows go: looked up under the product
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const int j = x * kTile + r8 + 16 * e;
                    nout[e] = direct && j < it.n_sel ? (sel ? __ldg(sel + j) : j) : -1;
                }
                ok &= warp_wait_relaxed(bar_g, t & 1);
                if (warp == 4 && x + 1 == n_q && lane == 0) mbar_arrive(bar_kv_free);
                tc_fence_after();
#pragma unroll 1
                for (int c = 0; c < P.D; c += kDrain) {
                    float v[kDrain];
                    tmem_ld16(tm + c, v);
                    tmem_ld_wait();
                    if (!direct) {                       // fp32, 32-column panels of 128-byte swizzled rows
                        unsigned char* to = sDQ + (c >> 5) * kTileBytes + row * kRowBytes;
#pragma unroll
                        for (int e = 0; e < kDrain / 4; ++e)
                            *reinterpret_cast<float4*>(to + (((c & 31) / 4 + e) ^ (row & 7)) * 16) = make_float4(v[4 * e], v[4 * e + 1], v[4 * e + 2], v[4 * e + 3]);
                    } else {
                        unsigned char* to = sDQ + row * kRowBytes;
#pragma unroll
                        for (int e = 0; e < kDrain / 8; ++e)
                            *reinterpret_cast<uint4*>(to + (((c >> 3) + e) ^ (row & 7)) * 16) =
                                make_uint4(pack2(v[8 * e] * P.scale, v[8 * e + 1] * P.scale), pack2(v[8 * e + 2] * P.scale, v[8 * e + 3] * P.scale),
                                           pack2(v[8 * e + 4] * P.scale, v[8 * e + 5] * P.scale), pack2(v[8 * e + 6] * P.scale, v[8 * e + 7] * P.scale));
                    }
                }
                tc_fence_before();
                fence_proxy_async_smem();
                ok = drain_sync_and(ok);                 // the staging tile is complete
                if (!direct) {
                    if (owner) {
                        tma_reduce_add_4d(&map_acc, sDQ, 0, it.h, x * kTile, it.b);
                        if (P.D > 32) tma_reduce_add_4d(&map_acc, sDQ + kTileBytes, 32, it.h, x * kTile, it.b);
                        bulk_commit_group();
                    }
                } else if (c8 * 8 < P.D) {
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        const int r = r8 + 16 * e;
                        if (nout[e] >= 0)
                            *reinterpret_cast<uint4*>(P.dq + ((static_cast<size_t>(it.b) * P.N + nout[e]) * P.H + it.h) * P.D + c8 * 8) =
                                *reinterpret_cast<const uint4*>(sDQ + r * kRowBytes + ((c8 ^ (r & 7)) << 4));
                    }
                }
            }
            if (!ok) break;
            if (!direct && owner) {                     // dQ' of this (instance, head) is complete once all its items are: the teams of the last convert it
                bulk_wait_group0();                      // this item's reductions have landed
                __threadfence();
                const int n = s_flag[2]++;               // items with an accumulated dQ' before this one
                if (n > 0 && !mbar_wait_relaxed(bar_flag, (n - 1) & 1)) set_status(P.status, VARDROP_ERR_TIMEOUT);     // the teams have read that one's flag
                *s_flag = atomicAdd(P.tile_done + it.b * P.H + it.h, 1) == (n_q - 1) / per_item;
                mbar_arrive(bar_conv);
            }
        }
        if (owner) bulk_wait_group0();                   // the last dQ reductions have landed
        asm volatile("cp.async.wait_all;" ::: "memory");
    }
    if (singles) {
        if (kMixed && pipeline) phase_sync();
        if (warp < 2)                                    // (four warps at it hold the teams' loads up: 20 us against 18.8 at 119 of 321 kept)
#pragma unroll 1
            while (write_zero_row(P, zeros)) {}
    }
    } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kBwdBigRegs));
    begin();
    const int w = (warp - 8) >> 3, gt = tid & (kBwdGroup - 1);
    if (pipeline) {
        // ------------------------------------------------------------ teams ---------------------------------------------
        const int row = gt & (kTile - 1), half = gt >> 7, id = w + 1;
        const uint32_t tm = tmem + w * kTeamCols + (static_cast<uint32_t>((warp & 3) * 32) << 16);
        const int r8 = gt >> 3;
        unsigned char* panels = sdS + 2 * w * kTileBytes;
        const uint64_t scale2 = pair_of(P.scale_log2, P.scale_log2);
        uint32_t t = 0, u = 0, n_conv = 0;               // query tiles, steps of this team, items with an accumulated dQ' so far
        auto load_kv = [&](const Item& it) {             // this team's K and V rows, 32 a warp
            const int x = (warp >> 2) & 1, g = (warp & 3) * 32;
            copy_32_rows(sKV + (2 * w + x) * kTileBytes + g * kRowBytes, (x == 0 ? P.k : P.v) + it.b * P.sB + it.h * P.sH, P.sN,
                         P.sel_idx + static_cast<size_t>(P.S > 1 ? it.b : 0) * P.N, key0_of(it, w) + g, it.n_sel, P.D);
            cp_async_arrive(bar_kv_full + w);
        };
        item_wait(0);
        ok = group_sync_and(id, ok);
#pragma unroll 1
        for (uint32_t i = 0; ok; ++i) {
            const Item it = item_read(i);
            if (it.n_sel < 0) break;
            const int n_q = (it.n_sel + kTile - 1) / kTile, key0 = key0_of(it, w);
            if (!boxes && i > 0) ok &= warp_wait_relaxed(bar_kv_free, (i - 1) & 1);
            // dQ' of an (instance, head) of more than two tiles: both teams of the CTA that brought its last part
            auto convert_dq = [&]() {
                if (n_q <= per_item) return;
                if (!warp_wait_relaxed(bar_conv, n_conv & 1)) set_status(P.status, VARDROP_ERR_TIMEOUT);
                ++n_conv;
                const int c8 = gt & 7;
                const bool last = *s_flag != 0;
                warp_arrive(bar_flag);
                if (!last || c8 * 8 >= P.D) return;
                __threadfence();
                const int32_t* sel = P.sel_idx ? P.sel_idx + static_cast<size_t>(P.S > 1 ? it.b : 0) * P.N : nullptr;
                const float4* acc = reinterpret_cast<const float4*>(P.dq_acc + (static_cast<size_t>(it.b) * P.Ncap * P.H + it.h) * kDP) + c8 * 2;
                __nv_bfloat16* out = P.dq + (static_cast<size_t>(it.b) * P.N * P.H + it.h) * P.D + c8 * 8;
#pragma unroll 1
                for (int j0 = w * 32 + (gt >> 3); j0 < it.n_sel; j0 += 128) {        // two rows a thread in flight
                    float4 a[2][2];
                    int n[2];
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int j = min(j0 + 64 * e, it.n_sel - 1);
                        n[e] = sel ? __ldg(sel + j) : j;
                        a[e][0] = __ldcg(acc + static_cast<size_t>(j) * P.H * (kDP / 4));
                        a[e][1] = __ldcg(acc + static_cast<size_t>(j) * P.H * (kDP / 4) + 1);
                    }
#pragma unroll
                    for (int e = 0; e < 2; ++e)
                        if (j0 + 64 * e < it.n_sel)
                            *reinterpret_cast<uint4*>(out + static_cast<size_t>(n[e]) * P.H * P.D) =
                                make_uint4(pack2(a[e][0].x * P.scale, a[e][0].y * P.scale), pack2(a[e][0].z * P.scale, a[e][0].w * P.scale),
                                           pack2(a[e][1].x * P.scale, a[e][1].y * P.scale), pack2(a[e][1].z * P.scale, a[e][1].w * P.scale));
                }
            };
            if (key0 >= it.n_sel) {                      // no key tile: nothing else ties this team to the others' pace, and it waits by parity
                if (boxes && i > 0) ok &= warp_wait_relaxed(bar_kv_free, (i - 1) & 1);
                item_wait(i + 1);
                ok = group_sync_and(id, ok);
                if (gt == 0) mbar_arrive(bar_skip + w);
                t += n_q;
                convert_dq();
                continue;
            }
            const int32_t* sel = P.sel_idx ? P.sel_idx + static_cast<size_t>(P.S > 1 ? it.b : 0) * P.N : nullptr;
            if (!boxes) load_kv(it);
            const bool key_valid = key0 + row < it.n_sel;
            // After an item it had no key tile in, a team may be two phases ahead of a query slot's barrier, which would let it through: its own
            // scores come after the phase it wants.
            ok &= warp_wait(bar_x + w, 0);
            bool s_ready = true;                         // a poll takes a hundred cycles to answer: polls go out ahead of where they are needed
#pragma unroll 1
            for (int x = 0; x < n_q && ok; ++x, ++t) {
                const int nh = steps_of(it, x), slot = t & 1;
#pragma unroll 1
                for (int hs = 0; hs < nh; ++hs, ++u) {
                    const int q0 = hs * 64 + half * 32;  // this thread's queries of the tile
                    const uint32_t lse = smem_u32(key_valid ? s_lse + slot * kTile + q0 : s_none), dlt = smem_u32(s_delta + slot * kTile + q0);
                    if (hs == 0) ok &= warp_wait(bar_q_full + slot, (t >> 1) & 1);       // the row statistics come with the tile
                    uint64_t l[16];                      // all asked for ahead: a load behind the tensor core's operands takes a hundred cycles
#pragma unroll
                    for (int e = 0; e < 16; ++e) l[e] = lds_pair(lse + 8 * e);
                    if (!__all_sync(0xffffffffu, s_ready)) ok &= warp_wait(bar_x + w, 0);
                    tc_fence_after();
                    float s[32], d[32];
                    tmem_ld32(tm + half * 32, s);
                    tmem_ld_wait();
                    tc_fence_before();
                    warp_arrive(bar_xfree + w);          // S^T is in registers: dP^T may be produced
                    uint32_t pk[16];
                    const bool dk_done = u == 0 || mbar_test(bar_dk + w, (u - 1) & 1);
                    exp_step(s, pk, l, scale2);
                    const bool dp_ready = mbar_test(bar_x + w, 1);
                    if (!__all_sync(0xffffffffu, dk_done)) ok &= warp_wait(bar_dk + w, (u - 1) & 1);     // dV of the previous step has read P^T, dK its dS^T
                    tc_fence_after();
                    tmem_st16(tm + kColP + half * 16, pk);
                    if (!__all_sync(0xffffffffu, dp_ready)) ok &= warp_wait(bar_x + w, 1);
                    tc_fence_after();
                    tmem_ld32(tm + half * 32, d);
                    const bool g_done = hs > 0 || x == 0 || mbar_test(bar_g, (t - 1) & 1);
                    if (hs == 0) ok &= warp_wait(bar_delta + slot, (t >> 1) & 1);
                    uint64_t dl[2][4];                   // Delta of eight queries, the next eight on their way
#pragma unroll
                    for (int e = 0; e < 4; ++e) dl[0][e] = lds_pair(dlt + 8 * e);
                    tmem_st_wait();
                    tmem_ld_wait();
                    tc_fence_before();
                    warp_arrive(bar_xfree + w);          // dP^T is in registers, P^T in tensor memory: dV and the next S^T may go
                    ds_step(s, d, pk, dl, dlt);
                    if (!__all_sync(0xffffffffu, g_done)) ok &= warp_wait(bar_g, (t - 1) & 1);   // dQ of the previous tile has read the panels
                    store_panel(panels + hs * kTileBytes, row, half, pk);
                    s_ready = mbar_test(bar_x + w, 0);
                    fence_proxy_async_smem();
                    warp_arrive(bar_ds + w);             // dK may go
                    if (hs + 1 == nh && lane == 0) mbar_arrive(bar_tile + w);    // and dQ
                    if (!ok) break;
                }
            }
            ok = group_sync_and(id, ok);
            if (!ok) break;
            // dV and dK of the key tile, staged over dS^T
            int nout[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int key = key0 + r8 + 32 * e;
                nout[e] = key < it.n_sel ? (sel ? __ldg(sel + key) : key) : -1;
            }
            ok &= warp_wait(bar_dk + w, (u - 1) & 1);
            ok &= warp_wait(bar_g, (t - 1) & 1);
            tc_fence_after();
#pragma unroll 1
            for (int e = 0; e < 2; ++e) stage_acc(panels + e * kTileBytes, tm + (e == 0 ? kColDv : kColDk), e == 0 ? 1.f : P.scale, row, half);
            tc_fence_before();
            warp_arrive(bar_accfree + w);
            ok = group_sync_and(id, ok);
            if (!ok) break;
#pragma unroll 1
            for (int e = 0; e < 2; ++e) store_rows(panels + e * kTileBytes, e == 0 ? P.dv : P.dk, nout, gt, P, it.b, it.h);
            item_wait(i + 1);
            ok = group_sync_and(id, ok);                 // the staging tiles are free
            convert_dq();
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
    }
    if (singles) {
        if (kMixed && pipeline) phase_sync();
        bwd_single<kMixed>(P, kept, sKV, reinterpret_cast<float*>(sDQ), bar_team + 2 * w, tmem + w * 256, w, gt, s_first, s_stride, s_count, ok);
    }
    }
    if (warp >= 8 || pipeline || !singles)       // (a warp that zeroed rows while it waited may have some of its group left)
#pragma unroll 1
        while (write_zero_row(P, zeros)) {}              // what is left
    if (!ok) set_status(P.status, VARDROP_ERR_TIMEOUT);
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, kBwdTmemCols);
}

}  // namespace

int attn_bwd_launch(const void* q, const void* k, const void* v, const void* o, const float* lse, const void* d_o,
                    const int32_t* sel_idx, const int32_t* n_sel, const int32_t* inv_idx, const vardrop_attn_cfg& c, void* dq,
                    void* dk, void* dv, void* ws, cudaStream_t stream) {
    if (attn_many_tiles(c, sel_idx)) return attn_bwd_many_launch(q, k, v, o, lse, d_o, sel_idx, n_sel, inv_idx, c, dq, dk, dv, ws, stream);
    const AttnWs w = attn_layout(c);
    const QkvLayout L = qkv_layout(c);
    const BwdParams P = bwd_params(q, k, v, o, lse, d_o, sel_idx, n_sel, inv_idx, c, dq, dk, dv, ws);
    CUtensorMap mq{}, mk{}, mv{}, mdo{}, macc;
    const long long HD = static_cast<long long>(c.H) * c.D;
    if (!sel_idx) {
        if (int st = make_tile_map(&mq, q, c.D, c.B, c.N, c.H, L.sB, L.sN, L.sH)) return st;
        if (int st = make_tile_map(&mk, k, c.D, c.B, c.N, c.H, L.sB, L.sN, L.sH)) return st;
        if (int st = make_tile_map(&mv, v, c.D, c.B, c.N, c.H, L.sB, L.sN, L.sH)) return st;
        if (int st = make_tile_map(&mdo, d_o, c.D, c.B, c.N, c.H, c.N * HD, HD, c.D)) return st;
    }
    if (int st = make_acc_map(&macc, static_cast<char*>(ws) + w.dq_acc, c.B, w.Ncap, c.H)) return st;
    const long long worst = static_cast<long long>(w.Ncap / kTile) * c.H * c.B;
    const int grid = static_cast<int>(worst < sm_count() ? worst : sm_count());          // one CTA per SM (all of tensor memory)
    auto launch = [&](auto kernel, int& attr_dev) {
        int dev = 0;
        cudaGetDevice(&dev);
        if (attr_dev != dev) {
            if (int st = check_cuda(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kBwdSmemBytes), "attention: smem attribute")) return st;
            attr_dev = dev;
        }
        LaunchScope ls_(K_ATTN_BWD, stream);
        return check_cuda(launch_chained(kernel, dim3(grid), dim3(kBwdThreads), kBwdSmemBytes, stream, mq, mk, mv, mdo, macc, P), "attention: backward launch");
    };
    static thread_local int attr_few = -1, attr_mixed = -1;
    return sel_idx && P.S > 1 ? launch(attn_bwd_kernel<true>, attr_mixed) : launch(attn_bwd_kernel<false>, attr_few);
}

}  // namespace vardrop
