// Attention backward over many key tiles of kept variate tokens (attn_bwd.cu: few).
//
// bwd_prep_kernel     Delta_i = sum_d dO'_id O'_id, the kept rows laid out as tiles (selection), and the cleared dQ' accumulator (no selection: with one
//                     the forward pass clears it).
// bwd_many_kernel     one persistent CTA per SM over work items of one 128-key tile of a (head, instance); dQ is added into an fp32 accumulator by bulk
//                     reduce-adds.
// bwd_convert_kernel  the zero rows of every dropped variate; dQ' accumulator to bf16 rows of dq.
//
// Each row of dq / dk / dv is written exactly once.
#include "attn_bwd.cuh"
#include "attn_zero_rows.h"

namespace vardrop {

namespace {

// ---------------------------------------------------------------------------------------------------------
// prep
// ---------------------------------------------------------------------------------------------------------
struct PrepParams {
    const uint4* o;         // [B, N, H, D] bf16
    const uint4* d_o;       // [B, N, H, D] bf16
    const __nv_bfloat16* q;
    float* delta;           // [B, H, Ncap]
    float4* dq_acc;         // [B, Ncap, H, 64] fp32; NULL: cleared by the forward pass
    uint4* staged[2];       // [B, Ncap, H, D] bf16 copies of the kept rows of Q, and of dO: with a selection
    const int32_t* sel_idx; // [S, N]; NULL: identity, nothing is staged
    const int32_t* n_sel;   // [S] kept counts; NULL: N
    long long sB, sN, sH;
    int N, Ncap, H, D, S;
};

// One thread per 16-byte chunk of a (token, head) row of 64; the 8 threads of a row reduce Delta by shuffles.  With a selection the rows
// that the main kernel reads again for every key tile (Q, dO) are laid out here once, zeros up to the tile's end (rows of dO past the kept ones
// may hold anything), so that it takes boxes.  K and V it reads once an item, as rows, under the products of the item before.  (Both measured with an earlier
// main kernel, of two key tiles an item: Q and dO by row copies 250 us at 1423 kept of 8192 against 170, K and V laid out here too a step of 8192 variates 311.8 us
// against 304.6.)
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
        uint4 vo = make_uint4(0u, 0u, 0u, 0u), vd = vo, vq = vo;
        if (i < n_sel && dc < src_chunks_head) {
            const size_t src = (static_cast<size_t>(b) * P.N + i) * (P.H * src_chunks_head) + h * src_chunks_head + dc;
            vo = __ldg(P.o + src);
            vd = __ldg(P.d_o + src);
            if (sel) vq = __ldg(reinterpret_cast<const uint4*>(P.q + (b * P.sB + __ldg(sel + i) * P.sN + h * P.sH + dc * 8)));
        }
        if (sel && dc < src_chunks_head) {
            const size_t to = ((static_cast<size_t>(b) * P.Ncap + i) * P.H + h) * src_chunks_head + dc;
            P.staged[0][to] = vq; P.staged[1][to] = vd;
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
struct ManyParams {
    const __nv_bfloat16 *k, *v;       // read by the row copies of a selection (boxes go through the tensor maps)
    const float* lse;                 // [B, H, N]
    const float* delta;               // [B, H, Ncap]
    __nv_bfloat16 *dk, *dv;           // [B, N, H, D]
    const int32_t* sel_idx;           // [S, N]; NULL: identity
    const int32_t* n_sel;             // [S]; NULL: N
    int* status;
    long long sB, sN, sH;             // element strides of k and v
    int B, N, Ncap, H, D, S;
    float scale, scale_log2, half_inv_scale;      // of dK; in the exponents, and 0.5 / scale there
};

constexpr int kManyThreads = 896;
// Register split (setmaxnreg works on whole warpgroups): launched with 896 x 72 = 64512 registers; the first warpgroup keeps 56 a
// thread, the two that take results out 64, the teams take 80: 128 x 56 + 256 x 64 + 512 x 80 = 64512.
constexpr int kManySmallRegs = 56;
constexpr int kManyOutRegs = 64;
constexpr int kManyBigRegs = 80;
constexpr uint32_t kManyTmemCols = 512;
constexpr int kManyStages = 3;         // ring of (Q, dO) tiles
constexpr int kManyTeamWarps = 8;
constexpr int kManyHeader = 13312;     // barriers, item list, row statistics
constexpr int kManySmemBytes = kManyHeader + 3 * kTileBytes /*K of two items, V*/ + 2 * kManyStages * kTileBytes /*ring*/ + 2 * kTileBytes /*dS^T, two 64-query panels*/ +
                               2 * kTileBytes /*staging: dQ as fp32, two 32-column panels; dV, dK as bf16*/;

// The first 32 bytes (16 bf16) of 128 rows of a swizzled tile to eight columns of tensor memory, row r to lane r: the A operand of a k-step.
__device__ __forceinline__ void tc_copy_128x256b(uint32_t taddr, uint64_t desc) {
    asm volatile("tcgen05.cp.cta_group::1.128x256b [%0], %1;" ::"r"(taddr), "l"(desc) : "memory");
}
// Shared-memory matrix descriptor without swizzle, K-major: rows of 16 bytes (8 bf16 of K), eight rows in a row; lbo = bytes to the other half of a k-step,
// sbo = bytes between 8-row groups.
__device__ __forceinline__ uint64_t umma_desc_plain(uint32_t smem_addr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
    return umma_desc_sw128(smem_addr, lbo_bytes, sbo_bytes) & ~(7ull << 61);
}
// x as three bf16 terms (24 bits), each in the low half of a word; one that is not finite as a single one.  (Below 1.7e38 in magnitude no term rounds to infinity.)
__device__ __forceinline__ void split3(float x, uint32_t& a, uint32_t& b, uint32_t& c) {
    const __nv_bfloat16 h = __float2bfloat16_rn(x);
    const float r = fabsf(x) < INFINITY ? x - __bfloat162float(h) : 0.f;
    const __nv_bfloat16 m = __float2bfloat16_rn(r);
    a = __bfloat16_as_ushort(h);
    b = __bfloat16_as_ushort(m);
    c = __bfloat16_as_ushort(__float2bfloat16_rn(r - __bfloat162float(m)));
}
// P^T = exp2(S^T scale) of a thread's 32 queries, in place, and as bf16, in batches of eight like exp_step.
__device__ __forceinline__ void exp_step_folded(float (&s)[32], uint32_t (&pk)[16], uint64_t scale2) {
#pragma unroll
    for (int g = 0; g < 6; ++g) {
        if (g < 4) {
#pragma unroll
            for (int e = 8 * g; e < 8 * g + 8; e += 2) halves_of(mul_pair(pair_of(s[e], s[e + 1]), scale2), s[e], s[e + 1]);
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
__device__ __forceinline__ bool group_sync_and(int id, bool ok) {     // barrier among a warpgroup, with an and-reduction of ok
    uint32_t r;
    asm volatile(
        "{\n.reg .pred p, q;\n"
        "setp.ne.b32 q, %1, 0;\n"
        "bar.red.and.pred p, %2, 128, q;\n"
        "selp.u32 %0, 1, 0, p;\n}"
        : "=r"(r)
        : "r"(static_cast<uint32_t>(ok)), "r"(id)
        : "memory");
    return r != 0;
}

// A work item is one 128-key tile of a (head, instance) over all its query tiles.  Two teams of 256 threads share the key tile; team w takes the queries
// 64 w to 64 w + 63 of every query tile.
//   warp 0       issues S^T = K Q^T and dV += P^T dO of both teams (all lanes run the issue code, an elected lane executes a group of products)
//   warp 1       issues dP^T = V dO^T and dK += dS^T Q of both teams
//   warp 2       issues dQ = dS K of a query tile once both teams have handed over their dS^T; copies K and V of the next item to tensor memory
//   warp 3       loads K, V of the items (boxes) and a ring of (Q, dO) tiles with their row statistics; decodes the items
//   warps 4-7    columns 0 to 31 of dQ from tensor memory into the accumulator; dV of a finished item; K rows of a selection
//   warps 8-11   columns 32 to 63; dK of a finished item; V rows of a selection
//   warps 12-19  team 0, warps 20-27  team 1: two threads a key row, 32 queries each.  A step: S^T to registers, P^T = exp2(S^T scale - lse) over it,
//                dP^T to registers, dS^T = P^T o (dP^T - Delta) over it and to shared memory (for dQ, through the transposed view)
// What bounds a step of 128 x 128 scores (2700 cycles): the shared-memory pipe, 128 bytes a cycle, of which 1109 go to the tensor core's operands, 875 to the threads' own
// accesses and 533 to the copy engine (2500 of 2800 under ncu, all of 1423 variates, B = 8); with every variate kept, B = 8, N = 8192, the power limit.
//   - A operands come from tensor memory wherever they can (K and V copied there once an item, P^T, dS^T): a product of N = 64 then takes 32 cycles instead of 48
//     and reads 2 KB instead of 6; 1600 cycles a step instead of 1920.
//   - -lse / scale and -Delta of a query are three bf16 terms each (24 bits) of a fifth k-step of S^T and dP^T, against rows of ones: no thread reads them
//     (64 broadcast loads a row and step), and without their registers nothing spills.  Each product has rows of its own and meets them with ones and with the
//     zeros behind the terms only: a row of both, picked from by ones and zeros, takes a Delta that is not finite into S^T (0 times infinity), and so into every
//     column of dV.  (6 KB more of shared memory; by events, 32 x 862 325.1 us -> 325.2, scale step 287.4 -> 287.8.)
//   - S^T of the next query tile is issued over P^T right behind the dV that reads it, dP^T over dS^T behind dK, so a team hands over three times a step and waits for
//     neither.  This takes for given that the products of one thread run in the order of their issue also where accumulators and shapes differ; the instruction set
//     documents the order for the same accumulator and shape.  Held by gradients that are the same bit for bit from run to run, at both head sizes and with several
//     items a CTA (test_attention_backward_is_reproducible).
//   - At the end of an item the next K and V are copied in behind the last products that read the old ones; the teams never leave the steps.
// Two 128-key tiles a CTA, a team each, with K and V from shared memory (before this), took 3500 cycles for as many scores: forward and backward by graphs, H = 8, all of
// 8192 variates, B = 8 4720 -> 4450 us, 1423 of 8192 kept 247.0 -> 227.5, 700 of 8192 158.5 -> 109.4; all of 862, B = 32 338.5 -> 294.
// Tensor memory: K 32 | V 32 | dV 64 | dK 64 | dQ 64 | team 0: S^T, P^T 64, dP^T, dS^T 64 | team 1.
constexpr uint32_t kColK = 0, kColV = 32, kColDv = 64, kColDk = 128, kColDq = 192, kColTeam = 256;

// kRows: with a selection, K and V come as rows.
template <bool kRows>
__global__ void __launch_bounds__(kManyThreads, 1) bwd_many_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                                                                   const __grid_constant__ CUtensorMap map_v, const __grid_constant__ CUtensorMap map_do,
                                                                   const __grid_constant__ CUtensorMap map_acc, const ManyParams P) {
    extern __shared__ __align__(1024) unsigned char smem_dyn[];      // (every address below is a constant then: no registers)
    // Set-up first: it touches nothing another kernel produces, so it runs while the previous kernel of the stream is still finishing.
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem_dyn);
    uint64_t* bar_k_full = bars;                    // [2] K of an item in shared memory
    uint64_t* bar_k_free = bars + 2;                // [2] its last dQ is done
    uint64_t* bar_v_full = bars + 4;                // V of an item in shared memory
    uint64_t* bar_v_free = bars + 5;                // and in tensor memory
    uint64_t* bar_q_full = bars + 6;                // [kManyStages] slot holds a query tile
    uint64_t* bar_q_free = bars + 9;                // [kManyStages] every product reading the slot is done (both issuing warps)
    uint64_t* bar_s = bars + 12;                    // [2] S^T of team w's step complete
    uint64_t* bar_dp = bars + 14;                   // [2] dP^T
    uint64_t* bar_p = bars + 16;                    // [2] P^T in tensor memory
    uint64_t* bar_ds = bars + 18;                   // [2] dS^T in tensor memory
    uint64_t* bar_g = bars + 20;                    // dQ of a query tile complete
    uint64_t* bar_dv_done = bars + 21;              // dV of an item complete
    uint64_t* bar_dv_free = bars + 22;              // and in registers
    uint64_t* bar_dk_done = bars + 23;
    uint64_t* bar_dk_free = bars + 24;
    uint64_t* bar_gfree = bars + 25;                // dQ of a query tile in registers
    uint64_t* bar_panel = bars + 26;                // [2] dS^T in shared memory
    uint64_t* bar_kv = bars + 28;                   // [2] K, V of an item in tensor memory
    uint64_t* bar_item = bars + 30;                 // [8] entry of the item list is written
    uint64_t* bar_left = bars + 39;                 // [3] what an issuing warp whose wait gave up has issued is done
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 38);
    struct alignas(16) Item { int jt, h, b, n_sel; };               // n_sel < 0 ends the list
    Item* s_item = reinterpret_cast<Item*>(smem_dyn + 384);         // [8]
    uint4* s_ones = reinterpret_cast<uint4*>(smem_dyn + 512);       // [8] bf16 rows of three ones
    uint4* s_stats = s_ones + 8;                                    // [2][kManyStages][128] three bf16 terms of half of -lse / scale, of half of -Delta, of the slot's rows
    static_assert(42 * 8 <= 512 - 8 * sizeof(Item) && 512 + (8 + 2 * kManyStages * kTile) * sizeof(uint4) <= kManyHeader, "header too small");
    unsigned char* sK = smem_dyn + kManyHeader;                     // K of two items
    unsigned char* sV = sK + 2 * kTileBytes;
    unsigned char* sQ = sV + kTileBytes;                            // slots of (Q tile, dO tile)
    unsigned char* sdS = sQ + 2 * kManyStages * kTileBytes;         // dS^T: rows = keys, a 64-query panel of each team
    unsigned char* sOut = sdS + 2 * kTileBytes;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (smem_u32(smem_dyn) & 1023u) {
        chain_wait();
        if (tid == 0) set_status(P.status, VARDROP_ERR_CUDA);
        return;
    }
    if (warp == 0) {
        tmem_alloc(tmem_slot, kManyTmemCols);
        tmem_relinquish();
    }
    if (tid == 0) {
        for (int w = 0; w < 2; ++w) {
            mbar_init(bar_k_full + w, kRows ? 128 : 1);      // a box: one announcing arrival; row copies: every thread of a warpgroup
            mbar_init(bar_k_free + w, 1);
            mbar_init(bar_s + w, 1);
            mbar_init(bar_dp + w, 1);
            mbar_init(bar_p + w, kManyTeamWarps);
            mbar_init(bar_ds + w, kManyTeamWarps);
            mbar_init(bar_panel + w, kManyTeamWarps);
            mbar_init(bar_kv + w, 1);
        }
        mbar_init(bar_v_full, kRows ? 128 : 1);
        mbar_init(bar_v_free, 1);
        for (int s = 0; s < kManyStages; ++s) {
            mbar_init(bar_q_full + s, 2);                     // the boxes' announcing arrival, the statistics
            mbar_init(bar_q_free + s, 2);
        }
        mbar_init(bar_g, 1);
        mbar_init(bar_dv_done, 1);
        mbar_init(bar_dv_free, 4);
        mbar_init(bar_dk_done, 1);
        mbar_init(bar_dk_free, 4);
        mbar_init(bar_gfree, 8);
        for (int i = 0; i < 8; ++i) mbar_init(bar_item + i, 1);
        for (int w = 0; w < 3; ++w) mbar_init(bar_left + w, 1);
        mbar_fence_init();
        tma_prefetch_desc(&map_q);
        tma_prefetch_desc(&map_do);
        if (!kRows) {
            tma_prefetch_desc(&map_k);
            tma_prefetch_desc(&map_v);
        }
        tma_prefetch_desc(&map_acc);
    }
    if (tid < 8) s_ones[tid] = make_uint4(0x3f803f80u, 0x00003f80u, 0u, 0u);
    fence_proxy_async_smem();
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
        n_t = (kept + kTile - 1) / kTile;
        n_items = n_t * P.H * P.B;                             // (short instances skip some)
    };
    auto item_wait = [&](uint32_t i) { ok &= warp_wait_relaxed(bar_item + (i & 7), (i >> 3) & 1); };
    auto item_read = [&](uint32_t i) {
        const int4 x = *reinterpret_cast<const int4*>(s_item + (i & 7));
        return Item{x.x, x.y, x.z, x.w};
    };
    auto item_at = [&](uint32_t i) {                           // n_sel -1 for an item that did not come
        item_wait(i);
        Item it = item_read(i);
        if (!ok) it.n_sel = -1;
        return it;
    };
    auto warp_arrive = [&](uint64_t* bar) {                    // all lanes are done
        __syncwarp();
        if (lane == 0) mbar_arrive(bar);
    };
    auto next_slot = [](uint32_t& st, uint32_t& ph) {
        if (++st == kManyStages) { st = 0; ph ^= 1; }
    };

    if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kManySmallRegs));
    begin();
    // One backward pass per forward pass: the forward kernel left a mark (and cleared this workspace's counters); a backward pass that
    // does not find it (a second backward for the same forward, or two forwards sharing the workspace before their backwards) would
    // add into stale state, so it reports the call instead of returning wrong gradients.
    if (blockIdx.x == 0 && tid == 0 && atomicExch(P.status + kWsPairingWord, 0) != 1) set_status(P.status, VARDROP_ERR_INVALID_ARG);
    if (warp < 2) {
        // ------------------------------------------------------------ issue ---------------------------------------------
        // Warp 0: S^T from K and Q, dV from P^T and dO.  Warp 1: dP^T from V and dO, dK from dS^T and Q.  One body: `first` is the product that opens a
        // step, `second` the one that adds up.
        const uint32_t idesc_first = umma_idesc_bf16(128, 64, 0, 0), idesc_second = umma_idesc_bf16(128, P.D, 0, 1);
        const uint64_t d_q = umma_desc_sw128(smem_u32(sQ) + (warp == 0 ? 0 : kTileBytes), 16, 1024);                 // operand of the first product
        const uint64_t m_q = umma_desc_sw128(smem_u32(sQ) + (warp == 0 ? kTileBytes : 0), kTileBytes, 1024);         // of the second
        const uint32_t c_kv = tmem + (warp == 0 ? kColK : kColV), c_acc = tmem + (warp == 0 ? kColDv : kColDk), c_team = tmem + kColTeam + warp * 64;
        // A k-step is two rows of eight: both are the same one, whence the halves.
        const uint64_t d_ones = umma_desc_plain(smem_u32(s_ones), 0, 0), d_stats = umma_desc_plain(smem_u32(s_stats + warp * kManyStages * kTile), 0, 128);
        uint64_t* bar_first = warp == 0 ? bar_s : bar_dp;
        uint64_t* bar_handed = warp == 0 ? bar_p : bar_ds;
        uint64_t* bar_done = warp == 0 ? bar_dv_done : bar_dk_done;
        uint64_t* bar_free = warp == 0 ? bar_dv_free : bar_dk_free;
        uint32_t t = 0, st = 0, ph = 0, sn = 0, pn = 0;        // query tiles so far, their slot; slot of the tile whose first products come next
        auto wait_slot = [&]() {
            ok &= warp_wait_relaxed(bar_q_full + sn, pn);
            tc_fence_after();
        };
        auto first = [&](int w) {
            if (elect_one()) {
                const uint64_t bd = umma_desc_advance(d_q, sn * 2 * kTileBytes + w * 64 * kRowBytes);
                const uint32_t to = c_team + w * 128;
                tc_mma_bf16_ta(to, c_kv, bd, idesc_first, 0u);
                tc_mma_bf16_ta(to, c_kv + 8, umma_desc_advance(bd, 32), idesc_first, 1u);
                if (P.D > 32) {
                    tc_mma_bf16_ta(to, c_kv + 16, umma_desc_advance(bd, 64), idesc_first, 1u);
                    tc_mma_bf16_ta(to, c_kv + 24, umma_desc_advance(bd, 96), idesc_first, 1u);
                }
                tc_mma_bf16(to, d_ones, umma_desc_advance(d_stats, (sn * kTile + w * 64) * 16), idesc_first, 1u);
                tc_commit(bar_first + w);
            }
            __syncwarp();
        };
        Item it = item_at(0);
        if (it.n_sel >= 0) {
            ok &= warp_wait(bar_kv + warp, 0);
            wait_slot();
            first(0);
            first(1);
            next_slot(sn, pn);
        }
#pragma unroll 1
        for (uint32_t i = 0; ok && it.n_sel >= 0; ++i) {
            const int n_q = (it.n_sel + kTile - 1) / kTile;
            it = item_at(i + 1);
#pragma unroll 1
            for (int x = 0; x < n_q && ok; ++x, ++t) {
                const bool last = x + 1 == n_q, more = !last || it.n_sel >= 0;
#pragma unroll 1
                for (int w = 0; w < 2; ++w) {
                    ok &= warp_wait(bar_handed + w, t & 1);
                    if (i > 0 && x + w == 0) ok &= warp_wait(bar_free, (i - 1) & 1);       // the previous item's sum is out
                    tc_fence_after();
                    if (elect_one()) {
                        const uint64_t bd = umma_desc_advance(m_q, st * 2 * kTileBytes + w * 64 * kRowBytes);
                        const uint32_t a = c_team + w * 128;
#pragma unroll
                        for (int ks = 0; ks < 4; ++ks)
                            tc_mma_bf16_ta(c_acc, a + (ks >> 1) * 32 + (ks & 1) * 8, umma_desc_advance(bd, ks * 2048), idesc_second, ks > 0 ? 1u : (x + w > 0 ? 1u : 0u));
                        if (w == 1) {
                            tc_commit(bar_q_free + st);
                            if (last) tc_commit(bar_done);
                        }
                    }
                    __syncwarp();
                    if (!more) continue;
                    if (w == 0) {
                        if (last) ok &= warp_wait(bar_kv + warp, (i + 1) & 1);
                        wait_slot();
                    }
                    first(w);
                }
                if (more) next_slot(sn, pn);
                next_slot(st, ph);
            }
        }
    } else if (warp == 2) {
        const uint32_t idesc_mnmn = umma_idesc_bf16(128, P.D, 1, 1);       // A MN-major, B MN-major
        const uint64_t a_ds = umma_desc_sw128(smem_u32(sdS), kTileBytes, 1024), b_k = umma_desc_sw128(smem_u32(sK), kTileBytes, 1024);
        const uint64_t k_from = umma_desc_sw128(smem_u32(sK), 16, 1024), v_from = umma_desc_sw128(smem_u32(sV), 16, 1024);
        auto copy_kv = [&](uint32_t i, bool v) {               // an item's K or V to tensor memory
            ok &= v ? warp_wait_relaxed(bar_v_full, i & 1) : warp_wait_relaxed(bar_k_full + (i & 1), (i >> 1) & 1);
            if (kRows) fence_proxy_async_smem();               // rows written by asynchronous copies are read by the tensor core
            tc_fence_after();
            if (elect_one()) {
                const uint64_t from = v ? v_from : umma_desc_advance(k_from, (i & 1) * kTileBytes);
#pragma unroll
                for (int ks = 0; ks < 4; ++ks)
                    if (ks < 2 || P.D > 32) tc_copy_128x256b(tmem + (v ? kColV : kColK) + ks * 8, umma_desc_advance(from, ks * 32));
                tc_commit(bar_kv + (v ? 1 : 0));
                if (v) tc_commit(bar_v_free);
            }
            __syncwarp();
        };
        uint32_t t = 0;
        Item it = item_at(0);
        if (it.n_sel >= 0) {
            copy_kv(0, false);
            copy_kv(0, true);
        }
#pragma unroll 1
        for (uint32_t i = 0; ok && it.n_sel >= 0; ++i) {
            const int n_q = (it.n_sel + kTile - 1) / kTile;
            const uint64_t bk = umma_desc_advance(b_k, (i & 1) * kTileBytes);
            it = item_at(i + 1);
#pragma unroll 1
            for (int x = 0; x < n_q && ok; ++x, ++t) {
                if (x + 1 == n_q && it.n_sel >= 0) {           // the last products that read this K (V) are both teams' first ones of this tile
                    ok &= warp_wait(bar_s + 1, t & 1);
                    copy_kv(i + 1, false);
                    ok &= warp_wait(bar_dp + 1, t & 1);
                    copy_kv(i + 1, true);
                }
                if (t > 0) ok &= warp_wait_relaxed(bar_gfree, (t - 1) & 1);
                ok &= warp_wait(bar_panel, t & 1);
                ok &= warp_wait(bar_panel + 1, t & 1);
                tc_fence_after();
                if (elect_one()) {                       // dQ = dS K, dS the transposed view of dS^T
#pragma unroll
                    for (int ks = 0; ks < 8; ++ks)
                        tc_mma_bf16(tmem + kColDq, umma_desc_advance(a_ds, ks * 2048), umma_desc_advance(bk, ks * 2048), idesc_mnmn, ks > 0 ? 1u : 0u);
                    tc_commit(bar_g);
                    if (x + 1 == n_q) tc_commit(bar_k_free + (i & 1));
                }
                __syncwarp();
            }
        }
    } else {
        // ------------------------------------------------------------ loads, items --------------------------------------
        int k = blockIdx.x;                              // next item to publish, in grid steps
        auto publish = [&](uint32_t i) {
            Item it{0, 0, 0, -1};
#pragma unroll 1
            for (; it.n_sel < 0 && k < n_items; k += gridDim.x) {
                const int hb = small_div(k, n_t);
                it.b = small_div(hb, P.H);
                it.jt = k - hb * n_t;
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
        auto load_kv = [&](uint32_t i, const Item& it) {
            ok &= warp_wait_relaxed(bar_k_free + (i & 1), ((i >> 1) & 1) ^ 1);
            ok &= warp_wait_relaxed(bar_v_free, (i & 1) ^ 1);
            if (ok && lane == 0) {
                mbar_expect_tx(bar_k_full + (i & 1), kTileBytes);
                tma_load_4d(sK + (i & 1) * kTileBytes, &map_k, bar_k_full + (i & 1), 0, it.h, it.jt * kTile, it.b);
                mbar_expect_tx(bar_v_full, kTileBytes);
                tma_load_4d(sV, &map_v, bar_v_full, 0, it.h, it.jt * kTile, it.b);
            }
            __syncwarp();
        };
        uint32_t st = 0, ph = 0;
        publish(0);
        Item next = item_at(0);
        if (!kRows && next.n_sel >= 0) load_kv(0, next);
#pragma unroll 1
        for (uint32_t i = 0; ok; ++i) {
            const Item it = next;
            if (it.n_sel < 0) break;
            publish(i + 1);
            next = item_at(i + 1);
            const int n_q = (it.n_sel + kTile - 1) / kTile;
            const float* lse_row = P.lse + (static_cast<size_t>(it.b) * P.H + it.h) * P.N;
            const float* delta_row = P.delta + (static_cast<size_t>(it.b) * P.H + it.h) * P.Ncap;
            // Row statistics of a query tile travel with it, four rows a lane; those of the next tile are asked for ahead of the wait for this one's slot.
            float st_lse[4], st_delta[4];
            auto stats_load = [&](int x) {
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int r = x * kTile + e * 32 + lane;
                    st_lse[e] = r < it.n_sel ? __ldg(lse_row + r) : 0.f;       // (missing queries have zero rows of Q and dO: any P will do)
                    st_delta[e] = r < it.n_sel ? __ldg(delta_row + r) : 0.f;
                }
            };
            stats_load(0);
#pragma unroll 1
            for (int x = 0; x < n_q; ++x) {
                ok &= warp_wait_relaxed(bar_q_free + st, ph ^ 1);
                if (!ok) break;
                if (lane == 0) {                         // the tiles first: the products wait for them a step ahead of anything the statistics are for
                    mbar_expect_tx(bar_q_full + st, 2 * kTileBytes);
                    tma_load_4d(sQ + st * 2 * kTileBytes, &map_q, bar_q_full + st, 0, it.h, x * kTile, it.b);
                    tma_load_4d(sQ + st * 2 * kTileBytes + kTileBytes, &map_do, bar_q_full + st, 0, it.h, x * kTile, it.b);
                }
                __syncwarp();
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    uint32_t l[3], d[3];
                    split3(-st_lse[e] * P.half_inv_scale, l[0], l[1], l[2]);
                    split3(-0.5f * st_delta[e], d[0], d[1], d[2]);
                    s_stats[st * kTile + e * 32 + lane] = make_uint4(l[0] | l[1] << 16, l[2], 0u, 0u);
                    s_stats[(kManyStages + st) * kTile + e * 32 + lane] = make_uint4(d[0] | d[1] << 16, d[2], 0u, 0u);
                }
                fence_proxy_async_smem();
                warp_arrive(bar_q_full + st);
                stats_load(x + 1);
                next_slot(st, ph);
                if (!kRows && x == (n_q > 1 ? 1 : 0) && next.n_sel >= 0) load_kv(i + 1, next);
            }
        }
    }
    } else if (warp < 12) {
        // ------------------------------------------------------------ dQ; dV, dK of an item -----------------------------
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kManyOutRegs));
        begin();
        const int g = (warp >> 2) - 1, id = 1 + g, row = tid & (kTile - 1);
        const uint32_t tm = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16);
        const bool owner = row == 0, columns = g * 32 < P.D;     // the one thread of the warpgroup that owns its bulk reductions; there are such columns
        unsigned char* panel = sOut + g * kTileBytes;            // this warpgroup's staging panel of 128-byte swizzled rows
        unsigned char* rowp = panel + row * kRowBytes;
        auto panel_free = [&]() {
            if (owner) bulk_wait_group_read0();
            ok = group_sync_and(id, ok);
        };
        // K (V) rows of an item, 32 a warp
        auto load_rows = [&](uint32_t i, const Item& it) {
            if (!kRows || it.n_sel < 0) return;
            const int key = it.jt * kTile + row;
            const int pick = key < it.n_sel ? __ldg(P.sel_idx + static_cast<size_t>(P.S > 1 ? it.b : 0) * P.N + key) : -1;
            ok &= g == 0 ? warp_wait_relaxed(bar_k_free + (i & 1), ((i >> 1) & 1) ^ 1) : warp_wait_relaxed(bar_v_free, (i & 1) ^ 1);
            if (!ok) return;
            copy_32_picked((g == 0 ? sK + (i & 1) * kTileBytes : sV) + (warp & 3) * 32 * kRowBytes, (g == 0 ? P.k : P.v) + it.b * P.sB + it.h * P.sH, P.sN, pick, P.D);
            cp_async_arrive(g == 0 ? bar_k_full + (i & 1) : bar_v_full);
        };
        // Nothing bounds a named barrier.  A warp whose wait gave up goes on to the last barrier of its query tile, where all four learn of it, and all leave there: no
        // other exit but the end of the list, which all see, since each waits for the entry of the next item ahead of that barrier.
        load_rows(0, item_at(0));
        ok = group_sync_and(id, ok);
        uint32_t t = 0;
#pragma unroll 1
        for (uint32_t i = 0; ok; ++i) {
            const Item it = item_read(i);
            if (it.n_sel < 0) break;
            const int n_q = (it.n_sel + kTile - 1) / kTile;
            // dV or dK of the item's keys: a warp's 32 rows through its part of the panel, eight lanes a row
            auto rows_out = [&](uint32_t col, uint64_t* done, uint64_t* freed, float mul, __nv_bfloat16* dst) {
                int n[8];                                // variates of this lane's rows, -1: none
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const int key = it.jt * kTile + (warp & 3) * 32 + 4 * e + (lane >> 3);
                    n[e] = key < it.n_sel ? (kRows ? __ldg(P.sel_idx + static_cast<size_t>(P.S > 1 ? it.b : 0) * P.N + key) : key) : -1;
                }
                panel_free();
                ok &= warp_wait_relaxed(done, i & 1);
                tc_fence_after();
#pragma unroll 1
                for (int c = 0; c < P.D; c += 32) {
                    float v[32];
                    tmem_ld32(tm + col + c, v);
                    tmem_ld_wait();
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        *reinterpret_cast<uint4*>(rowp + (((c / 8 + q) ^ (row & 7)) << 4)) =
                            make_uint4(pack2(v[8 * q + 0] * mul, v[8 * q + 1] * mul), pack2(v[8 * q + 2] * mul, v[8 * q + 3] * mul),
                                       pack2(v[8 * q + 4] * mul, v[8 * q + 5] * mul), pack2(v[8 * q + 6] * mul, v[8 * q + 7] * mul));
                }
                tc_fence_before();
                warp_arrive(freed);                      // the next item's products wait for these columns
                const int c8 = lane & 7;
                if (c8 * 8 < P.D) {
                    __nv_bfloat16* out = dst + (static_cast<size_t>(it.b) * P.N * P.H + it.h) * P.D + c8 * 8;
                    const unsigned char* from = panel + ((warp & 3) * 32 + (lane >> 3)) * kRowBytes;
#pragma unroll
                    for (int e = 0; e < 8; ++e)
                        if (n[e] >= 0)
                            *reinterpret_cast<uint4*>(out + static_cast<size_t>(n[e]) * P.H * P.D) =
                                *reinterpret_cast<const uint4*>(from + 4 * e * kRowBytes + ((c8 ^ ((4 * e + (lane >> 3)) & 7)) << 4));
                }
            };
            // The next item's rows ahead of anything that waits for this one's products: those of its last query tile come behind them.
            if (kRows) load_rows(i + 1, item_at(i + 1));
            int x = 0;
#pragma unroll 1
            do {
                if (x + 1 == n_q) {                      // complete ahead of the item's last dQ, and about when it is
                    if (g == 0) rows_out(kColDv, bar_dv_done, bar_dv_free, 1.f, P.dv);
                    else rows_out(kColDk, bar_dk_done, bar_dk_free, P.scale, P.dk);
                }
                panel_free();
                ok &= warp_wait_relaxed(bar_g, t & 1);
                tc_fence_after();
                if (columns) {
                    float v[32];
                    tmem_ld32(tm + kColDq + g * 32, v);
                    tmem_ld_wait();
                    tc_fence_before();
                    warp_arrive(bar_gfree);
#pragma unroll
                    for (int e = 0; e < 8; ++e)
                        *reinterpret_cast<float4*>(rowp + ((e ^ (row & 7)) << 4)) = make_float4(v[4 * e], v[4 * e + 1], v[4 * e + 2], v[4 * e + 3]);
                    fence_proxy_async_smem();
                } else {
                    warp_arrive(bar_gfree);
                }
                if (!kRows && x == 0) item_wait(i + 1);  // (behind the hand-off that the next dQ waits for)
                ok = group_sync_and(id, ok);             // the panel is complete
                if (owner && columns) {
                    tma_reduce_add_4d(&map_acc, panel, g * 32, it.h, x * kTile, it.b);
                    bulk_commit_group();
                }
                ++t;
            } while (++x < n_q && ok);
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        if (owner) bulk_wait_group0();                   // the last reductions of dQ have landed
    } else {
        // ------------------------------------------------------------ teams ---------------------------------------------
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kManyBigRegs));
        begin();
        const int w = (warp - 12) >> 3, row = tid & (kTile - 1), half = ((warp - 12) >> 2) & 1;
        const uint32_t tm_s = tmem + kColTeam + w * 128 + half * 32 + (static_cast<uint32_t>((warp & 3) * 32) << 16), tm_d = tm_s + 64;
        unsigned char* panel = sdS + w * kTileBytes;
        uint32_t t = 0;
        bool s_ready = false;                            // a poll takes a hundred cycles to answer: polls go out ahead of where they are needed
#pragma unroll 1
        for (uint32_t i = 0; ok; ++i) {
            const Item it = item_at(i);
            if (it.n_sel < 0) break;
            const int n_q = (it.n_sel + kTile - 1) / kTile;
            // Rows of keys that do not exist are zeros and their dV, dK go nowhere; P^T = 1 keeps what they add to dQ at zero.
            const float scale = it.jt * kTile + row < it.n_sel ? P.scale_log2 : 0.f;
            const uint64_t scale2 = pair_of(scale, scale);
#pragma unroll 1
            for (int x = 0; x < n_q && ok; ++x, ++t) {
                if (!__all_sync(0xffffffffu, s_ready)) ok &= warp_wait(bar_s + w, t & 1);
                tc_fence_after();
                float s[32], d[32];
                uint32_t pk[16];
                tmem_ld32(tm_s, s);
                tmem_ld_wait();
                exp_step_folded(s, pk, scale2);
                const bool dp_ready = mbar_test(bar_dp + w, t & 1);
                tmem_st16(tm_s, pk);
                tmem_st_wait();
                tc_fence_before();
                warp_arrive(bar_p + w);                  // dV may go, and the next S^T over P^T behind it
                if (!__all_sync(0xffffffffu, dp_ready)) ok &= warp_wait(bar_dp + w, t & 1);
                tc_fence_after();
                tmem_ld32(tm_d, d);
                const bool g_done = t == 0 || mbar_test(bar_g, (t - 1) & 1);
                tmem_ld_wait();
#pragma unroll
                for (int e = 0; e < 32; e += 2) {        // dP^T has -Delta in it
                    halves_of(mul_pair(pair_of(s[e], s[e + 1]), pair_of(d[e], d[e + 1])), d[e], d[e + 1]);
                    pk[e >> 1] = pack_bf16(d[e], d[e + 1]);
                }
                tmem_st16(tm_d, pk);
                tmem_st_wait();
                tc_fence_before();
                warp_arrive(bar_ds + w);                 // dK may go, the next dP^T over dS^T behind it
                if (!__all_sync(0xffffffffu, g_done)) ok &= warp_wait(bar_g, (t - 1) & 1);   // dQ of the previous tile has read the panels
                store_panel(panel, row, half, pk);
                s_ready = mbar_test(bar_s + w, (t + 1) & 1);
                fence_proxy_async_smem();
                warp_arrive(bar_panel + w);              // and dQ
            }
        }
    }
    if (!ok) {
        set_status(P.status, VARDROP_ERR_TIMEOUT);
        if (warp < 3) {                                  // what it has issued is done before tensor memory is given back
            tc_commit_w(bar_left + warp);
            warp_wait(bar_left + warp, 0);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, kManyTmemCols);
}

// ---------------------------------------------------------------------------------------------------------
// dq from the accumulator (paths with many key tiles)
// ---------------------------------------------------------------------------------------------------------
struct ConvertParams {
    const float4* dq_acc;    // [B, Ncap, H, 64] fp32
    uint4* dq;               // [B, N, H, D] bf16
    const int32_t* sel_idx;  // [S, N]; NULL: identity
    const int32_t* n_sel;    // [S]; NULL: N
    const int32_t* inv_idx;  // [S, N]; NULL: nothing dropped
    uint4 *dk, *dv;
    int main_grid;           // CTAs of the main kernel
    int B, N, Ncap, H, D, S;
    float scale;
};

// What bounds it is memory: the accumulator's kept rows in, 16-byte results, two in flight a thread.
// Ahead of that, and of the wait for the main kernel, the zero rows of dq, dk, dv for every dropped variate, a warp a row: CTAs come in here as that
// kernel's run out of items, and it writes no row of a dropped variate.  (What these rows hang on, the selection and whoever used the buffers before, is
// done: the main kernel itself has waited for it before it let this one in.)  Beside the items, by a warp of the main kernel, they cost as much as the memory
// takes for them: ordinary stores hold up the queue that every barrier of the SM goes through, bulk stores the copy engine (1423 of 8192 kept, B = 8, a
// call: 175 us beside the items, 159 here).
constexpr int kConvertPerSm = 5;       // CTAs that an SM holds (48 registers a thread)
__global__ void __launch_bounds__(256, kConvertPerSm) bwd_convert_kernel(const ConvertParams P) {
    if (P.inv_idx) {
        const int lane = threadIdx.x & 31, rows = P.B * P.N, row_chunks = P.H * (P.D / 8);
        const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
        // The first CTAs come in where the main kernel has an item less, as many as those SMs hold: they stay there until it is done, and the others come behind it.
        // They take as many rows more as an item is long (2700 cycles a query tile, 25 bytes written a cycle and SM), as long as the late ones keep the early ones'
        // part of an even share.  (By graphs, forward and backward, counted as eight an SM | five | six, with 40 registers | eight, with 32: 1423 of 8192 kept, B = 8
        // 232.9 us | 227.5 | 227.8 | 231.6, 400 of 4000, B = 16 102.2 | 101.9 | 103.7 | 104.5, 300 of 3000, B = 8 47.4 | 46.2 | 46.6 | 47.8.)
        const int kept = largest_kept(P.n_sel, P.S, P.N), n_t = (kept + kTile - 1) / kTile, n_long = n_t * P.H * P.B % P.main_grid;
        const int ctas = static_cast<int>(gridDim.x * gridDim.y), cta = static_cast<int>(blockIdx.y * gridDim.x + blockIdx.x);
        const int n_early = n_long ? min(ctas, kConvertPerSm * (P.main_grid - n_long)) : 0;
        const RowShares shares = row_shares(rows, ctas, n_early, 2700.f * 25.f / kConvertPerSm * n_t / (48.f * row_chunks) * P.N / max(1, P.N - kept));
        const int end = first_row(shares, cta + 1);
#pragma unroll 1
        for (int at = first_row(shares, cta) + static_cast<int>(threadIdx.x >> 5) * 8; at < end; at += 64) {
            bool dropped = false;
            if (lane < 8 && at + lane < end) {
                const int b = small_div(at + lane, P.N);
                dropped = __ldcg(P.inv_idx + static_cast<size_t>(P.S > 1 ? b : 0) * P.N + (at + lane - b * P.N)) < 0;
            }
#pragma unroll 1
            for (unsigned mask = __ballot_sync(0xffffffffu, dropped); mask; mask &= mask - 1) {
                const size_t to = static_cast<size_t>(at + __ffs(mask) - 1) * row_chunks;
#pragma unroll 1
                for (int c = lane; c < row_chunks; c += 32) {
                    P.dq[to + c] = zero;
                    P.dk[to + c] = zero;
                    P.dv[to + c] = zero;
                }
            }
        }
    }
    chain_wait();
    chain_release();
    const int b = blockIdx.y, srow = P.S > 1 ? b : 0;
    const int n_sel = P.n_sel ? P.n_sel[srow] : P.N;
    const int32_t* sel = P.sel_idx ? P.sel_idx + static_cast<size_t>(srow) * P.N : nullptr;
    const int sh = P.D > 32 ? 3 : 2, chunks_row = P.H << sh;        // 16-byte results per row
    const int total = n_sel * chunks_row, stride = gridDim.x * blockDim.x;
    const float4* acc = P.dq_acc + static_cast<size_t>(b) * P.Ncap * P.H * (kDP / 4);
    uint4* dq = P.dq + static_cast<size_t>(b) * P.N * chunks_row;
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += 2 * stride) {
        float4 a[2][2];
        size_t to[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int at = min(idx + e * stride, total - 1);
            const int j = small_div(at, chunks_row), c = at - j * chunks_row, h = c >> sh, dc = c & ((1 << sh) - 1);
            to[e] = static_cast<size_t>(sel ? __ldg(sel + j) : j) * chunks_row + c;
            const float4* src = acc + (static_cast<size_t>(j) * P.H + h) * (kDP / 4) + dc * 2;
            a[e][0] = __ldcg(src);
            a[e][1] = __ldcg(src + 1);
        }
#pragma unroll
        for (int e = 0; e < 2; ++e)
            if (idx + e * stride < total)
                dq[to[e]] = make_uint4(pack2(a[e][0].x * P.scale, a[e][0].y * P.scale), pack2(a[e][0].z * P.scale, a[e][0].w * P.scale),
                                       pack2(a[e][1].x * P.scale, a[e][1].y * P.scale), pack2(a[e][1].z * P.scale, a[e][1].w * P.scale));
    }
}

}  // namespace

int attn_bwd_many_launch(const void* q, const void* k, const void* v, const void* o, const float* lse, const void* d_o, const int32_t* sel_idx, const int32_t* n_sel,
                         const int32_t* inv_idx, const vardrop_attn_cfg& c, void* dq, void* dk, void* dv, void* ws, cudaStream_t stream) {
    const AttnWs w = attn_layout(c);
    const QkvLayout L = qkv_layout(c);
    char* base = static_cast<char*>(ws);
    ManyParams P{};
    P.k = static_cast<const __nv_bfloat16*>(k); P.v = static_cast<const __nv_bfloat16*>(v);
    P.lse = lse; P.delta = reinterpret_cast<const float*>(base + w.delta);
    P.dk = static_cast<__nv_bfloat16*>(dk); P.dv = static_cast<__nv_bfloat16*>(dv);
    P.sel_idx = sel_idx; P.n_sel = sel_idx ? n_sel : nullptr;
    P.status = reinterpret_cast<int*>(base);
    P.sB = L.sB; P.sN = L.sN; P.sH = L.sH;
    P.B = c.B; P.N = c.N; P.Ncap = w.Ncap; P.H = c.H; P.D = c.D; P.S = attn_sel_rows(c, sel_idx);
    P.scale = c.sm_scale > 0.f ? c.sm_scale : 1.f / sqrtf(static_cast<float>(c.D));
    // -lse / scale has to be finite: in the exponents a scale counts as 2^-120 at least, against which any score below 2^90 is nothing (lse is the logarithm of the
    // kept count then).  dQ and dK get the scale as it is.
    const float least = fmaxf(P.scale, 7.5231638e-37f);
    P.scale_log2 = least * 1.4426950408889634f;
    P.half_inv_scale = 0.5f / least;
    const int gx = max(1, 8 * sm_count() / c.B);                   // of prep and convert: about eight CTAs per SM in total
    {
        PrepParams R{};
        R.o = static_cast<const uint4*>(o); R.d_o = static_cast<const uint4*>(d_o);
        R.delta = reinterpret_cast<float*>(base + w.delta);
        R.dq_acc = attn_fwd_clears(c, sel_idx) ? nullptr : reinterpret_cast<float4*>(base + w.dq_acc);
        R.q = static_cast<const __nv_bfloat16*>(q);
        for (int i = 0; i < 2; ++i) R.staged[i] = reinterpret_cast<uint4*>(base + w.staged[i]);
        R.sel_idx = sel_idx;
        R.sB = L.sB; R.sN = L.sN; R.sH = L.sH;
        R.n_sel = P.n_sel;
        R.N = c.N; R.Ncap = w.Ncap; R.H = c.H; R.D = c.D; R.S = P.S;
        const long long blocks = (static_cast<long long>(w.Ncap) * c.H * 8 + 255) / 256;
        cudaError_t err;
        { LaunchScope ls_(K_BWD_PREP, stream); err = launch_chained(bwd_prep_kernel, dim3(static_cast<int>(blocks < gx ? blocks : gx), c.B), dim3(256), 0, stream, R); }
        if (int st = check_cuda(err, "attention: backward prep launch")) return st;
    }
    CUtensorMap mq{}, mk{}, mv{}, mdo{}, macc;
    const long long HD = static_cast<long long>(c.H) * c.D;
    if (sel_idx) {
        CUtensorMap* const maps[2] = {&mq, &mdo};
        for (int i = 0; i < 2; ++i)
            if (int st = make_tile_map(maps[i], base + w.staged[i], c.D, c.B, w.Ncap, c.H, w.Ncap * HD, HD, c.D)) return st;
    } else {
        if (int st = make_tile_map(&mq, q, c.D, c.B, c.N, c.H, L.sB, L.sN, L.sH)) return st;
        if (int st = make_tile_map(&mk, k, c.D, c.B, c.N, c.H, L.sB, L.sN, L.sH)) return st;
        if (int st = make_tile_map(&mv, v, c.D, c.B, c.N, c.H, L.sB, L.sN, L.sH)) return st;
        if (int st = make_tile_map(&mdo, d_o, c.D, c.B, c.N, c.H, c.N * HD, HD, c.D)) return st;
    }
    if (int st = make_acc_map(&macc, base + w.dq_acc, c.B, w.Ncap, c.H)) return st;
    const long long worst = static_cast<long long>(w.Ncap / kTile) * c.H * c.B;
    const int grid = static_cast<int>(worst < sm_count() ? worst : sm_count());          // one CTA per SM (all of tensor memory)
    auto launch = [&](auto kernel, int& attr_dev) {
        int dev = 0;
        cudaGetDevice(&dev);
        if (attr_dev != dev) {
            if (int st = check_cuda(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kManySmemBytes), "attention: smem attribute")) return st;
            attr_dev = dev;
        }
        LaunchScope ls_(K_ATTN_BWD, stream);
        return check_cuda(launch_chained(kernel, dim3(grid), dim3(kManyThreads), kManySmemBytes, stream, mq, mk, mv, mdo, macc, P), "attention: backward launch");
    };
    static thread_local int attr_all = -1, attr_rows = -1;
    if (int st = sel_idx ? launch(bwd_many_kernel<true>, attr_rows) : launch(bwd_many_kernel<false>, attr_all)) return st;
    ConvertParams F{};
    F.dq_acc = reinterpret_cast<const float4*>(base + w.dq_acc);
    F.dq = static_cast<uint4*>(dq);
    F.sel_idx = sel_idx;
    F.n_sel = P.n_sel;
    F.inv_idx = sel_idx ? inv_idx : nullptr;
    F.main_grid = grid;
    F.dk = static_cast<uint4*>(dk); F.dv = static_cast<uint4*>(dv);
    F.B = c.B; F.N = c.N; F.Ncap = w.Ncap; F.H = c.H; F.D = c.D; F.S = P.S; F.scale = P.scale;
    const long long blocks = (static_cast<long long>(c.N) * c.H * (c.D / 8) + 255) / 256;
    cudaError_t err;
    { LaunchScope ls_(K_BWD_CONVERT, stream); err = launch_chained(bwd_convert_kernel, dim3(static_cast<int>(blocks < gx ? blocks : gx), c.B), dim3(256), 0, stream, F); }
    return check_cuda(err, "attention: backward convert launch");
}

}  // namespace vardrop
