// Attention forward (Eq. 3) over the kept variate tokens.
//
// attn_fwd_tile_kernel   few tiles (the kept sets of the paper's workloads): 128-thread CTAs, four to an SM, one 128-query tile each.
// attn_fwd_kernel        many tiles: one persistent CTA per SM over pairs of 128-query tiles, a warp role for each part of the work.
//
// Both form S = Q K^T and O += P V on the tcgen05 tensor cores with the accumulators, and P itself, in tensor memory; operand rows come
// straight from the caller's tensors (boxes, or the kept rows by asynchronous copies).
#include "attn_common.cuh"

namespace vardrop {

// ---------------------------------------------------------------------------------------------------------
// host: tensor maps
// ---------------------------------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_tiled_fn() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qres) == cudaSuccess &&
            qres == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    }
    return fn;
}

// Encoding a tensor map costs a driver call of a microsecond or two and a training loop passes the same buffers step after
// step: a small per-thread cache, keyed by everything the encoding depends on, returns the map of a known buffer.
namespace {
struct MapKey {
    const void* base;
    long long a;
    int kind, b, c, d;
    bool operator==(const MapKey& o) const { return base == o.base && a == o.a && kind == o.kind && b == o.b && c == o.c && d == o.d; }
};
struct alignas(64) MapSlot {
    CUtensorMap map;
    MapKey key;
    long long aux[3];      // strides of a tile map (the key only carries a mix of them)
    bool used;
};
constexpr int kMapSlots = 256;
MapSlot* map_slot(const MapKey& k) {
    static thread_local MapSlot slots[kMapSlots] = {};
    const uintptr_t h = (reinterpret_cast<uintptr_t>(k.base) >> 8) * 0x9E3779B97F4A7C15ull + static_cast<uintptr_t>(k.kind) * 0x632BE5ABull;
    return &slots[(h >> 40) % kMapSlots];
}
}  // namespace

int sm_count() {
    static thread_local int cached_dev = -1, cached = 148;
    int dev = 0;
    if (cudaGetDevice(&dev) == cudaSuccess && dev != cached_dev) {
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && n > 0) cached = n;
        cached_dev = dev;
    }
    return cached;
}

int make_tile_map(CUtensorMap* map, const void* base, int D, int B, int tokens, int H, long long sB, long long sN, long long sH) {
    const MapKey key{base, (sB * 131 + sN * 31 + sH) * 128 + D, 1, B, tokens, H};
    MapSlot* slot = map_slot(key);
    if (slot->used && slot->key == key && slot->aux[0] == sB && slot->aux[1] == sN && slot->aux[2] == sH) { *map = slot->map; return VARDROP_OK; }
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return fail(VARDROP_ERR_CUDA, "attention: cuTensorMapEncodeTiled entry point not available");
    const cuuint64_t dims[4] = {static_cast<cuuint64_t>(D), static_cast<cuuint64_t>(H), static_cast<cuuint64_t>(tokens),
                                static_cast<cuuint64_t>(B)};
    const cuuint64_t strides[3] = {static_cast<cuuint64_t>(sH) * 2, static_cast<cuuint64_t>(sN) * 2, static_cast<cuuint64_t>(sB) * 2};
    const cuuint32_t box[4] = {kDP, 1, kTile, 1};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    const CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return fail(VARDROP_ERR_CUDA, "attention: cuTensorMapEncodeTiled failed with code %d", static_cast<int>(r));
    slot->map = *map; slot->key = key; slot->used = true;
    slot->aux[0] = sB; slot->aux[1] = sN; slot->aux[2] = sH;
    return VARDROP_OK;
}

int make_acc_map(CUtensorMap* map, const void* base, int B, int Ncap, int H) {
    const MapKey key{base, 0, 2, B, Ncap, H};
    MapSlot* slot = map_slot(key);
    if (slot->used && slot->key == key) { *map = slot->map; return VARDROP_OK; }
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return fail(VARDROP_ERR_CUDA, "attention: cuTensorMapEncodeTiled entry point not available");
    const cuuint64_t dims[4] = {static_cast<cuuint64_t>(kDP), static_cast<cuuint64_t>(H), static_cast<cuuint64_t>(Ncap), static_cast<cuuint64_t>(B)};
    const cuuint64_t strides[3] = {static_cast<cuuint64_t>(kDP) * 4, static_cast<cuuint64_t>(H) * kDP * 4, static_cast<cuuint64_t>(Ncap) * H * kDP * 4};
    const cuuint32_t box[4] = {32, 1, kTile, 1};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    const CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                          CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return fail(VARDROP_ERR_CUDA, "attention: cuTensorMapEncodeTiled (accumulator) failed with code %d", static_cast<int>(r));
    slot->map = *map; slot->key = key; slot->used = true;
    return VARDROP_OK;
}

int attn_validate(const vardrop_attn_cfg& c) {
    if (c.B < 1 || c.N < 1 || c.H < 1) return fail(VARDROP_ERR_INVALID_ARG, "attention: B, N, H >= 1 required (B=%d N=%d H=%d)", c.B, c.N, c.H);
    if (c.D != 32 && c.D != 64) return fail(VARDROP_ERR_UNSUPPORTED, "attention: head dimension %d (32 or 64 supported)", c.D);
    if (c.N > 65536) return fail(VARDROP_ERR_UNSUPPORTED, "attention: N=%d above 65536", c.N);
    if (static_cast<long long>(c.B) * c.N * c.H >= (1ll << 31)) return fail(VARDROP_ERR_UNSUPPORTED, "attention: B*N*H above 2^31");
    if (c.H > 65535 || c.B > 65535) return fail(VARDROP_ERR_UNSUPPORTED, "attention: B or H above 65535");
    if (c.S != 0 && c.S != 1 && c.S != c.B) return fail(VARDROP_ERR_INVALID_ARG, "attention: S=%d must be 1 (shared selection) or B (one per instance)", c.S);
    if (!(c.sm_scale >= 0.f)) return fail(VARDROP_ERR_INVALID_ARG, "attention: sm_scale must be >= 0 (0 selects 1/sqrt(D))");
    if (c.sB != 0 || c.sN != 0 || c.sH != 0) {
        if (c.sH < c.D || c.sN < c.sH || c.sB < c.sN || (c.sH | c.sN | c.sB) % 8 != 0)
            return fail(VARDROP_ERR_INVALID_ARG, "attention: strides sB=%lld sN=%lld sH=%lld must be multiples of 8 with sB >= sN >= sH >= D (or all 0)",
                        static_cast<long long>(c.sB), static_cast<long long>(c.sN), static_cast<long long>(c.sH));
        if (c.sB > (1ll << 38)) return fail(VARDROP_ERR_UNSUPPORTED, "attention: sB above 2^38 elements");
    }
    return VARDROP_OK;
}

size_t attn_workspace_bytes(const vardrop_attn_cfg& c) { return attn_layout(c).total; }

namespace {

// ---------------------------------------------------------------------------------------------------------
// forward
// ---------------------------------------------------------------------------------------------------------
struct FwdParams {
    const __nv_bfloat16 *q, *k, *v;    // read by the row copies of a selection (boxes go through the tensor maps)
    __nv_bfloat16* o;
    float* lse;
    const int32_t* sel_idx; // [S, N] kept variates; NULL: all N tokens
    const int32_t* n_sel;   // [S] kept counts; NULL: all N tokens
    int* status;
    float4* dq_acc;         // [B, Ncap, H, 64] fp32: zeroed here where the backward pass will accumulate into it (NULL: the backward pass does)
    int32_t* tile_done;     // few tiles: [B, H] completion counters of the backward pass, zeroed here
    long long sB, sN, sH;   // element strides of q, k, v
    int B, N, Ncap, H, D, S;
    float scale_log2;       // sm_scale * log2(e)
};

// Work items: two 128-query tiles each, either two neighbouring tiles of one (head, instance) over the same keys, or (what an odd
// tile count leaves over, and all there is when the kept set is a single tile) the last tile of two
// neighbouring heads, each with keys of its own.  Roles of a CTA (one per SM, persistent over the items):
//   warps 0, 1       issue the tensor-core products of tile 0, 1 (every lane runs the issue code so that operands stay in
//                    uniform registers, an elected lane executes each product); first in the CTA because the schedulers favour the
//                    oldest ready warp and their short chains sit on the critical path
//   warps 2, 3       load Q (double-buffered across items) and a four-stage ring of K/V tiles
//   warps 4-7        finish an item: O / l, rounded to bf16 and written as whole rows, while the softmax warpgroups are already in
//                    the next one (done by the softmax warpgroups it was 5000 cycles an item, more than a step and a half of seven)
//   warps 8-23       four softmax warpgroups, two to a query tile: one thread per row and 64-key half of a step
// The limit is the special-function unit: 16 exponentials a cycle and SM make 1024 cycles per 128 x 128 scores where the products
// need 512 (N = 128 scores at 64 cycles, N = 64 P V at 32 with P in tensor memory).  What it takes to get near it:
//   - a softmax thread never waits for a product: it copies its scores to registers and frees their columns at once, so the next
//     S = Q K^T runs under the exponentials, and P has columns of its own, so P V of the step before does too;
//   - four warps a scheduler: what surrounds the exponentials of one (tensor-memory loads, maximum, hand-offs: as long as the
//     exponentials themselves) runs under those of the others (two threads a row share its reference maximum through shared memory);
//   - little code: a warp's step is some 300 instructions (one thread per row made it 1300, and short items, which run every path
//     once, then spend their time on instruction fetch).
// Measured, events around the launch: 8192 variates, B = 8, 1380 us (1528 with one thread per row and the staged form), 862 variates, B = 32, 104 us
// (120); 1423 kept of 8192 83 us and no gather launch (94 + 20).  Back to back the last two take 98 and 75.
// Tensor memory of tile w (256 columns): S 128 | P 64 | O 64.
constexpr int kFwdTiles = 2;                     // query tiles of an item
constexpr int kFwdGroupThreads = 128;
constexpr int kFwdTileThreads = 2 * kFwdGroupThreads;      // softmax threads of a tile
constexpr int kFwdThreads = 2 * kFwdGroupThreads + kFwdTiles * kFwdTileThreads;
// Register split (setmaxnreg works on whole warpgroups): launched with 768 x 80 = 61440 registers; the softmax warpgroups take 96 a
// thread, the others keep 48: 512 x 96 + 256 x 48 = 61440.
constexpr int kFwdSoftmaxRegs = 96;
constexpr int kFwdOtherRegs = 48;
constexpr int kFwdStages = 4;                    // K/V ring (stages of one 128-key K tile and V tile)
constexpr uint32_t kFwdTmemCols = 512;
constexpr int kFwdSmemBytes = 8192 /*barriers, row maxima and sums, alignment*/ + 2 * kFwdTiles * kTileBytes /*Q tiles of two items*/ + kFwdStages * 2 * kTileBytes /*K, V ring*/ +
                              kTileBytes /*O staging*/;
constexpr int kFwdLoadWarps = 2;
constexpr float kRescaleStep = 8.f;              // the reference maximum of a row moves only when the running maximum has grown by 2^8
// It starts as the maximum over the row's first 64 keys: which keys it is taken over decides how P is rounded to bf16, and so the last bits of O
// (which calls without a selection keep whichever kernel serves them).
__device__ __forceinline__ float first_reference(float m_first64, float m_rest) { return m_rest > m_first64 + kRescaleStep ? m_rest : m_first64; }

// The arithmetic of the softmax, written as instructions that keep their order (volatile): left to itself the compiler places the
// consumers of a pair of exponentials right behind it, and a warp then runs at the latency of the special-function unit (20 cycles
// an exponential, measured) instead of its rate (8): see the batches in the kernel.
// 2^x by the special-function unit (relative error about 2^-22; -inf gives 0)
__device__ __forceinline__ float fast_exp2(float x) {
    float y;
    asm volatile("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Two fp32 values in one 64-bit register pair, for the packed fp32 instructions of sm_100 (one issue slot for two results;
// each half is the IEEE operation of the scalar instruction, so results do not change).
__device__ __forceinline__ uint64_t pair_of(float lo, float hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void halves_of(uint64_t v, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }
__device__ __forceinline__ uint64_t fma_pair(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t d;
    asm volatile("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ uint64_t add_pair(uint64_t a, uint64_t b) {
    uint64_t d;
    asm volatile("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
    float d;
    asm volatile("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    uint32_t d;
    asm volatile("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
    return d;
}

// every lane of the warp waits; the result is the same in all of them
__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity) { return __all_sync(0xffffffffu, mbar_wait(bar, parity)); }
// the same with a sleep between polls: for warps whose reaction time is not on the critical path
__device__ __forceinline__ bool warp_wait_relaxed(uint64_t* bar, uint32_t parity) { return __all_sync(0xffffffffu, mbar_wait_relaxed(bar, parity)); }

// barrier among the 256 softmax threads of tile w
__device__ __forceinline__ void tile_sync(int w) {
    if (w == 0) asm volatile("bar.sync 2, 256;" ::: "memory");
    else asm volatile("bar.sync 3, 256;" ::: "memory");
}
__device__ __forceinline__ void tile_arrive(int w) {
    if (w == 0) asm volatile("bar.arrive 2, 256;" ::: "memory");
    else asm volatile("bar.arrive 3, 256;" ::: "memory");
}

__global__ void __launch_bounds__(kFwdThreads, 1) attn_fwd_kernel(const __grid_constant__ CUtensorMap map_q,
                                                                   const __grid_constant__ CUtensorMap map_k,
                                                                   const __grid_constant__ CUtensorMap map_v, const FwdParams P) {
    extern __shared__ unsigned char smem_dyn[];
    // Set-up first (shared-memory carve-up, barriers, tensor memory): it touches nothing another kernel produces, so it runs
    // while the previous kernel of the stream is still finishing.
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem_dyn);     // barriers and the TMEM slot sit in front of the tiles
    uint64_t* bar_q_full = bars + 0;                // [2] Q tiles of an item have landed
    uint64_t* bar_q_free = bars + 2;                // [2] every S product of the item has completed (both issue warps)
    uint64_t* bar_kv_full = bars + 4;               // [kFwdStages]
    uint64_t* bar_kv_free = bar_kv_full + kFwdStages;  // [kFwdStages] every product reading the stage has completed (both issue warps)
    uint64_t* bar_s = bar_kv_free + kFwdStages;     // [2] S of tile w's next step is in tensor memory
    uint64_t* bar_sfree = bar_s + kFwdTiles;       // [2] tile w's threads hold S in registers (256 arrivals)
    uint64_t* bar_p = bar_sfree + kFwdTiles;       // [2] P of tile w is in tensor memory (256 arrivals)
    uint64_t* bar_pv = bar_p + kFwdTiles;          // [2] O += P V of tile w's step has completed
    uint64_t* bar_l = bar_pv + kFwdTiles;          // [2] row sums and maxima of tile w's item are in shared memory (256 arrivals)
    uint64_t* bar_ofree = bar_l + kFwdTiles;       // [2] they and O have been read (128 arrivals): the next item may overwrite them
    uint64_t* bar_first = bar_ofree + kFwdTiles;    // the first item's row copies have landed
    uint64_t* bar_item = bar_first + 1;             // [8] entry of the item list is written
    uint64_t* bar_stagger = bar_item + 8;           // P of tile 0's first step is in tensor memory; completes once
    uint64_t* bar_skip = bar_stagger + 1;           // [2] tile 1's softmax warps (8), its issue warp are in an item without a second tile
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bar_skip + 2);
    float* s_max = reinterpret_cast<float*>(smem_dyn + 768);    // [tile][step parity][half][row] maxima of a step
    float* s_ref = s_max + kFwdTiles * 4 * kTile;               // [tile][row] reference maximum (log2 domain)
    float* s_sum = s_ref + kFwdTiles * kTile;                   // [tile][half][row] sums
    unsigned char* sQ = align_tiles(reinterpret_cast<unsigned char*>(s_sum + kFwdTiles * 2 * kTile));
    unsigned char* sK = sQ + 2 * kFwdTiles * kTileBytes;       // kFwdStages stages of (K tile, V tile)
    unsigned char* sOut = sK + kFwdStages * 2 * kTileBytes;     // staging tile
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (sOut + kTileBytes > smem_dyn + kFwdSmemBytes) {     // dynamic shared memory base not 1024-byte aligned
        chain_wait();
        if (tid == 0) set_status(P.status, VARDROP_ERR_CUDA);
        return;
    }
    const bool boxes = P.sel_idx == nullptr;
    if (warp == 0) {
        tmem_alloc(tmem_slot, kFwdTmemCols);
        tmem_relinquish();
    }
    if (tid == 0) {
        const uint32_t n_load = boxes ? 1 : 32 * kFwdLoadWarps;      // a box: one announcing arrival; row copies: one of every loader lane
        for (int i = 0; i < 2; ++i) {
            mbar_init(bar_q_full + i, n_load);
            mbar_init(bar_q_free + i, 2);
        }
        for (int st = 0; st < kFwdStages; ++st) {
            mbar_init(bar_kv_full + st, n_load);
            mbar_init(bar_kv_free + st, 2);
        }
        for (int w = 0; w < kFwdTiles; ++w) {
            mbar_init(bar_s + w, 1);
            mbar_init(bar_sfree + w, kFwdTileThreads);
            mbar_init(bar_p + w, kFwdTileThreads);
            mbar_init(bar_pv + w, 1);
            mbar_init(bar_l + w, kFwdTileThreads);
            mbar_init(bar_ofree + w, kFwdGroupThreads);
        }
        mbar_init(bar_first, kFwdThreads - 128);
        for (int i = 0; i < 8; ++i) mbar_init(bar_item + i, 1);
        mbar_init(bar_stagger, 1);
        mbar_init(bar_skip, kFwdTileThreads / 32);
        mbar_init(bar_skip + 1, 1);
        mbar_fence_init();
        if (boxes) {
            tma_prefetch_desc(&map_q);
            tma_prefetch_desc(&map_k);
            tma_prefetch_desc(&map_v);
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    bool ok = true;
    // Work items, decoded by the first loader warp one ahead and passed to the other roles through shared memory (decoding takes a few
    // divisions, whose conversions and reciprocals queue behind the exponentials in the special-function unit: 1000 to 2000 cycles
    // an item when every role did it).  Eight entries: the loads run at most two items ahead of the products, these one of the rows
    // leaving, so an entry has been read long before its place is taken again.
    // Tile w of an item: query tile qt + w of head h, or (split) tile qt of head h + w.  n_act: tiles that exist; -1 ends the list.
    struct alignas(16) Item { int b, h, qt, n_sel, n_kv, n_act, split, pad; };
    Item* s_item = reinterpret_cast<Item*>(smem_dyn + 512);
    auto item_at = [&](uint32_t i) {
        Item it;
        ok &= warp_wait_relaxed(bar_item + (i & 7), (i >> 3) & 1);
        const int4* from = reinterpret_cast<const int4*>(s_item + (i & 7));
        const int4 x = from[0], y = from[1];
        it.b = x.x; it.h = x.y; it.qt = x.z; it.n_sel = x.w; it.n_kv = y.x; it.n_act = ok ? y.y : -1; it.split = y.z;
        return it;
    };
    // Behind every role's entry code, so that fetching that code overlaps the previous kernel.
    auto begin = [&]() {
        chain_wait();
        chain_release();
    };

    // The first item's Q tiles and first K/V stages (one, or one of each warpgroup) of a selection: all warps but the issuing and the
    // loading ones share the row copies.
    auto load_first = [&]() {
        if (boxes) return;
        const Item it = item_at(0);
        if (it.n_act < 0) return;
        const int32_t* idx = P.sel_idx + static_cast<size_t>(P.S > 1 ? it.b : 0) * P.N;
        const int n_tiles = it.n_act + (it.split ? 2 * it.n_act : 2);
#pragma unroll 1
        for (int task = warp - 4; task < 4 * n_tiles; task += kFwdThreads / 32 - 4) {
            const int tile = task >> 2, g = task & 3, kv = tile - it.n_act, w = kv < 0 ? tile : kv >> 1;
            const __nv_bfloat16* from = (kv < 0 ? P.q : (kv & 1) ? P.v : P.k) + it.b * P.sB + (it.h + (it.split ? w : 0)) * P.sH;
            unsigned char* to = (kv < 0 ? sQ + tile * kTileBytes : sK + kv * kTileBytes) + g * 32 * kRowBytes;
            copy_32_rows(to, from, P.sN, idx, (kv < 0 ? (it.split ? it.qt : it.qt + w) * kTile : 0) + g * 32, it.n_sel, P.D);
        }
        cp_async_arrive(bar_first);
    };

    if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kFwdOtherRegs));
    if (warp >= 2) {
        // ---------------------------------------------------------------- loads ----------------------------------
        const int part = warp - 2;
        uint32_t stage_n = 0, n_done = 0;
        begin();
        if (blockIdx.x == 0 && tid == 64) P.status[kWsPairingWord] = 1;     // this workspace now holds a forward pass that no backward pass has consumed
        const int kept = largest_kept(P.n_sel, P.S, P.N);
        const int n_t = (kept + kTile - 1) / kTile, hs = (P.H + 1) >> 1;    // tiles of the longest selection
        const int per_b = (n_t >> 1) * P.H + (n_t & 1) * hs;                // items of an instance of that length (shorter ones skip some)
        int k = blockIdx.x;                              // next item to publish, in grid steps
        auto publish = [&](uint32_t i) {
            Item it;
            it.n_act = -1;
#pragma unroll 1
            for (; it.n_act < 0 && k < per_b * P.B; k += gridDim.x) {
                it.b = small_div(k, per_b);
                int r = k - it.b * per_b;
                it.n_sel = P.S > 1 ? P.n_sel[it.b] : kept;
                it.n_kv = (it.n_sel + kTile - 1) / kTile;
                const int pairs = it.n_kv >> 1;
                it.split = r >= pairs * P.H;
                if (!it.split) {
                    it.h = small_div(r, pairs);
                    it.qt = 2 * (r - it.h * pairs);
                    it.n_act = 2;
                } else {
                    it.h = 2 * (r - pairs * P.H);
                    it.qt = it.n_kv - 1;
                    if ((it.n_kv & 1) && it.h < P.H) it.n_act = min(2, P.H - it.h);      // otherwise a shorter instance has no such item
                }
            }
            if (lane == 0) {
                int4* to = reinterpret_cast<int4*>(s_item + (i & 7));
                to[0] = make_int4(it.b, it.h, it.qt, it.n_sel);
                to[1] = make_int4(it.n_kv, it.n_act, it.split, 0);
                mbar_arrive(bar_item + (i & 7));
            }
            __syncwarp();
        };
        if (part == 0) publish(0);
        if (!boxes || part == 0) {
#pragma unroll 1
            for (uint32_t i = 0; ok; ++i) {
                if (part == 0) publish(i + 1);
                const Item it = item_at(i);
                if (it.n_act < 0) break;
                const uint32_t qb = n_done & 1;
                ok = warp_wait_relaxed(bar_q_free + qb, ((n_done >> 1) & 1) ^ 1);
                if (!ok) break;
                unsigned char* sq = sQ + qb * kFwdTiles * kTileBytes;
                if (boxes) {
                    auto tile = [&](unsigned char* to, const CUtensorMap* map, uint64_t* bar, int h, int tok0) {
                        if (lane == 0) tma_load_4d(to, map, bar, 0, h, tok0, it.b);
                    };
                    if (lane == 0) mbar_expect_tx(bar_q_full + qb, it.n_act * kTileBytes);
                    __syncwarp();
#pragma unroll 1
                    for (int w = 0; w < it.n_act; ++w)
                        tile(sq + w * kTileBytes, &map_q, bar_q_full + qb, it.split ? it.h + w : it.h, (it.split ? it.qt : it.qt + w) * kTile);
                    int x = 0, j = 0;
#pragma unroll 1
                    for (int l = 0; l < it.n_kv * (it.split ? it.n_act : 1); ++l, ++stage_n) {
                        const uint32_t st = stage_n % kFwdStages;
                        ok = warp_wait_relaxed(bar_kv_free + st, ((stage_n / kFwdStages) & 1) ^ 1);
                        if (!ok) break;
                        if (lane == 0) mbar_expect_tx(bar_kv_full + st, 2 * kTileBytes);
                        __syncwarp();
#pragma unroll 1
                        for (int kv = 0; kv < 2; ++kv)
                            tile(sK + (2 * st + kv) * kTileBytes, kv ? &map_v : &map_k, bar_kv_full + st, it.h + x, j * kTile);
                        if (++x == (it.split ? it.n_act : 1)) { x = 0; ++j; }
                    }
                } else {
                    const int32_t* idx = P.sel_idx + static_cast<size_t>(P.S > 1 ? it.b : 0) * P.N;
                    const long long base = it.b * P.sB + it.h * P.sH;
                    const int per_step = it.split ? it.n_act : 1;
                    int l = 0, x = 0, j = 0;
                    if (i == 0) {       // brought in by the other warps: pass it on
                        ok = warp_wait(bar_first, 0);
                        if (!ok) break;
                        mbar_arrive(bar_q_full);
                        for (; static_cast<int>(stage_n) < per_step; ++stage_n) mbar_arrive(bar_kv_full + stage_n);
                        l = per_step;
                        j = 1;
                    } else {
#pragma unroll 1
                        for (int w = 0; w < it.n_act; ++w)
                            copy_tile_rows<false>(sq + w * kTileBytes, P.q + base + (it.split ? w * P.sH : 0), nullptr, P.sN,
                                                  tile_picks(idx, (it.split ? it.qt : it.qt + w) * kTile, it.n_sel, part), P.D, part);
                        cp_async_arrive(bar_q_full + qb);
                    }
#pragma unroll 1
                    for (; l < it.n_kv * per_step; ++l, ++stage_n) {
                        const uint32_t st = stage_n % kFwdStages;
                        const RowPicks picks = tile_picks(idx, j * kTile, it.n_sel, part);
                        ok = warp_wait_relaxed(bar_kv_free + st, ((stage_n / kFwdStages) & 1) ^ 1);
                        if (!ok) break;
                        copy_tile_rows<true>(sK + st * 2 * kTileBytes, P.k + base + x * P.sH, P.v + base + x * P.sH, P.sN, picks, P.D, part);
                        cp_async_arrive(bar_kv_full + st);
                        if (++x == per_step) { x = 0; ++j; }
                    }
                }
                ++n_done;
            }
            asm volatile("cp.async.wait_all;" ::: "memory");
        }
    } else {
        // ---------------------------------------------------------------- tensor-core issue ----------------------
        // Issue warp w serves softmax warpgroup w.  Both warps follow every stage of the ring and release it with a commit of their own
        // (a commit with nothing outstanding arrives at once), so the release counts are fixed at two.
        const int w = warp;
        begin();
        uint32_t stage_n = 0, n_done = 0, n_mine = 0, t = 0;      // ring stages passed, items, items and steps of this warpgroup
        const int ks_head = P.D / 16;
        // Operand descriptors are built once and stepped by additions.
        const uint64_t d_q = umma_desc_sw128(smem_u32(sQ), 16, 1024);                       // K-major: + 32 bytes per 16 head dimensions
        const uint64_t d_k = umma_desc_sw128(smem_u32(sK), 16, 1024);
        const uint64_t d_v = umma_desc_sw128(smem_u32(sK + kTileBytes), kTileBytes, 1024);  // MN-major: + 2048 bytes per 16 keys
        const uint32_t tm_s = tmem + w * 256, tm_p = tm_s + 128, tm_o = tm_s + 192;
        const uint32_t idesc_o = umma_idesc_bf16(128, P.D, 0, 1);
        auto issue_scores = [&](uint64_t a, uint32_t st, int n_keys) {      // S_w = Q_w K^T, the key count rounded up to 16
            const uint64_t bdesc = umma_desc_advance(d_k, st * 2 * kTileBytes);
            const uint32_t idesc = umma_idesc_bf16(128, (n_keys + 15) & ~15, 0, 0);
            if (elect_one()) {
                tc_mma_bf16(tm_s, a, bdesc, idesc, 0u);
                tc_mma_bf16(tm_s, umma_desc_advance(a, 32), umma_desc_advance(bdesc, 32), idesc, 1u);
                if (ks_head > 2) {
                    tc_mma_bf16(tm_s, umma_desc_advance(a, 64), umma_desc_advance(bdesc, 64), idesc, 1u);
                    tc_mma_bf16(tm_s, umma_desc_advance(a, 96), umma_desc_advance(bdesc, 96), idesc, 1u);
                }
                tc_commit(bar_s + w);
            }
            __syncwarp();
        };
        auto issue_pv = [&](uint32_t st, int n_keys, uint32_t acc) {        // O_w (+)= P_w V
            const uint64_t bdesc = umma_desc_advance(d_v, st * 2 * kTileBytes);
            const int k_steps = (n_keys + 15) >> 4;
            if (elect_one()) {
                if (k_steps == 8) {                 // the usual case, straight-line
#pragma unroll
                    for (int ks = 0; ks < 8; ++ks)
                        tc_mma_bf16_ta(tm_o, tm_p + ks * 8, umma_desc_advance(bdesc, ks * 2048), idesc_o, ks > 0 ? 1u : acc);
                } else {
#pragma unroll 1
                    for (int ks = 0; ks < k_steps; ++ks)
                        tc_mma_bf16_ta(tm_o, tm_p + ks * 8, umma_desc_advance(bdesc, ks * 2048), idesc_o, ks > 0 ? 1u : acc);
                }
                tc_commit(bar_pv + w);
            }
            __syncwarp();
        };
        auto wait_full = [&](uint64_t* bar, uint32_t parity) {
            ok &= warp_wait_relaxed(bar, parity);
            if (!boxes) fence_proxy_async_smem();        // rows written by asynchronous copies are read by the tensor core
            tc_fence_after();
        };
#pragma unroll 1
        for (uint32_t i = 0; ok; ++i) {
            const Item it = item_at(i);
            if (it.n_act < 0) break;
            const uint32_t qb = n_done & 1;
            const int per_step = it.split ? it.n_act : 1;                // ring stages of a step
            if (w < it.n_act) {
                const uint64_t a = umma_desc_advance(d_q, (qb * kFwdTiles + w) * kTileBytes);
                const uint32_t mine = it.split ? w : 0;
                wait_full(bar_q_full + qb, (n_done >> 1) & 1);
                uint32_t sn = stage_n + mine;
                wait_full(bar_kv_full + sn % kFwdStages, (sn / kFwdStages) & 1);
                // The second tile starts a softmax later than the first: in step, both tiles' exponentials queue up and then both tiles'
                // hand-offs leave the special-function unit idle (3400 cycles a step of 128 keys against 2600).  Not worth its delay for a few steps.
                // (On a barrier of one phase: bar_p may have gone two phases on by the time this warp's first stage has landed, and its third waits for
                // a stage of the ring that this warp has yet to release.)
                if (i == 0 && w == 1 && it.n_kv >= 4) ok &= warp_wait_relaxed(bar_stagger, 0);
                issue_scores(a, sn % kFwdStages, min(kTile, it.n_sel));
                if (it.n_kv == 1) tc_commit_w(bar_q_free + qb);
#pragma unroll 1
                for (int j = 0; j < it.n_kv && ok; ++j, ++t) {
                    if (j + 1 < it.n_kv) {               // the next S, as soon as the warpgroup holds this one
                        const uint32_t s1 = sn + per_step;
                        wait_full(bar_kv_full + s1 % kFwdStages, (s1 / kFwdStages) & 1);
                        ok &= warp_wait_relaxed(bar_sfree + w, t & 1);
                        tc_fence_after();
                        issue_scores(a, s1 % kFwdStages, min(kTile, it.n_sel - (j + 1) * kTile));
                        if (j + 2 == it.n_kv) tc_commit_w(bar_q_free + qb);
                    }
                    ok &= warp_wait_relaxed(bar_p + w, t & 1);
                    if (t == 0 && w == 0 && lane == 0) mbar_arrive(bar_stagger);
                    if (j == 0 && n_mine > 0) ok &= warp_wait_relaxed(bar_ofree + w, (n_mine - 1) & 1);     // O of the previous item has been read
                    tc_fence_after();
                    issue_pv(sn % kFwdStages, min(kTile, it.n_sel - j * kTile), j > 0);
#pragma unroll 1
                    for (int x = 0; x < per_step; ++x) {                 // this step's stages: mine is read by the products above
                        const uint32_t so = stage_n + j * per_step + x;
                        if (x != static_cast<int>(mine)) ok &= warp_wait_relaxed(bar_kv_full + so % kFwdStages, (so / kFwdStages) & 1);
                        tc_commit_w(bar_kv_free + so % kFwdStages);
                    }
                    sn += per_step;
                }
                ++n_mine;
            } else {                                     // nothing to compute in this item: keep up with its barriers
                ok &= warp_wait_relaxed(bar_q_full + qb, (n_done >> 1) & 1);
                ok &= warp_wait_relaxed(bar_skip, (n_done - n_mine) & 1);      // its softmax warps are here too
                if (lane == 0) mbar_arrive(bar_skip + 1);
                tc_commit_w(bar_q_free + qb);
#pragma unroll 1
                for (int l = 0; l < it.n_kv * per_step && ok; ++l) {
                    const uint32_t so = stage_n + l;
                    ok &= warp_wait_relaxed(bar_kv_full + so % kFwdStages, (so / kFwdStages) & 1);
                    tc_commit_w(bar_kv_free + so % kFwdStages);
                }
            }
            stage_n += it.n_kv * per_step;
            ++n_done;
        }
    }
    } else if (warp < 8) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kFwdOtherRegs));
        // ---------------------------------------------------------------- O / l, rounded to bf16 ------------------
        // through a staging tile, so that whole 128-byte rows are written; a warp writes the rows it has staged
        const int r = tid & (kFwdGroupThreads - 1);
        const uint32_t lane_sel = static_cast<uint32_t>((warp & 3) * 32) << 16;
        uint32_t t0 = 0, t1 = 0, n0 = 0, n1 = 0;        // steps and items of the two softmax warpgroups so far
        const int c = r & 7, r0 = (r & ~31) + (lane >> 3);
        begin();
        load_first();
#pragma unroll 1
        for (uint32_t i = 0; ok; ++i) {
            const Item it = item_at(i);
            if (it.n_act < 0) break;
#pragma unroll 1
            for (int w = 0; w < it.n_act; ++w) {
                const uint32_t t_last = (w ? t1 : t0) + it.n_kv - 1, n_mine = w ? n1 : n0;
                const int qt = it.split ? it.qt : it.qt + w, h = it.split ? it.h + w : it.h;
                unsigned char* stage = sOut;
                ok &= warp_wait_relaxed(bar_l + w, n_mine & 1);
                ok &= warp_wait(bar_pv + w, t_last & 1);
                if (!ok) break;
                tc_fence_after();
                const float m_ref = s_ref[w * kTile + r], l_sum = s_sum[2 * w * kTile + r] + s_sum[(2 * w + 1) * kTile + r];
                const float inv_l = 1.f / l_sum;
                const int row = qt * kTile + r;
                unsigned char* rowp = stage + r * kRowBytes;
#pragma unroll 1
                for (int c16 = 0; c16 < P.D / 16; ++c16) {
                    float ov[16];
                    tmem_ld16(tmem + w * 256 + 192 + lane_sel + c16 * 16, ov);
                    tmem_ld_wait();
#pragma unroll
                    for (int q = 0; q < 2; ++q)
                        *reinterpret_cast<uint4*>(rowp + (((c16 * 2 + q) ^ (r & 7)) << 4)) =
                            make_uint4(pack_bf16(ov[8 * q + 0] * inv_l, ov[8 * q + 1] * inv_l), pack_bf16(ov[8 * q + 2] * inv_l, ov[8 * q + 3] * inv_l),
                                       pack_bf16(ov[8 * q + 4] * inv_l, ov[8 * q + 5] * inv_l), pack_bf16(ov[8 * q + 6] * inv_l, ov[8 * q + 7] * inv_l));
                }
                tc_fence_before();
                mbar_arrive(bar_ofree + w);                  // O, maximum and sum are in registers or in the staging tile
                if (row < it.n_sel) P.lse[(static_cast<size_t>(it.b) * P.H + h) * P.N + row] = (m_ref + log2f(l_sum)) * 0.6931471805599453f;
                __syncwarp();
                if (c * 8 < P.D) {
                    __nv_bfloat16* out = P.o + ((static_cast<size_t>(it.b) * P.N + qt * kTile + r0) * P.H + h) * P.D + c * 8;
                    const unsigned char* from = stage + r0 * kRowBytes;
                    const int left = it.n_sel - qt * kTile - r0;             // rows 4 apart, as long as they exist
#pragma unroll 1
                    for (int x = 0; x < 8; x += 4) {
                        uint4 v[4];
#pragma unroll
                        for (int u = 0; u < 4; ++u) v[u] = *reinterpret_cast<const uint4*>(from + (x + u) * 4 * kRowBytes + ((c ^ ((r0 + 4 * u) & 7)) << 4));
#pragma unroll
                        for (int u = 0; u < 4; ++u)
                            if ((x + u) * 4 < left) *reinterpret_cast<uint4*>(out + static_cast<size_t>(x + u) * 4 * P.H * P.D) = v[u];
                    }
                }
                __syncwarp();                                // its rows of the staging tile are free
            }
            t0 += it.n_kv; ++n0;
            if (it.n_act > 1) { t1 += it.n_kv; ++n1; }
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kFwdSoftmaxRegs));
        // ---------------------------------------------------------------- softmax --------------------------------
        const int w = (warp - 8) >> 3, half = ((warp - 8) >> 2) & 1;     // query tile of the item, 64-key half of a step
        const int r = tid & (kFwdGroupThreads - 1);     // query row inside the tile = tensor-memory lane
        const uint32_t lane_sel = static_cast<uint32_t>((warp & 3) * 32) << 16;
        const uint32_t tm_s = tmem + w * 256 + half * 64 + lane_sel, tm_p = tmem + w * 256 + 128 + half * 32 + lane_sel, tm_o = tmem + w * 256 + 192 + lane_sel;
        float* my_max = s_max + w * 4 * kTile + r;
        begin();
        load_first();
        uint32_t n_mine = 0, t = 0;                     // items and steps of this tile so far
#pragma unroll 1
        for (uint32_t i = 0; ok; ++i) {
            const Item it = item_at(i);
            if (it.n_act < 0) break;
            if (w >= it.n_act) {                        // nothing else ties the warps of a tile that an item lacks to the others' pace, and they wait by parity
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_skip);
                ok = warp_wait_relaxed(bar_skip + 1, (i - n_mine) & 1);
                continue;
            }
            if (half == 0) {
                const int qt = it.split ? it.qt : it.qt + w, h = it.split ? it.h + w : it.h;
                if (P.dq_acc) {     // the backward pass adds per-key-tile pieces of dQ' into the accumulator: clear this tile's rows
                    float4* rows = P.dq_acc + ((static_cast<size_t>(it.b) * P.Ncap + qt * kTile + (r >> 4)) * P.H + h) * (kDP / 4) + (r & 15);
#pragma unroll 1
                    for (int x = 0; x < kDP / 4; ++x, rows += static_cast<size_t>(kFwdGroupThreads / 16) * P.H * (kDP / 4))
                        *rows = make_float4(0.f, 0.f, 0.f, 0.f);         // 16 consecutive threads clear one 256-byte row
                }
            }
            float m_ref = -INFINITY, l_run = 0.f;       // exponentials are taken against m_ref (log2 domain), which trails the running maximum
            bool s_ready = false;                       // a poll's answer takes a hundred cycles: polls go out ahead of where they are needed
#pragma unroll 1
            for (int j = 0; j < it.n_kv; ++j, ++t) {
                if (!__all_sync(0xffffffffu, s_ready)) ok = warp_wait(bar_s + w, t & 1);
                if (!ok) break;
                tc_fence_after();
                const int valid = it.n_sel - j * kTile - half * 64;      // keys of this half that exist (may be none)
                float s[64];
                tmem_ld32(tm_s, s);
                tmem_ld32(tm_s + 32, s + 32);
                tmem_ld_wait();
                tc_fence_before();
                mbar_arrive(bar_sfree + w);              // S is in registers: the next one may be produced
                if (valid < 64) {                                     // ragged last step: keys past n_sel never win the max
#pragma unroll
                    for (int i = 0; i < 64; ++i)
                        if (i >= valid) s[i] = -INFINITY;
                }
                float mx[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) mx[i] = s[i];
#pragma unroll
                for (int i = 4; i < 60; i += 8) {                     // three-input maximum: two new values per instruction
#pragma unroll
                    for (int u = 0; u < 4; ++u) mx[u] = max3(mx[u], s[i + u], s[i + 4 + u]);
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) mx[u] = fmaxf(mx[u], s[60 + u]);
                // the other half's maximum of the row, through shared memory (arrays of the two step parities, so one barrier a step is enough)
                float* ex = my_max + (t & 1) * 2 * kTile;
                const float m_mine = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * P.scale_log2;
                ex[half * kTile] = m_mine;
                const bool pv_done = t == 0 || mbar_test(bar_pv + w, (t - 1) & 1);
                tile_sync(w);
                const float m_tile = fmaxf(m_mine, ex[(half ^ 1) * kTile]);
                if (j == 0) {
                    m_ref = first_reference(ex[0], m_tile);
                } else {
                    // O accumulates in tensor memory against m_ref.  It is rescaled only when a row's maximum has outgrown m_ref by
                    // 2^8 (probabilities then stay below 256, exact enough in bf16 and far from overflow); each half takes its
                    // share of the columns.
                    const bool grow = m_tile > m_ref + kRescaleStep;
                    if (__any_sync(0xffffffffu, grow)) {
                        ok = warp_wait(bar_pv + w, (t - 1) & 1);          // O of the previous step is complete
                        tc_fence_after();
                        const float alpha = grow ? fast_exp2(m_ref - m_tile) : 1.f;
                        if (grow) m_ref = m_tile;
                        l_run *= alpha;
#pragma unroll 1
                        for (int c = half * (P.D / 2); c < (half + 1) * (P.D / 2); c += 16) {     // sixteen columns at a time: the scores stay in registers
                            float ov[16];
                            tmem_ld16(tm_o + c, ov);
                            tmem_ld_wait();
#pragma unroll
                            for (int d = 0; d < 16; ++d) ov[d] *= alpha;
                            tmem_st16(tm_o + c, reinterpret_cast<const uint32_t*>(ov));
                        }
                    }
                }
                const uint64_t scale2 = pair_of(P.scale_log2, P.scale_log2), shift2 = pair_of(-m_ref, -m_ref);
                uint64_t l2[2] = {pair_of(0.f, 0.f), pair_of(0.f, 0.f)};          // four running sums: keys i = 0..3 mod 4
                uint32_t pk[32];
                // three batches of eight scores in flight: exponents of batch g, exponentials of batch g - 1, sums and rounding of batch g - 2
#pragma unroll
                for (int g = 0; g < 10; ++g) {
                    if (g < 8) {
#pragma unroll
                        for (int i = 8 * g; i < 8 * g + 8; i += 2) halves_of(fma_pair(pair_of(s[i], s[i + 1]), scale2, shift2), s[i], s[i + 1]);
                    }
                    if (g >= 1 && g < 9) {
#pragma unroll
                        for (int i = 8 * g - 8; i < 8 * g; ++i) s[i] = fast_exp2(s[i]);       // exp2(-inf) = 0 for the masked keys
                    }
                    if (g >= 2) {
#pragma unroll
                        for (int i = 8 * g - 16; i < 8 * g - 8; i += 2) {
                            l2[(i >> 1) & 1] = add_pair(l2[(i >> 1) & 1], pair_of(s[i], s[i + 1]));
                            pk[i >> 1] = pack_bf16(s[i], s[i + 1]);
                        }
                    }
                }
                if (!__all_sync(0xffffffffu, pv_done)) ok &= warp_wait(bar_pv + w, (t - 1) & 1);      // P V of the previous step has read P
                tc_fence_after();
                s_ready = mbar_test(bar_s + w, (t + 1) & 1);
                tmem_st32(tm_p, pk);                                  // keys 2 c and 2 c + 1 in column c
                {
                    float a0, a1, a2, a3;
                    halves_of(l2[0], a0, a1);
                    halves_of(l2[1], a2, a3);
                    l_run += (a0 + a1) + (a2 + a3);
                }
                tmem_st_wait();
                tc_fence_before();
                mbar_arrive(bar_p + w);
                if (!ok) break;
            }
            if (!ok) break;
            if (n_mine > 0) ok = warp_wait(bar_ofree + w, (n_mine - 1) & 1);         // the previous item's have been read
            if (half == 0) s_ref[w * kTile + r] = m_ref;
            s_sum[(2 * w + half) * kTile + r] = l_run;
            mbar_arrive(bar_l + w);
            ++n_mine;
        }
    }

    if (!ok) {
        set_status(P.status, VARDROP_ERR_TIMEOUT);
        // A softmax warp whose wait gave up has left by itself, and nothing bounds a named barrier: it arrives once more in passing.  The others reach
        // at most one more: the scores of the step behind that one wait for this warp's arrivals too.
        if (warp >= 8) tile_arrive((warp - 8) >> 3);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, kFwdTmemCols);
}

// ---------------------------------------------------------------------------------------------------------
// forward, few tiles
// ---------------------------------------------------------------------------------------------------------
// With one or two tiles per head and instance the step is a chain of latencies (kept count, row indices, rows, scores, softmax, P V,
// rows out), each a few hundred cycles, and every path runs once or twice, at the speed of instruction fetch.  So: no roles and no
// hand-offs but __syncthreads, rolled loops over 32 scores (the scores stay in tensor memory and are read twice), one stage, 48 KB
// and 128 columns a CTA, so that four CTAs share an SM and fill each other's waits.
// B = 32, H = 8, D = 64: 119 kept 7.1 us back to back (10 in the persistent kernel of the first form), 200 kept 15.3 us without a gather
// launch (19 and a gather of 16).
// Tensor memory: S 128; P (bf16) over S's columns 0 .. 63 as they are consumed, P V into columns 64 .. 127.
constexpr int kTileFwdThreads = 128;
constexpr uint32_t kTileFwdTmemCols = 128;
constexpr int kTileFwdSmemBytes = 1024 /*alignment*/ + 3 * kTileBytes /*Q, K, V*/;
constexpr int kTileFwdPerSm = 4;

// kLag: more than two tiles without a selection, where a row's reference maximum is that of its first 64 keys until the running maximum has outgrown
// it by 2^8; O then goes back to tensor memory for the next P V to add to; and the next key tile's K comes in under the softmax, its V under the step
// after (all of 321 variates, B = 32: 28.2 -> 27.6 us back to back).  Otherwise it is the running maximum over whole key tiles, and the tiles' parts
// of O are added up in registers; a second tile's rows come when the first is done (under its softmax, the code of it cost calls of one and
// two tiles 1 to 4 %: 128 variates, B = 32 5.98 -> 6.15, 555 of 1500 kept, B = 32 65.6 -> 66.8).
template <bool kLag>
__global__ void __launch_bounds__(kTileFwdThreads, kTileFwdPerSm) attn_fwd_tile_kernel(const FwdParams P) {
    extern __shared__ unsigned char smem_dyn[];
    __shared__ uint64_t bar_s, bar_o;
    __shared__ uint32_t tmem_slot;
    unsigned char* sQ = align_tiles(smem_dyn);
    unsigned char* sK = sQ + kTileBytes;
    unsigned char* sV = sK + kTileBytes;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (warp == 0) {
        tmem_alloc(&tmem_slot, kTileFwdTmemCols);
        tmem_relinquish();
    }
    if (tid == 0) {
        mbar_init(&bar_s, 1);
        mbar_init(&bar_o, 1);
        mbar_fence_init();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot, tm = tmem + (static_cast<uint32_t>(warp * 32) << 16);
    const uint32_t idesc_o = umma_idesc_bf16(128, P.D, 0, 1);
    const uint64_t d_q = umma_desc_sw128(smem_u32(sQ), 16, 1024), d_k = umma_desc_sw128(smem_u32(sK), 16, 1024);
    const uint64_t d_v = umma_desc_sw128(smem_u32(sV), kTileBytes, 1024);
    const uint64_t scale2 = pair_of(P.scale_log2, P.scale_log2);
    chain_wait();
    chain_release();
    if (blockIdx.x == 0 && tid == 0) P.status[kWsPairingWord] = 1;      // this workspace now holds a forward pass that no backward pass has consumed
    const int kept = largest_kept(P.n_sel, P.S, P.N);
    const int n_t = (kept + kTile - 1) / kTile, n_items = n_t * P.H * P.B;
    bool ok = true;
    uint32_t t = 0;                                     // key tiles of this CTA so far: parity of bar_s and bar_o

#pragma unroll 1
    for (int item = blockIdx.x; item < n_items; item += gridDim.x) {
        const int hb = small_div(item, n_t), qt = item - hb * n_t, b = small_div(hb, P.H), h = hb - b * P.H;
        const int n_sel = P.S > 1 ? P.n_sel[b] : kept, n_kv = (n_sel + kTile - 1) / kTile;
        if (qt >= n_kv) continue;
        const int32_t* idx = P.sel_idx ? P.sel_idx + static_cast<size_t>(P.S > 1 ? b : 0) * P.N : nullptr;
        const long long base = b * P.sB + h * P.sH;
        if (qt == 0 && tid == 0) P.tile_done[b * P.H + h] = 0;
        if ((n_kv > 2 || (n_kv == 2 && P.S > 1)) && P.dq_acc) {             // the backward pass adds per-key-tile pieces of dQ' into the accumulator (it completes dQ of two tiles in place, if no instance has more): clear this tile's rows
            float4* rows = P.dq_acc + ((static_cast<size_t>(b) * P.Ncap + qt * kTile + (tid >> 4)) * P.H + h) * (kDP / 4) + (tid & 15);
#pragma unroll 1
            for (int x = 0; x < kDP / 4; ++x, rows += static_cast<size_t>(kTileFwdThreads / 16) * P.H * (kDP / 4))
                *rows = make_float4(0.f, 0.f, 0.f, 0.f);                 // 16 consecutive threads clear one 256-byte row
        }
        // every warp copies its 32 rows of a tile
        auto load_rows = [&](unsigned char* tile, const __nv_bfloat16* from, int t0) {
            copy_32_rows(tile + warp * 32 * kRowBytes, from + base, P.sN, idx, t0 * kTile + warp * 32, n_sel, P.D);
        };
        load_rows(sQ, P.q, qt);
        load_rows(sK, P.k, 0);
        asm volatile("cp.async.commit_group;" ::: "memory");
        load_rows(sV, P.v, 0);
        asm volatile("cp.async.commit_group;" ::: "memory");
        float o_acc[kDP];                                // more than one key tile: the sum over the tiles before the current one
        float m_run = -INFINITY, l_run = 0.f;
#pragma unroll 1
        for (int j = 0; j < n_kv; ++j, ++t) {
            const int n_keys = min(kTile, n_sel - j * kTile);
            if (!kLag && j > 0) {
#pragma unroll 1
                for (int x = 1; x < 3; ++x) {            // K, V
                    load_rows(sQ + x * kTileBytes, x == 1 ? P.k : P.v, j);
                    asm volatile("cp.async.commit_group;" ::: "memory");
                }
            }
            asm volatile("cp.async.wait_group 1;" ::: "memory");         // Q and K have landed
            fence_proxy_async_smem();
            tc_fence_before();
            __syncthreads();
            if (warp == 0) {
                tc_fence_after();
                if (elect_one()) {
                    const uint32_t idesc = umma_idesc_bf16(128, (n_keys + 15) & ~15, 0, 0);
#pragma unroll 1
                    for (int ks = 0; ks < P.D / 16; ++ks)
                        tc_mma_bf16(tmem, umma_desc_advance(d_q, ks * 32), umma_desc_advance(d_k, ks * 32), idesc, ks > 0);
                    tc_commit(&bar_s);
                }
                __syncwarp();
            }
            ok &= mbar_wait(&bar_s, t & 1);
            tc_fence_after();
            const bool more = kLag && j + 1 < n_kv;
            if (more) {                                  // K has been read: the next one comes in under the softmax
                load_rows(sK, P.k, j + 1);
                asm volatile("cp.async.commit_group;" ::: "memory");
            }
            // ---- row maximum, 32 scores at a time ----
            float m_first = -INFINITY, m_tile = -INFINITY;           // kLag: of the first 64 keys of the tile, of the others
#pragma unroll 1
            for (int c = 0; c < n_keys; c += 32) {
                float s[32];
                if (kLag && c == 64) { m_first = m_tile; m_tile = -INFINITY; }
                tmem_ld32(tm + c, s);
                tmem_ld_wait();
                if (n_keys - c < 32) {                                // ragged end: keys past n_sel never win the maximum
#pragma unroll
                    for (int i = 0; i < 32; ++i)
                        if (c + i >= n_keys) s[i] = -INFINITY;
                }
                float mx[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) mx[u] = s[u];
#pragma unroll
                for (int i = 4; i < 28; i += 8) {
#pragma unroll
                    for (int u = 0; u < 4; ++u) mx[u] = max3(mx[u], s[i + u], s[i + 4 + u]);
                }
                m_tile = max3(m_tile, max3(mx[0], s[28], mx[1]), max3(max3(s[29], mx[2], s[30]), mx[3], s[31]));
            }
            float m_new, alpha;
            if (kLag) {
                if (n_keys <= 64) { m_first = m_tile; m_tile = -INFINITY; }
                m_new = first_reference(j == 0 ? m_first * P.scale_log2 : first_reference(m_run, m_first * P.scale_log2), m_tile * P.scale_log2);
                alpha = m_new == m_run ? 1.f : fast_exp2(m_run - m_new);
                l_run *= alpha;
            } else {
                m_new = fmaxf(m_run, m_tile * P.scale_log2);
                alpha = fast_exp2(m_run - m_new);
            }
            m_run = m_new;
            // ---- P = exp2(S scale - maximum), rounded to bf16, over the columns of S that have been read ----
            const uint64_t shift2 = pair_of(-m_new, -m_new);
            uint64_t l2[2] = {pair_of(0.f, 0.f), pair_of(0.f, 0.f)};
            auto l_sum = [&]() {
                float a0, a1, a2, a3;
                halves_of(l2[0], a0, a1);
                halves_of(l2[1], a2, a3);
                return (a0 + a1) + (a2 + a3);
            };
#pragma unroll 1
            for (int c = 0; c < n_keys; c += 32) {
                float s[32];
                uint32_t pk[16];
                if (kLag && c == 64) {                   // 64 keys a sum
                    l_run += l_sum();
                    l2[0] = l2[1] = pair_of(0.f, 0.f);
                }
                tmem_ld32(tm + c, s);
                tmem_ld_wait();
                if (n_keys - c < 32) {
#pragma unroll
                    for (int i = 0; i < 32; ++i)
                        if (c + i >= n_keys) s[i] = -INFINITY;
                }
#pragma unroll
                for (int g = 0; g < 6; ++g) {            // batches of eight: exponents of g, exponentials of g - 1, sums and rounding of g - 2
                    if (g < 4) {
#pragma unroll
                        for (int i = 8 * g; i < 8 * g + 8; i += 2) halves_of(fma_pair(pair_of(s[i], s[i + 1]), scale2, shift2), s[i], s[i + 1]);
                    }
                    if (g >= 1 && g < 5) {
#pragma unroll
                        for (int i = 8 * g - 8; i < 8 * g; ++i) s[i] = fast_exp2(s[i]);       // exp2(-inf) = 0 for the masked keys
                    }
                    if (g >= 2) {
#pragma unroll
                        for (int i = 8 * g - 16; i < 8 * g - 8; i += 2) {
                            l2[(i >> 1) & 1] = add_pair(l2[(i >> 1) & 1], pair_of(s[i], s[i + 1]));
                            pk[i >> 1] = pack_bf16(s[i], s[i + 1]);
                        }
                    }
                }
                tmem_st16(tm + (c >> 1), pk);            // keys 2 c' and 2 c' + 1 in column c'
            }
            if (kLag) {
                l_run += l_sum();
                if (j > 0) {                             // O so far, for P V to add to
                    if (__any_sync(0xffffffffu, alpha != 1.f)) {
#pragma unroll
                        for (int d = 0; d < kDP; ++d) o_acc[d] *= alpha;
                    }
                    tmem_st32(tm + 64, reinterpret_cast<const uint32_t*>(o_acc));
                    if (P.D > 32) tmem_st32(tm + 96, reinterpret_cast<const uint32_t*>(o_acc + 32));
                }
            } else {
                l_run = l_run * alpha + l_sum();
            }
            if (more) asm volatile("cp.async.wait_group 1;" ::: "memory");         // V has landed
            else asm volatile("cp.async.wait_group 0;" ::: "memory");
            fence_proxy_async_smem();
            tmem_st_wait();
            tc_fence_before();
            ok = __syncthreads_and(ok);
            if (!ok) { item = n_items; break; }          // a wait gave up somewhere in the CTA: stop
            if (warp == 0) {
                tc_fence_after();
                if (elect_one()) {
#pragma unroll 1
                    for (int ks = 0; ks < (n_keys + 15) >> 4; ++ks)
                        tc_mma_bf16_ta(tmem + 64, tmem + ks * 8, umma_desc_advance(d_v, ks * 2048), idesc_o, (kLag && j > 0) || ks > 0);
                    tc_commit(&bar_o);
                }
                __syncwarp();
            }
            ok &= mbar_wait(&bar_o, t & 1);              // (agreed on at the next such barrier: no thread leaves by itself)
            tc_fence_after();
            if (more) {                                  // and V
                load_rows(sV, P.v, j + 1);
                asm volatile("cp.async.commit_group;" ::: "memory");
            }
            if (kLag ? j + 1 < n_kv : n_kv > 1) {
                if (kLag || j == 0) {
                    tmem_ld32(tm + 64, o_acc);
                    if (P.D > 32) tmem_ld32(tm + 96, o_acc + 32);
                    tmem_ld_wait();
                } else {
                    const uint64_t alpha2 = pair_of(alpha, alpha);
#pragma unroll
                    for (int c = 0; c < kDP; c += 32) {
                        if (c < P.D) {
                            float ov[32];
                            tmem_ld32(tm + 64 + c, ov);
                            tmem_ld_wait();
#pragma unroll
                            for (int d = 0; d < 32; d += 2)          // rescale and add in one step
                                halves_of(fma_pair(pair_of(o_acc[c + d], o_acc[c + d + 1]), alpha2, pair_of(ov[d], ov[d + 1])), o_acc[c + d], o_acc[c + d + 1]);
                        }
                    }
                    if (j + 1 == n_kv) {                 // back where a single tile leaves it
                        tmem_st32(tm + 64, reinterpret_cast<const uint32_t*>(o_acc));
                        if (P.D > 32) tmem_st32(tm + 96, reinterpret_cast<const uint32_t*>(o_acc + 32));
                        tmem_st_wait();
                    }
                }
            }
            tc_fence_before();
            if (j + 1 < n_kv) __syncthreads();           // the next step's S goes over these columns
        }
        if (item == n_items) break;
        // ---- O / l, rounded to bf16, through Q's tile so that whole rows are written ----
        {
            const float inv_l = 1.f / l_run;
            unsigned char* rowp = sQ + tid * kRowBytes;
            const int row = qt * kTile + tid;
            if (row < n_sel) P.lse[(static_cast<size_t>(b) * P.H + h) * P.N + row] = (m_run + log2f(l_run)) * 0.6931471805599453f;
#pragma unroll 1
            for (int c16 = 0; c16 < P.D / 16; ++c16) {
                float ov[16];
                tmem_ld16(tm + 64 + c16 * 16, ov);
                tmem_ld_wait();
#pragma unroll
                for (int q = 0; q < 2; ++q)
                    *reinterpret_cast<uint4*>(rowp + (((c16 * 2 + q) ^ (tid & 7)) << 4)) =
                        make_uint4(pack_bf16(ov[8 * q + 0] * inv_l, ov[8 * q + 1] * inv_l), pack_bf16(ov[8 * q + 2] * inv_l, ov[8 * q + 3] * inv_l),
                                   pack_bf16(ov[8 * q + 4] * inv_l, ov[8 * q + 5] * inv_l), pack_bf16(ov[8 * q + 6] * inv_l, ov[8 * q + 7] * inv_l));
            }
            tc_fence_before();
            __syncwarp();                                // a warp writes the rows it has staged
            const int c = lane & 7, r0 = warp * 32 + (lane >> 3);
            if (c * 8 < P.D) {
                __nv_bfloat16* out = P.o + ((static_cast<size_t>(b) * P.N + qt * kTile + r0) * P.H + h) * P.D + c * 8;
                const unsigned char* from = sQ + r0 * kRowBytes + ((c ^ (r0 & 7)) << 4);
                const unsigned char* from4 = sQ + (r0 + 4) * kRowBytes + ((c ^ ((r0 + 4) & 7)) << 4);
                const int left = min(32 - (lane >> 3), n_sel - qt * kTile - r0);
                const size_t step = static_cast<size_t>(4) * P.H * P.D;
#pragma unroll 1
                for (int x = 0; x < left; x += 8, out += 2 * step, from += 8 * kRowBytes, from4 += 8 * kRowBytes) {     // rows 4 apart
                    const uint4 v0 = *reinterpret_cast<const uint4*>(from), v1 = *reinterpret_cast<const uint4*>(from4);
                    *reinterpret_cast<uint4*>(out) = v0;
                    if (x + 4 < left) *reinterpret_cast<uint4*>(out + step) = v1;
                }
            }
            __syncthreads();                             // Q's tile is free for the next item
        }
    }
    if (!ok) set_status(P.status, VARDROP_ERR_TIMEOUT);
    asm volatile("cp.async.wait_all;" ::: "memory");
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, kTileFwdTmemCols);
}

}  // namespace

// Which kernel: with a selection as the backward pass (see attn_many_tiles).  Without one, up to three tiles: all of 384 variates take 10.4 us against 12.4 at B = 4 (27.9 and 27.2 at B = 32); at four it turns.
static bool attn_fwd_few_tiles(const vardrop_attn_cfg& c, const int32_t* sel_idx) { return sel_idx ? !attn_many_tiles(c, sel_idx) : c.N <= 3 * kTile; }

int attn_fwd_launch(const void* q, const void* k, const void* v, const int32_t* sel_idx, const int32_t* n_sel,
                    const vardrop_attn_cfg& c, void* o, float* lse, void* ws, cudaStream_t stream) {
    const AttnWs w = attn_layout(c);
    const QkvLayout L = qkv_layout(c);
    char* base = static_cast<char*>(ws);
    const bool few = attn_fwd_few_tiles(c, sel_idx);
    CUtensorMap mq{}, mk{}, mv{};
    if (!sel_idx && !few) {
        if (int st = make_tile_map(&mq, q, c.D, c.B, c.N, c.H, L.sB, L.sN, L.sH)) return st;
        if (int st = make_tile_map(&mk, k, c.D, c.B, c.N, c.H, L.sB, L.sN, L.sH)) return st;
        if (int st = make_tile_map(&mv, v, c.D, c.B, c.N, c.H, L.sB, L.sN, L.sH)) return st;
    }
    FwdParams P{};
    P.q = static_cast<const __nv_bfloat16*>(q); P.k = static_cast<const __nv_bfloat16*>(k); P.v = static_cast<const __nv_bfloat16*>(v);
    P.o = static_cast<__nv_bfloat16*>(o); P.lse = lse; P.sel_idx = sel_idx; P.n_sel = sel_idx ? n_sel : nullptr;
    P.status = reinterpret_cast<int*>(base);
    P.dq_acc = attn_fwd_clears(c, sel_idx) ? reinterpret_cast<float4*>(base + w.dq_acc) : nullptr;
    P.tile_done = reinterpret_cast<int32_t*>(base + w.delta);
    P.sB = L.sB; P.sN = L.sN; P.sH = L.sH;
    P.B = c.B; P.N = c.N; P.Ncap = w.Ncap; P.H = c.H; P.D = c.D; P.S = attn_sel_rows(c, sel_idx);
    const float scale = c.sm_scale > 0.f ? c.sm_scale : 1.f / sqrtf(static_cast<float>(c.D));
    P.scale_log2 = scale * 1.4426950408889634f;
    static thread_local int attr_dev = -1;
    int dev = 0;
    cudaGetDevice(&dev);
    if (attr_dev != dev) {
        if (int st = check_cuda(cudaFuncSetAttribute(attn_fwd_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kFwdSmemBytes), "attention: smem attribute")) return st;
        for (auto kernel : {attn_fwd_tile_kernel<false>, attn_fwd_tile_kernel<true>})
            if (int st = check_cuda(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kTileFwdSmemBytes), "attention: smem attribute")) return st;
        attr_dev = dev;
    }
    const int n_t = w.Ncap / kTile;
    LaunchScope ls_(K_ATTN_FWD, stream);
    if (few) {
        const long long worst = static_cast<long long>(n_t) * c.H * c.B, cap = static_cast<long long>(kTileFwdPerSm) * sm_count();
        const bool lag = !sel_idx && c.N > 2 * kTile;
        return check_cuda(launch_chained(lag ? attn_fwd_tile_kernel<true> : attn_fwd_tile_kernel<false>, dim3(static_cast<unsigned>(worst < cap ? worst : cap)), dim3(kTileFwdThreads), kTileFwdSmemBytes, stream, P),
                          "attention: forward launch");
    }
    const long long worst = (static_cast<long long>(n_t / 2) * c.H + (n_t & 1 ? (c.H + 1) / 2 : 0)) * c.B;
    const long long most = worst > static_cast<long long>((c.H + 1) / 2) * c.B ? worst : static_cast<long long>((c.H + 1) / 2) * c.B;
    const int grid = static_cast<int>(most < sm_count() ? most : sm_count());                 // one CTA per SM
    return check_cuda(launch_chained(attn_fwd_kernel, dim3(grid), dim3(kFwdThreads), kFwdSmemBytes, stream, mq, mk, mv, P), "attention: forward launch");
}

}  // namespace vardrop
