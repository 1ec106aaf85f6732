// Variate redundancy of a batch (Appendix A, Eq. 4): for every instance and variate, the largest Pearson correlation
// coefficient with any other variate of the same window, and how many variates exceed a threshold (Sec. 1 quotes the
// share above 0.9).  This is the O(N^2 T) similarity the paper argues against computing per batch; here it checks how
// redundant a workload is.
//
// pearson_normalize_kernel   one warp per (instance, variate): mean and centred norm in fp32, then the unit vector
//                            z = (x - mean) / |x - mean| is stored as two bf16 terms, z = hi + lo (16 mantissa bits).
// pearson_max_kernel         persistent, one CTA per SM: rho = z_v . z_w is a dense contraction, so it runs on the tcgen05 tensor cores (hi hi +
//                            hi lo + lo hi, fp32 accumulator in tensor memory) in units of 128 x 256 variates of an instance.
#include "attn_common.cuh"

namespace vardrop {

namespace {

struct PearsonParams {
    const float* x;          // [B, N, L]
    __nv_bfloat16* z_hi;     // [B, N, Lrow]
    __nv_bfloat16* z_lo;
    float* max_rho;          // [B, N]
    int32_t* n_above;        // [B]
    int32_t* done;           // [B] units of an instance that are in max_rho
    int* status;
    int B, N, L, Lrow;
    float threshold;
};

// What bounds it is memory (each window read once, two bf16 terms written): rows of up to 1024 steps stay in registers between the mean, the
// norm and the division.  B = 32, N = 862, L = 96: 10.8 us, 18.8 with three passes over a row and zero padding written (events around the
// launch).
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}
__device__ __forceinline__ void split_bf16(float z, __nv_bfloat16& hi, __nv_bfloat16& lo) {
    hi = __float2bfloat16_rn(z);
    lo = __float2bfloat16_rn(z - __bfloat162float(hi));
}
// kQuads 16-byte pieces a lane and row; 0: rows of any length and alignment, read three times.  Several short rows a warp, so that enough loads
// are in flight.
template <int kQuads>
struct NormalizeRows { static constexpr int value = kQuads == 0 || kQuads == 8 ? 1 : kQuads == 4 ? 2 : 4; };
template <int kQuads>
__global__ void __launch_bounds__(256) pearson_normalize_kernel(const PearsonParams P) {
    chain_wait();
    chain_release();
    constexpr int kRows = NormalizeRows<kQuads>::value;
    const int b = blockIdx.y, lane = threadIdx.x & 31;
    const int n0 = (blockIdx.x * 8 + (threadIdx.x >> 5)) * kRows;
    if (blockIdx.x == 0 && threadIdx.x == 0) { P.n_above[b] = 0; P.done[b] = 0; }
    if (n0 >= P.N) return;
    const size_t r0 = static_cast<size_t>(b) * P.N + n0;
    const int rows = min(kRows, P.N - n0);
    if (lane < rows) P.max_rho[r0 + lane] = -2.f;
    if constexpr (kQuads > 0) {
        const int quads = P.L >> 2;
        float4 v[kRows][kQuads];
        float s[kRows], ss[kRows];
#pragma unroll
        for (int r = 0; r < kRows; ++r) {
#pragma unroll
            for (int i = 0; i < kQuads; ++i)
                v[r][i] = r < rows && lane + 32 * i < quads ? __ldg(reinterpret_cast<const float4*>(P.x + (r0 + r) * P.L) + lane + 32 * i) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int r = 0; r < kRows; ++r) {
            s[r] = 0.f;
#pragma unroll
            for (int i = 0; i < kQuads; ++i) s[r] += (v[r][i].x + v[r][i].y) + (v[r][i].z + v[r][i].w);
        }
#pragma unroll
        for (int r = 0; r < kRows; ++r) s[r] = warp_sum(s[r]);
#pragma unroll
        for (int r = 0; r < kRows; ++r) {
            const float mean = s[r] / static_cast<float>(P.L);
            ss[r] = 0.f;
#pragma unroll
            for (int i = 0; i < kQuads; ++i) {
                if (lane + 32 * i < quads) {
                    float4& q = v[r][i];
                    q.x -= mean; q.y -= mean; q.z -= mean; q.w -= mean;
                    ss[r] += (q.x * q.x + q.y * q.y) + (q.z * q.z + q.w * q.w);
                }
            }
        }
#pragma unroll
        for (int r = 0; r < kRows; ++r) ss[r] = warp_sum(ss[r]);
#pragma unroll
        for (int r = 0; r < kRows; ++r) {
            if (r >= rows) break;
            if (!isfinite(ss[r]) && lane == 0) set_status(P.status, VARDROP_ERR_NONFINITE);
            const float inv = ss[r] > 0.f ? 1.f / sqrtf(ss[r]) : 0.f;    // a constant variate correlates 0 with everything
#pragma unroll
            for (int i = 0; i < kQuads; ++i) {
                if (lane + 32 * i < quads) {
                    __nv_bfloat16 h[4], l[4];
                    split_bf16(v[r][i].x * inv, h[0], l[0]);
                    split_bf16(v[r][i].y * inv, h[1], l[1]);
                    split_bf16(v[r][i].z * inv, h[2], l[2]);
                    split_bf16(v[r][i].w * inv, h[3], l[3]);
                    reinterpret_cast<uint2*>(P.z_hi + (r0 + r) * P.Lrow)[lane + 32 * i] = *reinterpret_cast<const uint2*>(h);
                    reinterpret_cast<uint2*>(P.z_lo + (r0 + r) * P.Lrow)[lane + 32 * i] = *reinterpret_cast<const uint2*>(l);
                }
            }
        }
    } else {
        __nv_bfloat16* hi = P.z_hi + r0 * P.Lrow;
        __nv_bfloat16* lo = P.z_lo + r0 * P.Lrow;
        const float* row = P.x + r0 * P.L;
        float s = 0.f, ss = 0.f;
        for (int t = lane; t < P.L; t += 32) s += row[t];
        const float mean = warp_sum(s) / static_cast<float>(P.L);
        for (int t = lane; t < P.L; t += 32) {
            const float d = row[t] - mean;
            ss = fmaf(d, d, ss);
        }
        ss = warp_sum(ss);
        if (!isfinite(ss) && lane == 0) set_status(P.status, VARDROP_ERR_NONFINITE);
        const float inv = ss > 0.f ? 1.f / sqrtf(ss) : 0.f;
        for (int t = lane; t < P.L; t += 32) split_bf16((row[t] - mean) * inv, hi[t], lo[t]);
    }
}

// A unit is a 128-variate row tile against a 256-variate column tile of an instance, all time steps; the CTAs take equal runs of units in the
// order (instance, column tile, row tile), so that they finish together.  Windows of up to 128 steps (two chunks of 64) keep the column tile,
// two thirds of the operands, in shared memory from unit to unit.
//   warp 0        loads: rings of two row-tile chunks and two column-tile chunks, hi and lo, by the copy engine, zeros outside
//   warp 1        products: 3 x 4 of M = 128, N = 256 (fewer at the edges) a chunk, into one of two accumulators
//   warps 4-11    maxima of a finished unit under the products of the next, to max_rho by atomics; whoever brings the last unit of an instance
//                 counts the variates above the threshold
// What bounds it is the tensor core (three executed products per algorithmic one, the price of 1e-4 accuracy from a bf16 pipe).
// B = 32, N = 862, L = 96: 24 us, 43.5 with one CTA per row tile and operands through registers (events around the launch).
constexpr int kPearsonThreads = 384;
constexpr int kColTile = 256;
constexpr int kPearsonSlots = 2;                                  // of either ring (a third row-tile slot changed nothing)
constexpr int kPearsonRowBytes = 2 * kTileBytes, kPearsonColBytes = 4 * kTileBytes;      // a chunk of a row tile (hi, lo), of a column tile (hi 2, lo 2)
constexpr int kPearsonSmemBytes = 1024 + kPearsonSlots * (kPearsonRowBytes + kPearsonColBytes);
constexpr uint32_t kPearsonTmemCols = 512;

__device__ __forceinline__ void atomic_max_float(float* at, float v) {
    v += 0.f;                                                     // -0 orders as an integer below every negative number
    if (v >= 0.f) atomicMax(reinterpret_cast<int*>(at), __float_as_int(v));
    else atomicMin(reinterpret_cast<unsigned int*>(at), __float_as_uint(v));
}
__device__ __forceinline__ bool epilogue_sync_and(bool ok) {
    uint32_t r;
    asm volatile(
        "{\n.reg .pred p, q;\n"
        "setp.ne.b32 q, %1, 0;\n"
        "bar.red.and.pred p, 1, 256, q;\n"
        "selp.u32 %0, 1, 0, p;\n}"
        : "=r"(r)
        : "r"(static_cast<uint32_t>(ok))
        : "memory");
    return r != 0;
}

__global__ void __launch_bounds__(kPearsonThreads, 1) pearson_max_kernel(const __grid_constant__ CUtensorMap map_hi, const __grid_constant__ CUtensorMap map_lo,
                                                                         const PearsonParams P) {
    extern __shared__ unsigned char smem_dyn[];
    uint64_t* bar_full = reinterpret_cast<uint64_t*>(smem_dyn);      // [2] the step's tiles are there
    uint64_t* bar_free = bar_full + 2;                               // [2] its products are done
    uint64_t* bar_acc = bar_free + 2;                                // [2] accumulator of a unit complete
    uint64_t* bar_accfree = bar_acc + 2;                             // [2] and read (8 warps)
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bar_accfree + 2);
    int* s_last = reinterpret_cast<int*>(tmem_slot + 1);
    unsigned char* tiles = align_tiles(smem_dyn + 128);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tiles + kPearsonSlots * (kPearsonRowBytes + kPearsonColBytes) > smem_dyn + kPearsonSmemBytes) {    // dynamic shared memory base not 1024-byte aligned
        chain_wait();
        if (tid == 0) set_status(P.status, VARDROP_ERR_CUDA);
        return;
    }
    if (warp == 0) {
        tmem_alloc(tmem_slot, kPearsonTmemCols);
        tmem_relinquish();
    }
    if (tid == 0) {
        for (int i = 0; i < 2; ++i) {
            mbar_init(bar_full + i, 1);
            mbar_init(bar_free + i, 1);
            mbar_init(bar_acc + i, 1);
            mbar_init(bar_accfree + i, 8);
        }
        mbar_fence_init();
        tma_prefetch_desc(&map_hi);
        tma_prefetch_desc(&map_lo);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    chain_wait();
    chain_release();

    const int row_tiles = (P.N + kTile - 1) / kTile, col_tiles = (P.N + kColTile - 1) / kColTile, n_chunks = (P.L + 63) / 64;
    const long long units = static_cast<long long>(P.B) * row_tiles * col_tiles;
    const long long u0 = units * blockIdx.x / gridDim.x, u1 = units * (blockIdx.x + 1) / gridDim.x;
    struct Unit { long long group; int b, ti, tj, cols; };           // group: (instance, column tile)
    const bool resident = n_chunks <= 2;
    // where chunk kc of the unit's column tile lies (the ring slot of the step, where it does not stay)
    auto col_slot = [&](const Unit& x, int kc, uint32_t step) { return !resident ? step & 1 : n_chunks == 2 ? static_cast<uint32_t>(kc) : static_cast<uint32_t>(x.group) & 1; };
    auto unit_at = [&](long long u) {
        Unit x;
        x.group = u / row_tiles;
        x.ti = static_cast<int>(u - x.group * row_tiles);
        x.b = static_cast<int>(x.group / col_tiles);
        x.tj = static_cast<int>(x.group - static_cast<long long>(x.b) * col_tiles);
        x.cols = min(kColTile, P.N - x.tj * kColTile);
        return x;
    };
    bool ok = true;
    if (warp == 0) {
        if (lane == 0) {
            uint32_t step = 0;
#pragma unroll 1
            for (long long u = u0; u < u1 && ok; ++u) {
                const Unit x = unit_at(u);
                const int halves = x.cols > kTile ? 2 : 1;
#pragma unroll 1
                for (int kc = 0; kc < n_chunks; ++kc, ++step) {
                    const uint32_t st = step & 1;
                    const bool bring = !resident || u == u0 || x.ti == 0;        // the column tile changes with the first row tile
                    ok = mbar_wait_relaxed(bar_free + st, ((step >> 1) & 1) ^ 1);     // two steps ago: the last to read either place
                    if (!ok) break;
                    unsigned char* rows = tiles + st * kPearsonRowBytes;
                    unsigned char* cols = tiles + 2 * kPearsonRowBytes + col_slot(x, kc, step) * kPearsonColBytes;
                    mbar_expect_tx(bar_full + st, (2 + (bring ? 2 * halves : 0)) * kTileBytes);
                    tma_load_4d(rows, &map_hi, bar_full + st, kc * 64, 0, x.ti * kTile, x.b);
                    tma_load_4d(rows + kTileBytes, &map_lo, bar_full + st, kc * 64, 0, x.ti * kTile, x.b);
                    if (!bring) continue;
#pragma unroll 1
                    for (int h = 0; h < halves; ++h) {
                        tma_load_4d(cols + h * kTileBytes, &map_hi, bar_full + st, kc * 64, 0, x.tj * kColTile + h * kTile, x.b);
                        tma_load_4d(cols + (2 + h) * kTileBytes, &map_lo, bar_full + st, kc * 64, 0, x.tj * kColTile + h * kTile, x.b);
                    }
                }
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        const uint64_t d0 = umma_desc_sw128(smem_u32(tiles), 16, 1024);
        uint32_t step = 0, i = 0;
#pragma unroll 1
        for (long long u = u0; u < u1 && ok; ++u, ++i) {
            const Unit x = unit_at(u);
            const uint32_t idesc = umma_idesc_bf16(128, (x.cols + 15) & ~15, 0, 0), d = tmem + (i & 1) * kColTile;
            ok = __all_sync(0xffffffffu, mbar_wait_relaxed(bar_accfree + (i & 1), ((i >> 1) & 1) ^ 1));
            if (!ok) break;
            tc_fence_after();
#pragma unroll 1
            for (int kc = 0; kc < n_chunks; ++kc, ++step) {
                const uint32_t st = step & 1;
                ok = __all_sync(0xffffffffu, mbar_wait(bar_full + st, (step >> 1) & 1));
                if (!ok) break;
                tc_fence_after();
                const int k_steps = min(4, (P.L - kc * 64 + 15) / 16);
                if (elect_one()) {                                   // rho += hi hi + hi lo + lo hi over these time steps
                    const uint64_t ah = umma_desc_advance(d0, st * kPearsonRowBytes), al = umma_desc_advance(ah, kTileBytes);
                    const uint64_t bh = umma_desc_advance(d0, 2 * kPearsonRowBytes + col_slot(x, kc, step) * kPearsonColBytes), bl = umma_desc_advance(bh, 2 * kTileBytes);
#pragma unroll 1
                    for (int ks = 0; ks < k_steps; ++ks) {
                        tc_mma_bf16(d, umma_desc_advance(ah, ks * 32), umma_desc_advance(bh, ks * 32), idesc, (kc > 0 || ks > 0) ? 1u : 0u);
                        tc_mma_bf16(d, umma_desc_advance(ah, ks * 32), umma_desc_advance(bl, ks * 32), idesc, 1u);
                        tc_mma_bf16(d, umma_desc_advance(al, ks * 32), umma_desc_advance(bh, ks * 32), idesc, 1u);
                    }
                    tc_commit(bar_free + st);
                    if (kc + 1 == n_chunks) tc_commit(bar_acc + (i & 1));
                }
                __syncwarp();
            }
        }
    } else if (warp >= 4) {
        // two threads a row, 128 of the 256 columns each
        const int row = tid & (kTile - 1), half = (warp - 4) >> 2;
        const uint32_t tm = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16) + half * kTile;
        // (These warps share a named barrier, which nothing bounds: one whose wait gives up goes on to it, without work or further waits, and all leave there.)
        int taken = 0;                                               // units of the current instance
        uint32_t i = 0;
#pragma unroll 1
        for (long long u = u0; u < u1; ++u, ++i) {
            const Unit x = unit_at(u);
            const int v = x.ti * kTile + row;
            float best = -2.f;
            ok = ok && __all_sync(0xffffffffu, mbar_wait(bar_acc + (i & 1), (i >> 1) & 1));
            tc_fence_after();
#pragma unroll 1
            for (int c = 0; c < kTile && ok; c += 32) {
                const int w0 = x.tj * kColTile + half * kTile + c;
                if (w0 >= P.N) break;
                float r[32];
                tmem_ld32(tm + (i & 1) * kColTile + c, r);
                tmem_ld_wait();
                if (w0 + 32 <= P.N && (w0 + 32 <= x.ti * kTile || w0 >= (x.ti + 1) * kTile)) {
                    float m[4] = {best, r[0], r[1], r[2]};
#pragma unroll
                    for (int e = 3; e < 32; ++e) m[e & 3] = fmaxf(m[e & 3], r[e]);
                    best = fmaxf(fmaxf(m[0], m[1]), fmaxf(m[2], m[3]));
                } else {                                             // the diagonal, or columns past the last variate
#pragma unroll
                    for (int e = 0; e < 32; ++e)
                        if (w0 + e < P.N && w0 + e != v) best = fmaxf(best, r[e]);
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0 && ok) mbar_arrive(bar_accfree + (i & 1));
            if (v < P.N && best > -2.f) atomic_max_float(P.max_rho + static_cast<size_t>(x.b) * P.N + v, best);
            ++taken;
            if (u + 1 == u1 || (x.ti + 1 == row_tiles && x.tj + 1 == col_tiles)) {           // the run leaves this instance
                __threadfence();
                ok = epilogue_sync_and(ok);
                if (!ok) break;
                if (tid == 128) {
                    __threadfence();
                    *s_last = atomicAdd(P.done + x.b, taken) + taken == row_tiles * col_tiles;
                }
                epilogue_sync_and(true);
                if (*s_last) {
                    __threadfence();
                    int above = 0;
                    for (int n = tid - 128; n < P.N; n += 256) above += __ldcg(P.max_rho + static_cast<size_t>(x.b) * P.N + n) >= P.threshold;
                    above = __reduce_add_sync(0xffffffffu, above);
                    if (lane == 0 && above) atomicAdd(P.n_above + x.b, above);
                }
                taken = 0;
                epilogue_sync_and(true);                             // the flag is free
            }
        }
    }
    if (!ok) set_status(P.status, VARDROP_ERR_TIMEOUT);
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, kPearsonTmemCols);
}

struct PearsonWs {
    size_t z_hi, z_lo, done, total;
    int Lrow;
};
PearsonWs pearson_layout(const vardrop_pearson_cfg& c) {
    PearsonWs w;
    w.Lrow = (c.L + 7) / 8 * 8;                                      // rows start on 16-byte boundaries
    const size_t bytes = align_up(static_cast<size_t>(c.B) * c.N * w.Lrow * sizeof(__nv_bfloat16), 1024);
    w.z_hi = kWsHeaderBytes;
    w.z_lo = w.z_hi + bytes;
    w.done = w.z_lo + bytes;
    w.total = w.done + align_up(sizeof(int32_t) * c.B, 1024);
    return w;
}

}  // namespace

int pearson_validate(const vardrop_pearson_cfg& c) {
    if (c.B < 1 || c.N < 1 || c.L < 2) return fail(VARDROP_ERR_INVALID_ARG, "pearson: B, N >= 1 and L >= 2 required (B=%d N=%d L=%d)", c.B, c.N, c.L);
    if (c.B > 65535) return fail(VARDROP_ERR_UNSUPPORTED, "pearson: B=%d above 65535", c.B);
    if (c.L > 65536 || c.N > (1 << 22)) return fail(VARDROP_ERR_UNSUPPORTED, "pearson: L=%d or N=%d too large", c.L, c.N);
    if (!(c.threshold >= -1.f && c.threshold <= 1.f)) return fail(VARDROP_ERR_INVALID_ARG, "pearson: threshold must lie in [-1, 1]");
    return VARDROP_OK;
}

size_t pearson_workspace_bytes(const vardrop_pearson_cfg& c) { return pearson_layout(c).total; }

int pearson_launch(const float* x, const vardrop_pearson_cfg& c, float* max_rho, int32_t* n_above, void* ws, cudaStream_t stream) {
    const PearsonWs w = pearson_layout(c);
    char* base = static_cast<char*>(ws);
    PearsonParams P{};
    P.x = x; P.z_hi = reinterpret_cast<__nv_bfloat16*>(base + w.z_hi); P.z_lo = reinterpret_cast<__nv_bfloat16*>(base + w.z_lo);
    P.max_rho = max_rho; P.n_above = n_above; P.status = reinterpret_cast<int*>(base);
    P.done = reinterpret_cast<int32_t*>(base + w.done);
    P.B = c.B; P.N = c.N; P.L = c.L; P.Lrow = w.Lrow; P.threshold = c.threshold;
    CUtensorMap hi, lo;                                              // [B, N, L], zeros outside
    if (int st = make_tile_map(&hi, P.z_hi, c.L, c.B, c.N, 1, static_cast<long long>(c.N) * w.Lrow, w.Lrow, w.Lrow)) return st;
    if (int st = make_tile_map(&lo, P.z_lo, c.L, c.B, c.N, 1, static_cast<long long>(c.N) * w.Lrow, w.Lrow, w.Lrow)) return st;
    cudaError_t err;
    {
        LaunchScope ls_(K_PEARSON_NORM, stream);
        auto launch = [&](auto kernel, int rows) { return launch_chained(kernel, dim3((c.N + 8 * rows - 1) / (8 * rows), c.B), dim3(256), 0, stream, P); };
        err = (c.L & 3) != 0 || c.L > 1024 ? launch(pearson_normalize_kernel<0>, NormalizeRows<0>::value)
              : c.L <= 128                 ? launch(pearson_normalize_kernel<1>, NormalizeRows<1>::value)
              : c.L <= 256                 ? launch(pearson_normalize_kernel<2>, NormalizeRows<2>::value)
              : c.L <= 512                 ? launch(pearson_normalize_kernel<4>, NormalizeRows<4>::value)
                                           : launch(pearson_normalize_kernel<8>, NormalizeRows<8>::value);
    }
    if (int st = check_cuda(err, "pearson: normalize launch")) return st;
    static thread_local int attr_dev = -1;
    int dev = 0;
    cudaGetDevice(&dev);
    if (attr_dev != dev) {
        if (int st = check_cuda(cudaFuncSetAttribute(pearson_max_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kPearsonSmemBytes), "pearson: smem attribute")) return st;
        attr_dev = dev;
    }
    const long long units = static_cast<long long>(c.B) * ((c.N + kTile - 1) / kTile) * ((c.N + kColTile - 1) / kColTile);
    const int grid = static_cast<int>(units < sm_count() ? units : sm_count());
    { LaunchScope ls_(K_PEARSON_MAX, stream); err = launch_chained(pearson_max_kernel, dim3(grid), dim3(kPearsonThreads), kPearsonSmemBytes, stream, hi, lo, P); }
    return check_cuda(err, "pearson: launch");
}

}  // namespace vardrop
