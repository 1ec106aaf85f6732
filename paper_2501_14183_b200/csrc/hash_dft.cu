// k-dominant frequency hashing (Algorithm 1) for lookback lengths with a large prime factor: the candidate bins of the discrete Fourier transform
// as what they are, a product of the folded windows with a matrix of cosines and sines.
//
//   e_j = x_j + x_{L-j},  o_j = x_j - x_{L-j}  (0 < j < L / 2);   Re X_f = x_0 + sum_j e_j cos(2 pi j f / L) (+- x_{L/2}),   Im X_f = -sum_j o_j sin(2 pi j f / L)
//
// A quarter of the bins are candidates, so a window costs about L^2 / 4 multiply-adds; they run as a register-tiled fp32 product, two results an
// instruction.  (A mixed-radix transform pays a prime factor p with p complex multiply-adds for each of the L points, each operand read from
// shared memory.)  What bounds it is the reading of the two operands from shared memory beside the products, and with few windows the latency
// of a block.  B = 8, N = 2000, L = 1021: 310 us, 5690 with the transform; N = 500, L = 313: 21 us, 197.
//
// A CTA takes kW windows (whole hash rows) and tiles of kF bins: 16-step blocks of folded windows from global memory and of the matrix, gathered
// from a table of L entries, both double-buffered; 4 x 4 outputs a thread, summed 16 steps at a time and then block by block: one chain of L / 2
// additions left the amplitudes up to three times as far from fp64 as the transform does (L = 858: 3.1e-7 of the spectrum, 1.0e-7 so and with the
// transform).  Amplitudes are summed over the batch in ascending instance order in
// shared memory and ranked by eight lanes a row.  With few windows the bin tiles are dealt out over a cluster, whose first CTA ranks.
#include "common.cuh"
#include "kernels.h"

namespace vardrop {

namespace {

constexpr int kStep = 16;                        // time steps a block

struct DftParams {
    const float* x;
    uint64_t* keys;
    int32_t* freqs;
    float* amp_dbg;
    int* status;
    int N, L, k, f_lo, nf, scope;
    int rows_total;       // S * N
    int rows_per_cta;     // hash rows per CTA (cluster)
    int win_per_row;      // windows averaged into one row (B or 1)
    int chunk;            // windows of a row taken per pass: rows_per_cta * chunk <= kW
    int tiles;            // bin tiles
    int split;            // CTAs of a cluster
};

__device__ __forceinline__ uint64_t pair_of(float lo, float hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void halves_of(uint64_t v, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }
__device__ __forceinline__ void fma_pair(uint64_t& d, uint64_t a, uint64_t b) { asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b)); }
__device__ __forceinline__ void add_pair(uint64_t& d, uint64_t a) { asm("add.rn.f32x2 %0, %0, %1;" : "+l"(d) : "l"(a)); }
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// the same place in the shared memory of the cluster's first CTA
__device__ __forceinline__ uint32_t first_cta_addr(const void* p) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"(smem_u32(p)));
    return r;
}

template <int kW, int kF>
struct DftShape {
    static constexpr int kThreads = kW * kF / 16;
    static constexpr int kPitchW = kW + 2, kPitchF = kF + 2;                 // even (8-byte reads), and stores of a transposed block hit distinct banks
    static constexpr int kBlock = 2 * kStep * (kPitchW + kPitchF);           // floats: e, o, cos, sin
    static constexpr int kAmpPitch = kF + 1;
    // table [L] pairs, two blocks (the amplitudes of a tile go over them), sums [rows][nf]
    static constexpr int kBlocks = 2 * kBlock > kW * kAmpPitch ? 2 * kBlock : (kW * kAmpPitch + 1) / 2 * 2;
    static size_t smem_bytes(int L, int rows, int nf) { return sizeof(float2) * L + sizeof(float) * (kBlocks + static_cast<size_t>(rows) * nf); }
};

template <int kW, int kF>
__global__ void __launch_bounds__(kW * kF / 16, kW == 16 ? 8 : 8192 / (kW * kF)) hash_dft_kernel(const DftParams P) {
    using S = DftShape<kW, kF>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int L = P.L, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int T = S::kThreads;
    float2* tw = reinterpret_cast<float2*>(smem_raw);
    float* blocks = reinterpret_cast<float*>(tw + L);
    float* sums = blocks + S::kBlocks;                                       // [rows][nf], in the cluster's first CTA
    for (int m = tid; m < L; m += T) {          // cos and sin of 2 pi m / L; the angle is folded to |m'| <= L / 2 first, what rounding it leaves is put in after
        const int mf = 2 * m > L ? m - L : m;
        const float turn = 2.f * static_cast<float>(mf) / static_cast<float>(L);
        const float rest = fmaf(-turn, static_cast<float>(L), 2.f * static_cast<float>(mf)) / static_cast<float>(L) * 3.14159265f;
        float s, c;
        sincospif(turn, &s, &c);
        tw[m] = make_float2(fmaf(-s, rest, c), fmaf(c, rest, s));
    }
    const int group = blockIdx.x / P.split, rank = blockIdx.x - group * P.split;
    const int row0 = group * P.rows_per_cta, rows = min(P.rows_per_cta, P.rows_total - row0);
    const int half = (L - 1) / 2;                                            // folded steps 1 .. half
    const int n_blocks = (half + kStep - 1) / kStep;
    chain_wait();
    chain_release();
    if (P.split > 1) cluster_sync();                                         // every CTA of the cluster runs: its shared memory may be written

    // this thread's outputs: windows 4 tw4 .. + 3, bins 4 tf4 .. + 3 of a tile; a warp covers 16 windows x 32 bins
    constexpr int kWarpsF = kF / 32;
    const int tf4 = (warp % kWarpsF) * 8 + (lane & 7), tw4 = (warp / kWarpsF) * 4 + (lane >> 3);
    // what it loads of a block: steps lane % 16 of windows (tid / 16) + i (T / 16), and bins tid % kF of steps (tid / kF) + 4 i
    constexpr int kLoads = kW * kStep / T;
    const int lj = tid & (kStep - 1), lw = tid / kStep;
    const int mf = tid % kF, mj = tid / kF;
    constexpr int kRowsF = T / kF, kMat = kStep / kRowsF;                    // matrix rows a pass, passes

    for (int b0 = 0; b0 < P.win_per_row; b0 += P.chunk) {
        const int cw = min(P.chunk, P.win_per_row - b0), n_win = rows * cw;
        // window wl of the pass: instance b0 + wl % cw of row wl / cw
        auto window = [&](int wl) {
            const int r = wl / cw, bi = wl - r * cw;
            const size_t w = P.scope == 0 ? static_cast<size_t>(b0 + bi) * P.N + (row0 + r) : static_cast<size_t>(row0 + r);
            return P.x + w * L;
        };
        const float* src[kLoads];
#pragma unroll
        for (int i = 0; i < kLoads; ++i) {
            const int wl = lw + i * (T / kStep);
            src[i] = wl < n_win ? window(wl) : nullptr;
        }
        for (int tile = rank; tile < P.tiles; tile += P.split) {
            const int f0 = P.f_lo + tile * kF;
            uint32_t at = static_cast<uint32_t>((static_cast<long long>(mj + 1) * (f0 + mf)) % L);       // (step index) f mod L of this thread's matrix rows
            const uint32_t at_step = static_cast<uint32_t>((static_cast<long long>(kRowsF) * (f0 + mf)) % L);
            float e[kLoads], o[kLoads];
            auto fetch = [&](int blk) {
                const int j = 1 + blk * kStep + lj;
#pragma unroll
                for (int i = 0; i < kLoads; ++i) {
                    const bool live = src[i] && j <= half;
                    const float a = live ? __ldg(src[i] + j) : 0.f, b = live ? __ldg(src[i] + L - j) : 0.f;
                    e[i] = a + b;
                    o[i] = a - b;
                }
            };
            auto park = [&](int blk) {
                float* to = blocks + (blk & 1) * S::kBlock;
                float* se = to + lj * S::kPitchW + lw;
#pragma unroll
                for (int i = 0; i < kLoads; ++i) {
                    se[i * (T / kStep)] = e[i];
                    se[kStep * S::kPitchW + i * (T / kStep)] = o[i];
                }
                float* sc = to + 2 * kStep * S::kPitchW + mj * S::kPitchF + mf;
#pragma unroll
                for (int i = 0; i < kMat; ++i) {
                    const float2 v = tw[at];
                    sc[i * kRowsF * S::kPitchF] = v.x;
                    sc[(kStep + i * kRowsF) * S::kPitchF] = v.y;
                    at += at_step;
                    if (at >= static_cast<uint32_t>(L)) at -= L;
                }
            };
            uint64_t re[4][2], im[4][2];                                     // [bin][window pair]
#pragma unroll
            for (int f = 0; f < 4; ++f) re[f][0] = re[f][1] = im[f][0] = im[f][1] = 0ull;
            if (n_blocks > 0) {
                fetch(0);
                __syncthreads();                                             // the blocks are free (and the table complete)
                park(0);
            }
            for (int blk = 0; blk < n_blocks; ++blk) {
                if (blk + 1 < n_blocks) fetch(blk + 1);
                __syncthreads();
                const float* from = blocks + (blk & 1) * S::kBlock;
                const float* pe = from + 4 * tw4;
                const float* pc = from + 2 * kStep * S::kPitchW + 4 * tf4;
                uint64_t bre[4][2], bim[4][2];                               // this block's sums
#pragma unroll
                for (int f = 0; f < 4; ++f) bre[f][0] = bre[f][1] = bim[f][0] = bim[f][1] = 0ull;
#pragma unroll 4
                for (int j = 0; j < kStep; ++j) {
                    const uint64_t e0 = *reinterpret_cast<const uint64_t*>(pe + j * S::kPitchW), e1 = *reinterpret_cast<const uint64_t*>(pe + j * S::kPitchW + 2);
                    const uint64_t o0 = *reinterpret_cast<const uint64_t*>(pe + (kStep + j) * S::kPitchW), o1 = *reinterpret_cast<const uint64_t*>(pe + (kStep + j) * S::kPitchW + 2);
                    const float2 c01 = *reinterpret_cast<const float2*>(pc + j * S::kPitchF), c23 = *reinterpret_cast<const float2*>(pc + j * S::kPitchF + 2);
                    const float2 s01 = *reinterpret_cast<const float2*>(pc + (kStep + j) * S::kPitchF), s23 = *reinterpret_cast<const float2*>(pc + (kStep + j) * S::kPitchF + 2);
                    const float c[4] = {c01.x, c01.y, c23.x, c23.y}, s[4] = {s01.x, s01.y, s23.x, s23.y};
#pragma unroll
                    for (int f = 0; f < 4; ++f) {
                        const uint64_t cc = pair_of(c[f], c[f]), ss = pair_of(s[f], s[f]);
                        fma_pair(bre[f][0], e0, cc);
                        fma_pair(bre[f][1], e1, cc);
                        fma_pair(bim[f][0], o0, ss);
                        fma_pair(bim[f][1], o1, ss);
                    }
                }
#pragma unroll
                for (int f = 0; f < 4; ++f) {
                    add_pair(re[f][0], bre[f][0]);
                    add_pair(re[f][1], bre[f][1]);
                    add_pair(im[f][0], bim[f][0]);
                    add_pair(im[f][1], bim[f][1]);
                }
                if (blk + 1 < n_blocks) park(blk + 1);
            }
            __syncthreads();                                                 // the amplitudes go over the blocks
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                const int wl = 4 * tw4 + p;
                if (wl < n_win) {
                    const float* x = window(wl);
                    const float x0 = __ldg(x), xh = (L & 1) == 0 ? __ldg(x + L / 2) : 0.f;
#pragma unroll
                    for (int f = 0; f < 4; ++f) {
                        float r2[2], i2[2];
                        halves_of(re[f][p >> 1], r2[0], r2[1]);
                        halves_of(im[f][p >> 1], i2[0], i2[1]);
                        const float r = r2[p & 1] + (x0 + (((f0 + 4 * tf4 + f) & 1) ? -xh : xh)), i = i2[p & 1];
                        blocks[wl * S::kAmpPitch + 4 * tf4 + f] = sqrtf(fmaf(r, r, i * i));
                    }
                }
            }
            __syncthreads();
            // batch sum, ascending instance order
            for (int i = tid; i < rows * kF; i += T) {
                const int r = i / kF, f = i - r * kF, fi = tile * kF + f;
                if (fi >= P.nf) continue;
                float* to = sums + r * P.nf + fi;
                const float* amp = blocks + r * cw * S::kAmpPitch + f;
                if (P.split == 1) {
                    float a = b0 > 0 ? *to : 0.f;
                    for (int bi = 0; bi < cw; ++bi) a += amp[bi * S::kAmpPitch];
                    *to = a;
                } else {
                    const uint32_t addr = first_cta_addr(to);
                    float a = 0.f;
                    if (b0 > 0) asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(a) : "r"(addr));
                    for (int bi = 0; bi < cw; ++bi) a += amp[bi * S::kAmpPitch];
                    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(a) : "memory");
                }
            }
            __syncthreads();
        }
    }
    if (P.split > 1) cluster_sync();
    if (rank != 0) return;

    // ---- top-k ranking (descending amplitude, lower bin first on ties), packing: eight lanes a row ------------
    const float inv_n = 1.f / static_cast<float>(P.win_per_row);
    const int l8 = lane & 7;
    for (int r0 = warp * 4; r0 < rows; r0 += T / 8) {
        const int r = r0 + (lane >> 3), row = row0 + r;
        const bool live = r < rows;
        float* a = sums + (live ? r : 0) * P.nf;
        bool bad = false;
        if (live) {
            for (int fi = l8; fi < P.nf; fi += 8) {
                bad |= !isfinite(a[fi]);
                if (P.amp_dbg) P.amp_dbg[static_cast<size_t>(row) * P.nf + fi] = a[fi] * inv_n;
            }
        }
        if (__any_sync(0xffffffffu, bad) && lane == 0) set_status(P.status, VARDROP_ERR_NONFINITE);
        uint64_t key = 0;
        for (int rk = 0; rk < P.k; ++rk) {
            // the largest amplitude left, then the lowest bin that has it; amplitudes are non-negative, so their bit patterns order like the
            // values; taken bins are negative, code 0 = nothing left
            unsigned top = 0;
            int bin = 0;
#pragma unroll 4
            for (int fi = l8; fi < P.nf; fi += 8) {
                const float v = a[fi];
                const unsigned code = v >= 0.f ? __float_as_uint(v) + 1u : 0u;
                if (code > top) { top = code; bin = fi; }
            }
#pragma unroll
            for (int m = 1; m < 8; m <<= 1) {
                const unsigned t2 = __shfl_xor_sync(0xffffffffu, top, m);
                const int b2 = __shfl_xor_sync(0xffffffffu, bin, m);
                if (t2 > top || (t2 == top && b2 < bin)) { top = t2; bin = b2; }
            }
            if (live && l8 == 0) {
                a[bin] = -1.f;                                               // removes the winner (bin 0 only with non-finite input)
                if (P.freqs) P.freqs[static_cast<size_t>(row) * P.k + rk] = P.f_lo + bin;
            }
            key = (key << 12) | static_cast<uint64_t>(P.f_lo + bin);
            __syncwarp();
        }
        if (live && l8 == 0) P.keys[row] = key;
    }
}

template <int kW, int kF>
int launch_dft(const DftParams& P, cudaStream_t stream) {
    using S = DftShape<kW, kF>;
    const size_t smem = S::smem_bytes(P.L, P.rows_per_cta, P.nf);
    static thread_local int attr_dev = -1;
    int dev = 0;
    cudaGetDevice(&dev);
    if (attr_dev != dev) {
        if (int st = check_cuda(cudaFuncSetAttribute(hash_dft_kernel<kW, kF>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024), "hash: smem attribute")) return st;
        attr_dev = dev;
    }
    const int groups = (P.rows_total + P.rows_per_cta - 1) / P.rows_per_cta;
    cudaError_t err;
    {
        LaunchScope ls_(K_HASH, stream);
        cudaLaunchAttribute attr[2];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = P.split; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(groups * P.split);
        cfg.blockDim = dim3(S::kThreads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = stream;
        cfg.attrs = attr;
        cfg.numAttrs = P.split > 1 ? 2 : 1;
        err = cudaLaunchKernelEx(&cfg, hash_dft_kernel<kW, kF>, P);
    }
    return check_cuda(err, "hash: launch");
}

}  // namespace

// Returns -1 where the transform in shared memory is the better one (or the sums do not fit).
int hash_dft_launch(const float* x, const vardrop_hash_cfg& c, int f_lo, int f_hi, uint64_t* keys, int32_t* freqs, float* amp_dbg, int* status,
                    cudaStream_t stream) {
    int large = 0;                               // sum of the prime factors above 7, which the transform takes as plain sums
    for (int rem = c.L, p = 2; rem > 1; ++p)
        while (rem % p == 0) { rem /= p; large += p > 7 ? p : 0; }
    if (large == 0) return -1;                   // (16000 windows of 300 steps: 23 us there, 58 here)
    DftParams P{};
    P.x = x; P.keys = keys; P.freqs = freqs; P.amp_dbg = amp_dbg; P.status = status;
    P.N = c.N; P.L = c.L; P.k = c.k; P.f_lo = f_lo; P.nf = f_hi - f_lo; P.scope = c.scope;
    const HashSplit there = hash_split(c);
    P.rows_total = there.rows_total; P.win_per_row = there.win_per_row;
    const bool narrow = P.nf <= 32;
    P.tiles = (P.nf + (narrow ? 31 : 63)) / (narrow ? 32 : 64);
    // 64 windows a CTA, or 16 where that leaves SMs idle, and then the bin tiles over a cluster as well
    const long long windows = static_cast<long long>(c.B) * c.N;
    const int W = windows >= 1000 ? 64 : 16;
    P.chunk = P.win_per_row < W ? P.win_per_row : W;
    P.rows_per_cta = W / P.chunk;
    const size_t sums = sizeof(float) * static_cast<size_t>(P.rows_per_cta) * P.nf;
    if (sums + sizeof(float2) * c.L > 160 * 1024) return -1;
    const long long groups = (P.rows_total + P.rows_per_cta - 1) / P.rows_per_cta;
    P.split = 1;
    while (P.split < 8 && P.split < P.tiles && groups * P.split < 2ll * sm_count()) P.split *= 2;
    // What either costs, in microseconds: rounds of CTAs, each its blocks and rows here (the first of a cluster ranks for all), its complex transforms
    // there (plain sums over an even length read shared memory with bank conflicts).  The terms are fitted to 1100 measured calls of 33 to 1021 steps,
    // 100 to 32000 windows and three bands, with stages of fours and primes there: the choice so made costs about 1 % more than the better of the two.  With
    // the stages that some lengths save since (radix_plan), 484 calls of 70 such lengths: 2.0 % more, and 1.6 % by terms fitted to those.  Where it turns, there | here: 4384
    // windows of 715 = 5 11 13 steps 41 | 63 us, of 391 = 17 23 37 | 25, of 1021 1642 | 86; 100 of 313 14 | 21, of 1021 107 | 50.
    auto rounds = [](long long ctas, int at_once) { return static_cast<double>((ctas + at_once - 1) / at_once); };
    const int passes_there = (there.win_per_row + there.chunk - 1) / there.chunk;
    const int transforms = there.rows_per_cta > 1 ? (there.rows_per_cta * there.chunk + 1) / 2 : passes_there * ((there.chunk + 1) / 2);
    const double cost_there = 4.3 + rounds((there.rows_total + there.rows_per_cta - 1) / there.rows_per_cta, sm_count()) * transforms * c.L *
                                       ((c.L & 1 ? 1.17e-4 : 1.5e-4) * large + 1.1e-3);
    const int passes = (P.win_per_row + P.chunk - 1) / P.chunk, blocks = ((c.L - 1) / 2 + kStep - 1) / kStep;
    const double work = static_cast<double>((P.tiles + P.split - 1) / P.split) * passes * blocks;
    const double cost = W == 16 ? (narrow ? 3.2 + rounds(groups * P.split, 3 * sm_count()) * (1.24 * work + 0.42 * P.rows_per_cta)
                                          : 4.0 + rounds(groups * P.split, 3 * sm_count()) * (1.32 * work + 0.22 * P.rows_per_cta))
                                : (narrow ? 4.5 + rounds(groups * P.split, 2 * sm_count()) * (1.24 * work + 0.07 * P.rows_per_cta)
                                          : 6.1 + rounds(groups * P.split, sm_count()) * (1.365 * work + 0.048 * P.rows_per_cta) + (P.split > 1 ? 0.25 * P.rows_per_cta : 0.0));
    if (cost >= cost_there) return -1;
    if (W == 64) return narrow ? launch_dft<64, 32>(P, stream) : launch_dft<64, 64>(P, stream);
    return narrow ? launch_dft<16, 32>(P, stream) : launch_dft<16, 64>(P, stream);
}

}  // namespace vardrop
