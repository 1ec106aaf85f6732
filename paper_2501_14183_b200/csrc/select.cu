// Grouping by hash value and stratified sampling (Eq. 1, Eq. 2), without a spin-wait.
//
// Up to 1024 variates (2048 with many rows): one CTA per hash row does everything in shared memory (select_small_kernel).
// Up to 8192: two launches, every variate's sorted position by comparing all pairs of keys over the whole GPU (select_place_kernel), then a
// cluster of eight CTAs per hash row (select_cluster_kernel).
// Larger ones take three launches behind a clear:
//   select_count_kernel   every CTA compares a slice of variates against a slice of keys and adds, per variate n,
//                         lt[n] = #{m : key_m < key_n} and eq[n] = #{m < n : key_m = key_n} with integer atomics.  lt[n] is
//                         the start of n's group in (key, index) order and eq[n] is n's rank inside its group, so lt + eq
//                         is n's sorted position.
//   select_group_kernel   one CTA per hash row scatters the members, scans the group heads into dense group ids and
//                         offsets, and draws each member's Philox priority.
//   select_sample_kernel  every member counts the members of its own group with a smaller (priority, rank) pair; it is
//                         kept when that count is below the group's quota.  The CTA that finishes last for a hash row
//                         compacts the kept variates into sel_idx / inv_idx with one scan.
#include <mutex>
#include <type_traits>

#include "common.cuh"
#include "kernels.h"

namespace vardrop {

namespace {

constexpr int kSelThreads = 256;    // select_count_kernel
constexpr int kTailThreads = 1024;  // select_group_kernel, select_sample_kernel: one CTA walks a whole hash row, so the
                                    // round trips to memory are spread over as many threads as a CTA can have
constexpr int kTailChunks = 8;      // positions per thread in a batch of the ordered compaction (64 registers a thread)
constexpr int kKeyChunk = 128;      // keys compared per CTA by select_count_kernel
constexpr size_t kGroupMaxSmem = 216 * 1024;   // select_group_kernel keeps 12 bytes per variate in shared memory up to this

struct SelectParams {
    const uint64_t* keys;
    int32_t *group_id, *group_offsets, *members, *n_groups, *sel_idx, *n_sel, *inv_idx;
    // workspace
    int* status;
    unsigned int* done2;   // [S]
    uint64_t* sorted_keys; // [S, N] (in the place of lt and eq)
    int32_t* lt;           // [S, N]
    int32_t* eq;           // [S, N]
    uint32_t* prio;        // [S, N] priority by sorted position
    int32_t* keep;         // [S, N] by variate
    int S, N, gs;
    long long rate_ppm;
    uint32_t seed_lo, seed_hi, step;
};

// Philox4x32-10 (Salmon et al., SC'11): ten rounds of two 32x32->64 multiplies, xors with the key, and a
// Weyl key schedule.  Returns word 0 of the output block.
__device__ __forceinline__ uint32_t philox4x32_10_word0(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, uint32_t k0, uint32_t k1) {
#pragma unroll 2
    for (int round = 0; round < 10; ++round) {
        const uint32_t hi0 = __umulhi(0xD2511F53u, c0), lo0 = 0xD2511F53u * c0;
        const uint32_t hi1 = __umulhi(0xCD9E8D57u, c2), lo1 = 0xCD9E8D57u * c2;
        const uint32_t n0 = hi1 ^ c1 ^ k0, n2 = hi0 ^ c3 ^ k1;
        c0 = n0; c1 = lo1; c2 = n2; c3 = lo0;
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
    return c0;
}

__device__ __forceinline__ int quota_of(int size, int gs, long long rate_ppm) {
    long long by_rate = (static_cast<long long>(size) * rate_ppm + 999999ll) / 1000000ll;
    if (by_rate < 1) by_rate = 1;
    long long q = size;
    if (gs > 0 && gs < q) q = gs;
    if (by_rate < q) q = by_rate;
    return static_cast<int>(q);
}

__device__ __forceinline__ uint32_t quota_small(uint32_t size, int gs, uint32_t rate_ppm) {        // the same for size <= 2048: 32 bits are enough
    uint32_t q = max(1u, (size * rate_ppm + 999999u) / 1000000u);
    if (gs > 0) q = min(q, static_cast<uint32_t>(gs));
    return min(q, size);
}

// Inclusive scan of one int per thread across the CTA (kThreads threads); returns this thread's inclusive value
// and the CTA total through `total`.
template <int kThreads>
__device__ __forceinline__ int block_scan_inclusive(int v, int* warp_sums, int* total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int o = __shfl_up_sync(0xffffffffu, v, off);
        if (lane >= off) v += o;
    }
    __syncthreads();
    if (lane == 31) warp_sums[warp] = v;
    __syncthreads();
    int base = 0, tot = 0;
#pragma unroll
    for (int w = 0; w < kThreads / 32; ++w) {
        const int s = warp_sums[w];
        if (w < warp) base += s;
        tot += s;
    }
    *total = tot;
    return v + base;
}

// True in every thread of exactly one CTA per hash row: the one whose arrival completes the count.
__device__ __forceinline__ bool last_cta_of_row(unsigned int* counter, unsigned int ctas_per_row, int* flag_smem) {
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned int prev = atomicAdd(counter, 1u);
        *flag_smem = (prev + 1u == ctas_per_row);
    }
    __syncthreads();
    const bool last = *flag_smem != 0;
    if (last) __threadfence();
    return last;
}

// Ordered compaction by one CTA of kThreads threads: for every position p < N, in ascending order,
// `emit(p, set, before, payload)` is called with (set, payload) = flag(p) and before = number of set flags at positions
// below p; returns the number of set flags.  Positions are dealt to the threads round-robin (position = batch base +
// chunk * kThreads + thread) and a batch of kChunks chunks is handled with fully unrolled loops, so the (dependent) loads
// behind the flags of a thread are coalesced and all in flight at once instead of one memory round trip per position; a
// batch is ordered with warp ballots and one scan of the per-warp counts.
template <int kThreads, int kChunks, class FlagFn, class EmitFn>
__device__ __forceinline__ int ordered_compact(int N, FlagFn flag, EmitFn emit) {
    constexpr int kWarps = kThreads / 32;
    static_assert(kChunks <= 32 && kChunks * kWarps <= kThreads, "one ballot word per thread at most");
    __shared__ uint32_t s_mask[kChunks * kWarps];  // ballot of chunk k, warp w at [k * kWarps + w]: position order
    __shared__ int s_excl[kChunks * kWarps];       // set flags of the batch before that (chunk, warp)
    __shared__ int s_warp[kWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int done = 0;                                  // set flags of the batches before this one
    for (int base = 0; base < N; base += kChunks * kThreads) {
        uint32_t bits = 0;                         // bit k: flag of position base + k * kThreads + thread
        int payload[kChunks];
#pragma unroll
        for (int k = 0; k < kChunks; ++k) {
            const int p = base + k * kThreads + static_cast<int>(threadIdx.x);
            payload[k] = 0;
            if (p < N && flag(p, &payload[k])) bits |= 1u << k;
        }
        uint32_t mine = 0;
#pragma unroll
        for (int k = 0; k < kChunks; ++k) {
            const uint32_t m = __ballot_sync(0xffffffffu, (bits >> k) & 1u);
            if (lane == k) mine = m;
        }
        __syncthreads();                           // the tables of the previous batch are no longer read
        if (lane < kChunks) s_mask[lane * kWarps + warp] = mine;
        __syncthreads();
        int total = 0;
        const bool entry = static_cast<int>(threadIdx.x) < kChunks * kWarps;      // one (chunk, warp) ballot per thread
        const int cnt = entry ? __popc(s_mask[threadIdx.x]) : 0;
        const int incl = block_scan_inclusive<kThreads>(cnt, s_warp, &total);
        if (entry) s_excl[threadIdx.x] = incl - cnt;
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kChunks; ++k) {
            const int p = base + k * kThreads + static_cast<int>(threadIdx.x);
            if (p < N) {
                const uint32_t m = s_mask[k * kWarps + warp];
                emit(p, ((bits >> k) & 1u) != 0, done + s_excl[k * kWarps + warp] + __popc(m & ((1u << lane) - 1u)), payload[k]);
            }
        }
        done += total;
    }
    return done;
}

__global__ void __launch_bounds__(kSelThreads) select_count_kernel(const SelectParams P) {
    __shared__ uint64_t skeys[kKeyChunk];
    chain_wait();
    chain_release();
    const int s = blockIdx.z, N = P.N;
    const uint64_t* keys = P.keys + static_cast<size_t>(s) * N;
    int32_t* lt = P.lt + static_cast<size_t>(s) * N;
    int32_t* eq = P.eq + static_cast<size_t>(s) * N;
    const int n = blockIdx.x * kSelThreads + threadIdx.x;
    const int m0 = blockIdx.y * kKeyChunk;
    const int mcount = min(kKeyChunk, N - m0);
    for (int i = threadIdx.x; i < mcount; i += blockDim.x) skeys[i] = keys[m0 + i];
    __syncthreads();
    if (n < N) {
        const uint64_t mine = keys[n];
        int c_lt = 0, c_eq = 0;
        const int n_first = blockIdx.x * kSelThreads;
        if (m0 >= n_first + kSelThreads) {                 // every key of the slice has a higher index than every variate here
            for (int i = 0; i < mcount; ++i) c_lt += skeys[i] < mine;
        } else if (m0 + mcount <= n_first) {               // every key of the slice has a lower index
            for (int i = 0; i < mcount; ++i) {
                const uint64_t other = skeys[i];
                c_lt += other < mine;
                c_eq += other == mine;
            }
        } else {
            for (int i = 0; i < mcount; ++i) {
                const uint64_t other = skeys[i];
                c_lt += other < mine;
                c_eq += (other == mine) & (m0 + i < n);
            }
        }
        if (c_lt) atomicAdd(lt + n, c_lt);
        if (c_eq) atomicAdd(eq + n, c_eq);
    }
}

// One CTA per hash row, after the counts are complete: members, group heads -> ids and offsets, priorities.
// The three passes reach members / eq / group ids through the sorted positions, i.e. in scattered order.  A single SM
// turns every scattered warp access to global memory into 32 separate requests, which is what this kernel's time used
// to be; with kShared the three arrays live in shared memory (12 bytes per variate) and global memory only sees
// coalesced reads and writes.  Rows too long for that work on the global arrays directly.
template <bool kShared>
__global__ void __launch_bounds__(kTailThreads) select_group_kernel(const SelectParams P) {
    extern __shared__ int32_t s_rows[];
    chain_wait();
    chain_release();
    const int s = blockIdx.x, N = P.N;
    const int32_t* lt = P.lt + static_cast<size_t>(s) * N;
    int32_t* eq = P.eq + static_cast<size_t>(s) * N;
    int32_t* members = P.members + static_cast<size_t>(s) * N;
    int32_t* gid = P.group_id + static_cast<size_t>(s) * N;
    int32_t* off = P.group_offsets + static_cast<size_t>(s) * (N + 1);
    uint32_t* prio = P.prio + static_cast<size_t>(s) * N;
    int32_t* gid_by_pos = P.lt + static_cast<size_t>(s) * N;       // lt is dead after the first pass: group id by position
    int32_t* w_eq = kShared ? s_rows : eq;                         // working copies, by variate / position / variate
    int32_t* w_members = kShared ? s_rows + N : members;
    int32_t* w_gid = kShared ? s_rows + 2 * N : gid;
    // every loop of this kernel takes several positions per thread at a time: the loads of a batch are issued together, so
    // a batch costs one or two memory round trips instead of one per position
    constexpr int U = 4;
    for (int base = 0; base < N; base += U * kTailThreads) {
        int dst[U], rank[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int i = base + u * kTailThreads + static_cast<int>(threadIdx.x);
            rank[u] = i < N ? __ldcg(eq + i) : 0;
            dst[u] = i < N ? __ldcg(lt + i) + rank[u] : -1;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int i = base + u * kTailThreads + static_cast<int>(threadIdx.x);
            if (dst[u] >= 0) {
                w_members[dst[u]] = i;
                if (kShared) w_eq[i] = rank[u];
            }
        }
    }
    __syncthreads();
    // group heads over the sorted positions: the first member of every group has no equal key before it
    const int total_groups = ordered_compact<kTailThreads, kTailChunks>(
        N, [&](int p, int* nn) { *nn = w_members[p]; return w_eq[*nn] == 0; },
        [&](int p, bool head, int before, int nn) {
            if (head) off[before] = p;
            const int g = before - (head ? 0 : 1);       // heads at or below p, minus one
            w_gid[nn] = g;
            gid_by_pos[p] = g;
            if (kShared) members[p] = nn;
        });
    for (int i = total_groups + threadIdx.x; i <= N; i += blockDim.x) off[i] = N;
    if (threadIdx.x == 0) P.n_groups[s] = total_groups;
    __syncthreads();
    for (int base = 0; base < N; base += U * kTailThreads) {
        int rank[U], g[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int p = base + u * kTailThreads + static_cast<int>(threadIdx.x);
            const int nn = p < N ? w_members[p] : 0;
            rank[u] = w_eq[nn];
            g[u] = w_gid[nn];
            if (kShared && p < N) gid[p] = w_gid[p];     // position p doubles as a variate index for the copy-out
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int p = base + u * kTailThreads + static_cast<int>(threadIdx.x);
            if (p < N)
                prio[p] = philox4x32_10_word0(static_cast<uint32_t>(rank[u]), static_cast<uint32_t>(g[u]), static_cast<uint32_t>(s), P.step,
                                              P.seed_lo, P.seed_hi);
        }
    }
}

__global__ void __launch_bounds__(kTailThreads) select_sample_kernel(const SelectParams P) {
    __shared__ int flag;
    chain_wait();
    chain_release();
    const int s = blockIdx.z, N = P.N;
    const int32_t* members = P.members + static_cast<size_t>(s) * N;
    const int32_t* gid_by_pos = P.lt + static_cast<size_t>(s) * N;      // written by select_group_kernel
    const int32_t* off = P.group_offsets + static_cast<size_t>(s) * (N + 1);
    const uint32_t* prio = P.prio + static_cast<size_t>(s) * N;
    int32_t* keep = P.keep + static_cast<size_t>(s) * N;
    const int p = blockIdx.x * kTailThreads + threadIdx.x;
    if (p < N) {
        const int nn = members[p];
        const int g = gid_by_pos[p];
        const int begin = off[g], end = off[g + 1];
        const uint32_t mine = prio[p];
        int smaller = 0;
        for (int o = begin; o < end; ++o) {
            const uint32_t other = __ldg(prio + o);
            smaller += (other < mine) | ((other == mine) & (o < p));
        }
        keep[nn] = smaller < quota_of(end - begin, P.gs, P.rate_ppm);
    }
    if (!last_cta_of_row(P.done2 + s, gridDim.x, &flag)) return;

    // ---- the last CTA of this hash row: compaction of the kept variates in ascending index order --------
    int32_t* sel = P.sel_idx + static_cast<size_t>(s) * N;
    int32_t* inv = P.inv_idx + static_cast<size_t>(s) * N;
    const int total = ordered_compact<kTailThreads, kTailChunks>(
        N, [&](int i, int*) { return __ldcg(keep + i) != 0; },
        [&](int i, bool kept, int before, int) {
            if (kept) sel[before] = i;
            inv[i] = kept ? before : -1;
        });
    for (int i = total + threadIdx.x; i < N; i += blockDim.x) sel[i] = -1;
    if (threadIdx.x == 0) P.n_sel[s] = total;
}

// ---------------------------------------------------------------------------------------------------------
// Long groups (up to a few per CTA): a member's sampling rank only matters near the quota.  The priorities are uniform 32-bit numbers: a count of members
// by their top bits finds the bucket in which the quota ends; members in the buckets below are kept, those above are not, and the few in
// it are ranked among themselves.  Counting a rank over the whole group would be size^2 comparisons.
// ---------------------------------------------------------------------------------------------------------
constexpr int kCountMaxGroup = 64;             // longest group whose ranks are counted over all of it
constexpr int kBucketShift = 26, kBuckets = 64;
template <int kMax>
struct LongGroups {
    int n;                                     // zeroed ahead
    int start[kMax], size[kMax], quota[kMax];  // the group's priorities are prio[start ..]
    int cut[kMax], below[kMax], n_cand[kMax];  // the bucket, members below it, members in it
    int hist[kMax * kBuckets];                 // zeroed ahead
};
template <int kMax>
__device__ __forceinline__ void add_long_group(LongGroups<kMax>& G, int start, int size, int quota) {      // by one thread
    const int l = atomicAdd(&G.n, 1);
    G.start[l] = start; G.size[l] = size; G.quota[l] = quota; G.n_cand[l] = 0;
}
// By the whole CTA of T threads, behind a barrier and with one at its end.  cand[start ..]: members in the bucket, in any order.
template <int T, int kMax>
__device__ __noinline__ void rank_long_groups(LongGroups<kMax>& G, const uint32_t* prio, uint16_t* cand) {
    const int tid = threadIdx.x, lane = tid & 31;
    for (int l = 0; l < G.n; ++l)
        for (int o = tid; o < G.size[l]; o += T) atomicAdd(G.hist + l * kBuckets + (prio[G.start[l] + o] >> kBucketShift), 1);
    __syncthreads();
    for (int l = tid >> 5; l < G.n; l += T / 32) {
        const int quota = G.quota[l], h0 = G.hist[l * kBuckets + 2 * lane], h1 = G.hist[l * kBuckets + 2 * lane + 1];
        int run = h0 + h1;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, run, o);
            if (lane >= o) run += v;
        }
        const int b0 = run - h0 - h1, b1 = run - h1;           // members below the lane's two buckets
        if (b0 < quota && quota <= b1) { G.cut[l] = 2 * lane; G.below[l] = b0; }
        if (b1 < quota && quota <= run) { G.cut[l] = 2 * lane + 1; G.below[l] = b1; }
    }
    __syncthreads();
    for (int l = 0; l < G.n; ++l)
        for (int o = G.start[l] + tid; o < G.start[l] + G.size[l]; o += T)
            if (static_cast<int>(prio[o] >> kBucketShift) == G.cut[l]) cand[G.start[l] + atomicAdd(G.n_cand + l, 1)] = static_cast<uint16_t>(o);
    __syncthreads();
}
// Whether prio[o] of the group from `start` on is within the quota; equal priorities rank by place.
template <int kMax>
__device__ __noinline__ bool long_group_keeps(const LongGroups<kMax>& G, const uint32_t* prio, const uint16_t* cand, int start, int o) {
    int l = 0;
    while (G.start[l] != start) ++l;
    const uint32_t mine = prio[o];
    const int bucket = static_cast<int>(mine >> kBucketShift);
    if (bucket != G.cut[l]) return bucket < G.cut[l];
    int below = G.below[l];
    for (int i = 0; i < G.n_cand[l]; ++i) {
        const int c = cand[start + i];
        below += (prio[c] < mine) | ((prio[c] == mine) & (c < o));
    }
    return below < G.quota[l];
}

// ---------------------------------------------------------------------------------------------------------
// Small problems (N <= 1024, or 2048 with many rows): one CTA per hash row does everything in shared memory.
//
// The distinct keys are found with a hash table and ranked against each other, which gives the group ids and offsets; a bitmap of its
// members per distinct key gives a variate's place in its group; the sampling rank of a member is counted over its group.  More distinct keys than a
// few hundred (small_max_groups) are sorted instead:
//   sort 1: (key, variate)                      -> members, group heads -> ids, offsets
//   sort 2: (group id, Philox priority, rank j) -> position inside the group = sampling rank
// Then the kept flags are compacted.  No scratch in global memory, no global atomics.
// ---------------------------------------------------------------------------------------------------------
constexpr int kSmallMaxN = 2048;

// Bitonic sort of M (a power of two >= 64) items by M / 2 threads, which are all that is left of the CTA.  Thread t keeps items 2t and 2t + 1 in
// registers.
// Compare-exchange distance j = 1 stays inside the thread, j = 2 .. 32 goes through warp shuffles (the partner of item
// i is item i ^ j = slot (i & 1) of lane t ^ (j / 2)), and only j >= 64 passes through shared memory.
// Items are (key, payload) pairs ordered by key, then payload; kPayload = false sorts bare keys.
template <bool kPayload>
__device__ __forceinline__ void bitonic_sort_regs(uint64_t& k0, uint32_t& p0, uint64_t& k1, uint32_t& p1, uint64_t* sk, uint32_t* sp, int M) {
    const int t = threadIdx.x;
    auto greater = [](uint64_t ka, uint32_t pa, uint64_t kb, uint32_t pb) { return ka > kb || (kPayload && ka == kb && pa > pb); };
    // keep the smaller of (mine, other) when `want_min`, else the larger
    auto keep = [&](uint64_t& km, uint32_t& pm, uint64_t ko, uint32_t po, bool want_min) {
        const bool mine_greater = greater(km, pm, ko, po);
        if (mine_greater == want_min) { km = ko; pm = po; }
    };
    for (int k = 2; k <= M; k <<= 1) {
        const bool up = ((2 * t) & k) == 0;              // the same for both items of the thread once k >= 2
        int j = k >> 1;
        for (; j >= 64; j >>= 1) {                       // partners live in another warp
            sk[2 * t] = k0; sk[2 * t + 1] = k1;
            if (kPayload) { sp[2 * t] = p0; sp[2 * t + 1] = p1; }
            __syncthreads();
            const int l = (2 * t) ^ j;
            const uint64_t ok0 = sk[l], ok1 = sk[l + 1];
            const uint32_t op0 = kPayload ? sp[l] : 0u, op1 = kPayload ? sp[l + 1] : 0u;
            __syncthreads();
            const bool lower = ((2 * t) & j) == 0;
            keep(k0, p0, ok0, op0, lower == up);
            keep(k1, p1, ok1, op1, lower == up);
        }
        for (; j >= 2; j >>= 1) {                        // partners live in the same warp
            const int m = j >> 1;
            const uint64_t ok0 = __shfl_xor_sync(0xffffffffu, k0, m), ok1 = __shfl_xor_sync(0xffffffffu, k1, m);
            const uint32_t op0 = kPayload ? __shfl_xor_sync(0xffffffffu, p0, m) : 0u, op1 = kPayload ? __shfl_xor_sync(0xffffffffu, p1, m) : 0u;
            const bool lower = (t & m) == 0;
            keep(k0, p0, ok0, op0, lower == up);
            keep(k1, p1, ok1, op1, lower == up);
        }
        if (greater(k0, p0, k1, p1) == up) {             // distance 1: the thread's own pair (up is taken at k >= 2; k = 2 sorts pairs
            const uint64_t tk = k0; k0 = k1; k1 = tk;    //              alternately up and down by bit 1 of the item index)
            const uint32_t tp = p0; p0 = p1; p1 = tp;
        }
    }
}

// exclusive scan of two values per thread (positions 2 tid and 2 tid + 1) over the CTA's first kThreads threads; returns the exclusive prefix
// of position 2 tid and the total
template <int kThreads>
__device__ __forceinline__ int block_scan_pair(int v0, int v1, int* warp_sums, int* total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int v = v0 + v1;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int o = __shfl_up_sync(0xffffffffu, v, off);
        if (lane >= off) v += o;
    }
    __syncthreads();
    if (lane == 31) warp_sums[warp] = v;
    __syncthreads();
    int base = 0, tot = 0;
#pragma unroll 1
    for (int w = 0; w < kThreads / 32; ++w) {
        const int sw = warp_sums[w];
        if (w < warp) base += sw;
        tot += sw;
    }
    *total = tot;
    return v + base - v0 - v1;
}

// Most distinct keys the table path takes: ranking G keys is G^2 / 4 cycles, the sort does not depend on G.  Table | sort: 200 variates, 100 keys 3.9 | 5.2 us,
// 200 6.2 | 5.4; 512, 256 keys 6.4 | 6.6, 512 13.8 | 7.0; 600, 300 keys 8.0 | 9.3; 862, 431 keys 11.7 | 10.0; above 1024 variates the bitmaps fill shared
// memory first.  (A call with more has paid for the table when it comes to sort: 512 variates, all distinct, 4.9 us by sorting alone.)
__host__ __device__ constexpr int small_max_groups(int M) { return M <= 128 ? M : M <= 256 ? 160 : M <= 512 ? 256 : M <= 1024 ? 352 : 360; }

// Shared memory of the table path (the sorting path uses less, over it).
struct SmallLayout {
    int table, list, info, bits, prio, size, before, slot_id, rank, at_pos, cand, total;       // byte offsets
};
__host__ __device__ constexpr SmallLayout small_layout(int M) {
    SmallLayout l{};
    const int G = small_max_groups(M), pitch = (M / 32) | 1, pitch2 = (M / 64) | 1;
    int o = 0;
    l.table = o; o += 2 * M * 8;                   // [2M] keys
    l.bits = o; o += (G * pitch + 3) / 4 * 16;     // [G][pitch] members of an entry, by variate
    l.size = o; o += (G + 16) * 4;                 // [G] members of an entry, 1 << 16 added
    l.prio = o; o += (M + 7 * G + 8) * 4;          // priorities, a group's from a multiple of eight on, all ones between groups
    l.list = o; o += (G + 16) * 8;                 // [G] distinct keys, in any order: the entries; all ones behind them
    l.info = o; o += G * 8;                        // [G] first sorted position | size << 16, quota | place of its priorities << 16
    l.before = o; o += G * pitch2 * 4;             // [G][pitch2] members of an entry in the chunks of 32 variates before each, two chunks a word
    l.slot_id = o; o += (2 * M + 2) * 2;           // [2M + 1] slot -> entry
    l.rank = o; o += G * 2;                        // [G] group id of an entry
    l.total = (o + 15) & ~15;
    l.at_pos = l.table;                            // [M] by sorted position: variate | entry << 16 (the table is not looked up any more by then)
    l.cand = l.bits;                               // [M + 7 G + 8] (nor these)
    return l;
}

// launched with min(M, 1024) threads (M >= 64 a power of two, N <= M), kItems variates or sorted positions a thread
//
// What bounds it is the instructions of eight short steps between barriers: 21000 warp instructions for 862 variates on one SM, at half of its
// issue rate, and for a few dozen variates their latency.  So the steps are dependent accesses of shared memory without searches (the bitmaps
// give places, a group's priorities are read eight at a time), ranked keys are held four to a thread, and the sizes of the tables are constants
// of the instantiation (as arguments, index arithmetic and loop remainders were half of the instructions).
// Between other launches, with the bitonic sort (up to 512) or the counts per chunk and searches (above) of before: 321 variates in 26 groups 5.4 -> 3.4 us, 862
// in 71 7.1 -> 4.9, in 172 10.0 -> 6.0; all distinct 321 4.9 -> 6.2, 862 10.1 -> 10.6; 32 rows of 321 in 26 5.6 -> 3.5.
template <int M>
__global__ void __launch_bounds__(M < 1024 ? M : 1024) select_small_kernel(const SelectParams P) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    constexpr int T = M < 1024 ? M : 1024, kItems = M / T;
    constexpr SmallLayout L = small_layout(M);
    constexpr bool kSort = small_max_groups(M) < M;
    constexpr int G_max = small_max_groups(M), W = M >> 5, pitch = W | 1, pitch2 = (W / 2) | 1;
    constexpr int kMaxLong = M / (kCountMaxGroup + 1) + 1;
    static_assert(G_max * pitch * 4 >= (M + 7 * G_max + 8) * 2 || M <= kCountMaxGroup, "candidates fit the place of the bitmaps");
    __shared__ int warp_sums[32];
    __shared__ uint32_t keep_bits[W];
    __shared__ int n_entries, all_ones, n_keep;
    __shared__ LongGroups<kMaxLong> long_groups;
    __shared__ __align__(4) bool kept[M];
    const int s = blockIdx.x, N = P.N, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr uint64_t kEmpty = ~0ull;             // marks a free slot; as a key it has a slot of its own behind the table's
    constexpr int kHashShift = M == 64 ? 25 : M == 128 ? 24 : M == 256 ? 23 : M == 512 ? 22 : M == 1024 ? 21 : 20;
    static_assert(1u << (32 - kHashShift) == 2u * M, "a hash value is a slot");
    uint64_t* table = reinterpret_cast<uint64_t*>(sm_raw + L.table);
    uint64_t* list = reinterpret_cast<uint64_t*>(sm_raw + L.list);
    uint2* info = reinterpret_cast<uint2*>(sm_raw + L.info);
    uint32_t* bits = reinterpret_cast<uint32_t*>(sm_raw + L.bits);
    uint32_t* prio = reinterpret_cast<uint32_t*>(sm_raw + L.prio);
    uint32_t* size_s = reinterpret_cast<uint32_t*>(sm_raw + L.size);
    uint32_t* before = reinterpret_cast<uint32_t*>(sm_raw + L.before);
    uint16_t* slot_id = reinterpret_cast<uint16_t*>(sm_raw + L.slot_id);
    uint16_t* rank = reinterpret_cast<uint16_t*>(sm_raw + L.rank);
    uint32_t* at_pos = reinterpret_cast<uint32_t*>(sm_raw + L.at_pos);
    uint16_t* cand = reinterpret_cast<uint16_t*>(sm_raw + L.cand);
    // cleared ahead of the wait: the table, the priorities and the list of keys all ones, bitmaps and sizes zero
#pragma unroll
    for (int i = tid; i < M; i += T) reinterpret_cast<uint4*>(table)[i] = make_uint4(~0u, ~0u, ~0u, ~0u);
#pragma unroll 1
    for (int i = L.bits / 16 + tid; i < L.prio / 16; i += T) reinterpret_cast<uint4*>(sm_raw)[i] = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll 1
    for (int i = tid; i < M + 7 * G_max + 8; i += T) prio[i] = ~0u;
#pragma unroll 1
    for (int i = tid; i < G_max + 16; i += T) list[i] = ~0ull;
#pragma unroll 1
    for (int i = tid; i < kMaxLong * kBuckets; i += T) long_groups.hist[i] = 0;
#pragma unroll
    for (int i = tid; i < M; i += T) kept[i] = false;
    if (tid == 0) { n_entries = 0; all_ones = 0; n_keep = 0; long_groups.n = 0; }
    __syncthreads();
    chain_wait();
    chain_release();
    const uint64_t* keys = P.keys + static_cast<size_t>(s) * N;
    int32_t* members = P.members + static_cast<size_t>(s) * N;
    int32_t* gid = P.group_id + static_cast<size_t>(s) * N;
    int32_t* off = P.group_offsets + static_cast<size_t>(s) * (N + 1);
    int32_t* sel = P.sel_idx + static_cast<size_t>(s) * N;
    int32_t* inv = P.inv_idx + static_cast<size_t>(s) * N;

    // ---- the distinct keys: whoever takes a slot opens an entry ------------------------------------------------
    uint64_t key[kItems];
    int at[kItems];                                // slot, then entry of this thread's variates
#pragma unroll
    for (int e = 0; e < kItems; ++e) key[e] = tid + e * T < N ? keys[tid + e * T] : 0ull;
#pragma unroll
    for (int e = 0; e < kItems; ++e) {
        at[e] = 2 * M;
        if (tid + e * T >= N || (kSort && e > 0 && *reinterpret_cast<volatile int*>(&n_entries) > G_max)) continue;         // (too many already: to the sort)
        bool mine = false;
        if (key[e] == kEmpty) {
            mine = atomicExch(&all_ones, 1) == 0;
        } else {
            at[e] = static_cast<int>((static_cast<uint32_t>(key[e]) + static_cast<uint32_t>(key[e] >> 32) * 0x85EBCA6Bu) * 0x9E3779B9u >> kHashShift);
#pragma unroll 1
            for (;;) {                             // at most half of the slots are ever taken
                const uint64_t cur = atomicCAS(reinterpret_cast<unsigned long long*>(table + at[e]), kEmpty, key[e]);
                mine = cur == kEmpty;
                if (mine || cur == key[e]) break;
                at[e] = (at[e] + 1) & (2 * M - 1);
            }
        }
        if (mine) {
            const int d = atomicAdd(&n_entries, 1);
            if (d < G_max) { list[d] = key[e]; slot_id[at[e]] = static_cast<uint16_t>(d); }
        }
    }
    __syncthreads();
    const int G = n_entries;
    if (!kSort || G <= G_max) {
        // ---- members of an entry ---------------------------------------------------------------------------------
#pragma unroll
        for (int e = 0; e < kItems; ++e) {
            if (tid + e * T >= N) continue;
            at[e] = slot_id[at[e]];
            atomicOr(bits + at[e] * pitch + warp + 32 * e, 1u << lane);
        }
        __syncthreads();
        // ---- four lanes an entry: members in the chunks of 32 variates before each, and all of them ------------------
        constexpr int kShare = W >= 8 ? W / 4 : 2;             // a lane's chunks
#pragma unroll 1
        for (int base = 0; base + (tid & ~31) / 4 < G; base += T / 4) {        // (warps with no entry go ahead)
            const int d = base + (tid >> 2), sub = tid & 3;
            const bool has = d < G && sub * kShare < W;
            const int from = min(d, G_max - 1) * pitch + sub * kShare, to = min(d, G_max - 1) * pitch2 + sub * (kShare / 2);
            int count[kShare], run = 0;
#pragma unroll
            for (int c = 0; c < kShare; ++c) {
                count[c] = has ? __popc(bits[from + c]) : 0;
                run += count[c];
            }
            const int own = run;
            int v = __shfl_up_sync(0xffffffffu, run, 1);
            if (sub >= 1) run += v;
            v = __shfl_up_sync(0xffffffffu, run, 2);
            if (sub >= 2) run += v;
            if (sub == 3 && d < G) size_s[d] = 1u << 16 | static_cast<uint32_t>(run);
            run -= own;
#pragma unroll
            for (int c = 0; c < kShare; c += 2) {
                if (has) before[to + c / 2] = static_cast<uint32_t>(run) | static_cast<uint32_t>(run + count[c]) << 16;
                run += count[c] + count[c + 1];
            }
        }
        __syncthreads();
        // ---- group id and first position of an entry: the entries with smaller keys and their members; quota -----------
        // Eight lanes rank four entries at a time: a key read from shared memory is compared with four in registers.
        bool any_long = false;
#pragma unroll 1
        for (int base = 0; base + (tid & ~31) / 2 < G; base += T / 2) {
            const int d0 = base + (tid >> 3) * 4, part = tid & 7;
            uint64_t mine[4];
            uint32_t below[4] = {0u, 0u, 0u, 0u};              // smaller keys << 16 | their members
#pragma unroll
            for (int i = 0; i < 4; ++i) mine[i] = list[min(d0, G_max) + i];
#pragma unroll 2
            for (int e = part; e < G; e += 8) {
                const uint64_t other = list[e];
                const uint32_t one = size_s[e];
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (other < mine[i]) below[i] += one;
            }
#pragma unroll
            for (int o = 1; o < 8; o <<= 1) {
#pragma unroll
                for (int i = 0; i < 4; ++i) below[i] += __shfl_xor_sync(0xffffffffu, below[i], o);
            }
            const int d = d0 + part;
            if (part < 4 && d < G) {
                const uint32_t sums = part < 2 ? (part == 0 ? below[0] : below[1]) : part == 2 ? below[2] : below[3];
                const uint32_t size = size_s[d] & 0xFFFFu, first = sums & 0xFFFFu, g = sums >> 16, q = quota_small(size, P.gs, static_cast<uint32_t>(P.rate_ppm));
                const uint32_t start = (first + 7 * g + 7) & ~7u;              // of its priorities: at least `size` before the next group's
                rank[d] = static_cast<uint16_t>(g);
                info[d] = make_uint2(first | size << 16, q | start << 16);
                atomicAdd(&n_keep, static_cast<int>(q));
                if (size > kCountMaxGroup && q < size) {
                    add_long_group(long_groups, static_cast<int>(start), static_cast<int>(size), static_cast<int>(q));
                    any_long = true;
                }
            }
        }
        any_long = __syncthreads_or(any_long) && M > kCountMaxGroup;
        // ---- sorted positions and priorities ---------------------------------------------------------------------
#pragma unroll
        for (int e = 0; e < kItems; ++e) {
            const int n = tid + e * T, d = at[e], chunk = warp + 32 * e;
            if (n >= N) continue;
            const int g = rank[d];
            const uint2 f = info[d];
            const int j = ((before[d * pitch2 + chunk / 2] >> (chunk & 1) * 16) & 0xFFFFu) + __popc(bits[d * pitch + chunk] & ((1u << lane) - 1u));
            prio[(f.y >> 16) + j] = philox4x32_10_word0(static_cast<uint32_t>(j), static_cast<uint32_t>(g), static_cast<uint32_t>(s), P.step, P.seed_lo, P.seed_hi);
            at_pos[(f.x & 0xFFFFu) + j] = static_cast<uint32_t>(n) | static_cast<uint32_t>(d) << 16;
            gid[n] = g;
        }
        if (tid < G) off[rank[tid]] = static_cast<int>(info[tid].x & 0xFFFFu);
        for (int i = G + tid; i <= N; i += T) off[i] = N;
        if (tid == 0) P.n_groups[s] = G;
        __syncthreads();
        // ---- sampling ranks ----------------------------------------------------------------------------------------
        if (any_long) rank_long_groups<T>(long_groups, prio, cand);
        // Equal priorities rank by place.  That is a matter of one call in thousands, so it is left out at first: two members of a group with the
        // same priority on either side of its quota then make one kept variate too many.
        int total, kept_before[kItems];                // kept variates, and those in the chunks before this warp's
#pragma unroll 1
        for (bool exact = false;; exact = true) {
#pragma unroll
            for (int e = 0; e < kItems; ++e) {
                const int p = tid + e * T;
                if (p >= N) continue;
                const int n = static_cast<int>(at_pos[p] & 0xFFFFu), d = static_cast<int>(at_pos[p] >> 16);
                const uint2 f = info[d];
                const int size = static_cast<int>(f.x >> 16), quota = static_cast<int>(f.y & 0xFFFFu);
                const int start = static_cast<int>(f.y >> 16), j = p - static_cast<int>(f.x & 0xFFFFu);
                members[p] = n;
                bool keep = quota == size;
                if (!keep && size <= kCountMaxGroup) {
                    const uint32_t* of_group = prio + start;
                    const uint32_t mine = of_group[j];
                    int below = 0;                     // (what lies behind the group is all ones)
#pragma unroll 1
                    for (int o = 0; o < size; o += 8) {
                        const uint4 u = *reinterpret_cast<const uint4*>(of_group + o), v = *reinterpret_cast<const uint4*>(of_group + o + 4);
                        below += (u.x < mine) + (u.y < mine) + (u.z < mine) + (u.w < mine) + (v.x < mine) + (v.y < mine) + (v.z < mine) + (v.w < mine);
                    }
                    if (exact) {
#pragma unroll 1
                        for (int o = 0; o < j; ++o) below += of_group[o] == mine;
                    }
                    keep = below < quota;
                } else if (!keep) {
                    keep = long_group_keeps(long_groups, prio, cand, start, start + j);
                }
                kept[n] = keep;
            }
            __syncthreads();
            // ---- the kept variates in ascending order ---------------------------------------------------------------
#pragma unroll
            for (int e = 0; e < kItems; ++e) {
                const uint32_t word = __ballot_sync(0xffffffffu, kept[tid + e * T]);
                if (lane == 0) keep_bits[warp + 32 * e] = word;
            }
            __syncthreads();
            total = 0;
#pragma unroll
            for (int e = 0; e < kItems; ++e) {
                const int v = lane < W ? __popc(keep_bits[lane + 32 * e]) : 0;
                int both = v << 16 | (lane < warp ? v : 0);
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) both += __shfl_xor_sync(0xffffffffu, both, o);
                kept_before[e] = total + (both & 0xFFFF);
                total += both >> 16;
            }
            if (exact || total == n_keep) break;
        }
#pragma unroll
        for (int e = 0; e < kItems; ++e) {
            const int n = tid + e * T;
            if (n >= N) continue;
            const uint32_t word = keep_bits[warp + 32 * e];
            const bool keep = (word >> lane) & 1u;
            const int pos = kept_before[e] + __popc(word & ((1u << lane) - 1u));
            if (keep) sel[pos] = n;
            inv[n] = keep ? pos : -1;
        }
        for (int i = total + tid; i < N; i += T) sel[i] = -1;
        if (tid == 0) P.n_sel[s] = total;
        return;
    }
    if constexpr (kSort) {
    // ---- the sorting path: two items a thread, the rest of the threads are done ----------------------------
    constexpr int kSortThreads = M / 2;
    if (tid >= kSortThreads) return;               // (whole warps; a barrier waits for those that have not left)
    uint64_t* a = reinterpret_cast<uint64_t*>(sm_raw);            // [M] sorted keys, later sorted (group, priority, rank) codes
    uint32_t* idx = reinterpret_cast<uint32_t*>(a + M);           // [M] variate by sorted position
    int* gpos = reinterpret_cast<int*>(idx + M);                  // [M] group id by sorted position
    int* off_s = gpos + M;                                        // [M + 1] group offsets
    int* keep_s = off_s + M + 1;                                  // [M] kept flag by variate
    const int p0 = 2 * tid, p1 = 2 * tid + 1;                     // the two items / positions this thread owns
    uint64_t k0 = p0 < N ? keys[p0] : ~0ull, k1 = p1 < N ? keys[p1] : ~0ull;
    uint32_t n0 = p0, n1 = p1;
    // Keys of up to 53 bits (k <= 4 frequencies of 12 bits, say) leave room for the variate index below them: one 64-bit
    // word per item orders by (key, index), and the sort moves a third less data per compare-exchange.
    constexpr int kIndexBits = 11;
    static_assert((1 << kIndexBits) >= kSmallMaxN, "index field too narrow");
    const bool wide = __syncthreads_or((p0 < N && (k0 >> (64 - kIndexBits)) != 0) || (p1 < N && (k1 >> (64 - kIndexBits)) != 0));
    if (!wide) {
        if (p0 < N) k0 = (k0 << kIndexBits) | n0;
        if (p1 < N) k1 = (k1 << kIndexBits) | n1;
        bitonic_sort_regs<false>(k0, n0, k1, n1, a, idx, M);
        n0 = static_cast<uint32_t>(k0) & ((1u << kIndexBits) - 1u);       // padding items (all ones) sort last and are never read
        n1 = static_cast<uint32_t>(k1) & ((1u << kIndexBits) - 1u);
        k0 >>= kIndexBits;
        k1 >>= kIndexBits;
    } else {
        bitonic_sort_regs<true>(k0, n0, k1, n1, a, idx, M);
    }
    a[p0] = k0; a[p1] = k1; idx[p0] = n0; idx[p1] = n1;
    __syncthreads();

    // group heads -> dense ids and offsets
    const int h0 = (p0 < N) && (p0 == 0 || k0 != a[p0 - 1]);
    const int h1 = (p1 < N) && (k1 != k0);
    int groups = 0;
    const int heads_before = block_scan_pair<kSortThreads>(h0, h1, warp_sums, &groups);
    const int g0 = heads_before + h0 - 1, g1 = heads_before + h0 + h1 - 1;
    if (p0 < N) {
        gpos[p0] = g0;
        if (h0) { off_s[g0] = p0; off[g0] = p0; }
        members[p0] = n0;
        gid[n0] = g0;
    }
    if (p1 < N) {
        gpos[p1] = g1;
        if (h1) { off_s[g1] = p1; off[g1] = p1; }
        members[p1] = n1;
        gid[n1] = g1;
    }
    if (tid == 0) { off_s[groups] = N; P.n_groups[s] = groups; }
    for (int i = groups + tid; i <= N; i += kSortThreads) off[i] = N;
    __syncthreads();

    // sampling rank: sort (group, priority, j)
    uint64_t c0 = ~0ull, c1 = ~0ull;
    if (p0 < N) {
        const int j = p0 - off_s[g0];
        const uint32_t pri = philox4x32_10_word0(static_cast<uint32_t>(j), static_cast<uint32_t>(g0), static_cast<uint32_t>(s), P.step, P.seed_lo, P.seed_hi);
        c0 = (static_cast<uint64_t>(g0) << 43) | (static_cast<uint64_t>(pri) << 11) | static_cast<uint64_t>(j);
    }
    if (p1 < N) {
        const int j = p1 - off_s[g1];
        const uint32_t pri = philox4x32_10_word0(static_cast<uint32_t>(j), static_cast<uint32_t>(g1), static_cast<uint32_t>(s), P.step, P.seed_lo, P.seed_hi);
        c1 = (static_cast<uint64_t>(g1) << 43) | (static_cast<uint64_t>(pri) << 11) | static_cast<uint64_t>(j);
    }
    uint32_t d0 = 0, d1 = 0;
    __syncthreads();                                              // everyone is done reading the sorted keys in `a`
    // Where groups are small a member's sampling rank is the number of codes of its group below its own, counted over the group's
    // few positions.  Only when some group is long does the second sort pay.
    const int size0 = p0 < N ? off_s[g0 + 1] - off_s[g0] : 0, size1 = p1 < N ? off_s[g1 + 1] - off_s[g1] : 0;
    a[p0] = c0; a[p1] = c1;
    if (!__syncthreads_or(size0 > kCountMaxGroup || size1 > kCountMaxGroup)) {
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int p = 2 * tid + e;
            if (p < N) {
                const uint64_t mine = e ? c1 : c0;
                const int g = e ? g1 : g0;
                const int begin = off_s[g], end = off_s[g + 1];
                int below = 0;
                for (int o = begin; o < end; ++o) below += a[o] < mine;
                keep_s[idx[p]] = below < quota_of(end - begin, P.gs, P.rate_ppm);
            }
        }
    } else {
        bitonic_sort_regs<false>(c0, d0, c1, d1, a, nullptr, M);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int q = 2 * tid + e;
            const uint64_t c = e ? c1 : c0;
            if (q < N) {
                const int g = static_cast<int>(c >> 43), j = static_cast<int>(c & 2047u);
                const int begin = off_s[g], size = off_s[g + 1] - begin;
                keep_s[idx[begin + j]] = (q - begin) < quota_of(size, P.gs, P.rate_ppm);
            }
        }
    }
    __syncthreads();

    // compaction in ascending variate order
    const int kp0 = p0 < N ? keep_s[p0] : 0, kp1 = p1 < N ? keep_s[p1] : 0;
    int total = 0;
    int pos = block_scan_pair<kSortThreads>(kp0, kp1, warp_sums, &total);
    if (p0 < N) { if (kp0) { sel[pos] = p0; inv[p0] = pos; ++pos; } else inv[p0] = -1; }
    if (p1 < N) { if (kp1) { sel[pos] = p1; inv[p1] = pos; } else inv[p1] = -1; }
    for (int i = total + tid; i < N; i += kSortThreads) sel[i] = -1;
    if (tid == 0) P.n_sel[s] = total;
    }
}

// ---------------------------------------------------------------------------------------------------------
// Middle sizes, two launches.
//
// select_place_kernel     the sorted position of every variate, by comparing every pair of keys: N^2 comparisons of a few instructions are a matter
//                         of one to seven microseconds for the whole GPU, and nothing has to be cleared or exchanged
// select_cluster_kernel   a cluster of eight CTAs per hash row, each with an eighth of the positions (n_loc, a multiple of 32), a thread to a
//                         position: group heads, ids, priorities, sampling ranks, compaction
// What bounds the second is latency: a few short steps and three barriers of the cluster (a fourth, that says that all of its CTAs run, is
// arrived at where the kernel begins and waited for behind the keys' loads).  One CTA with several variates a thread is bound by its
// instruction rate (2000 variates in 100 groups 9.4 us, in 500 27; so 11 in either), sorting an eighth of the keys in every CTA of the cluster and
// searching the eight lists took 31 us for 8192.  In a training step: 8192 variates 43.8 us by the three launches below and their clear -> 20.8; 3000
// 22.5 -> 11.5; 1200 12.9 (one CTA) -> 8.3.
// ---------------------------------------------------------------------------------------------------------
constexpr int kClusterCtas = 8;
constexpr int kClusterMaxN = 8192;
constexpr int kTwoLaunchRows = 4;                // from 1025 to 2048 variates: hash rows up to which the two launches are taken
constexpr int kPlaceThreads = 1024;

// What bounds it is the integer and comparison rate (64 results a cycle and SM).  Sixteen lanes hold kV variates each, the half warps of the CTA compare them
// with different keys, two a shared-memory load.  Keys are compared as doubles, whose bit patterns order like the values as long as none is
// negative, infinite or not a number: one instruction, on a pipe of its own, where two 64-bit integers take two that share theirs with the counting
// (8192 variates 12.0 -> 10.4 us).  Keys of up to five 12-bit bins are such numbers; others are compared as integers.
template <int kV>
__global__ void __launch_bounds__(kPlaceThreads) select_place_kernel(const SelectParams P) {
    extern __shared__ __align__(16) uint64_t s_keys[];         // [N rounded up to 2]
    __shared__ int s_pos[16 * kV];
    constexpr int kParts = kPlaceThreads / 16;
    const int N = P.N, s = blockIdx.y, tid = threadIdx.x, lane = tid & 31, part = tid >> 4;
    if (tid < 16 * kV) s_pos[tid] = 0;
    chain_wait();
    chain_release();
    const uint64_t* keys = P.keys + static_cast<size_t>(s) * N;
    bool special = false;
#pragma unroll 4
    for (int i = tid; i < N; i += kPlaceThreads) {
        const uint64_t key = keys[i];
        s_keys[i] = key;
        special |= key >= 0x7FF0000000000000ull;
    }
    if (tid == 0 && (N & 1)) s_keys[N] = ~0ull;      // (never below another key: the largest integer, and not a number)
    special = __syncthreads_or(special);
    const int base = blockIdx.x * 16 * kV;
    int pos[kV];
#pragma unroll
    for (int i = 0; i < kV; ++i) pos[i] = 0;
    const int n_pairs = (N + 1) >> 1, first = min(base >> 1, n_pairs), last = min((base >> 1) + 8 * kV, n_pairs);
    auto count = [&](auto as) {
        using T = decltype(as(uint64_t{}));
        T mine[kV];
#pragma unroll
        for (int i = 0; i < kV; ++i) mine[i] = as(s_keys[min(base + (lane & 15) + 16 * i, N - 1)]);
        const ulonglong2* pairs = reinterpret_cast<const ulonglong2*>(s_keys);
        // keys of lower index than every variate here count where they are not above, those of higher index where they are below
#pragma unroll 4
        for (int t = part; t < first; t += kParts) {
            const ulonglong2 o = pairs[t];
            const T x = as(o.x), y = as(o.y);
#pragma unroll
            for (int i = 0; i < kV; ++i) {
                if (x <= mine[i]) ++pos[i];
                if (y <= mine[i]) ++pos[i];
            }
        }
#pragma unroll 1
        for (int t = first + part; t < last; t += kParts) {
            const ulonglong2 o = pairs[t];
            const T x = as(o.x), y = as(o.y);
#pragma unroll
            for (int i = 0; i < kV; ++i) {
                const int n = base + (lane & 15) + 16 * i;
                pos[i] += (x < mine[i] || (x == mine[i] && 2 * t < n)) + (y < mine[i] || (y == mine[i] && 2 * t + 1 < n));
            }
        }
#pragma unroll 4
        for (int t = last + part; t < n_pairs; t += kParts) {
            const ulonglong2 o = pairs[t];
            const T x = as(o.x), y = as(o.y);
#pragma unroll
            for (int i = 0; i < kV; ++i) {
                if (x < mine[i]) ++pos[i];
                if (y < mine[i]) ++pos[i];
            }
        }
    };
    if (special) count([](uint64_t v) { return v; });
    else count([](uint64_t v) { return __longlong_as_double(static_cast<long long>(v)); });
#pragma unroll
    for (int i = 0; i < kV; ++i) {
        pos[i] += __shfl_xor_sync(0xffffffffu, pos[i], 16);
        if (lane < 16) atomicAdd(s_pos + lane + 16 * i, pos[i]);
    }
    __syncthreads();
    const int n = base + tid;
    if (tid < 16 * kV && n < N) {
        const size_t to = static_cast<size_t>(s) * N + s_pos[tid];
        P.sorted_keys[to] = s_keys[n];
        P.members[to] = n;
    }
}

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync() {
    cluster_arrive();
    cluster_wait();
}
// address of this CTA's shared variable `p` in CTA `cta` of the cluster
__device__ __forceinline__ uint32_t peer_addr(const void* p, int cta) {
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(cta));
    return a;
}
__device__ __forceinline__ void peer_store4(uint32_t a, int v) { asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory"); }
__device__ __forceinline__ void peer_store1(uint32_t a, int v) { asm volatile("st.shared::cluster.u8 [%0], %1;" ::"r"(a), "r"(v) : "memory"); }

template <int M>                                               // n_loc <= M
__global__ void __launch_bounds__(M) select_cluster_kernel(const SelectParams P, int n_loc, FastDiv div_loc) {
    constexpr int kWarps = M / 32;
    constexpr int kMaxLong = M / (kCountMaxGroup + 1) + 2;
    extern __shared__ __align__(16) unsigned char sm_raw[];
    uint32_t* prio = reinterpret_cast<uint32_t*>(sm_raw);      // [8 M] by sorted position: the CTA's own, and the rest of the groups that reach beyond them
    uint16_t* cand = reinterpret_cast<uint16_t*>(sm_raw + kClusterCtas * M * 4);       // [8 M]
    __shared__ LongGroups<kMaxLong> long_groups;
    __shared__ uint32_t bits[kWarps];                          // heads by own position; then kept flags by own variate
    __shared__ int cta_heads[kClusterCtas], cta_first[kClusterCtas], cta_last[kClusterCtas], cta_kept[kClusterCtas];
    __shared__ unsigned char kept[M];
    const int r = blockIdx.x, s = blockIdx.y, N = P.N, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int lo = r * n_loc, cnt = max(0, min(n_loc, N - lo)), p = lo + tid;
    const bool mine = tid < cnt;
    cluster_arrive();                                          // this CTA runs: its shared memory may be written (the others wait for it ahead of their first store)
    kept[tid] = 0;
#pragma unroll 1
    for (int i = tid; i < kMaxLong * kBuckets; i += M) long_groups.hist[i] = 0;
    if (tid == 0) long_groups.n = 0;
    chain_wait();
    chain_release();
    const uint64_t* keys = P.sorted_keys + static_cast<size_t>(s) * N;
    int32_t* gid = P.group_id + static_cast<size_t>(s) * N;
    int32_t* off = P.group_offsets + static_cast<size_t>(s) * (N + 1);
    int32_t* sel = P.sel_idx + static_cast<size_t>(s) * N;
    int32_t* inv = P.inv_idx + static_cast<size_t>(s) * N;
    auto below_lane = [&](uint32_t word) { return word & ((1u << lane) - 1u); };
    // this warp's sum over the warps before it, and the CTA's
    auto warp_prefix = [&](int* total) {
        const int v = lane < kWarps ? __popc(bits[lane]) : 0;
        int both = v << 16 | (lane < warp ? v : 0);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) both += __shfl_xor_sync(0xffffffffu, both, o);
        *total = both >> 16;
        return both & 0xFFFF;
    };

    // ---- group heads -----------------------------------------------------------------------------------------------
    const uint64_t key = mine ? __ldcg(keys + p) : 0ull, prev = mine && p > 0 ? __ldcg(keys + p - 1) : 0ull;
    const int n = mine ? __ldcg(P.members + static_cast<size_t>(s) * N + p) : 0;
    const uint32_t word = __ballot_sync(0xffffffffu, mine && (p == 0 || key != prev));
    if (lane == 0) bits[warp] = word;
    __syncthreads();
    int heads = 0;
    const int heads_before = warp_prefix(&heads);
    const uint32_t with_heads = __ballot_sync(0xffffffffu, lane < kWarps && bits[lane < kWarps ? lane : 0] != 0u);       // warps that hold a head
    cluster_wait();                                            // every CTA of the cluster runs (the launch chain and the keys' loads hide it)
    if (tid < kClusterCtas) {
        int first = N, last = -1;                              // the CTA's first and last head
        if (with_heads) {
            const int w0 = __ffs(with_heads) - 1, w1 = 31 - __clz(with_heads);
            first = lo + w0 * 32 + __ffs(bits[w0]) - 1;
            last = lo + w1 * 32 + 31 - __clz(bits[w1]);
        }
        peer_store4(peer_addr(cta_heads + r, tid), heads);
        peer_store4(peer_addr(cta_first + r, tid), first);
        peer_store4(peer_addr(cta_last + r, tid), last);
    }
    cluster_sync();
    // ---- group ids, places and priorities ----------------------------------------------------------------------------
    int groups = 0, heads_lower = 0, last_lower = -1, first_higher = N;
#pragma unroll
    for (int q = 0; q < kClusterCtas; ++q) {
        groups += cta_heads[q];
        if (q < r) { heads_lower += cta_heads[q]; last_lower = max(last_lower, cta_last[q]); }
        if (q > r) first_higher = min(first_higher, cta_first[q]);
    }
    const uint32_t upto = word & (0xFFFFFFFFu >> (31 - lane)), above = lane < 31 ? word >> (lane + 1) << (lane + 1) : 0u;
    const int g = heads_lower + heads_before + __popc(upto) - 1;
    int start = last_lower, end = first_higher;
    {
        const uint32_t lower = with_heads & ((1u << warp) - 1u), higher = warp < 31 ? with_heads >> (warp + 1) << (warp + 1) : 0u;
        if (upto) start = lo + warp * 32 + 31 - __clz(upto);
        else if (lower) { const int w = 31 - __clz(lower); start = lo + w * 32 + 31 - __clz(bits[w]); }
        if (above) end = lo + warp * 32 + __ffs(above) - 1;
        else if (higher) { const int w = __ffs(higher) - 1; end = lo + w * 32 + __ffs(bits[w]) - 1; }
    }
    auto priority = [&](int j, int group) {
        return philox4x32_10_word0(static_cast<uint32_t>(j), static_cast<uint32_t>(group), static_cast<uint32_t>(s), P.step, P.seed_lo, P.seed_hi);
    };
    const uint32_t pr = priority(p - start, g);
    if (mine) {
        prio[p] = pr;
        gid[n] = g;
        if (p == start) off[g] = p;
    }
    // the rest of the group that began before the CTA's positions, and of the one that ends behind them
    if (cnt > 0) {
        const int first_here = with_heads ? lo + (__ffs(with_heads) - 1) * 32 + __ffs(bits[__ffs(with_heads) - 1]) - 1 : N;
        if (first_here != lo) {
#pragma unroll 1
            for (int o = last_lower + tid; o < lo; o += M) prio[o] = priority(o - last_lower, heads_lower - 1);
        }
        const int w1 = 31 - __clz(with_heads), last_start = with_heads ? lo + w1 * 32 + 31 - __clz(bits[w1]) : last_lower;
#pragma unroll 1
        for (int o = lo + cnt + tid; o < first_higher; o += M) prio[o] = priority(o - last_start, heads_lower + heads - 1);
    }
    for (int i = groups + r * M + tid; i <= N; i += kClusterCtas * M) off[i] = N;
    if (r == 0 && tid == 0) P.n_groups[s] = groups;
    const int size = end - start, quota = quota_of(size, P.gs, P.rate_ppm);
    const bool is_long = mine && size > kCountMaxGroup && quota < size;
    if (is_long && p == max(start, lo)) add_long_group(long_groups, start, size, quota);
    // ---- sampling ranks ------------------------------------------------------------------------------------------------
    if (__syncthreads_or(is_long)) rank_long_groups<M>(long_groups, prio, cand);
    if (mine) {
        bool keep = quota == size;
        if (is_long) {
            keep = long_group_keeps(long_groups, prio, cand, start, p);
        } else if (!keep) {
            int below = 0;
#pragma unroll 4
            for (int o = start; o < p; ++o) below += prio[o] <= pr;        // equal priorities rank by place
#pragma unroll 4
            for (int o = p + 1; o < end; ++o) below += prio[o] < pr;
            keep = below < quota;
        }
        const int owner = static_cast<int>(fd_div(static_cast<uint32_t>(n), div_loc));
        if (keep) peer_store1(peer_addr(kept + (n - owner * n_loc), owner), 1);
    }
    cluster_sync();
    // ---- the kept variates in ascending order ----------------------------------------------------------------------------
    const uint32_t kept_word = __ballot_sync(0xffffffffu, kept[tid] != 0);
    if (lane == 0) bits[warp] = kept_word;
    __syncthreads();
    int kept_here = 0, base = warp_prefix(&kept_here), total = 0;
    if (tid < kClusterCtas) peer_store4(peer_addr(cta_kept + r, tid), kept_here);
    cluster_sync();
#pragma unroll
    for (int q = 0; q < kClusterCtas; ++q) {
        base += q < r ? cta_kept[q] : 0;
        total += cta_kept[q];
    }
    if (mine) {
        const bool keep = (kept_word >> lane) & 1u;
        const int pos = base + __popc(below_lane(kept_word));
        if (keep) sel[pos] = p;
        inv[p] = keep ? pos : -1;
    }
    for (int i = total + r * M + tid; i < N; i += kClusterCtas * M) sel[i] = -1;
    if (r == 0 && tid == 0) P.n_sel[s] = total;
}

struct SelectWs {
    size_t done2, lt, eq, prio, keep, total, zero_begin, zero_bytes;
};
SelectWs select_layout(int S, int N) {
    SelectWs w;
    size_t o = kWsHeaderBytes;
    w.zero_begin = o;
    w.done2 = o; o += align_up(sizeof(unsigned int) * S, 16);
    w.lt = o;    o += align_up(sizeof(int32_t) * S * N, 16);
    w.eq = o;    o += align_up(sizeof(int32_t) * S * N, 16);
    w.zero_bytes = o - w.zero_begin;
    w.prio = o;  o += align_up(sizeof(uint32_t) * S * N, 16);
    w.keep = o;  o += align_up(sizeof(int32_t) * S * N, 16);
    w.total = o;
    return w;
}

}  // namespace

int select_validate(const vardrop_select_cfg& c) {
    if (c.S < 1 || c.S > 65535) return fail(VARDROP_ERR_INVALID_ARG, "select: S=%d outside 1..65535", c.S);
    if (c.N < 1 || c.N > 65536) return fail(VARDROP_ERR_INVALID_ARG, "select: N=%d outside 1..65536", c.N);
    if (!(c.rate > 0.0) || c.rate > 1.0) return fail(VARDROP_ERR_INVALID_ARG, "select: rate=%g outside (0, 1]", c.rate);
    return VARDROP_OK;
}

size_t select_workspace_bytes(const vardrop_select_cfg& c) { return select_layout(c.S, c.N).total; }

int select_launch(const uint64_t* keys, const vardrop_select_cfg& c, int32_t* group_id, int32_t* group_offsets, int32_t* members,
                  int32_t* n_groups, int32_t* sel_idx, int32_t* n_sel, int32_t* inv_idx, void* ws, cudaStream_t stream, bool one_cta) {
    const SelectWs w = select_layout(c.S, c.N);
    char* base = static_cast<char*>(ws);
    SelectParams P{};
    P.keys = keys; P.group_id = group_id; P.group_offsets = group_offsets; P.members = members; P.n_groups = n_groups;
    P.sel_idx = sel_idx; P.n_sel = n_sel; P.inv_idx = inv_idx;
    P.status = reinterpret_cast<int*>(base);
    P.done2 = reinterpret_cast<unsigned int*>(base + w.done2);
    P.lt = reinterpret_cast<int32_t*>(base + w.lt);
    P.eq = reinterpret_cast<int32_t*>(base + w.eq);
    P.sorted_keys = reinterpret_cast<uint64_t*>(base + w.lt);
    P.prio = reinterpret_cast<uint32_t*>(base + w.prio);
    P.keep = reinterpret_cast<int32_t*>(base + w.keep);
    P.S = c.S; P.N = c.N; P.gs = c.gs;
    P.rate_ppm = llround(c.rate * 1.0e6);
    P.seed_lo = static_cast<uint32_t>(c.seed & 0xFFFFFFFFu);
    P.seed_hi = static_cast<uint32_t>(c.seed >> 32);
    P.step = c.step;
    // From 1025 variates two launches over more SMs do not depend on the groups, and take as long as one CTA a row does with few groups until the rows
    // are many.  In 40 | 200 | all groups, one CTA a row takes 6.4 | 8.1 | 18 us at 1025 variates and 8.4 | 10 | 20 at 2048, with any number of rows;
    // two launches take, at 1025, 7.1 | 6.5 | 5.5 for one row, 9.3 | 8.7 | 7.4 for four, 11.8 | 10.6 | 9.1 for eight; at 2048 8.0 | 7.5 | 6.4 for one,
    // 11.9 | 11.0 | 10.1 for four.
    // (one_cta: the caller's scratch is shared by calls that may overlap, and may not be touched up to 2048 variates.)
    const bool small = c.N <= 1024 || (c.N <= kSmallMaxN && (one_cta || c.S > kTwoLaunchRows));
    if (small) {
        auto launch = [&](auto m) {
            constexpr int kM = decltype(m)::value, table = small_layout(kM).total;
            constexpr int sorting = small_max_groups(kM) < kM ? kM * (8 + 4 + 4 + 4 + 4) + 16 : 0, smem = table > sorting ? table : sorting;
            static thread_local int attr_dev = -1;
            int dev = 0;
            cudaGetDevice(&dev);
            if (smem > 40 * 1024 && attr_dev != dev) {         // (48 KB without asking, some of it the kernel's own)
                if (int st = check_cuda(cudaFuncSetAttribute(select_small_kernel<kM>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem), "select: smem attribute")) return st;
                attr_dev = dev;
            }
            LaunchScope ls_(K_SELECT_SMALL, stream);
            return check_cuda(launch_chained(select_small_kernel<kM>, dim3(c.S), dim3(kM < 1024 ? kM : 1024), smem, stream, P), "select: launch");
        };
        using std::integral_constant;
        return c.N <= 64    ? launch(integral_constant<int, 64>{})
               : c.N <= 128 ? launch(integral_constant<int, 128>{})
               : c.N <= 256 ? launch(integral_constant<int, 256>{})
               : c.N <= 512 ? launch(integral_constant<int, 512>{})
               : c.N <= 1024 ? launch(integral_constant<int, 1024>{})
                             : launch(integral_constant<int, kSmallMaxN>{});
    }
    if (c.N <= kClusterMaxN) {
        using std::integral_constant;
        // variates a lane of the first launch: as many as leave most SMs a CTA
        const long long rows = static_cast<long long>(c.N) * c.S;
        auto place = [&](auto v) {
            constexpr int kV = decltype(v)::value;
            static thread_local int attr_dev = -1;
            int dev = 0;
            cudaGetDevice(&dev);
            if (attr_dev != dev) {
                if (int st = check_cuda(cudaFuncSetAttribute(select_place_kernel<kV>, cudaFuncAttributeMaxDynamicSharedMemorySize, kClusterMaxN * 8), "select: smem attribute")) return st;
                attr_dev = dev;
            }
            LaunchScope ls_(K_SELECT_PLACE, stream);
            return check_cuda(launch_chained(select_place_kernel<kV>, dim3((c.N + 16 * kV - 1) / (16 * kV), c.S), dim3(kPlaceThreads), (static_cast<size_t>(c.N) + 1) / 2 * 16, stream, P),
                              "select: place launch");
        };
        if (int st = rows <= 16ll * sm_count() ? place(integral_constant<int, 1>{}) : rows <= 32ll * sm_count() ? place(integral_constant<int, 2>{}) : place(integral_constant<int, 4>{})) return st;
        const int n_loc = ((c.N + kClusterCtas - 1) / kClusterCtas + 31) / 32 * 32;
        auto groups = [&](auto m) {
            constexpr int kM = decltype(m)::value, smem = kClusterCtas * kM * 6;
            static thread_local int attr_dev = -1;
            int dev = 0;
            cudaGetDevice(&dev);
            if (smem > 40 * 1024 && attr_dev != dev) {
                if (int st = check_cuda(cudaFuncSetAttribute(select_cluster_kernel<kM>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem), "select: smem attribute")) return st;
                attr_dev = dev;
            }
            LaunchScope ls_(K_SELECT_CLUSTER, stream);
            return check_cuda(launch_chained_clusters(kClusterCtas, select_cluster_kernel<kM>, dim3(kClusterCtas, c.S), dim3(kM), smem, stream, P, n_loc, make_fastdiv(n_loc)), "select: group launch");
        };
        return n_loc <= 256 ? groups(integral_constant<int, 256>{}) : n_loc <= 512 ? groups(integral_constant<int, 512>{}) : groups(integral_constant<int, 1024>{});
    }
    if (int st = check_cuda(cudaMemsetAsync(base + w.zero_begin, 0, w.zero_bytes, stream), "select: clear counters")) return st;
    const dim3 grid1((c.N + kSelThreads - 1) / kSelThreads, (c.N + kKeyChunk - 1) / kKeyChunk, c.S);
    cudaError_t err;
    { LaunchScope ls_(K_SELECT_COUNT, stream); err = launch_chained(select_count_kernel, grid1, dim3(kSelThreads), 0, stream, P); }
    if (int st = check_cuda(err, "select: count launch")) return st;
    const size_t group_smem = 3 * sizeof(int32_t) * static_cast<size_t>(c.N);
    if (group_smem <= kGroupMaxSmem) {
        static thread_local int group_attr_dev = -1;
        int dev = 0;
        cudaGetDevice(&dev);
        if (group_attr_dev != dev) {
            if (int st = check_cuda(cudaFuncSetAttribute(select_group_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kGroupMaxSmem)),
                                    "select: smem attribute")) return st;
            group_attr_dev = dev;
        }
        LaunchScope ls_(K_SELECT_GROUP, stream);
        err = launch_chained(select_group_kernel<true>, dim3(c.S), dim3(kTailThreads), group_smem, stream, P);
    } else {
        LaunchScope ls_(K_SELECT_GROUP, stream);
        err = launch_chained(select_group_kernel<false>, dim3(c.S), dim3(kTailThreads), 0, stream, P);
    }
    if (int st = check_cuda(err, "select: group launch")) return st;
    const dim3 grid2((c.N + kTailThreads - 1) / kTailThreads, 1, c.S);
    { LaunchScope ls_(K_SELECT_SAMPLE, stream); err = launch_chained(select_sample_kernel, grid2, dim3(kTailThreads), 0, stream, P); }
    return check_cuda(err, "select: sample launch");
}

// ---- allocation-free variant ------------------------------------------------------------------------------
// Scratch for vardrop_select_static: a fixed array that is part of the loaded module, so a caller that may not
// allocate device memory still has somewhere for the counters, ranks, priorities and keep flags to live.
// Sized for S * N <= kStaticMaxRows (worst case S = kStaticMaxRows, N = 1).
static __device__ __align__(256) unsigned char g_select_static_scratch[kStaticSelectBytes];

int select_static_launch(const uint64_t* keys, const vardrop_select_cfg& c, int32_t* group_id, int32_t* group_offsets, int32_t* members,
                         int32_t* n_groups, int32_t* sel_idx, int32_t* n_sel, int32_t* inv_idx, cudaStream_t stream) {
    if (static_cast<long long>(c.S) * c.N > kStaticMaxRows)
        return fail(VARDROP_ERR_UNSUPPORTED, "select_static: S*N = %lld exceeds the built-in scratch limit of %d; use vardrop_select with a workspace",
                    static_cast<long long>(c.S) * c.N, kStaticMaxRows);
    if (select_workspace_bytes(c) > static_cast<size_t>(kStaticSelectBytes))
        return fail(VARDROP_ERR_UNSUPPORTED, "select_static: layout of %zu bytes exceeds the built-in scratch of %d bytes",
                    select_workspace_bytes(c), kStaticSelectBytes);
    // The array's name is only a handle on the host; the device address is looked up once per device, with that
    // device current, and remembered.
    constexpr int kMaxDevices = 64;
    static std::mutex mu;
    static void* dev_ptr[kMaxDevices] = {};
    int dev = -1;
    if (int st = check_cuda(cudaGetDevice(&dev), "select_static: cudaGetDevice")) return st;
    if (dev < 0 || dev >= kMaxDevices) return fail(VARDROP_ERR_UNSUPPORTED, "select_static: device ordinal %d not supported", dev);
    void* ptr = nullptr;
    {
        std::lock_guard<std::mutex> lock(mu);
        if (!dev_ptr[dev]) {
            void* p = nullptr;
            if (int st = check_cuda(cudaGetSymbolAddress(&p, g_select_static_scratch), "select_static: cudaGetSymbolAddress")) return st;
            dev_ptr[dev] = p;
        }
        ptr = dev_ptr[dev];
    }
    return select_launch(keys, c, group_id, group_offsets, members, n_groups, sel_idx, n_sel, inv_idx, ptr, stream, true);
}

}  // namespace vardrop
