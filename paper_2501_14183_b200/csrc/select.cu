// Grouping by hash value and stratified sampling (Eq. 1, Eq. 2), without a spin-wait.
//
// Small problems (N <= 2048): one CTA per hash row does everything in shared memory (select_small_kernel).
// Larger ones take three launches:
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
#pragma unroll
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
// Small problems (N <= 2048): one CTA per hash row does everything in shared memory.
//
// More than 512, in few groups (the point of the method): the distinct keys are found with a hash table and ranked by counting, which gives the group ids; a
// variate's place in its group is the number of equal keys in the 32-variate chunks before its own plus those below it in the chunk; its
// sampling rank is counted over its group, or, with a long group, found by sorting (group, priority, place).
// Fewer variates, or many groups: two bitonic sorts.
//   sort 1: (key, variate)                      -> members, group heads -> ids, offsets
//   sort 2: (group id, Philox priority, rank j) -> position inside the group = sampling rank
// Then the kept flags are compacted with one scan.  No scratch in global memory, no global atomics.
// ---------------------------------------------------------------------------------------------------------
constexpr int kSmallMaxN = 2048;

// Bitonic sort of M (a power of two >= 64) items by M / 2 threads.  Thread t keeps items 2t and 2t + 1 in registers.
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

// exclusive scan of two values per thread (positions 2 tid and 2 tid + 1) over the CTA; returns the exclusive prefix
// of position 2 tid and the total
__device__ __forceinline__ int block_scan_pair(int v0, int v1, int* warp_sums, int* total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
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
    for (int w = 0; w < n_warps; ++w) {
        const int sw = warp_sums[w];
        if (w < warp) base += sw;
        tot += sw;
    }
    *total = tot;
    return v + base - v0 - v1;
}

// Most groups the counting path takes.  Ranking G keys is G^2 / 32 cycles; the sort does not depend on G.  Counting | sorting, 862 variates: 60 groups
// 7.2 | 8.8 us, 130 8.0 | 8.6, 160 8.4 | 8.7, 200 10.3 | 8.7; 2048 variates: 100 11.7 | 18.6, 300 15.6 | 17.6, 362 17.5 | 17.6, 420 19.8 | 17.6.  A call
// with more has paid for the table when it comes to sort: 862 distinct keys 9.7 us instead of 8.1, 2048 19.1 instead of 16.6.
__host__ __device__ constexpr int small_max_groups(int M) { return M <= 1024 ? 160 : 360; }
// Longest group whose sampling ranks are counted: 128 positions take some 4000 cycles, the sort of 1024 codes 8000.
constexpr int kCountMaxGroup = 128, kSortCountMaxGroup = 64;

// Shared memory of the counting path (the sorting path uses less, over it).
struct SmallLayout {
    int table, list, prio, size, off, count, slot_id, rank, quota, slot, place, member, entry, total;       // byte offsets
};
__host__ __device__ inline SmallLayout small_layout(int M) {
    SmallLayout l{};
    const int G = (small_max_groups(M) + 1) & ~1;
    int o = 0;
    l.table = o; o += 2 * M * 8;                   // [2M] keys
    l.list = o; o += G * 8;                        // [G] distinct keys, in any order: the entries
    l.prio = o; o += M * 4;                        // [M] priority by sorted position
    l.size = o; o += G * 4;                        // [G] members of an entry
    l.off = o; o += G * 4;                         // [G] sorted position of its first member
    l.count = o; o += M / 32 * G * 2;              // [M / 32][G] members of an entry in a chunk; then in the chunks before it
    l.slot_id = o; o += (2 * M + 2) * 2;           // [2M + 1] slot -> entry
    l.rank = o; o += G * 2;                        // [G] group id of an entry
    l.quota = o; o += G * 2;                       // [G] members of an entry to keep
    l.slot = o; o += M * 2;                        // [M] by variate: its slot, then its entry
    l.place = o; o += M;                           // [M] by variate: its place among the equal keys of its chunk
    l.member = o; o += M * 2;                      // [M] by sorted position: variate
    l.entry = o; o += M * 2;                       // [M] by sorted position: entry
    l.total = (o + 15) & ~15;
    return l;
}

// launched with M / 2 threads (M >= 64 a power of two, N <= M)
//
// What bounds it is latency: half a dozen short steps between barriers, each run once, at the speed of instruction fetch.  So the steps are
// few (sizes and offsets come out of the ranking of the distinct keys, without scans) and their loops rolled, with what a variate
// carries from step to step in shared memory.
// Measured, counting | sorting: 862 variates in one group 9.2 | 11.6 us, in 16 groups 7.5 | 11.8, in 60 7.2 | 8.8; 2048 in one 15.8 | 24.3; events around
// the launch, 32 rows of 321 11.6 | 10.7, 21 8.6 | 8.7: up to 512 items it sorts.
constexpr int kSortOnlyItems = 512;
template <bool kCounting>
__global__ void __launch_bounds__(kSmallMaxN / 2) select_small_kernel(const SelectParams P, int M) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    __shared__ int warp_sums[kSmallMaxN / 64];
    __shared__ uint32_t keep_bits[kSmallMaxN / 32];
    __shared__ int n_entries, all_ones;
    const int s = blockIdx.x, N = P.N, tid = threadIdx.x, T = blockDim.x, lane = tid & 31;
    const SmallLayout L = small_layout(M);
    const int G_max = small_max_groups(M), G_row = (G_max + 1) & ~1;
    constexpr uint64_t kEmpty = ~0ull;             // marks a free slot; as a key it has a slot of its own behind the table's
    uint64_t* table = reinterpret_cast<uint64_t*>(sm_raw + L.table);
    uint64_t* list = reinterpret_cast<uint64_t*>(sm_raw + L.list);
    uint32_t* prio = reinterpret_cast<uint32_t*>(sm_raw + L.prio);
    int* size_s = reinterpret_cast<int*>(sm_raw + L.size);
    int* first_s = reinterpret_cast<int*>(sm_raw + L.off);
    uint32_t* count2 = reinterpret_cast<uint32_t*>(sm_raw + L.count);              // two entries a word
    uint16_t* count = reinterpret_cast<uint16_t*>(sm_raw + L.count);
    uint16_t* slot_id = reinterpret_cast<uint16_t*>(sm_raw + L.slot_id);
    uint16_t* rank = reinterpret_cast<uint16_t*>(sm_raw + L.rank);
    uint16_t* quota_s = reinterpret_cast<uint16_t*>(sm_raw + L.quota);
    uint16_t* slot_s = reinterpret_cast<uint16_t*>(sm_raw + L.slot);
    unsigned char* place_s = sm_raw + L.place;
    uint16_t* member_s = reinterpret_cast<uint16_t*>(sm_raw + L.member);
    uint16_t* entry_s = reinterpret_cast<uint16_t*>(sm_raw + L.entry);
    if (kCounting) {
        for (int i = tid; i < M; i += T) reinterpret_cast<uint4*>(table)[i] = make_uint4(~0u, ~0u, ~0u, ~0u);
#pragma unroll 1
        for (int i = tid; i < M / 32 * (G_row / 2); i += T) count2[i] = 0u;
#pragma unroll 1
        for (int i = tid; i < G_row; i += T) size_s[i] = 0;
        if (tid < M / 32) keep_bits[tid] = 0u;
        if (tid == 0) { n_entries = 0; all_ones = 0; }
        __syncthreads();
    }
    chain_wait();
    chain_release();
    const uint64_t* keys = P.keys + static_cast<size_t>(s) * N;
    int32_t* members = P.members + static_cast<size_t>(s) * N;
    int32_t* gid = P.group_id + static_cast<size_t>(s) * N;
    int32_t* off = P.group_offsets + static_cast<size_t>(s) * (N + 1);
    int32_t* sel = P.sel_idx + static_cast<size_t>(s) * N;
    int32_t* inv = P.inv_idx + static_cast<size_t>(s) * N;

    if (kCounting) {
        // ---- the distinct keys: whoever takes a slot opens an entry --------------------------------------------
#pragma unroll 1
        for (int n = tid; n < N; n += T) {
            if (n >= T && *reinterpret_cast<volatile int*>(&n_entries) > G_max) break;       // too many already: to the sort
            const uint64_t key = keys[n];
            int at = 2 * M;
            bool mine = false;
            if (key == kEmpty) {
                mine = atomicExch(&all_ones, 1) == 0;
            } else {
                at = static_cast<int>((key * 0x9E3779B97F4A7C15ull) >> (64 - (31 - __clz(2 * M))));
#pragma unroll 1
                for (;;) {                             // at most half of the slots are ever taken
                    uint64_t cur = *reinterpret_cast<volatile uint64_t*>(table + at);
                    if (cur == kEmpty) {
                        cur = atomicCAS(reinterpret_cast<unsigned long long*>(table + at), kEmpty, key);
                        mine = cur == kEmpty;
                    }
                    if (mine || cur == key) break;
                    at = (at + 1) & (2 * M - 1);
                }
            }
            if (mine) {
                const int d = atomicAdd(&n_entries, 1);
                if (d < G_max) { list[d] = key; slot_id[at] = static_cast<uint16_t>(d); }
            }
            slot_s[n] = static_cast<uint16_t>(at);
        }
        __syncthreads();
        const int G = n_entries;
        if (G <= G_max) {
            // equal keys within a chunk of 32 consecutive variates
#pragma unroll 1
            for (int n = tid; n - lane < N; n += T) {
                const int d = n < N ? slot_id[slot_s[n]] : 0x10000 + lane;
                const unsigned same = __match_any_sync(0xffffffffu, d);
                if (n < N) {
                    const int place = __popc(same & ((1u << lane) - 1u));
                    slot_s[n] = static_cast<uint16_t>(d);
                    place_s[n] = static_cast<unsigned char>(place);
                    if (place == 0) {
                        count[(n >> 5) * G_row + d] = static_cast<uint16_t>(__popc(same));
                        atomicAdd(size_s + d, __popc(same));
                    }
                }
            }
            __syncthreads();
            // entries 2 i and 2 i + 1: members in the chunks before each chunk
            if (2 * tid < G) {
                uint32_t run = 0;
#pragma unroll 1
                for (int c = 0; c < (N + 31) / 32; c += 4) {
                    uint32_t v[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) v[i] = c + i < M / 32 ? count2[(c + i) * (G_row / 2) + tid] : 0u;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        if (c + i < M / 32) count2[(c + i) * (G_row / 2) + tid] = run;
                        run += v[i];
                    }
                }
            }
            // group id and first position of an entry: entries with smaller keys and their members, counted by `parts` lanes to an entry
            int parts_log = 0;
            while (parts_log < 5 && (G << (parts_log + 1)) <= T) ++parts_log;
            int longest = 0;
#pragma unroll 1
            for (int base = 0; base < (G << parts_log); base += T) {
                const int d = (base + tid) >> parts_log;
                uint32_t below = 0, before = 0;
                if (d < G) {
                    const uint64_t mine = list[d];
                    longest = max(longest, size_s[d]);
#pragma unroll 4
                    for (int e = tid & ((1 << parts_log) - 1); e < G; e += 1 << parts_log) {
                        const uint32_t less = list[e] < mine ? 1u : 0u;
                        below += less;
                        before += less * static_cast<uint32_t>(size_s[e]);
                    }
                }
                uint32_t both = below << 16 | before;          // below < 2^9, before <= 2^11
#pragma unroll 1
                for (int m = 1; m < 1 << parts_log; m <<= 1) both += __shfl_xor_sync(0xffffffffu, both, m);
                if (d < G && (tid & ((1 << parts_log) - 1)) == 0) {
                    rank[d] = static_cast<uint16_t>(both >> 16);
                    first_s[d] = static_cast<int>(both & 0xFFFFu);
                    quota_s[d] = static_cast<uint16_t>(quota_of(size_s[d], P.gs, P.rate_ppm));
                }
            }
            const bool long_group = __syncthreads_or(longest > kCountMaxGroup);
            // sorted positions
#pragma unroll 1
            for (int n = tid; n < N; n += T) {
                const int d = slot_s[n], g = rank[d], first = first_s[d];
                const int j = count[(n >> 5) * G_row + d] + place_s[n];
                prio[first + j] = philox4x32_10_word0(static_cast<uint32_t>(j), static_cast<uint32_t>(g), static_cast<uint32_t>(s), P.step, P.seed_lo, P.seed_hi);
                member_s[first + j] = static_cast<uint16_t>(n);
                entry_s[first + j] = static_cast<uint16_t>(d);
                gid[n] = g;
            }
            uint32_t* by_rank = reinterpret_cast<uint32_t*>(list);       // first position | quota << 16 of a group (the keys are no longer read)
            for (int d = tid; d < G; d += T) {
                off[rank[d]] = first_s[d];
                if (long_group) by_rank[rank[d]] = static_cast<uint32_t>(first_s[d]) | static_cast<uint32_t>(quota_s[d]) << 16;
            }
            for (int i = G + tid; i <= N; i += T) off[i] = N;
            if (tid == 0) P.n_groups[s] = G;
            __syncthreads();
            if (!long_group) {
                // sampling ranks, by sorted position: neighbours read the same priorities
#pragma unroll 1
                for (int p = tid; p < N; p += T) {
                    const int d = entry_s[p], begin = first_s[d], size = size_s[d], n = member_s[p];
                    members[p] = n;
                    const int quota = quota_s[d];
                    int below = 0;
                    if (quota < size) {
                        const uint32_t mine = prio[p];
#pragma unroll 8
                        for (int o = begin; o < begin + size; ++o) {
                            const uint32_t other = prio[o];
                            below += (other < mine) | ((other == mine) & (o < p));
                        }
                    }
                    if (below < quota) atomicOr(keep_bits + (n >> 5), 1u << (n & 31));
                }
            } else {
                // some group is long: the codes (group, priority, place) are sorted, over the hash table's slots
                uint64_t c[2];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int p = 2 * tid + e;
                    c[e] = ~0ull;
                    if (p < N) {
                        const int d = entry_s[p];
                        members[p] = member_s[p];
                        c[e] = static_cast<uint64_t>(rank[d]) << 43 | static_cast<uint64_t>(prio[p]) << 11 | static_cast<uint64_t>(p - first_s[d]);
                    }
                }
                uint32_t none0 = 0, none1 = 0;
                bitonic_sort_regs<false>(c[0], none0, c[1], none1, table, nullptr, M);
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int q = 2 * tid + e;
                    if (q < N) {
                        const uint32_t group = by_rank[c[e] >> 43];
                        const int begin = static_cast<int>(group & 0xFFFFu), n = member_s[begin + static_cast<int>(c[e] & 2047u)];
                        if (q - begin < static_cast<int>(group >> 16)) atomicOr(keep_bits + (n >> 5), 1u << (n & 31));
                    }
                }
            }
            __syncthreads();
            const uint32_t w0 = lane < M / 32 ? keep_bits[lane] : 0u, w1 = lane + 32 < M / 32 ? keep_bits[lane + 32] : 0u;
            const int v0 = __popc(w0), v1 = __popc(w1);
            const int total = __reduce_add_sync(0xffffffffu, v0 + v1);
#pragma unroll 1
            for (int n = tid; n - lane < N; n += T) {
                const int c = n >> 5;
                const int base = __reduce_add_sync(0xffffffffu, (lane < c ? v0 : 0) + (lane + 32 < c ? v1 : 0));
                const uint32_t word = keep_bits[c];
                const bool keep = (word >> lane) & 1u;
                const int pos = base + __popc(word & ((1u << lane) - 1u));
                if (keep) sel[pos] = n;
                if (n < N) inv[n] = keep ? pos : -1;
            }
            for (int i = total + tid; i < N; i += T) sel[i] = -1;
            if (tid == 0) P.n_sel[s] = total;
            return;
        }
    }

    // ---- the sorting path --------------------------------------------------------------------------------
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
    const int before = block_scan_pair(h0, h1, warp_sums, &groups);
    const int g0 = before + h0 - 1, g1 = before + h0 + h1 - 1;
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
    for (int i = groups + tid; i <= N; i += blockDim.x) off[i] = N;
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
    if (!__syncthreads_or(size0 > kSortCountMaxGroup || size1 > kSortCountMaxGroup)) {
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
    int pos = block_scan_pair(kp0, kp1, warp_sums, &total);
    if (p0 < N) { if (kp0) { sel[pos] = p0; inv[p0] = pos; ++pos; } else inv[p0] = -1; }
    if (p1 < N) { if (kp1) { sel[pos] = p1; inv[p1] = pos; } else inv[p1] = -1; }
    for (int i = total + tid; i < N; i += blockDim.x) sel[i] = -1;
    if (tid == 0) P.n_sel[s] = total;
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
                  int32_t* n_groups, int32_t* sel_idx, int32_t* n_sel, int32_t* inv_idx, void* ws, cudaStream_t stream) {
    const SelectWs w = select_layout(c.S, c.N);
    char* base = static_cast<char*>(ws);
    SelectParams P{};
    P.keys = keys; P.group_id = group_id; P.group_offsets = group_offsets; P.members = members; P.n_groups = n_groups;
    P.sel_idx = sel_idx; P.n_sel = n_sel; P.inv_idx = inv_idx;
    P.status = reinterpret_cast<int*>(base);
    P.done2 = reinterpret_cast<unsigned int*>(base + w.done2);
    P.lt = reinterpret_cast<int32_t*>(base + w.lt);
    P.eq = reinterpret_cast<int32_t*>(base + w.eq);
    P.prio = reinterpret_cast<uint32_t*>(base + w.prio);
    P.keep = reinterpret_cast<int32_t*>(base + w.keep);
    P.S = c.S; P.N = c.N; P.gs = c.gs;
    P.rate_ppm = llround(c.rate * 1.0e6);
    P.seed_lo = static_cast<uint32_t>(c.seed & 0xFFFFFFFFu);
    P.seed_hi = static_cast<uint32_t>(c.seed >> 32);
    P.step = c.step;
    if (c.N <= kSmallMaxN) {
        int M = 64;
        while (M < c.N) M <<= 1;
        const size_t sorting = static_cast<size_t>(M) * (8 + 4 + 4 + 4 + 4) + 16, counting = small_layout(M).total;
        const bool count = M > kSortOnlyItems;
        const size_t smem = count && counting > sorting ? counting : sorting;
        static thread_local int attr_dev = -1;
        int dev = 0;
        cudaGetDevice(&dev);
        if (attr_dev != dev) {
            if (int st = check_cuda(cudaFuncSetAttribute(select_small_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024), "select: smem attribute")) return st;
            attr_dev = dev;
        }
        cudaError_t err;
        { LaunchScope ls_(K_SELECT_SMALL, stream); err = launch_chained(count ? select_small_kernel<true> : select_small_kernel<false>, dim3(c.S), dim3(M / 2), smem, stream, P, M); }
        return check_cuda(err, "select: launch");
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
    return select_launch(keys, c, group_id, group_offsets, members, n_groups, sel_idx, n_sel, inv_idx, ptr, stream);
}

}  // namespace vardrop
