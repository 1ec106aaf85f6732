// Host-side plan of the transform in shared memory (hash_kernel): the radices of a length and the threads of a CTA.  Plain C++, no CUDA.
#pragma once

#include <initializer_list>

namespace vardrop {

constexpr int kMaxStages = 16;

// Radices in the order of the stages.  Prime factors above 7 come last, as stages of plain sums (behind a copy-in stage, radix 1, when there is
// no small factor to read the windows with).
struct RadixPlan {
    int n = 0, radix[kMaxStages] = {};
    bool wide = false;                           // has radices of 6 and 8 to 10
    bool sums = false;                           // has stages of plain sums
    void push(int r) { radix[n++] = r; }
    void push_sums(int rem) {
        if (rem > 1 && n == 0) push(1);
        for (int p = 11; rem > 1; p += 2)
            for (; rem % p == 0; rem /= p) { push(p); sums = true; }
    }
};

inline RadixPlan fours_and_primes(int L) {
    RadixPlan plan;
    for (int r : {4, 2, 3, 5, 7})
        for (; L % r == 0; L /= r) plan.push(r);
    plan.push_sums(L);
    return plan;
}

// Fewest stages: u twos go with a five to a radix of 10, v with a three to 6; the threes left make nines, the twos eights (and fours, where an eight
// would leave a single two: a stage more of two-point butterflies, and larger errors).
inline RadixPlan radices_to_ten(int L) {
    int exps[4] = {0, 0, 0, 0};
    const int primes[4] = {2, 3, 5, 7};
    for (int i = 0; i < 4; ++i)
        for (; L % primes[i] == 0; L /= primes[i]) ++exps[i];
    int tens = 0, sixes = 0, fewest = 99;
    for (int u = 0; u <= exps[0] && u <= exps[2]; ++u)
        for (int v = 0; u + v <= exps[0] && v <= exps[1]; ++v) {
            const int stages = v + (exps[0] - u - v + 2) / 3 + (exps[1] - v + 1) / 2;      // (a ten takes a five's place)
            if (stages < fewest) { fewest = stages; tens = u; sixes = v; }
        }
    int twos = exps[0] - tens - sixes, threes = exps[1] - sixes;
    RadixPlan plan;
    plan.wide = true;
    for (int i = 0; i < tens; ++i) plan.push(10);
    for (; threes >= 2; threes -= 2) plan.push(9);
    for (; twos >= 3 && twos != 4; twos -= 3) plan.push(8);
    for (int i = 0; i < sixes; ++i) plan.push(6);
    for (; twos >= 2; twos -= 2) plan.push(4);
    if (twos == 1) plan.push(2);
    if (threes == 1) plan.push(3);
    for (int i = tens; i < exps[2]; ++i) plan.push(5);
    for (int i = 0; i < exps[3]; ++i) plan.push(7);
    plan.push_sums(L);
    return plan;
}

// A stage is a pass over shared memory and a barrier, but the radices above 7 cost registers: they are taken where they save a stage.
// (Between other launches, with fours and primes and with them: 137 rows of 32 windows of 168 steps 6.5 -> 6.0 us, 862 of 16 of 250 16.6 -> 11.0, 200 of 8 of
// 1000 11.2 -> 9.1.  2500 rows of 4 of 140 steps, which save none: 8.0, and 11.9 with 8 more registers.)
// Not two eights for three fours: their stores conflict eight ways (862 rows of 16 of 64 steps 5.3 us, 5.7 so), and the error is 1 % larger.
inline RadixPlan radix_plan(int L) {
    const RadixPlan narrow = fours_and_primes(L), wide = radices_to_ten(L);
    const bool eights = wide.n == 2 && wide.radix[0] == 8 && wide.radix[1] == 8;
    return wide.n < narrow.n && !eights ? wide : narrow;
}

// Threads of a CTA.  transforms: of a pass; ctas: of the launch; smem: bytes a CTA; few_rows: passes are long because the rows are few.
inline int hash_threads(const RadixPlan& plan, int L, int transforms, int rows_per_cta, int ctas, int smem, bool few_rows, int sms) {
    int most = 1;                                // butterflies (plain sums: outputs) of the largest stage
    for (int i = 0; i < plan.n; ++i) {
        const int tasks = transforms * (plan.radix[i] > 10 ? L : L / plan.radix[i]);
        most = tasks > most ? tasks : most;
    }
    // By the rounds that the CTAs take: as far as shared memory goes, an SM holds nine of 128 threads and five of 256; of the narrow form, ten and five with plain
    // sums, twelve and six without.
    // 862 rows of 16 windows of 90 steps, 128 | 256 threads: 5.8 | 9.0 us; of 1000 steps, where five fit either way, 53.8 | 42.4.
    const int per_sm = (ctas + sms - 1) / sms, room = 227 * 1024 / (smem + 1024);
    auto rounds = [&](int n) {
        n = n < room ? n : room > 1 ? room : 1;
        return (per_sm + n - 1) / n;
    };
    const bool lean = !plan.wide && !plan.sums;
    if (per_sm > 2 && rounds(plan.wide ? 9 : lean ? 12 : 10) < rounds(lean ? 6 : 5) && most <= (rows_per_cta > 4 ? 384 : 512)) return 128;
    if (!plan.wide) {
        // A CTA that is mostly idle in its last round keeps others from the SM: 128 instead of 256 where that wastes less (2500 rows of 4 windows of 560 steps
        // in this form 27.1 -> 22.2 us); 512 for a long pass when CTAs are few.  Not with many rows to a CTA, which its warps rank one after the other
        // (10272 rows of one window of 45 steps 7.9 us with 256 threads, 8.3 with 128), nor where the CTAs are few anyway (100 rows of 2 of 945 steps
        // 6.3 | 7.6; with fewer than one an SM a stage of plain sums has a task for every output).
        const int tasks = transforms * (plan.sums && ctas < sms ? L : L / plan.radix[0]);
        auto idle = [&](int t) { return (tasks + t - 1) / t * t; };
        const bool small = tasks <= 128 || (ctas >= 8 * sms && 5 * idle(128) < 4 * idle(256));
        return few_rows && tasks > 256 ? 512 : small && rows_per_cta <= 4 ? 128 : 256;
    }
    // Up to two CTAs an SM as many threads as find work; with many rows to a CTA, or as many rounds either way, 256 but for the shortest stages.  Fitted to 900
    // calls of 32 to 1024 steps, 30 to 10272 rows and 1 to 32 windows a row, between other launches: 0.4 % above the best of 128, 256 and 512.
    // 100 rows of 2 of 1000 steps 6.4 | 5.7 | 5.6 us, 137 of 32 of 168 7.6 | 6.6 | 6.2, 2500 of 4 of 360 14.9 | 13.8 | 24.2.
    if (per_sm <= 2) return most <= 64 ? 128 : most <= 256 ? 256 : 512;
    return per_sm <= 4 || rows_per_cta > 4 || most > 192 ? 256 : 128;
}

}  // namespace vardrop
