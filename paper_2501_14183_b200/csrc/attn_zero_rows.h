// How the CTAs of the many-tile backward's last launch share out the rows of the gradients.  Plain C++, for the device and the host.
#pragma once

#ifdef __CUDACC__
#define VARDROP_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define VARDROP_HOST_DEVICE inline
#endif

namespace vardrop {

// Rows a CTA in 1/1024: `late` for every one and `more` for the first `n_early`.
struct RowShares {
    int rows, ctas, n_early;
    long long late, more;
};
// `wanted` rows more for each of the first n_early CTAs, as long as the others keep their part of an even share.
VARDROP_HOST_DEVICE RowShares row_shares(int rows, int ctas, int n_early, float wanted) {
    const float even = static_cast<float>(rows) / ctas, most = even * (ctas - n_early) / (n_early > 1 ? n_early : 1);
    const float more = n_early == 0 ? 0.f : wanted < most ? wanted : most;
    return {rows, ctas, n_early, static_cast<long long>(1024.f * (even - more * n_early / ctas)), static_cast<long long>(1024.f * more)};
}
// First row of CTA c, and the end of CTA c - 1: in whole numbers, so that both come to the same one.  (The sum in floating point, as it was, depends on which
// of its products the compiler fuses, for one boundary in 1600.)
VARDROP_HOST_DEVICE int first_row(const RowShares& s, int c) {
    if (c >= s.ctas) return s.rows;
    const long long at = (c * s.late + (c < s.n_early ? c : s.n_early) * s.more) >> 10;
    return at < s.rows ? static_cast<int>(at) : s.rows;
}

}  // namespace vardrop
