// Short DFTs in registers, every index and twiddle a compile-time constant.
#pragma once

#include "common.cuh"

namespace vardrop {

namespace {

// ---- compile-time trigonometry ------------------------------------------------------------------------------
namespace ct {
constexpr double kPi = 3.14159265358979323846264338327950288;
constexpr double sin_small(double x) {          // |x| <= pi / 4
    const double x2 = x * x;
    double term = x, sum = x;
    for (int i = 1; i <= 12; ++i) {
        term *= -x2 / static_cast<double>((2 * i) * (2 * i + 1));
        sum += term;
    }
    return sum;
}
constexpr double cos_small(double x) {
    const double x2 = x * x;
    double term = 1.0, sum = 1.0;
    for (int i = 1; i <= 12; ++i) {
        term *= -x2 / static_cast<double>((2 * i - 1) * (2 * i));
        sum += term;
    }
    return sum;
}
// cos and sin of 2 pi num / den for 0 <= num < den, reduced to the first half-quadrant with integers
constexpr double cos_turn(long long num, long long den);
constexpr double sin_turn(long long num, long long den) {
    if (2 * num > den) return -sin_turn(den - num, den);            // sin(2 pi - a) = -sin a
    if (4 * num > den) return sin_turn(den - 2 * num, 2 * den);     // sin(pi - a) = sin a ; (den/2 - num)/den = (den - 2 num)/(2 den)
    if (8 * num > den) return cos_turn(den - 4 * num, 4 * den);     // sin a = cos(pi/2 - a)
    return sin_small(2.0 * kPi * static_cast<double>(num) / static_cast<double>(den));
}
constexpr double cos_turn(long long num, long long den) {
    if (2 * num > den) return cos_turn(den - num, den);
    if (4 * num > den) return -cos_turn(den - 2 * num, 2 * den);
    if (8 * num > den) return sin_turn(den - 4 * num, 4 * den);
    return cos_small(2.0 * kPi * static_cast<double>(num) / static_cast<double>(den));
}
}  // namespace ct

template <int NUM, int DEN>
struct Turn {                                   // cos and sin of 2 pi NUM / DEN as float constants
    static constexpr float c = static_cast<float>(ct::cos_turn(NUM, DEN));
    static constexpr float s = static_cast<float>(ct::sin_turn(NUM, DEN));
};

// m2 = 2 m for the angle 2 pi m / L, folded to |m| <= L / 2.
__device__ __forceinline__ float folded_half_turns(int m, int L) { return static_cast<float>(2 * (2 * m > L ? m - L : m)); }
// cos and sin of pi m2 / L to their last bit; turn: m2 / L to a rounding or two.  What it is off by (known exactly from its product with L) is put in after.
__device__ __forceinline__ float2 cos_sin_turn(float m2, float turn, int L, float inv_L) {
    const float rest = fmaf(-turn, static_cast<float>(L), m2) * (3.14159265f * inv_L);
    float s, c;
    sincospif(turn, &s, &c);
    return make_float2(fmaf(-s, rest, c), fmaf(c, rest, s));
}

template <int I>
struct Int {
    static constexpr int value = I;
};
template <int B, int E, class F>
__device__ __forceinline__ void static_for(F&& f) {
    if constexpr (B < E) {
        f(Int<B>{});
        static_for<B + 1, E>(f);
    }
}

// Complex sums and differences as one packed instruction each (two IEEE fp32 results per issue slot: the kernel is bound by
// instruction issue, not by the fp32 pipe).
__device__ __forceinline__ unsigned long long pack_c(float2 a) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a.x), "f"(a.y));
    return r;
}
__device__ __forceinline__ float2 unpack_c(unsigned long long v) {
    float2 a;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a.x), "=f"(a.y) : "l"(v));
    return a;
}
__device__ __forceinline__ float2 cadd(float2 a, float2 b) {
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(pack_c(a)), "l"(pack_c(b)));
    return unpack_c(d);
}
__device__ __forceinline__ float2 csub(float2 a, float2 b) {
    unsigned long long d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(pack_c(a)), "l"(pack_c(b)));
    return unpack_c(d);
}

// v * exp(-2 pi i NUM / DEN)
template <int NUM, int DEN>
__device__ __forceinline__ float2 rotate(float2 v) {
    constexpr int n = ((NUM % DEN) + DEN) % DEN;
    if constexpr (n == 0) return v;
    else if constexpr (4 * n == DEN) return make_float2(v.y, -v.x);
    else if constexpr (2 * n == DEN) return make_float2(-v.x, -v.y);
    else if constexpr (4 * n == 3 * DEN) return make_float2(-v.y, v.x);
    else {
        constexpr float c = Turn<n, DEN>::c, s = Turn<n, DEN>::s;
        return make_float2(fmaf(v.y, s, v.x * c), fmaf(-v.x, s, v.y * c));
    }
}

// ---- prime-size butterflies: y_m = sum_j v_j exp(-2 pi i j m / R), in place --------------------------------
template <int R>
__device__ __forceinline__ void butterfly(float2* v);

template <>
__device__ __forceinline__ void butterfly<2>(float2* v) {
    const float2 a = v[0], b = v[1];
    v[0] = cadd(a, b);
    v[1] = csub(a, b);
}
template <>
__device__ __forceinline__ void butterfly<4>(float2* v) {
    const float2 s02 = cadd(v[0], v[2]), d02 = csub(v[0], v[2]);
    const float2 s13 = cadd(v[1], v[3]), d13 = csub(v[1], v[3]);
    v[0] = cadd(s02, s13);
    v[2] = csub(s02, s13);
    v[1] = make_float2(d02.x + d13.y, d02.y - d13.x);
    v[3] = make_float2(d02.x - d13.y, d02.y + d13.x);
}
// odd prime: pair j with R - j;  y_m = a_m - i b_m,  y_{R-m} = a_m + i b_m  with
// a_m = v_0 + sum_j cos(2 pi j m / R) (v_j + v_{R-j}),  b_m = sum_j sin(2 pi j m / R) (v_j - v_{R-j})
template <int R>
__device__ __forceinline__ void odd_butterfly(float2* v) {
    constexpr int Hh = (R - 1) / 2;
    float2 p[Hh], m[Hh];
    static_for<0, Hh>([&](auto J) {
        constexpr int j = decltype(J)::value;
        p[j] = cadd(v[j + 1], v[R - 1 - j]);
        m[j] = csub(v[j + 1], v[R - 1 - j]);
    });
    float2 out[R];
    out[0] = v[0];
    static_for<0, Hh>([&](auto J) { out[0] = cadd(out[0], p[decltype(J)::value]); });
    static_for<1, Hh + 1>([&](auto M) {
        constexpr int mm = decltype(M)::value;
        float2 a = v[0], b = make_float2(0.f, 0.f);
        static_for<1, Hh + 1>([&](auto J) {
            constexpr int j = decltype(J)::value;
            constexpr int idx = (j * mm) % R;
            constexpr float c = Turn<idx, R>::c, s = Turn<idx, R>::s;
            a.x = fmaf(c, p[j - 1].x, a.x);
            a.y = fmaf(c, p[j - 1].y, a.y);
            b.x = fmaf(s, m[j - 1].x, b.x);
            b.y = fmaf(s, m[j - 1].y, b.y);
        });
        out[mm] = make_float2(a.x + b.y, a.y - b.x);
        out[R - mm] = make_float2(a.x - b.y, a.y + b.x);
    });
    static_for<0, R>([&](auto J) { v[decltype(J)::value] = out[decltype(J)::value]; });
}
template <>
__device__ __forceinline__ void butterfly<3>(float2* v) { odd_butterfly<3>(v); }
template <>
__device__ __forceinline__ void butterfly<5>(float2* v) { odd_butterfly<5>(v); }
template <>
__device__ __forceinline__ void butterfly<7>(float2* v) { odd_butterfly<7>(v); }

template <int N>
struct Radix {                                  // outermost radix of the decimation
    static constexpr int value = N % 4 == 0 ? 4 : N % 2 == 0 ? 2 : N % 3 == 0 ? 3 : N % 5 == 0 ? 5 : 7;
};

// N-point DFT of in[0], in[IS], ... to out[0], out[OS], ... (decimation in time; all indices are constants)
template <int N, int IS, int OS>
__device__ __forceinline__ void dft(const float2* in, float2* out) {
    if constexpr (N == 1) {
        out[0] = in[0];
    } else if constexpr (N == 2 || N == 3 || N == 4 || N == 5 || N == 7) {
        float2 v[N];
        static_for<0, N>([&](auto J) { v[decltype(J)::value] = in[decltype(J)::value * IS]; });
        butterfly<N>(v);
        static_for<0, N>([&](auto J) { out[decltype(J)::value * OS] = v[decltype(J)::value]; });
    } else {
        constexpr int R = Radix<N>::value, M = N / R;
        static_assert(R * M == N, "length must factor into 2, 3, 5, 7");
        float2 sub[N];                                       // sub[r M + k]: DFT of the samples congruent to r
        static_for<0, R>([&](auto Rr) {
            constexpr int r = decltype(Rr)::value;
            dft<M, IS * R, 1>(in + r * IS, sub + r * M);
        });
        static_for<0, M>([&](auto K) {
            constexpr int k = decltype(K)::value;
            float2 v[R];
            static_for<0, R>([&](auto Rr) {
                constexpr int r = decltype(Rr)::value;
                v[r] = rotate<r * k, N>(sub[r * M + k]);
            });
            butterfly<R>(v);
            static_for<0, R>([&](auto Q) {
                constexpr int q = decltype(Q)::value;
                out[(k + M * q) * OS] = v[q];
            });
        });
    }
}

}  // namespace

}  // namespace vardrop
