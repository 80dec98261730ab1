// Small DFTs on registers, in FP32 or FP64, with compile-time twiddles: the building blocks of
// every FFT kernel whose length is split into factors of at most 20.
#pragma once

#include "common.cuh"

namespace hmc {

// cos and sin of 2 pi m / R at compile time. The angle is reduced to at most pi / 4 in whole
// numbers (the quadrant of 4 m / R, then the complement past half a quadrant), where the Taylor
// sums below, taken from the smallest term up, are good to the last bit or so.
constexpr double kPi = 3.14159265358979323846264338327950288;
__host__ __device__ constexpr double ct_sin_series(double x) {   // |x| <= pi / 4
    double s = 1.0;
    for (int n = 11; n >= 1; --n) s = 1.0 - x * x / ((2.0 * n) * (2.0 * n + 1.0)) * s;
    return x * s;
}
__host__ __device__ constexpr double ct_cos_series(double x) {
    double s = 1.0;
    for (int n = 11; n >= 1; --n) s = 1.0 - x * x / ((2.0 * n - 1.0) * (2.0 * n)) * s;
    return s;
}
__host__ __device__ constexpr double ct_cos2pi(int m, int R) {
    m %= R;
    if (m < 0) m += R;
    const int q = 4 * m / R, rem = 4 * m - q * R;   // quadrant; angle past it: (pi / 2) rem / R
    const bool flip = 2 * rem > R;
    const double x = 0.5 * kPi * (flip ? R - rem : rem) / R;
    const double c = flip ? ct_sin_series(x) : ct_cos_series(x), s = flip ? ct_cos_series(x) : ct_sin_series(x);
    return q == 0 ? c : q == 1 ? -s : q == 2 ? -c : s;
}
__host__ __device__ constexpr double ct_sin2pi(int m, int R) {
    m %= R;
    if (m < 0) m += R;
    const int q = 4 * m / R, rem = 4 * m - q * R;
    const bool flip = 2 * rem > R;
    const double x = 0.5 * kPi * (flip ? R - rem : rem) / R;
    const double c = flip ? ct_sin_series(x) : ct_cos_series(x), s = flip ? ct_cos_series(x) : ct_sin_series(x);
    return q == 0 ? s : q == 1 ? c : q == 2 ? -s : -c;
}
template <typename T, int R> struct TwR { T c[R], s[R]; };   // cos, sin of 2 pi m / R
template <typename T, int R> __host__ __device__ constexpr TwR<T, R> make_tw() {
    TwR<T, R> t{};
    for (int m = 0; m < R; ++m) { t.c[m] = (T)ct_cos2pi(m, R); t.s[m] = (T)ct_sin2pi(m, R); }
    return t;
}

template <typename C> struct RealOf;
template <> struct RealOf<float2> { using T = float; };
template <> struct RealOf<double2> { using T = double; };

template <typename C, typename T> __device__ __forceinline__ C mulcs(C a, T c, T s) {   // a * (c + i s)
    C o;
    o.x = a.x * c - a.y * s;
    o.y = a.x * s + a.y * c;
    return o;
}

// a * (DIR i)^q: a product with these twiddles would keep its multiplications by 0
template <int DIR, typename C> __device__ __forceinline__ C turn(C a, int q) {
    q &= 3;
    if (q == 0) return a;
    if (q == 2) return mk<C>(-a.x, -a.y);
    return (q == 1) == (DIR > 0) ? mk<C>(-a.y, a.x) : mk<C>(a.y, -a.x);
}

// Prime-size DFTs on registers: v[p] <- sum_q v[q] w^{pq}, w = e^{DIR 2 pi i / R}.
template <int R, int DIR, typename C>
__device__ __forceinline__ void bfly_prime(C* v) {
    using T = typename RealOf<C>::T;
    if constexpr (R == 2) {
        const C a = v[0], b = v[1];
        v[0] = cadd(a, b);
        v[1] = csub(a, b);
    } else if constexpr (R == 4) {
        const C a = v[0], b = v[1], c = v[2], d = v[3];
        const C s0 = cadd(a, c), s1 = csub(a, c), s2 = cadd(b, d), s3 = csub(b, d);
        const C s3r = mk<C>(-DIR * s3.y, DIR * s3.x);   // s3 * (DIR i)
        v[0] = cadd(s0, s2);
        v[2] = csub(s0, s2);
        v[1] = cadd(s1, s3r);
        v[3] = csub(s1, s3r);
    } else if constexpr (R == 3) {
        // X1,2 = v0 - (v1 + v2)/2 +- DIR i (sqrt3/2)(v1 - v2)
        constexpr T h = (T)ct_sin2pi(1, 3);
        const C t1 = cadd(v[1], v[2]), e = csub(v[1], v[2]);
        const T dx = DIR * h * e.x, dy = DIR * h * e.y;
        const T mx = v[0].x - (T)0.5 * t1.x, my = v[0].y - (T)0.5 * t1.y;
        v[0] = cadd(v[0], t1);
        v[1].x = mx - dy; v[1].y = my + dx;
        v[2].x = mx + dy; v[2].y = my - dx;
    } else if constexpr (R == 5) {
        // pairs (1, 4) and (2, 3): X_{1,4} = m1 +- i n1, X_{2,3} = m2 +- i n2
        constexpr T c1 = (T)ct_cos2pi(1, 5), c2 = (T)ct_cos2pi(2, 5);
        constexpr T s1 = (T)ct_sin2pi(1, 5), s2 = (T)ct_sin2pi(2, 5);
        const C a1 = cadd(v[1], v[4]), a2 = cadd(v[2], v[3]), b1 = csub(v[1], v[4]), b2 = csub(v[2], v[3]);
        const T m1x = v[0].x + c1 * a1.x + c2 * a2.x, m1y = v[0].y + c1 * a1.y + c2 * a2.y;
        const T m2x = v[0].x + c2 * a1.x + c1 * a2.x, m2y = v[0].y + c2 * a1.y + c1 * a2.y;
        const T n1x = DIR * (s1 * b1.x + s2 * b2.x), n1y = DIR * (s1 * b1.y + s2 * b2.y);
        const T n2x = DIR * (s2 * b1.x - s1 * b2.x), n2y = DIR * (s2 * b1.y - s1 * b2.y);
        v[0] = cadd(v[0], cadd(a1, a2));
        v[1].x = m1x - n1y; v[1].y = m1y + n1x;
        v[4].x = m1x + n1y; v[4].y = m1y - n1x;
        v[2].x = m2x - n2y; v[2].y = m2y + n2x;
        v[3].x = m2x + n2y; v[3].y = m2y - n2x;
    } else {
        // odd R: pairs (q, R - q): with a = v_q + v_{R-q}, b = v_q - v_{R-q},
        // X_{p, R-p} = v0 + sum_q cos(2 pi p q / R) a_q +- DIR i sum_q sin(2 pi p q / R) b_q
        static_assert(R % 2 == 1, "odd prime");
        constexpr TwR<T, R> W = make_tw<T, R>();
        constexpr int H = R / 2;
        C a[H], b[H];
        C s0 = v[0];
#pragma unroll
        for (int q = 0; q < H; ++q) {
            a[q] = cadd(v[q + 1], v[R - 1 - q]);
            b[q] = csub(v[q + 1], v[R - 1 - q]);
            s0 = cadd(s0, a[q]);
        }
#pragma unroll
        for (int p = 1; p <= H; ++p) {
            C m = v[0], n = mk<C>(0, 0);
#pragma unroll
            for (int q = 0; q < H; ++q) {
                const T c = W.c[(p * (q + 1)) % R], s = DIR * W.s[(p * (q + 1)) % R];
                m.x += c * a[q].x; m.y += c * a[q].y;
                n.x += s * b[q].x; n.y += s * b[q].y;
            }
            // both outputs need v[0] only; v[p] and v[R - p] are already folded into a, b
            v[p].x = m.x - n.y; v[p].y = m.y + n.x;
            v[R - p].x = m.x + n.y; v[R - p].y = m.y - n.x;
        }
        v[0] = s0;
    }
}

// R = R1 * R2 point DFT on registers by one Cooley-Tukey split: with n = n1 + R1 n2 and
// k = k2 + R2 k1, X[k] = sum_n1 w_R1^{n1 k1} w_R^{n1 k2} sum_n2 v[n] w_R2^{n2 k2}.
template <int R1, int R2, int DIR, typename C>
__device__ __forceinline__ void bfly_split(C* v) {
    using T = typename RealOf<C>::T;
    constexpr int R = R1 * R2;
    constexpr TwR<T, R> W = make_tw<T, R>();
    C u[R];
#pragma unroll
    for (int n1 = 0; n1 < R1; ++n1) {
        C w[R2];
#pragma unroll
        for (int n2 = 0; n2 < R2; ++n2) w[n2] = v[n1 + R1 * n2];
        bfly_prime<R2, DIR>(w);
#pragma unroll
        for (int k2 = 0; k2 < R2; ++k2)
            u[n1 * R2 + k2] = (4 * n1 * k2) % R == 0
                                  ? turn<DIR>(w[k2], 4 * n1 * k2 / R)
                                  : mulcs(w[k2], W.c[(n1 * k2) % R], (T)DIR * W.s[(n1 * k2) % R]);
    }
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) {
        C z[R1];
#pragma unroll
        for (int n1 = 0; n1 < R1; ++n1) z[n1] = u[n1 * R2 + k2];
        bfly_prime<R1, DIR>(z);
#pragma unroll
        for (int k1 = 0; k1 < R1; ++k1) v[k2 + R2 * k1] = z[k1];
    }
}

// R = R1 * R2 with coprime factors: the index maps n = R2 a + R1 b and k = k1 (mod R1), k2 (mod R2) leave no
// twiddles between the two steps (Good, 1958; Thomas, 1963).
__host__ __device__ constexpr int crt(int k1, int R1, int k2, int R2) {
    for (int k = 0; k < R1 * R2; ++k)
        if (k % R1 == k1 && k % R2 == k2) return k;
    return 0;
}
template <int R1, int R2, int DIR, typename C>
__device__ __forceinline__ void bfly_coprime(C* v) {
    constexpr int R = R1 * R2;
    C u[R];
#pragma unroll
    for (int b = 0; b < R2; ++b) {
        C w[R1];
#pragma unroll
        for (int a = 0; a < R1; ++a) w[a] = v[(R2 * a + R1 * b) % R];
        bfly_prime<R1, DIR>(w);
#pragma unroll
        for (int a = 0; a < R1; ++a) u[a * R2 + b] = w[a];
    }
#pragma unroll
    for (int a = 0; a < R1; ++a) {
        C w[R2];
#pragma unroll
        for (int b = 0; b < R2; ++b) w[b] = u[a * R2 + b];
        bfly_prime<R2, DIR>(w);
#pragma unroll
        for (int b = 0; b < R2; ++b) v[crt(a, R1, b, R2)] = w[b];
    }
}

template <int R, int DIR, typename C>
__device__ __forceinline__ void bfly(C* v) {
    if constexpr (R == 2 || R == 3 || R == 4 || R == 5 || R == 7) bfly_prime<R, DIR>(v);
    else if constexpr (R == 6) bfly_coprime<2, 3, DIR>(v);
    else if constexpr (R == 8) bfly_split<2, 4, DIR>(v);
    else if constexpr (R == 9) bfly_split<3, 3, DIR>(v);
    else if constexpr (R == 10) bfly_coprime<2, 5, DIR>(v);
    else if constexpr (R == 12) bfly_coprime<4, 3, DIR>(v);
    else if constexpr (R == 14) bfly_coprime<2, 7, DIR>(v);
    else if constexpr (R == 15) bfly_coprime<3, 5, DIR>(v);
    else if constexpr (R == 16) bfly_split<4, 4, DIR>(v);
    else if constexpr (R == 20) bfly_coprime<4, 5, DIR>(v);
    else static_assert(R == 2, "unsupported radix");
}

}  // namespace hmc
