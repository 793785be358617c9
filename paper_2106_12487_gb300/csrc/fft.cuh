// Register DFTs of small radices and the radix schedule of an axis.
//
// Radix kernels: powers of two (2..16) by unrolled radix-2 decimation in time
// with literal twiddles; 3, 5, 7 from the symmetric and antisymmetric parts of
// their inputs with literal cosines and sines; 6, 10, 12, 14, 15 as coprime
// products of those by the prime-factor map of Good (1958), which needs no
// twiddles; 9 as 3 x 3.
// Direction: DIR = -1 forward (exp(-2 pi i ...)), DIR = +1 inverse; both
// unnormalised.
#pragma once

#include <type_traits>

#include "common.cuh"

namespace bloch {

// Division of n < 2^31 by an invariant divisor d >= 1 with one high multiply,
// an add and a shift (Granlund & Montgomery 1994, division by invariant
// integers): l = ceil(log2 d), m = floor(2^32 (2^l - d) / d) + 1,
// n / d = (umulhi(m, n) + n) >> l.
struct FastDiv {
    unsigned m = 1;
    int l = 0;
};
inline FastDiv make_fastdiv(unsigned d) {
    FastDiv f;
    int l = 0;
    while ((1ull << l) < (unsigned long long)d) ++l;
    f.l = l;
    f.m = (unsigned)((((1ull << 32) * ((1ull << l) - d)) / d) + 1);
    return f;
}
__device__ __forceinline__ unsigned fdiv(unsigned n, const FastDiv& f) { return (__umulhi(f.m, n) + n) >> f.l; }

// Radix schedule N = r1 * r2 * r3 of an axis (r2 = 1: two stages).  The first
// and the last radix come from {1..10, 12, 14, 15, 16} (float-float: without
// 12 and 14), the middle one from {1, 3, 5, 6, 7, 8} (float-float: and 4); every
// length up to 512 with prime factors in {2,3,5,7} has one.
struct AxisPlan {
    int N;
    int r1, r2, r3;
    FastDiv d1, d2, d3;      // division by the radices
    FastDiv m1, m2, m3;      // division by N / radix (butterflies of a stage per pencil)
};

// cos(2 pi m / 16), m taken modulo 16
template <typename R>
__device__ __forceinline__ R cos16(int m) {
    switch (m & 15) {
        case 0: return R(1.0);
        case 1: case 15: return R(0.92387953251128675613);
        case 2: case 14: return R(0.70710678118654752440);
        case 3: case 13: return R(0.38268343236508977173);
        case 4: case 12: return R(0.0);
        case 5: case 11: return R(-0.38268343236508977173);
        case 6: case 10: return R(-0.70710678118654752440);
        case 7: case 9: return R(-0.92387953251128675613);
        default: return R(-1.0);
    }
}

// float-float values: hi = cos rounded to float, lo = the rounded remainder
template <>
__device__ __forceinline__ dfloat cos16<dfloat>(int m) {
    switch (m & 15) {
        case 0: return dfloat(1.0f, 0.0f);
        case 1: case 15: return dfloat(0.9238795042037964f, 2.830748968563057e-08f);
        case 2: case 14: return dfloat(0.7071067690849304f, 1.2101617485882343e-08f);
        case 3: case 13: return dfloat(0.3826834261417389f, 6.2233507236442165e-09f);
        case 4: case 12: return dfloat(0.0f, 0.0f);
        case 5: case 11: return dfloat(-0.3826834261417389f, -6.2233507236442165e-09f);
        case 6: case 10: return dfloat(-0.7071067690849304f, -1.2101617485882343e-08f);
        case 7: case 9: return dfloat(-0.9238795042037964f, -2.830748968563057e-08f);
        default: return dfloat(-1.0f, 0.0f);
    }
}

// x * exp(DIR * 2 pi i k / R) for power-of-two R <= 16 (k compile-time after unrolling)
template <int R, int DIR, typename C>
__device__ __forceinline__ C twiddle_pow2(C x, int k) {
    using T = decltype(x.x);
    if (k == 0) return x;
    if (4 * k == R) return cmul_i<DIR>(x);
    const int m = k * (16 / R);
    const T c = cos16<T>(m);
    const T s = T(DIR) * cos16<T>(m - 4);   // sin(2 pi m/16) = cos(2 pi (m-4)/16)
    if constexpr (std::is_same<T, dfloat>::value) {
        if ((m & 3) == 2) {   // 45 and 135 degrees: sum first, then one product each (four roundings, not six)
            const C d = mk(x.x - x.y, x.y + x.x), e = mk(x.x + x.y, x.y - x.x);
            // times c (1 + DIR i), with cos = sin (45 degrees) or cos = -sin (135)
            return cscale((DIR > 0) == (m == 2) ? d : e, c);
        }
    }
    return cmul(x, mk(c, s));
}

// Butterfly v_k = e + w o, v_{k+H} = e - w o with w = exp(DIR 2 pi i k / R), k
// and R compile time.  With w = m (1 + i t) or m (t + i), |t| <= 1, the product
// costs two fused multiply-adds and both outputs two each: 6 instead of 8
// operations (Linzer & Feig 1993).  Float-float has no fused multiply-add to
// gain from and keeps the plain product.
template <int R, int DIR, typename C>
__device__ __forceinline__ void butterfly(C e, C o, int k, C& lo, C& hi) {
    using T = decltype(e.x);
    if (k == 0 || 4 * k == R || std::is_same<T, dfloat>::value) {
        const C t = twiddle_pow2<R, DIR>(o, k);
        lo = cadd(e, t);
        hi = csub(e, t);
        return;
    }
    const int m16 = k * (16 / R);   // 1..7
    const T c = cos16<T>(m16), s = T(DIR) * cos16<T>(m16 - 4);
    // tan or cot of the angle, folded into [-1, 1]: 45 degrees 1, 22.5 degrees sqrt(2) - 1
    const T q = T((m16 & 1) ? 0.41421356237309504880 : 1.0);
    T m, ux, uy;
    if (m16 <= 2 || m16 >= 6) {     // |cos| >= |sin|
        const T t = T(DIR) * (m16 <= 2 ? q : -q);
        m = c;
        ux = fma(-t, o.y, o.x);
        uy = fma(t, o.x, o.y);
    } else {
        const T t = T(DIR) * (m16 < 4 ? q : -q);
        m = s;
        ux = fma(t, o.x, -o.y);
        uy = fma(t, o.y, o.x);
    }
    lo = mk(fma(m, ux, e.x), fma(m, uy, e.y));
    hi = mk(fma(-m, ux, e.x), fma(-m, uy, e.y));
}

// cosines and sines 2 pi k / R of the odd radices, k = 1 .. (R - 1) / 2
template <int R> __host__ __device__ constexpr double odd_cos(int k) {
    constexpr double c3[] = {1.0, -0.5};
    constexpr double c5[] = {1.0, 0.30901699437494742410, -0.80901699437494742410};
    constexpr double c7[] = {1.0, 0.62348980185873353053, -0.22252093395631440429, -0.90096886790241912624};
    k %= R;
    if (k > R / 2) k = R - k;
    return R == 3 ? c3[k < 2 ? k : 0] : R == 5 ? c5[k < 3 ? k : 0] : c7[k];
}
template <int R> __host__ __device__ constexpr double odd_sin(int k) {
    constexpr double s3[] = {0.0, 0.86602540378443864676};
    constexpr double s5[] = {0.0, 0.95105651629515357212, 0.58778525229247312917};
    constexpr double s7[] = {0.0, 0.78183148246802980871, 0.97492791218182360702, 0.43388373911755812048};
    k %= R;
    const bool neg = k > R / 2;
    if (neg) k = R - k;
    const double v = R == 3 ? s3[k < 2 ? k : 0] : R == 5 ? s5[k < 3 ? k : 0] : s7[k];
    return neg ? -v : v;
}

// coprime factors of the prime-factor radices
template <int R> struct Coprime { static constexpr int a = 1, b = 1; };
template <> struct Coprime<6> { static constexpr int a = 2, b = 3; };
template <> struct Coprime<10> { static constexpr int a = 2, b = 5; };
template <> struct Coprime<12> { static constexpr int a = 4, b = 3; };
template <> struct Coprime<14> { static constexpr int a = 2, b = 7; };
template <> struct Coprime<15> { static constexpr int a = 3, b = 5; };

__host__ __device__ constexpr int inv_mod(int x, int m) {
    for (int i = 1; i < m; ++i)
        if ((x * i) % m == 1) return i;
    return 1;
}

template <int R, int DIR, typename C>
struct RegDFT {
    __device__ __forceinline__ static void run(C* v) {
        using T = decltype(v[0].x);
        if constexpr (R == 1) {
            return;
        } else if constexpr (R == 2) {
            C a = v[0], b = v[1];
            v[0] = cadd(a, b);
            v[1] = csub(a, b);
        } else if constexpr ((R & (R - 1)) == 0) {
            constexpr int H = R / 2;
            C e[H], o[H];
#pragma unroll
            for (int i = 0; i < H; ++i) {
                e[i] = v[2 * i];
                o[i] = v[2 * i + 1];
            }
            RegDFT<H, DIR, C>::run(e);
            RegDFT<H, DIR, C>::run(o);
#pragma unroll
            for (int k = 0; k < H; ++k) butterfly<R, DIR>(e[k], o[k], k, v[k], v[k + H]);
        } else if constexpr (R == 3 || R == 5 || R == 7) {
            // X_k = a_k + DIR i b_k, X_{R-k} = a_k - DIR i b_k from t_n = v_n + v_{R-n}, d_n = v_n - v_{R-n}
            constexpr int H = (R - 1) / 2;
            C t[H], d[H];
            C x0 = v[0];
#pragma unroll
            for (int n = 0; n < H; ++n) {
                t[n] = cadd(v[n + 1], v[R - 1 - n]);
                d[n] = csub(v[n + 1], v[R - 1 - n]);
                x0 = cadd(x0, t[n]);
            }
#pragma unroll
            for (int k = 1; k <= H; ++k) {
                C a = v[0], b = cscale(d[0], T(odd_sin<R>(k)));
#pragma unroll
                for (int n = 0; n < H; ++n) {
                    const T c = T(odd_cos<R>((n + 1) * k));
                    a = mk(fma(c, t[n].x, a.x), fma(c, t[n].y, a.y));
                    if (n > 0) {
                        const T s = T(odd_sin<R>((n + 1) * k));
                        b = mk(fma(s, d[n].x, b.x), fma(s, d[n].y, b.y));
                    }
                }
                const C ib = cmul_i<DIR>(b);
                v[k] = cadd(a, ib);         // v[1..H], v[R-H..] are read only through t and d
                v[R - k] = csub(a, ib);
            }
            v[0] = x0;
        } else if constexpr (R == 9) {
            constexpr double c9[5] = {1.0, 0.76604444311897803520, 0.17364817766693034885, -0.5,
                                      -0.93969262078590838405};
            constexpr double s9[5] = {0.0, 0.64278760968653932632, 0.98480775301220805937, 0.86602540378443864676,
                                      0.34202014332566873304};
            C w[3][3];
#pragma unroll
            for (int n2 = 0; n2 < 3; ++n2) {
#pragma unroll
                for (int n1 = 0; n1 < 3; ++n1) w[n2][n1] = v[3 * n1 + n2];
                RegDFT<3, DIR, C>::run(w[n2]);
#pragma unroll
                for (int k1 = 1; k1 < 3; ++k1)
                    if (n2 > 0) w[n2][k1] = cmul(w[n2][k1], mk(T(c9[n2 * k1]), T(DIR * s9[n2 * k1])));
            }
#pragma unroll
            for (int k1 = 0; k1 < 3; ++k1) {
                C x[3] = {w[0][k1], w[1][k1], w[2][k1]};
                RegDFT<3, DIR, C>::run(x);
#pragma unroll
                for (int k2 = 0; k2 < 3; ++k2) v[k1 + 3 * k2] = x[k2];
            }
        } else {
            // Good's map: input n = (B i + A j) mod R, output k = (B inv_A(B) p + A inv_B(A) q) mod R
            constexpr int A = Coprime<R>::a, B = Coprime<R>::b;
            static_assert(A * B == R && A > 1, "no register DFT of this radix");
            constexpr int ua = B * inv_mod(B % A, A), ub = A * inv_mod(A % B, B);
            C w[A][B];
#pragma unroll
            for (int i = 0; i < A; ++i) {
#pragma unroll
                for (int j = 0; j < B; ++j) w[i][j] = v[(B * i + A * j) % R];
                RegDFT<B, DIR, C>::run(w[i]);
            }
#pragma unroll
            for (int q = 0; q < B; ++q) {
                C x[A];
#pragma unroll
                for (int i = 0; i < A; ++i) x[i] = w[i][q];
                RegDFT<A, DIR, C>::run(x);
#pragma unroll
                for (int p = 0; p < A; ++p) v[(ua * p + ub * q) % R] = x[p];
            }
        }
    }
};

}  // namespace bloch
