// Register-resident DFTs of sizes 1..16 with compile-time twiddle constants.
//
// Dft<N, INV>::run(v) transforms N complex values in place, natural order in
// and out: forward X[k] = sum_n v[n] exp(-2 pi i n k / N) (INV = false) or
// the unnormalised inverse with exp(+2 pi i n k / N) (INV = true).
//
// Primes use the symmetric form X[k] = v0 + sum_j a_j cos(2 pi jk/P)
// +/- i sum_j b_j sin(2 pi jk/P) with a_j = v_j + v_{P-j}, b_j = v_j - v_{P-j};
// composite sizes use one Cooley-Tukey split N = A*B done entirely in
// registers.  The cos/sin constants are evaluated at compile time from their
// Taylor series after an exact quadrant reduction of the rational angle.
#pragma once
#include <stdint.h>
#include <type_traits>
#include <utility>

namespace psatd {

template <typename T>
struct alignas(2 * sizeof(T)) cpx {
    T x, y;
};

__device__ __forceinline__ float fma_t(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_t(double a, double b, double c) { return __fma_rn(a, b, c); }

template <typename T>
__host__ __device__ __forceinline__ cpx<T> mk(T x, T y) { cpx<T> r; r.x = x; r.y = y; return r; }
template <typename T>
__device__ __forceinline__ cpx<T> operator+(cpx<T> a, cpx<T> b) { return mk(a.x + b.x, a.y + b.y); }
template <typename T>
__device__ __forceinline__ cpx<T> operator-(cpx<T> a, cpx<T> b) { return mk(a.x - b.x, a.y - b.y); }
template <typename T>
__device__ __forceinline__ cpx<T> cmul(cpx<T> a, cpx<T> b) {
    return mk(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
template <typename T>   // a * conj(b)
__device__ __forceinline__ cpx<T> cmulc(cpx<T> a, cpx<T> b) {
    return mk(a.x * b.x + a.y * b.y, a.y * b.x - a.x * b.y);
}
template <typename T>
__device__ __forceinline__ cpx<T> conj(cpx<T> a) { return mk(a.x, -a.y); }
template <typename T>   // i * a
__device__ __forceinline__ cpx<T> mul_i(cpx<T> a) { return mk(-a.y, a.x); }
template <typename T>
__device__ __forceinline__ cpx<T> scale(cpx<T> a, T s) { return mk(a.x * s, a.y * s); }

// ---- compile-time trigonometry of rational angles ------------------------
constexpr double kPi = 3.141592653589793238462643383279502884;

constexpr double taylor_sin(double x) {
    double x2 = x * x, term = x, sum = x;
    for (int n = 1; n < 22; ++n) { term *= -x2 / ((2.0 * n) * (2.0 * n + 1.0)); sum += term; }
    return sum;
}
constexpr double taylor_cos(double x) {
    double x2 = x * x, term = 1.0, sum = 1.0;
    for (int n = 1; n < 22; ++n) { term *= -x2 / ((2.0 * n - 1.0) * (2.0 * n)); sum += term; }
    return sum;
}
// 2 pi m / N = q pi/2 + phi with phi in [0, pi/2)
constexpr long quad_of(long m, long N) { return (4 * (((m % N) + N) % N)) / N; }
constexpr double phi_of(long m, long N) {
    return (kPi / 2) * double(4 * (((m % N) + N) % N) - quad_of(m, N) * N) / double(N);
}
// +-1/2 exactly at multiples of 30 degrees (the series ends within an ulp of it)
constexpr double snap_half(double v) {
    return v > 0.5 - 1e-15 && v < 0.5 + 1e-15 ? 0.5 : v > -0.5 - 1e-15 && v < -0.5 + 1e-15 ? -0.5 : v;
}
constexpr double cos2pi(long m, long N) {
    return snap_half(quad_of(m, N) == 0 ? taylor_cos(phi_of(m, N))
                   : quad_of(m, N) == 1 ? -taylor_sin(phi_of(m, N))
                   : quad_of(m, N) == 2 ? -taylor_cos(phi_of(m, N))
                                        : taylor_sin(phi_of(m, N)));
}
constexpr double sin2pi(long m, long N) {
    return snap_half(quad_of(m, N) == 0 ? taylor_sin(phi_of(m, N))
                   : quad_of(m, N) == 1 ? taylor_cos(phi_of(m, N))
                   : quad_of(m, N) == 2 ? -taylor_sin(phi_of(m, N))
                                        : -taylor_cos(phi_of(m, N)));
}

// ---- compile-time loop ----------------------------------------------------
template <int I, int N, class F>
__device__ __forceinline__ void static_for_impl(F&& f) {
    if constexpr (I < N) {
        f(std::integral_constant<int, I>{});
        static_for_impl<I + 1, N>(f);
    }
}
template <int N, class F>
__device__ __forceinline__ void static_for(F&& f) { static_for_impl<0, N>(f); }

// FP32 constants are split into hi + lo (lo = the FP32 rounding of the
// remainder), so that a product with a constant carries no systematic
// quantisation error; in FP64 the lo part is dropped.  PSATD_DFT_HILO 0
// keeps only the FP32 rounding.
#ifndef PSATD_DFT_HILO
#define PSATD_DFT_HILO 1
#endif
template <typename T>
struct Split32 {
    static constexpr bool kOn = sizeof(T) == 4 && PSATD_DFT_HILO;
};
template <typename T>
constexpr T hi_of(double v) { return T(v); }
template <typename T>
constexpr T lo_of(double v) { return T(v - double(T(v))); }
// Whether the FP32 constant v needs its lo part (+-1/2 and the like do not).
template <typename T>
constexpr bool has_lo(double v) { return Split32<T>::kOn && v - double(float(v)) != 0.0; }
constexpr double abs_c(double v) { return v < 0 ? -v : v; }

// Constants are applied by magnitude, so that c and -c share one register; the
// sign goes to the other operand (free).
template <bool NEG, typename T>
__device__ __forceinline__ T sgn(T v) {
    if constexpr (NEG) return -v;
    else return v;
}

// multiply by exp(sgn 2 pi i M / N), sgn = -1 forward, +1 inverse
template <int M, int N, bool INV, typename T>
__device__ __forceinline__ cpx<T> twiddle(cpx<T> v) {
    constexpr int m = ((M % N) + N) % N;
    if constexpr (m == 0) {
        return v;
    } else if constexpr (2 * m == N) {
        return mk(-v.x, -v.y);
    } else if constexpr (4 * m == N) {          // exp(sgn i pi/2) = sgn i
        return INV ? mk(-v.y, v.x) : mk(v.y, -v.x);
    } else if constexpr (4 * m == 3 * N) {      // exp(sgn i 3pi/2) = -sgn i
        return INV ? mk(v.y, -v.x) : mk(-v.y, v.x);
    } else {
        constexpr double c = cos2pi(m, N);
        constexpr double s = INV ? sin2pi(m, N) : -sin2pi(m, N);
        if constexpr (!Split32<T>::kOn) {
            constexpr T cc = T(c), ss = T(s);
            return mk(v.x * cc - v.y * ss, v.x * ss + v.y * cc);
        }
        constexpr double cm = abs_c(c), sm = abs_c(s);
        // (x c - y s) + i (x s + y c), the lo parts first
        const T xc = sgn<(c < 0)>(v.x), yc = sgn<(c < 0)>(v.y);
        const T xs = sgn<(s < 0)>(v.x), ys = sgn<(s > 0)>(v.y);
        if constexpr (Split32<T>::kOn && 8 * m % N == 0) {   // c = +-s: one product (hi + lo) for each part
            const T u = xc + ys, w = yc + xs;
            return mk(fma_t(u, hi_of<T>(cm), u * lo_of<T>(cm)), fma_t(w, hi_of<T>(cm), w * lo_of<T>(cm)));
        }
        T re, im;
        if constexpr (has_lo<T>(cm) && has_lo<T>(sm)) {
            re = fma_t(xc, lo_of<T>(cm), ys * lo_of<T>(sm));
            im = fma_t(yc, lo_of<T>(cm), xs * lo_of<T>(sm));
            re = fma_t(ys, hi_of<T>(sm), re);
            im = fma_t(xs, hi_of<T>(sm), im);
        } else if constexpr (has_lo<T>(cm)) {
            re = fma_t(ys, hi_of<T>(sm), xc * lo_of<T>(cm));
            im = fma_t(xs, hi_of<T>(sm), yc * lo_of<T>(cm));
        } else if constexpr (has_lo<T>(sm)) {
            re = fma_t(ys, hi_of<T>(sm), ys * lo_of<T>(sm));
            im = fma_t(xs, hi_of<T>(sm), xs * lo_of<T>(sm));
        } else {
            re = ys * hi_of<T>(sm);
            im = xs * hi_of<T>(sm);
        }
        return mk(fma_t(xc, hi_of<T>(cm), re), fma_t(yc, hi_of<T>(cm), im));
    }
}

template <int N, bool INV>
struct Dft;

template <bool INV>
struct Dft<1, INV> {
    template <typename T>
    __device__ __forceinline__ static void run(cpx<T>*) {}
};

template <bool INV>
struct Dft<2, INV> {
    template <typename T>
    __device__ __forceinline__ static void run(cpx<T>* v) {
        cpx<T> a = v[0];
        v[0] = a + v[1];
        v[1] = a - v[1];
    }
};

template <bool INV>
struct Dft<4, INV> {
    template <typename T>
    __device__ __forceinline__ static void run(cpx<T>* v) {
        const cpx<T> a = v[0] + v[2], b = v[0] - v[2], c = v[1] + v[3], d = v[1] - v[3];
        v[0] = a + c;
        v[2] = a - c;
        // b -/+ i d
        const cpx<T> bm = mk(b.x + d.y, b.y - d.x), bp = mk(b.x - d.y, b.y + d.x);
        if (INV) { v[1] = bp; v[3] = bm; }
        else     { v[1] = bm; v[3] = bp; }
    }
};

template <int P, bool INV>
struct DftPrime {
    template <typename T>
    __device__ __forceinline__ static void run(cpx<T>* v) {
        constexpr int H = (P - 1) / 2;
        cpx<T> a[H], b[H];
        static_for<H>([&](auto jc) {
            constexpr int j = decltype(jc)::value;
            a[j] = v[j + 1] + v[P - 1 - j];
            b[j] = v[j + 1] - v[P - 1 - j];
        });
        const cpx<T> x0 = v[0];
        cpx<T> s0 = x0 + a[0];
        static_for<H - 1>([&](auto jc) { s0 = s0 + a[decltype(jc)::value + 1]; });
        v[0] = s0;
        static_for<H>([&](auto kc) {
            constexpr int k = decltype(kc)::value + 1;
            cpx<T> R = x0, Q;
            cpx<T> Rl, Ql;                       // lo parts of the constants, summed apart
            static_for<H>([&](auto jc) {
                constexpr int j = decltype(jc)::value + 1;
                constexpr double c = cos2pi((long)j * k, P), s = sin2pi((long)j * k, P);
                if constexpr (!Split32<T>::kOn) {
                    constexpr T cc = T(c), ss = T(s);
                    if constexpr (j == 1) Q = mk(T(0), T(0));
                    R.x += a[j - 1].x * cc; R.y += a[j - 1].y * cc;
                    Q.x += b[j - 1].x * ss; Q.y += b[j - 1].y * ss;
                    return;
                }
                constexpr double cm = abs_c(c), sm = abs_c(s);
                const cpx<T> ac = mk(sgn<(c < 0)>(a[j - 1].x), sgn<(c < 0)>(a[j - 1].y));
                const cpx<T> bs = mk(sgn<(s < 0)>(b[j - 1].x), sgn<(s < 0)>(b[j - 1].y));
                if constexpr (has_lo<T>(cm)) {
                    constexpr T cl = lo_of<T>(cm);
                    if constexpr (j == 1) Rl = mk(ac.x * cl, ac.y * cl);
                    else Rl = mk(fma_t(ac.x, cl, Rl.x), fma_t(ac.y, cl, Rl.y));
                }
                if constexpr (has_lo<T>(sm)) {
                    constexpr T sl = lo_of<T>(sm);
                    if constexpr (j == 1) Ql = mk(bs.x * sl, bs.y * sl);
                    else Ql = mk(fma_t(bs.x, sl, Ql.x), fma_t(bs.y, sl, Ql.y));
                }
                constexpr T ch = hi_of<T>(cm), sh = hi_of<T>(sm);
                R = mk(fma_t(ac.x, ch, R.x), fma_t(ac.y, ch, R.y));
                // P = 3 has one sine: its lo product starts the sum
                if constexpr (j == 1 && H == 1 && has_lo<T>(sm)) Q = mk(fma_t(bs.x, sh, Ql.x), fma_t(bs.y, sh, Ql.y));
                else if constexpr (j == 1) Q = mk(bs.x * sh, bs.y * sh);
                else Q = mk(fma_t(bs.x, sh, Q.x), fma_t(bs.y, sh, Q.y));
            });
            // every constant but the cosine of P = 3 (-1/2) has a lo part
            if constexpr (Split32<T>::kOn && H > 1) { R = R + Rl; Q = Q + Ql; }
            // X_k = R + sgn i Q, X_{P-k} = R - sgn i Q
            if (INV) { v[k] = mk(R.x - Q.y, R.y + Q.x); v[P - k] = mk(R.x + Q.y, R.y - Q.x); }
            else     { v[k] = mk(R.x + Q.y, R.y - Q.x); v[P - k] = mk(R.x - Q.y, R.y + Q.x); }
        });
    }
};

template <int N, int A, bool INV>
struct DftSplit {
    template <typename T>
    __device__ __forceinline__ static void run(cpx<T>* v) {
        constexpr int B = N / A;
        cpx<T> y[N];
        // A-point DFTs over n1 of v[B n1 + n2], then twiddle w_N^{n2 k1}
        static_for<B>([&](auto n2c) {
            constexpr int n2 = decltype(n2c)::value;
            cpx<T> t[A];
            static_for<A>([&](auto n1c) { t[decltype(n1c)::value] = v[B * decltype(n1c)::value + n2]; });
            Dft<A, INV>::run(t);
            static_for<A>([&](auto k1c) {
                constexpr int k1 = decltype(k1c)::value;
                y[n2 * A + k1] = twiddle<n2 * k1, N, INV>(t[k1]);
            });
        });
        // B-point DFTs over n2, output X[k1 + A k2]
        static_for<A>([&](auto k1c) {
            constexpr int k1 = decltype(k1c)::value;
            cpx<T> t[B];
            static_for<B>([&](auto n2c) { t[decltype(n2c)::value] = y[decltype(n2c)::value * A + k1]; });
            Dft<B, INV>::run(t);
            static_for<B>([&](auto k2c) { v[k1 + A * decltype(k2c)::value] = t[decltype(k2c)::value]; });
        });
    }
};

template <bool INV> struct Dft<3, INV> : DftPrime<3, INV> {};
template <bool INV> struct Dft<5, INV> : DftPrime<5, INV> {};
template <bool INV> struct Dft<7, INV> : DftPrime<7, INV> {};
template <bool INV> struct Dft<11, INV> : DftPrime<11, INV> {};
template <bool INV> struct Dft<13, INV> : DftPrime<13, INV> {};
template <bool INV> struct Dft<6, INV> : DftSplit<6, 2, INV> {};
template <bool INV> struct Dft<8, INV> : DftSplit<8, 2, INV> {};
template <bool INV> struct Dft<9, INV> : DftSplit<9, 3, INV> {};
template <bool INV> struct Dft<10, INV> : DftSplit<10, 2, INV> {};
template <bool INV> struct Dft<12, INV> : DftSplit<12, 4, INV> {};
template <bool INV> struct Dft<14, INV> : DftSplit<14, 2, INV> {};
template <bool INV> struct Dft<15, INV> : DftSplit<15, 3, INV> {};
template <bool INV> struct Dft<16, INV> : DftSplit<16, 4, INV> {};
template <bool INV> struct Dft<20, INV> : DftSplit<20, 4, INV> {};
template <bool INV> struct Dft<24, INV> : DftSplit<24, 3, INV> {};

// Call f(integral_constant<int, n>) for a runtime n in 1..16.
template <class F>
__device__ __forceinline__ void with_size(int n, F&& f) {
    switch (n) {
        case 1: f(std::integral_constant<int, 1>{}); break;
        case 2: f(std::integral_constant<int, 2>{}); break;
        case 3: f(std::integral_constant<int, 3>{}); break;
        case 4: f(std::integral_constant<int, 4>{}); break;
        case 5: f(std::integral_constant<int, 5>{}); break;
        case 6: f(std::integral_constant<int, 6>{}); break;
        case 7: f(std::integral_constant<int, 7>{}); break;
        case 8: f(std::integral_constant<int, 8>{}); break;
        case 9: f(std::integral_constant<int, 9>{}); break;
        case 10: f(std::integral_constant<int, 10>{}); break;
        case 11: f(std::integral_constant<int, 11>{}); break;
        case 12: f(std::integral_constant<int, 12>{}); break;
        case 13: f(std::integral_constant<int, 13>{}); break;
        case 14: f(std::integral_constant<int, 14>{}); break;
        case 15: f(std::integral_constant<int, 15>{}); break;
        case 16: f(std::integral_constant<int, 16>{}); break;
        default: break;
    }
}

}  // namespace psatd
