// Device building blocks of the FFT path: compile-time trigonometry,
// in-register DFTs of small radices, and block transforms that exchange data
// in place through shared memory.
//
// The transform computed is the DFT of Sec. 2.3 Eq. (10) (0-based indices),
// F[k] = sum_n f[n] exp(DIR * i 2 pi k n / N), DIR = -1 forward, +1 inverse
// (unnormalised both ways), evaluated by the Cooley-Tukey factorisation the
// paper cites for FFTs (Sec. 2.3), one butterfly stage per factor of N: in
// place, three factors at most, for the FP32 passes (block transforms
// below), and in the self-sorting (Stockham) order, stage s of
// N = R_0 R_1 ... R_{S-1}, for the tensor-core column pass: with Ns = R_0 ... R_{s-1} and butterfly j in [0, N/R_s)
//   inputs   x[j + m N/R_s],                      m = 0..R_s-1
//   twiddle  x_m *= exp(DIR i 2 pi (j mod Ns) m / (Ns R_s))
//   DFT of size R_s in registers
//   outputs  y[(j div Ns) Ns R_s + (j mod Ns) + m Ns]
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "lp_internal.h"

namespace lpk {

// ---------------------------------------------------------------------------
// Compile-time trigonometry: cos / sin of 2 pi t / n for integer t, n.
// The angle is reduced to a quadrant in exact integer arithmetic, then a
// Taylor series in double precision (16 terms on |x| <= pi/4, truncation far
// below 1e-17) is summed.  Only used to build constants at compile time.
// ---------------------------------------------------------------------------
constexpr double kHalfPi = 1.57079632679489661923132169163975;

__host__ __device__ constexpr double taylor_sin(double x)
{
    double term = x, sum = x;
    for (int k = 1; k < 16; ++k) {
        term *= -x * x / ((2.0 * k) * (2.0 * k + 1.0));
        sum += term;
    }
    return sum;
}

__host__ __device__ constexpr double taylor_cos(double x)
{
    double term = 1.0, sum = 1.0;
    for (int k = 1; k < 16; ++k) {
        term *= -x * x / ((2.0 * k - 1.0) * (2.0 * k));
        sum += term;
    }
    return sum;
}

// cos(phi), sin(phi) for phi = (pi/2) r / n, 0 <= r < n, with the argument
// kept in [0, pi/4] by the complementary-angle identity.
__host__ __device__ constexpr double quad_cos(long r, long n)
{
    return (2 * r <= n) ? taylor_cos(kHalfPi * (double)r / (double)n)
                        : taylor_sin(kHalfPi * (double)(n - r) / (double)n);
}
__host__ __device__ constexpr double quad_sin(long r, long n)
{
    return (2 * r <= n) ? taylor_sin(kHalfPi * (double)r / (double)n)
                        : taylor_cos(kHalfPi * (double)(n - r) / (double)n);
}

__host__ __device__ constexpr double cos2pi(long t, long n)
{
    t = ((t % n) + n) % n;
    const long q = (4 * t) / n, r = 4 * t - q * n;
    const double c = quad_cos(r, n), s = quad_sin(r, n);
    return q == 0 ? c : q == 1 ? -s : q == 2 ? -c : s;
}
__host__ __device__ constexpr double sin2pi(long t, long n)
{
    t = ((t % n) + n) % n;
    const long q = (4 * t) / n, r = 4 * t - q * n;
    const double c = quad_cos(r, n), s = quad_sin(r, n);
    return q == 0 ? s : q == 1 ? c : q == 2 ? -s : -c;
}

// ---------------------------------------------------------------------------
// Compile-time loop helper: calls f(integral_constant<int, I>) for I in [B, E).
// ---------------------------------------------------------------------------
template <int B, int E, class F>
__device__ __forceinline__ void sfor(F&& f)
{
    if constexpr (B < E) {
        f(std::integral_constant<int, B>{});
        sfor<B + 1, E>(f);
    }
}

// ---------------------------------------------------------------------------
// Complex helpers, generic over float2 / double2.
// ---------------------------------------------------------------------------
template <class C> struct Scalar;
template <> struct Scalar<float2> { using type = float; };
template <> struct Scalar<double2> { using type = double; };

template <class C>
__device__ __forceinline__ C mk(typename Scalar<C>::type x, typename Scalar<C>::type y)
{
    C r;
    r.x = x;
    r.y = y;
    return r;
}
template <class C> __device__ __forceinline__ C cadd(C a, C b) { return mk<C>(a.x + b.x, a.y + b.y); }
template <class C> __device__ __forceinline__ C csub(C a, C b) { return mk<C>(a.x - b.x, a.y - b.y); }
// a * c (c real) and a * c + acc
template <class C> __device__ __forceinline__ C cscale(C a, typename Scalar<C>::type c)
{
    return mk<C>(a.x * c, a.y * c);
}
template <class C> __device__ __forceinline__ C cfma(C a, typename Scalar<C>::type c, C acc)
{
    return mk<C>(a.x * c + acc.x, a.y * c + acc.y);
}

// FP32 complex values {re, im} are a natural pair for the packed FP32x2
// instructions: an addition, a subtraction, a real scaling or a real
// multiply-add of a complex value is one add / sub / mul / fma .f32x2.
// A plan chooses per length (LP_PACKED_FP32, set by the length's translation
// unit, whose device code is compiled on its own): the packed constants take
// registers, which costs more than it saves in the register-bound kernels of
// some lengths.
#ifndef LP_PACKED_FP32
#define LP_PACKED_FP32 1
#endif
#if LP_PACKED_FP32
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 csub(float2 a, float2 b)
{
    unsigned long long ra, rb, rd;
    asm("mov.b64 %0, {%1, %2};" : "=l"(ra) : "f"(a.x), "f"(a.y));
    asm("mov.b64 %0, {%1, %2};" : "=l"(rb) : "f"(b.x), "f"(b.y));
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(rd) : "l"(ra), "l"(rb));
    float2 d;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(d.x), "=f"(d.y) : "l"(rd));
    return d;
}
__device__ __forceinline__ float2 cscale(float2 a, float c) { return __fmul2_rn(a, make_float2(c, c)); }
__device__ __forceinline__ float2 cfma(float2 a, float c, float2 acc) { return __ffma2_rn(a, make_float2(c, c), acc); }
#endif
template <class C> __device__ __forceinline__ C cmul(C a, C b)
{
    return mk<C>(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// multiply by i*DIR (DIR = +-1)
template <int DIR, class C> __device__ __forceinline__ C mul_idir(C a)
{
    if constexpr (DIR > 0) return mk<C>(-a.y, a.x);
    else return mk<C>(a.y, -a.x);
}

// Constants of the FP32 butterflies.  The rounding error of a table's twiddle
// differs from place to place and averages out; a butterfly's constant is the
// same for all data, and rounded alike in the forward transform F and the
// inverse G it scales whatever passes both (G F - R I has a diagonal).  So the
// two directions round them such that G F comes as close to R I as FP32
// allows, at no cost:
//   * a turn by (c, s): the inverse takes the value whose error cancels the
//     forward one's best, c rounded about (cos(pi/8): -2.8e-8, then +3.2e-8);
//   * radices 3, 5, 7: the choice of |G F - R I| smallest among all roundings
//     of their constants up or down in either direction: 3.6 -> 3.3e-8 of R
//     (Frobenius), 5.0 -> 2.8e-8, 6.1 -> 4.3e-8.
// Maps of one spectrum at N x N, rms error against 64 bits with both
// directions rounded to nearest = 1: 0.83 at 1024 and 8192, 0.86 at 4096, 0.80
// at 16384, 0.88 at 4704, 8640 and 17280, 0.94 at 13440, 0.99 at 2250.
__host__ __device__ constexpr float fp32_other(double c)  // of the two FP32 values around c, the farther one
{
    const float f = (float)c;
    double ulp = 1.0;
    while (ulp > (c < 0 ? -c : c)) ulp *= 0.5;
    ulp *= 1.0 / 8388608.0;
    return (float)((double)f < c ? (double)f + ulp : (double)f - ulp);
}
template <int DIR, class S>
__host__ __device__ constexpr S turn_const(double c)
{
    return std::is_same<S, float>::value && DIR > 0 ? (S)(2.0 * c - (double)(S)c) : (S)c;
}
// cos and sin of 2 pi q / P
template <int P, int DIR, class S>
__host__ __device__ constexpr S prime_cos(long q)
{
    q = q % P;
    if (2 * q > P) q = P - q;
    const bool other = std::is_same<S, float>::value && ((P == 5 && q == 1 && DIR > 0) || (P == 7 && q == 2));
    return other ? (S)fp32_other(cos2pi(q, P)) : (S)cos2pi(q, P);
}
template <int P, int DIR, class S>
__host__ __device__ constexpr S prime_sin(long q)
{
    q = q % P;
    const bool neg = 2 * q > P;
    if (neg) q = P - q;
    const bool other =
        std::is_same<S, float>::value && ((P == 3 && DIR > 0) || P == 5 || (P == 7 && q == 3 && DIR > 0));
    const S v = other ? (S)fp32_other(sin2pi(q, P)) : (S)sin2pi(q, P);
    return neg ? -v : v;
}

// An odd eighth turn is exp(DIR i 2 pi t / n) = (+-1 +- i) sqrt(1/2).
__host__ __device__ constexpr bool odd_eighth(long t, long n) { return (8 * t) % n == 0 && (8 * t / n) % 2 != 0; }
constexpr double kSqrtHalf = 0.70710678118654752440084436210485;

// a * exp(DIR i 2 pi t / n) / sqrt(1/2) for an odd eighth turn: a sum and a
// difference.  The butterfly that follows multiplies by sqrt(1/2) in the
// multiply-add that adds it: one rounding instead of two, and one instruction
// less.  (Packed arithmetic has no contraction of its own: with products of
// their own here and in radix 3 the maps' errors were 1-3 % larger than with
// scalar arithmetic.)
template <int T, int N, int DIR, class C>
__device__ __forceinline__ C eighth_unscaled(C a)
{
    using S = typename Scalar<C>::type;
    constexpr S cs = (S)(cos2pi(T, N) > 0 ? 1 : -1);
    constexpr S sn = (S)((sin2pi(T, N) > 0 ? 1 : -1) * DIR);
    return mk<C>(cs * a.x - sn * a.y, sn * a.x + cs * a.y);
}

// a * exp(DIR i 2 pi t / n), with t, n compile-time.  Exact quarter turns are
// done by swaps, eighth turns with one shared factor, the rest by a complex
// multiply against rounded constants.
template <int T, int N, int DIR, class C>
__device__ __forceinline__ C rot(C a)
{
    using S = typename Scalar<C>::type;
    constexpr int t = ((T % N) + N) % N;
    if constexpr (t == 0) {
        return a;
    } else if constexpr (2 * t == N) {
        return mk<C>(-a.x, -a.y);
    } else if constexpr (4 * t == N) {
        return mul_idir<DIR>(a);
    } else if constexpr (4 * t == 3 * N) {
        return mul_idir<-DIR>(a);
    } else if constexpr ((8 * t) % N == 0) {
        // odd multiple of an eighth turn: cos, sin = +-sqrt(1/2)
        constexpr S h = (S)kSqrtHalf;
        constexpr S cs = (S)(cos2pi(t, N) > 0 ? 1 : -1);
        constexpr S sn = (S)((sin2pi(t, N) > 0 ? 1 : -1) * DIR);
        // (x + i y)(cs + i sn) h
        return mk<C>(h * (cs * a.x - sn * a.y), h * (sn * a.x + cs * a.y));
    } else {
        constexpr S c = turn_const<DIR, S>(cos2pi(t, N));
        constexpr S s = DIR * turn_const<DIR, S>(sin2pi(t, N));
        return mk<C>(a.x * c - a.y * s, a.x * s + a.y * c);
    }
}

// ---------------------------------------------------------------------------
// In-register DFT of size R (unnormalised), natural order in and out.
// ---------------------------------------------------------------------------
__host__ __device__ constexpr int gcd_i(int a, int b) { return b == 0 ? a : gcd_i(b, a % b); }

// Split of a composite radix r = a * b for the in-register DFT: coprime
// factors when there are any (prime-factor algorithm, no internal
// twiddles), the largest such a with a*a <= r; otherwise the largest
// divisor a with a*a <= r (4 x r/4 for powers of two).  1 for primes.
__host__ __device__ constexpr int small_factor(int r)
{
    int coprime = 1;
    for (int a = 2; a < r; ++a)
        if (r % a == 0 && gcd_i(a, r / a) == 1 && (coprime == 1 || a * a <= r)) coprime = a;
    if (coprime > 1) {
        // prefer the smaller of the two coprime factors first
        const int b = r / coprime;
        return coprime < b ? coprime : b;
    }
    if (r % 4 == 0 && r > 4) return 4;
    int best = 1;
    for (int a = 2; a * a <= r; ++a)
        if (r % a == 0) best = a;
    return best;
}

// modular inverse of a mod m (a, m coprime), compile time
__host__ __device__ constexpr int inv_mod(int a, int m)
{
    for (int x = 1; x < m; ++x)
        if ((a * x) % m == 1) return x;
    return 1;
}

template <int R, int DIR, class C> struct Dft;

// DFT of size R whose inputs in the mask PEND still lack a factor sqrt(1/2)
template <int R, int DIR, int PEND, class C> __device__ __forceinline__ void dft_pending(C* v);

// of the inputs B n1 + n2 (n1 < A): those in the mask
template <int A, int B>
__host__ __device__ constexpr int pending_inputs(int mask, int n2)
{
    int m = 0;
    for (int n1 = 0; n1 < A; ++n1) m |= ((mask >> (B * n1 + n2)) & 1) << n1;
    return m;
}
// the n2 < B whose turn n2 k1 / R is an odd eighth
template <int B, int R>
__host__ __device__ constexpr int pending_turns(int k1)
{
    int m = 0;
    for (int n2 = 0; n2 < B; ++n2) m |= (odd_eighth((long)n2 * k1, R) ? 1 : 0) << n2;
    return m;
}

template <int DIR, class C> struct Dft<1, DIR, C> {
    __device__ __forceinline__ static void run(C*) {}
};

template <int DIR, class C> struct Dft<2, DIR, C> {
    __device__ __forceinline__ static void run(C* v)
    {
        C a = v[0], b = v[1];
        v[0] = cadd(a, b);
        v[1] = csub(a, b);
    }
};

template <int DIR, class C> struct Dft<4, DIR, C> {
    __device__ __forceinline__ static void run(C* v)
    {
        C t0 = cadd(v[0], v[2]), t1 = csub(v[0], v[2]);
        C t2 = cadd(v[1], v[3]), t3 = mul_idir<DIR>(csub(v[1], v[3]));
        v[0] = cadd(t0, t2);
        v[2] = csub(t0, t2);
        v[1] = cadd(t1, t3);
        v[3] = csub(t1, t3);
    }
};

// Odd prime P: pair x_k with x_{P-k}; y_m = x_0 + sum_k (x_k + x_{P-k}) cos
// + DIR i sum_k (x_k - x_{P-k}) sin, and y_{P-m} the conjugate combination.
template <int P, int DIR, class C>
__device__ __forceinline__ void dft_odd_prime(C* v)
{
    using S = typename Scalar<C>::type;
    constexpr int H = (P - 1) / 2;
    C a[H], b[H];
    sfor<1, H + 1>([&](auto K_) {
        constexpr int k = decltype(K_)::value;
        a[k - 1] = cadd(v[k], v[P - k]);
        b[k - 1] = csub(v[k], v[P - k]);
    });
    C y[P];
    y[0] = v[0];
    sfor<0, H>([&](auto K_) { y[0] = cadd(y[0], a[decltype(K_)::value]); });
    sfor<1, H + 1>([&](auto M_) {
        constexpr int m = decltype(M_)::value;
        C re = v[0];
        if constexpr (H == 1 && std::is_same<C, float2>::value) {
            // one sine: in the multiply-add that adds it (one rounding less)
            constexpr S s = prime_sin<P, DIR, S>(1);
            re = cfma(a[0], (S)cos2pi(1, P), re);
            const C ib = mul_idir<DIR>(b[0]);
            y[m] = cfma(ib, s, re);
            y[P - m] = cfma(ib, -s, re);
            return;
        }
        C im;
        sfor<1, H + 1>([&](auto K_) {
            constexpr int k = decltype(K_)::value;
            constexpr S c = prime_cos<P, DIR, S>((long)k * m);
            constexpr S s = prime_sin<P, DIR, S>((long)k * m);
            re = cfma(a[k - 1], c, re);
            im = (k == 1) ? cscale(b[0], s) : cfma(b[k - 1], s, im);
        });
        // y_m = re + DIR i im ; y_{P-m} = re - DIR i im
        C ii = mul_idir<DIR>(im);
        y[m] = cadd(re, ii);
        y[P - m] = csub(re, ii);
    });
    sfor<0, P>([&](auto K_) { v[decltype(K_)::value] = y[decltype(K_)::value]; });
}

// Composite R = A * B.
//  * gcd(A, B) = 1: prime-factor (Good-Thomas) algorithm.  With input index
//    n = (B n1 + A n2) mod R and output index k = k1 B (B^-1 mod A) +
//    k2 A (A^-1 mod B) mod R (k1 = k mod A, k2 = k mod B), the R-point DFT
//    is A-point DFTs over n1 followed by B-point DFTs over n2 with no
//    twiddles in between; both index maps are compile-time permutations.
//  * otherwise Cooley-Tukey in registers: n = B n1 + n2, k = k1 + A k2;
//    A-point DFTs over n1, twiddle exp(DIR i 2pi n2 k1 / R), B-point DFTs
//    over n2.
template <int R, int DIR, class C> struct Dft {
    static constexpr int A = small_factor(R);
    static constexpr int B = R / A;
    __device__ __forceinline__ static void run(C* v)
    {
        if constexpr (A == 1) {
            static_assert(R % 2 == 1, "prime radix must be odd here");
            dft_odd_prime<R, DIR, C>(v);
        } else if constexpr (gcd_i(A, B) == 1) {
            constexpr int EA = B * inv_mod(B % A, A);  // k -> k1 component of the CRT
            constexpr int EB = A * inv_mod(A % B, B);
            C t[R];
            sfor<0, B>([&](auto N2_) {
                constexpr int n2 = decltype(N2_)::value;
                C a[A];
                sfor<0, A>([&](auto N1_) {
                    constexpr int n1 = decltype(N1_)::value;
                    a[n1] = v[(B * n1 + A * n2) % R];
                });
                Dft<A, DIR, C>::run(a);
                sfor<0, A>([&](auto K1_) { t[n2 * A + decltype(K1_)::value] = a[decltype(K1_)::value]; });
            });
            sfor<0, A>([&](auto K1_) {
                constexpr int k1 = decltype(K1_)::value;
                C b[B];
                sfor<0, B>([&](auto N2_) { b[decltype(N2_)::value] = t[decltype(N2_)::value * A + k1]; });
                Dft<B, DIR, C>::run(b);
                sfor<0, B>([&](auto K2_) {
                    constexpr int k2 = decltype(K2_)::value;
                    v[(k1 * EA + k2 * EB) % R] = b[k2];
                });
            });
        } else {
            run_pending<0>(v);
        }
    }
    // Cooley-Tukey with the factor sqrt(1/2) of the inputs in the mask PEND
    // still to come; the eighth turns between the factors leave theirs to the
    // second factor's butterflies.
    template <int PEND>
    __device__ __forceinline__ static void run_pending(C* v)
    {
        constexpr bool FP32 = std::is_same<C, float2>::value;
        C t[R];
        sfor<0, B>([&](auto N2_) {
            constexpr int n2 = decltype(N2_)::value;
            C a[A];
            sfor<0, A>([&](auto N1_) { a[decltype(N1_)::value] = v[B * decltype(N1_)::value + n2]; });
            dft_pending<A, DIR, pending_inputs<A, B>(PEND, n2)>(a);
            sfor<0, A>([&](auto K1_) {
                constexpr int k1 = decltype(K1_)::value;
                if constexpr (FP32 && odd_eighth(n2 * k1, R)) t[n2 * A + k1] = eighth_unscaled<n2 * k1, R, DIR>(a[k1]);
                else t[n2 * A + k1] = rot<n2 * k1, R, DIR>(a[k1]);
            });
        });
        sfor<0, A>([&](auto K1_) {
            constexpr int k1 = decltype(K1_)::value;
            C b[B];
            sfor<0, B>([&](auto N2_) { b[decltype(N2_)::value] = t[decltype(N2_)::value * A + k1]; });
            dft_pending<B, DIR, FP32 ? pending_turns<B, R>(k1) : 0>(b);
            sfor<0, B>([&](auto K2_) { v[k1 + A * decltype(K2_)::value] = b[decltype(K2_)::value]; });
        });
    }
};

template <int R, int DIR, int PEND, class C>
__device__ __forceinline__ void dft_pending(C* v)
{
    using S = typename Scalar<C>::type;
    constexpr S h = (S)kSqrtHalf;
    if constexpr (PEND == 0) {
        Dft<R, DIR, C>::run(v);
    } else if constexpr (R == 2 && PEND == 2) {
        const C a = v[0], b = v[1];
        v[0] = cfma(b, h, a);
        v[1] = cfma(b, -h, a);
    } else if constexpr (R == 4 && PEND == 4) {
        const C t0 = cfma(v[2], h, v[0]), t1 = cfma(v[2], -h, v[0]);
        const C t2 = cadd(v[1], v[3]), t3 = mul_idir<DIR>(csub(v[1], v[3]));
        v[0] = cadd(t0, t2);
        v[2] = csub(t0, t2);
        v[1] = cadd(t1, t3);
        v[3] = csub(t1, t3);
    } else if constexpr (R == 4 && PEND == 10) {
        const C t0 = cadd(v[0], v[2]), t1 = csub(v[0], v[2]);
        const C t2 = cadd(v[1], v[3]), t3 = mul_idir<DIR>(csub(v[1], v[3]));
        v[0] = cfma(t2, h, t0);
        v[2] = cfma(t2, -h, t0);
        v[1] = cfma(t3, h, t1);
        v[3] = cfma(t3, -h, t1);
    } else if constexpr (R == 8) {
        Dft<R, DIR, C>::template run_pending<PEND>(v);
    } else {
        sfor<0, R>([&](auto K_) {
            constexpr int k = decltype(K_)::value;
            if constexpr ((PEND >> k) & 1) v[k] = cscale(v[k], h);
        });
        Dft<R, DIR, C>::run(v);
    }
}

// ---------------------------------------------------------------------------
// Radix sequences
// ---------------------------------------------------------------------------
template <int... Rs> struct Seq {};

template <class In, class Out> struct RevImpl;
template <int... Out> struct RevImpl<Seq<>, Seq<Out...>> { using type = Seq<Out...>; };
template <int H, int... T, int... Out> struct RevImpl<Seq<H, T...>, Seq<Out...>> {
    using type = typename RevImpl<Seq<T...>, Seq<H, Out...>>::type;
};
template <class S> using Reverse = typename RevImpl<S, Seq<>>::type;

template <class S> struct SeqInfo;
template <int H, int... T> struct SeqInfo<Seq<H, T...>> {
    static constexpr int first = H;
    static constexpr int last = sizeof...(T) == 0 ? H : SeqInfo<Seq<T...>>::last;
    static constexpr int min_r = (sizeof...(T) == 0 || H < SeqInfo<Seq<T...>>::min_r) ? H : SeqInfo<Seq<T...>>::min_r;
    static constexpr int max_r = (sizeof...(T) == 0 || H > SeqInfo<Seq<T...>>::max_r) ? H : SeqInfo<Seq<T...>>::max_r;
    static constexpr int product = H * SeqInfo<Seq<T...>>::product;
    static constexpr int stages = 1 + sizeof...(T);
};
template <> struct SeqInfo<Seq<>> {
    static constexpr int first = 1, last = 1, min_r = 1 << 30, max_r = 0, product = 1, stages = 0;
};

// ---------------------------------------------------------------------------
// Block transforms: N = R0 R1 R2 (R0 = 1: two factors), in place in shared
// memory.  With N1 = R1 R2, input n = j + N1 q (j < N1, q < R0), j = i + R2 l
// (i < R2, l < R1), and frequency k = m + R0 (k1 + R1 k2):
//
//   stage 1   for each j: DFT of size R0 over q -> m
//   stage 2   for each m, i: times exp(-i 2 pi l m / (R0 R1)), DFT of size R1
//             over l -> k1, times exp(-i 2 pi i (m + R0 k1) / N)
//   stage 3   for each m, k1: DFT of size R2 over i -> k2
//
// (decimation in frequency; the inverse runs the mirror image, decimation in
// time, with the conjugate twiddles).  Element (m, l, i) sits at
// m S0 + l S1 + i, and every butterfly writes where it read: stage 2 leaves
// k1 in l's place, stage 3 leaves k2 in i's place.  So an exchange needs no
// second buffer and no barrier before its writes, and the R1 R2-point
// sub-transform of one m (stages 2 and 3) stays within one group of G lanes
// of a warp (8, 16 or 32, the smallest that holds max(R1, R2)): its exchange
// is ordered by __syncwarp alone.  Only the exchange between stage 1 and the
// sub-transforms crosses warps, which leaves one block barrier per transform
// where the self-sorting order needs two per exchange.
//
// Twiddles: the factor exp(-i 2 pi (i + R2 l) m / N) between stages 1 and 2
// is split into its l part, R0 R1 values that a block keeps in shared memory
// (w1; the lanes of a group read one address), and its i part, which is the
// same for the whole butterfly and joins the table of stage 2's outputs (w2,
// N values).  The passes are bound by shared-memory and L1 bandwidth: a
// table of stage 1 of its own would add 8 bytes per point and direction.
// ---------------------------------------------------------------------------
template <int N_, int R0_, int R1_, int R2_>
struct Geo {
    static constexpr int N = N_, R0 = R0_, R1 = R1_, R2 = R2_, N1 = R1_ * R2_;
    static_assert(R0 * R1 * R2 == N, "radices must multiply to N");
    static constexpr int RM = R1 > R2 ? R1 : R2;
    static_assert(RM <= 32, "a sub-transform's lanes are one warp at most");
    static constexpr int G = RM <= 8 ? 8 : RM <= 16 ? 16 : 32;  // lanes of a sub-transform
    static constexpr int GPW = 32 / G;                          // sub-transforms per warp and round
    static constexpr int R1P = (R1 + 1) / 2 * 2;                // entries of w1 per m (16-byte rows)
    static constexpr int W1 = R0 > 1 ? (R0 * R1P + 7) / 8 * 8 : 0;  // shared-memory entries of w1
    static constexpr bool STREAM = 4ll * N * N <= 129ll << 20;  // see ld_once
    // position in a spectrum column of frequency (m, k1, k2): the lanes of
    // a sub-transform (k1) read VK consecutive k2 each, side by side
    static constexpr int VK = R2 % 4 == 0 ? 4 : R2 % 2 == 0 ? 2 : 1;
    static constexpr __host__ __device__ int kpos(int m, int k1, int k2)
    {
        return ((m * (R2 / VK) + k2 / VK) * R1 + k1) * VK + k2 % VK;
    }
};

// Strides of the in-place layout.  Where R2 is even, stage 3 moves its R2
// consecutive elements 16 bytes at a time: S1 is even with S1 / 2 odd, and S0
// likewise (eight lanes of a 16-byte access on consecutive k1, or on
// consecutive m in the row passes' sweep, then hit distinct banks); S1 = R2
// wherever that is so already, which keeps stage 1's writes consecutive.
// Where R2 is odd the accesses are 8 bytes, and S1 and S0 are odd.
template <class Ge>
struct Lay {
    static constexpr bool VEC = Ge::R2 % 2 == 0;
    static constexpr int S1 = !VEC ? Ge::R2 : (Ge::R2 / 2) % 2 ? Ge::R2 : Ge::R2 + 2;
    static constexpr int S0_ = Ge::R1 * S1;
    static constexpr int S0 = !VEC ? S0_ | 1 : (S0_ / 2) % 2 ? S0_ : S0_ + 2;
    // elements of one transform, ELEMS mod 16 = 8: two transforms taken by
    // alternating lanes do not share banks (and starts stay 16-byte aligned)
    static constexpr int ELEMS = (Ge::R0 * S0 + 7) / 16 * 16 + 8;
    static_assert(ELEMS >= Ge::R0 * S0, "layout extent");
};

template <class C> __device__ __forceinline__ C cmulc(C a, C w)  // a conj(w)
{
    return mk<C>(a.x * w.x + a.y * w.y, a.y * w.x - a.x * w.y);
}

// address of stage 1's butterfly j within a transform (its outputs m: + m S0)
template <class Ge>
__device__ __forceinline__ int stage1_addr(int j)
{
    return Lay<Ge>::S1 == Ge::R2 ? j : j + (j / Ge::R2) * (Lay<Ge>::S1 - Ge::R2);
}

// Loads that pass through once.  Where a square map's U (4 N^2 bytes) stays in
// the 129 MB L2, T, U and the spectra are kept out of L1, which holds the
// table w2: inverse row pass 41.3 -> 37.7 us at 4704, 51.5 -> 46.5 at 5376,
// 73 -> 70 with eight spectra at 2250.  Beyond that the same loads cost more
// (inverse row pass 709 -> 748, column pass 989 -> 1044 us at 17280: without
// L1 allocation they fetch less of a line from memory at a time), and stay
// plain.  The volatile forms are for what the previous grid
// wrote: they stay behind the wait for it.
template <class Ge, class V>
__device__ __forceinline__ V ld_once(const V* p)
{
    V v;
    if constexpr (!Ge::STREAM) {
        v = *p;
    } else if constexpr (sizeof(V) == 8) {
        asm volatile("ld.global.L1::no_allocate.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
    } else {
        asm volatile("ld.global.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];"
                     : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
    }
    return v;
}
template <class Ge, class V>
__device__ __forceinline__ V ld_spectrum(const V* p)
{
    V v;
    if constexpr (!Ge::STREAM || sizeof(V) == 4) {
        v = __ldg(p);
    } else if constexpr (sizeof(V) == 8) {
        asm("ld.global.nc.L1::no_allocate.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
    } else {
        asm("ld.global.nc.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];"
            : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
    }
    return v;
}

// the block's copy of w1 (read after the barrier that follows stage 1)
template <class Ge>
__device__ __forceinline__ void load_w1(float2* w1, const float2* __restrict__ table, int t, int th)
{
    if constexpr (Ge::R0 > 1)
        for (int i = t; i < Ge::R0 * Ge::R1P; i += th) w1[i] = __ldg(table + i);
}

// x[l] *= w1[m][l] (CONJ: its conjugate)
template <class Ge, bool CONJ>
__device__ __forceinline__ void twiddle_in(float2 (&x)[Ge::R1], const float2* w1m)
{
    if constexpr (Ge::R0 > 1) {
#pragma unroll
        for (int l = 0; l < Ge::R1; l += 2) {
            const float4 w = *reinterpret_cast<const float4*>(w1m + l);
            if (l > 0) x[l] = CONJ ? cmulc(x[l], make_float2(w.x, w.y)) : cmul(x[l], make_float2(w.x, w.y));
            if (l + 1 < Ge::R1)
                x[l + 1] = CONJ ? cmulc(x[l + 1], make_float2(w.z, w.w)) : cmul(x[l + 1], make_float2(w.z, w.w));
        }
    }
}

// stage 2 of lane i of sub-transform m at b (x loaded): twiddles and DFT over l, in place
template <class Ge>
__device__ __forceinline__ void stage2_fwd(float2 (&x)[Ge::R1], float2* b, int m, int i, const float2* w1,
                                           const float2* __restrict__ w2)
{
    constexpr int K0 = Ge::R0 > 1 ? 0 : 1;  // (m = 0: output k1 = 0 has no twiddle)
    twiddle_in<Ge, false>(x, w1 + m * Ge::R1P);
    Dft<Ge::R1, -1, float2>::run(x);
    const float2* w = w2 + m * Ge::N1 + i;
    if constexpr (K0 == 1) b[i] = x[0];
#pragma unroll
    for (int k = K0; k < Ge::R1; ++k) b[i + k * Lay<Ge>::S1] = cmul(x[k], __ldg(w + k * Ge::R2));
}
template <class Ge>
__device__ __forceinline__ void stage2_inv(float2 (&x)[Ge::R1], const float2* b, int m, int i, const float2* w1,
                                           const float2* __restrict__ w2)
{
    constexpr int K0 = Ge::R0 > 1 ? 0 : 1;
    const float2* w = w2 + m * Ge::N1 + i;
    if constexpr (K0 == 1) x[0] = b[i];
#pragma unroll
    for (int k = K0; k < Ge::R1; ++k) x[k] = cmulc(b[i + k * Lay<Ge>::S1], __ldg(w + k * Ge::R2));
    Dft<Ge::R1, 1, float2>::run(x);
    twiddle_in<Ge, true>(x, w1 + m * Ge::R1P);
}

// the R2 consecutive elements of lane k1
template <class Ge>
__device__ __forceinline__ void load_run(float2 (&f)[Ge::R2], const float2* b, int k1)
{
    const float2* p = b + k1 * Lay<Ge>::S1;
    if constexpr (Lay<Ge>::VEC) {
#pragma unroll
        for (int k = 0; k < Ge::R2; k += 2) {
            const float4 q = *reinterpret_cast<const float4*>(p + k);
            f[k] = make_float2(q.x, q.y);
            f[k + 1] = make_float2(q.z, q.w);
        }
    } else {
#pragma unroll
        for (int k = 0; k < Ge::R2; ++k) f[k] = p[k];
    }
}
template <class Ge>
__device__ __forceinline__ void store_run(const float2 (&f)[Ge::R2], float2* b, int k1)
{
    float2* p = b + k1 * Lay<Ge>::S1;
    if constexpr (Lay<Ge>::VEC) {
#pragma unroll
        for (int k = 0; k < Ge::R2; k += 2)
            *reinterpret_cast<float4*>(p + k) = make_float4(f[k].x, f[k].y, f[k + 1].x, f[k + 1].y);
    } else {
#pragma unroll
        for (int k = 0; k < Ge::R2; ++k) p[k] = f[k];
    }
}

}  // namespace lpk
