// Mixed-radix FFTs of lines of at most 256 points (sm_103a), two register
// passes per line with one exchange through shared memory between them.
//
// A line of n = P1 P2 points is the Stockham autosort algorithm over a list of
// small radices (2, 3, 4, 5, and for some lengths in-register 8, 9, 12, 15,
// 16), its consecutive radices taken in two groups whose products are P1 and
// P2.  One thread does a whole group for one butterfly in registers: it loads
// the P inputs x[j + q n/P], runs the group's radices one after another and
// stores the P outputs, so that the shared-memory traffic is that of two
// passes however many radices there are.
//
// Group of radices A, B, C after Ns = product of the radices before it
// (j in [0, n/P), k = j mod Ns):
//   input q = (ra B + rb) C + rc        at j + q n/P
//   radix A over ra, twiddle W_{Ns A}^(ra k),              output digit ka
//   radix B over rb, twiddle W_{Ns A B}^(rb (k + ka Ns)),  output digit kb
//   radix C over rc, twiddle W_{Ns P}^(rc (k + (ka + A kb) Ns)), digit kc
//   output q' = ka + A kb + A B kc      at (j - k) P + k + q' Ns
// In the first group Ns = 1 and k = 0: its twiddles are constants.  Forward
// uses W_n = exp(-2 pi i/n), inverse its conjugate; neither scales.
//
// Every constant of a transform (table twiddles, the sines and cosines inside
// the radix 3, 5, 8, 9 and 16 butterflies) is held as a pair hi + lo of FP32
// numbers whose sum is the FP64 value, and a product x W is formed as
// x W_hi + x W_lo.  With the constants rounded to FP32 alone, the rounding
// errors of the few twiddles a smooth field's low frequencies go through add
// up coherently: the transform's low-frequency amplitudes come out biased by
// a few 1e-8, which shifts the energy of Eq. (Eoffk) (dominated by those
// frequencies) by ~1e-7 of itself.  With the pair the constants are exact to
// ~1e-15 and only the (unbiased) rounding of the arithmetic remains.
#pragma once

#include "common.cuh"

#include <type_traits>
#include <utility>

namespace vdw {

// packed FP32 pairs: one instruction for both parts (the transforms are bound
// by issue slots and shared memory; 1-5 % of the plane kernels' time)
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return __fadd2_rn(a, make_float2(-b.x, -b.y)); }
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
// a * conj(b)
__device__ __forceinline__ float2 cmulc(float2 a, float2 b) {
    return make_float2(fmaf(a.x, b.x, a.y * b.y), fmaf(a.y, b.x, -a.x * b.y));
}
// -i a (forward) or +i a (inverse)
template <bool INV>
__device__ __forceinline__ float2 mul_mi(float2 a) {
    return INV ? make_float2(-a.y, a.x) : make_float2(a.y, -a.x);
}

// A twiddle W as {W_hi.x, W_hi.y, W_lo.x, W_lo.y}, W = W_hi + W_lo.
using Tw = float4;
// a W (the small product a W_lo first, then the main one accumulated on it)
__device__ __forceinline__ float2 cmul_tw(float2 a, Tw w) {
    const float lr = fmaf(a.x, w.z, -a.y * w.w);
    const float li = fmaf(a.x, w.w, a.y * w.z);
    return make_float2(fmaf(a.x, w.x, fmaf(-a.y, w.y, lr)), fmaf(a.x, w.y, fmaf(a.y, w.x, li)));
}
// a conj(W)
__device__ __forceinline__ float2 cmulc_tw(float2 a, Tw w) {
    const float lr = fmaf(a.x, w.z, a.y * w.w);
    const float li = fmaf(a.y, w.z, -a.x * w.w);
    return make_float2(fmaf(a.x, w.x, fmaf(a.y, w.y, lr)), fmaf(a.y, w.x, fmaf(-a.x, w.y, li)));
}
template <bool INV>
__device__ __forceinline__ float2 tw_mul(float2 a, Tw w) {
    return INV ? cmulc_tw(a, w) : cmul_tw(a, w);
}
// A twiddle held as its FP32 value only (transforms whose results tolerate
// the constant rounding: the inverse transforms and those of w).
template <bool INV>
__device__ __forceinline__ float2 tw_mul(float2 a, float2 w) {
    return INV ? cmulc(a, w) : cmul(a, w);
}
// store a hi/lo twiddle as a table entry of either kind
__device__ __forceinline__ void tw_put(Tw* d, Tw s) { *d = s; }
__device__ __forceinline__ void tw_put(float2* d, Tw s) { *d = make_float2(s.x, s.y); }
// Real constant c = hi + lo from its FP64 value.
struct KPair {
    float h, l;
};
__host__ __device__ constexpr KPair kpair(double c) { return KPair{(float)c, (float)(c - (double)(float)c)}; }
// x c
__device__ __forceinline__ float kmul(float x, KPair c) { return fmaf(x, c.h, x * c.l); }
// x c + y d (one rounding of the main products' sum)
__device__ __forceinline__ float kmul2(float x, KPair c, float y, KPair d) {
    return fmaf(x, c.h, fmaf(y, d.h, fmaf(x, c.l, y * d.l)));
}

template <int R, bool INV>
__device__ __forceinline__ void dft(float2* v);

template <>
__device__ __forceinline__ void dft<2, false>(float2* v) {
    float2 a = cadd(v[0], v[1]), b = csub(v[0], v[1]);
    v[0] = a; v[1] = b;
}
template <>
__device__ __forceinline__ void dft<2, true>(float2* v) { dft<2, false>(v); }

template <bool INV>
__device__ __forceinline__ void dft3(float2* v) {
    constexpr KPair s3 = kpair(0.86602540378443864676);  // sin(2 pi/3)
    float2 s = cadd(v[1], v[2]);
    float2 d = csub(v[1], v[2]);
    float2 x0 = cadd(v[0], s);
    float2 t = make_float2(fmaf(-0.5f, s.x, v[0].x), fmaf(-0.5f, s.y, v[0].y));
    const float2 dm = mul_mi<INV>(d);
    float2 u = make_float2(kmul(dm.x, s3), kmul(dm.y, s3));
    v[0] = x0;
    v[1] = cadd(t, u);
    v[2] = csub(t, u);
}
template <>
__device__ __forceinline__ void dft<3, false>(float2* v) { dft3<false>(v); }
template <>
__device__ __forceinline__ void dft<3, true>(float2* v) { dft3<true>(v); }

template <bool INV>
__device__ __forceinline__ void dft4(float2* v) {
    float2 a = cadd(v[0], v[2]), b = csub(v[0], v[2]);
    float2 c = cadd(v[1], v[3]), d = mul_mi<INV>(csub(v[1], v[3]));
    v[0] = cadd(a, c);
    v[2] = csub(a, c);
    v[1] = cadd(b, d);
    v[3] = csub(b, d);
}
template <>
__device__ __forceinline__ void dft<4, false>(float2* v) { dft4<false>(v); }
template <>
__device__ __forceinline__ void dft<4, true>(float2* v) { dft4<true>(v); }

template <bool INV>
__device__ __forceinline__ void dft5(float2* v) {
    constexpr KPair c1 = kpair(0.30901699437494742410);   // cos(2 pi/5)
    constexpr KPair c2 = kpair(-0.80901699437494742410);  // cos(4 pi/5)
    constexpr KPair s1 = kpair(0.95105651629515357212);   // sin(2 pi/5)
    constexpr KPair s2 = kpair(0.58778525229247312917);   // sin(4 pi/5)
    constexpr KPair ms1 = kpair(-0.95105651629515357212);
    float2 a1 = cadd(v[1], v[4]), b1 = csub(v[1], v[4]);
    float2 a2 = cadd(v[2], v[3]), b2 = csub(v[2], v[3]);
    float2 x0 = cadd(v[0], cadd(a1, a2));
    float2 t1 = make_float2(v[0].x + kmul2(a1.x, c1, a2.x, c2), v[0].y + kmul2(a1.y, c1, a2.y, c2));
    float2 t2 = make_float2(v[0].x + kmul2(a1.x, c2, a2.x, c1), v[0].y + kmul2(a1.y, c2, a2.y, c1));
    float2 u1 = mul_mi<INV>(make_float2(kmul2(b1.x, s1, b2.x, s2), kmul2(b1.y, s1, b2.y, s2)));
    float2 u2 = mul_mi<INV>(make_float2(kmul2(b1.x, s2, b2.x, ms1), kmul2(b1.y, s2, b2.y, ms1)));
    v[0] = x0;
    v[1] = cadd(t1, u1);
    v[4] = csub(t1, u1);
    v[2] = cadd(t2, u2);
    v[3] = csub(t2, u2);
}
template <>
__device__ __forceinline__ void dft<5, false>(float2* v) { dft5<false>(v); }
template <>
__device__ __forceinline__ void dft<5, true>(float2* v) { dft5<true>(v); }

// ---- in-register radices ---------------------------------------------------
template <bool INV>
__device__ __forceinline__ void dft8(float2* v) {
    constexpr KPair r2 = kpair(0.70710678118654752440);
    // two radix-4 transforms of the even and odd samples
    float2 e[4] = {v[0], v[2], v[4], v[6]};
    float2 o[4] = {v[1], v[3], v[5], v[7]};
    dft4<INV>(e);
    dft4<INV>(o);
    // odd twiddles W8^k, k = 1..3 (conjugate for the inverse)
    const float s = INV ? 1.f : -1.f;
    const float2 o1 = make_float2(kmul(o[1].x - s * o[1].y, r2), kmul(o[1].y + s * o[1].x, r2));
    const float2 o2 = make_float2(-s * o[2].y, s * o[2].x);
    const float2 o3 = make_float2(kmul(-o[3].x - s * o[3].y, r2), kmul(-o[3].y + s * o[3].x, r2));
    v[0] = cadd(e[0], o[0]);
    v[4] = csub(e[0], o[0]);
    v[1] = cadd(e[1], o1);
    v[5] = csub(e[1], o1);
    v[2] = cadd(e[2], o2);
    v[6] = csub(e[2], o2);
    v[3] = cadd(e[3], o3);
    v[7] = csub(e[3], o3);
}
template <>
__device__ __forceinline__ void dft<8, false>(float2* v) { dft8<false>(v); }
template <>
__device__ __forceinline__ void dft<8, true>(float2* v) { dft8<true>(v); }

// ---- composite radices, evaluated in registers ----------------------------
// W_N^e = exp(-2 pi i e / N) (conjugated for the inverse) for the few
// exponents the Cooley-Tukey splits 3x3 and 4x4 need.
template <int N, int E>
__device__ __forceinline__ Tw wconst() {
    static_assert(N == 9 || N == 16, "no constants for this length");
    double c = 1.0, s = 0.0;  // cos, sin of 2 pi E / N
    if (N == 9) {
        if (E == 1) { c = 0.766044443118978035202; s = 0.642787609686539326323; }
        if (E == 2) { c = 0.173648177666930348852; s = 0.984807753012208059367; }
        if (E == 4) { c = -0.939692620785908384054; s = 0.342020143325668733044; }
    } else {
        if (E == 1) { c = 0.923879532511286756128; s = 0.382683432365089771728; }
        if (E == 2) { c = 0.707106781186547524401; s = 0.707106781186547524401; }
        if (E == 3) { c = 0.382683432365089771728; s = 0.923879532511286756128; }
        if (E == 4) { c = 0.0; s = 1.0; }
        if (E == 6) { c = -0.707106781186547524401; s = 0.707106781186547524401; }
        if (E == 9) { c = -0.923879532511286756128; s = -0.382683432365089771728; }
    }
    const KPair cr = kpair(c), ci = kpair(-s);
    return make_float4(cr.h, ci.h, cr.l, ci.l);
}

// Cooley-Tukey in registers, N = R1 R2, input index R2 n1 + n2, output
// k1 + R1 k2: R2 transforms of length R1, twiddles W_N^(n2 k1), R1
// transforms of length R2.
template <int R1, int R2, bool INV, int N2 = 0, int K1 = 1>
__device__ __forceinline__ void ct_twiddle(float2 (&Y)[R1 * R2]) {
    if constexpr (N2 < R2) {
        if constexpr (K1 < R1) {
            if constexpr (N2 > 0) {
                const Tw w = wconst<R1 * R2, N2 * K1>();
                Y[N2 * R1 + K1] = tw_mul<INV>(Y[N2 * R1 + K1], w);
            }
            ct_twiddle<R1, R2, INV, N2, K1 + 1>(Y);
        } else {
            ct_twiddle<R1, R2, INV, N2 + 1, 1>(Y);
        }
    }
}

template <int R1, int R2, bool INV>
__device__ __forceinline__ void dft_ct(float2* v) {
    float2 Y[R1 * R2];
#pragma unroll
    for (int n2 = 0; n2 < R2; ++n2) {
        float2 t[R1];
#pragma unroll
        for (int n1 = 0; n1 < R1; ++n1) t[n1] = v[R2 * n1 + n2];
        dft<R1, INV>(t);
#pragma unroll
        for (int k1 = 0; k1 < R1; ++k1) Y[n2 * R1 + k1] = t[k1];
    }
    ct_twiddle<R1, R2, INV>(Y);
#pragma unroll
    for (int k1 = 0; k1 < R1; ++k1) {
        float2 t[R2];
#pragma unroll
        for (int n2 = 0; n2 < R2; ++n2) t[n2] = Y[n2 * R1 + k1];
        dft<R2, INV>(t);
#pragma unroll
        for (int k2 = 0; k2 < R2; ++k2) v[k1 + R1 * k2] = t[k2];
    }
}

constexpr int inv_mod(int a, int m) {
    for (int x = 1; x < m; ++x)
        if ((a * x) % m == 1) return x;
    return 1;
}

// Good-Thomas (prime-factor) split for coprime R1, R2: input index
// (R2 n1 + R1 n2) mod N, output index by the Chinese remainder theorem; no
// twiddles between the two sets of short transforms.
template <int R1, int R2, bool INV>
__device__ __forceinline__ void dft_pfa(float2* v) {
    constexpr int N = R1 * R2;
    constexpr int i1 = inv_mod(R2 % R1, R1), i2 = inv_mod(R1 % R2, R2);
    float2 Y[N];
#pragma unroll
    for (int n2 = 0; n2 < R2; ++n2) {
        float2 t[R1];
#pragma unroll
        for (int n1 = 0; n1 < R1; ++n1) t[n1] = v[(R2 * n1 + R1 * n2) % N];
        dft<R1, INV>(t);
#pragma unroll
        for (int k1 = 0; k1 < R1; ++k1) Y[n2 * R1 + k1] = t[k1];
    }
#pragma unroll
    for (int k1 = 0; k1 < R1; ++k1) {
        float2 t[R2];
#pragma unroll
        for (int n2 = 0; n2 < R2; ++n2) t[n2] = Y[n2 * R1 + k1];
        dft<R2, INV>(t);
#pragma unroll
        for (int k2 = 0; k2 < R2; ++k2) v[(k1 * R2 * i1 + k2 * R1 * i2) % N] = t[k2];
    }
}

template <> __device__ __forceinline__ void dft<9, false>(float2* v) { dft_ct<3, 3, false>(v); }
template <> __device__ __forceinline__ void dft<9, true>(float2* v) { dft_ct<3, 3, true>(v); }
template <> __device__ __forceinline__ void dft<12, false>(float2* v) { dft_pfa<4, 3, false>(v); }
template <> __device__ __forceinline__ void dft<12, true>(float2* v) { dft_pfa<4, 3, true>(v); }
template <> __device__ __forceinline__ void dft<15, false>(float2* v) { dft_pfa<5, 3, false>(v); }
template <> __device__ __forceinline__ void dft<15, true>(float2* v) { dft_pfa<5, 3, true>(v); }
template <> __device__ __forceinline__ void dft<16, false>(float2* v) { dft_ct<4, 4, false>(v); }
template <> __device__ __forceinline__ void dft<16, true>(float2* v) { dft_ct<4, 4, true>(v); }

// ---------------------------------------------------------------------------
// groups of radices
// ---------------------------------------------------------------------------
// f(integral_constant<int, i>) for i = 0 .. N-1
template <class F, int... I>
__device__ __forceinline__ void static_for_impl(F&& f, std::integer_sequence<int, I...>) {
    (f(std::integral_constant<int, I>{}), ...);
}
template <int N, class F>
__device__ __forceinline__ void static_for(F&& f) {
    static_for_impl(f, std::make_integer_sequence<int, N>{});
}

// cos and sin of 2 pi e/n for the constant twiddles of a first group, by
// their series on [0, pi/4] after reduction to the first octant (exact at the
// multiples of a quarter turn)
constexpr double series_cos(double x) {
    double s = 0.0, t = 1.0;
    for (int k = 0; k < 14; ++k) {
        s += t;
        t *= -x * x / ((2.0 * k + 1.0) * (2.0 * k + 2.0));
    }
    return s;
}
constexpr double series_sin(double x) {
    double s = 0.0, t = x;
    for (int k = 0; k < 14; ++k) {
        s += t;
        t *= -x * x / ((2.0 * k + 2.0) * (2.0 * k + 3.0));
    }
    return s;
}
constexpr double turn_cos(int e, int n);
constexpr double turn_sin(int e, int n) {
    e %= n;
    if (2 * e > n) return -turn_sin(n - e, n);                 // second half: odd
    if (4 * e > n) return turn_sin(n - 2 * e, 2 * n);          // sin(pi - x)
    if (8 * e > n) return series_cos(6.28318530717958647692 * (n - 4 * e) / (4.0 * n));
    return series_sin(6.28318530717958647692 * e / (double)n);
}
constexpr double turn_cos(int e, int n) { return turn_sin(4 * e + n, 4 * n); }

// a W_N^E (conjugated for the inverse) with a constant twiddle: hi/lo pairs
// (W = Tw) or the FP32 value (W = float2)
template <int N, int E, bool INV, class W>
__device__ __forceinline__ float2 mul_root(float2 a) {
    constexpr int e = ((E % N) + N) % N;
    if constexpr (e == 0) return a;
    else if constexpr (4 * e == N) return mul_mi<INV>(a);
    else if constexpr (2 * e == N) return make_float2(-a.x, -a.y);
    else if constexpr (4 * e == 3 * N) return mul_mi<!INV>(a);
    else {
        constexpr KPair cr = kpair(turn_cos(e, N)), ci = kpair(-turn_sin(e, N));
        if constexpr (sizeof(W) == sizeof(float4)) return tw_mul<INV>(a, make_float4(cr.h, ci.h, cr.l, ci.l));
        else return tw_mul<INV>(a, make_float2(cr.h, ci.h));
    }
}

template <int A_, int B_ = 1, int C_ = 1>
struct Grp {
    static constexpr int A = A_, B = B_, C = C_, P = A_ * B_ * C_;
    // output digit q' of register i (the radices run in place: register
    // (ka B + kb) C + kc ends with output ka + A kb + A B kc)
    static constexpr int digit(int i) { return i / (B * C) + A * ((i / C) % B) + A * B * (i % C); }
    // register of output digit d
    static constexpr int reg(int d) { return ((d % A) * B + (d / A) % B) * C + d / (A * B); }
};

// The group's transform of v (input q in register q).  FIRST: Ns = 1,
// constant twiddles.  Otherwise tw points at the group's table (k_twiddles)
// plus k: the twiddle of entry i is tw[i Ns].
template <class G, bool INV, bool FIRST, class W>
__device__ __forceinline__ void group_fft(float2 (&v)[G::P], const W* tw, int Ns) {
    constexpr int A = G::A, B = G::B, C = G::C, BC = B * C;
    if constexpr (A > 1) {
        static_for<BC>([&](auto S) {
            constexpr int s = decltype(S)::value;
            float2 t[A];
#pragma unroll
            for (int r = 0; r < A; ++r) {
                t[r] = v[r * BC + s];
                if (!FIRST && r > 0) t[r] = tw_mul<INV>(t[r], tw[(r - 1) * Ns]);
            }
            dft<A, INV>(t);
#pragma unroll
            for (int r = 0; r < A; ++r) v[r * BC + s] = t[r];
        });
    }
    if constexpr (B > 1) {
        static_for<A>([&](auto KA) {
            constexpr int ka = decltype(KA)::value;
            static_for<C>([&](auto S) {
                constexpr int s = decltype(S)::value;
                float2 t[B];
                static_for<B>([&](auto R) {
                    constexpr int r = decltype(R)::value;
                    t[r] = v[ka * BC + r * C + s];
                    if constexpr (FIRST) t[r] = mul_root<A * B, r * ka, INV, W>(t[r]);
                    else if constexpr (r > 0) t[r] = tw_mul<INV>(t[r], tw[(A - 1 + (r - 1) * A + ka) * Ns]);
                });
                dft<B, INV>(t);
#pragma unroll
                for (int r = 0; r < B; ++r) v[ka * BC + r * C + s] = t[r];
            });
        });
    }
    if constexpr (C > 1) {
        static_for<A * B>([&](auto K) {
            constexpr int ka = decltype(K)::value / B, kb = decltype(K)::value % B, kk = ka + A * kb;
            float2 t[C];
            static_for<C>([&](auto R) {
                constexpr int r = decltype(R)::value;
                t[r] = v[ka * BC + kb * C + r];
                if constexpr (FIRST) t[r] = mul_root<A * B * C, r * kk, INV, W>(t[r]);
                else if constexpr (r > 0) t[r] = tw_mul<INV>(t[r], tw[(A * B - 1 + (r - 1) * A * B + kk) * Ns]);
            });
            dft<C, INV>(t);
#pragma unroll
            for (int r = 0; r < C; ++r) v[ka * BC + kb * C + r] = t[r];
        });
    }
}

// ---------------------------------------------------------------------------
// line schedules
// ---------------------------------------------------------------------------
// Compile-time lengths (the grids 180 x 180 x 72 and 256 x 256 x 96): two
// in-register radices each.  Any other length takes its groups at run time
// from the list 4, .., 4, 2, 3, .., 3, 5, .., 5 (make_line_plan).
// CtLine<N, true>: the order of the inverse x transforms of u and D.w
// (LinePlan p1i, merge_swaps).
template <int CN> struct CtGroups { using G1 = Grp<1>; using G2 = Grp<1>; };
template <> struct CtGroups<180> { using G1 = Grp<15>; using G2 = Grp<12>; };
template <> struct CtGroups<72> { using G1 = Grp<9>; using G2 = Grp<8>; };
template <> struct CtGroups<256> { using G1 = Grp<16>; using G2 = Grp<16>; };
template <> struct CtGroups<96> { using G1 = Grp<12>; using G2 = Grp<8>; };
template <int CN, bool XI = false>
struct CtLine {
    using A = typename CtGroups<CN>::G1;
    using B = typename CtGroups<CN>::G2;
    static constexpr bool SWAP = XI && merge_swaps(A::P, B::P, MERGE_CT);
    using G1 = std::conditional_t<SWAP, B, A>;
    using G2 = std::conditional_t<SWAP, A, B>;
};

// Run-time lengths: any, or (ANY16) with no group above 16.  The second kind
// leaves the larger groups' registers out of a kernel.
constexpr int ANY = 0, ANY16 = -1;

// f(group of product P) for a run-time P.  A product stands for one list of
// radices; P1 of an even length is one of the first set, of an odd one also
// of the second, and P2 one of the third.
template <bool ODD, bool BIG, class F>
__device__ __forceinline__ void first_group(int P, F&& f) {
    switch (P) {
        case 2: f(Grp<2>{}); break;
        case 4: f(Grp<4>{}); break;
        case 6: f(Grp<2, 3>{}); break;
        case 8: f(Grp<4, 2>{}); break;
        case 10: f(Grp<2, 5>{}); break;
        case 12: f(Grp<4, 3>{}); break;
        case 16: f(Grp<4, 4>{}); break;
        default:
            if constexpr (BIG) {
                switch (P) {
                    case 18: f(Grp<2, 3, 3>{}); break;
                    case 20: f(Grp<4, 5>{}); break;
                    case 24: f(Grp<4, 2, 3>{}); break;
                    default: break;
                }
            }
            if constexpr (ODD) {
                switch (P) {
                    case 3: f(Grp<3>{}); break;
                    case 5: f(Grp<5>{}); break;
                    case 9: f(Grp<3, 3>{}); break;
                    case 15: f(Grp<3, 5>{}); break;
                    default: break;
                }
            }
            if constexpr (ODD && BIG) {
                switch (P) {
                    case 25: f(Grp<5, 5>{}); break;
                    case 27: f(Grp<3, 3, 3>{}); break;
                    default: break;
                }
            }
    }
}
// WIDE: also the groups that are second only in an inverse x transform
template <bool BIG, bool WIDE, class F>
__device__ __forceinline__ void second_group(int P, F&& f) {
    switch (P) {
        case 1: f(Grp<1>{}); break;
        case 2: f(Grp<2>{}); break;
        case 3: f(Grp<3>{}); break;
        case 4: f(Grp<4>{}); break;
        case 5: f(Grp<5>{}); break;
        case 6: f(Grp<2, 3>{}); break;
        case 8: f(Grp<4, 2>{}); break;
        case 9: f(Grp<3, 3>{}); break;
        case 10: f(Grp<2, 5>{}); break;
        case 12: f(Grp<4, 3>{}); break;
        case 15: f(Grp<3, 5>{}); break;
        case 16: f(Grp<4, 4>{}); break;
        default:
            if constexpr (BIG) {
                if (P == 25) f(Grp<5, 5>{});
            }
            if constexpr (BIG && WIDE) {
                if (P == 18) f(Grp<2, 3, 3>{});
                if (P == 20) f(Grp<4, 5>{});
                if (P == 24) f(Grp<4, 2, 3>{});
            }
    }
}
template <int CN, bool ODD, bool XI = false, class F>
__device__ __forceinline__ void on_first(const LinePlan& lp, F&& f) {
    if constexpr (CN > 0) f(typename CtLine<CN, XI>::G1{});
    else first_group<ODD || XI, CN == ANY>(lp.P1, f);
}
template <int CN, bool XI = false, class F>
__device__ __forceinline__ void on_second(const LinePlan& lp, F&& f) {
    if constexpr (CN > 0) f(typename CtLine<CN, XI>::G2{});
    else second_group<CN == ANY, XI>(lp.P2, f);
}

}  // namespace vdw
