// Shared pieces of the transform kernels: block reductions, twiddle loads, and
// the forward / inverse transform of one y plane (N3 rows of N1 reals <->
// N3 x Nh half spectrum) through shared memory.
#pragma once
#include "fft.cuh"

namespace vdw {

// ---------------------------------------------------------------------------
// reductions
// ---------------------------------------------------------------------------
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// Deterministic block sum (fixed order); result valid in thread 0.
__device__ inline double block_sum(double v, double* red) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    v = warp_sum(v);
    __syncthreads();
    if (lane == 0) red[warp] = v;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x == 0)
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s += red[i];
    return s;
}

// A line's second-group twiddle table (n - P1 entries) into shared memory;
// W = Tw keeps the hi/lo pairs, W = float2 the FP32 values only.
template <class W>
__device__ __forceinline__ void load_twiddles(W* dst, const Tw* __restrict__ src, int n) {
    for (int i = threadIdx.x; i < n; i += blockDim.x) tw_put(dst + i, src[i]);
}

// i / d for a small divisor (1 <= d < 256) and 0 <= i < 2^24 by one
// multiply-high with m = ceil(2^32 / d): the error term i (m d - 2^32) / 2^32 /
// d stays below 1/d, so the quotient is exact in that range.
struct SmallDiv {
    unsigned m;
    int d;
};
__device__ __forceinline__ SmallDiv small_div(int d) {
    SmallDiv s;
    s.d = d;
    s.m = d == 1 ? 0u : 0xFFFFFFFFu / (unsigned)d + 1u;
    return s;
}
__device__ __forceinline__ int sdiv(int i, SmallDiv s) { return s.d == 1 ? i : (int)__umulhi((unsigned)i, s.m); }
// the same with the divisor known at compile time when C > 0
template <int C>
__device__ __forceinline__ int cdiv(int i, SmallDiv s) {
    if constexpr (C > 0) return (int)((unsigned)i / (unsigned)C);
    else return sdiv(i, s);
}

// ---------------------------------------------------------------------------
// plane helpers (one y plane, N3 rows of N1 reals <-> N3 x Nh half spectrum)
// ---------------------------------------------------------------------------
// Points in packed order: q = ((y (N3/2) + j) N1 + x) 2 + s is the point
// (x, y, z = 2j + s).  A field written in this order fills the packed real
// rows of its y plane (real rows 2j and 2j + 1 interleaved in complex row j)
// with consecutive addresses.  Sets (y, z, x, j); returns the flat index
// (z N2 + y) N1 + x.
__device__ __forceinline__ long long packed_point(long long q, const GridArgs& g, int& y, int& z, int& x, int& j) {
    const int s = (int)(q & 1);
    const int nh3 = g.N3 >> 1;
    if (g.fast) {
        const unsigned t = (unsigned)(q >> 1);
        const unsigned rr = __umulhi(t, g.m1);
        x = (int)(t - rr * (unsigned)g.N1);
        y = (int)__umulhi(rr, g.mh3);
        j = (int)(rr - (unsigned)y * (unsigned)nh3);
    } else {
        const long long t = q >> 1;
        const long long rr = t / g.N1;
        x = (int)(t - rr * g.N1);
        y = (int)(rr / nh3);
        j = (int)(rr - (long long)y * nh3);
    }
    z = 2 * j + s;
    return ((long long)z * g.N2 + y) * g.N1 + x;
}
// (x, y, z) of flat index i = (z N2 + y) N1 + x
__device__ __forceinline__ void flat_point(long long i, const GridArgs& g, int& x, int& y, int& z) {
    if (g.fast) {
        const unsigned r = __umulhi((unsigned)i, g.m1);
        x = (int)((unsigned)i - r * (unsigned)g.N1);
        z = (int)__umulhi(r, g.m2);
        y = (int)(r - (unsigned)z * (unsigned)g.N2);
    } else {
        const long long r = i / g.N1;
        x = (int)(i - r * g.N1);
        z = (int)(r / g.N2);
        y = (int)(r - (long long)z * g.N2);
    }
}
// Packed real rows: real rows 2j and 2j+1 of a plane are the real and
// imaginary parts of complex row j, which starts at complex offset 2 Nh j.
// This is the float offset, within its plane, of real point (x, z = 2j + s).
__device__ __forceinline__ int packed_offset(int x, int j, int s, int Nh) { return 4 * j * Nh + 2 * x + s; }

// ---------------------------------------------------------------------------
// y lines (pencils)
// ---------------------------------------------------------------------------
// Shared-memory lines of the pencil kernels: point k1 + P1 k2 of a line sits
// at k1 + (P1 | 1) k2, a line takes pencil_stride values, and the C lines of
// a field C pencil_stride values plus a pad.  The stride is 2 (mod 16): the
// lanes that take 8 columns and 2 neighbouring points of each then hit the
// 16 distinct 8-byte banks, and the field pads do the same for lanes that
// take 4 fields and 4 neighbouring points.
__host__ __device__ __forceinline__ int pencil_stride(const LinePlan& p) {
    const int n = (p.P1 | 1) * p.P2;
    return n + ((2 - n) % 16 + 16) % 16;
}

// ---------------------------------------------------------------------------
// one y plane
// ---------------------------------------------------------------------------
// Shared memory of a plane transform: N3/2 rows, row j holding the complex
// row j = (real row 2j) + i (real row 2j + 1), and later the half spectra of
// those two rows.  Element k of a row sits at slot(k) = k plus one for every
// 2^sh runs of P elements before it, where P is the step that one pass takes
// from lane to lane and has a factor of 4 or more in common with the 16
// 8-byte banks (16 / that factor = 2^sh runs come back to the same bank); no
// pads for other P.  A row takes an odd number of slots, so that lanes on
// consecutive rows hit distinct banks.  Half spectra: real row 2j's
// value at kx takes slot(kx) of row j, real row 2j + 1's takes slot(N1 - kx)
// (two extra slots at the row's end for kx = 0 and N1/2), so that every pass
// writes where the same thread read and no pass needs a second buffer.
struct PlaneGeo {
    int run, sh;
    int len;          // slots of a row before the two extra ones
    int S;            // slots of a row
    // offset of the first element of run q, and slot of element k (dP: division by run)
    __host__ __device__ __forceinline__ constexpr int at(int q) const { return q * run + (q >> sh); }
    __device__ __forceinline__ int slot(int k, SmallDiv dP) const { return k + (sdiv(k, dP) >> sh); }
};
// forward: run P1 (the row transform's first group stores steps of P1);
// inverse: run P2 (its second group reads steps of P2).  Without the pads
// where they would not fit in shared memory (wide planes).
__host__ __device__ constexpr PlaneGeo plane_geo(int P1, int P2, bool inverse, bool pad) {
    const int run = inverse ? P2 : P1, cnt = inverse ? P1 : P2;
    const int sh = !pad ? 31 : run % 16 == 0 ? 0 : run % 8 == 0 ? 1 : run % 4 == 0 ? 2 : 31;
    const int len = run * cnt + ((cnt - 1) >> sh);
    return PlaneGeo{run, sh, len, pad ? ((len + 2) | 1) : len + 2};
}
template <int CN1, bool INVERSE, bool XI = false>
__device__ __forceinline__ PlaneGeo geo_of(const GridArgs& g) {
    if constexpr (CN1 > 0) {
        constexpr PlaneGeo p = plane_geo(CtLine<CN1, XI>::G1::P, CtLine<CN1, XI>::G2::P, INVERSE, true);
        return p;
    } else {
        const LinePlan& l = XI ? g.p1i : g.p1;
        return plane_geo(l.P1, l.P2, INVERSE, INVERSE ? g.pad_inv : g.pad_fwd);
    }
}
// the slots of kx for the even and the odd real row
__device__ __forceinline__ void half_slots(const PlaneGeo& G, SmallDiv dP, int N1, int kx, int& se, int& so) {
    const int km = N1 - kx;
    se = G.slot(kx, dP);
    so = kx == 0 ? G.len : (kx == km ? G.len + 1 : G.slot(km, dP));
}
// A second group of at most this many points is transformed for k and N1 - k
// in one thread and split into the two half spectra in its registers, which
// takes a quarter off the shared-memory accesses (180 x 180 x 72: 108 -> 101
// us, 128^3: 114 -> 100 us forward); above it the split is a pass of its own
// (registers).  So it is for the w planes (W = float2), a single wave of
// blocks where the longer thread is slower (35 against 29 us).
template <int CN1, class W>
constexpr int FUSE_P = sizeof(W) < sizeof(Tw) ? 0 : CN1 > 0 ? 12 : 9;
// The half spectra's values from Z_k = f and Z_{-k} = s:
// (Z_k + conj Z_{-k})/2 and -i (Z_k - conj Z_{-k})/2
__device__ __forceinline__ float2 split_even(float2 f, float2 s) {
    return make_float2(0.5f * (f.x + s.x), 0.5f * (f.y - s.y));
}
__device__ __forceinline__ float2 split_odd(float2 f, float2 s) {
    return make_float2(0.5f * (f.y + s.y), -0.5f * (f.x - s.x));
}
// The inverse: Z_k and Z_{-k} of Z = A + i B from A_k = a and B_k = b.  A first
// group of at most MERGE_P points does it in registers, for k and N1 - k in
// one thread; otherwise it is a pass of its own.
template <int CN1>
constexpr int MERGE_P = CN1 > 0 ? MERGE_CT : MERGE_RT;
__device__ __forceinline__ float2 merge_pos(float2 a, float2 b) { return make_float2(a.x - b.y, a.y + b.x); }
__device__ __forceinline__ float2 merge_neg(float2 a, float2 b) { return make_float2(a.x + b.y, b.x - a.y); }
// position of (z, kx): even and odd real rows of a complex row at slots se, so
__device__ __forceinline__ int zpos(int z, int S, int se, int so) { return (z >> 1) * S + ((z & 1) ? so : se); }

// Twiddles in shared memory after n float2 values, on a 16-byte boundary.
__host__ __device__ __forceinline__ size_t tw_offset(size_t n) { return (n + 1) & ~(size_t)1; }
template <class W = Tw>
__device__ __forceinline__ W* twiddles_after(float2* base, size_t n) {
    return reinterpret_cast<W*>(base + tw_offset(n));
}

// Forward transform of one plane: complex rows from ld(row, x) (R2C along x
// of the two real rows in each, C2C along z), results to st(kz, kx, value).
// Each phase is one register pass over all lines of the plane; a block-wide
// barrier separates the phases.  The x passes' first group takes neighbouring
// x in neighbouring lanes (the loads), the second neighbouring rows (one
// twiddle for all lanes), the z passes neighbouring kx (the same, and the
// stores).
template <int CN1, int CN3, class W, class LD, class ST>
__device__ __forceinline__ void plane_forward(float2* sm, const GridArgs& g, const Tw* __restrict__ tw, LD ld, ST st) {
    const int N1 = CN1 > 0 ? CN1 : g.N1, N3 = CN3 > 0 ? CN3 : g.N3;
    const int Nh = N1 / 2 + 1, nr = N3 / 2;
    const PlaneGeo G = geo_of<CN1, false>(g);
    const int S = G.S;
    const int P1 = G.run, Q1 = CN3 > 0 ? CtLine<CN3>::G1::P : g.p3.P1;
    W* tw1 = twiddles_after<W>(sm, (size_t)nr * S);
    W* tw3 = tw1 + (N1 - P1);
    load_twiddles(tw1, tw, N1 - P1);
    load_twiddles(tw3, tw + g.N1 + g.N2, N3 - Q1);
    pdl_wait();
    const int t0 = threadIdx.x, nt = blockDim.x;
    on_first<CN1, false>(g.p1, [&](auto tag) {
        using R = decltype(tag);
        constexpr int CM = CN1 > 0 ? CN1 / R::P : 0;
        const int m = CN1 > 0 ? CM : g.p1.P2;
        const SmallDiv dm = small_div(m);
        for (int it = t0; it < nr * m; it += nt) {
            const int row = cdiv<CM>(it, dm), j = it - row * m;
            float2 v[R::P];
#pragma unroll
            for (int q = 0; q < R::P; ++q) v[q] = ld(row, j + q * m);
            group_fft<R, false, true, W>(v, (const W*)nullptr, 1);
            float2* d = sm + row * S + G.at(j);
#pragma unroll
            for (int i = 0; i < R::P; ++i) d[R::digit(i)] = v[i];
        }
    });
    __syncthreads();
    constexpr int CR = CN3 > 0 ? CN3 / 2 : 0;
    const SmallDiv dr = small_div(nr);
    const SmallDiv dP = small_div(G.run);
    on_second<CN1>(g.p1, [&](auto tag) {
        using R = decltype(tag);
        constexpr int P = R::P;
        if constexpr (P <= FUSE_P<CN1, W>) {
            // k1 = ka and P1 - ka: digit d of one is -(digit P - 1 - d of the
            // other); k1 = 0 and P1/2 are their own partners
            for (int it = t0; it < (P1 / 2 + 1) * nr; it += nt) {
                const int ka = cdiv<CR>(it, dr), row = it - ka * nr;
                float2* d = sm + row * S;
                float2* da = d + ka;
                float2 a[P];
#pragma unroll
                for (int q = 0; q < P; ++q) a[q] = da[G.at(q)];
                group_fft<R, false, false, W>(a, tw1 + ka, P1);
                if (ka == 0) {
                    da[0] = split_even(a[0], a[0]);
                    d[G.len] = split_odd(a[0], a[0]);
                    static_for<P / 2>([&](auto Q) {
                        constexpr int q = decltype(Q)::value + 1, m = P - q;
                        const float2 f = a[R::reg(q)], s = a[R::reg(m)];
                        da[G.at(q)] = split_even(f, s);
                        (q == m ? d[G.len + 1] : da[G.at(m)]) = split_odd(f, s);
                    });
                } else if (2 * ka == P1) {
                    static_for<(P + 1) / 2>([&](auto Q) {
                        constexpr int q = decltype(Q)::value, m = P - 1 - q;
                        const float2 f = a[R::reg(q)], s = a[R::reg(m)];
                        da[G.at(q)] = split_even(f, s);
                        (q == m ? d[G.len + 1] : da[G.at(m)]) = split_odd(f, s);
                    });
                } else {
                    const int kb = P1 - ka;
                    float2* db = d + kb;
                    float2 b[P];
#pragma unroll
                    for (int q = 0; q < P; ++q) b[q] = db[G.at(q)];
                    group_fft<R, false, false, W>(b, tw1 + kb, P1);
                    static_for<P>([&](auto Q) {
                        constexpr int q = decltype(Q)::value, m = P - 1 - q;
                        const float2 x = a[R::reg(q)], y = b[R::reg(m)];
                        if constexpr (q <= m) {  // k = ka + P1 q below N1/2
                            da[G.at(q)] = split_even(x, y);
                            db[G.at(m)] = split_odd(x, y);
                        } else {
                            db[G.at(m)] = split_even(y, x);
                            da[G.at(q)] = split_odd(y, x);
                        }
                    });
                }
            }
        } else {
            for (int it = t0; it < P1 * nr; it += nt) {
                const int k1 = cdiv<CR>(it, dr), row = it - k1 * nr;
                float2* d = sm + row * S + k1;
                float2 v[P];
#pragma unroll
                for (int q = 0; q < P; ++q) v[q] = d[G.at(q)];
                group_fft<R, false, false, W>(v, tw1 + k1, P1);
#pragma unroll
                for (int i = 0; i < P; ++i) d[G.at(R::digit(i))] = v[i];
            }
        }
    });
    __syncthreads();
    if (N1 / P1 > FUSE_P<CN1, W>) {
        for (int it = t0; it < Nh * nr; it += nt) {
            const int k = cdiv<CR>(it, dr), row = it - k * nr;
            float2* d = sm + row * S;
            int se, so;
            half_slots(G, dP, N1, k, se, so);
            const float2 zk = d[se], zm = d[k == 0 || 2 * k == N1 ? se : so];
            d[se] = split_even(zk, zm);
            d[so] = split_odd(zk, zm);
        }
        __syncthreads();
    }
    constexpr int CH = CN1 > 0 ? CN1 / 2 + 1 : 0;
    const SmallDiv dh = small_div(Nh);
    on_first<CN3, false>(g.p3, [&](auto tag) {
        using R = decltype(tag);
        const int m = CN3 > 0 ? CN3 / R::P : g.p3.P2;
        for (int it = t0; it < m * Nh; it += nt) {
            const int j = cdiv<CH>(it, dh), kx = it - j * Nh;
            int se, so;
            half_slots(G, dP, N1, kx, se, so);
            float2* d0 = sm + zpos(j, S, se, so);
            float2* d1 = sm + zpos(j + m, S, se, so);
            float2 v[R::P];
#pragma unroll
            for (int q = 0; q < R::P; ++q) v[q] = (q & 1 ? d1 : d0)[(q >> 1) * m * S];
            group_fft<R, false, true, W>(v, (const W*)nullptr, 1);
#pragma unroll
            for (int i = 0; i < R::P; ++i) (R::digit(i) & 1 ? d1 : d0)[(R::digit(i) >> 1) * m * S] = v[i];
        }
    });
    __syncthreads();
    on_second<CN3>(g.p3, [&](auto tag) {
        using R = decltype(tag);
        for (int it = t0; it < Q1 * Nh; it += nt) {
            const int k1 = cdiv<CH>(it, dh), kx = it - k1 * Nh;
            int se, so;
            half_slots(G, dP, N1, kx, se, so);
            const float2* d0 = sm + zpos(k1 * R::P, S, se, so);
            const float2* d1 = sm + zpos(k1 * R::P + 1, S, se, so);
            float2 v[R::P];
#pragma unroll
            for (int q = 0; q < R::P; ++q) v[q] = (q & 1 ? d1 : d0)[(q >> 1) * S];
            group_fft<R, false, false, W>(v, tw3 + k1, Q1);
#pragma unroll
            for (int i = 0; i < R::P; ++i) st(k1 + Q1 * R::digit(i), kx, v[i]);
        }
    });
}

// Inverse transform of one plane (unscaled): half spectrum from ld(kz, kx),
// C2C along z, C2R along x of the two real rows of each complex row (the
// imaginary parts at kx = 0 and N1/2 are dropped, as a complex-to-real
// transform does), st(row, x, {real row 2 row, real row 2 row + 1}).
template <int CN1, int CN3, class W, class LD, class ST>
__device__ __forceinline__ void plane_inverse(float2* sm, const GridArgs& g, const Tw* __restrict__ tw, LD ld, ST st) {
    const int N1 = CN1 > 0 ? CN1 : g.N1, N3 = CN3 > 0 ? CN3 : g.N3;
    const int Nh = N1 / 2 + 1, nr = N3 / 2;
    constexpr bool XI = sizeof(W) < sizeof(Tw);  // (the gradient keeps the forward order)
    const LinePlan& lx = XI ? g.p1i : g.p1;
    const PlaneGeo G = geo_of<CN1, true, XI>(g);
    const int S = G.S;
    const int P1 = CN1 > 0 ? CtLine<CN1, XI>::G1::P : lx.P1, Q1 = CN3 > 0 ? CtLine<CN3>::G1::P : g.p3.P1;
    W* tw1 = twiddles_after<W>(sm, (size_t)nr * S);
    W* tw3 = tw1 + (N1 - P1);
    load_twiddles(tw1, tw + (XI ? tw_off_xi(g) : 0), N1 - P1);
    load_twiddles(tw3, tw + g.N1 + g.N2, N3 - Q1);
    pdl_wait();
    const int t0 = threadIdx.x, nt = blockDim.x;
    constexpr int CH = CN1 > 0 ? CN1 / 2 + 1 : 0;
    const SmallDiv dh = small_div(Nh), dP = small_div(G.run);
    on_first<CN3, false>(g.p3, [&](auto tag) {
        using R = decltype(tag);
        const int m = CN3 > 0 ? CN3 / R::P : g.p3.P2;
        for (int it = t0; it < m * Nh; it += nt) {
            const int j = cdiv<CH>(it, dh), kx = it - j * Nh;
            float2 v[R::P];
#pragma unroll
            for (int q = 0; q < R::P; ++q) v[q] = ld(j + q * m, kx);
            int se, so;
            half_slots(G, dP, N1, kx, se, so);
            float2* d0 = sm + zpos(R::P * j, S, se, so);
            float2* d1 = sm + zpos(R::P * j + 1, S, se, so);
            group_fft<R, true, true, W>(v, (const W*)nullptr, 1);
#pragma unroll
            for (int i = 0; i < R::P; ++i) (R::digit(i) & 1 ? d1 : d0)[(R::digit(i) >> 1) * S] = v[i];
        }
    });
    __syncthreads();
    on_second<CN3>(g.p3, [&](auto tag) {
        using R = decltype(tag);
        for (int it = t0; it < Q1 * Nh; it += nt) {
            const int k1 = cdiv<CH>(it, dh), kx = it - k1 * Nh;
            int se, so;
            half_slots(G, dP, N1, kx, se, so);
            float2* d0 = sm + zpos(k1, S, se, so);
            float2* d1 = sm + zpos(k1 + Q1, S, se, so);
            float2 v[R::P];
#pragma unroll
            for (int q = 0; q < R::P; ++q) v[q] = (q & 1 ? d1 : d0)[(q >> 1) * Q1 * S];
            group_fft<R, true, false, W>(v, tw3 + k1, Q1);
#pragma unroll
            for (int i = 0; i < R::P; ++i) (R::digit(i) & 1 ? d1 : d0)[(R::digit(i) >> 1) * Q1 * S] = v[i];
        }
    });
    __syncthreads();
    constexpr int CR = CN3 > 0 ? CN3 / 2 : 0;
    const SmallDiv dr = small_div(nr);
    const bool merged = XI && P1 <= MERGE_P<CN1>;
    if (!merged) {
        // Z = A + i B on the full circle from the two half spectra
        for (int it = t0; it < Nh * nr; it += nt) {
            const int k = cdiv<CR>(it, dr), row = it - k * nr;
            int se, so;
            half_slots(G, dP, N1, k, se, so);
            float2* d = sm + row * S;
            float2 a = d[se], b = d[so];
            const bool edge = k == 0 || 2 * k == N1;
            if (edge) a.y = b.y = 0.f;
            d[se] = merge_pos(a, b);
            if (!edge) d[so] = merge_neg(a, b);
        }
        __syncthreads();
    }
    on_first<CN1, false, XI>(lx, [&](auto tag) {
        using R = decltype(tag);
        constexpr int P = R::P;
        const int m = CN1 > 0 ? CN1 / P : lx.P2;
        const auto run = [&](float2* d, float2 (&v)[P]) {
            group_fft<R, true, true, W>(v, (const W*)nullptr, 1);
#pragma unroll
            for (int i = 0; i < P; ++i) d[G.at(R::digit(i))] = v[i];
        };
        if constexpr (XI && P <= MERGE_P<CN1>) {
            // j and m - j: element r of one is -(element P - 1 - r of the
            // other); j = 0 and m/2 are their own partners
            for (int it = t0; it < (m / 2 + 1) * nr; it += nt) {
                const int j = cdiv<CR>(it, dr), row = it - j * nr;
                float2* d = sm + row * S;
                float2* da = d + j;
                float2 a[P];
#pragma unroll
                for (int r = 0; r < P; ++r) a[r] = da[G.at(r)];
                if (j == 0) {
                    a[0].y = d[G.len].x;
                    static_for<P / 2>([&](auto Q) {
                        constexpr int r = decltype(Q)::value + 1, s = P - r;
                        if constexpr (r == s) {
                            a[r].y = d[G.len + 1].x;
                        } else {
                            const float2 x = a[r], y = a[s];
                            a[r] = merge_pos(x, y);
                            a[s] = merge_neg(x, y);
                        }
                    });
                    run(da, a);
                } else if (2 * j == m) {
                    static_for<(P + 1) / 2>([&](auto Q) {
                        constexpr int r = decltype(Q)::value, s = P - 1 - r;
                        if constexpr (r == s) {
                            a[r].y = d[G.len + 1].x;
                        } else {
                            const float2 x = a[r], y = a[s];
                            a[r] = merge_pos(x, y);
                            a[s] = merge_neg(x, y);
                        }
                    });
                    run(da, a);
                } else {
                    float2* db = d + (m - j);
                    float2 b[P];
#pragma unroll
                    for (int r = 0; r < P; ++r) b[r] = db[G.at(r)];
                    static_for<P>([&](auto Q) {
                        constexpr int r = decltype(Q)::value, s = P - 1 - r;
                        const float2 x = a[r], y = b[s];
                        if constexpr (r <= s) {  // k = j + r m below N1/2
                            a[r] = merge_pos(x, y);
                            b[s] = merge_neg(x, y);
                        } else {
                            b[s] = merge_pos(y, x);
                            a[r] = merge_neg(y, x);
                        }
                    });
                    run(da, a);
                    run(db, b);
                }
            }
        } else {
            for (int it = t0; it < m * nr; it += nt) {
                const int j = cdiv<CR>(it, dr), row = it - j * nr;
                float2* d = sm + row * S + j;
                float2 v[P];
#pragma unroll
                for (int r = 0; r < P; ++r) v[r] = d[G.at(r)];
                run(d, v);
            }
        }
    });
    __syncthreads();
    const SmallDiv dk = small_div(P1);
    constexpr int CK = CN1 > 0 ? CtLine<CN1, XI>::G1::P : 0;
    on_second<CN1, XI>(lx, [&](auto tag) {
        using R = decltype(tag);
        for (int it = t0; it < P1 * nr; it += nt) {
            const int row = cdiv<CK>(it, dk), k1 = it - row * P1;
            const float2* d = sm + row * S + G.at(k1);
            float2 v[R::P];
#pragma unroll
            for (int q = 0; q < R::P; ++q) v[q] = d[q];
            group_fft<R, true, false, W>(v, tw1 + k1, P1);
#pragma unroll
            for (int i = 0; i < R::P; ++i) st(row, k1 + P1 * R::digit(i), v[i]);
        }
    });
}

// Threads of the plane kernels at most; two such blocks (64 registers per
// thread) or more smaller ones per SM, plane_block (pipeline.cu).
constexpr int PLANE_THREADS = 512;

// f(Dims) with the line kinds of a plan: the compile-time grids, else per
// plane (x and z together) and per y line the run-time kind.
template <int N1_, int N2_, int N3_>
struct Dims {
    static constexpr int N1 = N1_, N2 = N2_, N3 = N3_;
};
template <class F>
auto on_grid(const GridArgs& g, F&& f) {
    if (sized_grid(g.N1, g.N2, g.N3)) return g.N1 == 180 ? f(Dims<180, 180, 72>{}) : f(Dims<256, 256, 96>{});
    const auto small = [](const LinePlan& l) { return l.P1 <= 16 && l.P2 <= 16; };
    if (small(g.p1) && small(g.p3))
        return small(g.p2) ? f(Dims<ANY16, ANY16, ANY16>{}) : f(Dims<ANY16, ANY, ANY16>{});
    return small(g.p2) ? f(Dims<ANY, ANY16, ANY>{}) : f(Dims<ANY, ANY, ANY>{});
}

}  // namespace vdw
