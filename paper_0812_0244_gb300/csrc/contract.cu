// The y stage of the 3D transforms and the per-G contraction of Eqs. (Eoffk),
// (epsofk) in |G| order.
//
// The kernel phi_ab(|G|) depends on G only through |G|, by a cubic spline on
// a uniform k mesh (the radial table, text after Eq. Eoffk).  In the natural
// (kx, ky, kz) order neighbouring points fall in unrelated intervals of that
// table, so the 32 lanes of a warp would fetch 32 different table rows at
// every step of the Nq (Nq + 1) / 2 pair loop.  Here the points of the half
// spectrum are sorted once per plan by |G|: consecutive points then share
// their table interval, a warp's table fetch is one broadcast row, and the
// contraction is a plain stream over the sorted points.
//
//   P2a k_pencil_fwd      C2C along y of 4 fields for C columns; each point's
//                         4 values (32 bytes) go to its sorted position
//   P2b k_contract_sorted per sorted point: u_a = sum_b phi_ab(|G|) theta_b,
//                         the energy of Eq. (Eoffk) in FP64, u / N written back
//   P2c k_pencil_inv      gathers the 4 values of each point of C columns from
//                         the sorted records, inverse C2C along y, back into
//                         the plane layout
//
// Record layout ("quads"): field a = 4 q + i of sorted point r is float2 i of
// the 32-byte record r of quad q: Q[q * qstride + 2 r], Q[... + 2 r + 1]
// (float4 units), qstride = 2 Npad.  Npad is the number of half-spectrum
// points N2 N3 (N1/2 + 1) rounded up to a whole number of contraction blocks;
// the padding records stay zero.  (Writing u in pencil order instead, so that
// the inverse y kernel reads contiguous runs, moves the scattered accesses
// into the contraction's stores and measured no faster.)
#include "plane.cuh"

#include <algorithm>
#include <cmath>
#include <numeric>
#include <vector>

namespace vdw {

constexpr int SORT_THREADS = SORTED_BLOCK;  // points per contraction block
constexpr int PEN_COLS = 8;        // columns per y-pencil block (64-byte runs per plane row)
// Threads of the y-pencil kernels at most.  A block's work is 32 lines of P1
// or P2 butterflies per pass.
constexpr int PEN_THREADS = 256;
// Shared-memory share (%) of the SM's memory under the pencil kernels.  us
// forward / inverse at 44, 58, 72 %: 180 x 180 x 72 99/102, 84/92, 89/102; 256
// x 256 x 96 322/352, 229/274, 242/308; 144 x 144 x 72 53/51, 53/54, 53/61.
constexpr int PEN_CARVEOUT = 58;

// field stride of the lines [4][PEN_COLS][pencil_stride]: lanes that take 4
// fields and 4 neighbouring points (steps of 1 in the forward kernel's
// second pass, of P1 | 1 in the inverse kernel's first) hit distinct banks
__host__ __device__ __forceinline__ int pencil_field_stride(const LinePlan& p, bool inverse) {
    return PEN_COLS * pencil_stride(p) + (inverse ? (4 * (p.P1 | 1)) & 15 : 4);
}
template <int CN2>
__device__ __forceinline__ LinePlan line_of(const GridArgs& g) {
    if constexpr (CN2 > 0) return LinePlan{CN2, CtLine<CN2>::G1::P, CtLine<CN2>::G2::P};
    else return g.p2;
}

// ---------------------------------------------------------------------------
// P2a: forward y transforms of one quad of fields, records in |G| order
// ---------------------------------------------------------------------------
// Block (column tile, quad q): the fields 4q .. 4q+3 of 8 consecutive
// half-spectrum columns, all N2 rows.  First pass: neighbouring lanes take
// neighbouring columns (64-byte runs of the plane rows), straight from global
// memory into the butterflies.  Second pass: neighbouring lanes take the four
// fields, so that four lanes write one point's 32-byte record.
//
// Bound by the latency of its scattered accesses: the share of the SM's memory
// left to L1 decides how many loads are in flight (PEN_CARVEOUT; at 180 x 180
// x 72 the inverse kernel takes 154 us with four blocks' shared memory
// resident and 92 us with two).  us per launch, 20 fields, before (lines
// staged by asynchronous copies, a shared-memory pass per radix) and after,
// forward / inverse: 180 x 180 x 72 117 / 135 -> 84 / 90; 256 x 256 x 96 387 /
// 413 -> 228 / 273; 144 x 144 x 72 (per density) 154 / 154 -> 50 / 54; 200 x
// 200 x 72 279 / 281 -> 144 / 136 (its radix-25 group); 128^3 220 / 216 -> 77 / 80.
template <int CN2>
__global__ void __launch_bounds__(PEN_THREADS, 3) k_pencil_fwd(const float2* __restrict__ spec, GridArgs g,
                                                               const Tw* __restrict__ tw,
                                                               const unsigned* __restrict__ pos,
                                                               float4* __restrict__ Q, long long qstride) {
    extern __shared__ float2 sm[];
    const LinePlan L = line_of<CN2>(g);
    const int N2 = L.n, P1 = L.P1, ps = P1 | 1;
    const int S = pencil_stride(L), LS = pencil_field_stride(L, false);
    Tw* tw2 = twiddles_after(sm, (size_t)4 * LS);
    load_twiddles(tw2, tw, N2 - P1);
    pdl_wait();
    const int c0 = blockIdx.x * PEN_COLS, q = blockIdx.y;
    spec += blockIdx.z * g.bs_spec + (long long)4 * q * N2 * g.ncols;  // density blockIdx.z of a batch
    float2* Qf = reinterpret_cast<float2*>(Q + blockIdx.z * g.bs_Q + q * qstride);
    on_first<CN2, true>(L, [&](auto tag) {
        using R = decltype(tag);
        constexpr int CM = CN2 > 0 ? CN2 / R::P : 0;
        const int m = CN2 > 0 ? CM : L.P2;
        const SmallDiv dm = small_div(m);
        const long long step = (long long)m * g.ncols;
        for (int it = threadIdx.x; it < 4 * PEN_COLS * m; it += blockDim.x) {
            const int cc = it & (PEN_COLS - 1), t = it / PEN_COLS, a = cdiv<CM>(t, dm), j = t - a * m;
            const int col = c0 + cc;
            float2 v[R::P];
            const float2* src = spec + (long long)(a * N2 + j) * g.ncols + col;
#pragma unroll
            for (int i = 0; i < R::P; ++i) v[i] = col < g.ncols ? __ldcg(src + i * step) : make_float2(0.f, 0.f);
            group_fft<R, false, true, Tw>(v, (const Tw*)nullptr, 1);
            float2* d = sm + a * LS + cc * S + ps * j;
#pragma unroll
            for (int i = 0; i < R::P; ++i) d[R::digit(i)] = v[i];
        }
    });
    __syncthreads();
    on_second<CN2>(L, [&](auto tag) {
        using R = decltype(tag);
        constexpr int CP = CN2 > 0 ? CN2 / R::P : 0;
        const SmallDiv dp = small_div(P1);
        for (int it = threadIdx.x; it < 4 * PEN_COLS * P1; it += blockDim.x) {
            const int a = it & 3, t = it >> 2, cc = cdiv<CP>(t, dp), k1 = t - cc * P1;
            const int col = c0 + cc;
            if (col >= g.ncols) continue;
            const unsigned* pp = pos + (long long)col * N2 + k1;
            unsigned r[R::P];
#pragma unroll
            for (int i = 0; i < R::P; ++i) r[i] = __ldg(pp + P1 * R::digit(i));
            const float2* d = sm + a * LS + cc * S + k1;
            float2 v[R::P];
#pragma unroll
            for (int i = 0; i < R::P; ++i) v[i] = d[i * ps];
            group_fft<R, false, false, Tw>(v, tw2 + k1, P1);
#pragma unroll
            for (int i = 0; i < R::P; ++i) Qf[4 * (long long)r[i] + a] = v[i];
        }
    });
}

// ---------------------------------------------------------------------------
// P2c: records in |G| order -> inverse y transforms -> plane layout
// ---------------------------------------------------------------------------
// The forward kernel's mirror image: four lanes read one point's record into
// the first pass, the second pass writes 64-byte runs of the plane rows.
template <int CN2>
__global__ void __launch_bounds__(PEN_THREADS, 3) k_pencil_inv(float2* __restrict__ spec, GridArgs g,
                                                               const Tw* __restrict__ tw,
                                                               const unsigned* __restrict__ pos,
                                                               const float4* __restrict__ Q, long long qstride) {
    extern __shared__ float2 sm[];
    const LinePlan L = line_of<CN2>(g);
    const int N2 = L.n, P1 = L.P1, ps = P1 | 1;
    const int S = pencil_stride(L), LS = pencil_field_stride(L, true);
    float2* tw2 = twiddles_after<float2>(sm, (size_t)4 * LS);
    load_twiddles(tw2, tw, N2 - P1);
    pdl_wait();
    const int c0 = blockIdx.x * PEN_COLS, q = blockIdx.y;
    spec += blockIdx.z * g.bs_spec + (long long)4 * q * N2 * g.ncols;  // density blockIdx.z of a batch
    const float2* Qf = reinterpret_cast<const float2*>(Q + blockIdx.z * g.bs_Q + q * qstride);
    on_first<CN2, true>(L, [&](auto tag) {
        using R = decltype(tag);
        constexpr int CM = CN2 > 0 ? CN2 / R::P : 0;
        const int m = CN2 > 0 ? CM : L.P2;
        const SmallDiv dm = small_div(m);
        for (int it = threadIdx.x; it < 4 * PEN_COLS * m; it += blockDim.x) {
            const int a = it & 3, t = it >> 2, cc = cdiv<CM>(t, dm), j = t - cc * m;
            const int col = c0 + cc;
            float2 v[R::P];
            if (col < g.ncols) {
                const unsigned* pp = pos + (long long)col * N2 + j;
                unsigned r[R::P];
#pragma unroll
                for (int i = 0; i < R::P; ++i) r[i] = __ldg(pp + i * m);
#pragma unroll
                for (int i = 0; i < R::P; ++i) v[i] = __ldcg(Qf + 4 * (long long)r[i] + a);
            } else {
#pragma unroll
                for (int i = 0; i < R::P; ++i) v[i] = make_float2(0.f, 0.f);
            }
            group_fft<R, true, true, float2>(v, (const float2*)nullptr, 1);
            float2* d = sm + a * LS + cc * S + ps * j;
#pragma unroll
            for (int i = 0; i < R::P; ++i) d[R::digit(i)] = v[i];
        }
    });
    __syncthreads();
    on_second<CN2>(L, [&](auto tag) {
        using R = decltype(tag);
        constexpr int CP = CN2 > 0 ? CN2 / R::P : 0;
        const SmallDiv dp = small_div(P1);
        const long long step = (long long)P1 * g.ncols;
        for (int it = threadIdx.x; it < 4 * PEN_COLS * P1; it += blockDim.x) {
            const int cc = it & (PEN_COLS - 1), t = it / PEN_COLS, a = cdiv<CP>(t, dp), k1 = t - a * P1;
            const int col = c0 + cc;
            const float2* d = sm + a * LS + cc * S + k1;
            float2 v[R::P];
#pragma unroll
            for (int i = 0; i < R::P; ++i) v[i] = d[i * ps];
            group_fft<R, true, false, float2>(v, tw2 + k1, P1);
            float2* dst = spec + (long long)(a * N2 + k1) * g.ncols + col;
            if (col < g.ncols) {
#pragma unroll
                for (int i = 0; i < R::P; ++i) dst[R::digit(i) * step] = v[i];
            }
        }
    });
}

// ---------------------------------------------------------------------------
// P2b: the contraction over the sorted points
// ---------------------------------------------------------------------------
// gs[r] = |G| of sorted point r (bohr^-1), negative (or -0) where the point
// counts once in the energy (kx = 0 or kx = N1/2) and positive where it
// stands for itself and its conjugate -G (weight 2); non-decreasing in |G|
// (the padding repeats the last |G|).  kcoef: the radial table as cubic
// coefficients in the local position t, [Nk-1][NQ(NQ+1)/2] float4, pair order
// a <= b row by row.  E partial: sum over the block of
// w_G sum_a Re(conj theta_a u_a), unscaled.
//
// The block's points lie in a contiguous run of table intervals [jlo, jhi]
// (|G| is sorted), whose rows are one contiguous piece of the table.  STAGED:
// they are staged in shared memory, CONTRACT_ROWS at a time, so that the pair
// loop reads them by broadcast instead of waiting on the L2 cache; nearly
// every block of a large grid needs one window.  Otherwise (small grids, whose
// blocks span many intervals) each lane reads its own row from global memory:
// one pass of the pair loop per warp instead of one per window (23 -> 12 us at
// 24^3, 25 -> 14 us at 48^3).
constexpr int CONTRACT_ROWS = 4;  // table rows staged per block at most

// One record (four fields of a point): 32 bytes by one access.  As two 16-byte
// accesses every lane's half sector went through L1 twice (contraction of 8 x
// 144 x 144 x 72 518 us against 498, 256 x 256 x 96 274 against 268).
__device__ __forceinline__ void load_record(const float4* p, float2* v) {
    asm volatile("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(v[0].x), "=f"(v[0].y), "=f"(v[1].x), "=f"(v[1].y), "=f"(v[2].x), "=f"(v[2].y), "=f"(v[3].x),
                   "=f"(v[3].y)
                 : "l"(__cvta_generic_to_global(p))
                 : "memory");
}
__device__ __forceinline__ void store_record(float4* p, const float2* v, float s) {
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(__cvta_generic_to_global(p)),
                 "f"(v[0].x * s), "f"(v[0].y * s), "f"(v[1].x * s), "f"(v[1].y * s), "f"(v[2].x * s), "f"(v[2].y * s),
                 "f"(v[3].x * s), "f"(v[3].y * s)
                 : "memory");
}

// u += Phi(t) theta with the row's pair coefficients cf; the real and the
// imaginary part by one packed instruction (the loop is bound by issue: 112 ->
// 104 us at 180 x 180 x 72, 268 -> 250 at 256 x 256 x 96, the same bits; phi of
// two pairs at a time packed as well took 136)
template <int NQ>
__device__ __forceinline__ void pair_loop(const float4* cf, float t, const float2 (&th)[NQ], float2 (&u)[NQ]) {
    int p = 0;
#pragma unroll
    for (int a = 0; a < NQ; ++a) {
#pragma unroll
        for (int b = a; b < NQ; ++b, ++p) {
            const float4 c = cf[p];
            const float phi = fmaf(t, fmaf(t, fmaf(t, c.w, c.z), c.y), c.x);
            const float2 pp = make_float2(phi, phi);
            u[a] = __ffma2_rn(pp, th[b], u[a]);
            if (b != a) u[b] = __ffma2_rn(pp, th[a], u[b]);
        }
    }
}

template <int NQ, bool STAGED>
__global__ void __launch_bounds__(SORT_THREADS, 4) k_contract_sorted(float4* __restrict__ Q, long long qstride,
                                                                    const float* __restrict__ gs,
                                                                    const float4* __restrict__ kcoef, float inv_dk,
                                                                    int Nk, float invN, double* __restrict__ epart,
                                                                    int write_back, long long bsQ, int bsE) {
    constexpr int NP = NQ * (NQ + 1) / 2;
    __shared__ double red[32];
    __shared__ float4 rows[STAGED ? CONTRACT_ROWS * NP : 1];
    Q += blockIdx.y * bsQ;  // density blockIdx.y of a batch
    epart += blockIdx.y * bsE;
    pdl_wait();
    const long long r0 = (long long)blockIdx.x * SORT_THREADS;
    const long long r = r0 + threadIdx.x;
    float2 th[NQ];
#pragma unroll
    for (int q = 0; q < NQ / 4; ++q) load_record(Q + q * qstride + 2 * r, th + 4 * q);
    const float gm = gs[r];
    const float wgt = signbit(gm) ? 1.f : 2.f;
    const float s = fabsf(gm) * inv_dk;
    const int j = min((int)s, Nk - 2);
    const float t = s - (float)j;
    float2 u[NQ];
#pragma unroll
    for (int a = 0; a < NQ; ++a) u[a] = make_float2(0.f, 0.f);
    if constexpr (STAGED) {
        const int jlo = min((int)(fabsf(gs[r0]) * inv_dk), Nk - 2);
        const int jhi = min((int)(fabsf(gs[r0 + SORT_THREADS - 1]) * inv_dk), Nk - 2);
        for (int w = jlo; w <= jhi; w += CONTRACT_ROWS) {
            const int nr = min(CONTRACT_ROWS, jhi - w + 1);
            if (w != jlo) __syncthreads();  // the previous window's rows are read
            const float4* src = kcoef + (long long)w * NP;
            for (int i = threadIdx.x; i < nr * NP; i += SORT_THREADS) rows[i] = __ldg(src + i);
            __syncthreads();
            if (j >= w && j < w + nr) pair_loop<NQ>(rows + (j - w) * NP, t, th, u);
        }
    } else {
        pair_loop<NQ>(kcoef + (long long)j * NP, t, th, u);
    }
    float e = 0.f;
#pragma unroll
    for (int a = 0; a < NQ; ++a) e = fmaf(th[a].x, u[a].x, fmaf(th[a].y, u[a].y, e));
    const double es = block_sum((double)(wgt * e), red);
    if (threadIdx.x == 0) epart[blockIdx.x] = es;
    if (!write_back) return;
#pragma unroll
    for (int q = 0; q < NQ / 4; ++q) store_record(Q + q * qstride + 2 * r, u + 4 * q, invN);
}

// The same with two points per thread, r and r + 64 of the block's 128, in
// packed FP32 pairs: one instruction for both points' products, and one read
// of a row for both.  Blocks of a large grid nearly always hold one or two
// intervals; a thread whose points differ in theirs takes them one by one.
// The staged rows hold each coefficient twice ({w, w, z, z}, {y, y, x, x}).
// Eight fields at 180 x 180 x 72: 48.6 -> 42.5 us.  With 20 fields the two
// points' values take 255 registers, two warps per scheduler, and 178 us
// against 114: there the kernel above stays.
constexpr int PAIR_THREADS = SORTED_BLOCK / 2;

template <int NQ>
__device__ __forceinline__ void pair_loop2(const float4* cf, float2 t, const float2 (&thx)[NQ],
                                           const float2 (&thy)[NQ], float2 (&ux)[NQ], float2 (&uy)[NQ]) {
    int p = 0;
#pragma unroll
    for (int a = 0; a < NQ; ++a) {
#pragma unroll
        for (int b = a; b < NQ; ++b, ++p) {
            const float4 hi = cf[2 * p], lo = cf[2 * p + 1];
            float2 phi = __ffma2_rn(t, make_float2(hi.x, hi.y), make_float2(hi.z, hi.w));
            phi = __ffma2_rn(t, phi, make_float2(lo.x, lo.y));
            phi = __ffma2_rn(t, phi, make_float2(lo.z, lo.w));
            ux[a] = __ffma2_rn(phi, thx[b], ux[a]);
            uy[a] = __ffma2_rn(phi, thy[b], uy[a]);
            if (b != a) {
                ux[b] = __ffma2_rn(phi, thx[a], ux[b]);
                uy[b] = __ffma2_rn(phi, thy[a], uy[b]);
            }
        }
    }
}
// one of the two points (S = 0, 1) from the table itself
template <int NQ, int S>
__device__ __forceinline__ void pair_loop1(const float4* __restrict__ cf, float t, const float2 (&thx)[NQ],
                                           const float2 (&thy)[NQ], float2 (&ux)[NQ], float2 (&uy)[NQ]) {
    const auto at = [](const float2& v) { return S ? v.y : v.x; };
    const auto add = [&](float2& v, float phi, float x) {
        if (S) v.y = fmaf(phi, x, v.y);
        else v.x = fmaf(phi, x, v.x);
    };
    int p = 0;
#pragma unroll
    for (int a = 0; a < NQ; ++a) {
#pragma unroll
        for (int b = a; b < NQ; ++b, ++p) {
            const float4 c = __ldg(cf + p);
            const float phi = fmaf(t, fmaf(t, fmaf(t, c.w, c.z), c.y), c.x);
            add(ux[a], phi, at(thx[b]));
            add(uy[a], phi, at(thy[b]));
            if (b != a) {
                add(ux[b], phi, at(thx[a]));
                add(uy[b], phi, at(thy[a]));
            }
        }
    }
}

template <int NQ>
__global__ void __launch_bounds__(PAIR_THREADS, 6) k_contract_pairs(
    float4* __restrict__ Q, long long qstride, const float* __restrict__ gs, const float4* __restrict__ kcoef,
    float inv_dk, int Nk, float invN, double* __restrict__ epart, int write_back, long long bsQ, int bsE) {
    constexpr int NP = NQ * (NQ + 1) / 2;
    __shared__ double red[32];
    __shared__ float4 rows[CONTRACT_ROWS * NP * 2];
    Q += blockIdx.y * bsQ;  // density blockIdx.y of a batch
    epart += blockIdx.y * bsE;
    pdl_wait();
    const long long r0 = (long long)blockIdx.x * SORT_THREADS;
    const long long r = r0 + threadIdx.x, r1 = r + PAIR_THREADS;
    float2 thx[NQ], thy[NQ], ux[NQ], uy[NQ];
#pragma unroll
    for (int q = 0; q < NQ / 4; ++q) {
        const float4* b = Q + q * qstride;
        const float4 a0 = b[2 * r], a1 = b[2 * r + 1], b0 = b[2 * r1], b1 = b[2 * r1 + 1];
        thx[4 * q] = make_float2(a0.x, b0.x);
        thy[4 * q] = make_float2(a0.y, b0.y);
        thx[4 * q + 1] = make_float2(a0.z, b0.z);
        thy[4 * q + 1] = make_float2(a0.w, b0.w);
        thx[4 * q + 2] = make_float2(a1.x, b1.x);
        thy[4 * q + 2] = make_float2(a1.y, b1.y);
        thx[4 * q + 3] = make_float2(a1.z, b1.z);
        thy[4 * q + 3] = make_float2(a1.w, b1.w);
    }
    const float g0 = gs[r], g1 = gs[r1];
    const float s0 = fabsf(g0) * inv_dk, s1 = fabsf(g1) * inv_dk;
    const int j0 = min((int)s0, Nk - 2), j1 = min((int)s1, Nk - 2);
    const float2 t = make_float2(s0 - (float)j0, s1 - (float)j1);
#pragma unroll
    for (int a = 0; a < NQ; ++a) ux[a] = uy[a] = make_float2(0.f, 0.f);
    const int jlo = min((int)(fabsf(gs[r0]) * inv_dk), Nk - 2);
    const int jhi = min((int)(fabsf(gs[r0 + SORT_THREADS - 1]) * inv_dk), Nk - 2);
    const int nr = min(jhi - jlo + 1, CONTRACT_ROWS);
    const float4* src = kcoef + (long long)jlo * NP;
    for (int i = threadIdx.x; i < nr * NP; i += PAIR_THREADS) {
        const float4 c = __ldg(src + i);
        rows[2 * i] = make_float4(c.w, c.w, c.z, c.z);
        rows[2 * i + 1] = make_float4(c.y, c.y, c.x, c.x);
    }
    __syncthreads();
    if (j0 == j1 && j0 - jlo < nr) {
        pair_loop2<NQ>(rows + (j0 - jlo) * NP * 2, t, thx, thy, ux, uy);
    } else {
        pair_loop1<NQ, 0>(kcoef + (long long)j0 * NP, t.x, thx, thy, ux, uy);
        pair_loop1<NQ, 1>(kcoef + (long long)j1 * NP, t.y, thx, thy, ux, uy);
    }
    float2 e = make_float2(0.f, 0.f);
#pragma unroll
    for (int a = 0; a < NQ; ++a) e = __ffma2_rn(thx[a], ux[a], __ffma2_rn(thy[a], uy[a], e));
    const double es = block_sum((double)((signbit(g0) ? 1.f : 2.f) * e.x) + (double)((signbit(g1) ? 1.f : 2.f) * e.y), red);
    if (threadIdx.x == 0) epart[blockIdx.x] = es;
    if (!write_back) return;
#pragma unroll
    for (int q = 0; q < NQ / 4; ++q) {
        float4* b = Q + q * qstride;
        const int a = 4 * q;
        b[2 * r] = make_float4(ux[a].x * invN, uy[a].x * invN, ux[a + 1].x * invN, uy[a + 1].x * invN);
        b[2 * r + 1] = make_float4(ux[a + 2].x * invN, uy[a + 2].x * invN, ux[a + 3].x * invN, uy[a + 3].x * invN);
        b[2 * r1] = make_float4(ux[a].y * invN, uy[a].y * invN, ux[a + 1].y * invN, uy[a + 1].y * invN);
        b[2 * r1 + 1] = make_float4(ux[a + 2].y * invN, uy[a + 2].y * invN, ux[a + 3].y * invN, uy[a + 3].y * invN);
    }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
size_t sorted_pencil_smem(const GridArgs& g) {
    const size_t n = 4 * (size_t)std::max(pencil_field_stride(g.p2, false), pencil_field_stride(g.p2, true));
    return sizeof(float2) * tw_offset(n) + sizeof(Tw) * (size_t)(g.p2.n - g.p2.P1);
}
// |G| order of the half spectrum: pos[col N2 + y] = sorted position of the
// point (kx, y, kz), col = kz Nh + kx; gs[sorted position] = |G| with the
// energy weight in its sign.  Ties (equal |G|) keep the (col, y) order, so
// the permutation is deterministic.
int sorted_plan(vdw_ctx* c) {
    const GridArgs& g = c->g;
    const long long nG = (long long)g.ncols * g.N2;
    const long long Npad = (nG + SORT_THREADS - 1) / SORT_THREADS * SORT_THREADS;
    const double PI_D = 3.14159265358979323846;
    const double b1 = 2.0 * PI_D / c->L[0], b2 = 2.0 * PI_D / c->L[1], b3 = 2.0 * PI_D / c->L[2];
    std::vector<double> key((size_t)nG);
    for (int col = 0; col < g.ncols; ++col) {
        const int kx = col % g.Nh, kz = col / g.Nh;
        const int mz = (2 * kz <= g.N3) ? kz : kz - g.N3;
        const double ax = b1 * kx, az = b3 * mz;
        for (int y = 0; y < g.N2; ++y) {
            const int my = (2 * y <= g.N2) ? y : y - g.N2;
            const double ay = b2 * my;
            key[(size_t)col * g.N2 + y] = ax * ax + ay * ay + az * az;
        }
    }
    std::vector<unsigned> idx((size_t)nG);
    std::iota(idx.begin(), idx.end(), 0u);
    std::stable_sort(idx.begin(), idx.end(), [&](unsigned a, unsigned b) { return key[a] < key[b]; });
    std::vector<unsigned> pos((size_t)nG);
    std::vector<float> gs((size_t)Npad, 0.f);
    for (long long s = 0; s < nG; ++s) {
        const unsigned i = idx[(size_t)s];
        pos[i] = (unsigned)s;
        const int col = (int)(i / g.N2), kx = col % g.Nh;
        const bool single = (kx == 0) || (2 * kx == g.N1);
        const float m = (float)std::sqrt(key[i]);
        gs[(size_t)s] = single ? -m : m;
    }
    // padding records (theta = 0): the last |G| again, so that |gs| stays sorted
    for (long long s = nG; s < Npad; ++s) gs[(size_t)s] = std::fabs(gs[(size_t)(nG - 1)]);
    c->nG = nG;
    c->Npad = Npad;
    c->nb_sorted = (int)(Npad / SORT_THREADS);
    VDW_CUDA(cudaMalloc(&c->d_pos, sizeof(unsigned) * (size_t)nG));
    VDW_CUDA(cudaMalloc(&c->d_gs, sizeof(float) * (size_t)Npad));
    VDW_CUDA(cudaMemcpy(c->d_pos, pos.data(), sizeof(unsigned) * (size_t)nG, cudaMemcpyHostToDevice));
    VDW_CUDA(cudaMemcpy(c->d_gs, gs.data(), sizeof(float) * (size_t)Npad, cudaMemcpyHostToDevice));
    c->bytes += sizeof(unsigned) * (size_t)nG + sizeof(float) * (size_t)Npad;
    return VDW_OK;
}

void sorted_free(vdw_ctx* c) {
    cudaFree(c->d_pos);
    cudaFree(c->d_gs);
    c->d_pos = nullptr;
    c->d_gs = nullptr;
}

template <int CN2>
static int configure_sorted_sized(vdw_ctx* c) {
    int rc = raise_smem_limit(k_pencil_fwd<CN2>, (int)sorted_pencil_smem(c->g));
    if (!rc) rc = raise_smem_limit(k_pencil_inv<CN2>, (int)sorted_pencil_smem(c->g));
    if (rc) return rc;
    // The scattered 32-byte records reserve a 128-byte L1 line each while they
    // are in flight: with all of the SM's memory given to shared memory, what
    // is left for L1 bounds the loads in flight.
    VDW_CUDA(cudaFuncSetAttribute(k_pencil_fwd<CN2>, cudaFuncAttributePreferredSharedMemoryCarveout, PEN_CARVEOUT));
    VDW_CUDA(cudaFuncSetAttribute(k_pencil_inv<CN2>, cudaFuncAttributePreferredSharedMemoryCarveout, PEN_CARVEOUT));
    int dev = 0;
    VDW_CUDA(cudaGetDevice(&dev));
    VDW_CUDA(cudaDeviceGetAttribute(&c->nsm, cudaDevAttrMultiProcessorCount, dev));
    return VDW_OK;
}

int sorted_configure(vdw_ctx* c) {
    return on_grid(c->g, [&](auto d) { return configure_sorted_sized<decltype(d)::N2>(c); });
}

int sorted_forward(vdw_ctx* c, int nfields, cudaStream_t s, int B) {
    const GridArgs& g = c->g;
    const dim3 grid((g.ncols + PEN_COLS - 1) / PEN_COLS, nfields / 4, B);
    on_grid(g, [&](auto d) {
        launch(early_launch(g, B), k_pencil_fwd<decltype(d)::N2>, grid, PEN_THREADS, sorted_pencil_smem(g), s, c->d_spec, g, c->d_tw + tw_off_y(g), c->d_pos, c->d_Q, 2 * c->Npad);
    });
    VDW_CUDA(cudaGetLastError());
    return VDW_OK;
}

int sorted_inverse(vdw_ctx* c, int nfields, cudaStream_t s, int B) {
    const GridArgs& g = c->g;
    const dim3 grid((g.ncols + PEN_COLS - 1) / PEN_COLS, nfields / 4, B);
    on_grid(g, [&](auto d) {
        launch(early_launch(g, B), k_pencil_inv<decltype(d)::N2>, grid, PEN_THREADS, sorted_pencil_smem(g), s, c->d_spec, g, c->d_tw + tw_off_y(g), c->d_pos, c->d_Q, 2 * c->Npad);
    });
    VDW_CUDA(cudaGetLastError());
    return VDW_OK;
}

int sorted_contract(vdw_ctx* c, double* epart, int write_back, cudaStream_t s, int B) {
    return sorted_contract_table(c, c->p.Nq, c->d_kcoef, c->g.inv_dk, c->g.Nk, epart, write_back, s, B);
}

int sorted_contract_table(vdw_ctx* c, int nq, const float4* table, float inv_dk, int nk, double* epart,
                          int write_back, cudaStream_t s, int B) {
    const GridArgs& g = c->g;
    const long long qs = 2 * c->Npad;
    // large grids: a block's points share one or two intervals (at least twice
    // as many blocks as the intervals they span)
    const double gmax = M_PI * std::sqrt(std::pow(g.N1 / c->L[0], 2) + std::pow(g.N2 / c->L[1], 2) +
                                         std::pow(g.N3 / c->L[2], 2));
    const bool staged = c->nb_sorted >= 2.0 * gmax * inv_dk;
#define VDW_CONTRACT_K(KERNEL, THREADS)                                                                  \
    launch(early_launch(g, B), KERNEL, dim3(c->nb_sorted, B), THREADS, 0, s, c->d_Q, qs, c->d_gs, table, inv_dk, nk, g.invN, epart, \
           write_back, g.bs_Q, g.bs_epart)
#define VDW_CONTRACT(NQ)                                                                                 \
    if (staged) VDW_CONTRACT_K((k_contract_sorted<NQ, true>), SORT_THREADS);                             \
    else VDW_CONTRACT_K((k_contract_sorted<NQ, false>), SORT_THREADS)
    switch (nq) {
        case 20: VDW_CONTRACT(20); break;
        case 8:
            // two points per thread, where the blocks fill the SMs at half the threads
            if (staged && (long long)c->nb_sorted * B >= 8LL * c->nsm)
                VDW_CONTRACT_K(k_contract_pairs<8>, PAIR_THREADS);
            else
                VDW_CONTRACT(8);
            break;
        case 12: VDW_CONTRACT(12); break;
        case 16: VDW_CONTRACT(16); break;
        default: set_error("Nq not compiled in"); return VDW_ERR_UNSUPPORTED;
    }
#undef VDW_CONTRACT
#undef VDW_CONTRACT_K
    VDW_CUDA(cudaGetLastError());
    return VDW_OK;
}

}  // namespace vdw
