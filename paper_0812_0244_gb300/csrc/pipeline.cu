// The hot path of the Roman-Perez--Soler evaluation on one GB300.
//
//   P0 k_pointwise      n, grad n -> q, mesh interval k, position t (Eq. Sat,
//                       Eq. fofx), theta_a = n p_a(q) (text after Eq. Eoffk)
//                       into packed real planes; Delta E partial sums
//                       (Eqs. DEnl, Depsnl)
//   P1 (planes.cu)      forward plane transforms of theta_a in place: R2C
//                       along x and C2C along z through shared memory
//   P2 (contract.cu)    C2C along y of all Nq fields, points written in |G|
//                       order; per G: u_a(G) = sum_b phi_ab(|G|) theta_b(G)
//                       with phi_ab from the radial table, energy of Eq.
//                       (Eoffk) in FP64; inverse C2C along y (Eqs. epsilon,
//                       epsofk)
//   P3 (planes.cu)      inverse plane transform of u_a (in place)
//      k_u_sum          Eq. (Vi) per point: v_loc and g of w = g grad n
//      k_w_planes       forward plane transform of w
//   P4 k_pencil_div     y transform of w, i G' . w(G), inverse y transform
//   P5 k_div_final      inverse plane transform, v = v_loc - D . w
//
// Layouts: real fields [N3][N2][N1] flat (x fastest); spectra
// [field][N2][N3][Nh] with Nh = N1/2+1 (a y plane of the half spectrum is one
// contiguous block, a pencil along y strides by N3 Nh).
//
// The transform kernels are templates over the line lengths (CN1, CN2, CN3):
// the grids 180 x 180 x 72 and 256 x 256 x 96 get compile-time lengths, any
// other size one of the two run-time kinds of fft.cuh.
#include "plane.cuh"
#include "pointwise.cuh"

#include <algorithm>
#include <initializer_list>
#include <string>
#include <vector>

namespace vdw {

constexpr int XC_BLOCKS = 1024;  // blocks (and partial-sum slots) of the semilocal kernel

// ---------------------------------------------------------------------------
// P0: pointwise
// ---------------------------------------------------------------------------
// q, its mesh interval k and position t per point (flat order out), theta_a
// = n p_a(q) (text after Eq. Eoffk) into the packed real rows of the
// spectrum buffer, and the Delta E partial sums.  aux (flat order) keeps
// what the assembly of Eq. (Vi) needs besides the field sums:
// {n dq/dn, n (dq/d|grad n|)/|grad n|, d(Delta eps)/dn, its grad n coefficient}.
// The grid is cut into slabs of nj complex rows (z = 2 j0 .. 2 (j0 + nj) - 1
// for slab j0 / nj), each walked in packed order within the slab: q = ((y nj
// + (j - j0)) N1 + x) 2 + s, by nbs blocks of which block b writes its
// Delta E partial sum to epart[slab nbs + b].  A launch with slab >= 0 does
// that slab alone (grid nbs); with slab < 0 the grid holds nbs blocks for
// every slab, block b doing block b mod nbs of slab b / nbs, so that both
// forms give the same partial sums.  mnj = ceil(2^32 / nj) when g.fast.
// Bound by issue slots (64 % of the cycles), not by HBM (a third of its
// bandwidth).  Four blocks of 256 threads per SM at 62 registers, the two z of
// a packed row to a thread (8-byte stores), the interval counted: 80 us at 180
// x 180 x 72.  One point per thread took 100 us at 40 registers and six blocks,
// 112 at 64 registers and four.
template <int NQ>
__global__ void __launch_bounds__(256, POINT_BLOCKS) k_pointwise(const float* __restrict__ n, const float* __restrict__ grad,
                                                   GridArgs g, PointParams P, int slab, int nj, unsigned mnj,
                                                   int nbs, float* __restrict__ t_out, uint8_t* __restrict__ k_out,
                                                   float4* __restrict__ aux, float2* __restrict__ spec,
                                                   double* __restrict__ epart,
                                                   unsigned* __restrict__ badp) {
    __shared__ double red[32];
    __shared__ SplineMesh sp;
    __shared__ float2 mp[NQ * MP_LD];
    {
        // density blockIdx.y of a batch
        const long long b = blockIdx.y;
        n += b * g.N;
        grad += 3 * b * g.N;
        t_out += b * g.N;
        k_out += b * g.N;
        aux += b * g.N;
        spec += b * g.bs_spec;
        epart += b * g.bs_epart;
    }
    load_spline_mesh(&sp, P);
    load_spline_pairs<NQ>(mp, P);
    pdl_wait();
    __syncthreads();
    const int sl = slab >= 0 ? slab : (int)blockIdx.x / nbs;
    const int lb = slab >= 0 ? (int)blockIdx.x : (int)blockIdx.x - sl * nbs;
    const int j0 = sl * nj;
    const long long N = g.N, zs = (long long)g.N1 * g.N2;
    const long long Nc = (long long)g.N2 * nj * g.N1;     // pairs of points of the slab
    const long long fstride = (long long)g.N2 * g.ncols;  // values between the planes of two fields
    double acc = 0.0;
    unsigned int bad = 0;
    for (long long q = lb * (long long)blockDim.x + threadIdx.x; q < Nc; q += (long long)nbs * blockDim.x) {
        int y, x, jj;
        if (g.fast) {
            const unsigned rr = __umulhi((unsigned)q, g.m1);
            x = (int)((unsigned)q - rr * (unsigned)g.N1);
            y = nj == 1 ? (int)rr : (int)__umulhi(rr, mnj);
            jj = (int)(rr - (unsigned)y * (unsigned)nj);
        } else {
            const long long rr = q / g.N1;
            x = (int)(q - rr * g.N1);
            y = (int)(rr / nj);
            jj = (int)(rr - (long long)y * nj);
        }
        const int j = j0 + jj;
        const long long i0 = (2LL * j * g.N2 + y) * g.N1 + x;
        // per point: the spline's coefficients at its interval
        float nn[2], A[2], B[2], cA[2], cB[2], h26[2];
        int kk[2];
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const long long i = i0 + s * zs;
            const float ni = n[i];
            bad += (!(ni >= 0.f) || !isfinite(ni)) ? 1u : 0u;
            const QPoint qp = q_point<NQ>(ni, grad[i], grad[N + i], grad[2 * N + i], P, sp.qm);
            t_out[i] = qp.t;
            k_out[i] = (uint8_t)qp.k;
            const bool ok = qp.k != K_INVALID;
            float4 ax = make_float4(0.f, 0.f, 0.f, 0.f);
            if (ok) {
                const float qv = qp.q, q3 = qv * qv * qv, q4 = q3 * qv;
                acc += (double)(0.5f * P.C_s * ni * ni / q3);
                const float cn = 1.5f * P.C_s * ni * ni / q4;
                ax = make_float4(ni * qp.dq_dn, ni * qp.dq_dg, P.C_s * ni / q3 - cn * qp.dq_dn, -cn * qp.dq_dg);
            }
            aux[i] = ax;
            nn[s] = ok ? ni : 0.f;
            kk[s] = ok ? qp.k : 0;
            A[s] = 1.f - qp.t;
            B[s] = qp.t;
            cA[s] = A[s] * A[s] * A[s] - A[s];
            cB[s] = B[s] * B[s] * B[s] - B[s];
            h26[s] = sp.h26[kk[s]];
        }
        float2* dst = spec + ((long long)y * g.ncols + (2 * j * g.Nh + x));
        const float2* m0 = mp + kk[0];
        const float2* m1 = mp + kk[1];
#pragma unroll
        for (int a = 0; a < NQ; ++a) {
            // p_a = (A at a = k, B at a = k + 1) + (cA M_ak + cB M_a,k+1) h^2/6
            const float2 u = m0[a * MP_LD], w = m1[a * MP_LD];
            const float y0 = a == kk[0] ? A[0] : (a == kk[0] + 1 ? B[0] : 0.f);
            const float y1 = a == kk[1] ? A[1] : (a == kk[1] + 1 ? B[1] : 0.f);
            const float p0 = fmaf(fmaf(cA[0], u.x, cB[0] * u.y), h26[0], y0);
            const float p1 = fmaf(fmaf(cA[1], w.x, cB[1] * w.y), h26[1], y1);
            dst[a * fstride] = make_float2(nn[0] * p0, nn[1] * p1);
        }
    }
    const double s = block_sum(acc, red);
    if (threadIdx.x == 0) epart[sl * nbs + lb] = s;
    __syncthreads();
    const double b = block_sum((double)bad, red);
    if (threadIdx.x == 0) {
        const int nb = (int)(slab >= 0 ? gridDim.x * (g.N3 / 2 / nj) : gridDim.x);  // blocks of a density
        badp[1 + blockIdx.y * nb + sl * nbs + lb] = (unsigned)b;
        if (blockIdx.x == 0 && blockIdx.y == 0) badp[0] = nb * gridDim.y;
    }
}

// P1 (the forward plane transforms of theta_a) is in planes.cu; P2 (y
// transforms and the contraction) in contract.cu.

// ---------------------------------------------------------------------------
// P3': the assembly of Eq. (Vi)
// ---------------------------------------------------------------------------
// S0 = sum_a u_a p_a(q), S1 = sum_a u_a p_a'(q) from the packed real u_a planes
// left in the spectrum buffer by the inverse k_planes_inplace.  On interval k with
// A = 1 - t, B = t, p_a = A d_ak + B d_a,k+1 + [(A^3 - A) M_ak + (B^3 - B)
// M_a,k+1] h^2/6 is linear in the second derivatives M, so both sums need
// only u_k, u_k+1 and the two dot products m0 = sum_a u_a M_ak, m1 = sum_a
// u_a M_a,k+1.  Then, with aux from the pointwise pass,
//   v_loc = S0 + S1 n dq/dn + d(Delta eps)/dn,   g = S1 n dq/d|grad n| / |grad n| + ...
// mode 0: v_loc to v (if v), w = g grad n to w_out (if w_out), both times
// gE[0] dOmega if gE; mode 1: v_loc to v, g to
// g_out (the plane transforms of w follow in k_w_planes).
constexpr int USUM_THREADS = 256;

// One thread takes the two points z = 2 j, 2 j + 1 of a packed row, so that a
// field's two values come by one 8-byte load.
template <int NQ>
__global__ void __launch_bounds__(USUM_THREADS, 4) k_u_sum(const float2* __restrict__ uf, const float* __restrict__ grad,
                                                        const float* __restrict__ tk, const uint8_t* __restrict__ kk,
                                                        const float4* __restrict__ aux, GridArgs g, PointParams P,
                                                        float* __restrict__ v, float* __restrict__ w_out,
                                                        float* __restrict__ g_out, int mode,
                                                        const double* __restrict__ gE, double dOmega) {
    __shared__ SplineMesh sp;
    __shared__ float2 mp[NQ * MP_LD];
    {
        // density blockIdx.y of a batch
        const long long b = blockIdx.y;
        uf += b * g.bs_spec;
        grad += 3 * b * g.N;
        tk += b * g.N;
        kk += b * g.N;
        aux += b * g.N;
        if (v) v += b * g.N;
        if (w_out) w_out += 3 * b * g.N;
        if (g_out) g_out += b * g.N;
    }
    load_spline_mesh(&sp, P);
    load_spline_pairs<NQ>(mp, P);
    pdl_wait();
    __syncthreads();
    const float scale = gE ? (float)(gE[0] * dOmega) : 1.f;
    const long long N = g.N;
    const long long fstride = (long long)g.N2 * g.ncols;  // values between the planes of two fields
    const long long zs = (long long)g.N1 * g.N2;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N / 2; i += (long long)gridDim.x * blockDim.x) {
        int x, y, j;
        flat_point(i, g, x, y, j);  // (x, y) of the plane z = 2 j
        const float2* up = uf + (long long)y * g.ncols + (2 * j * g.Nh + x);
        const long long i0 = i + j * zs;
        const int k0 = kk[i0], k1 = kk[i0 + zs];
        const int c0 = k0 == K_INVALID ? 0 : k0, c1 = k1 == K_INVALID ? 0 : k1;
        float2 uk = make_float2(0.f, 0.f), uk1 = uk, m0 = uk, m1 = uk;
#pragma unroll
        for (int a = 0; a < NQ; ++a) {
            const float2 u = up[a * fstride];
            const float2 M0 = mp[a * MP_LD + c0], M1 = mp[a * MP_LD + c1];
            m0.x = fmaf(u.x, M0.x, m0.x);
            m1.x = fmaf(u.x, M0.y, m1.x);
            m0.y = fmaf(u.y, M1.x, m0.y);
            m1.y = fmaf(u.y, M1.y, m1.y);
            uk.x = (a == c0) ? u.x : uk.x;
            uk1.x = (a == c0 + 1) ? u.x : uk1.x;
            uk.y = (a == c1) ? u.y : uk.y;
            uk1.y = (a == c1 + 1) ? u.y : uk1.y;
        }
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const long long ii = i0 + s * zs;
            const int k = s ? c1 : c0;
            const float t = tk[ii];
            const float4 ax = aux[ii];
            const float a0 = s ? uk.y : uk.x, a1 = s ? uk1.y : uk1.x, b0 = s ? m0.y : m0.x, b1 = s ? m1.y : m1.x;
            const float A = 1.f - t, B = t;
            const float s0 = A * a0 + B * a1 + ((A * A * A - A) * b0 + (B * B * B - B) * b1) * sp.h26[k];
            const float s1 = (a1 - a0) * sp.ih[k] + ((3.f * B * B - 1.f) * b1 - (3.f * A * A - 1.f) * b0) * sp.h6[k];
            const bool ok = (s ? k1 : k0) != K_INVALID;
            const float vl = ok ? s0 + ax.x * s1 + ax.z : 0.f, gg = ok ? ax.y * s1 + ax.w : 0.f;
            if (v) v[ii] = vl * scale;
            if (mode == 0 && w_out) {
                w_out[ii] = gg * grad[ii] * scale;
                w_out[N + ii] = gg * grad[N + ii] * scale;
                w_out[2 * N + ii] = gg * grad[2 * N + ii] * scale;
            }
            if (mode == 1) g_out[ii] = gg;
        }
    }
}

// ---------------------------------------------------------------------------
// P3b: forward plane transforms of the three components of w = g grad n
// ---------------------------------------------------------------------------
template <int CN1, int CN3>
__global__ void __launch_bounds__(PLANE_THREADS, 2)
    k_w_planes(const float* __restrict__ gfield, const float* __restrict__ grad, GridArgs g, const Tw* __restrict__ tw,
               float2* __restrict__ wspec) {
    extern __shared__ float2 sm[];
    const int N1 = CN1 > 0 ? CN1 : g.N1, Nh = N1 / 2 + 1;
    const int y = blockIdx.x, c = blockIdx.y;
    const int zs = N1 * g.N2;  // flat distance between rows z and z + 1
    // density blockIdx.z of a batch
    const float* gf = gfield + blockIdx.z * g.N + (long long)N1 * y;
    const float* gc = grad + (3 * blockIdx.z + c) * g.N + (long long)N1 * y;
    float2* dst = wspec + blockIdx.z * g.bs_wspec + ((long long)c * g.N2 + y) * g.ncols;
    plane_forward<CN1, CN3, float2>(
        sm, g, tw,
        [&](int row, int x) {
            const long long i = 2LL * row * zs + x;
            return make_float2(gf[i] * gc[i], gf[i + zs] * gc[i + zs]);
        },
        [&](int kz, int kx, float2 w) { dst[kz * Nh + kx] = w; });
}

// ---------------------------------------------------------------------------
// P4: spectral divergence along pencils
// ---------------------------------------------------------------------------
// Block: the three components of 8 columns.  The forward transform's second
// group, d = i G' . w / N and the inverse transform's first group (the same
// radices: the inverse takes the two groups in the other order) stay in one
// thread's registers.  180 x 180 x 72: 26 -> 18 us; 100^3: 29 -> 25 us.
constexpr int DIV_COLS = 8;
constexpr int DIV_THREADS = 128;

template <int CN2>
__global__ void __launch_bounds__(DIV_THREADS) k_pencil_div(float2* __restrict__ wspec, GridArgs g,
                                                            const Tw* __restrict__ tw, const Tw* __restrict__ tw_swap) {
    extern __shared__ float2 sm[];
    constexpr int C = DIV_COLS;
    LinePlan L = g.p2;
    if constexpr (CN2 > 0) L = LinePlan{CN2, CtLine<CN2>::G1::P, CtLine<CN2>::G2::P};
    const int N2 = L.n, P1 = L.P1, P2 = L.P2, ps = P1 | 1;
    const int S = pencil_stride(L);
    float2* tw2 = twiddles_after<float2>(sm, (size_t)3 * C * S);
    float2* tw2s = tw2 + (N2 - P1);
    load_twiddles(tw2, tw, N2 - P1);
    load_twiddles(tw2s, tw_swap, N2 - P2);
    pdl_wait();
    wspec += blockIdx.y * g.bs_wspec;  // density blockIdx.y of a batch
    const int c0 = blockIdx.x * C;
    on_first<CN2, true>(L, [&](auto tag) {
        using R = decltype(tag);
        constexpr int CM = CN2 > 0 ? CN2 / R::P : 0;
        const int m = CN2 > 0 ? CM : L.P2;
        const SmallDiv dm = small_div(m);
        const long long step = (long long)m * g.ncols;
        for (int it = threadIdx.x; it < 3 * C * m; it += blockDim.x) {
            const int cc = it & (C - 1), t = it / C, c = cdiv<CM>(t, dm), j = t - c * m;
            const int col = c0 + cc;
            float2 v[R::P];
            const float2* src = wspec + (long long)(c * N2 + j) * g.ncols + col;
#pragma unroll
            for (int i = 0; i < R::P; ++i) v[i] = col < g.ncols ? src[i * step] : make_float2(0.f, 0.f);
            group_fft<R, false, true, float2>(v, (const float2*)nullptr, 1);
            float2* d = sm + (c * C + cc) * S + ps * j;
#pragma unroll
            for (int i = 0; i < R::P; ++i) d[R::digit(i)] = v[i];
        }
    });
    __syncthreads();
    on_second<CN2>(L, [&](auto tag) {
        using R = decltype(tag);
        for (int it = threadIdx.x; it < C * P1; it += blockDim.x) {
            const int cc = it & (C - 1), k1 = it / C;
            const int col = min(c0 + cc, g.ncols - 1);
            const int kx = col % g.Nh, kz = col / g.Nh;
            // derivative wave numbers with the Nyquist components removed
            const int mx = (2 * kx == g.N1) ? 0 : kx;
            const int mz = (2 * kz == g.N3) ? 0 : ((2 * kz < g.N3) ? kz : kz - g.N3);
            const float Gx = g.gx * mx, Gz = g.gz * mz;
            float2* l = sm + cc * S + k1;
            float2 dv[R::P];  // i G . w / N at k = k1 + P1 i
#pragma unroll 1
            for (int c = 0; c < 3; ++c) {
                float2 v[R::P];
#pragma unroll
                for (int i = 0; i < R::P; ++i) v[i] = l[c * C * S + i * ps];
                group_fft<R, false, false, float2>(v, tw2 + k1, P1);
#pragma unroll
                for (int i = 0; i < R::P; ++i) {
                    const int k = k1 + P1 * R::digit(i);
                    const int my = (2 * k == N2) ? 0 : ((2 * k < N2) ? k : k - N2);
                    const float G = (c == 0 ? Gx : c == 1 ? g.gy * my : Gz) * g.invN;
                    float2& d = dv[R::digit(i)];
                    d.x = c == 0 ? -G * v[i].y : fmaf(-G, v[i].y, d.x);
                    d.y = c == 0 ? G * v[i].x : fmaf(G, v[i].x, d.y);
                }
            }
            group_fft<R, true, true, float2>(dv, (const float2*)nullptr, 1);
#pragma unroll
            for (int i = 0; i < R::P; ++i) l[R::digit(i) * ps] = dv[i];
        }
    });
    __syncthreads();
    on_first<CN2, true>(L, [&](auto tag) {
        using R = decltype(tag);
        const long long step = (long long)P2 * g.ncols;
        for (int it = threadIdx.x; it < C * P2; it += blockDim.x) {
            const int cc = it & (C - 1), j = it / C;
            const int col = c0 + cc;
            const float2* l = sm + cc * S + ps * j;
            float2 v[R::P];
#pragma unroll
            for (int i = 0; i < R::P; ++i) v[i] = l[i];
            group_fft<R, true, false, float2>(v, tw2s + j, P2);
            float2* dst = wspec + (long long)j * g.ncols + col;
            if (col < g.ncols) {
#pragma unroll
                for (int i = 0; i < R::P; ++i) dst[R::digit(i) * step] = v[i];
            }
        }
    });
}

// ---------------------------------------------------------------------------
// P5: inverse plane transform of D.w, v = v_loc - D.w
// ---------------------------------------------------------------------------
template <int CN1, int CN3>
__global__ void __launch_bounds__(PLANE_THREADS, 2)
    k_div_final(const float2* __restrict__ wspec, GridArgs g, const Tw* __restrict__ tw, float* __restrict__ v) {
    extern __shared__ float2 sm[];
    const int N1 = CN1 > 0 ? CN1 : g.N1, Nh = N1 / 2 + 1;
    const int y = blockIdx.x;
    const int zs = N1 * g.N2;
    // density blockIdx.y of a batch
    const float2* src = wspec + blockIdx.y * g.bs_wspec + (long long)y * g.ncols;
    float* vp = v + blockIdx.y * g.N + (long long)N1 * y;
    plane_inverse<CN1, CN3, float2>(
        sm, g, tw, [&](int kz, int kx) { return src[kz * Nh + kx]; },
        [&](int row, int x, float2 d) {
            const long long i = 2LL * row * zs + x;
            vp[i] -= d.x;
            vp[i + zs] -= d.y;
        });
}

// ---------------------------------------------------------------------------
// finite-difference gradient (the paper's own): central differences on the
// periodic grid, and the chain term of Eq. (Vi) as the transposed stencil
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_stencil_gradient(const float* __restrict__ f, GridArgs g, float3 ih2,
                                                          float* __restrict__ grad) {
    const long long N = g.N;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x) {
        int x, y, z;
        flat_point(i, g, x, y, z);
        const long long rowz = (long long)z * g.N2;
        const long long xm = i - x + (x == 0 ? g.N1 - 1 : x - 1), xp = i - x + (x == g.N1 - 1 ? 0 : x + 1);
        const long long ym = ((rowz + (y == 0 ? g.N2 - 1 : y - 1)) * g.N1) + x;
        const long long yp = ((rowz + (y == g.N2 - 1 ? 0 : y + 1)) * g.N1) + x;
        const long long zm = (((long long)(z == 0 ? g.N3 - 1 : z - 1) * g.N2 + y) * g.N1) + x;
        const long long zp = (((long long)(z == g.N3 - 1 ? 0 : z + 1) * g.N2 + y) * g.N1) + x;
        grad[i] = (f[xp] - f[xm]) * ih2.x;
        grad[N + i] = (f[yp] - f[ym]) * ih2.y;
        grad[2 * N + i] = (f[zp] - f[zm]) * ih2.z;
    }
}

// v -= sum_c D_c (g grad_c n): with the antisymmetric central-difference D,
// D^T w = -D w (w = g grad n, g from the assembly)
__global__ void __launch_bounds__(256) k_stencil_div_sub(const float* __restrict__ gg, const float* __restrict__ grad,
                                                         GridArgs g, float3 ih2, float* __restrict__ v) {
    const long long N = g.N;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x) {
        int x, y, z;
        flat_point(i, g, x, y, z);
        const long long rowz = (long long)z * g.N2;
        const long long xm = i - x + (x == 0 ? g.N1 - 1 : x - 1), xp = i - x + (x == g.N1 - 1 ? 0 : x + 1);
        const long long ym = ((rowz + (y == 0 ? g.N2 - 1 : y - 1)) * g.N1) + x;
        const long long yp = ((rowz + (y == g.N2 - 1 ? 0 : y + 1)) * g.N1) + x;
        const long long zm = (((long long)(z == 0 ? g.N3 - 1 : z - 1) * g.N2 + y) * g.N1) + x;
        const long long zp = (((long long)(z == g.N3 - 1 ? 0 : z + 1) * g.N2 + y) * g.N1) + x;
        const float d = (gg[xp] * grad[xp] - gg[xm] * grad[xm]) * ih2.x +
                        (gg[yp] * grad[N + yp] - gg[ym] * grad[N + ym]) * ih2.y +
                        (gg[zp] * grad[2 * N + zp] - gg[zm] * grad[2 * N + zm]) * ih2.z;
        v[i] -= d;
    }
}

// ---------------------------------------------------------------------------
// semilocal partner terms of Eq. (Exc): revPBE exchange (kappa = 1.245,
// mu = 0.066725 pi^2/3) and LDA correlation (the PW92 eps_c of q0)
// ---------------------------------------------------------------------------
// Adds de/dn to v and the coefficient of grad n in de/d(grad n) to g (so that
// the divergence stage takes it with the nonlocal w); FP64 block sums of
// e_x and e_c into epart[block] and epart[nb + block].
__global__ void __launch_bounds__(256) k_semilocal(const float* __restrict__ n, const float* __restrict__ grad,
                                                   long long N, float n_min, float* __restrict__ v,
                                                   float* __restrict__ gg, double* __restrict__ epart) {
    __shared__ double red[32];
    const float PI_F = 3.14159265358979f;
    const float KAPPA = 1.245f, MU = 0.066725f * PI_F * PI_F / 3.f;
    const float AX = -0.75f * 0.98474502184269641f;  // -(3/4) (3/pi)^(1/3)
    const float A = 0.031091f, a1 = 0.21370f;
    const float b1 = 7.5957f, b2 = 3.5876f, b3 = 1.6382f, b4 = 0.49294f;
    double sx = 0.0, sc = 0.0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x) {
        const float ni = n[i];
        if (!(ni > n_min) || !isfinite(ni)) continue;
        const float gx = grad[i], gy = grad[N + i], gz = grad[2 * N + i];
        const float cb = cbrtf(ni);
        const float kF = cbrtf(3.f * PI_F * PI_F) * cb;
        const float inv_n = 1.f / ni;
        const float s2 = (gx * gx + gy * gy + gz * gz) * (0.25f * inv_n * inv_n) / (kF * kF);
        const float den = 1.f + MU * s2 / KAPPA;
        const float Fx = 1.f + KAPPA - KAPPA / den;
        const float dF = MU / (den * den);
        const float e0 = AX * ni * cb;
        const float ex = e0 * Fx;
        const float dex = (4.f / 3.f) * AX * cb * Fx + e0 * dF * (-(8.f / 3.f) * s2 * inv_n);
        const float gex = e0 * dF * 2.f * (0.25f * inv_n * inv_n) / (kF * kF);
        const float rs = cbrtf(3.f / (4.f * PI_F * ni));
        const float srs = sqrtf(rs);
        const float Q = 2.f * A * (b1 * srs + b2 * rs + b3 * rs * srs + b4 * rs * rs);
        const float dQ = 2.f * A * (0.5f * b1 / srs + b2 + 1.5f * b3 * srs + 2.f * b4 * rs);
        const float Lg = log1pf(1.f / Q);
        const float ec = -2.f * A * (1.f + a1 * rs) * Lg;
        const float dec = -2.f * A * a1 * Lg + 2.f * A * (1.f + a1 * rs) * dQ / (Q * Q + Q);
        if (v) v[i] += dex + ec + ni * dec * (-rs * inv_n * (1.f / 3.f));
        if (gg) gg[i] += gex;
        sx += (double)ex;
        sc += (double)(ni * ec);
    }
    const double tx = block_sum(sx, red);
    __syncthreads();
    const double tcs = block_sum(sc, red);
    if (threadIdx.x == 0) {
        epart[blockIdx.x] = tx;
        epart[gridDim.x + blockIdx.x] = tcs;
    }
}

// E[4] = {E_xc, E_c^nl, E_x, E_c^LDA} from the nonlocal E[0] and the partials
__global__ void k_xc_final(const double* __restrict__ Enl, const double* __restrict__ epart, int nb, double dOmega,
                           double* __restrict__ E) {
    __shared__ double red[32];
    double a = 0.0, b = 0.0;
    for (int i = threadIdx.x; i < nb; i += blockDim.x) {
        a += epart[i];
        b += epart[nb + i];
    }
    const double ta = block_sum(a, red);
    __syncthreads();
    const double tb = block_sum(b, red);
    if (threadIdx.x == 0) {
        const double Ex = dOmega * ta, Ec = dOmega * tb;
        E[0] = Enl[0] + Ex + Ec;
        E[1] = Enl[0];
        E[2] = Ex;
        E[3] = Ec;
    }
}

// ---------------------------------------------------------------------------
// energy: fixed-order FP64 reduction of the block partials (the GPU's FP64
// rate is low: one block summing all partials took 17 us)
// ---------------------------------------------------------------------------
constexpr int ESPLIT_THREADS = 256;

// Block b of density blockIdx.y sums the share [b n / EPART_SPLIT, (b + 1) n /
// EPART_SPLIT) of each partial-sum array; the last block to finish adds the
// shares in index order, scaled into {E, E_soft, Delta E} (E alone if !all).
// One launch: a second one for the 64 shares cost 4 us of a small call.
__global__ void __launch_bounds__(ESPLIT_THREADS) k_energy(const double* __restrict__ epart, int nb0, int nb2,
                                                           double* escr, unsigned* __restrict__ count, double s0,
                                                           double s2, double* __restrict__ E, int all, int bs_epart) {
    __shared__ double red[32];
    __shared__ bool last;
    pdl_wait();
    epart += (long long)blockIdx.y * bs_epart;  // density blockIdx.y of a batch
    escr += (long long)blockIdx.y * bs_epart;
    E += (all ? 3 : 1) * blockIdx.y;
    count += blockIdx.y;
    const long long b = blockIdx.x;
    const int lo0 = (int)(b * nb0 / EPART_SPLIT), hi0 = (int)((b + 1) * nb0 / EPART_SPLIT);
    const int lo2 = (int)(b * nb2 / EPART_SPLIT), hi2 = (int)((b + 1) * nb2 / EPART_SPLIT);
    double a0 = 0.0, a2 = 0.0;
    for (int i = lo0 + threadIdx.x; i < hi0; i += blockDim.x) a0 += epart[i];
    for (int i = lo2 + threadIdx.x; i < hi2; i += blockDim.x) a2 += epart[nb0 + i];
    const double t0 = block_sum(a0, red);
    __syncthreads();
    const double t2 = block_sum(a2, red);
    if (threadIdx.x == 0) {
        __stcg(escr + b, t0);
        __stcg(escr + EPART_SPLIT + b, t2);
        __threadfence();
        last = atomicAdd(count, 1u) == EPART_SPLIT - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    const int i = threadIdx.x;
    const double u0 = block_sum(i < EPART_SPLIT ? __ldcg(escr + i) : 0.0, red);
    __syncthreads();
    const double u2 = block_sum(i < EPART_SPLIT ? __ldcg(escr + EPART_SPLIT + i) : 0.0, red);
    if (threadIdx.x == 0) {
        const double dE = s0 * u0, Es = s2 * u2;
        E[0] = Es + dE;
        if (all) {
            E[1] = Es;
            E[2] = dE;
        }
        *count = 0;
    }
}

// Twiddle table of a line's second group with radices A, B, C after Ns (order
// as group_fft reads it): W_n^e = exp(-2 pi i e / n) in FP64, stored as the
// hi/lo FP32 pair of each part.
__global__ void k_twiddles(Tw* tw, int n, int Ns, int A, int B, int C) {
    const int tot = (A * B * C - 1) * Ns;
    for (int i = threadIdx.x + blockIdx.x * blockDim.x; i < tot; i += blockDim.x * gridDim.x) {
        int q = i / Ns;
        const int k = i - q * Ns;
        int e;
        if (q < A - 1) {
            e = (q + 1) * k * (n / (Ns * A));
        } else if (q < A * B - 1) {
            q -= A - 1;
            e = (q / A + 1) * (k + (q % A) * Ns) * (n / (Ns * A * B));
        } else {
            q -= A * B - 1;
            e = (q / (A * B) + 1) * (k + (q % (A * B)) * Ns) * (n / (Ns * A * B * C));
        }
        double s, c;
        sincospi(-2.0 * (double)e / (double)n, &s, &c);
        const float ch = (float)c, sh = (float)s;
        tw[i] = make_float4(ch, sh, (float)(c - (double)ch), (float)(s - (double)sh));
    }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
// The groups fft.cuh has (second_group / first_group): the radices of a
// product, {1, 1, 1} where it has none.
struct Radices {
    int a, b, c;
};
static Radices radices_of(int P) {
    switch (P) {
        case 6: return {2, 3, 1};
        case 8: return {4, 2, 1};
        case 9: return {3, 3, 1};
        case 10: return {2, 5, 1};
        case 12: return {4, 3, 1};
        case 15: return {3, 5, 1};
        case 16: return {4, 4, 1};
        case 18: return {2, 3, 3};
        case 20: return {4, 5, 1};
        case 24: return {4, 2, 3};
        case 25: return {5, 5, 1};
        case 27: return {3, 3, 3};
        default: return {P, 1, 1};  // 1 .. 5
    }
}

// The radices of n are 4, .., 4, 2, 3, .., 3, 5, .., 5 in this order.  Of the
// places where that list can be cut into two groups that exist, the one with
// the smallest larger group is taken (registers and work per thread), the
// larger second group on a tie (longer runs in the first pass's loads).
int make_line_plan(int n, bool sized, LinePlan* lp) {
    lp->n = n;
    lp->P1 = lp->P2 = 0;
    if (sized) {
        lp->P1 = n == 180 ? 15 : n == 72 ? 9 : n == 256 ? 16 : 12;
        lp->P2 = n / lp->P1;
        return VDW_OK;
    }
    int rad[16], nr = 0, m = n;
    for (int r : {4, 2, 3, 5})
        while (m % r == 0) {
            rad[nr++] = r;
            m /= r;
        }
    if (m != 1) return VDW_ERR_SIZE;
    const auto is_group = [&](int i0, int i1, bool first) {
        int P = 1;
        for (int i = i0; i < i1; ++i) P *= rad[i];
        if (P > 27 || i1 - i0 > 3) return 0;
        if (P == 1) return first ? 0 : 1;
        const Radices r = radices_of(P);
        const int want[3] = {r.a, r.b, r.c};
        for (int i = 0; i < 3; ++i)
            if ((i0 + i < i1 ? rad[i0 + i] : 1) != want[i]) return 0;
        if (!first && (P == 18 || P == 20 || P == 24 || P == 27)) return 0;
        return P;
    };
    for (int cut = 1; cut <= nr; ++cut) {
        const int a = is_group(0, cut, true), b = is_group(cut, nr, false);
        if (!a || !b) continue;
        const int big = std::max(a, b), cur = std::max(lp->P1, lp->P2);
        if (lp->P1 == 0 || big < cur || (big == cur && b > lp->P2)) {
            lp->P1 = a;
            lp->P2 = b;
        }
    }
    return lp->P1 ? VDW_OK : VDW_ERR_SIZE;
}

// Block size in [lo, hi] (whole warps) with the fewest thread slots over
// passes of items of a given cost each, the largest on a tie.
struct Pass {
    int items, cost;
};
static int best_threads(std::initializer_list<Pass> passes, int lo, int hi) {
    int best = hi;
    long long least = -1;
    for (int t = hi; t >= lo; t -= 32) {
        long long c = 0;
        for (const Pass& p : passes) c += (long long)((p.items + t - 1) / t) * t * p.cost;
        if (least < 0 || c < least) {
            least = c;
            best = t;
        }
    }
    return best;
}

// shared memory of a plane kernel, forward or inverse, with hi/lo (exact) or
// FP32 twiddles
static size_t smem_plane_of(const GridArgs& g, bool inverse, bool exact, bool pad) {
    const LinePlan& l = inverse && !exact ? g.p1i : g.p1;
    const PlaneGeo p = plane_geo(l.P1, l.P2, inverse, pad);
    return sizeof(float2) * tw_offset((size_t)(g.N3 / 2) * p.S) +
           (exact ? sizeof(Tw) : sizeof(float2)) * ((size_t)(g.N1 - l.P1) + (g.N3 - g.p3.P1));
}
size_t smem_plane(const GridArgs& g, bool inverse, bool exact) {
    return smem_plane_of(g, inverse, exact, inverse ? g.pad_inv : g.pad_fwd);
}

// Block size of a plane kernel launched on nblocks planes: as many threads
// per SM as its registers allow, over the blocks that shared memory and the
// grid allow there, and among the sizes near that the one that wastes the
// fewest thread slots over the passes.
int plane_block(const vdw_ctx* c, long long nblocks, bool inverse, bool exact) {
    const GridArgs& g = c->g;
    const int nr = g.N3 / 2;
    const long long nsm = std::max(c->nsm, 1);
    const long long smem = (long long)smem_plane(g, inverse, exact) + 1024;
    // three blocks may fill the SM's memory; a fourth only where it leaves
    // some for L1, through which the planes are loaded (w planes of 180 x 180
    // x 72: 29 us with three blocks of 288 threads, 37 with four of 256)
    const long long fit = std::max(1LL, std::min(228 * 1024 / smem, std::max(3LL, 192 * 1024 / smem)));
    const int most = PLANE_THREADS;
    // small planes, many of them: a block keeps at least one warp (32 densities
    // of 24^3 213 us; two warps 229, four 240)
    const long long per_sm = std::clamp<long long>(std::min(fit, (nblocks + nsm - 1) / nsm), 1, 2 * most / 32);
    const bool fused = !inverse && exact && on_grid(g, [&](auto d) { return g.p1.P2 <= FUSE_P<decltype(d)::N1, Tw>; });
    const int items = std::max({nr * g.p1.P2, nr * g.p1.P1, g.Nh * g.p3.P2, g.Nh * g.p3.P1});
    const int hi = std::min((int)std::min<long long>(most, 2 * most / per_sm) / 32 * 32, (items + 31) / 32 * 32);
    const int lo = std::min(hi, (int)(2 * most / (per_sm + 1)) / 32 * 32 + 32);  // no room for another block
    const bool merged = inverse && !exact && on_grid(g, [&](auto d) { return g.p1i.P1 <= MERGE_P<decltype(d)::N1>; });
    const LinePlan& l = inverse && !exact ? g.p1i : g.p1;
    const Pass first = merged ? Pass{nr * (l.P2 / 2 + 1), 2 * l.P1} : Pass{nr * l.P2, l.P1};
    const Pass second = fused ? Pass{nr * (l.P1 / 2 + 1), 2 * l.P2} : Pass{nr * l.P1, l.P2};
    return best_threads({first, second, {fused || merged ? 0 : g.Nh * nr, 2}, {g.Nh * g.p3.P2, g.p3.P1},
                         {g.Nh * g.p3.P1, g.p3.P2}},
                        lo, hi);
}
static size_t smem_div(const GridArgs& g) {
    return sizeof(float2) * tw_offset((size_t)3 * DIV_COLS * pencil_stride(g.p2)) +
           sizeof(float2) * ((size_t)2 * g.N2 - g.p2.P1 - g.p2.P2);
}

// dynamic shared memory per block, leaving room for the kernels' static arrays
static const size_t SMEM_MAX = 227 * 1024 - 1024;

int pipeline_plan_check(vdw_ctx* c) {
    GridArgs& g = c->g;
    g.pad_fwd = smem_plane_of(g, false, true, true) <= SMEM_MAX;
    g.pad_inv = smem_plane_of(g, true, true, true) <= SMEM_MAX && smem_plane_of(g, true, false, true) <= SMEM_MAX;
    // the whole-plane limit of the unpadded rows
    if (sizeof(float2) * (size_t)g.N3 * g.Nh + sizeof(Tw) * (g.N1 + g.N3) > 222 * 1024 ||
        smem_plane(g, false, true) > SMEM_MAX || smem_plane(g, true, true) > SMEM_MAX ||
        smem_plane(g, true, false) > SMEM_MAX || sorted_pencil_smem(g) > SMEM_MAX || smem_div(g) > SMEM_MAX)
        return VDW_ERR_SIZE;
    return VDW_OK;
}

int pipeline_make_twiddles(vdw_ctx* c) {
    const GridArgs& g = c->g;
    const bool sized = sized_grid(g.N1, g.N2, g.N3);
    const auto make = [&](int off, int n, int Ns, int P) {
        const Radices r = sized ? Radices{P, 1, 1} : radices_of(P);
        if (P > 1) k_twiddles<<<4, 256>>>(c->d_tw + off, n, Ns, r.a, r.b, r.c);
    };
    make(0, g.N1, g.p1.P1, g.p1.P2);
    make(tw_off_y(g), g.N2, g.p2.P1, g.p2.P2);
    make(g.N1 + g.N2, g.N3, g.p3.P1, g.p3.P2);
    make(tw_off_swap(g), g.N2, g.p2.P2, g.p2.P1);
    make(tw_off_xi(g), g.N1, g.p1i.P1, g.p1i.P2);
    VDW_CUDA(cudaGetLastError());
    VDW_CUDA(cudaDeviceSynchronize());
    return VDW_OK;
}

static float3 stencil_ih2(const vdw_ctx* c) {
    return make_float3((float)(c->g.N1 / (2.0 * c->L[0])), (float)(c->g.N2 / (2.0 * c->L[1])),
                       (float)(c->g.N3 / (2.0 * c->L[2])));
}
static int stencil_blocks(const GridArgs& g) { return (int)std::min<long long>((g.N + 255) / 256, 8192); }

int pipeline_stencil_gradient(vdw_ctx* c, const float* f, float* grad, cudaStream_t s) {
    k_stencil_gradient<<<stencil_blocks(c->g), 256, 0, s>>>(f, c->g, stencil_ih2(c), grad);
    VDW_CUDA(cudaGetLastError());
    return VDW_OK;
}

// one wave of resident blocks, each thread striding over several points: the
// spline table is staged once per block
static int u_sum_blocks(const vdw_ctx* c) {
    const GridArgs& g = c->g;
    return (int)std::min<long long>((g.N / 2 + USUM_THREADS - 1) / USUM_THREADS,
                                    (long long)std::max(c->usum_per_sm, 1) * std::max(c->nsm, 1));
}

static int launch_u_sum(vdw_ctx* c, const float* grad, float* v, float* w, int mode, cudaStream_t s, int B,
                        GradScale gs) {
    const GridArgs& g = c->g;
    const int nb = u_sum_blocks(c);
    const double dOmega = c->L[0] * c->L[1] * c->L[2] / (double)g.N;
#define VDW_U_SUM(NQ) \
    launch(early_launch(g, B), k_u_sum<NQ>, dim3(nb, B), USUM_THREADS, 0, s, c->d_spec, grad, c->d_t, c->d_k, c->d_aux, g, c->pp, v, w, \
           c->d_gg, mode, gs.on ? gs.gE : nullptr, dOmega)
    switch (c->pp.Nq) {
        case 20: VDW_U_SUM(20); break;
        case 8: VDW_U_SUM(8); break;
        case 12: VDW_U_SUM(12); break;
        case 16: VDW_U_SUM(16); break;
        default: set_error("Nq not compiled in"); return VDW_ERR_UNSUPPORTED;
    }
#undef VDW_U_SUM
    return VDW_OK;
}

template <int CN1, int CN2, int CN3>
static int run_sized(vdw_ctx* c, const float* n, const float* grad, double* E, float* v, float* w, cudaStream_t s,
                     int fd, int xc, const cudaEvent_t* slab_ready, int B, GradScale gs) {
    const GridArgs& g = c->g;
    const PointParams& P = c->pp;
    const bool want_pot = (v != nullptr) || (w != nullptr);
    // stage marks for vdw_profile_read (event k+1 closes stage k)
    auto mark = [&](int stage) {
        if (c->prof) {
            cudaEventRecord(c->ev[stage + 1], s);
            c->ev_done[stage] = 1;
        }
    };
    if (c->prof) {
        for (int i = 0; i < VDW_NSTAGES; ++i) c->ev_done[i] = 0;
        cudaEventRecord(c->ev[0], s);
    }
    // one launch over all slabs, or (host entry point) one per slab as its inputs arrive
    const int nlaunch = slab_ready ? c->p0_chunks : 1;
    for (int sl = 0; sl < nlaunch; ++sl) {
        if (slab_ready) VDW_CUDA(cudaStreamWaitEvent(s, slab_ready[sl], 0));
        const int slab = slab_ready ? sl : -1;
        const int nblk = slab_ready ? c->nb_p0 : c->nb_point;
#define VDW_POINTWISE(NQ)                                                                                  \
    launch(early_launch(g, B), k_pointwise<NQ>, dim3(nblk, B), 256, 0, s, n, grad, g, P, slab, c->p0_nj, c->p0_mnj, c->nb_p0, c->d_t, \
           c->d_k, c->d_aux, c->d_spec, c->d_epart, c->d_bad)
        switch (P.Nq) {
            case 20: VDW_POINTWISE(20); break;
            case 8: VDW_POINTWISE(8); break;
            case 12: VDW_POINTWISE(12); break;
            case 16: VDW_POINTWISE(16); break;
            default: set_error("Nq not compiled in"); return VDW_ERR_UNSUPPORTED;
        }
#undef VDW_POINTWISE
    }
    mark(ST_POINTWISE);

    int rc = planes_inplace(c, P.Nq, false, s, B);
    if (rc) return rc;
    mark(ST_PLANES_FWD);

    // y transforms, contraction in |G| order, inverse y transforms (contract.cu)
    rc = sorted_forward(c, P.Nq, s, B);
    if (rc) return rc;
    mark(ST_PENCILS_FWD);
    rc = sorted_contract(c, c->d_epart + c->nb_point, want_pot ? 1 : 0, s, B);
    if (rc) return rc;
    mark(ST_CONTRACT);
    // With a potential to follow (and no stage timing), the energy reduction
    // runs on the context's side stream beside the inverse transforms, which
    // do not touch the partial sums; the caller's stream waits for it before
    // the call returns (so the next call's partial sums come after it).
    bool forked = false;
    auto join = [&]() {
        if (forked) cudaStreamWaitEvent(s, c->ev_join, 0);
        forked = false;
    };
    if (E) {
        const double Omega = c->L[0] * c->L[1] * c->L[2];
        const double Nd = (double)g.N;
        double* escr = c->d_epart + c->nb_point + c->nb_sorted;
        cudaStream_t se = s;
        if (want_pot && !c->prof) {
            VDW_CUDA(cudaEventRecord(c->ev_fork, s));
            VDW_CUDA(cudaStreamWaitEvent(c->s_side, c->ev_fork, 0));
            se = c->s_side;
        }
        launch(se == s && early_launch(g, B), k_energy, dim3(EPART_SPLIT, B), ESPLIT_THREADS, 0, se, c->d_epart,
               c->nb_point, c->nb_sorted, escr, c->d_ecount, Omega / Nd, 0.5 * Omega / (Nd * Nd), E, gs.on ? 0 : 1,
               g.bs_epart);
        if (se != s) {
            VDW_CUDA(cudaEventRecord(c->ev_join, se));
            forked = true;
        }
        mark(ST_ENERGY);
    }
    if (xc && !want_pot)
        k_semilocal<<<XC_BLOCKS, 256, 0, s>>>(n, grad, g.N, P.n_min, nullptr, nullptr, c->d_xc + 4);
    if (want_pot) {
        rc = sorted_inverse(c, P.Nq, s, B);
        if (rc) {
            join();
            return rc;
        }
        mark(ST_PENCILS_INV);
        const int mode = (w != nullptr || gs.on) ? 0 : 1;
        rc = planes_inplace(c, P.Nq, true, s, B);
        if (rc) {
            join();
            return rc;
        }
        mark(ST_PLANES_INV);
        const int rcs = launch_u_sum(c, grad, v, w, mode, s, B, gs);
        if (rcs) {
            join();
            return rcs;
        }
        if (xc)
            k_semilocal<<<XC_BLOCKS, 256, 0, s>>>(n, grad, g.N, P.n_min, v, mode == 1 ? c->d_gg : nullptr,
                                                  c->d_xc + 4);
        mark(ST_USUM);
        if (mode == 1 && fd) {
            // finite-difference gradient: the chain term is a stencil, no transforms
            k_stencil_div_sub<<<stencil_blocks(g), 256, 0, s>>>(c->d_gg, grad, g, stencil_ih2(c), v);
            mark(ST_DIV_FINAL);
        } else if (mode == 1) {
            launch(early_launch(g, B), k_w_planes<CN1, CN3>, dim3(g.N2, 3, B), plane_block(c, 3LL * g.N2 * B, false, false),
                   smem_plane(g, false, false), s, c->d_gg, grad, g, c->d_tw, c->d_wspec);
            mark(ST_W_PLANES);
            launch(early_launch(g, B), k_pencil_div<CN2>, dim3((g.ncols + DIV_COLS - 1) / DIV_COLS, B), DIV_THREADS, smem_div(g), s,
                   c->d_wspec, g, c->d_tw + tw_off_y(g), c->d_tw + tw_off_swap(g));
            mark(ST_PENCIL_DIV);
            launch(early_launch(g, B), k_div_final<CN1, CN3>, dim3(g.N2, B), plane_block(c, (long long)g.N2 * B, true, false),
                   smem_plane(g, true, false), s, c->d_wspec, g, c->d_tw, v);
            mark(ST_DIV_FINAL);
        }
    }
    join();
    VDW_CUDA(cudaGetLastError());
    return VDW_OK;
}

template <int CN1, int CN2, int CN3>
static int configure_sized(vdw_ctx* c) {
    const GridArgs& g = c->g;
    const int sf = (int)smem_plane(g, false, false), sp = (int)smem_plane(g, true, false);
    const int sd = (int)smem_div(g);
    int rc = planes_configure(c);
    if (!rc) rc = set_and_check(k_pencil_div<CN2>, "k_pencil_div", sd, DIV_THREADS);
    if (!rc) rc = set_and_check(k_div_final<CN1, CN3>, "k_div_final", sp, PLANE_THREADS);
    if (!rc) rc = set_and_check(k_w_planes<CN1, CN3>, "k_w_planes", sf, PLANE_THREADS);
    if (rc) return rc;
    rc = sorted_configure(c);
    if (rc) return rc;
    // resident blocks per SM of the field sum (its grid is one wave of them)
    int per_sm = 0;
    switch (c->p.Nq) {
        case 20: VDW_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_u_sum<20>, USUM_THREADS, 0)); break;
        case 16: VDW_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_u_sum<16>, USUM_THREADS, 0)); break;
        case 12: VDW_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_u_sum<12>, USUM_THREADS, 0)); break;
        default: VDW_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_u_sum<8>, USUM_THREADS, 0));
    }
    c->usum_per_sm = per_sm;
    return VDW_OK;
}

int pipeline_configure(vdw_ctx* c) {
    return on_grid(c->g, [&](auto d) {
        using D = decltype(d);
        return configure_sized<D::N1, D::N2, D::N3>(c);
    });
}

template <int CN1, int CN2, int CN3>
static void launch_divergence(vdw_ctx* c, float* v, cudaStream_t s) {
    const GridArgs& g = c->g;
    launch(early_launch(g, 1), k_pencil_div<CN2>, (g.ncols + DIV_COLS - 1) / DIV_COLS, DIV_THREADS, smem_div(g), s,
                   c->d_wspec, g, c->d_tw + tw_off_y(g), c->d_tw + tw_off_swap(g));
    launch(early_launch(g, 1), k_div_final<CN1, CN3>, g.N2, plane_block(c, g.N2, true, false),
                   smem_plane(g, true, false), s, c->d_wspec, g, c->d_tw, v);
}

template <int CN1, int CN3>
static void launch_w_planes(vdw_ctx* c, const float* grad, cudaStream_t s) {
    const GridArgs& g = c->g;
    launch(early_launch(g, 1), k_w_planes<CN1, CN3>, dim3(g.N2, 3), plane_block(c, 3LL * g.N2, false, false),
                   smem_plane(g, false, false), s, c->d_gg, grad, g, c->d_tw, c->d_wspec);
}

int pipeline_w_planes(vdw_ctx* c, const float* grad, cudaStream_t s) {
    on_grid(c->g, [&](auto d) {
        using D = decltype(d);
        launch_w_planes<D::N1, D::N3>(c, grad, s);
    });
    VDW_CUDA(cudaGetLastError());
    return VDW_OK;
}

int pipeline_divergence(vdw_ctx* c, float* v, cudaStream_t s) {
    on_grid(c->g, [&](auto d) {
        using D = decltype(d);
        launch_divergence<D::N1, D::N2, D::N3>(c, v, s);
    });
    VDW_CUDA(cudaGetLastError());
    return VDW_OK;
}

int pipeline_energy_final(vdw_ctx* c, const double* epart, int nb0, int nb2, double* E, cudaStream_t s) {
    const double Omega = c->L[0] * c->L[1] * c->L[2];
    const double Nd = (double)c->g.N;
    // the shares go to the context's own scratch (after density 0's partial sums)
    double* escr = c->d_epart + c->nb_point + c->nb_sorted;
    launch(early_launch(c->g, 1), k_energy, dim3(EPART_SPLIT, 1), ESPLIT_THREADS, 0, s, epart, nb0, nb2, escr, c->d_ecount,
           Omega / Nd, 0.5 * Omega / (Nd * Nd), E, 1, 0);
    VDW_CUDA(cudaGetLastError());
    return VDW_OK;
}

int pipeline_run(vdw_ctx* c, const float* n, const float* grad, double* E, float* v, float* w, cudaStream_t s,
                 int fd, int xc, const cudaEvent_t* slab_ready, int B, GradScale gs) {
    return on_grid(c->g, [&](auto d) {
        using D = decltype(d);
        return run_sized<D::N1, D::N2, D::N3>(c, n, grad, E, v, w, s, fd, xc, slab_ready, B, gs);
    });
}

int pipeline_xc_final(vdw_ctx* c, double* E, cudaStream_t s) {
    const double dOmega = c->L[0] * c->L[1] * c->L[2] / (double)c->g.N;
    k_xc_final<<<1, 256, 0, s>>>(c->d_xc, c->d_xc + 4, XC_BLOCKS, dOmega, E);
    VDW_CUDA(cudaGetLastError());
    return VDW_OK;
}

}  // namespace vdw
