// P1 and P3 of the hot path (pipeline.cu): the plane transforms of theta_a and
// u_a, in place.
#include "plane.cuh"

#include <algorithm>
#include <climits>

namespace vdw {

// One block per (y plane, field).  Both sides of the transform keep the
// packed real layout: real rows 2j and 2j + 1 are the real and imaginary
// parts of complex row j, which starts 2 Nh j values into the plane.
// Forward: those rows are replaced by their half spectrum; inverse: the half
// spectrum of u_a is replaced by the packed rows of its real values (unscaled:
// 1/N is folded into the contraction).
//
// Bound by shared memory (about eight 8-byte accesses per point) and issue
// slots, not by HBM (half its bandwidth).  The plane goes from global memory
// straight into the first pass's registers and from the last pass's back, so
// that only the three exchanges between the four register passes and the
// real/half-spectrum step touch shared memory (the form before staged the
// plane by a bulk copy and made every radix pass, 3 or 4 per line at a
// run-time length, a load and a store).  us per launch, 20 fields, before and
// after, forward / inverse: 180 x 180 x 72 156 / 154 -> 96 / 94; 256 x 256 x
// 96 358 / 323 -> 274 / 274; run-time lengths, 144 x 144 x 72 (per density)
// 304 / 288 -> 70 / 64, 200 x 200 x 72 545 / 506 -> 164 / 142, 128^3 303 /
// 266 -> 102 / 98, 100^3 174 / 171 -> 56 / 55.
template <int CN1, int CN3, bool INV>
__global__ void __launch_bounds__(PLANE_THREADS, 2)
    k_planes_inplace(float2* __restrict__ spec, GridArgs g, const Tw* __restrict__ tw, int ahead) {
    extern __shared__ float2 sm[];
    const int Nh = CN1 > 0 ? CN1 / 2 + 1 : g.Nh;
    const int y = blockIdx.x, a = blockIdx.y;
    float2* p = spec + blockIdx.z * g.bs_spec + ((long long)a * g.N2 + y) * g.ncols;
    // the planes of a launch are contiguous in block order
    const long long left = (long long)gridDim.x * gridDim.y * gridDim.z - 1 -
                           (y + (long long)gridDim.x * (a + (long long)gridDim.y * blockIdx.z));
    if (threadIdx.x == 0 && ahead <= left) prefetch_l2(p + (long long)ahead * g.ncols, (unsigned)sizeof(float2) * g.ncols);
    const auto row_at = [&](int row, int x) { return p + (row * 2 * Nh + x); };
    const auto pt_at = [&](int kz, int kx) { return p + (kz * Nh + kx); };
    // the forward transforms of theta feed the energy: hi/lo twiddles there
    if constexpr (INV)
        plane_inverse<CN1, CN3, float2>(
            sm, g, tw, [&](int kz, int kx) { return *pt_at(kz, kx); },
            [&](int row, int x, float2 u) { *row_at(row, x) = u; });
    else
        plane_forward<CN1, CN3, Tw>(
            sm, g, tw, [&](int row, int x) { return *row_at(row, x); },
            [&](int kz, int kx, float2 c) { *pt_at(kz, kx) = c; });
}

int planes_configure(vdw_ctx* c) {
    const int sf = (int)smem_plane(c->g, false, true), si = (int)smem_plane(c->g, true, false);
    return on_grid(c->g, [&](auto d) {
        using D = decltype(d);
        int rc = set_and_check(k_planes_inplace<D::N1, D::N3, true>, "k_planes_inplace", si, PLANE_THREADS);
        if (!rc) rc = set_and_check(k_planes_inplace<D::N1, D::N3, false>, "k_planes_inplace", sf, PLANE_THREADS);
        return rc;
    });
}

int planes_inplace(vdw_ctx* c, int nfields, bool inverse, cudaStream_t s, int B) {
    const GridArgs& g = c->g;
    const dim3 grid(g.N2, nfields, B);
    const int nt = plane_block(c, (long long)g.N2 * nfields * B, inverse, !inverse);
    const size_t sm = smem_plane(g, inverse, !inverse);
    // Where an SM holds two planes at most, a block asks L2 for the plane of the
    // block that follows it (256 x 256 x 96: 285 -> 274 us; with three blocks
    // per SM the others hide that latency, and 128^3 takes 104 us against 101);
    // with fewer fields than planned the densities are not contiguous.
    const int per_sm = std::max(1, std::min((int)(228 * 1024 / (sm + 1024)), 2 * PLANE_THREADS / nt));
    const int ahead = per_sm > 2 || (B > 1 && nfields != c->p.Nq) ? INT_MAX : std::max(1, c->nsm) * per_sm;
    on_grid(g, [&](auto d) {
        using D = decltype(d);
        if (inverse) launch(early_launch(g, B), k_planes_inplace<D::N1, D::N3, true>, grid, nt, sm, s, c->d_spec, g, c->d_tw, ahead);
        else launch(early_launch(g, B), k_planes_inplace<D::N1, D::N3, false>, grid, nt, sm, s, c->d_spec, g, c->d_tw, ahead);
    });
    VDW_CUDA(cudaGetLastError());
    return VDW_OK;
}

}  // namespace vdw
