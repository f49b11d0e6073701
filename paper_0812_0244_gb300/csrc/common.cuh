// Shared definitions of the vdwnl CUDA library (sm_103a).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>
#include <stddef.h>
#include <string>

#include "../../include/vdwnl.h"

namespace vdw {

// Stages of one call, for vdw_profile_read (include/vdwnl.h lists them).
enum Stage {
    ST_POINTWISE = 0,
    ST_PLANES_FWD,
    ST_PENCILS_FWD,
    ST_CONTRACT,
    ST_ENERGY,
    ST_PENCILS_INV,
    ST_PLANES_INV,
    ST_USUM,
    ST_W_PLANES,
    ST_PENCIL_DIV,
    ST_DIV_FINAL,
    ST_COUNT
};
static_assert(ST_COUNT == VDW_NSTAGES, "stage list");

constexpr int MAX_NQ = 32;     // largest interpolation mesh the kernels take
constexpr int MAX_MC = 32;     // largest order m_c of the saturation sum of Eq. (Sat)
constexpr int MAX_DIM = 256;   // largest grid dimension (FFT line length)
constexpr int POINT_BLOCKS = 4;  // blocks of the pointwise kernel per SM
constexpr uint8_t K_INVALID = 255;  // interval code of a point with theta = 0

// Schedule of one line length n = P1 P2: the products of the two groups of
// radices its transform takes in registers (fft.cuh, make_line_plan).
struct LinePlan {
    int n;
    int P1, P2;
};

// Pointwise constants, passed by value (kernel parameter space).
struct PointParams {
    int Nq;
    int m_c;
    float q_c;
    float n_min;
    float C_s;
    float inv_m[MAX_MC + 1];     // 1/m, m = 1 .. m_c (terms of the saturation sum)
    float qm[MAX_NQ];            // q mesh
    // device, [MAX_NQ][MAX_NQ]: Mq[a MAX_NQ + k] = second derivative of p_a at
    // knot k (a block copies what it needs to shared memory)
    const float* Mq;
};

// Grid geometry shared by the plane and pencil kernels.
struct GridArgs {
    int N1, N2, N3, Nh;    // Nh = N1/2 + 1
    long long N;           // N1 N2 N3
    int ncols;             // N3 * Nh: columns of the half spectrum per y
    float gx, gy, gz;      // 2 pi / L_d
    // Flat-index divisions by N1, N2 and N3/2 as multiply-high by
    // m = ceil(2^32 / d), exact for i d < 2^32; fast = 0 (plain division)
    // when N max(N1, N2, N3) reaches 2^32 or a divisor is 1.
    unsigned m1, m2, mh3;
    float inv_dk;          // 1 / Delta k of the radial table
    int Nk;                // points of the radial table
    float invN;            // 1 / N
    LinePlan p1, p2, p3;   // line transforms along x, y, z
    LinePlan p1i;          // inverse along x of u and D.w (its groups may be in the other order)
    int pad_fwd, pad_inv;  // plane transforms with padded rows (plane_geo)
    int fast;              // flat-index divisions by m1, m2, mh3
    // batches (vdw_energy_potential_batched): density b of a batch uses the
    // workspaces at these element offsets times b; the kernels take b from
    // their last grid dimension (0 for a single density)
    long long bs_spec;   // float2 values between two densities' spectrum buffers
    long long bs_wspec;  // float2 values between two w-spectrum buffers
    long long bs_Q;      // float4 values between two record buffers (contract.cu)
    int bs_epart;        // energy partial sums per density
};

// Learned reduced basis: sizes fixed at compile time.
constexpr int LRN_H = 64;                          // hidden units of the channel network
constexpr int LRN_M = 8;                           // channels
constexpr int LRN_P = LRN_M * (LRN_M + 1) / 2;     // learned pair kernels m <= n
constexpr int LRN_N3 = 16;                         // last layer padded to a legal MMA width
// offsets in the flat parameter vector: W1 [H][2], b1, W2 [H][H], b2, W3 [M][H], b3, K [P][J]
constexpr int LRN_OFF_W1 = 0;
constexpr int LRN_OFF_B1 = LRN_OFF_W1 + LRN_H * 2;
constexpr int LRN_OFF_W2 = LRN_OFF_B1 + LRN_H;
constexpr int LRN_OFF_B2 = LRN_OFF_W2 + LRN_H * LRN_H;
constexpr int LRN_OFF_W3 = LRN_OFF_B2 + LRN_H;
constexpr int LRN_OFF_B3 = LRN_OFF_W3 + LRN_M * LRN_H;
constexpr int LRN_OFF_K = LRN_OFF_B3 + LRN_M;

// Device view of a loaded learned model (kernel parameter).  The bf16
// operands are stored in the tensor-core layout (tc.cuh) as raw 16-bit words.
struct LearnedArgs {
    int J;                  // knots
    float dk, inv_dk;       // knot spacing and its inverse
    float mu1, inv_sig1, mu2, inv_sig2, eps2;  // feature standardisation, eps^2
    const float* w1;        // [H][2] bf16-rounded values
    const float* b1;        // [H]
    const float* b2;        // [H]
    const float* b3;        // [M]
    const uint16_t* w2f;    // forward operand W2 [H out][H in]
    const uint16_t* w3f;    // forward operand W3 [16 (M padded)][H]
    const float* w3r;       // W3 bf16-rounded values, row-major [M][H]
    const float4* knots;    // [J-1][P]: cubic coefficients in t of the Catmull-Rom piece on interval j
    int* err;               // set when a tensor-core wait gives up
    int base;               // channel weights = spline base + network (1) or network alone (0)
    // the network tabulated on the feature nodes (vdw_learned_tabulate): node
    // (i1, i2), i = 0 .. T + 1, at x = -D + (i - 1) h, its 8 outputs at
    // node (i1, i2): channels 0-3 at tab[i1 (T + 2) + i2], 4-7 at the same
    // index + (T + 2)^2; tabT = 0: no table
    const float4* tab;
    int tabT;
    float tabD, tab_h, tab_inv_h;
    float bqm[LRN_M];       // base mesh
    float bMq[LRN_M * LRN_M];  // bMq[m * M + k]: second derivative of base spline m at knot k
};

}  // namespace vdw

// The context behind the opaque vdw_handle.
struct vdw_ctx {
    vdw_params p;
    int device;
    // tables
    vdw::PointParams pp;        // host copy of the pointwise constants
    double phi0, C_s;
    float4* d_kcoef;            // [Nk-1][npairs] cubic coefficients in local t
    float* d_Mq;                // behind pp.Mq
    // plan
    int planned;
    vdw::GridArgs g;
    double L[3];
    float4* d_tw;               // twiddle tables (hi/lo pairs): x, y, z lines, y lines with their groups swapped
    float2* d_spec;             // [Nq][N2][N3][Nh] theta(G), then u(G), then real u (packed rows), in place
    float2* d_wspec;            // [3][N2][N3][Nh] w(G); component 0 then D.w
    float* d_t;                 // [N] position of q inside its mesh interval
    uint8_t* d_k;               // [N] mesh interval of q (K_INVALID: theta = 0)
    float4* d_aux;              // [N] n dq/dn, n dq/d|grad n| / |grad n|, and the Delta E derivatives
    double* d_epart;            // per-block energy partial sums
    unsigned* d_ecount;         // per density: blocks of the running energy reduction that are done
    int nb_point;               // their count for the pointwise kernel
    // points of the half spectrum in |G| order (contract.cu)
    long long nG, Npad;         // N2 N3 (N1/2 + 1), rounded up to whole contraction blocks
    int nb_sorted;              // contraction blocks (and energy partials)
    unsigned* d_pos;            // [N3 Nh][N2] sorted position of point (col, y)
    float* d_gs;                // [Npad] |G| of each sorted point, sign = energy weight
    float4* d_Q;                // [Nq/4][Npad][2] field quads of the sorted points
    int batch_max;              // densities the per-density workspaces hold (vdw_plan_batch)
    int nsm;                    // SMs of the device (persistent grids)
    int usum_per_sm;            // resident blocks per SM of the field-sum kernel
    // the pointwise pass runs in p0_chunks slabs of p0_nj complex rows (2 p0_nj
    // z values) with nb_p0 blocks each, so that the host entry point can copy
    // slab c + 1 while slab c is processed (nb_point = p0_chunks * nb_p0)
    int p0_chunks, p0_nj, nb_p0;
    unsigned p0_mnj;            // ceil(2^32 / p0_nj) (multiply-high division)
    cudaStream_t s_copy;        // copy stream of the host entry point
    cudaEvent_t ev_in;          // orders the copy stream after the caller's stream
    cudaEvent_t ev_slab[4];     // slab c of the inputs is on the device
    cudaStream_t s_side;        // the energy reduction beside the inverse transforms
    cudaEvent_t ev_fork, ev_join;
    // negative or non-finite densities of the last call: [0] the number of
    // entries, then one count per block of its pointwise kernel
    unsigned* d_bad;
    int bad_cap;                // entries d_bad has room for
    float* d_gg;                // [N] g of w = g grad n (assembly -> w plane transforms)
    // give-up flags of the bounded waits, in mapped page-locked host memory so
    // that an entry point can read them without synchronising: [1] the
    // tensor-core waits of the learned path ([0] unused)
    int* h_flags;               // host view
    int* d_flags;               // device view of the same two words
    int wait_seen;              // a give-up was reported since vdw_plan
    double* d_xc;               // [4 + 2 XC_BLOCKS] nonlocal E and semilocal partial sums
    // buffers of the host-pointer entry point (allocated on first use)
    float* d_in;                // [4N]
    float* d_v;                 // [N]
    double* d_E;                // [3]
    float* d_gtmp;              // [3N] spectral gradient when the caller passes none
    size_t bytes;
    // learned reduced basis (vdw_learned_load)
    int lrn_loaded;
    int lrn_J;
    double lrn_kmax;
    void* d_lrn;                // one allocation behind the LearnedArgs pointers
    vdw::LearnedArgs la;
    float* d_U;                 // [M][N] real-space u_m for the parameter gradient (on first use)
    float* d_lw;                // [2M + 2][N] per-point coefficients of the learned assembly (on first use)
    double* d_gK;               // [P][J] knot-gradient accumulator (on first use)
    float4* d_lrn_tab;          // the tabulated network (vdw_learned_tabulate)
    size_t lrn_tab_bytes;
    // per-stage timing (vdw_profile_enable)
    int prof;
    cudaEvent_t ev[VDW_NSTAGES + 1];
    int ev_done[VDW_NSTAGES];
};

namespace vdw {

void set_error(const std::string& s);
int cuda_fail(cudaError_t e, const char* what);
// VDW_ERR_TIMEOUT (and clears the flags) if a kernel of an earlier call gave up
// a bounded wait since the last check, else VDW_OK
int check_wait(vdw_ctx* c);
// per-density workspaces for Bmax densities (api.cu)
int alloc_density_work(vdw_ctx* c, int Bmax);

// Programmatic dependent launch: a kernel started by launch() may begin while
// the kernel before it in the stream still runs its last blocks.  Such a
// kernel calls pdl_wait() before it touches anything that earlier work of the
// stream reads or writes (the wait ends when all of that work is complete and
// visible); ahead of it only tables that live as long as the plan are read
// (twiddles, the spline mesh, |G| order).  pdl_wait() also lets the kernel
// after it start in the same way.
__device__ __forceinline__ void pdl_wait() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
// Asks for bytes of global memory (16-byte aligned, a multiple of 16 bytes) to
// be brought into L2: one thread of a block does it for the block that will
// take its place on the SM, whose first loads then miss L1 only.
__device__ __forceinline__ void prefetch_l2(const void* p, unsigned bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(__cvta_generic_to_global(p)), "r"(bytes) : "memory");
}
// early: small grids only (early_launch), where launch latency and the first
// loads are a good part of a kernel; the blocks that wait take shared memory
// and L1 from the running kernel, which costs a large grid more (24^3 74 -> 53
// us a call, 100^3 497 -> 456; 256 x 256 x 96 2697 -> 2733, so not there).
template <class... K, class... A>
inline void launch(bool early, void (*kernel)(K...), dim3 grid, int block, size_t smem, cudaStream_t s, A&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = early ? 1 : 0;
    cudaLaunchKernelEx(&cfg, kernel, static_cast<K>(args)...);
}

#define VDW_CUDA(call)                                         \
    do {                                                       \
        cudaError_t _e = (call);                               \
        if (_e != cudaSuccess) return ::vdw::cuda_fail(_e, #call); \
    } while (0)

// Serialises raise_smem_limit across threads (api.cu).
void smem_limit_lock(bool lock);

// Raises (never lowers) a kernel's dynamic shared-memory limit to bytes.
// The limit belongs to the kernel, for the whole process, not to a context:
// contexts of different grids (or learned models of different knot counts)
// that share a kernel would otherwise lower each other's limit, and their
// launches would then fail.
template <class K>
int raise_smem_limit(K kernel, size_t bytes) {
    smem_limit_lock(true);
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, kernel);
    if (e == cudaSuccess && (size_t)fa.maxDynamicSharedSizeBytes < bytes)
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    smem_limit_lock(false);
    if (e != cudaSuccess) return cuda_fail(e, "raise_smem_limit");
    return VDW_OK;
}

// Sets a kernel's dynamic shared-memory limit and checks that the block size
// it will be launched with fits its register use.
template <class K>
int set_and_check(K kernel, const char* name, int smem, int threads) {
    if (const int rs = raise_smem_limit(kernel, (size_t)smem)) return rs;
    cudaFuncAttributes fa;
    VDW_CUDA(cudaFuncGetAttributes(&fa, kernel));
    if (fa.maxThreadsPerBlock < threads) {
        set_error(std::string(name) + ": " + std::to_string(threads) + " threads requested, " +
                  std::to_string(fa.maxThreadsPerBlock) + " possible with " + std::to_string(fa.numRegs) +
                  " registers");
        return VDW_ERR_UNSUPPORTED;
    }
    return VDW_OK;
}

inline bool early_launch(const GridArgs& g, int B) { return g.N * B <= (1LL << 21); }

// pipeline launchers (pipeline.cu)
// slab_ready (optional): per slab of the pointwise pass, an event to wait on
// before processing it (the host entry point's copies)
// B > 1: a batch of B densities (n [B][N], grad [B][3][N], E [B][3], v [B][N],
// w [B][3][N]), one launch per stage; needs the batch workspaces of vdw_plan_batch
// gs: gradient outputs (v_loc, w) times gE[0] dOmega, and E is E_c^nl alone
struct GradScale {
    bool on = false;
    const double* gE = nullptr;
};
int pipeline_run(vdw_ctx* c, const float* n, const float* grad, double* E, float* v, float* w,
                 cudaStream_t s, int fd = 0, int xc = 0, const cudaEvent_t* slab_ready = nullptr, int B = 1,
                 GradScale gs = {});
// E[4] of the functional from the nonlocal energy (d_xc[0]) and the semilocal sums
int pipeline_xc_final(vdw_ctx* c, double* E, cudaStream_t s);
// central-difference gradient of a field (into grad [3][N])
int pipeline_stencil_gradient(vdw_ctx* c, const float* f, float* grad, cudaStream_t s);
int pipeline_plan_check(vdw_ctx* c);
// shared memory and block size of a plane kernel on nblocks planes, forward or
// inverse, with hi/lo (exact) or FP32 twiddles
size_t smem_plane(const GridArgs& g, bool inverse, bool exact);
int plane_block(const vdw_ctx* c, long long nblocks, bool inverse, bool exact);
int pipeline_make_twiddles(vdw_ctx* c);
int pipeline_configure(vdw_ctx* c);
// the divergence term of a potential (w(G) in d_wspec) and the energy reduction
int pipeline_divergence(vdw_ctx* c, float* v, cudaStream_t s);
// in-place plane transforms of the first nfields fields of d_spec: inverse
// (half spectrum -> packed real rows) or forward (packed real rows -> half
// spectrum)
int planes_inplace(vdw_ctx* c, int nfields, bool inverse, cudaStream_t s, int B = 1);
int planes_configure(vdw_ctx* c);
// forward plane transforms of w = g grad n with g in d_gg (into d_wspec)
int pipeline_w_planes(vdw_ctx* c, const float* grad, cudaStream_t s);
int pipeline_energy_final(vdw_ctx* c, const double* epart, int nb0, int nb2, double* E, cudaStream_t s);

// y transforms and contraction in |G| order (contract.cu)
size_t sorted_pencil_smem(const GridArgs& g);
int sorted_plan(vdw_ctx* c);
void sorted_free(vdw_ctx* c);
int sorted_configure(vdw_ctx* c);
int sorted_forward(vdw_ctx* c, int nfields, cudaStream_t s, int B = 1);
int sorted_inverse(vdw_ctx* c, int nfields, cudaStream_t s, int B = 1);
int sorted_contract(vdw_ctx* c, double* epart, int write_back, cudaStream_t s, int B = 1);
// the same contraction of the first nq fields with another table of the same
// layout ([nk-1][nq(nq+1)/2] float4 cubic coefficients on a uniform mesh)
int sorted_contract_table(vdw_ctx* c, int nq, const float4* table, float inv_dk, int nk, double* epart,
                          int write_back, cudaStream_t s, int B = 1);
constexpr int SORTED_BLOCK = 128;  // sorted points per contraction block
// The energy's partial sums (one per block of the pointwise pass and of the
// contraction) are reduced by EPART_SPLIT blocks that each sum a fixed
// contiguous share of both arrays; the block that finishes last sums their
// EPART_SPLIT results in index order.  The per-density partial-sum array ends
// with those 2 EPART_SPLIT values.
constexpr int EPART_SPLIT = 64;

// learned reduced basis (learned.cu)
int learned_run(vdw_ctx* c, const float* n, const float* grad, double* E, float* v, float* w, cudaStream_t s);
void learned_free(vdw_ctx* c);

// table launchers (table.cu)
int table_build(const vdw_params* p, double* h_qmesh, double* h_phik, double* phi0, double* C_s);
int table_upload(vdw_ctx* c, const double* h_phik, double C_s);

// The inverse x transforms merge the two half spectra of a row in their first
// group's registers when it has at most this many points, with compile-time
// and with run-time groups (above 9 points the run-time kernels spill), so the
// smaller group goes first (us inverse planes: 180 x 180 x 72 106 -> 94, 128^3
// 104 -> 98, 100^3 65 -> 55); not where the rows then need a pad after every
// run (16 points) that they do not need otherwise (144: 514 against 520).
constexpr int MERGE_CT = 12, MERGE_RT = 9;
__host__ __device__ constexpr bool merge_swaps(int P1, int P2, int most) {
    return P1 > P2 && P2 > 1 && P2 <= most && !(P1 % 16 == 0 && P2 % 2 == 1);
}
// Groups of a line length ({2,3,5}-smooth, 4 <= n <= 256); sized: the
// compile-time schedule of the grids that have one.
int make_line_plan(int n, bool sized, LinePlan* lp);
// grids with compile-time line lengths
inline bool sized_grid(int n1, int n2, int n3) {
    return (n1 == 180 && n2 == 180 && n3 == 72) || (n1 == 256 && n2 == 256 && n3 == 96);
}
// offsets of the twiddle tables in d_tw (entries)
inline int tw_off_y(const GridArgs& g) { return g.N1; }
inline int tw_off_swap(const GridArgs& g) { return g.N1 + g.N2 + g.N3; }
__host__ __device__ inline int tw_off_xi(const GridArgs& g) { return g.N1 + 2 * g.N2 + g.N3; }

}  // namespace vdw
