// The library's host code on a machine without a GPU: the objects of the build
// linked against this stand-in for the CUDA runtime, which allocates host
// memory, runs no kernel and checks what each launch is given.
//
//   fake_cuda planes NQ   every call of planes that are small enough for many
//                         to share an SM, up to 32 densities per call
//   fake_cuda batch       a call on the caller's stream right after vdw_plan_batch
//   fake_cuda learned     the learned path's calls right after vdw_learned_load
//
// Exits 1 with a line per fault.
#include <cuda_runtime_api.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

#include "../include/vdwnl.h"

static std::map<const void*, std::string> g_names;
static std::string g_case;
static int g_faults = 0, g_launches = 0;
static bool g_pending = false;  // a memset was queued on the default stream and nothing waited for it

static void fault(const std::string& what) {
    if (++g_faults <= 20) std::printf("%s: %s\n", g_case.c_str(), what.c_str());
}
static cudaError_t launched(const void* f, dim3 grid, dim3 block, size_t smem, cudaStream_t s) {
    ++g_launches;
    if (g_pending && s) fault(g_names[f] + " does not wait for a memset on the default stream");
    const unsigned t = block.x * block.y * block.z;
    if (t < 1 || t > 1024 || grid.x < 1 || grid.y < 1 || grid.z < 1 || grid.y > 65535 || grid.z > 65535 ||
        smem > 227 * 1024)
        fault(g_names[f] + ": grid " + std::to_string(grid.x) + " " + std::to_string(grid.y) + " " +
              std::to_string(grid.z) + ", " + std::to_string(t) + " threads, " + std::to_string(smem) + " bytes");
    return cudaSuccess;
}

extern "C" {
// what the compiler's host stubs call
static dim3 g_grid, g_block;
static size_t g_smem;
static cudaStream_t g_stream;
void** __cudaRegisterFatBinary(void*) { return reinterpret_cast<void**>(&g_grid); }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
    g_names[host] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, cudaStream_t s) {
    g_grid = grid;
    g_block = block;
    g_smem = smem;
    g_stream = s;
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* s) {
    *grid = g_grid;
    *block = g_block;
    *smem = g_smem;
    *static_cast<cudaStream_t*>(s) = g_stream;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
    *k = (cudaKernel_t)f;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3 block, void**, size_t smem, cudaStream_t s) {
    return launched((const void*)k, grid, block, smem, s);
}
// the runtime
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) {
    return launched(f, c->gridDim, c->blockDim, c->dynamicSmemBytes, c->stream);
}
cudaError_t cudaMalloc(void** p, size_t n) {
    *p = std::malloc(n ? n : 1);
    return *p ? cudaSuccess : cudaErrorMemoryAllocation;
}
cudaError_t cudaFree(void* p) {
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) {
    *p = std::calloc(n, 1);
    return cudaSuccess;
}
cudaError_t cudaFreeHost(void* p) { return cudaFree(p); }
cudaError_t cudaHostGetDevicePointer(void** d, void* h, unsigned) {
    *d = h;
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) {
    std::memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void*, const void*, size_t, cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemset(void*, int, size_t) {
    g_pending = true;
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t s) {
    g_pending = g_pending || !s;
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() {
    g_pending = false;
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
    g_pending = g_pending && s;
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) {
    *d = 0;
    return cudaSuccess;
}
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : 0;
    return cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes* a, const void*) {
    std::memset(a, 0, sizeof(*a));
    a->maxThreadsPerBlock = 1024;
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
    *n = 4;
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) {
    *e = (cudaEvent_t)&g_grid;
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* t, cudaEvent_t, cudaEvent_t) {
    *t = 0.f;
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
    *s = (cudaStream_t)&g_block;
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaGetSymbolAddress(void** p, const void* s) {
    *p = const_cast<void*>(s);
    return cudaSuccess;
}
}

static void ok(int rc, const char* what) {
    if (rc) fault(std::string(what) + " returns " + std::to_string(rc) + " (" + vdw_last_error() + ")");
}
static vdw_handle context(int Nq) {
    vdw_params p;
    vdw_params_default(&p);
    p.Nq = Nq;
    p.Nk = 64;
    const std::vector<double> phi((size_t)Nq * Nq * p.Nk, 0.0);
    vdw_handle h = nullptr;
    ok(vdw_create(&h, &p, phi.data(), 1.0), "vdw_create");
    return h;
}
// the caller's stream (not the default one) and device arrays, never touched
static void* const STREAM = &g_stream;
static float g_buf[1];

static bool smooth(int n) {
    for (int r : {2, 3, 5})
        while (n % r == 0) n /= r;
    return n == 1;
}

static void planes(int Nq) {
    vdw_handle h = context(Nq);
    double E[1];
    for (int n1 = 4; n1 <= 256; n1 += 2)
        for (int n3 = 4; n3 <= 256; n3 += 2)
            for (int n2 : {4, 25, 96, 256}) {
                if (!smooth(n1) || !smooth(n3) || n1 * n3 > 2400) continue;
                const double L[3] = {0.5 * n1, 0.5 * n2, 0.5 * n3};
                g_case = std::to_string(n1) + " x " + std::to_string(n2) + " x " + std::to_string(n3);
                std::fflush(stdout);
                ok(vdw_plan(h, n1, n2, n3, L), "vdw_plan");
                ok(vdw_energy_potential(h, g_buf, nullptr, E, g_buf, nullptr, STREAM), "vdw_energy_potential");
                ok(vdw_energy_gradients(h, g_buf, g_buf, E, E, g_buf, g_buf, STREAM), "vdw_energy_gradients");
                ok(vdw_plan_batch(h, 32), "vdw_plan_batch");
                for (int B : {2, 3, 5, 8, 11, 16, 23, 32}) {
                    g_case += " B " + std::to_string(B);
                    ok(vdw_energy_potential_batched(h, B, g_buf, g_buf, E, g_buf, STREAM), "batched");
                    g_case.resize(g_case.rfind(" B "));
                }
            }
    vdw_destroy(h);
}

static void batch() {
    vdw_handle h = context(8);
    const double L[3] = {6.0, 6.0, 6.0};
    double E[1];
    ok(vdw_plan(h, 12, 12, 12, L), "vdw_plan");
    g_case = "after vdw_plan";
    ok(vdw_energy_potential(h, g_buf, g_buf, E, g_buf, nullptr, STREAM), "vdw_energy_potential");
    ok(vdw_plan_batch(h, 3), "vdw_plan_batch");
    g_case = "after vdw_plan_batch";
    ok(vdw_energy_potential_batched(h, 3, g_buf, g_buf, E, g_buf, STREAM), "batched");
    vdw_destroy(h);
}

static void learned() {
    vdw_handle h = context(8);
    const double L[3] = {6.0, 6.0, 6.0}, feat[5] = {0.0, 1.0, 0.0, 1.0, 1e-3};
    double E[1];
    ok(vdw_plan(h, 12, 12, 12, L), "vdw_plan");
    for (int J : {16, 16, 32}) {
        g_case = "J " + std::to_string(J);
        ok(vdw_learned_load(h, J, 40.0, feat, 0.1, 1.4, g_buf, STREAM), "vdw_learned_load");
        ok(vdw_learned_param_grad(h, g_buf, g_buf, 1.0, E, E, STREAM), "vdw_learned_param_grad");
        ok(vdw_learned_fit_grad(h, g_buf, g_buf, g_buf, g_buf, 1.0, E, STREAM), "vdw_learned_fit_grad");
        ok(vdw_learned_energy_potential(h, g_buf, g_buf, E, g_buf, nullptr, STREAM), "vdw_learned_energy_potential");
        ok(vdw_learned_tabulate(h, 16, 4.0, STREAM), "vdw_learned_tabulate");
        ok(vdw_learned_energy_potential(h, g_buf, g_buf, E, g_buf, nullptr, STREAM), "vdw_learned_energy_potential");
    }
    vdw_destroy(h);
}

int main(int argc, char** argv) {
    const std::string what = argc > 1 ? argv[1] : "";
    if (what == "planes") planes(std::atoi(argv[2]));
    else if (what == "batch") batch();
    else if (what == "learned") learned();
    else return 2;
    std::printf("%d launches, %d faults\n", g_launches, g_faults);
    return g_faults ? 1 : 0;
}
