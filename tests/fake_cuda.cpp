// A CUDA runtime of two devices on the host, under the library's host code (api.cu,
// step64.cu), for tests of who allocates and frees what, and on which device.
#include <cuda_runtime.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <map>
#include <string>
#include <vector>

#include "ds.h"
#include "ds_internal.h"
#include "step64.h"

static int g_current = 0, g_syncs[2];
static bool g_pool_full = false;           // the pool keeps what cudaMalloc would need
static std::map<void *, int> g_owner;      // allocations and their devices
static std::vector<std::string> g_faults;
static cudaError_t take(void **p, size_t bytes)
{
    *p = malloc(bytes ? bytes : 1);
    g_owner[*p] = g_current;
    return cudaSuccess;
}
static void give_back(void *p)
{
    if (!g_owner.erase(p)) g_faults.push_back("freed twice, or never allocated");
    free(p);
}
extern "C" {
cudaError_t cudaGetDevice(int *d) { *d = g_current; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { g_current = d; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int) { *v = a == cudaDevAttrComputeCapabilityMajor ? 10 : 3; return cudaSuccess; }
cudaError_t cudaMalloc(void **p, size_t b)
{
    *p = nullptr;
    return g_pool_full ? cudaErrorMemoryAllocation : take(p, b);
}
cudaError_t cudaMallocAsync(void **p, size_t b, cudaStream_t) { return take(p, b); }
cudaError_t cudaMallocFromPoolAsync(void **p, size_t b, cudaMemPool_t, cudaStream_t) { return take(p, b); }
cudaError_t cudaMemPoolCreate(cudaMemPool_t *p, const cudaMemPoolProps *) { *p = (cudaMemPool_t)1; return cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void *) { return cudaSuccess; }
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t, size_t) { g_pool_full = false; return cudaSuccess; }
// finds the device itself and waits for it
cudaError_t cudaFree(void *p) { if (p) give_back(p); return cudaSuccess; }
// orders itself on a stream of the current device
cudaError_t cudaFreeAsync(void *p, cudaStream_t)
{
    if (g_owner.count(p) && (g_owner[p] != g_current || !g_syncs[g_owner[p]])) g_faults.push_back("freed without waiting for its device");
    give_back(p);
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() { ++g_syncs[g_current]; return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return "error"; }
void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
}
namespace ds {
ds_status phi_batch_f64(int, const std::vector<PhiJob> &, cudaStream_t) { return DS_OK; }
ds_status phi_batch_cplx(int, const std::vector<PhiJobC> &, cudaStream_t) { return DS_OK; }
void launch_fold_cplx(int64_t, const double *, const double *, double, double, double *, double *, cudaStream_t) {}
namespace mm {
View tensor_view(int, const int64_t *n, int mu, const double *X)
{
    View v{};
    v.src[0] = X;
    v.scale[0] = 1.0;
    v.ncat = v.batch = 1;
    v.n = (int)n[mu];
    v.I = 1;
    v.rows = n[1 - mu];
    return v;
}
View matrix_view(int64_t n, const double *L, int, double scale)
{
    View v = tensor_view(2, &n, 0, L);
    v.scale[0] = scale;
    v.rows = n;
    return v;
}
bool use_digits(int64_t, int, int) { return true; }
int tile_cols(int64_t, int, int, int) { return 16; }
size_t scratch_bytes(int64_t, int64_t, int, int, bool) { return 4096; }
long long wait_limit_default() { return 1; }
void launch_split(const View *, const Image *, int, int *, cudaStream_t) {}
int run_products(const Context &, const Product *, int, cudaStream_t) { return 0; }
}
}

// the workspaces of a plan's sums where the pool has to give way first
static void scarce()
{
    {
        ds_phi_set set{};
        set.d = 2;
        set.n[0] = set.n[1] = 32;
        set.k = 1;
        set.tridiag[0] = set.tridiag[1] = true;
        static double P[1];
        set.P_dev = P;
        ds::Sums64 e;
        void *p = nullptr;
        ds::pool_alloc(&p, 16, nullptr);   // (makes the pool)
        cudaFree(p);
        g_pool_full = true;
        ds::sums_create(e, &set, 1024, {{ds::SumKind::plain, {0}}}, nullptr, 8, nullptr);
        if (!e.ctx.ws) g_faults.push_back("no scratch while the pool keeps memory");
        if (!e.mats || e.images.empty()) g_faults.push_back("no matrix images");
        ds::sums_destroy(e);
    }
}

int main(int argc, char **argv)
{
    if (argc > 1 && !strcmp(argv[1], "scarce")) {
        scarce();
        for (const std::string &f : g_faults) puts(f.c_str());
        return g_faults.empty() ? 0 : 1;
    }
    const ds_grid grid = {2, {5, 4, 0, 0}};
    std::vector<double> A(2 * (25 + 16), 0.5);
    for (int scheme : {DS_EXPRK3DS_REAL, DS_ETD2RKDS, DS_EXPRK3DS_CPLX}) {
        ds_phi_set *set = nullptr;
        cudaSetDevice(0);
        if (ds_phi_setup_ex(&grid, A.data(), 0, 1e-3, scheme, &set, nullptr) != DS_OK) g_faults.push_back(ds_last_error());
        cudaSetDevice(1);
        ds_phi_set_destroy(set);
        int now = -1;
        cudaGetDevice(&now);
        if (now != 1) g_faults.push_back("the caller's device changed");
        if (!g_owner.empty()) g_faults.push_back("memory left behind");
        if (g_syncs[1]) g_faults.push_back("waited for a device that does not hold the set");
    }
    for (const std::string &f : g_faults) puts(f.c_str());
    return g_faults.empty() ? 0 : 1;
}
