// A CUDA runtime of two devices on the host, under the library's host code (api.cu), for
// tests of who allocates and frees what, and on which device.
#include <cuda_runtime.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <map>
#include <string>
#include <vector>

#include "ds.h"
#include "ds_internal.h"

static int g_current = 0, g_syncs[2];
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
cudaError_t cudaMalloc(void **p, size_t b) { return take(p, b); }
cudaError_t cudaMallocAsync(void **p, size_t b, cudaStream_t) { return take(p, b); }
cudaError_t cudaMallocFromPoolAsync(void **p, size_t b, cudaMemPool_t, cudaStream_t) { return take(p, b); }
cudaError_t cudaMemPoolCreate(cudaMemPool_t *p, const cudaMemPoolProps *) { *p = (cudaMemPool_t)1; return cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void *) { return cudaSuccess; }
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t, size_t) { return cudaSuccess; }
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
}

int main()
{
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
