// What launch_host.cu calls of the CUDA runtime.  Function attributes are a device's, as in the real one: the last limit set
// holds for every caller.  An error stays pending until cudaGetLastError takes it.
#include <cuda_runtime_api.h>
#include <map>
#include "launch_host.h"

namespace fake {

std::set<int> refuse;
int launches = 0;
unsigned cluster = 1, grid_x = 0, grid_y = 0;
static cudaError_t pending = cudaSuccess;
static std::map<const void *, size_t> smem_limit;

static cudaError_t fail(cudaError_t e) { return pending = e; }
static cudaError_t launch(const void *f, size_t smem)
{
    const size_t limit = smem_limit.count(f) ? smem_limit[f] : 48 * 1024;
    if (refuse.count(launches++) || smem > limit) return fail(cudaErrorInvalidValue);
    return cudaSuccess;
}

}  // namespace fake

extern "C" {

cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **)
{
    fake::cluster = 1;
    fake::grid_x = c->gridDim.x;
    fake::grid_y = c->gridDim.y;
    for (unsigned k = 0; k < c->numAttrs; ++k)
        if (c->attrs[k].id == cudaLaunchAttributeClusterDimension) fake::cluster = c->attrs[k].val.clusterDim.x;
    return fake::launch(f, c->dynamicSmemBytes);
}
cudaError_t cudaLaunchKernel(const void *f, dim3, dim3, void **, size_t smem, cudaStream_t) { return fake::launch(f, smem); }
cudaError_t cudaFuncSetAttribute(const void *f, cudaFuncAttribute a, int v)
{
    if (a != cudaFuncAttributeMaxDynamicSharedMemorySize) return cudaSuccess;
    if (v > 227 * 1024) return fake::fail(cudaErrorInvalidValue);
    fake::smem_limit[f] = (size_t)v;
    return cudaSuccess;
}
cudaError_t cudaGetLastError(void)
{
    const cudaError_t e = fake::pending;
    fake::pending = cudaSuccess;
    return e;
}
cudaError_t cudaMemsetAsync(void *, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }

// what compiled kernels announce themselves with
void **__cudaRegisterFatBinary(void *)
{
    static void *handle;
    return &handle;
}
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, uint3 *, uint3 *, dim3 *, dim3 *, int *) {}
static size_t pushed_smem;
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t smem, struct CUstream_st *) { return pushed_smem = smem, 0; }
cudaError_t __cudaPopCallConfiguration(dim3 *grid, dim3 *block, size_t *smem, void *stream)
{
    *grid = *block = dim3(1);
    *smem = pushed_smem;
    *static_cast<cudaStream_t *>(stream) = nullptr;
    return cudaSuccess;
}
}
