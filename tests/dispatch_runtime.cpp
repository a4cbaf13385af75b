// Stand-in for the CUDA runtime without a GPU, for tests/test_dispatch_host.py:
// device memory is host memory that is never used again after it is freed, so
// that a launch that reads freed scratch can be told (held).
#include <cuda_runtime_api.h>

#include <cstdlib>
#include <cstring>
#include <string>
#include <vector>

namespace {

struct Block {
    char *p;
    size_t bytes;
    bool live;
};
std::vector<Block> blocks;
std::string journal;  // one word per launch; '!' marks a read outside live memory

}  // namespace

// [p, p + bytes) is the caller's, or wholly inside one allocation still held
bool held(const void *p, size_t bytes)
{
    const char *a = (const char *)p;
    for (const Block &b : blocks)
        if (a >= b.p && a < b.p + b.bytes) return b.live && a + bytes <= b.p + b.bytes;
    return true;
}

void note(const char *name, bool ok)
{
    journal += name;
    journal += ok ? " " : "! ";
}

extern "C" {

const char *dispatch_journal()
{
    static std::string out;
    out = journal;
    journal.clear();
    return out.c_str();
}

cudaError_t cudaMalloc(void **p, size_t bytes)
{
    *p = std::calloc(1, bytes);
    if (!*p) return cudaErrorMemoryAllocation;
    blocks.push_back({(char *)*p, bytes, true});
    return cudaSuccess;
}
cudaError_t cudaFree(void *p)
{
    for (Block &b : blocks)
        if (b.p == p) b.live = false;
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void **p, size_t bytes, unsigned)
{
    *p = std::calloc(1, bytes);
    return cudaSuccess;
}
cudaError_t cudaFreeHost(void *) { return cudaSuccess; }
cudaError_t cudaHostGetDevicePointer(void **d, void *h, unsigned)
{
    *d = h;
    return cudaSuccess;
}
// every host buffer is page-locked and mapped
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *p)
{
    a->type = cudaMemoryTypeHost;
    a->devicePointer = const_cast<void *>(p);
    return cudaSuccess;
}
cudaError_t cudaMemset(void *p, int v, size_t n)
{
    std::memset(p, v, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t) { return cudaMemset(p, v, n); }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t)
{
    std::memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int)
{
    *v = 152;
    return cudaSuccess;
}
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *) { return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *, cudaEvent_t, cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *, const void *, void **)
{
    return cudaSuccess;  // the kernel that publishes the status word
}

}  // extern "C"
