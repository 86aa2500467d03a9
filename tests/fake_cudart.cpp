// Stands in for the CUDA runtime under the library's host code, on a machine
// without a GPU: every call is written to a log instead of being carried out,
// and chosen ones return an error.  Nothing is launched.
#include <cuda_runtime.h>
#include <string.h>

extern "C" {

struct Entry {
    int kind;  // 1: launch, 2: memset
    void *ptr;
    size_t bytes;
    void *stream;
};
static Entry log_[4096];
static int nlog, launches, memsets;
static int fail_launch = -1, fail_memsets, capturing;

void fake_reset(int launch, int memset_failures, int capture)
{
    nlog = launches = memsets = 0;
    fail_launch = launch;
    fail_memsets = memset_failures;
    capturing = capture;
}
int fake_log(Entry *out)
{
    memcpy(out, log_, sizeof(Entry) * nlog);
    return nlog;
}
static void note(int kind, void *p, size_t n, void *s)
{
    if (nlog < 4096)
        log_[nlog++] = Entry{kind, p, n, s};
}

cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *cfg, const void *f, void **)
{
    if (launches++ == fail_launch)
        return cudaErrorLaunchOutOfResources;
    note(1, const_cast<void *>(f), 0, cfg->stream);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *p, int, size_t n, cudaStream_t s)
{
    if (memsets++ < fail_memsets)
        return cudaErrorUnknown;
    note(2, p, n, s);
    return cudaSuccess;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *st)
{
    *st = capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaGetDeviceProperties(cudaDeviceProp *p, int)
{
    memset(p, 0, sizeof *p);
    p->major = 10;
    p->minor = 3;
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *, const void *, size_t, cudaMemcpyKind, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *, const void *) { return cudaErrorNotSupported; }
cudaError_t cudaGetSymbolAddress(void **, const void *) { return cudaErrorNotSupported; }
cudaError_t cudaOccupancyMaxActiveClusters(int *, const void *, const cudaLaunchConfig_t *) { return cudaErrorNotSupported; }
cudaError_t cudaGetDriverEntryPointByVersion(const char *, void **, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult *)
{
    return cudaErrorNotSupported;
}

// what nvcc's host code calls to register and name kernels
void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, uint3 *, uint3 *, dim3 *, dim3 *, int *) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) { *k = (cudaKernel_t)f; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void **, size_t, cudaStream_t) { return cudaErrorNotSupported; }
unsigned __cudaPopCallConfiguration(dim3 *, dim3 *, size_t *, void *) { return 1; }

}  // extern "C"
