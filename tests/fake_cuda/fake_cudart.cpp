// A stand-in for the CUDA runtime, linked with the library's own objects by
// the CPU tests: device memory is host memory, no kernel runs, and every launch
// is recorded with its grid, cluster, stream and device.  Function attributes
// belong to a (function, device) pair, as in the runtime: a launch or an
// occupancy query that needs an attribute which its device's copy of the
// function was not given fails with an error.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <set>
#include <string>
#include <utility>
#include <vector>

namespace {

constexpr int kDevices = 2, kSms = 152, kMaxSmem = 232448, kDefaultSmem = 48 << 10;
// clusters of 1..16 such CTAs (one per SM) that a GB300 holds at once
constexpr int kClustersBySize[17] = {0, 152, 76, 46, 36, 28, 23, 15, 15, 7, 7, 7, 7, 7, 7, 7, 7};

struct Launch {
    std::string name;
    unsigned grid[3], block, cluster;
    unsigned long long smem, stream;
    int pdl, device;
};

std::mutex mu;
// the kernels register from static constructors that may run before this file's
std::map<const void *, std::string> &names()
{
    static std::map<const void *, std::string> m;
    return m;
}
std::set<std::pair<const void *, int>> large_smem, large_cluster;  // (function, device)
std::vector<Launch> launches;
std::string text;
thread_local int device = 0;
int cluster_limit[kDevices] = {kSms, kSms};  // clusters of any size that a device holds at once
unsigned long long next_handle = 0x1000;

cudaError_t check(const cudaLaunchConfig_t *cfg, const void *fn, unsigned *cluster, int *pdl)
{
    *cluster = 1;
    *pdl = 0;
    for (unsigned i = 0; i < cfg->numAttrs; ++i) {
        if (cfg->attrs[i].id == cudaLaunchAttributeClusterDimension)
            *cluster = cfg->attrs[i].val.clusterDim.x;
        if (cfg->attrs[i].id == cudaLaunchAttributeProgrammaticStreamSerialization)
            *pdl = cfg->attrs[i].val.programmaticStreamSerializationAllowed;
    }
    if (*cluster < 1 || *cluster > 16 || cfg->gridDim.x % *cluster)
        return cudaErrorInvalidConfiguration;
    if (*cluster > 8 && !large_cluster.count({fn, device}))
        return cudaErrorInvalidClusterSize;
    if (cfg->dynamicSmemBytes > kMaxSmem || (cfg->dynamicSmemBytes > kDefaultSmem && !large_smem.count({fn, device})))
        return cudaErrorInvalidValue;
    return cudaSuccess;
}

CUresult encode(CUtensorMap *map, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                CUtensorMapL2promotion, CUtensorMapFloatOOBfill)
{
    memset(map, 0, sizeof *map);
    return CUDA_SUCCESS;
}

}  // namespace

extern "C" {

// the launches since the last call: "name grid_x grid_y grid_z block cluster smem stream pdl device" a line
const char *fake_launches()
{
    std::lock_guard<std::mutex> lk(mu);
    text.clear();
    for (const Launch &l : launches) {
        text += l.name;
        for (unsigned long long x : {(unsigned long long)l.grid[0], (unsigned long long)l.grid[1],
                                     (unsigned long long)l.grid[2], (unsigned long long)l.block,
                                     (unsigned long long)l.cluster, l.smem, l.stream, (unsigned long long)l.pdl,
                                     (unsigned long long)l.device})
            text += " " + std::to_string(x);
        text += "\n";
    }
    launches.clear();
    return text.c_str();
}

// makes a device the calling thread's current one
void fake_set_device(int d)
{
    device = d;
}

// limits the clusters that a device holds at once
void fake_limit_clusters(int d, int n)
{
    cluster_limit[d] = n;
}

void **__cudaRegisterFatBinary(void *)
{
    static void *handle;
    return &handle;
}
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *fn, char *, const char *name, int, void *, void *, void *, void *,
                            int *)
{
    names()[fn] = name;
}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, void *)
{
    return 1;
}
cudaError_t __cudaPopCallConfiguration(dim3 *, dim3 *, size_t *, void *)
{
    return cudaErrorNotSupported;
}
cudaError_t __cudaGetKernel(cudaKernel_t *, const void *)
{
    return cudaErrorNotSupported;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void **, size_t, cudaStream_t)
{
    return cudaErrorNotSupported;  // the library launches through cudaLaunchKernelEx only
}

cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *cfg, const void *fn, void **)
{
    std::lock_guard<std::mutex> lk(mu);
    Launch l;
    const cudaError_t e = check(cfg, fn, &l.cluster, &l.pdl);
    if (e != cudaSuccess)
        return e;
    l.name = names().count(fn) ? names()[fn] : "?";
    l.grid[0] = cfg->gridDim.x, l.grid[1] = cfg->gridDim.y, l.grid[2] = cfg->gridDim.z;
    l.block = cfg->blockDim.x;
    l.smem = cfg->dynamicSmemBytes;
    l.stream = (unsigned long long)cfg->stream;
    l.device = device;
    launches.push_back(l);
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *fn, const cudaLaunchConfig_t *cfg)
{
    std::lock_guard<std::mutex> lk(mu);
    unsigned cluster;
    int pdl;
    const cudaError_t e = check(cfg, fn, &cluster, &pdl);
    if (e == cudaSuccess)
        *n = std::min(kClustersBySize[cluster], cluster_limit[device]);
    return e;
}
cudaError_t cudaFuncSetAttribute(const void *fn, cudaFuncAttribute attr, int value)
{
    std::lock_guard<std::mutex> lk(mu);
    if (attr == cudaFuncAttributeMaxDynamicSharedMemorySize && value > kDefaultSmem)
        large_smem.insert({fn, device});
    if (attr == cudaFuncAttributeNonPortableClusterSizeAllowed && value)
        large_cluster.insert({fn, device});
    return cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes *a, const void *)
{
    memset(a, 0, sizeof *a);
    return cudaSuccess;
}
cudaError_t cudaGetLastError()
{
    return cudaSuccess;
}
const char *cudaGetErrorString(cudaError_t e)
{
    static thread_local char s[32];
    snprintf(s, sizeof s, "cudaError %d", (int)e);
    return s;
}
cudaError_t cudaGetDeviceCount(int *n)
{
    *n = kDevices;
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int *d)
{
    *d = device;
    return cudaSuccess;
}
cudaError_t cudaSetDevice(int d)
{
    if (d < 0 || d >= kDevices)
        return cudaErrorInvalidDevice;
    device = d;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr attr, int)
{
    *v = attr == cudaDevAttrMultiProcessorCount ? kSms : attr == cudaDevAttrMaxSharedMemoryPerBlockOptin ? kMaxSmem : 0;
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize()
{
    return cudaSuccess;
}
cudaError_t cudaMalloc(void **p, size_t n)
{
    *p = malloc(n);
    return *p ? cudaSuccess : cudaErrorMemoryAllocation;
}
cudaError_t cudaFree(void *p)
{
    free(p);
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind)
{
    memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *, int, size_t, cudaStream_t)
{
    return cudaSuccess;
}
cudaError_t cudaMemcpyFromSymbolAsync(void *, const void *, size_t, size_t, cudaMemcpyKind, cudaStream_t)
{
    return cudaErrorNotSupported;
}
cudaError_t cudaGetSymbolAddress(void **, const void *)
{
    return cudaErrorNotSupported;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned)
{
    std::lock_guard<std::mutex> lk(mu);
    *s = (cudaStream_t)(next_handle += 0x10);
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t)
{
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t)
{
    return cudaSuccess;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *st)
{
    *st = cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned)
{
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned)
{
    std::lock_guard<std::mutex> lk(mu);
    *e = (cudaEvent_t)(next_handle += 0x10);
    return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t)
{
    return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t)
{
    return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char *, void **fn, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult *q)
{
    *fn = reinterpret_cast<void *>(encode);
    *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}

}  // extern "C"
