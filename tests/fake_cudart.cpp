// A CUDA runtime without a GPU, for tests of the library's host code: linked with the library's objects in
// place of the real one.  Two devices with different SM counts; addresses are made up and nothing is
// copied or run.  What the host code can get wrong is checked as on a device: a launch with more than 48 KB of
// dynamic shared memory fails unless that kernel was opted in to as much on the current device.  Launches
// and tensor maps (each encoding, and each address set) are logged, one line each (fake_log).
#include <cuda.h>
#include <cuda_runtime_api.h>

#include <cstdio>
#include <cstring>
#include <map>
#include <string>
#include <utility>

namespace {
int g_dev = 0;
constexpr int kSms[2] = {152, 100};
std::map<const void*, std::string> g_names;
std::map<std::pair<int, const void*>, int> g_smem;
std::string g_log;
int g_fail_opt_ins = 0;
uintptr_t g_next = 1ull << 40;
thread_local struct { dim3 grid, block; size_t smem; cudaStream_t st; } g_cfg;

cudaError_t launch(const void* f, dim3 g, dim3 b, size_t smem, int cluster, int pdl) {
    auto it = g_smem.find({g_dev, f});
    if (smem > 48 * 1024 && (it == g_smem.end() || (size_t)it->second < smem)) return cudaErrorInvalidValue;
    char line[512];
    std::snprintf(line, sizeof(line), "launch %d %s %u %u %u %u %zu %d %d\n", g_dev, g_names[f].c_str(), g.x, g.y, g.z, b.x, smem,
                  cluster, pdl);
    g_log += line;
    return cudaSuccess;
}

std::map<int, std::string> g_maps;  // dimensions of an encoded map, by the number written into it

CUresult replace(CUtensorMap* m, void* base) {
    if ((uintptr_t)base & 15) return CUDA_ERROR_INVALID_VALUE;
    int id;
    std::memcpy(&id, m, sizeof(id));
    g_log += "map " + std::to_string((uintptr_t)base) + g_maps.at(id) + "\n";
    return CUDA_SUCCESS;
}

CUresult encode(CUtensorMap* m, CUtensorMapDataType, cuuint32_t rank, void* base, const cuuint64_t* dims, const cuuint64_t* strides,
                const cuuint32_t* box, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                CUtensorMapFloatOOBfill) {
    if ((uintptr_t)base & 15) return CUDA_ERROR_INVALID_VALUE;
    std::string text;
    for (cuuint32_t i = 0; i < rank; ++i) {
        if (!dims[i] || dims[i] > 1ull << 32 || !box[i] || box[i] > 256) return CUDA_ERROR_INVALID_VALUE;
        if (i && (strides[i - 1] % 16 || strides[i - 1] >= 1ull << 40)) return CUDA_ERROR_INVALID_VALUE;
        text += " " + std::to_string(dims[i]) + ":" + std::to_string(i ? strides[i - 1] : 0) + ":" + std::to_string(box[i]);
    }
    const int id = (int)g_maps.size();
    g_maps[id] = text;
    std::memcpy(m, &id, sizeof(id));
    g_log += "encode\n";
    return replace(m, base);
}
}  // namespace

extern "C" {
void fake_set_device(int d) { g_dev = d; }
void fake_fail_opt_ins(int n) { g_fail_opt_ins = n; }  // the next n opt-ins fail
const char* fake_log() { return g_log.c_str(); }
void fake_clear() { g_log.clear(); }

void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* f, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) { g_names[f] = name; }
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t s, cudaStream_t st) { g_cfg = {g, b, s, st}; return 0; }
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* s, void* st) {
    *g = g_cfg.grid; *b = g_cfg.block; *s = g_cfg.smem; *(cudaStream_t*)st = g_cfg.st;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) { *k = (cudaKernel_t)f; return cudaSuccess; }
thread_local cudaError_t g_last = cudaSuccess;
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void**, size_t s, cudaStream_t) {
    const cudaError_t e = launch((const void*)k, g, b, s, 1, 0);
    if (e != cudaSuccess) g_last = e;
    return e;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) {
    int cluster = 1, pdl = 0;
    for (unsigned i = 0; i < c->numAttrs; ++i) {
        if (c->attrs[i].id == cudaLaunchAttributeClusterDimension) cluster = c->attrs[i].val.clusterDim.x;
        if (c->attrs[i].id == cudaLaunchAttributeProgrammaticStreamSerialization) pdl = c->attrs[i].val.programmaticStreamSerializationAllowed;
    }
    return launch(f, c->gridDim, c->blockDim, c->dynamicSmemBytes, cluster, pdl);
}
cudaError_t cudaGetLastError() { const cudaError_t e = g_last; g_last = cudaSuccess; return e; }
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute, int v) {
    if (g_fail_opt_ins > 0) { --g_fail_opt_ins; return cudaErrorUnknown; }
    g_smem[{g_dev, f}] = v;
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) { *d = g_dev; return cudaSuccess; }
cudaError_t cudaGetDeviceCount(int* n) { *n = 2; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int d) { *v = a == cudaDevAttrMultiProcessorCount ? kSms[d] : 0; return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t* c) {
    for (unsigned i = 0; i < c->numAttrs; ++i)
        if (c->attrs[i].id == cudaLaunchAttributeClusterDimension) *n = kSms[g_dev] / (int)c->attrs[i].val.clusterDim.x;
    return cudaSuccess;
}
cudaError_t cudaMalloc(void** p, size_t n) { *p = (void*)g_next; g_next += (n + 255) / 256 * 256; return cudaSuccess; }
cudaError_t cudaFree(void*) { return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void*, size_t n, cudaMemcpyKind k) { if (k == cudaMemcpyDeviceToHost) std::memset(d, 0, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t) { return cudaMemcpy(d, s, n, k); }
cudaError_t cudaMemset(void*, int, size_t) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void*) { return cudaMalloc(p, 1 << 24); }
cudaError_t cudaGetDriverEntryPointByVersion(const char* name, void** f, unsigned, unsigned long long, cudaDriverEntryPointQueryResult* q) {
    *f = std::strstr(name, "Replace") ? (void*)replace : (void*)encode; *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {  // every address: page-locked, device view = itself
    std::memset(a, 0, sizeof(*a));
    a->type = cudaMemoryTypeHost; a->devicePointer = (void*)p;
    return cudaSuccess;
}
const char* cudaGetErrorName(cudaError_t) { return "fake"; }
const char* cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = (cudaStream_t)(g_next += 16); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { *g = (cudaGraph_t)(g_next += 16); return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t, unsigned long long) { *x = (cudaGraphExec_t)(g_next += 16); return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = (cudaEvent_t)(g_next += 16); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* t, cudaEvent_t, cudaEvent_t) { *t = 0; return cudaSuccess; }
}
