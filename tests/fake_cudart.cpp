// A CUDA runtime without a GPU, linked with the library's own objects: two
// devices, device memory from the host's heap, kernels recorded instead of run.
// It checks what the host code owes the runtime: a launch with more than 48 KB of
// dynamic shared memory needs the opt-in of that kernel on that device.
#include <cuda_runtime_api.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <utility>
#include <vector>

namespace {
int g_device = 0;
cudaError_t g_last = cudaSuccess;
std::map<const void *, std::string> g_names;                       // host function -> kernel name
std::map<std::pair<const void *, int>, int> g_limit;               // (kernel, device) -> dynamic shared memory
std::map<char *, size_t> g_mem;                                    // live device allocations
std::vector<std::pair<char *, std::vector<char>>> g_uploads;       // host-to-device copies, as written
std::vector<std::string> g_launched;
int g_lowered = 0, g_frees = 0;
struct Config {
    dim3 grid, block;
    size_t smem;
    cudaStream_t stream;
};
std::vector<Config> g_config;

cudaError_t fail(cudaError_t e) { return g_last = e; }

cudaError_t launch(const void *f, size_t smem)
{
    const auto it = g_limit.find({f, g_device});
    if (smem > 48 * 1024 && (it == g_limit.end() || smem > (size_t)it->second)) return fail(cudaErrorInvalidValue);
    g_launched.push_back(g_names[f]);
    return cudaSuccess;
}
}  // namespace

// ---- what the tests read --------------------------------------------------
extern "C" {
int fake_launches() { return (int)g_launched.size(); }
const char *fake_launched(int k) { return g_launched[k].c_str(); }
int fake_limits_lowered() { return g_lowered; }
int fake_frees() { return g_frees; }
void fake_forget_uploads() { g_uploads.clear(); }
int fake_uploads() { return (int)g_uploads.size(); }
// copies whose destination has been freed or holds something else now
int fake_uploads_lost()
{
    int lost = 0;
    for (const auto &u : g_uploads) {
        bool live = false;
        for (const auto &m : g_mem) live = live || (u.first >= m.first && u.first + u.second.size() <= m.first + m.second);
        if (!live || memcmp(u.first, u.second.data(), u.second.size())) ++lost;
    }
    return lost;
}

// ---- the runtime ------------------------------------------------------------
cudaError_t cudaGetDeviceCount(int *n) { return *n = 2, cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { return *d = g_device, cudaSuccess; }
cudaError_t cudaSetDevice(int d) { return g_device = d, cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { return *v = 152, cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGetLastError()
{
    const cudaError_t e = g_last;
    g_last = cudaSuccess;
    return e;
}
cudaError_t cudaMalloc(void **p, size_t n)
{
    *p = calloc(n, 1);
    g_mem[(char *)*p] = n;
    return cudaSuccess;
}
cudaError_t cudaFree(void *p)
{
    ++g_frees;
    g_mem.erase((char *)p);
    free(p);
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { return *p = calloc(n, 1), cudaSuccess; }
cudaError_t cudaFreeHost(void *p) { return free(p), cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind kind, cudaStream_t)
{
    memcpy(d, s, n);
    if (kind == cudaMemcpyHostToDevice) g_uploads.push_back({(char *)d, std::vector<char>((char *)d, (char *)d + n)});
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) { return memset(d, v, n), cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void *f, cudaFuncAttribute a, int v)
{
    if (a != cudaFuncAttributeMaxDynamicSharedMemorySize) return cudaSuccess;
    int &limit = g_limit[{f, g_device}];
    g_lowered += v < limit;
    limit = v;
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void **, const void *) { return fail(cudaErrorInvalidSymbol); }
cudaError_t cudaGetDriverEntryPointByVersion(const char *, void **, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult *)
{
    return cudaErrorNotSupported;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **)
{
    return launch(f, c->dynamicSmemBytes);
}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, cudaStream_t s)
{
    g_config.push_back({grid, block, smem, s});
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *grid, dim3 *block, size_t *smem, void *s)
{
    const Config c = g_config.back();
    g_config.pop_back();
    *grid = c.grid;
    *block = c.block;
    *smem = c.smem;
    *(cudaStream_t *)s = c.stream;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) { return *k = (cudaKernel_t)f, cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void **, size_t smem, cudaStream_t)
{
    return launch((const void *)k, smem);
}
cudaError_t cudaLaunchKernel(const void *f, dim3, dim3, void **, size_t smem, cudaStream_t) { return launch(f, smem); }
void **__cudaRegisterFatBinary(void *)
{
    static void *handle;
    return &handle;
}
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *f, char *, const char *name, int, uint3 *, uint3 *, dim3 *, dim3 *, int *)
{
    g_names[f] = name;
}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
}
