// A stand-in for the CUDA runtime that runs no kernel, for host-side tests of libgpweno.so without a GPU (preloaded
// before libcudart): memory is host memory, launches are checked against the documented launch rules and
// recorded.  Two devices, 152 SMs each; as in the runtime, a kernel's limit on dynamic shared memory
// (cudaFuncAttributeMaxDynamicSharedMemorySize, 48 KB until it is set) belongs to one device.
#include <cuda_runtime_api.h>

#include <algorithm>
#include <atomic>
#include <chrono>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <thread>
#include <utility>
#include <vector>

namespace {
std::mutex g_m;
thread_local int g_device = 0;
std::map<std::pair<int, const void *>, int> g_limit;
std::map<const void *, std::pair<size_t, int>> g_blocks;   // allocation -> bytes, device
size_t g_bytes = 0, g_budget = ~size_t(0);
long g_launches = 0, g_lowered = 0;
std::atomic<int> g_hold{0}, g_held{0}, g_resident{0};
struct Config {
    dim3 grid, block;
    size_t smem;
    cudaStream_t st;
};
thread_local std::vector<Config> g_config;

cudaError_t launch(const void *f, dim3 block, size_t smem)
{
    std::lock_guard<std::mutex> l(g_m);
    const auto it = g_limit.find({g_device, f});
    const size_t limit = it == g_limit.end() ? 48 * 1024 : std::max(48 * 1024, it->second);
    if (smem > limit || block.x > 1024) return cudaErrorInvalidValue;
    ++g_launches;
    return cudaSuccess;
}
}  // namespace

extern "C" {

// ---- controls of the tests ----
void fake_device(int d) { g_device = d; }
long fake_launches() { return g_launches; }
long fake_lowered() { return g_lowered; }            // times a kernel's limit was set below an earlier value
size_t fake_bytes() { return g_bytes; }              // device memory held
void *fake_block(size_t bytes)                       // an allocation of that size
{
    for (const auto &b : g_blocks)
        if (b.second.first == bytes) return const_cast<void *>(b.first);
    return nullptr;
}
void fake_budget(size_t bytes) { g_budget = bytes; } // cudaMalloc fails beyond it
void fake_hold() { g_hold = 1; }                     // the next residency query returns only after fake_release()
int fake_held() { return g_held; }
void fake_release() { g_held = 0; }
void fake_resident(int n) { g_resident = n; }        // residency queries answer n

// ---- the runtime ----
const char *cudaGetErrorString(cudaError_t e) { return e == cudaSuccess ? "no error" : "fake runtime error"; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaGetDevice(int *d)
{
    *d = g_device;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int)
{
    *v = 152;
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMalloc(void **p, size_t n)
{
    std::lock_guard<std::mutex> l(g_m);
    if (g_bytes + n > g_budget) return cudaErrorMemoryAllocation;
    *p = std::malloc(n);
    g_blocks[*p] = {n, g_device};
    g_bytes += n;
    return cudaSuccess;
}
cudaError_t cudaFree(void *p)
{
    std::lock_guard<std::mutex> l(g_m);
    const auto it = g_blocks.find(p);
    if (it == g_blocks.end()) return p ? cudaErrorInvalidValue : cudaSuccess;
    g_bytes -= it->second.first;
    g_blocks.erase(it);
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaMallocHost(void **p, size_t n)
{
    *p = std::malloc(n);
    return cudaSuccess;
}
cudaError_t cudaFreeHost(void *p)
{
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaMemset(void *p, int v, size_t n)
{
    std::memset(p, v, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind)
{
    std::memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t)
{
    std::memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void **p, const void *s)
{
    *p = const_cast<void *>(s);
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void *f, cudaFuncAttribute, int v)
{
    std::lock_guard<std::mutex> l(g_m);
    const auto it = g_limit.find({g_device, f});
    if (it != g_limit.end() && v < it->second) ++g_lowered;
    g_limit[{g_device, f}] = v;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int block, size_t smem,
                                                                   unsigned)
{
    *n = g_resident ? g_resident.load() : std::max(1, std::min(512 / block, (int)(228 * 1024 / (smem + 1024))));
    if (g_hold.exchange(0)) {
        g_held = 1;
        for (int k = 0; k < 5000 && g_held; ++k) std::this_thread::sleep_for(std::chrono::milliseconds(1));
        g_held = 0;
    }
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **)
{
    return launch(f, c->blockDim, c->dynamicSmemBytes);
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f)
{
    *k = (cudaKernel_t)f;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3 block, void **, size_t smem, cudaStream_t)
{
    return launch((const void *)k, block, smem);
}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, cudaStream_t st)
{
    g_config.push_back({grid, block, smem, st});
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *grid, dim3 *block, size_t *smem, void *st)
{
    const Config c = g_config.back();
    g_config.pop_back();
    *grid = c.grid;
    *block = c.block;
    *smem = c.smem;
    *(cudaStream_t *)st = c.st;
    return cudaSuccess;
}
void **__cudaRegisterFatBinary(void *)
{
    static void *h;
    return &h;
}
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, uint3 *, uint3 *, dim3 *, dim3 *, int *) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
}
