// The tensor-core GEMMs' host code against a stand-in for the CUDA runtime with two devices: every launch has to find
// its kernel opted in to its shared memory on the device that is current, and a grid of that device's size.
#include <cstdio>
#include <map>
#include <set>
#include <utility>

#include "../../paper_2310_04559_gb300/csrc/cc_internal.cuh"

namespace {
int g_dev = 0, g_bad = 0, g_launches = 0;
unsigned g_grid = 0;
std::set<std::pair<int, const void*>> g_opted;

void launched(const void* fn, unsigned grid, size_t smem)
{
    ++g_launches;
    g_grid = grid;
    if (smem > 48 * 1024 && !g_opted.count({g_dev, fn})) ++g_bad;
}

int fake_encode(...) { return 0; }
}  // namespace

namespace cc {
void count_launch(int) {}
}

extern "C" {
cudaError_t cudaGetDevice(int* d) { *d = g_dev; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int d) { *v = d == 0 ? 140 : 10; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void* fn, cudaFuncAttribute, int) { g_opted.insert({g_dev, fn}); return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t*) { *n = g_dev == 0 ? 70 : 5; return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) { *n = 1; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** f, unsigned, unsigned long long, cudaDriverEntryPointQueryResult* q)
{
    *f = (void*)&fake_encode;
    *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* fn, void**)
{
    launched(fn, c->gridDim.x, c->dynamicSmemBytes);
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void* s) { *p = (void*)s; return cudaSuccess; }
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
// what nvcc's launch and registration stubs call
dim3 g_pushed;
size_t g_pushed_smem = 0;
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, uint3*, uint3*, dim3*, dim3*, int*) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 g, dim3, size_t s, void*) { g_pushed = g; g_pushed_smem = s; return 0; }
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* s, void*) { *g = g_pushed; *b = dim3(1); *s = g_pushed_smem; return cudaSuccess; }
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* fn) { *k = (cudaKernel_t)fn; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3, void**, size_t s, cudaStream_t) { launched((const void*)k, g.x, s); return cudaSuccess; }
}

int main()
{
    using namespace cc;
    static char mem[256];
    static int counter[2], status;
    for (int dev = 0; dev < 2; ++dev) {
        g_dev = dev;
        GemmCrt g{};
        g.M = g.N = 4096; g.K = 64; g.nm = 12;
        g.A = g.B = mem; g.pitchA = g.pitchB = 64; g.rowsA = g.rowsB = 4096;
        g.planes = (unsigned char*)mem; g.pitch = 4096;
        g.ksplit = 1; g.status = &status; g.counter = counter;
        int before = g_launches;
        if (gemm_crt(g, nullptr) != cudaSuccess || g_launches != before + 1) return printf("gemm_crt: no launch\n"), 2;
        if (g_grid != (dev == 0 ? 140u : 10u)) return printf("gemm_crt on device %d: %u CTAs\n", dev, g_grid), 3;
        GemmTc t{};
        t.kind = TC_BF16;
        t.M = t.N = 4096; t.K = 64;
        t.A = t.B = mem; t.pitchA = t.pitchB = 64; t.rowsA = t.rowsB = 4096;
        t.slices = 1; t.ngroups = 1; t.gn[0] = 1; t.epi = EPI_FP64_RMW; t.ksplit = 1;
        t.out = OutDesc{(double*)mem, plain_map(4096), plain_map(1), 0};
        t.status = &status;
        before = g_launches;
        if (gemm_tc(t, nullptr) != cudaSuccess || g_launches == before) return printf("gemm_tc: no launch\n"), 4;
        if (g_grid != (dev == 0 ? 140u : 10u)) return printf("gemm_tc on device %d: %u CTAs\n", dev, g_grid), 5;
    }
    printf("%d launches, %d without their shared memory\n", g_launches, g_bad);
    return g_bad ? 1 : 0;
}
