// gemm_f64.cu -- FP64 GEMM for the plain-FP64 precision mode.
//
// Computes C[rmap(m) + cmap(n)] (= or +=) sum_k A(m,k) B(n,k) for the two
// contractions of the integral-first order (Section 3.2): the integral block
// (ac|bd) = sum_P L_Pac L_Pbd (Eq. 5) and the ladder GEMM sum_cd (ac|bd) t_ijcd
// (Eq. 6), and for the other contractions.
//
// GB300 has two FP64 lanes per SM and clock: one warp-wide FMA keeps an SM sub-partition's FP64 pipe
// for about 64 clocks, and the tensor-core form (mma.m8n8k4.f64) runs on the same lanes at a lower measured rate
// (1.10 against 1.25 TFLOP/s for the whole GPU).  So the kernel uses plain FMAs, loads cost nothing
// next to them, and what matters is that every sub-partition of every SM has the same number of them:
//   - a warp owns 8 rows and 8 NT columns (2 x NT per thread), so rows are padded to 8 only (a ladder
//     GEMM has o(o+1)/2 rows: 55 rows cost 56, on 64-row tiles 64);
//   - a CTA's four warps take 32 rows, or split K between them where there are no more than 16 or 8 rows;
//   - NT and a split of K over a cluster of up to eight CTAs are chosen so that the CTAs fill whole
//     waves of the device; partial sums meet in distributed shared memory and are added in a fixed order.
// Against 64 x 64 tiles on mma.m8n8k4.f64: o=4/v=24/n=60 976 -> 157 us, o=10/v=100/n=500 62.1 -> 47.6 ms (1.21 TFLOP/s of the
// 1.25 that the FMA units reach), 55 x 5050 x 5050 6.6 -> 2.7 ms.
#include <algorithm>
#include <cmath>

#include "cc_internal.cuh"

namespace cc {
namespace {

constexpr int THREADS = 128, KT = 16;

__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ double peer_load(const double* p, uint32_t rank)
{
    uint32_t a;
    double x;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(x) : "r"(a) : "memory");
    return x;
}

// One R x KT tile into registers: the thread's elements q * THREADS + t, the contiguous index fastest.
template <int R>
struct Tile {
    static constexpr int N = (R * KT + THREADS - 1) / THREADS;
    double v[N];
    __device__ __forceinline__ void load(const double* __restrict__ X, const Map2& rm, const Map2& km, bool kmajor, int row0,
                                         int nrows, int k0, int kend)
    {
#pragma unroll
        for (int q = 0; q < N; ++q) {
            const int e = q * THREADS + (int)threadIdx.x;
            const int r = kmajor ? e / KT : e % R, k = kmajor ? e % KT : e / R;
            v[q] = (e < R * KT && row0 + r < nrows && k0 + k < kend) ? __ldg(X + map2(rm, row0 + r) + map2(km, k0 + k)) : 0.0;
        }
    }
    __device__ __forceinline__ void store(double* S, bool kmajor) const  // S[k][R + 1]
    {
#pragma unroll
        for (int q = 0; q < N; ++q) {
            const int e = q * THREADS + (int)threadIdx.x;
            const int r = kmajor ? e / KT : e % R, k = kmajor ? e % KT : e / R;
            if (e < R * KT) S[k * (R + 1) + r] = v[q];
        }
    }
};

// NT: columns per thread; WK: warps that split K (4 / WK warps side by side in rows).  Cluster rank: K split.
template <int NT, int WK>
__global__ void __launch_bounds__(THREADS) gemm_f64_kernel(const GemmF64 g, int kmajor_a, int kmajor_b, int ks, int kper)
{
    constexpr int TM = 32 / WK, TN = 8 * NT;
    constexpr int ASZ = KT * (TM + 1), BSZ = KT * (TN + 1);
    constexpr int RING = 2 * (ASZ + BSZ), PART = WK * TM * TN;
    __shared__ double sm[RING > PART ? RING : PART];

    // one-dimensional grid over tiles x K splits (no gridDim.y limit on M)
    const int tiles_n = (g.N + TN - 1) / TN;
    const long long tile = blockIdx.x / ks;
    const int rank = ks > 1 ? (int)cluster_rank() : 0;
    const int m0 = (int)(tile / tiles_n) * TM, n0 = (int)(tile % tiles_n) * TN;
    if (g.tri > 0 && (long long)min(g.N - 1, n0 + TN - 1) / g.tri < (long long)m0 / g.tri) return;  // (the whole cluster)
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int wm = warp / WK, wk = warp % WK;
    const int ra = wm * 8 + (lane >> 3) * 2, cb = lane & 7;  // rows ra, ra + 1; columns cb + 8 j
    const bool live = m0 + wm * 8 < g.M;                     // (uniform over the warp)
    const int kbeg = rank * kper, kend = min(g.K, kbeg + kper);

    double acc[2][NT];
#pragma unroll
    for (int j = 0; j < NT; ++j) acc[0][j] = acc[1][j] = 0.0;

    Tile<TM> ta;
    Tile<TN> tb;
    double* As = sm;
    double* Bs = sm + 2 * ASZ;
    ta.load(g.A, g.am, g.ak, kmajor_a, m0, g.M, kbeg, kend);
    tb.load(g.B, g.bm, g.bk, kmajor_b, n0, g.N, kbeg, kend);
    ta.store(As, kmajor_a);
    tb.store(Bs, kmajor_b);
    __syncthreads();
    int cur = 0;
    for (int k0 = kbeg; k0 < kend; k0 += KT, cur ^= 1) {
        const bool more = k0 + KT < kend;
        if (more) {
            ta.load(g.A, g.am, g.ak, kmajor_a, m0, g.M, k0 + KT, kend);
            tb.load(g.B, g.bm, g.bk, kmajor_b, n0, g.N, k0 + KT, kend);
        }
        if (live) {
            const double* a = As + cur * ASZ + ra;
            const double* b = Bs + cur * BSZ + cb;
            const int kn = min(KT, kend - k0);
            // (rounds of zeros at the end of K are left out: they would cost as much as any other)
            for (int kk = wk; kk < kn; kk += WK) {
                const double a0 = a[kk * (TM + 1)], a1 = a[kk * (TM + 1) + 1];
#pragma unroll
                for (int j = 0; j < NT; ++j) {
                    const double x = b[kk * (TN + 1) + 8 * j];
                    acc[0][j] = fma(a0, x, acc[0][j]);
                    acc[1][j] = fma(a1, x, acc[1][j]);
                }
            }
        }
        if (more) {
            ta.store(As + (cur ^ 1) * ASZ, kmajor_a);
            tb.store(Bs + (cur ^ 1) * BSZ, kmajor_b);
        }
        __syncthreads();
    }

    auto put = [&](int m, int n, double x) {
        double* p = g.out.C + map2(g.out.rmap, m) + map2(g.out.cmap, n);
        *p = g.out.accumulate ? *p + x : x;
    };
    if (WK == 1 && ks == 1) {
        if (!live) return;
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < NT; ++j)
                if (m0 + ra + i < g.M && n0 + cb + 8 * j < g.N) put(m0 + ra + i, n0 + cb + 8 * j, acc[i][j]);
        return;
    }
    // partial sums [wk][row][column], added over the warps and the cluster's CTAs in that order
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < NT; ++j) sm[(wk * TM + ra + i) * TN + cb + 8 * j] = acc[i][j];
    if (ks > 1) cluster_sync();
    else __syncthreads();
    for (int e = rank * THREADS + (int)threadIdx.x; e < TM * TN; e += ks * THREADS) {
        const int m = m0 + e / TN, n = n0 + e % TN;
        if (m >= g.M || n >= g.N) continue;
        double s = 0.0;
        for (int r = 0; r < ks; ++r)
#pragma unroll
            for (int w = 0; w < WK; ++w) {
                const double* q = sm + w * TM * TN + e;
                s += ks > 1 ? peer_load(q, (uint32_t)r) : *q;
            }
        put(m, n, s);
    }
    if (ks > 1) cluster_sync();  // no CTA leaves while a peer reads its sums
}

struct Shape {
    int nt, wk, ks;
};

// Fewest clocks on the busiest SM: CTAs per SM times a CTA's FMAs (64 clocks per warp-wide FMA and sub-partition) plus
// its start-up; many CTAs per SM even out.
Shape pick_shape(const GemmF64& g)
{
    const int sms = std::max(1, device_sm_count());
    Shape best{8, 1, 1};
    double best_t = 1e300;
    const int wk = g.M <= 8 ? 4 : (g.M <= 16 ? 2 : 1), tm = 32 / wk;
    for (int nt = 8; nt >= 1; nt /= 2)
        for (int ks = 1; ks <= 8; ks *= 2) {
            if (ks > 1 && g.K / ks < 2 * KT) continue;
            double tiles = std::ceil(g.M / (double)tm) * std::ceil(g.N / (8.0 * nt));
            if (g.tri > 0) tiles = 0.5 * tiles + 0.5 * std::ceil(g.N / (8.0 * nt));  // about half are skipped
            const double cta = 64.0 * 2 * nt * std::ceil(g.K / (double)ks) / wk + 3000.0 + (ks > 1 ? 4000.0 : 0.0);
            const double per_sm = tiles * ks / sms;
            const double t = (per_sm < 24 ? std::ceil(per_sm) : per_sm + 0.5) * cta;
            if (t < 0.98 * best_t) { best_t = t; best = Shape{nt, wk, ks}; }
        }
    return best;
}

template <int NT, int WK>
cudaError_t launch(const GemmF64& g, int ka, int kb, int ks, cudaStream_t s)
{
    const long long tiles = (long long)((g.N + 8 * NT - 1) / (8 * NT)) * ((g.M + 32 / WK - 1) / (32 / WK));
    if (tiles * ks > 0x7fffffffll) return cudaErrorInvalidConfiguration;
    const int kper = ((g.K + ks - 1) / ks + KT - 1) / KT * KT;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(tiles * ks));
    cfg.blockDim = dim3(THREADS);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)ks;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, gemm_f64_kernel<NT, WK>, g, ka, kb, ks, kper);
}

template <int NT>
cudaError_t launch_wk(const GemmF64& g, int ka, int kb, const Shape& sh, cudaStream_t s)
{
    if (sh.wk == 4) return launch<NT, 4>(g, ka, kb, sh.ks, s);
    if (sh.wk == 2) return launch<NT, 2>(g, ka, kb, sh.ks, s);
    return launch<NT, 1>(g, ka, kb, sh.ks, s);
}

}  // namespace

cudaError_t gemm_f64(const GemmF64& g, cudaStream_t s)
{
    if (g.M <= 0 || g.N <= 0) return cudaSuccess;
    // the index that is contiguous in memory runs fastest over the threads
    const int ka = g.ak.div == 0 && !g.ak.tab && g.ak.s1 == 1, kb = g.bk.div == 0 && !g.bk.tab && g.bk.s1 == 1;
    const Shape sh = pick_shape(g);
    cudaError_t err;
    if (sh.nt == 8) err = launch_wk<8>(g, ka, kb, sh, s);
    else if (sh.nt == 4) err = launch_wk<4>(g, ka, kb, sh, s);
    else if (sh.nt == 2) err = launch_wk<2>(g, ka, kb, sh, s);
    else err = launch_wk<1>(g, ka, kb, sh, s);
    if (err != cudaSuccess) return err;
    count_launch();
    return cudaGetLastError();
}

}  // namespace cc
