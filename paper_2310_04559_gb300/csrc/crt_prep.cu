// crt_prep.cu -- operands and results of the residue GEMM (crt.cuh, gemm_crt.cu): FP64 rows to bf16
// residue stacks D[l][row][pitch], the byte planes of an intermediate to the residues of its
// rounded rows, and the byte planes of a result to FP64.
//
// A row is rounded once to 42-bit integers X = round(x 2^(41 - e)), max |row| < 2^e, so every kernel here
// needs the row's maximum before it can write: the rows are walked twice, by a cluster of up to eight CTAs
// that exchange their maxima through distributed shared memory.  Spreading one row over a cluster keeps few
// rows in flight, so that the second walk finds the row in L2 and HBM sees it once.
//
// Four consecutive elements of a row form a quad, one thread's unit: its residues leave as one 8-byte store
// per modulus.  Quads must not straddle the segments a row consists of, so segments are padded to
// multiples of four with zeros (both operands of a GEMM use the same padded order, and zeros add nothing):
//   plain rows of K = (o, i):    k = o inner4 + i, inner4 = inner rounded up to four
//   packed c <= d rows: blocks of 8 x 8 entries (crt.cuh)
#include <climits>
#include <type_traits>

#include "cc_internal.cuh"
#include "crt.cuh"

namespace cc {
namespace {

constexpr int NT = 256;  // threads per CTA
constexpr size_t kMaxSmem = 227 * 1024;  // shared memory of one CTA at most
constexpr unsigned long long kAbs = 0x7fffffffffffffffull;
constexpr unsigned long long kInf = 0x7ff0000000000000ull;

__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

__device__ __forceinline__ uint32_t cluster_size()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}

// Maximum over the CTA's threads; every thread gets it.
__device__ __forceinline__ int block_max(int m, int* red)
{
    m = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
    __syncthreads();
    m = red[0];
    for (int w = 1; w < NT / 32; ++w) m = max(m, red[w]);
    __syncthreads();
    return m;
}

// Maximum over all threads of the cluster; every thread gets it.  `red`: NT / 32 + 1 values of shared memory, not reused
// before cluster_done().  The CTAs' values are exchanged through distributed shared memory; that everybody has read
// them is waited for only in cluster_done(), before the next exchange or the exit.
template <typename T>
__device__ __forceinline__ T cluster_max(T m, T* red)
{
    static_assert(sizeof(T) == 8, "64-bit values");
    for (int w = 16; w > 0; w >>= 1) {
        const T o = __shfl_xor_sync(0xffffffffu, m, w);
        m = o > m ? o : m;
    }
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
    __syncthreads();
    m = red[0];
    for (int w = 1; w < NT / 32; ++w) m = red[w] > m ? red[w] : m;
    const uint32_t cs = cluster_size();
    if (cs > 1) {
        if (threadIdx.x == 0) red[NT / 32] = m;
        asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
        const uint32_t mine = (uint32_t)__cvta_generic_to_shared(&red[NT / 32]);
        for (uint32_t r = 0; r < cs; ++r) {
            uint32_t a;
            unsigned long long o;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(mine), "r"(r));
            asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(o) : "r"(a) : "memory");
            m = (T)o > m ? (T)o : m;
        }
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    }
    return m;
}

__device__ __forceinline__ void cluster_done()
{
    if (cluster_size() > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    else __syncthreads();
}

__device__ __forceinline__ int exp_of_maxbits(unsigned long long b)
{
    if (b == 0) return 0;
    const int ex = (int)(b >> 52);
    return ex == 0 ? -1022 : ex - 1022;
}

// round(x * 2^(41 - e)) from the bit pattern of x (|x| < 2^e)
__device__ __forceinline__ long long fixed_of(double x, int e)
{
    const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
    const int ex = (int)((bits >> 52) & 0x7ff);
    unsigned long long mant = bits & 0x000fffffffffffffull;
    if (ex == 0 && mant == 0) return 0;
    int exe = ex;
    if (ex == 0) exe = 1; else mant |= 0x0010000000000000ull;
    const int sh = exe - 1075 + kCrtBits - 1 - e;
    long long X;
    if (sh >= 0) X = (long long)(mant << sh);
    else if (sh > -64) X = (long long)((mant + (1ull << (-sh - 1))) >> (-sh));
    else X = 0;
    return (bits >> 63) ? -X : X;
}

// y 2^-s rounded down
__device__ __forceinline__ long long shr_floor(long long y, int s) { return s >= 0 ? y >> min(s, 63) : y << -s; }

// Residues of N quads (u = X + kCrtBias): 8 bytes per modulus and quad at out[] + l * stride + k (elements).  out and
// stride are the same for the whole CTA, only the 32-bit k differs between threads.  Streaming stores: the rows in
// flight keep the L2.
template <int N>
__device__ __forceinline__ void put_quads(const unsigned long long (&u)[N][4], int nm, unsigned short* const (&out)[N],
                                          const long long (&stride)[N], uint32_t k)
{
    CrtPieces2 h[N][2] = {};
#pragma unroll
    for (int i = 0; i < N; ++i) {
        h[i][0] = CrtPieces2(u[i][0], u[i][1]);
        h[i][1] = CrtPieces2(u[i][2], u[i][3]);
    }
#pragma unroll
    for (int l = 0; l < kCrtMax; ++l) {
        if (l >= kCrtMin && l >= nm) break;
        const int p = crt_p(l);
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const uint2 v = make_uint2(crt_residues2(h[i][0], p), crt_residues2(h[i][1], p));
            unsigned short* row = out[i] + l * stride[i];
            __stcs(reinterpret_cast<uint2*>(row + k), v);
        }
    }
}

__device__ __forceinline__ void put_quad(const long long (&X)[4], int nm, unsigned short* out, long long stride, uint32_t k)
{
    const unsigned long long x[1][4] = {{X[0] + kCrtBias, X[1] + kCrtBias, X[2] + kCrtBias, X[3] + kCrtBias}};
    unsigned short* const o[1] = {out};
    const long long st[1] = {stride};
    put_quads<1>(x, nm, o, st, k);
}

// One byte of each of four consecutive elements from every plane, at base + off in plane 0, `ps` bytes between planes
// (a multiple of 16).  base is the same for the whole CTA where that matters.
template <bool AL>
struct RawQuad {
    uint32_t w[kCrtMax];
    __device__ __forceinline__ void load(const unsigned char* base, uint32_t off, long long ps, int nm)
    {
        const uint32_t mis = AL ? 0u : (uint32_t)((uintptr_t)base & 3);
        const unsigned char* q = base - mis;
        const uint32_t o = off + mis, sh = AL ? 0u : (o & 3) * 8, oa = AL ? o : o & ~3u;
#pragma unroll
        for (int l = 0; l < kCrtMax; ++l) {
            if (l >= kCrtMin && l >= nm) break;
            const uint32_t* s = reinterpret_cast<const uint32_t*>(q + l * ps + oa);
            w[l] = AL ? __ldg(s) : __funnelshift_r(__ldg(s), __ldg(s + 1), sh);
        }
    }
    // the elements as signed fractions of P, in units of 2^-64
    template <bool WIDE>
    __device__ __forceinline__ void fractions(const CrtRec& c, long long (&y)[4]) const
    {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            CrtAcc<WIDE> a(c);
#pragma unroll
            for (int l = 0; l < kCrtMax; ++l) {
                if (l >= kCrtMin && l >= c.nm) break;
                a.add(__byte_perm(w[l], 0, 0x4440 + j), c, l);
            }
            y[j] = a.fraction();
        }
    }
    // their top words: within nm * 128 of y >> 32
    __device__ __forceinline__ void tops(const CrtRec& c, int (&t)[4]) const
    {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            uint32_t a = c.t2;
#pragma unroll
            for (int l = 0; l < kCrtMax; ++l) {
                if (l >= kCrtMin && l >= c.nm) break;
                a += __byte_perm(w[l], 0, 0x4440 + j) * c.w2[l];
            }
            t[j] = (int)a;
        }
    }
};

// (i, j) of place p in the enumeration i-major of 0 <= i <= j < n: i n - i (i - 1) / 2 places lie before row i.
__device__ __forceinline__ void tri_index(long long p, long long n, long long& i, long long& j)
{
    const double b = 2.0 * (double)n + 1.0;
    i = (long long)(0.5 * (b - sqrt(fmax(b * b - 8.0 * (double)p, 0.0))));
    auto before = [&](long long q) { return q * n - q * (q - 1) / 2; };
    while (i > 0 && before(i) > p) --i;  // (the square root may be off by one)
    while (before(i + 1) <= p) ++i;
    j = i + (p - before(i));
}

// Row exponent of fractions y_k 2^(e_k): E with max |y_k| 2^(e_k) < 2^E, from one walk over the top words t_k of y_k.
// With e'_k = e_k - emax <= 0 and F = max |t_k| 2^(e'_k), max |y_k| 2^(e_k) is within (F +- slack) 2^(32 + emax),
// slack = nm * 128 + the rounding of F's float.  Where both ends give bit lengths at most one apart, the upper one
// stands (the rows carry 43 bits, one more than an FP64 row, for that); where they do not (a row far below the range
// of the integers), the row is walked again in full.  F is kept as float bits plus e' << 23, compared as integers
// (e' clamped to -200: what is smaller by 2^-200 ends in the second walk).
__device__ __forceinline__ int exp_code(int e) { return max(e, -100) * (1 << 23); }

__device__ __forceinline__ int top_code(int t, int ecode)
{
    return __float_as_int((float)(uint32_t)abs(t)) + ecode;  // (INT_MIN's magnitude is right as unsigned)
}

// E from the row's largest code; false: walk again.
__device__ __forceinline__ bool exponent_of(int code, int emax, int nm, int& E)
{
    const uint32_t slack = (uint32_t)nm * 128 + 512;
    const uint32_t F = code > 0 ? (uint32_t)__int_as_float(code) : 0u;  // < 2^31 + 256
    E = 64 - __clz(F + slack) + emax;
    return F > slack && 64 - __clz(F - slack) + emax >= E - 1;
}

// y 2^-s, rounded down, s >= 0
__device__ __forceinline__ long long shr_fast(long long y, int s) { return y >> min(s, 63); }

// Quads q, q + step, ... of a row of qi quads per outer index, as (o, i) without divisions.
struct QuadIter {
    uint32_t o, i, so, si, qi;
    __device__ QuadIter(uint32_t first, uint32_t step, uint32_t qi_) : o(first / qi_), i(first % qi_), so(step / qi_), si(step % qi_), qi(qi_) {}
    __device__ void next()
    {
        o += so;
        i += si;
        if (i >= qi) { i -= qi; ++o; }
    }
};

// Walk the quads of a row (outer indices below `outer`), each loaded one step before it is used: with the bytes of 12
// planes to gather per quad, the walks are bound by the latency of these loads.
template <bool AL, typename F>
__device__ __forceinline__ void walk_quads(QuadIter t, uint32_t outer, const unsigned char* X, long long pitch,
                                           long long plane, int nm, F&& use)
{
    RawQuad<AL> w;
    if (t.o < outer) w.load(X + (long long)t.o * pitch + t.i * 4, 0u, plane, nm);
    while (t.o < outer) {
        const RawQuad<AL> now = w;
        const uint32_t o = t.o, i = t.i;
        t.next();
        if (t.o < outer) w.load(X + (long long)t.o * pitch + t.i * 4, 0u, plane, nm);
        use(o, i, now);
    }
}

// ---------------------------------------------------------------- FP64 rows
struct RowsArg {
    RowSrc src;          // rm: row offsets; km unused
    long long ostride;   // elements between outer indices
    int outer, inner;
};

// Bound: HBM and the residues' arithmetic (96 rows of 46080: 37 us, 30% of HBM, 49% of the multipliers).
__global__ void __launch_bounds__(NT) crt_rows_kernel(const RowsArg a, int nm, unsigned short* __restrict__ D,
                                                      long long pitch, int* __restrict__ e_out, int* __restrict__ status)
{
    __shared__ unsigned long long red[NT / 32 + 1];
    const uint32_t cs = cluster_size(), rank = cluster_rank();
    const long long r = blockIdx.x / cs;
    const double* X = a.src.X + map2(a.src.rm, r);
    const uint32_t qi = (uint32_t)(a.inner + 3) / 4;
    const uint32_t step = cs * NT, first = rank * NT + threadIdx.x;
    unsigned long long mx = 0;
    for (QuadIter t(first, step, qi); t.o < (uint32_t)a.outer; t.next()) {
        const uint32_t i0 = t.i * 4;
        const double* x = X + (long long)t.o * a.ostride + i0;
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if ((int)i0 + j < a.inner) {
                const unsigned long long b = (unsigned long long)__double_as_longlong(x[j]) & kAbs;
                mx = b > mx ? b : mx;
            }
    }
    mx = cluster_max(mx, red);
    cluster_done();
    const int e = exp_of_maxbits(mx);
    if (rank == 0 && threadIdx.x == 0) {
        e_out[r] = e;
        if (status && mx >= kInf) atomicOr(status, kStatusNonfinite);
    }
    unsigned short* Dr = D + r * pitch;
    const long long stride = a.src.rows * pitch;
    for (QuadIter t(first, step, qi); t.o < (uint32_t)a.outer; t.next()) {
        const uint32_t i0 = t.i * 4;
        const double* x = X + (long long)t.o * a.ostride + i0;
        long long v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = (int)i0 + j < a.inner ? fixed_of(x[j], e) : 0;
        put_quad(v, nm, Dr, stride, (t.o * qi + t.i) * 4);
    }
}

// Rows of up to 4 * WQ * 32 elements: one warp per row, the row in registers (one walk).  A CTA per row of 96 elements
// spent its time on barriers and idle threads: 118 us for 46080 such rows, 41 now.
constexpr int WQ = 2;  // quads per lane

__global__ void __launch_bounds__(NT) crt_rows_warp_kernel(const RowsArg a, int nm, unsigned short* __restrict__ D,
                                                           long long pitch, int* __restrict__ e_out, int* __restrict__ status)
{
    const int lane = threadIdx.x & 31;
    const long long r = (long long)blockIdx.x * (NT / 32) + (threadIdx.x >> 5);
    if (r >= a.src.rows) return;
    const double* X = a.src.X + map2(a.src.rm, r);
    const uint32_t qi = (uint32_t)(a.inner + 3) / 4, nq = qi * (uint32_t)a.outer;
    double x[WQ][4];
    unsigned long long mx = 0;
#pragma unroll
    for (int w = 0; w < WQ; ++w) {
        const uint32_t q = lane + 32 * w, o = q / qi, i0 = (q % qi) * 4;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            x[w][j] = q < nq && (int)i0 + j < a.inner ? X[(long long)o * a.ostride + i0 + j] : 0.0;
            const unsigned long long b = (unsigned long long)__double_as_longlong(x[w][j]) & kAbs;
            mx = b > mx ? b : mx;
        }
    }
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) {
        const unsigned long long b = __shfl_xor_sync(0xffffffffu, mx, s);
        mx = b > mx ? b : mx;
    }
    const int e = exp_of_maxbits(mx);
    if (lane == 0) {
        e_out[r] = e;
        if (status && mx >= kInf) atomicOr(status, kStatusNonfinite);
    }
    unsigned short* Dr = D + r * pitch;
    const long long stride = a.src.rows * pitch;
#pragma unroll
    for (int w = 0; w < WQ; ++w) {
        const uint32_t q = lane + 32 * w;
        if (q >= nq) break;
        long long v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = fixed_of(x[w][j], e);
        put_quad(v, nm, Dr, stride, q * 4);
    }
}

// ------------------------------------------------------- FP64 columns (K strided)
__device__ __forceinline__ long long col_off(const ColSrc& s, long long r)
{
    if (s.brows == 0) return r;
    return map2(s.bmap, r / s.brows) + r % s.brows;
}

constexpr int CR = 32, CK = 64;  // transpose tile: 32 rows x 64 k

// Bound: the transposition's latency and HBM (o=8/v=160/n=800: 0.16 GB read twice, 0.49 GB written, 218 us, 42% of HBM).
// PREMAX: mx holds every row's largest |x| (over a K range longer than this call's); else it is found first, over the
// whole K by the cluster's CTAs, each taking every cs-th tile of k in both walks.
template <bool PREMAX>
__global__ void __launch_bounds__(NT) crt_cols_kernel(const ColSrc src, int nm, const unsigned long long* __restrict__ mx,
                                                      unsigned short* __restrict__ D, long long pitch,
                                                      int* __restrict__ e_out, int* __restrict__ status)
{
    __shared__ double S[CK][CR + 1];
    __shared__ unsigned long long part[NT / 32][CR], top[CR];
    __shared__ int ex[CR];
    const uint32_t cs = cluster_size(), rank = cluster_rank();
    const long long r0 = (long long)(blockIdx.x / cs) * CR;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const long long stride = src.rows * pitch;
    const long long roff = r0 + tx < src.rows ? col_off(src, r0 + tx) : -1;
    unsigned long long m = 0;
    if (PREMAX) {
        if (roff >= 0 && ty == 0) m = mx[r0 + tx];
    } else {
        if (roff >= 0)
            for (long long k0 = (long long)rank * CK; k0 < src.K; k0 += (long long)cs * CK)
#pragma unroll
                for (int y = 0; y < CK; y += NT / 32) {
                    const long long k = k0 + y + ty;
                    if (k >= src.K) break;
                    const unsigned long long b = (unsigned long long)__double_as_longlong(src.X[roff + k * src.ldk]) & kAbs;
                    m = b > m ? b : m;
                }
        part[ty][tx] = m;
        __syncthreads();
        if (ty == 0) {
            for (int w = 1; w < NT / 32; ++w) m = part[w][tx] > m ? part[w][tx] : m;
            top[tx] = m;
        }
        if (cs > 1) {
            asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
            if (ty == 0) {
                const uint32_t mine = (uint32_t)__cvta_generic_to_shared(&top[tx]);
                for (uint32_t r = 0; r < cs; ++r) {
                    uint32_t a;
                    unsigned long long o;
                    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(mine), "r"(r));
                    asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(o) : "r"(a) : "memory");
                    m = o > m ? o : m;
                }
            }
            asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");  // (waited for at the end)
        }
    }
    if (ty == 0) {
        ex[tx] = exp_of_maxbits(m);
        if (rank == 0 && roff >= 0) {
            e_out[r0 + tx] = ex[tx];
            if (status && m >= kInf) atomicOr(status, kStatusNonfinite);
        }
    }
    for (long long k0 = (long long)rank * CK; k0 < src.K; k0 += (long long)cs * CK) {
        __syncthreads();
#pragma unroll
        for (int y = 0; y < CK; y += NT / 32) {
            const long long k = k0 + y + ty;
            S[y + ty][tx] = (k < src.K && roff >= 0) ? src.X[roff + k * src.ldk] : 0.0;
        }
        __syncthreads();
        // 16 quads of k per row; 16 lanes write 128 contiguous bytes of one row per modulus
        const int q = threadIdx.x & 15;
#pragma unroll
        for (int y = threadIdx.x >> 4; y < CR; y += NT / 16) {
            const long long r = r0 + y, k = k0 + 4 * q;
            if (r >= src.rows || k >= src.K) continue;
            const int e = ex[y];
            long long v[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) v[j] = fixed_of(S[4 * q + j][y], e);
            put_quad(v, nm, D + r * pitch, stride, (uint32_t)k);
        }
    }
    if (!PREMAX) cluster_done();
}

// ------------------------------------------------ symmetric / antisymmetric packing
constexpr int TT = 32;  // tile edge

// Step t through the tile pairs (tc <= td) of nt tile rows, `by` pairs at a time.
struct TilePair {
    int tc, td, nt;
    __device__ TilePair(int nt_, int first) : tc(0), td(0), nt(nt_) { skip(first); }
    __device__ void skip(int by)
    {
        td += by;
        while (tc < nt && td >= nt) { td = td - nt + tc + 1; ++tc; }
    }
    __device__ bool ok() const { return tc < nt; }
};

// This thread's quad of a tile pair's output: entries (c, d .. d + 3) of tile (tc, td), local coordinates cl, dl, position k
// in the packed order.  16 threads make one 8 x 8 block, so every 16 lanes write one whole line per residue.
struct QuadPos {
    int cl, dl;
    uint32_t k;
    bool live;
    __device__ __forceinline__ QuadPos(const TilePair& t, int nb)
    {
        const int blk = (int)threadIdx.x >> 4, bi = blk >> 2, bj = blk & 3;
        const int n = min(4, nb - 4 * t.tc), m = min(4, nb - 4 * t.td);
        const bool diag = t.tc == t.td;
        live = bi < n && bj < m && (!diag || bj >= bi);
        cl = bi * 8 + (((int)threadIdx.x & 15) >> 1);
        dl = bj * 8 + ((int)threadIdx.x & 1) * 4;
        const int idx = diag ? bi * n - bi * (bi - 1) / 2 + (bj - bi) : bi * m + bj;
        k = (uint32_t)((crt_tile_off(t.tc, t.td, nb) + idx) * 64 + (cl & 7) * 8 + (dl & 7));
    }
};

// One pass over HBM: the second walk reads L2.  A small share everywhere (o=16/v=160: 82 us of 28 ms).
// T+ and T- of the pairs i <= j (or of all pairs, each with both rows): row p of D+ holds t_cd + t_dc (the diagonal t_cc), row p - (i + 1) - s0 of D-
// (pairs i < j) holds t_cd - t_dc; each with its own row exponent.
struct PmRows {
    const double* X;
    int all_pairs;            // every pair (i, j) has both rows, in the order i o + j
    int o, v;
    long long q0, s0;         // first pair of this call in the enumeration, first strict pair
};

__global__ void __launch_bounds__(NT) crt_pm_f64_kernel(const PmRows a, int nm, unsigned short* __restrict__ Dp,
                                                        int* __restrict__ ep, long long rows_p,
                                                        unsigned short* __restrict__ Dm, int* __restrict__ em,
                                                        long long rows_m, long long pitch, int* __restrict__ status)
{
    __shared__ double S1[TT][TT + 1], S2[TT][TT + 1];
    __shared__ unsigned long long red[NT / 32 + 1];
    const uint32_t cs = cluster_size(), rank = cluster_rank();
    const long long r = blockIdx.x / cs;
    const int v = a.v;
    long long i = 0, j = 1;
    if (!a.all_pairs) tri_index(a.q0 + r, a.o, i, j);
    const double* X = a.X + (a.all_pairs ? r : i * a.o + j) * v * v;
    const bool minus = i < j && Dm != nullptr;
    const long long rm = a.all_pairs ? r : a.q0 + r - (i + 1) - a.s0;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int nt = (v + TT - 1) / TT, nb = crt_blocks(v);
    unsigned long long m1 = 0, m2 = 0;
    int e1 = 0, e2 = 0;
    // one walk over the row's tile pairs: its maxima, or (PUT) its residues
    auto walk = [&](auto PUT, bool half) {
        for (TilePair t(nt, (int)rank); t.ok(); t.skip((int)cs)) {
            __syncthreads();
#pragma unroll
            for (int y = 0; y < TT; y += NT / 32) {
                const int c = t.tc * TT + y + ty, d = t.td * TT + tx;
                S1[y + ty][tx] = (c < v && d < v) ? X[(long long)c * v + d] : 0.0;
                const int d2 = t.td * TT + y + ty, c2 = t.tc * TT + tx;
                S2[y + ty][tx] = (d2 < v && c2 < v) ? X[(long long)d2 * v + c2] : 0.0;
            }
            __syncthreads();
            const QuadPos pos(t, nb);
            if (!pos.live) continue;
            const int c = t.tc * TT + pos.cl, d0 = t.td * TT + pos.dl;
            long long xp[4], xm[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int d = d0 + q;
                const bool in = d >= c && d < v;
                double x1 = S1[pos.cl][pos.dl + q], x2 = S2[pos.dl + q][pos.cl];
                if (half) { x1 *= 0.5; x2 *= 0.5; }
                const double zp = !in ? 0.0 : (d == c ? x1 : x1 + x2);
                const double zm = (!in || d == c || !minus) ? 0.0 : x1 - x2;
                if (!PUT.value) {
                    const unsigned long long bp = (unsigned long long)__double_as_longlong(zp) & kAbs;
                    const unsigned long long bm = (unsigned long long)__double_as_longlong(zm) & kAbs;
                    m1 = bp > m1 ? bp : m1;
                    m2 = bm > m2 ? bm : m2;
                } else {
                    xp[q] = fixed_of(zp, e1);
                    xm[q] = fixed_of(zm, e2);
                }
            }
            if (PUT.value) {
                put_quad(xp, nm, Dp + r * pitch, rows_p * pitch, pos.k);
                if (minus) put_quad(xm, nm, Dm + rm * pitch, rows_m * pitch, pos.k);
            }
        }
    };
    auto maxima = [&](bool half) {
        m1 = m2 = 0;
        walk(std::false_type(), half);
        m1 = cluster_max(m1, red);
        cluster_done();
        m2 = cluster_max(m2, red);
        cluster_done();
    };
    maxima(false);
    // A finite row whose sums t_cd +- t_dc pass 2^1024 goes by halves (exact, or below the row's last bit).
    const bool half = a.all_pairs && (m1 >= kInf || m2 >= kInf);  // (the same for the whole cluster)
    if (half) maxima(true);
    e1 = exp_of_maxbits(m1);
    e2 = exp_of_maxbits(m2);
    if (rank == 0 && threadIdx.x == 0) {
        ep[r] = e1 + (half ? 1 : 0);
        if (minus) em[rm] = e2 + (half ? 1 : 0);
        // NaN or Inf in the row (or, where pair symmetry is promised, an overflowing sum)
        if (status && (m1 >= kInf || m2 >= kInf)) atomicOr(status, kStatusNonfinite);
    }
    walk(std::true_type(), half);
}

// V+ and V- of the integral rows (a, b >= a) of one block from the byte planes of the integral GEMM,
// planes[l][(al, c)][(b', d)], each element's fraction y scaled by 2^(eA[al v + c] + eB[b' v + d]) (the factor CrtRec::frac is left to the result).  Both halves share the row exponent E of the largest |V|,
// as Y = round(V 2^(43 - E)) (one guard bit), V+- = (Y1 +- Y2) / 4.
// Bound: arithmetic and HBM together (o=16/v=160/n=800: alu 50%, FP32/integer multiply 57%, issue 61%, HBM 53% of
// their peaks, 10 ps per element): twelve 96-bit products to put an element together, 13 residues to take it apart, 12 bytes
// read and 26 written.  The row's second walk finds it in L2 (2.7 GB read for 4.1 GB of planes).  o=40/v=400/n=2000: 342 ms
// with one CTA per row, 205 with 4 x 4 blocks in registers, 171 with entries in the order of c and d, 157 now.
struct PmPlanes {
    const unsigned char* planes;
    long long plane, pitch_in;  // bytes between planes, per GEMM row
    int all_b;                  // rows (al, all b'), else (al, b' >= al)
    int Nb, v;
    const int* eA;
    const int* eB;
    int diag;                   // b' < al + diag: V- of (b, a)
};

// Its static shared memory: 33.9 KB, so that the exponents beside it pass 48 KB from about v = 950 on (launch_rows).
struct PmTiles {
    long long S[2][2][TT][TT + 1];  // two buffers: one barrier per tile pair
    long long red[NT / 32 + 1];
};

template <bool AL, bool WIDE>
__global__ void __launch_bounds__(NT, 4) crt_pm_planes_kernel(const PmPlanes a, const CrtRec rec, int nm,
                                                           unsigned short* __restrict__ Dp, int* __restrict__ ep,
                                                           unsigned short* __restrict__ Dm, int* __restrict__ em,
                                                           long long rows, long long pitch)
{
    extern __shared__ __align__(16) int esm[];  // exponents of c and of d, then their codes (each padded to a multiple of four)
    __shared__ PmTiles tiles;
    long long (&S)[2][2][TT][TT + 1] = tiles.S;
    long long (&red)[NT / 32 + 1] = tiles.red;
    const uint32_t cs = cluster_size(), rank = cluster_rank();
    const long long r = blockIdx.x / cs;
    const int v = a.v, v4 = (v + 3) & ~3;
    long long al = r / a.Nb, bq = r % a.Nb;
    if (!a.all_b) tri_index(r, a.Nb, al, bq);
    const bool flip = bq < al + a.diag;
    int* eo = esm;
    int* ei = esm + v4;
    int* co = esm + 2 * v4;
    int* ci = esm + 3 * v4;
    int m1 = INT_MIN, m2 = INT_MIN;
    for (int q = threadIdx.x; q < v4; q += NT) {
        const int e1 = q < v ? a.eA[al * v + q] : 0, e2 = q < v ? a.eB[bq * v + q] : 0;
        eo[q] = e1;
        ei[q] = e2;
        if (q < v) { m1 = max(m1, e1); m2 = max(m2, e2); }
    }
    m1 = block_max(m1, (int*)red);
    m2 = block_max(m2, (int*)red);
    for (int q = threadIdx.x; q < v4; q += NT) {
        co[q] = exp_code(eo[q] - m1);
        ci[q] = exp_code(ei[q] - m2);
    }
    __syncthreads();
    const int emax = m1 + m2;
    const unsigned char* X = a.planes + al * v * a.pitch_in + bq * v;
    const int qy = threadIdx.x >> 3, qx = (threadIdx.x & 7) * 4;
    const int nt = (v + TT - 1) / TT, nb = crt_blocks(v);
    // walk 1: the row exponent
    const uint32_t qi = (uint32_t)v4 / 4, step = cs * NT, first = rank * NT + threadIdx.x;
    int code = INT_MIN;
    walk_quads<AL>(QuadIter(first, step, qi), (uint32_t)v, X, a.pitch_in, a.plane, rec.nm,
                   [&](uint32_t c, uint32_t i, const RawQuad<AL>& w) {
        const int d0 = (int)i * 4;
        int tp[4];
        w.tops(rec, tp);
        const int cc = co[c];
        const int4 cd = *reinterpret_cast<const int4*>(ci + d0);
        const int cds[4] = {cd.x, cd.y, cd.z, cd.w};
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (AL || d0 + j < v) code = max(code, top_code(tp[j], cc + cds[j]));
    });
    code = (int)cluster_max((long long)code, red);
    int E;
    if (!exponent_of(code, emax, rec.nm, E)) {  // (the same for the whole cluster)
        cluster_done();
        int mx = INT_MIN;
        for (QuadIter t(first, step, qi); t.o < (uint32_t)v; t.next()) {
            const int d0 = (int)t.i * 4;
            RawQuad<AL> w;
            w.load(X + (long long)t.o * a.pitch_in + d0, 0u, a.plane, rec.nm);
            long long y[4];
            w.template fractions<WIDE>(rec, y);
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (d0 + j < v && y[j] != 0)
                    mx = max(mx, 64 - __clzll(y[j] < 0 ? -y[j] : y[j]) + eo[t.o] + ei[d0 + j]);
        }
        E = (int)cluster_max((long long)mx, red);
    }
    const bool zero = E == INT_MIN;
    if (zero) E = 0;
    if (rank == 0 && threadIdx.x == 0) {
        ep[r] = E;
        if (em) em[r] = E;
    }
    const int s0 = E - kPlaneBits;        // Y = y 2^(e - s0)
    const bool fast = s0 - emax >= 0;     // every element is shifted right
    unsigned short* Pr = Dp + r * pitch;
    unsigned short* Mr = Dm ? Dm + r * pitch : nullptr;
    const long long stride = rows * pitch;
    // one 32 x 32 tile of Y at rows row0.., columns col0.. (zero beyond v)
    auto tile = [&](long long (&T)[TT][TT + 1], int row0, int col0) {
        const int c = row0 + qy, d0 = col0 + qx;
        long long y[4] = {0, 0, 0, 0};
        if (!zero && c < v && d0 < v) {
            RawQuad<AL> w;
            // (one tile's rows span less than 4 GB)
            w.load(X + (long long)row0 * a.pitch_in + col0, (uint32_t)qy * (uint32_t)a.pitch_in + (uint32_t)qx, a.plane, rec.nm);
            w.template fractions<WIDE>(rec, y);
            const int sc = s0 - eo[c];
            const int4 e4 = *reinterpret_cast<const int4*>(ei + d0);
            const int es[4] = {e4.x, e4.y, e4.z, e4.w};
            if (fast) {
#pragma unroll
                for (int j = 0; j < 4; ++j) y[j] = (AL || d0 + j < v) ? shr_fast(y[j], sc - es[j]) : 0;
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j) y[j] = (AL || d0 + j < v) ? shr_floor(y[j], sc - es[j]) : 0;
            }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) T[qy][qx + j] = y[j];
    };
    int buf = 0;
    for (TilePair t(nt, (int)rank); t.ok(); t.skip((int)cs), buf ^= 1) {
        long long (&S1)[TT][TT + 1] = S[buf][0];
        long long (&S2)[TT][TT + 1] = S[buf][t.tc == t.td ? 0 : 1];
        tile(S1, t.tc * TT, t.td * TT);
        if (t.tc != t.td) tile(S2, t.td * TT, t.tc * TT);
        __syncthreads();
        const QuadPos pos(t, nb);
        if (!pos.live) continue;
        unsigned long long u[2][4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            // (entries beyond v are zero in the tiles)
            const long long Y1 = S1[pos.cl][pos.dl + j], Y2 = S2[pos.dl + j][pos.cl];
            // Y is rounded down, by half a unit on average: the sum of two makes up for it with 1 more
            u[0][j] = (unsigned long long)((Y1 + Y2 + (long long)(4 * kCrtBias + 3)) >> 2);
            u[1][j] = (unsigned long long)(((flip ? Y2 - Y1 : Y1 - Y2) + (long long)(4 * kCrtBias + 2)) >> 2);
            const int c = t.tc * TT + pos.cl, d = t.td * TT + pos.dl + j;
            if (t.tc == t.td && d <= c) {
                u[0][j] = d == c ? (unsigned long long)((Y1 + (long long)(2 * kCrtBias + 1)) >> 1) : kCrtBias;
                u[1][j] = kCrtBias;
            }
        }
        if (Mr) {
            unsigned short* const o[2] = {Pr, Mr};
            const long long st[2] = {stride, stride};
            put_quads<2>(u, nm, o, st, pos.k);
        } else {
            const unsigned long long u1[1][4] = {{u[0][0], u[0][1], u[0][2], u[0][3]}};
            unsigned short* const o[1] = {Pr};
            const long long st[1] = {stride};
            put_quads<1>(u1, nm, o, st, pos.k);
        }
    }
    cluster_done();
}

// ------------------------------------------- plain rows from the planes of an intermediate
// Row r = (al, q), K = (o, i): the fractions of planes[l][(al outer + o)][q inner + i], scaled by
// 2^(eA[al outer + o] + eB[q inner + i]) (the factor CrtRec::frac is left to the result).
// Bound as crt_pm_planes: 9.3 ps per element (o=16/v=160/n=800, M1 of the adjoint: 4.1 TB/s); five CTAs per SM (10.0 ms for
// all splits of that adjoint with four, 10.7 with five) or clusters twice as wide (11.6) are slower.
struct PlaneRows {
    const unsigned char* planes;
    long long plane, pitch_in;
    long long rows;
    int nal, nq;      // r = al * nq + q, or q * nal + al (q_major)
    int q_major;
    int outer, inner;
    const int* eA;
    const int* eB;
};

template <bool AL, bool WIDE>
__global__ void __launch_bounds__(NT, 4) crt_rows_planes_kernel(const PlaneRows a, const CrtRec rec, int nm,
                                                             unsigned short* __restrict__ D, long long pitch,
                                                             int* __restrict__ e_out)
{
    __shared__ long long red[NT / 32 + 1];
    const uint32_t cs = cluster_size(), rank = cluster_rank();
    // rows of one al next to each other: their pieces of a GEMM row are neighbours and share its sectors (960 rows of
    // 480 pieces of 96 elements: 2.0 GB read before, 0.9 now, 0.53 without overlap; 515 -> 440 us)
    const long long al = blockIdx.x / cs / a.nq, qr = blockIdx.x / cs % a.nq;
    const long long r = a.q_major ? qr * a.nal + al : al * a.nq + qr;
    const unsigned char* X = a.planes + al * a.outer * a.pitch_in + qr * a.inner;
    const int* eo = a.eA + al * a.outer;
    const int* ei = a.eB + qr * a.inner;
    const uint32_t qi = (uint32_t)(a.inner + 3) / 4, step = cs * NT, first = rank * NT + threadIdx.x;
    int m1 = INT_MIN, m2 = INT_MIN;
    for (int q = threadIdx.x; q < a.outer; q += NT) m1 = max(m1, __ldg(eo + q));
    for (int q = threadIdx.x; q < a.inner; q += NT) m2 = max(m2, __ldg(ei + q));
    m1 = block_max(m1, (int*)red);
    m2 = block_max(m2, (int*)red);
    const int emax = m1 + m2;
    int code = INT_MIN;
    walk_quads<AL>(QuadIter(first, step, qi), (uint32_t)a.outer, X, a.pitch_in, a.plane, rec.nm,
                   [&](uint32_t oo, uint32_t i, const RawQuad<AL>& w) {
        const int i0 = (int)i * 4;
        int tp[4];
        w.tops(rec, tp);
        const int cc = exp_code(__ldg(eo + oo) - m1);
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (AL || i0 + j < a.inner) code = max(code, top_code(tp[j], cc + exp_code(__ldg(ei + i0 + j) - m2)));
    });
    code = (int)cluster_max((long long)code, red);
    int E;
    if (!exponent_of(code, emax, rec.nm, E)) {  // (the same for the whole cluster)
        cluster_done();
        int mx = INT_MIN;
        for (QuadIter t(first, step, qi); t.o < (uint32_t)a.outer; t.next()) {
            const int i0 = (int)t.i * 4;
            RawQuad<AL> w;
            w.load(X + (long long)t.o * a.pitch_in + i0, 0u, a.plane, rec.nm);
            long long y[4];
            w.template fractions<WIDE>(rec, y);
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (i0 + j < a.inner && y[j] != 0)
                    mx = max(mx, 64 - __clzll(y[j] < 0 ? -y[j] : y[j]) + __ldg(eo + t.o) + __ldg(ei + i0 + j));
        }
        E = (int)cluster_max((long long)mx, red);
    }
    const bool zero = E == INT_MIN;
    if (zero) E = 0;
    if (rank == 0 && threadIdx.x == 0) e_out[r] = E;
    const int s0 = E - kPlaneBits;         // twice X = y 2^(e + 42 - E), rounded down; then halved, rounded
    const bool fast = s0 - emax >= 0;
    unsigned short* Dr = D + r * pitch;
    const long long stride = a.rows * pitch;
    walk_quads<AL>(QuadIter(first, step, qi), (uint32_t)a.outer, X, a.pitch_in, a.plane, rec.nm,
                   [&](uint32_t oo, uint32_t i, const RawQuad<AL>& w) {
        const int i0 = (int)i * 4;
        long long y[4];
        w.template fractions<WIDE>(rec, y);
        const int sc = s0 - __ldg(eo + oo);
        unsigned long long u[1][4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int s = sc - ((AL || i0 + j < a.inner) ? __ldg(ei + i0 + j) : 0);
            const long long Y = fast ? shr_fast(y[j], s) : shr_floor(y[j], s);
            u[0][j] = (zero || !(AL || i0 + j < a.inner)) ? kCrtBias
                                                          : (unsigned long long)((Y + (long long)(2 * kCrtBias + 1)) >> 1);
        }
        unsigned short* const o[1] = {Dr};
        const long long st[1] = {stride};
        put_quads<1>(u, nm, o, st, (oo * qi + i) * 4);
    });
    cluster_done();
}

// ------------------------------------------------------------------- results
// r * 2^e, rounded once, over the whole range of doubles: the exponent goes into r's own, and what leaves the normal
// numbers goes through scalbn.  (As x * 2^e * factor the first product passed 2^1024 for results from 2^972 on, their factor
// being about 2^-51.)
__device__ __forceinline__ double times_pow2(double r, int e)
{
    const int ex = (__double2hiint(r) >> 20) & 0x7ff, to = ex + e;
    if (ex != 0 && to > 0 && to < 0x7ff) return __hiloint2double(__double2hiint(r) + (e << 20), __double2loint(r));
    return scalbn(r, e);
}

// Bound: HBM and L2, nm bytes read per split and 8 written (o=40/v=400/n=2000, four splits: 3.4 ms of 650).
// C[rmap(m) + cmap(n)] (= or +=) x(m, n) * 2^(eA[m] + eB[n] + base) * factor, x from the planes summed over the K splits.
// MFAST: m is the output's contiguous index (the GEMM ran on the transposed problem).
template <bool MFAST>
__global__ void __launch_bounds__(NT) crt_to_f64_kernel(int M, int N, const unsigned char* __restrict__ planes,
                                                        long long pitch, int nsplit, const CrtRec rec, const OutDesc out,
                                                        int base, double factor, const int* __restrict__ eA, const int* __restrict__ eB)
{
    __shared__ double S[TT][TT + 1];
    const int qy = threadIdx.x >> 3, qx = (threadIdx.x & 7) * 4;
    const long long plane = (long long)M * pitch;
    const int tiles_n = (N + TT - 1) / TT;
    const int m0 = (int)(blockIdx.x / tiles_n) * TT, n0 = (int)(blockIdx.x % tiles_n) * TT;
    const int m = m0 + qy;
    if (m < M && n0 + qx < N) {
        // (a split's bytes carry the offset once each: the other splits' are taken off here)
        CrtAcc<true> a[4] = {CrtAcc<true>(rec), CrtAcc<true>(rec), CrtAcc<true>(rec), CrtAcc<true>(rec)};
        for (int s = 0; s < nsplit; ++s) {
            if (s > 0)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    a[j].a0 += rec.b0;
                    a[j].a1 += rec.b1;
                    a[j].a2 += rec.b2;
                }
            const unsigned char* p = planes + (long long)s * rec.nm * plane + m * pitch + n0 + qx;
#pragma unroll
            for (int l = 0; l < kCrtMax; ++l) {
                if (l >= kCrtMin && l >= rec.nm) break;
                const uint32_t w = __ldg(reinterpret_cast<const uint32_t*>(p + l * plane));
#pragma unroll
                for (int j = 0; j < 4; ++j) a[j].add((w >> (8 * j)) & 255u, rec, l);
            }
        }
        const int em = eA[m] + base;
        const long long ro = MFAST ? 0 : map2(out.rmap, m);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int n = n0 + qx + j;
            if (n >= N) continue;
            const double x = times_pow2((double)crt_scale(a[j].fraction(), rec) * factor, em + eB[n]);
            if (MFAST) {
                S[qy][qx + j] = x;
            } else {
                double* c = out.C + ro + map2(out.cmap, n);
                *c = out.accumulate ? *c + x : x;
            }
        }
    }
    if (MFAST) {
        __syncthreads();
        const int mm = m0 + (int)(threadIdx.x & 31);
        if (mm >= M) return;
        const long long ro = map2(out.rmap, mm);
#pragma unroll
        for (int y = 0; y < TT; y += NT / 32) {
            const int n = n0 + y + (int)(threadIdx.x >> 5);
            if (n >= N) continue;
            double* c = out.C + ro + map2(out.cmap, n);
            const double x = S[threadIdx.x & 31][n - n0];
            *c = out.accumulate ? *c + x : x;
        }
    }
}

// Clusters per row: enough CTAs for the device when rows are few, and few enough rows in flight (about 450
// CTAs are resident) for one walk's bytes to stay in L2 for the next; every CTA keeps at least 2048 elements.
int cluster_for(long long rows, long long elems, long long bytes)
{
    int cs = 1;
    while (cs < 8 && elems / (2 * cs) >= 2048 && (rows * cs < 4ll * device_sm_count() || bytes * 450 / cs > (64ll << 20)))
        cs *= 2;
    return cs;
}

// smem: dynamic shared memory; fixed: the static part of a kernel that takes any, or a little more.
template <typename... KArgs, typename... Args>
cudaError_t launch_rows(void (*kern)(KArgs...), long long rows, int cs, size_t smem, size_t fixed, cudaStream_t st, Args... args)
{
    if (rows * cs > 0x7fffffffll) return cudaErrorInvalidConfiguration;
    // (a launch gets 48 KB unasked, static and dynamic together; always the same opt-in, so that threads with different v
    // do not take it from each other)
    if (smem + fixed > kMaxSmem) return cudaErrorInvalidValue;
    if (smem + fixed > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(kMaxSmem - fixed));
        if (e != cudaSuccess) return e;
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(rows * cs));
    cfg.blockDim = dim3(NT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)cs;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...);
    if (e != cudaSuccess) return e;
    count_launch();
    return cudaGetLastError();
}

}  // namespace

cudaError_t crt_rows(const RowSrc& src, int outer, int inner, long long ostride, int nm, void* D, long long pitch, int* e,
                     int* status, cudaStream_t st)
{
    if (src.rows <= 0) return cudaSuccess;
    if ((long long)outer * ((inner + 3) / 4) > 0x7fffffffll) return cudaErrorInvalidValue;
    const RowsArg a{src, ostride, outer, inner};
    const long long elems = (long long)outer * inner;
    if ((long long)outer * ((inner + 3) / 4) <= 32 * WQ)
        return launch_rows(crt_rows_warp_kernel, (src.rows + NT / 32 - 1) / (NT / 32), 1, 0, 0, st, a, nm, (unsigned short*)D,
                           pitch, e, status);
    return launch_rows(crt_rows_kernel, src.rows, cluster_for(src.rows, elems, 8 * elems), 0, 0, st, a, nm,
                       (unsigned short*)D, pitch, e, status);
}

cudaError_t crt_cols(const ColSrc& src, int nm, void* D, long long pitch, int* e, const unsigned long long* premax,
                     int* status, cudaStream_t st)
{
    if (src.rows <= 0) return cudaSuccess;
    const long long blocks = (src.rows + CR - 1) / CR;
    // few blocks of rows: K is spread over a cluster
    int cs = 1;
    while (cs < 8 && blocks * cs < 4ll * device_sm_count() && src.K > 2ll * CK * cs) cs *= 2;
    if (premax)
        return launch_rows(crt_cols_kernel<true>, blocks, cs, 0, 0, st, src, nm, premax, (unsigned short*)D, pitch, e, status);
    return launch_rows(crt_cols_kernel<false>, blocks, cs, 0, 0, st, src, nm, (const unsigned long long*)nullptr,
                       (unsigned short*)D, pitch, e, status);
}

cudaError_t crt_pm_f64(const double* t2, bool all_pairs, int o, int v, long long q0, long long rows_p, long long s0,
                       long long rows_m, int nm, void* Dp, int* ep, void* Dm, int* em, long long pitch, int* status,
                       cudaStream_t st)
{
    if (rows_p <= 0) return cudaSuccess;
    const PmRows a{t2, all_pairs ? 1 : 0, o, v, q0, s0};
    const long long elems = (long long)v * v;
    return launch_rows(crt_pm_f64_kernel, rows_p, cluster_for(rows_p, elems, 8 * elems), 0, 0, st, a, nm, (unsigned short*)Dp,
                       ep, rows_p, rows_m > 0 ? (unsigned short*)Dm : nullptr, em, rows_m, pitch, status);
}

cudaError_t crt_pm_planes(const CrtPlanes& src, bool all_b, long long rows, int Nb, int v, const int* eA,
                          const int* eB, int diag, int nm, void* Dp, int* ep, void* Dm, int* em, long long pitch, cudaStream_t st)
{
    if (rows <= 0) return cudaSuccess;
    const size_t smem = sizeof(int) * 4 * (size_t)((v + 3) & ~3);  // v up to about 12400 (one `a` of such a block is 20 TB)
    const PmPlanes a{src.planes, src.plane, src.pitch, all_b ? 1 : 0, Nb, v, eA, eB, diag};
    const CrtRec rec = crt_rec(src.nm);
    const long long elems = (long long)v * v;
    const int cs = cluster_for(rows, elems, src.nm * elems);
    const bool al = v % 4 == 0 && src.pitch % 4 == 0 && src.plane % 4 == 0, wide = src.nm > 12;
    return launch_rows(al ? (wide ? crt_pm_planes_kernel<true, true> : crt_pm_planes_kernel<true, false>)
                          : (wide ? crt_pm_planes_kernel<false, true> : crt_pm_planes_kernel<false, false>),
                       rows, cs, smem, sizeof(PmTiles) + 1024, st, a, rec, nm, (unsigned short*)Dp, ep, (unsigned short*)Dm, em, rows, pitch);
}

cudaError_t crt_rows_planes(const CrtPlanes& src, int nal, int nq, bool q_major, int outer, int inner, const int* eA,
                            const int* eB, int nm, void* D, long long pitch, int* e, cudaStream_t st)
{
    const long long rows = (long long)nal * nq;
    if (rows <= 0) return cudaSuccess;
    if ((long long)outer * ((inner + 3) / 4) > 0x7fffffffll) return cudaErrorInvalidValue;
    const PlaneRows a{src.planes, src.plane, src.pitch, rows, nal, nq, q_major ? 1 : 0, outer, inner, eA, eB};
    const CrtRec rec = crt_rec(src.nm);
    const long long elems = (long long)outer * inner;
    const int cs = cluster_for(rows, elems, src.nm * elems);
    const bool al = inner % 4 == 0 && src.pitch % 4 == 0 && src.plane % 4 == 0, wide = src.nm > 12;
    return launch_rows(al ? (wide ? crt_rows_planes_kernel<true, true> : crt_rows_planes_kernel<true, false>)
                          : (wide ? crt_rows_planes_kernel<false, true> : crt_rows_planes_kernel<false, false>),
                       rows, cs, 0, 0, st, a, rec, nm, (unsigned short*)D, pitch, e);
}

cudaError_t crt_to_f64(int M, int N, const CrtPlanes& src, int nsplit, const OutDesc& out, int base, double factor,
                       bool mfast, const int* eA, const int* eB, cudaStream_t st)
{
    if (M <= 0 || N <= 0) return cudaSuccess;
    const long long tiles = (long long)((M + TT - 1) / TT) * ((N + TT - 1) / TT);
    if (tiles > 0x7fffffffll) return cudaErrorInvalidConfiguration;
    const CrtRec rec = crt_rec(src.nm);
    if (mfast)
        crt_to_f64_kernel<true><<<(unsigned)tiles, NT, 0, st>>>(M, N, src.planes, src.pitch, nsplit, rec, out, base, factor, eA, eB);
    else
        crt_to_f64_kernel<false><<<(unsigned)tiles, NT, 0, st>>>(M, N, src.planes, src.pitch, nsplit, rec, out, base, factor, eA, eB);
    count_launch();
    return cudaGetLastError();
}

}  // namespace cc
