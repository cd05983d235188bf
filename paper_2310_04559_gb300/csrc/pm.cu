// pm.cu -- symmetric / antisymmetric packing of the pair-symmetric ladder.
//
// For amplitudes with t[i,j,c,d] = t[j,i,d,c] the ladder term splits into a part
// symmetric and a part antisymmetric under c <-> d (closed-shell CC codes call these
// the t+ / t- amplitudes).  With V_ab[c,d] = (ac|bd) (Eq. 5) and, for c < d,
//
//     T+[ij][c<=d] = t_ijcd + t_ijdc  (t_ijcc on the diagonal)
//     T-[ij][c< d] = t_ijcd - t_ijdc
//     V+[ab][c<=d] = (V_ab[c,d] + V_ab[d,c]) / 2  (V_ab[c,c] on the diagonal)
//     V-[ab][c< d] = (V_ab[c,d] - V_ab[d,c]) / 2
//
// the sum of Eq. 6 is  sum_cd t_ijcd V_ab[c,d] = R+_ijab + R-_ijab  with
// R+ = sum_{c<=d} T+ V+ and R- = sum_{c<d} T- V-.  Because (ac|bd) = (bd|ac),
// V+ is symmetric and V- antisymmetric under a <-> b; T+ is symmetric and T-
// antisymmetric under i <-> j.  Hence R+ is needed for i <= j, a <= b only, R-
// for i < j, a < b only, and
//
//     R[i,j,a,b] = R[j,i,b,a] = R+ + R-,    R[j,i,a,b] = R[i,j,b,a] = R+ - R-.
//
// The two ladder GEMMs then have K = v(v+1)/2 and v(v-1)/2 and about o^2/2 rows,
// a quarter of the unpacked product each.  Packed column index of (c, d):
//     kp(c,d) = c*v - c(c-1)/2 + (d - c)       (c <= d, v(v+1)/2 entries)
//     km(c,d) = c*(v-1) - c(c-1)/2 + (d - c - 1)  (c < d, v(v-1)/2 entries)
//
// Rows of the integral block used here are the pairs (a, b) with b >= a of a block
// a0 <= a < a0 + A, b in [a0, v): packed row r = rowbase(al) + (b' - al) with
// al = a - a0, b' = b - a0, Nb = v - a0 and rowbase(al) = al*Nb - al(al-1)/2.
//
// Every v x v matrix is visited as pairs of 32 x 32 tiles (C, D) and (D, C) staged
// in shared memory, so that X[c][d] and X[d][c] are both read coalesced.
#include <cuda_bf16.h>

#include <cfloat>
#include <climits>
#include <type_traits>

#include "cc_internal.cuh"

namespace cc {
namespace {

constexpr int TT = 32;   // tile edge
constexpr int TY = 8;    // thread rows per tile (256 threads)
constexpr unsigned long long kAbs = 0x7fffffffffffffffull;

__device__ __forceinline__ long long kp_of(long long c, long long d, long long v) { return c * v - c * (c - 1) / 2 + (d - c); }
__device__ __forceinline__ long long km_of(long long c, long long d, long long v)
{
    return c * (v - 1) - c * (c - 1) / 2 + (d - c - 1);
}

// bf16 bit pattern of a small integer (|d| <= 256, exact): the float 1.5*2^23 + d has unit
// spacing, so subtracting 1.5*2^23 gives d exactly, and d has at most 8 significant bits.
__device__ __forceinline__ unsigned short bf16_small(int d)
{
    return (unsigned short)(__float_as_uint(__int_as_float(0x4B400000 + d) - 12582912.0f) >> 16);
}

// H = half * sum_{k<s} 2^(beta k): X + H holds the balanced digits of X plus `half` each as
// plain base-2^beta digits (no carries to propagate), for |X| <= 2^(beta s - 1) < H.
__device__ __forceinline__ long long digit_bias(int s, int beta)
{
    long long H = 0;
    for (int k = 0; k < s; ++k) H = (H << beta) | (1ll << (beta - 1));
    return H;
}

// Balanced base-2^beta digits of X (d_0 most significant) as bf16, same convention as
// the row splits: x ~= sum_k d_k 2^(e - beta + 1 - beta k) for X = round(x 2^(beta s - 1 - e)).
__device__ __forceinline__ void put_digits(long long X, long long H, int s, int beta, __nv_bfloat16* out,
                                           long long stride)
{
    const unsigned long long Y = (unsigned long long)(X + H);
    const int half = 1 << (beta - 1), mask = (1 << beta) - 1;
    unsigned short* o = (unsigned short*)out;
    o[0] = bf16_small((int)(Y >> (beta * (s - 1))) - half);
#pragma unroll
    for (int k = 1; k < 8; ++k) {
        if (k >= s) break;
        o[k * stride] = bf16_small(((int)(Y >> (beta * (s - 1 - k))) & mask) - half);
    }
}

// X * 2^sh rounded to an integer (round half up on right shifts).
__device__ __forceinline__ long long shr_round(long long X, int sh)
{
    if (sh >= 0) return X << sh;
    if (sh <= -63) return 0;
    return (X + (1ll << (-sh - 1))) >> (-sh);
}

// round(x * 2^(total - 1 - e)) from the bit pattern of x (|x| < 2^e).
__device__ __forceinline__ long long fixed_of(double x, int e, int total)
{
    const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
    const int ex = (int)((bits >> 52) & 0x7ff);
    unsigned long long mant = bits & 0x000fffffffffffffull;
    if (ex == 0 && mant == 0) return 0;
    int exe = ex;
    if (ex == 0) exe = 1; else mant |= 0x0010000000000000ull;
    const int sh = exe - 1075 + total - 1 - e;
    long long X;
    if (sh >= 0) X = (long long)(mant << sh);
    else if (sh > -64) X = (long long)((mant + (1ull << (-sh - 1))) >> (-sh));
    else X = 0;
    return (bits >> 63) ? -X : X;
}

__device__ __forceinline__ int exp_of_maxbits(unsigned long long b)
{
    if (b == 0) return 0;
    const int ex = (int)(b >> 52);
    return ex == 0 ? -1022 : ex - 1022;
}

__device__ __forceinline__ float tf32_round(float f)
{
    unsigned int u;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(u) : "f"(f));
    return __uint_as_float(u);
}
__device__ __forceinline__ float tf32_of(double x) { return tf32_round((float)x); }

__device__ __forceinline__ unsigned long long block_max_u64(unsigned long long m, unsigned long long* red)
{
    for (int w = 16; w > 0; w >>= 1) {
        const unsigned long long o = __shfl_xor_sync(0xffffffffu, m, w);
        m = o > m ? o : m;
    }
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
    __syncthreads();
    unsigned long long r = red[0];
    for (int w = 1; w < 8; ++w) r = red[w] > r ? red[w] : r;
    return r;
}

// Value of the packed entry (c, d) of one sign from x1 = X[c][d], x2 = X[d][c].
__device__ __forceinline__ double pm_value(double x1, double x2, bool diag, int sign, double h)
{
    if (diag) return x1;
    return sign > 0 ? (x1 + x2) * h : (x1 - x2) * h;
}

// FP64 source: one row r is the v x v matrix at X + rowtab[r] * rowmul (rowtab NULL: r * rowmul).
// kind: 0 = Ozaki digits (s slices, exponent per row), 1 = bf16 copy (e = 0), 2 = tf32 copy,
// 3 = FP64 copy.
__global__ void pm_f64_kernel(const double* __restrict__ X0, const long long* __restrict__ rowtab, long long rowmul,
                              int v, int sign, double h, int kind, int s, int beta, void* __restrict__ D,
                              long long pitch, long long rows, int* __restrict__ e_out, int* __restrict__ status)
{
    __shared__ double S1[TT][TT + 1], S2[TT][TT + 1];
    __shared__ unsigned long long red[8];
    const long long r = blockIdx.x;
    const double* X = X0 + (rowtab ? rowtab[r] : r) * rowmul;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int nt = (v + TT - 1) / TT;
    const long long vv = v;
    const long long slice_stride = rows * pitch;
    const int total = beta * s;
    const long long H = kind == 0 ? digit_bias(s, beta) : 0;
    int e = 0;
    for (int pass = (kind == 0 ? 0 : 1); pass < 2; ++pass) {
        unsigned long long mx = 0;
        for (int tc = 0; tc < nt; ++tc) {
            for (int td = tc; td < nt; ++td) {
                __syncthreads();
                for (int y = ty; y < TT; y += TY) {
                    const int c = tc * TT + y, d = td * TT + tx;
                    S1[y][tx] = (c < v && d < v) ? X[c * vv + d] : 0.0;
                    const int d2 = td * TT + y, c2 = tc * TT + tx;
                    S2[y][tx] = (d2 < v && c2 < v) ? X[d2 * vv + c2] : 0.0;
                }
                __syncthreads();
                for (int y = ty; y < TT; y += TY) {
                    const int c = tc * TT + y, d = td * TT + tx;
                    if (c >= v || d >= v || d < c || (sign < 0 && d == c)) continue;
                    const double z = pm_value(S1[y][tx], S2[tx][y], c == d, sign, h);
                    const long long k = sign > 0 ? kp_of(c, d, vv) : km_of(c, d, vv);
                    if (pass == 0) {
                        const unsigned long long b = (unsigned long long)__double_as_longlong(z) & kAbs;
                        mx = b > mx ? b : mx;
                    } else if (kind == 0) {
                        put_digits(fixed_of(z, e, total), H, s, beta, (__nv_bfloat16*)D + r * pitch + k, slice_stride);
                    } else if (kind == 1) {
                        ((__nv_bfloat16*)D)[r * pitch + k] = __double2bfloat16(z);
                    } else if (kind == 3) {
                        ((double*)D)[r * pitch + k] = z;
                    } else {
                        ((float*)D)[r * pitch + k] = tf32_of(z);
                    }
                }
            }
        }
        if (pass == 0) {
            const unsigned long long bm = block_max_u64(mx, red);
            e = exp_of_maxbits(bm);
            // NaN or Inf in the row (or an overflowing sum t_cd + t_dc): flag the call
            if (threadIdx.x == 0 && status && bm >= 0x7ff0000000000000ull) atomicOr(status, kStatusNonfinite);
        }
    }
    if (threadIdx.x == 0 && e_out) e_out[r] = e;
}

// Int64 fixed-point integral block (output of the integral GEMM kept as int64): packed
// row r is the unpacked row ru = rtab[r], X[c][d] = V[ru*ldx + c*v + d] * 2^(eo[c] + ei[d]
// + base) with eo = eA + amap(ru), ei = eB + bmap(ru).  Writes V+ and V- digits with one
// shared row exponent E (max |V| < 2^E bounds both halves).  Integer arithmetic only.
__global__ void pm_fixed_kernel(const PmFixedSrc src, int s, int beta, __nv_bfloat16* __restrict__ Dp,
                                long long pitchp, int* __restrict__ ep, __nv_bfloat16* __restrict__ Dm,
                                long long pitchm, int* __restrict__ em)
{
    extern __shared__ int esm[];  // eo[v], ei[v]
    __shared__ long long S1[TT][TT + 1], S2[TT][TT + 1];
    __shared__ int redi[8];
    const long long r = blockIdx.x;
    const long long ru = src.rtab[r];
    const int v = src.v;
    const long long vv = v;
    const long long ab = map2(src.amap, ru), bb = map2(src.bmap, ru);
    for (int q = threadIdx.x; q < v; q += 256) {
        esm[q] = src.eA[ab + q];
        esm[v + q] = src.eB[bb + q];
    }
    __syncthreads();
    const int* eo = esm;
    const int* ei = esm + v;
    const long long* X = src.X + ru * src.ldx;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // pass 1: E = max over the row of bitlength(|X|) + exponent, so max |V| < 2^E
    int mx = INT_MIN;
    for (int c = warp; c < v; c += 8) {
        const long long* Xc = X + c * vv;
        const int ec = eo[c];
#pragma unroll 4
        for (int d = lane; d < v; d += 32) {
            const long long x = __ldcs(Xc + d);
            const unsigned long long ax = x < 0 ? (unsigned long long)(-x) : (unsigned long long)x;
            const int b = x ? 64 - __clzll((long long)ax) + ec + ei[d] : INT_MIN;
            mx = b > mx ? b : mx;
        }
    }
    for (int w = 16; w > 0; w >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, w));
    if (lane == 0) redi[warp] = mx;
    __syncthreads();
    int m = redi[0];
    for (int w = 1; w < 8; ++w) m = max(m, redi[w]);
    const bool zero = m == INT_MIN;
    const int E = zero ? 0 : m + src.base;
    if (threadIdx.x == 0) {
        ep[r] = E;
        if (em) em[r] = E;
    }
    // pass 2: Y = round(V * 2^(total - E)) (one guard bit), V+- = (Y1 +- Y2) / 4 at the
    // digit scale 2^(total - 1 - E); the diagonal of V+ is Y1 / 2.  Tile pairs (tc <= td)
    // in order; the next pair's loads are issued before the current pair is split.
    const int total = beta * s;
    const long long H = digit_bias(s, beta);
    const int tx = lane, ty = warp;
    const int nt = (v + TT - 1) / TT;
    const long long sp = src.rows * pitchp, sm = src.rows * pitchm;
    const int sh0 = src.base + total - E;
    long long q1[TT / TY], q2[TT / TY];
    auto fetch = [&](int tc, int td) {
#pragma unroll
        for (int u = 0; u < TT / TY; ++u) {
            const int y = ty + u * TY;
            const int c = tc * TT + y, d = td * TT + tx;
            q1[u] = (!zero && c < v && d < v) ? __ldcs(X + c * vv + d) : 0;
            const int d2 = td * TT + y, c2 = tc * TT + tx;
            q2[u] = (!zero && d2 < v && c2 < v) ? __ldcs(X + d2 * vv + c2) : 0;
        }
    };
    int tc = 0, td = 0;
    fetch(0, 0);
    while (tc < nt) {
        __syncthreads();
#pragma unroll
        for (int u = 0; u < TT / TY; ++u) {
            S1[ty + u * TY][tx] = q1[u];
            S2[ty + u * TY][tx] = q2[u];
        }
        __syncthreads();
        int nc = tc, nd = td + 1;
        if (nd == nt) { ++nc; nd = nc; }
        if (nc < nt) fetch(nc, nd);
        for (int y = ty; y < TT; y += TY) {
            const int c = tc * TT + y, d = td * TT + tx;
            if (c >= v || d >= v || d < c) continue;
            const long long Y1 = shr_round(S1[y][tx], eo[c] + ei[d] + sh0);
            if (c == d) {
                put_digits((Y1 + 1) >> 1, H, s, beta, Dp + r * pitchp + kp_of(c, d, vv), sp);
            } else {
                const long long Y2 = shr_round(S2[tx][y], eo[d] + ei[c] + sh0);
                put_digits((Y1 + Y2 + 2) >> 2, H, s, beta, Dp + r * pitchp + kp_of(c, d, vv), sp);
                if (Dm) put_digits((Y1 - Y2 + 2) >> 2, H, s, beta, Dm + r * pitchm + km_of(c, d, vv), sm);
            }
        }
        tc = nc;
        td = nd;
    }
}

// Whether a bf16 rounding of h may differ from that of the number h stands for: h is next to, or exactly, the middle of two
// bf16 numbers (about one number in 22000).
__device__ __forceinline__ bool near_bf16_tie(float h) { return ((__float_as_uint(h) - 0x7fffu) & 0xffffu) <= 2u; }

// Integral block of the mixed modes in FP32 (the integral GEMM's own sums): V+ and V- of one row in one walk over its
// tile pairs, 4 bytes read and 2 (4) written per element.  Bound: HBM.  A row's tile pairs are shared by `share` CTAs,
// so that few rows are in flight: the 128-byte pieces of a tile start anywhere, and the sectors that two
// neighbouring tiles share are read once only if they are still in L2 when the second tile comes.  With one CTA per
// row and streaming loads 1.7 times the block was read; o=27/v=301/n=1501 in BF16 took 9.09 ms for the split, plain loads
// 7.66, 2 / 4 / 8 / 16 CTAs per row 6.74 / 6.16 / 5.96 / 6.23 (o=20/v=200/n=1000 in TF32: 2.38, 1.99, 1.86 / 1.73 / 1.61 / 1.71).
template <bool BF16>
__global__ void __launch_bounds__(TT * TY) pm_f32_kernel(const float* __restrict__ X0, long long ldx,
                                                         const long long* __restrict__ rtab, int Nb, int v,
                                                         void* __restrict__ Dp, long long pitchp, int* __restrict__ ep,
                                                         void* __restrict__ Dm, long long pitchm, int* __restrict__ em,
                                                         int share)
{
    typedef typename std::conditional<BF16, unsigned short, float>::type out_t;
    __shared__ float S[2][2][TT][TT + 1];  // two buffers: one barrier per tile pair
    const long long r = blockIdx.x / share;
    const long long ru = rtab[r];
    const float* X = X0 + (ru / Nb) * v * ldx + (ru % Nb) * v;
    out_t* P = (out_t*)Dp + r * pitchp;
    out_t* M = Dm ? (out_t*)Dm + r * pitchm : nullptr;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int nt = (v + TT - 1) / TT;
    const uint32_t ld = (uint32_t)ldx;  // (a tile's rows span less than 2^32 elements)
    // tile pairs (tc, td >= tc) in order, every share-th one
    int buf = 0, tc = 0, td = (int)(blockIdx.x % share);
    auto settle = [&] { while (tc < nt && td >= nt) { ++tc; td += tc - nt; } };
    settle();
    float q1[TT / TY], q2[TT / TY];
    auto fetch = [&](int c0, int d0) {
        const float* X1 = X + (long long)c0 * ldx + d0;
        const float* X2 = X + (long long)d0 * ldx + c0;
        if (d0 + TT <= v) {
#pragma unroll
            for (int u = 0; u < TT / TY; ++u) {
                const uint32_t o = (uint32_t)(ty + u * TY) * ld + (uint32_t)tx;
                q1[u] = __ldg(X1 + o);
                q2[u] = __ldg(X2 + o);
            }
        } else {
#pragma unroll
            for (int u = 0; u < TT / TY; ++u) {
                const int y = ty + u * TY;
                const uint32_t o = (uint32_t)y * ld + (uint32_t)tx;
                q1[u] = (c0 + y < v && d0 + tx < v) ? __ldg(X1 + o) : 0.0f;
                q2[u] = (d0 + y < v && c0 + tx < v) ? __ldg(X2 + o) : 0.0f;
            }
        }
    };
    for (; tc < nt; buf ^= 1) {
        const int c0 = tc * TT, d0 = td * TT;
        float (&S1)[TT][TT + 1] = S[buf][0];
        float (&S2)[TT][TT + 1] = S[buf][1];
        fetch(c0, d0);
#pragma unroll
        for (int u = 0; u < TT / TY; ++u) {
            S1[ty + u * TY][tx] = q1[u];
            S2[ty + u * TY][tx] = q2[u];
        }
        td += share;
        settle();
        // tf32: sums of numbers from 2^126 on may leave FP32's range before they are halved.  A tile pair that holds such a
        // number goes through FP64 as a whole (a test per element cost 1% of o=20/v=200/n=1000 in TF32).
        bool huge = false;
        if (BF16) {
            __syncthreads();
        } else {
            float top = 0.0f;
#pragma unroll
            for (int u = 0; u < TT / TY; ++u) top = fmaxf(top, fmaxf(fabsf(q1[u]), fabsf(q2[u])));
            huge = __syncthreads_or(top >= 0.25f * FLT_MAX);
        }
        auto put = [&](int y, bool diag) {
            const int c = c0 + y, d = d0 + tx;
            const float x1 = S1[y][tx], x2 = S2[tx][y];
            // packed positions kp_of and km_of (c, d)
            const uint32_t kp = (uint32_t)c * (uint32_t)v - (uint32_t)c * (uint32_t)(c - 1) / 2 - (uint32_t)c + (uint32_t)d;
            const uint32_t km = kp - (uint32_t)c - 1;
            if (BF16) {
                // A sum of halves: within a unit of FP32 of V+- (a half may lose a bit among the denormals), so only next to
                // a tie is the rounding to bf16 left to FP64.
                const float h1 = 0.5f * x1, h2 = 0.5f * x2;
                const float vp = diag && c == d ? x1 : __fadd_rn(h1, h2), vm = __fsub_rn(h1, h2);
                __nv_bfloat162 h = __floats2bfloat162_rn(vp, vm);
                if (near_bf16_tie(vp) | near_bf16_tie(vm)) {
                    const double y1 = x1, y2 = x2;
                    h = __nv_bfloat162(__double2bfloat16(diag && c == d ? y1 : 0.5 * (y1 + y2)), __double2bfloat16(0.5 * (y1 - y2)));
                }
                const uint32_t w = *reinterpret_cast<const uint32_t*>(&h);
                P[kp] = (out_t)(w & 0xffffu);
                if (M && !(diag && c == d)) M[km] = (out_t)(w >> 16);
            } else {
                // (FP64 sums of two FP32 values round to the same FP32 as the FP32 sum)
                P[kp] = (out_t)tf32_round(diag && c == d ? x1 : 0.5f * __fadd_rn(x1, x2));
                if (M && !(diag && c == d)) M[km] = (out_t)tf32_round(0.5f * __fsub_rn(x1, x2));
            }
        };
        if (!BF16 && huge) {
            for (int y = ty; y < TT; y += TY) {
                const int c = c0 + y, d = d0 + tx;
                if (c >= v || d >= v || d < c) continue;
                const double x1 = S1[y][tx], x2 = S2[tx][y];
                P[kp_of(c, d, v)] = (out_t)tf32_of(c == d ? x1 : 0.5 * (x1 + x2));
                if (M && d > c) M[km_of(c, d, v)] = (out_t)tf32_of(0.5 * (x1 - x2));
            }
        } else if (c0 < d0 && d0 + TT <= v) {
#pragma unroll
            for (int u = 0; u < TT / TY; ++u) put(ty + u * TY, false);
        } else {
#pragma unroll
            for (int u = 0; u < TT / TY; ++u) {
                const int y = ty + u * TY;
                if (c0 + y < v && d0 + tx < v && d0 + tx >= c0 + y) put(y, true);
            }
        }
    }
    if (threadIdx.x == 0 && blockIdx.x % share == 0) {
        if (ep) ep[r] = 0;
        if (em) em[r] = 0;
    }
}

// rtab[rowbase(al) + b' - al] = al * Nb + b' for b' in [al, Nb)
__global__ void fill_rtab_kernel(int Ab, int Nb, long long* __restrict__ rtab)
{
    const int al = blockIdx.x;
    const long long base = (long long)al * Nb - (long long)al * (al - 1) / 2;
    for (int b = al + threadIdx.x; b < Nb; b += blockDim.x) rtab[base + (b - al)] = (long long)al * Nb + b;
}

__device__ __forceinline__ void pair_ij(int o, int p, int& i, int& j)
{
    int ii = 0, rem = p;
    while (rem >= o - ii) { rem -= o - ii; ++ii; }
    i = ii;
    j = ii + rem;
}

// R from R+ (rows: pairs q0 <= p < q1, i <= j) and R- (rows: their pairs i < j, from strict index
// s0) of one block; columns are packed rows r (al, b' >= al).  Grid: x = tile (al, b'), y + z gridDim.y = pair p - q0.
// GEN: amplitudes without pair symmetry, every pair p = i o + j has its own R+ and R- row and writes R[p] only.
// A 32 x 32 tile (al, b') is written as it is and, through shared memory, transposed, so that both halves of R are
// written along the last index (entry by entry, the transposed half took host-resident R 4.3 ms of 19 at o=30, v=150,
// 8 bytes per write over the host link).
//
// Not finite: R+ and R- can overflow, or be two infinities of which one sum is NaN, where the plain product is neither
// (an infinite amplitude, or t_cd + t_dc beyond 2^1024).  With PLAIN (GEN in FP64) such entries are the plain product of the
// block's integrals and the amplitudes, by the entry's whole warp.
__device__ __forceinline__ double plain_product(const double* __restrict__ V, const double* __restrict__ T, int v, bool swap, int lane)
{
    double s = 0.0;
    for (int c = 0; c < v; ++c)
        for (int d = lane; d < v; d += 32) s = fma(V[swap ? (long long)d * v + c : (long long)c * v + d], T[(long long)c * v + d], s);
    for (int w = 16; w > 0; w >>= 1) s += __shfl_xor_sync(0xffffffffu, s, w);
    return s;
}

template <bool GEN, bool PLAIN>
__global__ void pm_combine_kernel(int o, int v, int a0, int Ab, int Nb, long long nr, long long np, long long q0,
                                  long long s0, const double* __restrict__ Rp, const double* __restrict__ Rm,
                                  double* __restrict__ R, int accumulate, const double* __restrict__ V,
                                  const double* __restrict__ T)
{
    __shared__ double E1[TT][TT + 1], E2[TT][TT + 1];
    const long long pl = (long long)blockIdx.y + (long long)blockIdx.z * gridDim.y;
    if (pl >= np) return;  // uniform over the block
    const int ntb = (Nb + TT - 1) / TT;
    const int ta = (int)(blockIdx.x / ntb) * TT, tb = (int)(blockIdx.x % ntb) * TT;
    if (tb + TT - 1 < ta) return;  // b' < al throughout
    int i = 0, j = 1;
    if (!GEN) pair_ij(o, (int)(q0 + pl), i, j);
    const long long vv = (long long)v * v;
    double* Rij = R + (GEN ? pl : (long long)i * o + j) * vv;
    double* Rji = GEN ? Rij : R + ((long long)j * o + i) * vv;
    const double* rp = Rp + pl * nr;
    const double* rm = GEN ? (Rm ? Rm + pl * nr : nullptr)
                           : ((i < j && Rm) ? Rm + (q0 + pl - (i + 1) - s0) * nr : nullptr);  // row among the pairs i < j
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    auto put = [&](double* p, double x) { *p = accumulate ? *p + x : x; };
#pragma unroll
    for (int y = ty; y < TT; y += TY) {
        const int al = ta + y, bq = tb + tx;
        const bool in = al < Ab && bq < Nb && bq >= al;
        const long long r = (long long)al * Nb - (long long)al * (al - 1) / 2 + (bq - al);
        const double plus = in ? rp[r] : 0.0;
        const double minus = (in && rm && bq != al) ? rm[r] : 0.0;
        double e1 = plus + minus, e2 = plus - minus;
        if (PLAIN) {
            for (unsigned bad = __ballot_sync(0xffffffffu, in && !(isfinite(e1) && isfinite(e2))); bad; bad &= bad - 1) {
                const int q = __ffs(bad) - 1;
                const double* row = V + ((long long)al * Nb + tb + q) * vv;
                const double x1 = plain_product(row, T + pl * vv, v, false, tx), x2 = plain_product(row, T + pl * vv, v, true, tx);
                if (tx == q) { e1 = x1; e2 = x2; }
            }
        }
        if (!in) continue;
        E1[y][tx] = e1;
        E2[y][tx] = e2;
        const long long ab = (long long)(a0 + al) * v + a0 + bq;
        put(Rij + ab, e1);
        if (!GEN && i != j && al != bq) put(Rji + ab, e2);
    }
    __syncthreads();
#pragma unroll
    for (int y = ty; y < TT; y += TY) {
        const int bq = tb + y, al = ta + tx;
        if (al >= Ab || bq >= Nb || bq < al) continue;
        const long long ba = (long long)(a0 + bq) * v + a0 + al;
        if (GEN) {
            if (al != bq) put(Rij + ba, E2[tx][y]);
        } else {
            if (i != j || al != bq) put(Rji + ba, E1[tx][y]);
            if (i != j && al != bq) put(Rij + ba, E2[tx][y]);
        }
    }
}

// Rows (al, all b) of a range of `a`: see pm_combine_rows.
__global__ void pm_combine_rows_kernel(long long np, int v, int a0, long long nr, const double* __restrict__ Rp,
                                       const double* __restrict__ Rm, double* __restrict__ R, int accumulate)
{
    const long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= nr) return;
    const int a = a0 + (int)(r / v), b = (int)(r % v);
    for (long long p = blockIdx.y; p < np; p += gridDim.y) {
        const double plus = Rp[p * nr + r], minus = Rm && a != b ? Rm[p * nr + r] : 0.0;
        double* dst = R + p * ((long long)v * v) + (long long)a0 * v + r;
        const double e = b < a ? plus - minus : plus + minus;
        *dst = accumulate ? *dst + e : e;
    }
}

// tab[q] = (i*o + j) * v*v for the pairs i < j (strict) or i <= j, i-major.
__global__ void fill_pairs_kernel(int o, int v, int strict, long long* __restrict__ tab)
{
    const int i = blockIdx.x;
    const long long vv = (long long)v * v;
    const long long base = strict ? (long long)i * (o - 1) - (long long)i * (i - 1) / 2
                                  : (long long)i * o - (long long)i * (i - 1) / 2;
    for (int j = i + strict + threadIdx.x; j < o; j += blockDim.x)
        tab[base + (j - i - strict)] = ((long long)i * o + j) * vv;
}

}  // namespace

cudaError_t pm_split_f64(const double* X, const long long* rowtab, long long rowmul, long long rows, int v, int sign,
                         double h, int kind, int s, int beta, void* D, long long pitch, int* e, int* status,
                         cudaStream_t st)
{
    if (rows <= 0) return cudaSuccess;
    if (v < 1 || (sign < 0 && v < 2)) return cudaErrorInvalidValue;
    if (kind == 0 && (s < 1 || s > 8 || beta < 2 || beta > 9 || beta * s > 62)) return cudaErrorInvalidValue;
    if (rows > 0x7fffffffll) return cudaErrorInvalidValue;
    pm_f64_kernel<<<(unsigned)rows, 256, 0, st>>>(X, rowtab, rowmul, v, sign, h, kind, s, beta, D, pitch, rows, e,
                                                   status);
    count_launch();
    return cudaGetLastError();
}

cudaError_t pm_split_fixed(const PmFixedSrc& src, int s, int beta, void* Dp, long long pitchp, int* ep, void* Dm,
                           long long pitchm, int* em, cudaStream_t st)
{
    if (src.rows <= 0) return cudaSuccess;
    if (s < 1 || s > 8 || beta < 2 || beta > 9 || beta * s > 62 || src.v < 1) return cudaErrorInvalidValue;
    // 8 v bytes of row / column exponents next to 17 KB of static tiles; above the 48 KB
    // default the kernel opts in to the larger dynamic shared memory (v up to about 26000)
    const size_t smem = sizeof(int) * 2 * (size_t)src.v;
    if (smem > 200 * 1024 || src.rows > 0x7fffffffll) return cudaErrorInvalidValue;
    if (smem > 30 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(pm_fixed_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    pm_fixed_kernel<<<(unsigned)src.rows, 256, smem, st>>>(src, s, beta, (__nv_bfloat16*)Dp, pitchp, ep,
                                                           (__nv_bfloat16*)Dm, pitchm, em);
    count_launch();
    return cudaGetLastError();
}

cudaError_t pm_split_f32(const float* X, long long ldx, const long long* rtab, long long rows, int Nb, int v, int kind,
                         void* Dp, long long pitchp, int* ep, void* Dm, long long pitchm, int* em, cudaStream_t st)
{
    if (rows <= 0) return cudaSuccess;
    if (v < 1 || (kind != 1 && kind != 2) || rows > 0x7fffffffll) return cudaErrorInvalidValue;
    const long long nt = (v + TT - 1) / TT, pairs = nt * (nt + 1) / 2;
    long long share = pairs < 8 ? pairs : 8;
    if (rows * share > 0x7fffffffll) share = 1;
    auto kern = kind == 1 ? pm_f32_kernel<true> : pm_f32_kernel<false>;
    kern<<<(unsigned)(rows * share), TT * TY, 0, st>>>(X, ldx, rtab, Nb, v, Dp, pitchp, ep, Dm, pitchm, em, (int)share);
    count_launch();
    return cudaGetLastError();
}

cudaError_t fill_rtab(int Ab, int Nb, long long* rtab, cudaStream_t st)
{
    if (Ab <= 0) return cudaSuccess;
    fill_rtab_kernel<<<Ab, 256, 0, st>>>(Ab, Nb, rtab);
    count_launch();
    return cudaGetLastError();
}

namespace {
// Tiles of a block by the pairs, within the grid limits for any number of pairs.
dim3 combine_grid(int Ab, int Nb, long long np)
{
    const long long gz = (np + 65534) / 65535, gy = (np + gz - 1) / gz;
    return dim3((unsigned)(((Ab + TT - 1) / TT) * ((Nb + TT - 1) / TT)), (unsigned)gy, (unsigned)gz);
}
}  // namespace

cudaError_t pm_combine(int o, int v, int a0, int Ab, int Nb, long long nr, long long q0, long long q1, long long s0,
                       const double* Rp, const double* Rm, double* R, int accumulate, cudaStream_t st)
{
    const long long np = q1 - q0;
    if (Ab <= 0 || np <= 0) return cudaSuccess;
    if (Ab > 65535 || np > 0x7fffffffll || q0 < 0 || q1 > (long long)o * (o + 1) / 2) return cudaErrorInvalidValue;
    pm_combine_kernel<false, false><<<combine_grid(Ab, Nb, np), TT * TY, 0, st>>>(o, v, a0, Ab, Nb, nr, np, q0, s0, Rp, Rm, R, accumulate,
                                                                          nullptr, nullptr);
    count_launch();
    return cudaGetLastError();
}

cudaError_t pm_combine_general(long long pairs, int v, int a0, int Ab, int Nb, long long nr, const double* Rp,
                               const double* Rm, double* R, int accumulate, const double* V, const double* T, cudaStream_t st)
{
    if (Ab <= 0 || pairs <= 0) return cudaSuccess;
    if (Ab > 65535 || pairs > 0x7fffffffll) return cudaErrorInvalidValue;
    auto kern = V ? pm_combine_kernel<true, true> : pm_combine_kernel<true, false>;
    kern<<<combine_grid(Ab, Nb, pairs), TT * TY, 0, st>>>(0, v, a0, Ab, Nb, nr, pairs, 0, 0, Rp, Rm, R, accumulate, V, T);
    count_launch();
    return cudaGetLastError();
}

cudaError_t pm_combine_rows(long long pairs, int v, int a0, long long nr, const double* Rp, const double* Rm, double* R,
                            int accumulate, cudaStream_t st)
{
    if (nr <= 0 || pairs <= 0) return cudaSuccess;
    pm_combine_rows_kernel<<<dim3((unsigned)((nr + 255) / 256), (unsigned)(pairs < 65535 ? pairs : 65535)), 256, 0, st>>>(
        pairs, v, a0, nr, Rp, Rm, R, accumulate);
    count_launch();
    return cudaGetLastError();
}

cudaError_t fill_pairs(int o, int v, int strict, long long* tab, cudaStream_t st)
{
    if (o - strict <= 0) return cudaSuccess;
    fill_pairs_kernel<<<o, 64, 0, st>>>(o, v, strict, tab);
    count_launch();
    return cudaGetLastError();
}

}  // namespace cc
