// crt.cuh -- residue arithmetic of the emulated-FP64 mode (the default, 42-bit precision).
//
// Every operand row is rounded once to 42-bit signed integers X = round(x 2^(41 - e)),
// |X| <= 2^41 (max |row| < 2^e), exactly as for the digit slices of split.cu.  Instead of cutting X
// into digits, X is reduced modulo nm pairwise coprime numbers p_l <= 256; one bf16 GEMM per modulus
// (gemm_crt.cu) gives C_l = (A_l B_l^T) mod p_l, and the Chinese remainder theorem returns the exact
// integer sum_k X_A X_B as long as it lies in (-P/2, P/2), P = prod p_l.  That holds for ANY input
// when K 2^82 < P/2, and crt_moduli() takes as many moduli as that needs: 12 up to K = 3574, 13 up
// to K = 754155.  (A second contraction, one of whose sides are 43-bit rows made from the first one's results, needs
// K 2^83 < P/2: 12 up to K = 1787, 13 up to 377077.)  So 12 or 13 bf16 GEMMs do what the digit slices do with 21, and
// nothing is dropped (the slices drop every level above 5).  This is the modular form of the Ozaki scheme (Ozaki, Uchino, Imamura,
// "Ozaki Scheme II", 2025), here with the fixed row scale of the slices and with partial sums kept exact by
// draining the FP32 accumulators every 1024 elements: |r| <= 128, so 1024 products stay within 2^24.
//
// Reconstruction: with M_l = P / p_l and m_l = M_l^-1 mod p_l, x / P = frac(sum_l r_l m_l / p_l).  The
// fractions W_l = m_l / p_l are tabulated as 96-bit fixed point and the sum taken modulo 1 (integer
// wrap-around), which yields x as a signed fraction of P; one 64 x 64 -> high multiply by P scales it to
// an int64 in units of 2^34 (12 moduli) of an X_A X_B product.  The error is below a quarter of that unit, so
// a sum that is a multiple of the unit (integer inputs) comes out exactly.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace cc {

constexpr int kCrtMax = 14;   // moduli in the table
constexpr int kCrtMin = 12;   // fewest ever used
constexpr int kCrtBits = 42;    // rows made from FP64: |X| <= 2^(kCrtBits - 1)
constexpr int kPlaneBits = 43;  // rows made from planes (crt_prep.cu): |X| <= 2^(kPlaneBits - 1)
constexpr int kCrtChunk = 1024;  // K elements whose products stay exact in FP32 (128 * 128 * 1024 = 2^24)

// 256 = 2^8, 255 = 3 5 17, 253 = 11 23, 247 = 13 19, 217 = 7 31; the others are prime.
__host__ __device__ constexpr int crt_p(int l)
{
    constexpr int t[kCrtMax] = {256, 255, 253, 251, 247, 241, 239, 233, 229, 227, 223, 217, 211, 199};
    return t[l];
}

// Everything the reconstruction from nm residues needs; a kernel parameter (uniform operands).
struct CrtRec {
    int nm;
    uint32_t w2[kCrtMax], w1[kCrtMax], w0[kCrtMax];  // W_l * 2^96, most significant word first
    uint32_t b2, b1, b0;  // sum_l W_l * 128 * 2^96, its negative: undoes the bytes' offset of 128
    uint32_t n2, n1;      // the same for the top two words alone
    uint32_t t2;          // the same for the top word alone
    long long mul;   // P * 2^-(unit - sh)
    int sh;          // x = (mulhi(y, mul) + 2^(sh-1)) >> sh
    int unit;        // result in units of 2^unit products
    double frac;     // P * 2^-64 * 2^(-2 (kCrtBits - 1)): one unit of y, before the row and column exponents
};

inline unsigned __int128 crt_product(int nm)
{
    unsigned __int128 P = 1;
    for (int l = 0; l < nm; ++l) P *= (unsigned)crt_p(l);
    return P;
}

// Moduli that keep sum_k X_A X_B (K terms of at most 2^(bits_a - 1 + bits_b - 1)) inside (-P/2, P/2); 0: more than
// the table has.
inline int crt_moduli(long long K, int bits_a = kCrtBits, int bits_b = kCrtBits)
{
    for (int nm = kCrtMin; nm <= kCrtMax; ++nm) {
        const unsigned __int128 need = (unsigned __int128)(unsigned long long)K << (bits_a + bits_b - 1);
        if (K < (1ll << 40) && need < crt_product(nm)) return nm;
    }
    return 0;
}

inline CrtRec crt_rec(int nm)
{
    CrtRec c{};
    c.nm = nm;
    const unsigned __int128 P = crt_product(nm);
    for (int l = 0; l < nm; ++l) {
        const unsigned p = (unsigned)crt_p(l);
        const unsigned r = (unsigned)((P / p) % p);
        unsigned inv = 1;
        while ((unsigned long long)r * inv % p != 1) ++inv;
        const unsigned __int128 w = (((unsigned __int128)inv << 96) + p / 2) / p;
        c.w2[l] = (uint32_t)(w >> 64);
        c.w1[l] = (uint32_t)(w >> 32);
        c.w0[l] = (uint32_t)w;
    }
    unsigned __int128 bias = 0;
    unsigned long long b64 = 0;
    for (int l = 0; l < nm; ++l) {
        b64 -= 128 * (((unsigned long long)c.w2[l] << 32) + c.w1[l]);
        bias += ((((unsigned __int128)c.w2[l] << 32) + c.w1[l]) << 32) + c.w0[l];
        c.t2 -= 128u * c.w2[l];
    }
    bias = (unsigned __int128)0 - 128 * bias;
    c.n2 = (uint32_t)(b64 >> 32);
    c.n1 = (uint32_t)b64;
    c.b2 = (uint32_t)(bias >> 64);
    c.b1 = (uint32_t)(bias >> 32);
    c.b0 = (uint32_t)bias;
    // the finest unit that the truncation of y, P 2^-64, stays a tenth of: 2^34, 2^42, 2^50 (|x| < 2^60 units)
    c.unit = 34 + 8 * (nm - kCrtMin);
    int bits = 0;
    for (unsigned __int128 q = P >> c.unit; q; q >>= 1) ++bits;
    c.sh = 62 - bits;
    c.mul = (long long)(c.sh <= c.unit ? P >> (c.unit - c.sh) : P << (c.sh - c.unit));
    c.frac = (double)P;
    for (int q = 0; q < 64 + 2 * (kCrtBits - 1); ++q) c.frac *= 0.5;
    return c;
}

// Exponent of one unit of the reconstructed integer, before the row and column exponents: a row's X
// counts 2^(e - (bits - 1)).
inline int crt_base(const CrtRec& c, int bits_a, int bits_b) { return c.unit - (bits_a - 1) - (bits_b - 1); }

// Packed order of the entries c <= d of a v x v matrix: 8 x 8 blocks (bc <= bd, 64 entries row by row, zero outside
// c <= d < v), one 128-byte line of bf16 each, the blocks of a 32 x 32 tile together, tiles (tc <= td) in order.  What a
// CTA makes of one tile pair is then one run of up to 2 KB in every residue's row, in whole lines (row by row in c it was
// 32 segments of 64 bytes, none aligned).  v = 400: 81600 entries for v(v+1)/2 = 80200.
__host__ __device__ inline int crt_blocks(int v) { return (v + 7) / 8; }
inline long long crt_kq_total(long long v)
{
    const long long nb = (v + 7) / 8;
    return nb * (nb + 1) / 2 * 64;
}
// Blocks before tile (tc, td) of nb x nb blocks.
__host__ __device__ inline int crt_tile_off(int tc, int td, int nb)
{
    const int b0 = 4 * tc, n = nb - b0 < 4 ? nb - b0 : 4;
    const int base = b0 * nb - b0 * (b0 - 1) / 2;
    return td == tc ? base : base + n * (n + 1) / 2 + n * 4 * (td - tc - 1);
}

#ifdef __CUDACC__
// Sum of r_l W_l modulo 1 as the top 64 bits, from bytes r_l + 128; add() one byte per modulus (and split).  WIDE sums
// 96 bits (error 2^-64); without, the 64-bit sum is off by up to nm * 128 units of 2^-64: for rows that are rounded to
// 43 bits.  With 12 moduli that is at most 2^41.4 of an X_A X_B product, 2^-40.6 of max|row A| max|row B| 4: an absolute
// error, so a row of integrals that all cancel to far below that product keeps fewer than 42 bits of its own largest entry
// (the digit slices resolve 2^44 there).
template <bool WIDE>
struct CrtAcc {
    unsigned long long a0, a1;
    uint32_t a2;
    __device__ __forceinline__ explicit CrtAcc(const CrtRec& c)
    {
        // (without the low words the offset's are left out as well: the same 64-bit weights are undone)
        a0 = WIDE ? c.b0 : 0;
        a1 = WIDE ? c.b1 : c.n1;
        a2 = WIDE ? c.b2 : c.n2;
    }
    __device__ __forceinline__ void add(uint32_t r, const CrtRec& c, int l)
    {
        if (WIDE) a0 += (unsigned long long)r * c.w0[l];
        a1 += (unsigned long long)r * c.w1[l];
        a2 += r * c.w2[l];
    }
    __device__ __forceinline__ long long fraction() const
    {
        return (long long)(((unsigned long long)a2 << 32) + a1 + (WIDE ? a0 >> 32 : 0));
    }
};

__device__ __forceinline__ long long crt_scale(long long y, const CrtRec& c)
{
    return (__mul64hi(y, c.mul) + (1ll << (c.sh - 1))) >> c.sh;
}

constexpr unsigned long long kCrtBias = 1ull << 42;  // residues are taken from X + kCrtBias

// X (|X| <= 2^42) as three pieces X = h2 2^28 + h1 2^14 + h0 in exact floats, for the residues below.
struct CrtPieces {
    float h2, h1, h0;
    // from u = X + 2^42, 0 .. 2^43
    __device__ __forceinline__ explicit CrtPieces(unsigned long long u)
    {
        // 2^23 + n as a float holds n < 2^23 exactly in its low bits
        h0 = __uint_as_float(0x4B000000u | ((uint32_t)u & 0x3fffu)) - 8388608.0f;
        h1 = __uint_as_float(0x4B000000u | ((uint32_t)(u >> 14) & 0x3fffu)) - 8388608.0f;
        h2 = __uint_as_float(0x4B000000u | (uint32_t)(u >> 28)) - (8388608.0f + 16384.0f);
    }
};

__host__ __device__ constexpr int crt_balanced(long long x, int p)
{
    const int r = (int)(x % p);
    return r > p / 2 ? r - p : r;
}

// Two floats in one register pair: the packed FP32 instructions of sm_100 and later do both at once.
__device__ __forceinline__ unsigned long long f2(float a, float b)
{
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c)
{
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b)
{
    unsigned long long r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

struct CrtPieces2 {
    unsigned long long h2, h1, h0;
    CrtPieces2() = default;
    __device__ __forceinline__ CrtPieces2(unsigned long long ua, unsigned long long ub)
    {
        const CrtPieces a(ua), b(ub);
        h2 = f2(a.h2, b.h2);
        h1 = f2(a.h1, b.h1);
        h0 = f2(a.h0, b.h0);
    }
};

// bf16 bits of X mod p for two X (the first in the low half), |r| <= 128.  t = h2 (2^28 mod p) + h1 (2^14 mod p)
// + h0 stays below 2^22, so every step is exact but the quotient, which is within 2^-9 of t / p: r is
// the balanced residue, or at most one beyond p / 2.  p is a compile-time constant wherever this is unrolled.
__device__ __forceinline__ uint32_t crt_residues2(const CrtPieces2& h, int p)
{
    const float c2 = (float)crt_balanced(1ll << 28, p), c1 = (float)crt_balanced(1ll << 14, p);
    const float inv = 1.0f / (float)p, big = 12582912.0f;
    const unsigned long long t = fma2(h.h2, f2(c2, c2), fma2(h.h1, f2(c1, c1), h.h0));
    const unsigned long long q = add2(fma2(t, f2(inv, inv), f2(big, big)), f2(-big, -big));
    const unsigned long long r = fma2(q, f2(-(float)p, -(float)p), t);
    return __byte_perm((uint32_t)r, (uint32_t)(r >> 32), 0x7632);
}
#endif

}  // namespace cc
