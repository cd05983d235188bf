// gemm_crt.cu -- Blackwell (sm_103a) residue GEMM of the emulated-FP64 mode (see crt.cuh):
//
//   planes[l][m][n] = 128 + ( sum_k A_l(m,k) B_l(n,k) ) mod p_l (balanced),   one byte each, l = 0 .. nm-1
//
// for K-major bf16 residue stacks A[l][row][pitch], B[l][row][pitch] with |A|, |B| <= 128.
//
// One pair of SMs (a cluster of two CTAs) owns a 256 x 256 output tile of one modulus at a time and
// issues tcgen05.mma.cta_group::2 (M = 256, N = 256, K = 16) into both SMs' tensor memory: per K-step
// of 64 each CTA stages only its 128 rows of A and 128 rows of B (32 KB) for 512 clocks of MMAs, so the
// copies ask for 64 B/clk/SM where 128 x 128 tiles of one CTA ask for 128.  The kernel is persistent:
// pairs take (modulus, K-split, tile) items in raster order from a global counter, so that the items
// resident at once share operand rows in L2.  The tile columns share N evenly in units of 32 columns: a ladder GEMM
// has o(o+1)/2 columns, and 820 of them become 224 + 224 + 192 + 192 instead of 3 x 256 + 64 (whose last tile
// would load 256 rows of A for 64 columns).
//
// Exactness: a pass covers at most kCrtChunk = 1024 K elements, so every FP32 partial sum is an integer
// of at most 128 * 128 * 1024 = 2^24 and exact for any input.  Two 256-column accumulators (all of
// TMEM) alternate between passes: the epilogue reduces pass p modulo p_l into registers while the MMAs of
// pass p + 1 run, and the item's sum once more, to the byte it stores.  The reductions are packed FP32
// (r = x - p rint(x / p), exact), 1.5 instructions per element and pass: converting to integers instead took 8000
// clocks per tile, as long as the MMAs of K = 1000 (8192 x 8192 x 1024, 12 moduli: 1518 TFLOP/s then, 2065 now).
//
// The same kernel runs the mixed modes' GEMMs (one bf16 or tf32 operand each, passes of 16384 elements in FP32, FP64
// across passes), storing the FP32 sums or FP64: on 128 x 128 tiles of single SMs they had no operand reuse and were
// bound by the copies (integral build of o=27/v=301/n=1501 in BF16: 37.2 ms then, 7.7 now).
//
// Bound: the tensor pipe, long calls its power cap (o=40/v=400/n=2000 integral blocks: 1930 TFLOP/s, against 1724 of
// a library GEMM that runs for seconds); below K = 512 the epilogue, 2.5 us per item.
//
// Roles (384 threads): warp 0 issues the A copies and fetches items (leader CTA), warp 3 the B copies,
// one thread of the leader's warp 2 the MMAs, warps 4-11 are the epilogue (one row and 128 columns per
// thread).  Copies of both CTAs complete on the leader's barriers; slot releases and accumulator
// hand-overs are multicast commits to both CTAs.
//
// Every wait is bounded (globaltimer); on expiry the CTA raises the pair's abort flags and the device
// status word, waits (again bounded) for what it has in flight, frees TMEM and exits.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>

#include "cc_internal.cuh"
#include "crt.cuh"

namespace cc {
namespace {

constexpr int BM = 128;                        // tile rows per CTA (256 per pair)
constexpr int TM = 2 * BM;                     // tile rows per pair
constexpr int TN = 256;                        // widest tile
constexpr int TILE_BYTES = 128 * 128;          // 128 rows x 128 bytes
// Two K-steps share a slot: one wait and one commit per 8 MMAs.  With a slot per step the thread that issues the MMAs was
// the bound (555 clocks per step of 512 clocks of MMAs; 8192 x 8192 x 2048: 1936 TFLOP/s then, 2108 now, with six slots or
// five alike).  Three steps in each of two slots copy too little ahead (1737).
constexpr int SUB = 2;                         // K-steps per ring slot
constexpr int NS = 3;                          // ring slots
constexpr int SLOT_BYTES = SUB * TILE_BYTES;   // of one operand
constexpr int RING_BYTES = NS * 2 * SLOT_BYTES;  // 192 KB
constexpr int QN = 16;                         // item queue slots
constexpr int EPI_WARPS = 8;
constexpr int THREADS = 128 + 32 * EPI_WARPS;  // 384
constexpr int TMEM_COLS = 512;                 // two accumulators of 256 columns
constexpr int CPT = TN / 2;                    // accumulator columns per epilogue thread
static_assert(kCrtChunk % (64 * SUB) == 0, "passes end with a ring slot");
constexpr int kReduceEvery = 60;               // passes between reductions of the running sums (far below 2^24)
// setmaxnreg split of the launch's 384 x 168 registers: 128 x 56 + 256 x 216 = 62464 <= 64512
constexpr int REG_LOW = 56, REG_HIGH = 216;
static_assert(128 * REG_LOW + 256 * REG_HIGH <= THREADS * 168, "register split exceeds the launch's share");
constexpr unsigned long long kSettleNs = 5000000ull;      // abort path: copies in flight land within this
constexpr unsigned long long kDrainLimitNs = 1000000000ull;  // abort path: bound on the MMA drain
constexpr int WARP_A = 0, WARP_MMA = 2, WARP_B = 3;

struct SmemCtl {
    unsigned long long full[NS], empty[NS];
    unsigned long long tfull[2], tempty[2];
    unsigned long long drain;
    unsigned long long item_q[QN];             // slot k % QN: k + 1 above this pair's item k (-1: no work left)
    unsigned int tmem_base;
    volatile int abort;
};
constexpr int STAGE_BYTES = 32 * CPT;          // residues of one epilogue warp: 32 rows x 128 columns
constexpr size_t SMEM_BYTES = 1024 + RING_BYTES + EPI_WARPS * STAGE_BYTES + sizeof(SmemCtl);
static_assert(SMEM_BYTES <= 227 * 1024, "shared memory");

// What a kernel stores: residue bytes, the FP32 sums themselves (one pass), or FP64 through an index map.
enum OutKind { OUT_RES = 0, OUT_F32 = 1, OUT_F64 = 2 };

// Division of 0 <= n < 2^31 by a fixed d >= 1: with 2^s < d <= 2^(s + 1), mul = ceil(2^(32 + s) / d) is less than d above
// the quotient, so n times the excess stays below 2^(32 + s).
struct FastDiv {
    uint32_t d, mul, s;
    FastDiv() = default;
    explicit FastDiv(long long div) : d((uint32_t)div), mul(0), s(0)
    {
        while (d > 1 && (2ull << s) < d) ++s;
        if (d > 1) mul = (uint32_t)(((1ull << (32 + s)) + d - 1) / d);
    }
    __device__ __forceinline__ int div(int n) const { return d == 1 ? n : (int)(__umulhi((uint32_t)n, mul) >> s); }
};

struct Params {
    int M, N, K, nm;
    int chunk;                       // K elements per pass
    long long rowA0, rowB0;
    int ksplit, kper;                // K split s owns [s*kper, min(K, (s+1)*kper))
    long long tri;                   // triangular tile skip (0 = off): b(n) = n / tri < a(m) = m / tri
    int tiles_m, tiles_n, group_m, nitems;
    FastDiv by_l, by_tiles, by_group, by_gm, by_last, by_tri;  // by_gm, by_last: rows of tiles in a group, in the last one
    uint32_t step_bytes;             // bytes both CTAs copy per K-step
    int ubase, urem;                 // tile column j: ubase units of 32 columns, one more where j < urem
    unsigned char* planes;           // [ksplit][nm][M][pitch]
    long long pitch;
    int accumulate;                  // add to the residues that are there (modulo p_l)
    float inv[kCrtMax], neg[kCrtMax];  // 1 / p_l, -p_l
    float* f32;                      // OUT_F32: [M][pitch]
    OutDesc out;                     // OUT_F64
    int* counter;                    // [0] items handed out beyond the first of each pair, [1] pairs done (both zero)
    int* status;
    unsigned long long wait_ns;
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

// shared::cluster address of the object at the same offset in CTA `rank` of the pair
__device__ __forceinline__ uint32_t in_cta(const void* p, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_u32(p)), "r"(rank));
    return r;
}

__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ unsigned long long gtime()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void mbar_init(unsigned long long* b, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(count));
}

__device__ __forceinline__ bool mbar_try(unsigned long long* b, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(b)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Raises the abort flag of both CTAs and the status word.
__device__ __forceinline__ void raise_abort(SmemCtl* ctl, uint32_t rank, int* status)
{
    ctl->abort = 1;
    asm volatile("st.volatile.shared::cluster.u32 [%0], %1;" ::"r"(in_cta((const void*)&ctl->abort, rank ^ 1)), "r"(1)
                 : "memory");
    atomicOr(status, kStatusWaitExpired);
}

// Bounded wait; false (and the abort flags raised) when the bound expires or another role has aborted.
__device__ __forceinline__ bool mbar_wait(unsigned long long* b, uint32_t parity, SmemCtl* ctl, uint32_t rank,
                                          const Params& p)
{
    if (mbar_try(b, parity)) return true;
    const unsigned long long t0 = gtime();
    for (unsigned it = 1;; ++it) {
        if (mbar_try(b, parity)) return true;
        if (it == 1 || (it & 7) == 0) {
            if (ctl->abort) return false;
            if (gtime() - t0 > p.wait_ns) {
                raise_abort(ctl, rank, p.status);
                return false;
            }
        }
    }
}

// Ring slot of the next K-step and the parity of its turn.
struct Ring {
    uint32_t slot = 0, phase = 0;
    __device__ __forceinline__ void next()
    {
        if (++slot == NS) { slot = 0; phase ^= 1; }
    }
};

// Item k of this pair (-1: no work left, or abort); bounded.
__device__ __forceinline__ int item_at(SmemCtl* ctl, uint32_t k, uint32_t rank, const Params& p)
{
    unsigned long long t0 = 0;
    for (unsigned it = 0;; ++it) {
        unsigned long long q;
        asm volatile("ld.relaxed.cluster.shared::cta.u64 %0, [%1];" : "=l"(q) : "r"(smem_u32(&ctl->item_q[k % QN])) : "memory");
        if ((uint32_t)(q >> 32) == k + 1) return (int)(uint32_t)q;
        if (it == 0) t0 = gtime();
        __nanosleep(32);
        if ((it & 15) == 15) {
            if (ctl->abort) return -1;
            if (gtime() - t0 > p.wait_ns) {
                raise_abort(ctl, rank, p.status);
                return -1;
            }
        }
    }
}

__device__ __forceinline__ void mbar_expect_tx(unsigned long long* b, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(b)), "r"(bytes) : "memory");
}

__device__ __forceinline__ void mbar_arrive_cluster(uint32_t addr)
{
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(addr) : "memory");
}

// Copy into this CTA's shared memory, completing on the barrier at shared::cluster address `bar`.
__device__ __forceinline__ void tma_load(void* dst, const CUtensorMap* map, uint32_t bar, int x, int y, int z)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(smem_u32(dst)), "l"((unsigned long long)map), "r"(x), "r"(y), "r"(z), "r"(bar)
        : "memory");
}

// tcgen05 shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row groups 1024 bytes apart.
__device__ __forceinline__ unsigned long long smem_desc(const void* p)
{
    const unsigned long long addr = smem_u32(p);
    return ((addr >> 4) & 0x3fffull) | (1ull << 16) | ((unsigned long long)(1024 >> 4) << 32) | (1ull << 46) | (2ull << 61);
}

// FP32 accumulate, A and B bf16 (1) or tf32 (2), both K-major, M = 256, N = width.
template <int KIND>
__device__ __forceinline__ uint32_t instr_desc(int width)
{
    const uint32_t fmt = KIND == TC_BF16 ? 1u : 2u;
    return (1u << 4) | (fmt << 7) | (fmt << 10) | ((uint32_t)(width >> 3) << 17) | ((uint32_t)(TM >> 4) << 24);
}

template <int KIND>
__device__ __forceinline__ void mma(uint32_t d, unsigned long long a, unsigned long long b, uint32_t idesc, uint32_t acc)
{
    if (KIND == TC_BF16)
        asm volatile(
            "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
            " tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}\n"
            ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"(acc));
    else
        asm volatile(
            "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
            " tcgen05.mma.cta_group::2.kind::tf32 [%0], %1, %2, %3, p;\n}\n"
            ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"(acc));
}

// Arrive on `bar` (same offset) in both CTAs once this thread's prior MMAs complete.
__device__ __forceinline__ void commit_both(unsigned long long* bar)
{
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
        ::"r"(smem_u32(bar)), "h"((unsigned short)3) : "memory");
}

// The same on this CTA's barrier alone.
__device__ __forceinline__ void commit_own(unsigned long long* bar)
{
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// The same lane of a converged warp each time; what it issues keeps its operands in uniform registers.
__device__ __forceinline__ bool elect_one()
{
    uint32_t r;
    asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(r));
    return r != 0;
}

__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// 32 lanes x 32 columns, waited for.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,"
        "%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
}

// 32 lanes x 8 columns, waited for.
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
        : "r"(taddr));
}

// One warp's staged 32-row box to the output at (x, y, z), unless all its rows lie beyond M.
__device__ __forceinline__ void store_box(const CUtensorMap* map, const void* src, int x, int y, int z, int M, int lane)
{
    if (lane != 0 || y >= M) return;
    asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%2, %3, %4}], [%1];"
                 ::"l"((unsigned long long)map), "r"(smem_u32(src)), "r"(x), "r"(y), "r"(z) : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}

// x - p rint(x / p) of two integers |x| <= 2^24 at once: exact, and at most p / 2 + 1 in magnitude (the quotient is
// within 2^-8 of x / p, so it is off by one at most next to a tie); at most p / 2 for |x| < 2^16.
__device__ __forceinline__ unsigned long long reduce2(unsigned long long x, unsigned long long inv, unsigned long long neg)
{
    const unsigned long long big = f2(12582912.0f, 12582912.0f), nbig = f2(-12582912.0f, -12582912.0f);
    return fma2(add2(fma2(x, inv, big), nbig), neg, x);
}

// The same with the quotient of x + 1/4 (|x| < 2^16): ties of even p go to -p / 2, and -p / 2 <= result < p / 2.
__device__ __forceinline__ unsigned long long reduce2_low(unsigned long long x, unsigned long long inv, unsigned long long neg)
{
    const unsigned long long big = f2(12582912.0f, 12582912.0f), nbig = f2(-12582912.0f, -12582912.0f);
    return fma2(add2(fma2(add2(x, f2(0.25f, 0.25f)), inv, big), nbig), neg, x);
}

// Item i: modulus-major, then K split, then tiles rastered in groups of group_m tile rows.  Every role decodes every item,
// so the divisions are multiplications (six 32-bit divisions: 0.2 us of an item's 2.6 at K = 64, and of its 5.7 at K = 1024).
struct Item {
    int l, split, m0, n0, width;  // width: columns of the MMAs (a multiple of 32)
    bool skip;
};

__device__ __forceinline__ Item item_of(const Params& p, int i)
{
    Item it;
    it.l = p.by_l.div(i);
    const int rem = i - it.l * (int)p.by_l.d;
    it.split = p.by_tiles.div(rem);
    const int t = rem - it.split * (int)p.by_tiles.d;
    const int g = p.by_group.div(t), in = t - g * (int)p.by_group.d;
    const int first_m = g * p.group_m;
    const bool last = p.tiles_m - first_m < p.group_m;
    const int j = last ? p.by_last.div(in) : p.by_gm.div(in);
    it.m0 = (first_m + in - j * (int)(last ? p.by_last.d : p.by_gm.d)) * TM;
    it.n0 = 32 * (j * p.ubase + min(j, p.urem));
    it.width = 32 * (p.ubase + (j < p.urem ? 1 : 0));
    // every element of the tile has b(n) < a(m)
    it.skip = p.tri > 0 && p.by_tri.div(min(p.N - 1, it.n0 + it.width - 1)) < p.by_tri.div(it.m0);
    return it;
}

// The first item after skipped item i that may not be skipped: a group's leading columns of tiles are skipped in all its
// rows together.
__device__ __forceinline__ int after_skipped(const Params& p, int i)
{
    const int rem = i - p.by_l.div(i) * (int)p.by_l.d, t = rem - p.by_tiles.div(rem) * (int)p.by_tiles.d;
    const int g = p.by_group.div(t), in = t - g * (int)p.by_group.d;
    const int first_m = g * p.group_m, gm = min(p.tiles_m - first_m, p.group_m);
    const int amin = p.by_tri.div(first_m * TM);
    auto end_of = [&](int j) { return min(p.N, 32 * ((j + 1) * p.ubase + min(j + 1, p.urem))); };  // columns up to tile j
    int j = max(0, amin * (int)p.by_tri.d / 32 / (p.ubase + 1) - 1);  // (a tile has at most ubase + 1 units)
    while (j < p.tiles_n && p.by_tri.div(end_of(j) - 1) < amin) ++j;
    return max(i + 1, i - in + j * gm);
}

// Number and index travel in one word: a count published with release semantics waited for the counter's answer, about
// 2 us per item.  Leader: publishes the pair's item k to both CTAs, `item` being the counter's answer (the first one the pair's own
// index), moved on past skipped tiles.  Slot k % QN is free: when item k is published, every copy of item k - 2 has
// been issued, so the MMAs of item k - 5 have completed (a ring of 3 slots, at least one per item), so both epilogues
// have drained item k - 7 and read its queue slot before.
__device__ __forceinline__ int publish_item(SmemCtl* ctl, const Params& p, uint32_t k, int item, int npairs)
{
    while (p.tri > 0 && item < p.nitems && item_of(p, item).skip) {
        // the counter jumps over a run of skipped items (one by one they took 1 us each, shared by the pairs)
        const int to = after_skipped(p, item);
        if (to > item + 1) atomicMax(p.counter, to - npairs);
        item = npairs + atomicAdd(p.counter, 1);
    }
    if (item >= p.nitems || ctl->abort) item = -1;
    const unsigned long long q = ((unsigned long long)(k + 1) << 32) | (uint32_t)item;
    for (uint32_t r = 0; r < 2; ++r)
        asm volatile("st.relaxed.cluster.shared::cluster.u64 [%0], %1;" ::"r"(in_cta(&ctl->item_q[k % QN], r)), "l"(q)
                     : "memory");
    return item;
}

template <int KIND, int OUT>
__global__ void __launch_bounds__(THREADS, 1)
gemm_crt_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                const __grid_constant__ CUtensorMap tmC, const Params p)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* base = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    unsigned char* aring = base;
    unsigned char* bring = base + NS * SLOT_BYTES;
    unsigned char* stage = base + RING_BYTES;
    SmemCtl* ctl = (SmemCtl*)(base + RING_BYTES + EPI_WARPS * STAGE_BYTES);
    constexpr int KSTEP = KIND == TC_BF16 ? 64 : 32;  // K elements per 128-byte swizzle atom

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank();
    const int pair = (int)(blockIdx.x >> 1), npairs = (int)(gridDim.x >> 1);

    if (threadIdx.x == 0) {
        for (int s = 0; s < NS; ++s) {
            mbar_init(&ctl->full[s], 1);
            mbar_init(&ctl->empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&ctl->tfull[b], 1);
            mbar_init(&ctl->tempty[b], 2 * EPI_WARPS);
        }
        mbar_init(&ctl->drain, 1);
        for (int q = 0; q < QN; ++q) ctl->item_q[q] = 0;
        ctl->abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == WARP_MMA) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&ctl->tmem_base)),
                     "r"(TMEM_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;");
    }
    fence_before();
    __syncthreads();
    cluster_sync();  // the peer's barriers are initialised before any copy, commit or store reaches them
    fence_after();
    const uint32_t tmem = ctl->tmem_base;

    if (warp < 4) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REG_LOW));
        if ((warp == WARP_A || warp == WARP_B) && lane == 0) {
            // ------------------------------------------------------------ producers
            const bool isA = warp == WARP_A;
            const CUtensorMap* map = isA ? &tmA : &tmB;
            asm volatile("prefetch.tensormap [%0];" ::"l"((unsigned long long)map) : "memory");
            unsigned char* ring = isA ? aring : bring;
            const bool fetcher = isA && rank == 0;
            uint32_t u = 0;  // K-steps issued
            Ring at;
            bool ok = true;
            // The fetcher publishes the item after the one being copied, and asks the counter for one more whose answer
            // it only looks at an item later: the atomic's latency (about 1 us, as long as an item of K = 256) then
            // overlaps the copies.
            uint32_t pub = 0;   // items published
            int raw = pair;     // the counter's next answer
            bool more = true;   // no -1 published yet
            for (uint32_t k = 0; ok; ++k) {
                if (fetcher) {
                    while (more && pub <= k + 1) {
                        more = publish_item(ctl, p, pub, raw, npairs) >= 0;
                        ++pub;
                        if (more) raw = npairs + atomicAdd(p.counter, 1);
                    }
                }
                const int item = item_at(ctl, k, rank, p);
                if (item < 0) break;
                const Item w = item_of(p, item);
                const int row = isA ? (int)(p.rowA0 + w.m0) + (int)rank * BM
                                    : (int)(p.rowB0 + w.n0) + (int)rank * (w.width >> 1);
                const int kbeg = w.split * p.kper, kend = min(p.K, kbeg + p.kper);
                for (int kb = kbeg; kb < kend; kb += SUB * KSTEP, ++u, at.next()) {
                    const uint32_t s = at.slot;
                    if (!mbar_wait(&ctl->empty[s], at.phase ^ 1, ctl, rank, p)) { ok = false; break; }
                    const bool both = kb + KSTEP < kend;
                    if (fetcher) mbar_expect_tx(&ctl->full[s], both ? SUB * p.step_bytes : p.step_bytes);  // A and B tiles of both CTAs
                    const uint32_t bar = in_cta(&ctl->full[s], 0);
                    tma_load(ring + s * SLOT_BYTES, map, bar, kb, row, w.l);
                    if (both) tma_load(ring + s * SLOT_BYTES + TILE_BYTES, map, bar, kb + KSTEP, row, w.l);
                }
            }
            // the last use of every slot is released: no commit still targets this CTA's barriers when it leaves
            for (uint32_t q = 1; q <= NS && q <= u && ok; ++q) {
                const uint32_t v = u - q;
                ok = mbar_wait(&ctl->empty[v % NS], (v / NS) & 1, ctl, rank, p);
            }
            if (fetcher) {
                // the last pair to finish leaves the counters zero for the next launch on them
                __threadfence();
                if (atomicAdd(p.counter + 1, 1) == npairs - 1) {
                    __threadfence();
                    p.counter[0] = 0;
                    p.counter[1] = 0;
                }
            }
            if (!ok) {
                // abort: copies into this CTA's ring may still be in flight, and the two CTAs may have stopped at
                // different K-steps, so the leader's barriers need not complete: give the copies time to land
                const unsigned long long t0 = gtime();
                while (gtime() - t0 < kSettleNs) __nanosleep(1000);
            }
        } else if (warp == WARP_MMA && rank == 0) {
            // ------------------------------------------------------------ MMA
            const unsigned long long adesc0 = smem_desc(aring), bdesc0 = smem_desc(bring);
            uint32_t npass = 0;
            Ring at;
            bool ok = true, any = false;
            for (uint32_t k = 0; ok; ++k) {
                const int item = __shfl_sync(0xffffffffu, item_at(ctl, k, rank, p), 0);
                if (item < 0) break;
                const Item w = item_of(p, item);
                const uint32_t idesc = instr_desc<KIND>(w.width);
                const int kbeg = w.split * p.kper, kend = min(p.K, kbeg + p.kper);
                for (int k0 = kbeg; k0 < kend && ok; k0 += p.chunk) {
                    const int buf = (int)(npass & 1);
                    ok = __all_sync(0xffffffffu, mbar_wait(&ctl->tempty[buf], ((npass >> 1) & 1) ^ 1, ctl, rank, p));
                    if (!ok) break;
                    fence_after();
                    const uint32_t d = tmem + (uint32_t)(buf * TN);
                    const int k1 = min(kend, k0 + p.chunk);
                    uint32_t acc = 0;
                    for (int kb = k0; kb < k1; kb += SUB * KSTEP, at.next()) {
                        const uint32_t s = at.slot;
                        ok = __all_sync(0xffffffffu, mbar_wait(&ctl->full[s], at.phase, ctl, rank, p));
                        if (!ok) break;
                        fence_after();
                        const unsigned long long ad = adesc0 + (unsigned long long)(s * (SLOT_BYTES >> 4));
                        const unsigned long long bd = bdesc0 + (unsigned long long)(s * (SLOT_BYTES >> 4));
                        any = true;
                        if (elect_one()) {
                            // four MMAs per 128-byte row: advance the start address by 32 bytes each
                            mma<KIND>(d, ad, bd, idesc, acc);
                            mma<KIND>(d, ad + 2, bd + 2, idesc, 1u);
                            mma<KIND>(d, ad + 4, bd + 4, idesc, 1u);
                            mma<KIND>(d, ad + 6, bd + 6, idesc, 1u);
                            if (kb + KSTEP < k1) {
                                constexpr unsigned long long next = TILE_BYTES >> 4;
                                mma<KIND>(d, ad + next, bd + next, idesc, 1u);
                                mma<KIND>(d, ad + next + 2, bd + next + 2, idesc, 1u);
                                mma<KIND>(d, ad + next + 4, bd + next + 4, idesc, 1u);
                                mma<KIND>(d, ad + next + 6, bd + next + 6, idesc, 1u);
                            }
                            commit_both(&ctl->empty[s]);
                        }
                        __syncwarp();
                        acc = 1;
                    }
                    if (!ok) break;
                    if (elect_one()) commit_both(&ctl->tfull[buf]);
                    __syncwarp();
                    ++npass;
                }
            }
            // both buffers' last drains (the peer's arrivals land here) are done
            for (uint32_t q = npass > 2 ? npass - 2 : 0; q < npass && ok; ++q)
                ok = __all_sync(0xffffffffu, mbar_wait(&ctl->tempty[q & 1], (q >> 1) & 1, ctl, rank, p));
            if (any) {
                // every MMA has completed before TMEM is released (on this CTA's barrier only: nobody in the peer would wait
                // for the arrival there, which might then find a CTA that has left)
                if (elect_one()) commit_own(&ctl->drain);
                __syncwarp();
                const unsigned long long t0 = gtime();
                while (!mbar_try(&ctl->drain, 0)) {
                    if (gtime() - t0 > kDrainLimitNs) { atomicOr(p.status, kStatusDrainExpired); break; }
                }
            }
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(REG_HIGH));
        // ------------------------------------------------------------ epilogue
        // Warp 4 + e reads TMEM lanes 32 (warp % 4) .. + 31 (one tile row per thread) and columns
        // 128 (e / 4) .. + 127.
        const int q4 = warp & 3, half = (warp - 4) >> 2;
        const int row = (int)rank * BM + q4 * 32 + lane;
        const int col0 = half * CPT;
        const uint32_t tl = tmem + ((uint32_t)(q4 * 32) << 16) + (uint32_t)col0;
        uint32_t npass = 0;
        unsigned long long sum[CPT / 2];  // two columns each
        bool ok = true;
        for (uint32_t k = 0; ok; ++k) {
            int item = -1;
            if (lane == 0) item = item_at(ctl, k, rank, p);
            item = __shfl_sync(0xffffffffu, item, 0);
            if (item < 0) break;
            const Item w = item_of(p, item);
            const int m = w.m0 + row;
            const unsigned long long inv = f2(p.inv[w.l], p.inv[w.l]), neg = f2(p.neg[w.l], p.neg[w.l]);
            const int kbeg = w.split * p.kper, kend = min(p.K, kbeg + p.kper);
            int pass = 0;
            for (int k0 = kbeg; k0 < kend; k0 += p.chunk, ++pass, ++npass) {
                const int buf = (int)(npass & 1);
                if (lane == 0) ok = mbar_wait(&ctl->tfull[buf], (npass >> 1) & 1, ctl, rank, p);
                ok = __shfl_sync(0xffffffffu, (int)ok, 0) != 0;
                if (!ok) break;
                fence_after();
                if (OUT == OUT_F64) {
                    // FP64 across the passes, in the output: first pass = (or +=), later ones +=
                    double* Crow = p.out.C + (m < p.M ? map2(p.out.rmap, m) : 0);
                    const bool add = pass > 0 || p.out.accumulate;
#pragma unroll 1
                    for (int c = 0; c < CPT && col0 + c < w.width; c += 8) {  // (uniform over the warp)
                        uint32_t r[8];
                        __syncwarp();
                        tmem_ld8(tl + (uint32_t)(buf * TN + c), r);
#pragma unroll
                        for (int q = 0; q < 8; ++q) {
                            const int n = w.n0 + col0 + c + q;
                            if (m >= p.M || n >= p.N) continue;
                            double* dst = Crow + map2(p.out.cmap, n);
                            const double x = (double)__uint_as_float(r[q]);
                            *dst = add ? *dst + x : x;
                        }
                    }
                } else if (OUT == OUT_F32) {
#pragma unroll
                    for (int c = 0; c < CPT; c += 32) {
                        if (col0 + c >= w.width) continue;  // (uniform over the warp; widths are multiples of 32)
                        uint32_t r[32];
                        __syncwarp();
                        tmem_ld32(tl + (uint32_t)(buf * TN + c), r);
                        // 32 rows x 32 columns (128 bytes) per TMA store, 128-byte swizzle; the map clips what lies outside
                        unsigned char* sb = stage + (warp - 4) * STAGE_BYTES;
                        if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
                        __syncwarp();
#pragma unroll
                        for (int q = 0; q < 8; ++q)
                            *reinterpret_cast<uint4*>(sb + lane * 128 + ((q ^ (lane & 7)) * 16)) =
                                make_uint4(r[4 * q], r[4 * q + 1], r[4 * q + 2], r[4 * q + 3]);
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                        __syncwarp();
                        store_box(&tmC, sb, w.n0 + col0 + c, w.m0 + (int)rank * BM + q4 * 32, 0, p.M, lane);
                    }
                } else if (col0 < w.width) {
                    // (columns beyond the width are read as well and never stored)
#pragma unroll
                    for (int c = 0; c < CPT; c += 32) {
                        uint32_t r[32];
                        tmem_ld32(tl + (uint32_t)(buf * TN + c), r);
#pragma unroll
                        for (int q = 0; q < 16; ++q) {
                            const unsigned long long x =
                                reduce2(f2(__uint_as_float(r[2 * q]), __uint_as_float(r[2 * q + 1])), inv, neg);
                            sum[c / 2 + q] = pass == 0 ? x : add2(sum[c / 2 + q], x);
                        }
                    }
                }
                fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(in_cta(&ctl->tempty[buf], 0));
                if (OUT == OUT_RES && pass % kReduceEvery == kReduceEvery - 1) {
#pragma unroll
                    for (int q = 0; q < CPT / 2; ++q) sum[q] = reduce2(sum[q], inv, neg);
                }
            }
            if (!ok) break;
            if (OUT != OUT_RES || col0 >= w.width) continue;
            // The bytes 128 + r, four columns to a word.  One pass leaves |r| <= (p + 1) / 2, which fits but for p = 256 and
            // 255; sums of passes (and those moduli) are reduced once more, to -p / 2 <= r < p / 2.
            const int plane = w.split * p.nm + w.l;
            unsigned char* dst = p.planes + ((long long)plane * p.M + m) * p.pitch + w.n0 + col0;
            if (p.accumulate && m < p.M) {
                // 64 of the row's old bytes at once, 16 per load (o=10/v=120/n=600 in chunks of 64 Cholesky vectors, integral
                // build: 19.5 ms with 4 bytes per load, 11.7 so; the digit slices take 12.7)
                const unsigned long long off = f2(-8388736.0f, -8388736.0f);
                // bytes 2 e, 2 e + 1 as the floats 2^23 + b
                auto pair = [](uint32_t o, int e) {
                    return f2(__uint_as_float(__byte_perm(o, 0x4B000000u, 0x7440 + 2 * e)),
                              __uint_as_float(__byte_perm(o, 0x4B000000u, 0x7441 + 2 * e)));
                };
#pragma unroll
                for (int c0 = 0; c0 < CPT / 16; c0 += 4) {
                    uint4 old[4];
#pragma unroll
                    for (int c = 0; c < 4; ++c)
                        old[c] = w.n0 + col0 + 16 * (c0 + c) < p.pitch ? *reinterpret_cast<const uint4*>(dst + 16 * (c0 + c))
                                                                       : make_uint4(0, 0, 0, 0);
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const uint32_t o[4] = {old[c].x, old[c].y, old[c].z, old[c].w};
#pragma unroll
                        for (int q = 0; q < 8; ++q) {
                            unsigned long long& x = sum[8 * (c0 + c) + q];
                            x = add2(x, add2(pair(o[q >> 1], q & 1), off));
                        }
                    }
                }
            }
            if (pass > 1 || w.l <= 1 || p.accumulate) {
#pragma unroll
                for (int q = 0; q < CPT / 2; ++q) sum[q] = reduce2_low(sum[q], inv, neg);
            }
            // columns c and c + 2 as 2^23 + (128 + r_c) + 256 (128 + r_c+2), so two packed instructions and a permute make a word
            auto word = [&](int q) {
                const unsigned long long off = f2(8421504.0f, 8421504.0f), shift = f2(256.0f, 256.0f);
                const unsigned long long a = fma2(sum[2 * q + 1], shift, add2(sum[2 * q], off));
                return __byte_perm((uint32_t)a, (uint32_t)(a >> 32), 0x5140);
            };
            if (col0 + CPT <= w.width) {
                // a whole half tile leaves as one TMA store per warp, 128-byte rows (16 bytes per lane and row straight
                // to memory are half sectors in 32 different lines per instruction): 32 rows x 128 bytes, 128-byte swizzle
                unsigned char* buf = stage + (warp - 4) * STAGE_BYTES;
                if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
                __syncwarp();
#pragma unroll
                for (int c = 0; c < CPT / 16; ++c)
                    *reinterpret_cast<uint4*>(buf + lane * CPT + ((c ^ (lane & 7)) * 16)) =
                        make_uint4(word(4 * c), word(4 * c + 1), word(4 * c + 2), word(4 * c + 3));
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                store_box(&tmC, buf, w.n0 + col0, w.m0 + (int)rank * BM + q4 * 32, plane, p.M, lane);
            } else if (m < p.M) {
#pragma unroll
                for (int c = 0; c < CPT / 16; ++c)
                    if (w.n0 + col0 + 16 * c < p.pitch && col0 + 16 * c < w.width)
                        *reinterpret_cast<uint4*>(dst + 16 * c) =
                            make_uint4(word(4 * c), word(4 * c + 1), word(4 * c + 2), word(4 * c + 3));
            }
        }
        // this warp's stores have left shared memory and are complete before the CTA exits
        if (OUT != OUT_F64 && lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    }

    fence_before();
    __syncthreads();
    cluster_sync();  // no CTA leaves while its peer may still read its shared memory or signal it
    fence_after();
    if (warp == WARP_MMA) {
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS));
    }
}

PFN_cuTensorMapEncodeTiled_v12000 get_encode()
{
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (PFN_cuTensorMapEncodeTiled_v12000)f;
    });
    return fn;
}

// 3-D map over a stack [nm][rows][pitch] of bf16 or tf32, extent K in the inner dimension; boxes of 128 bytes x box_rows.
bool make_map(CUtensorMap* m, const void* base, int kind, long long K, long long pitch, long long rows, int nm, int box_rows)
{
    auto enc = get_encode();
    if (!enc) return false;
    const int es = kind == TC_BF16 ? 2 : 4;
    cuuint64_t dims[3] = {(cuuint64_t)K, (cuuint64_t)rows, (cuuint64_t)nm};
    cuuint64_t strides[2] = {(cuuint64_t)(pitch * es), (cuuint64_t)(pitch * es * rows)};
    cuuint32_t box[3] = {(cuuint32_t)(128 / es), (cuuint32_t)box_rows, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    return enc(m, kind == TC_BF16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3,
               const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
               CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

struct Sides {  // operands of a launch
    const void* A; long long pitchA, rowsA;
    const void* B; long long pitchB, rowsB;
};

// Tiles, items, counter and launch; p holds everything else.
template <int KIND, int OUT>
cudaError_t launch(const Sides& g, Params& p, cudaStream_t s)
{
    p.tiles_m = (p.M + TM - 1) / TM;
    p.tiles_n = (p.N + TN - 1) / TN;
    const int units = (p.N + 31) / 32;
    p.ubase = units / p.tiles_n;
    p.urem = units % p.tiles_n;
    // Every group of tile rows reads all of B again, from memory unless B fits in L2: 16 rows read it half as often as 8, as
    // long as their own elements stay in L2 (integral build of o=40/v=400/n=2000 318 -> 312 ms, of o=20/v=200/n=1000 10.25
    // -> 10.15, o=27/v=301/n=1501 in BF16 7.86 -> 7.74).  Along a long K fewer rows at once are better (ladder GEMM at v=400,
    // K = 20160 per split: 170 ms with 8, 175 with 16).
    const int group = p.K <= 4096 ? 16 : 8;
    p.group_m = p.tiles_m < group ? p.tiles_m : group;
    const long long nitems = (long long)p.tiles_m * p.tiles_n * p.ksplit * p.nm;
    if (nitems > 0x7fffffffll - (1 << 20)) return cudaErrorInvalidConfiguration;
    p.nitems = (int)nitems;
    const long long ntiles = (long long)p.tiles_m * p.tiles_n;
    p.by_l = FastDiv(ntiles * p.ksplit);
    p.by_tiles = FastDiv(ntiles);
    p.by_group = FastDiv((long long)p.group_m * p.tiles_n);
    p.by_gm = FastDiv(p.group_m);
    p.by_last = FastDiv(p.tiles_m % p.group_m ? p.tiles_m % p.group_m : p.group_m);
    p.by_tri = FastDiv(p.tri > 0 ? std::min(p.tri, 0x7fffffffll) : 1);

    cudaLaunchConfig_t cfg{};
    cfg.blockDim = dim3(THREADS);
    cfg.dynamicSmemBytes = SMEM_BYTES;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    // persistent: as many pairs as are resident on the device at once
    static PerDevice resident;
    const int max_pairs = resident.get([&cfg] {
        if (cudaFuncSetAttribute(gemm_crt_kernel<KIND, OUT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_BYTES) != cudaSuccess)
            return 0;
        int n = 0;
        cfg.gridDim = dim3(2 * 64);
        if (cudaOccupancyMaxActiveClusters(&n, gemm_crt_kernel<KIND, OUT>, &cfg) != cudaSuccess || n <= 0) {
            cudaGetLastError();
            n = std::max(1, device_sm_count() / 2);
        }
        return n;
    });
    if (max_pairs == 0) return cudaErrorInvalidConfiguration;

    CUtensorMap ma, mb, mc{};
    if (OUT != OUT_F64) {
        // output planes, or the FP32 rows: 128 bytes x 32 rows per store
        const cuuint64_t es = OUT == OUT_RES ? 1 : 4, planes = OUT == OUT_RES ? (cuuint64_t)p.nm * p.ksplit : 1;
        auto enc = get_encode();
        cuuint64_t dims[3] = {(cuuint64_t)p.pitch, (cuuint64_t)p.M, planes};
        cuuint64_t strides[2] = {(cuuint64_t)p.pitch * es, (cuuint64_t)p.pitch * es * p.M};
        cuuint32_t box[3] = {(cuuint32_t)(128 / es), 32, 1}, estr[3] = {1, 1, 1};
        if (!enc || enc(&mc, OUT == OUT_RES ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3,
                        OUT == OUT_RES ? (void*)p.planes : (void*)p.f32, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                        CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
    // (narrow tiles, N <= 224, are bound by the copies: B's boxes hold only the rows a tile uses)
    const int brows = 16 * (p.ubase + (p.urem > 0 ? 1 : 0));
    p.step_bytes = 2u * (uint32_t)(TILE_BYTES + brows * 128);
    if (!make_map(&ma, g.A, KIND, p.K, g.pitchA, g.rowsA, p.nm, BM) ||
        !make_map(&mb, g.B, KIND, p.K, g.pitchB, g.rowsB, p.nm, brows))
        return cudaErrorInvalidValue;
    const int pairs = p.nitems < max_pairs ? p.nitems : max_pairs;
    cfg.gridDim = dim3((unsigned)(2 * pairs));
    const cudaError_t err = cudaLaunchKernelEx(&cfg, gemm_crt_kernel<KIND, OUT>, ma, mb, mc, p);
    if (err != cudaSuccess) return err;
    count_launch();
    return cudaGetLastError();
}

}  // namespace

cudaError_t gemm_crt(const GemmCrt& g, cudaStream_t s)
{
    if (g.M <= 0 || g.N <= 0) return cudaSuccess;
    if (g.K <= 0 || g.nm < 1 || g.nm > kCrtMax || g.pitch < g.N || g.pitch % 16 || g.tri < 0) return cudaErrorInvalidValue;
    Params p{};
    p.M = g.M; p.N = g.N; p.K = g.K; p.nm = g.nm;
    p.chunk = kCrtChunk;
    p.rowA0 = g.rowA0; p.rowB0 = g.rowB0;
    p.ksplit = g.ksplit > 1 ? g.ksplit : 1;
    p.kper = (int)((((long long)g.K + p.ksplit - 1) / p.ksplit + 63) / 64 * 64);
    if ((long long)p.kper * (p.ksplit - 1) >= g.K || (p.ksplit > 1 && g.accumulate)) return cudaErrorInvalidValue;
    p.tri = g.tri;
    p.planes = g.planes;
    p.pitch = g.pitch;
    p.accumulate = g.accumulate;
    for (int l = 0; l < g.nm; ++l) {
        p.inv[l] = 1.0f / (float)crt_p(l);
        p.neg[l] = -(float)crt_p(l);
    }
    p.status = g.status;
    p.wait_ns = g.wait_ns;
    p.counter = g.counter;
    return launch<TC_BF16, OUT_RES>(Sides{g.A, g.pitchA, g.rowsA, g.B, g.pitchB, g.rowsB}, p, s);
}

cudaError_t gemm_mix(const GemmMix& g, cudaStream_t s)
{
    if (g.M <= 0 || g.N <= 0) return cudaSuccess;
    const int kstep = g.kind == TC_BF16 ? 64 : 32;
    if (g.K <= 0 || g.chunk <= 0 || g.chunk % (SUB * kstep) || g.tri < 0) return cudaErrorInvalidValue;
    if (g.f32 && (g.K > g.chunk || g.pitch < g.N || g.pitch % 4)) return cudaErrorInvalidValue;
    Params p{};
    p.M = g.M; p.N = g.N; p.K = g.K; p.nm = 1;
    p.chunk = g.chunk;
    p.rowA0 = g.rowA0; p.rowB0 = g.rowB0;
    p.ksplit = 1;
    p.kper = (g.K + 63) / 64 * 64;
    p.tri = g.tri;
    p.f32 = g.f32;
    p.pitch = g.pitch;
    p.out = g.out;
    p.status = g.status;
    p.wait_ns = g.wait_ns;
    p.counter = g.counter;
    const Sides sd{g.A, g.pitchA, g.rowsA, g.B, g.pitchB, g.rowsB};
    if (g.kind == TC_BF16) return g.f32 ? launch<TC_BF16, OUT_F32>(sd, p, s) : launch<TC_BF16, OUT_F64>(sd, p, s);
    return g.f32 ? launch<TC_TF32, OUT_F32>(sd, p, s) : launch<TC_TF32, OUT_F64>(sd, p, s);
}

}  // namespace cc
