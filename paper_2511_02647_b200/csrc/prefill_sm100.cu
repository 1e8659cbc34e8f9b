// bf16 prefill attention for sm_100a (head_dim <= 128): TMA-fed, tcgen05 tensor cores, accumulators in TMEM,
// online softmax in fp32.  Serves fedattn_local (per-participant causal attention over packed
// segments) and fedattn_sync (queries over the aggregated KV, causal on global positions).
//
// Persistent kernel, one CTA per SM.  A work item is two "sub-tiles" of 128 query rows x one query head that share a
// KV head: two heads of a query tile; the last heads of an odd group in two neighbouring query tiles ("straddle"); or
// one head of one query tile, whose KV tiles the sub-tiles share ("halves").  Each sub-tile walks the key/value tiles
// its rows may see; tiles that the segment descriptors or the causal mask rule out are never loaded.  Items are sorted
// by cost and dealt to the CTAs in snake order.
//
// Per KV tile j and sub-tile t:
//     S_t = Q_t K_j^T          (tcgen05.mma, A/B from shared memory, D in TMEM)
//     P_t = exp2(S_t*c - m)    (softmax threads, TMEM -> registers -> TMEM, P aliases S)
//     O_t += P_t V_j           (tcgen05.mma, A = P from TMEM, B = V from shared memory)
// The tensor pipe alternates between the sub-tiles (PV_0 S_0 | PV_1 S_1 | ...); each sub-tile has a
// softmax warpgroup of its own, so while one warpgroup is in the serial part of its visit the other
// computes and the tensor pipe works for whichever sub-tile is ready.  O stays in TMEM for the whole
// tile walk and is rescaled only when a row's running maximum grows by more than 2^8 (the final
// normalisation uses the same reference, so the result is exact up to rounding).
//
// Warp roles: warps 0-3 softmax/epilogue of sub-tile 0, warps 4-7 of sub-tile 1: thread = query row =
// TMEM lane, all 128 key columns of the S tile (read from TMEM once, held in registers for the row
// maximum and then the exponentials) and the whole row of O; nothing is exchanged between threads (halves: the two
// partials of a row meet in the epilogue).  Warp 8
// TMA producer (+ TMEM allocation), warp 9 MMA issuer (the whole warp walks the loop, one elected lane
// issues); warp 10 checks the order of the key positions, warp 11 only fills that warpgroup, which
// hands most of its registers to the softmax warpgroups (setmaxnreg works on whole warpgroups).
// 2/8 of the exponentials of unmasked tiles are evaluated by a polynomial on the FMA pipe, because for
// this tile shape the ex2 unit alone is as slow as the tensor pipe.  The producer decodes every work
// item once and publishes it through shared memory for the softmax warps; finished rows leave through
// shared-memory staging and TMA stores (a warp with rows beyond its segment stores them directly).
// Every wait is bounded; on expiry the CTA sets the status word, stops waiting and runs to its normal
// end (TMEM is always released).
#include <cuda.h>

#include <stdio.h>
#include <stdlib.h>
#include <type_traits>

#include "attn_row.cuh"
#include "common.cuh"

namespace fedattn {

namespace {

constexpr int kTileM = 128;          // query rows per CTA
constexpr int kTileN = 128;          // keys per KV tile
constexpr int kBoxCols = 64;          // head-dim columns of one TMA box (128-byte swizzle); a tile is 1 or 2 boxes
// two softmax warpgroups, one per sub-tile.  (Both on the same S tile, split by columns with the row
// maxima exchanged through shared memory, was 2-4 % slower on dense sync; four warpgroups of 32 columns
// 20 %.)  P is handed to the MMA warp in kSplit halves, so that PV starts on the first.
constexpr int kSplit = 2;
constexpr int kSoftmaxThreads = 128 * kSplit;
constexpr int kThreads = kSoftmaxThreads + 128;  // then a warpgroup holding the TMA producer warp and the MMA issuer warp
// Registers move from that warpgroup to the softmax warpgroups once the roles split (setmaxnreg):
// 384 threads start with 168 each, and that allocation (3 x 168 = 504 registers per lane slot of a
// scheduler) is the pool the increases draw from.  setmaxnreg.inc waits, without limit, until the pool
// can give what it asks for, so the split must fit into it: 2 x kSoftmaxRegs + kOtherRegs <= 504; it
// keeps 8 spare.  (A 200 / 112 split asks for 512 per lane slot and never came back from the increase.)
constexpr int kSoftmaxRegs = 216, kOtherRegs = 64;
static_assert(2 * kSoftmaxRegs + kOtherRegs <= 496 && kSoftmaxRegs % 8 == 0 && kOtherRegs % 8 == 0, "register budget");
constexpr int kProducerWarp = 4 * kSplit, kMmaWarp = 4 * kSplit + 1;
static_assert(kSplit == 2 || kSplit == 4, "column split");
constexpr uint32_t kHalfBytes = kTileM * kBoxCols * 2;   // 16 KB: one 64-column TMA box of a Q, K or V tile
constexpr uint32_t kStageBytes = 32 * 128;            // output staging per softmax warp: 32 rows x 64 columns
constexpr uint32_t smem_bytes(int boxes)
{
    return 6 * boxes * kHalfBytes + 1024 /*alignment slack*/ + 1024 /*barriers, published items*/ + 2 * kSplit * 2 * kStageBytes;
}
// Keys per KV tile of an instance: weights in three bf16 parts take 3 x 16 columns of TMEM per 32 keys where S had 32; one
// box (head_dim <= 64) has the third part beside O, whose upper 64 columns are free, two boxes have room for 64 keys only.
__host__ __device__ constexpr int tile_keys(bool exact, int boxes) { return exact && boxes == 2 ? 64 : kTileN; }
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kColS = 0, kColO = 256;   // S (and P, aliased) of sub-tile t at kColS + 128 t; O at kColO + 128 t
// P (bf16 pairs) of keys 64 q .. 64 q + 63 sits at S column 64 q: every 32-key chunk of P
// lands in S columns that its thread has already read
constexpr uint32_t kWaitLimit = 1u << 20;
constexpr float kRescaleThreshold = 8.0f;

struct KernelParams {
    PrefillParams p;
    int32_t ord_seg[kMaxP];          // segments sorted by query-tile count, descending
    int32_t ord_nt[kMaxP];           // their query-tile counts
    int32_t band_rank[kMaxP + 1];    // tiles ranked above band b (levels ord_nt[b+1] < lv <= ord_nt[b])
    int32_t group;                   // query heads per KV head
    int32_t straddle;                // odd groups: ranked tiles have 256 rows, the last heads of their halves form an item
    uint64_t magic_per_tile, magic_ppk, magic_small[kMaxP];   // ceil(2^40 / d) for d = items per tile, per KV head, 1..kMaxP
    int32_t n_qtiles;                // total query tiles
    int32_t n_items;                 // ranked tiles x KV heads x items of one KV head
    int32_t n_kt;                    // KV tiles: ceil(total_kv / kTileN)
    int32_t *status;
    int32_t o_tma;                   // the output may leave through TMA stores (tensor map encoded)
    int32_t pairs;                   // exact instances: visibility is tested on explicit positions, in any order
    float sl2;                       // exact instances: logits to base 2 per unit of S
    GenericParams row;               // exact instances: the same call for the row routine that repairs non-finite rows
};

// Position tables of a general-position call (ints, in this order): minimum and maximum position of
// every query tile; then per KV position array (one per KV head when head-major, else one) the minimum and
// the maximum of every KV tile's key positions.  A query tile walks the KV tiles whose minimum does not exceed its
// largest position; those whose maximum does not exceed its smallest need no test.  A ragged last KV tile counts as
// never fully visible (maximum = INT_MAX).
struct PosTables {
    const int32_t *q_min, *q_max, *kv_min, *kv_max;
};
__device__ __host__ __forceinline__ PosTables pos_tables(const int32_t *tab, int n_qtiles, int n_arrays, int n_kt)
{
    PosTables t;
    t.q_min = tab; t.q_max = tab + n_qtiles;
    t.kv_min = tab + 2 * (size_t)n_qtiles; t.kv_max = t.kv_min + (size_t)n_arrays * n_kt;
    return t;
}
// Where an item's walk has tiles to skip, the producer leaves it in shared memory as a list (bit 15: the tile needs no
// test).  Longer lists than that has room for become "every tile up to the last visible one".  (Participants that hold
// alternate tokens of the sequence, four of 5001 rows in all, 32 / 8 heads: 955 us walking up to the last visible tile,
// 556 us with the list; contiguous members have nothing to skip.)
constexpr int kWalkMost = 128;

#ifdef FEDATTN_TRACE
// Debug build only: cycle stamps of one CTA's pipeline events, [tile][event].
__device__ long long g_trace[64 * 8];
#define TRACE(j, e) do { if (k == 0 && blockIdx.x == gridDim.x / 2 && (j) < 64) g_trace[(j) * 8 + (e)] = clock64(); } while (0)
#else
#define TRACE(j, e) do { } while (0)
#endif

// ---- PTX wrappers ---------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\t"
                 "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
    return ok != 0;
}
// Bounded wait.  Returns false (after flagging the status word once) when the limit is reached or
// another thread of this CTA already gave up.
__device__ __forceinline__ bool mbar_test_wait(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\t"
                 "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
    return ok != 0;
}
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, volatile int *abort_flag, int32_t *status,
                                          uint32_t limit = kWaitLimit)
{
    if (mbar_test_wait(bar, parity)) return true;        // phase already over: skip the suspending wait
    for (uint32_t it = 0; it < limit; ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if (*abort_flag) return false;
    }
    *abort_flag = 1;
    atomicMax(status, (int32_t)FEDATTN_ERR_TIMEOUT);
    return false;
}

// The same wait for the roles that hold few registers (producer, MMA issuer): the polling loop lives in
// one place instead of at every call site, which keeps those roles' code short.
__device__ __noinline__ bool mbar_wait_loop(uint64_t *bar, uint32_t parity, volatile int *abort_flag, int32_t *status)
{
    for (uint32_t it = 0; it < kWaitLimit; ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if (*abort_flag) return false;
    }
    *abort_flag = 1;
    atomicMax(status, (int32_t)FEDATTN_ERR_TIMEOUT);
    return false;
}
__device__ __forceinline__ bool mbar_wait_call(uint64_t *bar, uint32_t parity, volatile int *abort_flag, int32_t *status)
{
    if (mbar_test_wait(bar, parity)) return true;
    return mbar_wait_loop(bar, parity, abort_flag, status);
}

__device__ __forceinline__ void tma_load_3d(void *dst, const CUtensorMap *map, uint64_t *bar, int c0, int c1, int c2)
{
    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
                 " [%0], [%1, {%3, %4, %5}], [%2];"
                 ::"r"(smem_u32(dst)), "l"((uint64_t)map), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2)
                 : "memory");
}

__device__ __forceinline__ void tma_prefetch_3d(const CUtensorMap *map, int c0, int c1, int c2)
{
    asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global.tile [%0, {%1, %2, %3}];"
                 ::"l"((uint64_t)map), "r"(c0), "r"(c1), "r"(c2) : "memory");
}

// [32 rows x 64 columns] from shared memory (128-byte swizzle) to the output, one bulk group per call
__device__ __forceinline__ void tma_store_3d(const CUtensorMap *map, const void *src, int c0, int c1, int c2)
{
    asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.tile.bulk_group [%0, {%2, %3, %4}], [%1];"
                 ::"l"((uint64_t)map), "r"(smem_u32(src)), "r"(c0), "r"(c1), "r"(c2) : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
// the issuing thread's earlier bulk stores have read their shared memory
__device__ __forceinline__ void tma_store_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }

// true in exactly one lane of a converged warp
__device__ __forceinline__ bool elect_one()
{
    uint32_t pred;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(pred));
    return pred != 0;
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(uint64_t *bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// D[tmem] (+)= A[smem desc] * B[smem desc]
__device__ __forceinline__ void umma_ss(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t acc)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                 ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(acc) : "memory");
}
// D[tmem] (+)= A[tmem] * B[smem desc]
__device__ __forceinline__ void umma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t acc)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
                 ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(acc) : "memory");
}

#define FEDATTN_TMEM_LD32(taddr, r)                                                                          \
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 "                                                   \
                 "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"                                   \
                 "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"                  \
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),       \
                   "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),   \
                   "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]),             \
                   "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]),             \
                   "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])              \
                 : "r"(taddr) : "memory")

#define FEDATTN_TMEM_ST32(taddr, r)                                                                          \
    asm volatile("tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "                                             \
                 "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"                                  \
                 "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};"                         \
                 ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]),  \
                   "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]),          \
                   "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]),       \
                   "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]),       \
                   "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31]) : "memory")

#define FEDATTN_TMEM_ST16(taddr, r)                                                                          \
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "                                             \
                 "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"                                 \
                 ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]),  \
                   "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]),          \
                   "r"(r[14]), "r"(r[15]) : "memory")

#define FEDATTN_TMEM_LD16(taddr, r)                                                                          \
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 "                                                   \
                 "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"                           \
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),       \
                   "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),   \
                   "=r"(r[14]), "=r"(r[15])                                                                  \
                 : "r"(taddr) : "memory")

__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ float ex2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi)
{
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

__device__ __forceinline__ uint64_t pack_f32x2(float lo, float hi)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack_f32x2(uint64_t v, float &lo, float &hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t fma_f32x2(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ uint64_t add_f32x2(uint64_t a, uint64_t b)
{
    uint64_t r;
    asm("add.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ float max3(float a, float b, float c)
{
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// 2^x for a packed pair on the FMA/ALU pipes (no MUFU): x = n + f with n = round(x), |f| <= 1/2;
// 2^f by a degree-3 minimax polynomial (relative error 7.5e-5, far below the bf16 rounding of P),
// 2^n by adding n to the exponent field.  The magic constant 1.5 * 2^23 makes the low mantissa
// bits of x + magic hold n.  x is clamped at -125 so that the exponent arithmetic cannot wrap:
// anything smaller contributes 2^-125 instead of an even smaller value.  Needs x <= 100.
// bit (c & 7) set: column pair c takes the polynomial instead of ex2.approx.  2 of 8 pairs: 1, 2 and 3 of 8
// are within 1 % of each other (which is best depends on the board), none costs 2-3 %, 4 and 5 of 8 cost
// 2 and 5 % (the polynomial loads the ALU pipe as much as ex2 loads its own unit).
#ifndef FEDATTN_POLY_MASK
#define FEDATTN_POLY_MASK 0x11
#endif
constexpr uint32_t kPolyMask = FEDATTN_POLY_MASK;
__device__ __forceinline__ void exp2_poly_x2(uint64_t x2, float &p0, float &p1)
{
    float x0, x1;
    unpack_f32x2(x2, x0, x1);
    x0 = fmaxf(x0, -125.f); x1 = fmaxf(x1, -125.f);
    const uint64_t xc = pack_f32x2(x0, x1);
    const uint64_t magic = pack_f32x2(12582912.f, 12582912.f), neg_magic = pack_f32x2(-12582912.f, -12582912.f);
    const uint64_t neg_one = pack_f32x2(-1.f, -1.f);
    const uint64_t t2 = add_f32x2(xc, magic);
    const uint64_t f2 = fma_f32x2(add_f32x2(t2, neg_magic), neg_one, xc);
    uint64_t q2 = pack_f32x2(0.0551716685295105f, 0.0551716685295105f);
    q2 = fma_f32x2(q2, f2, pack_f32x2(0.2426111251115799f, 0.2426111251115799f));
    q2 = fma_f32x2(q2, f2, pack_f32x2(0.6932609677314758f, 0.6932609677314758f));
    q2 = fma_f32x2(q2, f2, pack_f32x2(0.9999280571937561f, 0.9999280571937561f));
    float q0, q1, t0, t1;
    unpack_f32x2(q2, q0, q1);
    unpack_f32x2(t2, t0, t1);
    p0 = __int_as_float(__float_as_int(q0) + (__float_as_int(t0) << 23));
    p1 = __int_as_float(__float_as_int(q1) + (__float_as_int(t1) << 23));
}

// Shared-memory matrix descriptor, 128-byte swizzle, 8-row groups 1024 bytes apart.
//   K-major operand (Q, K): rows of 64 bf16 = 128 B; a tile is two such [128 x 64] halves.
//   MN-major operand (V as B, N = head dim): 64 head-dim elements contiguous per key row;
//   lbo = distance between the two 64-wide head-dim halves.
__device__ __forceinline__ uint64_t make_desc(uint32_t saddr, uint32_t lbo_bytes, uint32_t sbo_bytes)
{
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3fff);
    d |= (uint64_t)((lbo_bytes >> 4) & 0x3fff) << 16;
    d |= (uint64_t)((sbo_bytes >> 4) & 0x3fff) << 32;
    d |= (uint64_t)1 << 46;            // descriptor version (Blackwell)
    d |= (uint64_t)2 << 61;            // SWIZZLE_128B
    return d;
}

// Instruction descriptor, kind::f16: D fp32, A/B bf16, M = 128, N columns.
__device__ __host__ constexpr uint32_t make_idesc(uint32_t n)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((n >> 3) << 17) | ((128u >> 4) << 24);
}
constexpr uint32_t kIdescPV = make_idesc(128) | (1u << 16);    // B (V) MN-major

// n / d for 0 <= n < 2^28 and 1 <= d <= 4096, with magic = ceil(2^40 / d)
__device__ __forceinline__ int fast_div(int n, uint64_t magic) { return (int)(((uint64_t)(uint32_t)n * magic) >> 40); }

// number of entries of the non-decreasing array pos[0..n) that are <= x
__device__ __forceinline__ int count_le(const int32_t *pos, int n, int x)
{
    int lo = 0, hi = n;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (ld_int(pos + mid) <= x) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// The same count, found by a converged warp together: every step probes 32 evenly spaced entries at
// once (one round trip to memory per step instead of one per halving), so 4096 entries take 3 steps.
// Every lane returns the count.
__device__ __forceinline__ int count_le_warp(const int32_t *pos, int n, int x, int lane)
{
    int lo = 0, hi = n;                                         // the count lies in [lo, hi]
    while (hi > lo) {
        const int width = hi - lo;
        if (width <= 32) {
            const bool le = lane < width && ld_int(pos + lo + lane) <= x;
            return lo + __popc(__ballot_sync(0xffffffffu, le));  // the entries <= x are a prefix
        }
        const int stride = (width + 31) >> 5;
        const int probe = min(lo + (lane + 1) * stride - 1, hi - 1);
        const int k = __popc(__ballot_sync(0xffffffffu, ld_int(pos + probe) <= x));
        if (k == 32) return hi;                                 // even the last entry is <= x
        hi = min(lo + (k + 1) * stride - 1, hi - 1);            // entry `hi` is > x: the count is at most hi
        lo = lo + k * stride;
    }
    return lo;
}

}  // namespace

// One unit of work: two sub-tiles of 128 query rows x one query head that share a KV head and a segment: two heads
// of one query tile, or (odd groups) the last head of two neighbouring query tiles.  Sub-tile 1 always has work and
// at least as many KV tiles as sub-tile 0, which may be missing (n_valid == 0).
struct Sub {
    int head, q_row0, n_valid, n_tiles;
};
struct Item {
    int kvh, seg, kv_begin;
    // The walk visits KV tiles 0 .. n_a-1 and then t_b0, t_b0+1, ...  (n_a == n_tiles unless the allowed
    // keys are two ranges: bidirectional remote-only attention, keys [0, a) and [b, T)).
    int n_a, t_b0, a, b;
    const int32_t *kvp;                // positions of this KV head's aggregated rows (sparse sync), or null
};
__device__ __forceinline__ int tile_of(const Item &it, int j) { return j < it.n_a ? j : it.t_b0 + (j - it.n_a); }

// allowed-prefix length c(row): keys kv_begin .. kv_begin + c - 1 are visible to query row r of the tile.
// Called by a converged warp with the same r in every lane (the searches are warp-cooperative).
__device__ __forceinline__ int prefix_len(const PrefillParams &p, const Item &it, const Sub &sub, int r, int lane)
{
    const int pos = sub.q_row0 + r;
    const int T = (int)p.total_kv;
    if (!p.sync) {
        const int seg_len = p.cu[it.seg + 1] - p.cu[it.seg];
        return p.causal ? min(pos - p.cu[it.seg] + 1, seg_len) : seg_len;
    }
    if (p.remote_only) {                               // what lies before the row's own segment
        const int before = p.cu[it.seg];
        return it.kvp ? count_le_warp(it.kvp, T, before - 1, lane) : min(before, T);
    }
    if (!p.causal) return T;
    if (!it.kvp) return min(pos + 1, T);
    return count_le_warp(it.kvp, T, pos, lane);
}

// Explicit positions without tables (exact instances): key x is visible to a row iff pos(x) <= lo, or, when
// two_sided, pos(x) >= hi.  lo depends on the row (explicit or implied position) or on its segment (remote-only).
struct PairRule {
    int lo, hi;
    bool two_sided;
    __device__ bool sees(int pos) const { return pos <= lo || (two_sided && pos >= hi); }
};
__device__ __forceinline__ PairRule pair_rule(const PrefillParams &p, const Item &it, const Sub &sub, int r)
{
    PairRule rule;
    rule.two_sided = p.remote_only && !p.causal;
    rule.hi = p.remote_only ? p.cu[it.seg + 1] : 0;
    if (p.remote_only) rule.lo = p.cu[it.seg] - 1;
    else {
        const int row = sub.q_row0 + min(r, sub.n_valid - 1);
        rule.lo = p.q_pos ? ld_int(p.q_pos + row) : row;
    }
    return rule;
}
// Number of KV tiles up to the last one with a key visible to some row of the sub-tile.  Walks the key
// positions backwards, 512 at a time (sixteen coalesced loads in flight per lane); called by a converged warp.
template <int kKeys>
__device__ __forceinline__ int last_visible_tile(const KernelParams &kp, const Item &it, const Sub &sub, int lane)
{
    const PrefillParams &p = kp.p;
    PairRule any = pair_rule(p, it, sub, lane);
    for (int r = lane + 32; r < kTileM; r += 32) any.lo = max(any.lo, pair_rule(p, it, sub, r).lo);
    any.lo = __reduce_max_sync(0xffffffffu, any.lo);
    const int T = (int)p.total_kv;
    for (int base = ((T - 1) / 512) * 512; base >= 0; base -= 512) {
        int last = -1;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const int key = base + 32 * i + lane;
            if (key < T && any.sees(it.kvp ? ld_int(it.kvp + key) : key)) last = key;
        }
        last = __reduce_max_sync(0xffffffffu, last);
        if (last >= 0) return last / kKeys + 1;
    }
    return 0;
}

// Called by a converged warp (all lanes get the same item).  kSpecial: the kernel instance that also
// serves explicit positions and bidirectional remote-only attention (two key ranges); the plain instance
// carries none of their state.  Causal remote-only attention is one more prefix mask: plain instance.
template <bool kSpecial, bool kExact, bool kHalves, int kKeys>
__device__ __forceinline__ Item decode_item(const KernelParams &kp, int item, int lane, Sub (&sub)[2], uint16_t *walk)
{
    const PrefillParams &p = kp.p;
    Item it;
    // divisions by launch constants go through host-computed reciprocals (kp.magic_*)
    const int g = kp.group;
    const int ppk = kHalves || kp.straddle ? g : (g + 1) >> 1;  // items per ranked tile and KV head
    const int per_tile = p.hkv * ppk;
    const int tile_rank = fast_div(item, kp.magic_per_tile);
    const int rem = item - tile_rank * per_tile;
    it.kvh = fast_div(rem, kp.magic_ppk);
    const int u = rem - it.kvh * ppk;
    // Heavy tiles first: query tiles are ranked by their index inside their segment, descending
    // (a causal tile's KV-tile count is that index + 1).  Level lv holds tile lv-1 of every segment
    // that has at least lv tiles.  With the segments sorted by tile count (ord_nt, descending), the
    // levels ord_nt[b+1] < lv <= ord_nt[b] form band b, in which every level holds the b+1 longest
    // segments; band_rank[b] = number of tiles above band b (host-computed).
    int b = 0;
    while (b + 1 < p.n_seg && tile_rank >= kp.band_rank[b + 1]) ++b;
    const int in_band = tile_rank - kp.band_rank[b];
    const int down = fast_div(in_band, kp.magic_small[b]);      // in_band / (b + 1): levels below the band's top
    const int lo = kp.ord_nt[b] - down;
    const int seg = kp.ord_seg[in_band - down * (b + 1)];
    const int end = p.cu[seg + 1];
    it.seg = seg;
    it.kvp = p.kv_pos ? p.kv_pos + (p.kv_head_major ? (int64_t)it.kvh * p.total_kv : 0) : nullptr;
    it.kv_begin = p.sync ? 0 : p.cu[seg];
    it.t_b0 = 0; it.a = 0; it.b = 0;
    const int row0 = p.cu[seg] + (lo - 1) * (!kHalves && kp.straddle ? 2 * kTileM : kTileM);
    bool two_rows = false;
    if (kHalves) {
        sub[0].head = sub[1].head = it.kvh * g + u;
        sub[0].q_row0 = sub[1].q_row0 = row0;
    } else if (kp.straddle) {
        // items 0 .. g-2: the head pairs of the first and of the second query tile; item g-1: both tiles' last head
        const int half = g >> 1;
        two_rows = u == g - 1;
        const int second = !two_rows && u >= half ? 1 : 0;
        const int h = two_rows ? g - 1 : 2 * (u - second * half);
        sub[0].head = it.kvh * g + h;
        sub[1].head = sub[0].head + (two_rows ? 0 : 1);
        sub[0].q_row0 = row0 + second * kTileM;
        sub[1].q_row0 = sub[0].q_row0 + (two_rows ? kTileM : 0);
    } else {
        sub[0].head = it.kvh * g + 2 * u;
        sub[1].head = sub[0].head + 1;
        sub[0].q_row0 = sub[1].q_row0 = row0;
    }
    sub[0].n_valid = max(0, min(kTileM, end - sub[0].q_row0));
    sub[1].n_valid = max(0, min(kTileM, end - sub[1].q_row0));
    if (!kHalves && !kp.straddle && 2 * u + 1 >= g) sub[1].n_valid = 0;     // odd group: the last pair is single
    if (sub[1].n_valid == 0) { const Sub x = sub[0]; sub[0] = sub[1]; sub[1] = x; }
    sub[0].n_tiles = sub[1].n_tiles = 0;
    it.n_a = 0;
    if (sub[1].n_valid == 0) return it;                         // no such query tile
    if (kSpecial && !kExact && p.general) {
        // both sub-tiles walk what either may see
        const PosTables pt = pos_tables(p.tab, kp.n_qtiles, p.kv_head_major ? p.hkv : 1, kp.n_kt);
        const size_t first = p.kv_head_major ? (size_t)it.kvh * kp.n_kt : 0;
        int q_max = ld_int(pt.q_max + (sub[1].q_row0 >> 7)), q_min = ld_int(pt.q_min + (sub[1].q_row0 >> 7));
        if (two_rows && sub[0].n_valid > 0) {
            q_max = max(q_max, ld_int(pt.q_max + (sub[0].q_row0 >> 7)));
            q_min = min(q_min, ld_int(pt.q_min + (sub[0].q_row0 >> 7)));
        }
        int n = 0, last = 0, run = 0;                           // visible tiles, end of the last, leading run without a test
        bool in_run = true;
        for (int t0 = 0; t0 < kp.n_kt; t0 += 32) {
            const int t = min(t0 + lane, kp.n_kt - 1);
            const bool in = t0 + lane < kp.n_kt;
            const uint32_t seen = __ballot_sync(0xffffffffu, in && ld_int(pt.kv_min + first + t) <= q_max);
            const uint32_t free = __ballot_sync(0xffffffffu, in && ld_int(pt.kv_max + first + t) <= q_min);
            const int at = n + __popc(seen & ((1u << lane) - 1u));
            if (((seen >> lane) & 1u) && at < kWalkMost) walk[at] = (uint16_t)(t | (((free >> lane) & 1u) << 15));
            n += __popc(seen);
            if (seen) last = t0 + 32 - __clz(seen);
            if (in_run) run += free == 0xffffffffu ? 32 : __ffs(~free) - 1;
            in_run = in_run && free == 0xffffffffu;
        }
        // nothing to skip (contiguous members), or no room for the list: a prefix of tiles, of which `run` need no test
        it.b = n == last || n > kWalkMost || kp.n_kt > 0x7fff ? run : -1;
        if (it.b >= 0) n = last;
        it.n_a = sub[1].n_tiles = n;
        sub[0].n_tiles = sub[0].n_valid > 0 ? n : 0;
    } else if (p.sync && p.remote_only && !(kExact && kp.pairs)) {
        // keys [0, a) lie before the rows' segment; when bidirectional (special instance only), keys [b, T)
        // after it count too
        const int T = (int)p.total_kv, n_t = (T + kKeys - 1) / kKeys;
        it.a = prefix_len(p, it, sub[1], 0, lane);
        it.n_a = (it.a + kKeys - 1) / kKeys;
        sub[1].n_tiles = it.n_a;
        it.b = T;
        if (kSpecial && !p.causal) {
            it.b = it.kvp ? count_le_warp(it.kvp, T, end - 1, lane) : min(end, T);
            it.t_b0 = it.b >= T ? n_t : max(it.b / kKeys, it.n_a);
            sub[1].n_tiles = it.n_a + (n_t - it.t_b0);
        }
        sub[0].n_tiles = sub[0].n_valid > 0 ? sub[1].n_tiles : 0;
    } else {
        // (one copy of the searches' code, walked a second time when the sub-tiles are different query tiles)
#pragma unroll 1
        for (int again = two_rows && sub[0].n_valid > 0 ? 1 : 0;; again = 0) {
            const Sub x = again ? sub[0] : sub[1];
            int n;
            if (kExact && kp.pairs) n = last_visible_tile<kKeys>(kp, it, x, lane);
            else n = (prefix_len(p, it, x, x.n_valid - 1, lane) + kKeys - 1) / kKeys;
            if (again) { sub[0].n_tiles = n; continue; }
            sub[1].n_tiles = n;
            break;
        }
        if (!two_rows && sub[0].n_valid > 0) sub[0].n_tiles = sub[1].n_tiles;
        if (sub[0].n_tiles > sub[1].n_tiles) { const Sub x = sub[0]; sub[0] = sub[1]; sub[1] = x; }
        it.n_a = sub[1].n_tiles;
    }
    if (kHalves) {                                              // sub-tile 1 walks tiles 0, 2, ..., sub-tile 0 tiles 1, 3, ...
        sub[0].n_tiles = sub[1].n_tiles >> 1;
        sub[1].n_tiles -= sub[0].n_tiles;
        if (sub[0].n_tiles == 0) sub[0].n_valid = 0;
    }
    return it;
}

// Persistent kernel: one CTA per SM walks the work items item = blockIdx.x, blockIdx.x + gridDim.x, ...
// Barrier phases run on: per-CTA counters of KV tiles (git) and of non-empty items (qn) give stages
// and parities, so the producer prefetches the next item's K/V and Q while the current item's last
// tiles and its epilogue are still in flight.
//
// kBoxes: 64-column boxes per tile (head_dim <= 64: one; <= 128: two).  kExact: the weights P keep their 24 bits (three
// bf16 parts, three PV products), every exponential is ex2, and rows that come out non-finite are redone by the row
// routine.  It serves the head dims below 128, whose users had fp32 weights from the SIMT kernel.  Bound by the chain
// softmax -> PV -> S, which carries the products (d = 64: 4 + 3 x 8 MMAs per tile, the latter of N = 64, no faster than of
// N = 128): two parts, 16 bits, take 20.7 and 47.1 us, three 24.7 and 55.9 for the local and the sync call of six ragged
// segments of 2160 tokens, 16 / 4 heads of 64 channels (2436 and 10994 us with one warp per row, fp32 FMA).  The error of o against fp64 is that of fp32 weights (the
// rounding of the bf16 output, 1.587459e-3 there; 1.587460e-3 with two parts), lse 3.2e-8 -> 2.9e-8 relative.
//
// kHalves: both sub-tiles are the SAME query tile of one head; sub-tile 1 walks the even KV tiles and sub-tile 0 the odd
// ones, and the epilogue merges the two partial rows (O_0 and O_1 have the same TMEM lanes, so every thread reads both;
// maximum and sum go through shared memory).  An item takes half as long as a pair of heads over the same keys: for
// launches whose longest walk, not their sum of work, decides.  K and V tiles then serve one product each, which
// doubles what the CTA reads from L2.
template <bool kSpecial, int kBoxes, bool kExact, bool kHalves>
__global__ void __launch_bounds__(kThreads, 1)
prefill_sm100_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                     const __grid_constant__ CUtensorMap map_v, const __grid_constant__ CUtensorMap map_o,
                     const __grid_constant__ KernelParams kp)
{
    extern __shared__ uint8_t smem_raw[];
    constexpr uint32_t kTileBytes = kBoxes * kHalfBytes;                            // a Q tile
    constexpr int kKeys = tile_keys(kExact, kBoxes), kChunks = kKeys / 32;         // keys of a KV tile, in chunks of 32
    constexpr int kPartKeys = kKeys / kSplit;                                      // keys of a half of P
    constexpr uint32_t kColP3 = (kBoxes == 1 ? kColO : kColS) + 64;                // exact instances: third parts of sub-tile 0's P
    constexpr uint32_t kKvBox = kKeys * kBoxCols * 2, kKvBytes = kBoxes * kKvBox;  // a K or V tile
    const PrefillParams &p = kp.p;
    const int d = kExact ? p.d : kBoxes * kBoxCols;
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t *sQ = smem;                                  // [2 sub-tiles][tile]
    uint8_t *sK = smem + 2 * kTileBytes;                 // [2 stages][tile]
    uint8_t *sV = sK + 2 * kKvBytes;                     // [2 stages][tile]
    uint64_t *bars = reinterpret_cast<uint64_t *>(sV + 2 * kKvBytes);
    uint64_t *q_full = bars + 0, *q_empty = bars + 1;
    uint64_t *k_full = bars + 2, *k_empty = bars + 4, *v_full = bars + 6, *v_empty = bars + 8;
    uint64_t *s_full = bars + 10, *o_done = bars + 12, *o_free = bars + 14;
    uint64_t *p_full = bars + 16;                        // [sub-tile][column part]
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 24);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(bars + 25);
    // what the producer tells the MMA issuer about an item, published before the item's Q load is issued
    // and read after q_full: {KV tiles of sub-tile 1, of sub-tile 0}; -1 tiles = no more items.  Two slots, like the phases.
    volatile int *item_info = reinterpret_cast<volatile int *>(bars + 26);
    // The producer decodes every work item once and publishes it here for the softmax warps (two slots of
    // 16 ints, filled an item ahead), so that decoding is not on their path between two items.
    uint64_t *item_full = bars + 20, *item_empty = bars + 22;
    uint64_t *halves_met = bars + 28;                    // halves: both warpgroups have left their partials' (m, l)
    volatile int *item_pub = reinterpret_cast<volatile int *>(bars + 32);
    uint16_t *walks = reinterpret_cast<uint16_t *>(bars + 48);      // general: [slot][kWalkMost]
    uint8_t *stage = sV + 2 * kKvBytes + 1024;           // [softmax warp][32 rows][128 B], 128-byte swizzle

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int n_items = kp.n_items;
    // Static schedule: round k hands item k*G + c to CTA c, in reversed CTA order on odd rounds, so
    // that with items sorted by cost every CTA gets a similar total.
    auto item_of = [&](int k) -> int {
        const int c = (k & 1) ? (int)gridDim.x - 1 - (int)blockIdx.x : (int)blockIdx.x;
        return k * (int)gridDim.x + c;
    };

    grid_wait();                                        // nothing is read or written before
    // ---- setup ------------------------------------------------------------------------------------
    if (tid == 0) {
        mbar_init(q_full, 1); mbar_init(q_empty, 1);
        for (int i = 0; i < 2; ++i) {
            mbar_init(k_full + i, 1); mbar_init(k_empty + i, 1); mbar_init(v_full + i, 1); mbar_init(v_empty + i, 1);
            mbar_init(s_full + i, 1); mbar_init(o_done + i, 1);
            mbar_init(o_free + i, kHalves ? 8 : 4);             // (halves: every warp reads both accumulators)
            for (int q = 0; q < kSplit; ++q) mbar_init(p_full + kSplit * i + q, 4);
            mbar_init(item_full + i, 1); mbar_init(item_empty + i, 2 * kSplit * 2);
        }
        mbar_init(halves_met, 8);
        *abort_flag = (*reinterpret_cast<volatile int32_t *>(kp.status) == FEDATTN_ERR_TIMEOUT) ? 1 : 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == kProducerWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(tmem_slot)), "r"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    // A timeout that an earlier kernel reported and nobody has polled yet: this launch does no work
    // (every wait would run out again) and leaves its outputs untouched.
    const int n_rounds = *abort_flag ? 0 : (n_items + (int)gridDim.x - 1) / (int)gridDim.x;

    // every warp of a warpgroup executes the same setmaxnreg (first thing in its role); the increase
    // waits for the decrease
    if (warp == kProducerWarp) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kOtherRegs));
        // ================= TMA producer =================
        // The whole warp decodes the work items (their searches are warp-cooperative); lane 0 waits and
        // issues the copies.
        if (lane == 0) {
            asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&map_q) : "memory");
            asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&map_k) : "memory");
            asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&map_v) : "memory");
        }
        int git = 0, qn = 0, pn = 0;
        // After a wait that ran out nothing is published or loaded any more: a slot may still be read, a buffer still be
        // written.  (All lanes get lane 0's answer.)
        auto slot_free = [&]() -> bool {
            bool ok = true;
            if (lane == 0 && pn >= 2) ok = mbar_wait_call(item_empty + (pn & 1), ((pn >> 1) - 1) & 1, abort_flag, kp.status);
            return __shfl_sync(0xffffffffu, ok, 0);
        };
        for (int k = 0; k < n_rounds; ++k) {
            const int item = item_of(k);
            if (item >= n_items) continue;
            Sub sub[2];
            const bool general = kSpecial && !kExact && p.general;
            if (general && !slot_free()) break;                 // the walk goes into the slot while decoding
            uint16_t *walk = walks + (pn & 1) * kWalkMost;
            const Item it = decode_item<kSpecial, kExact, kHalves, kKeys>(kp, item, lane, sub, walk);
            __syncwarp();
            const int n_tiles = sub[1].n_tiles + (kHalves ? sub[0].n_tiles : 0);
            if (!general && !slot_free()) break;
            if (lane == 0) {
                volatile int *slot = item_pub + (pn & 1) * 16;
                slot[0] = it.kvh; slot[1] = it.seg; slot[2] = it.kv_begin; slot[3] = it.n_a; slot[4] = it.t_b0;
                slot[5] = it.a; slot[6] = it.b;
#pragma unroll
                for (int t = 0; t < 2; ++t) {
                    slot[8 + 4 * t] = sub[t].head; slot[9 + 4 * t] = sub[t].q_row0; slot[10 + 4 * t] = sub[t].n_valid;
                    slot[11 + 4 * t] = sub[t].n_tiles;
                }
                mbar_arrive(item_full + (pn & 1));
                // this item's Q on its way into L2: the load itself has to wait for the Q buffer
#pragma unroll
                for (int t = kHalves ? 1 : 0; t < 2; ++t)
                    if (sub[t].n_tiles > 0) {
                        tma_prefetch_3d(&map_q, 0, sub[t].head, sub[t].q_row0);
                        if (kBoxes == 2) tma_prefetch_3d(&map_q, 64, sub[t].head, sub[t].q_row0);
                    }
            }
            ++pn;
            if (n_tiles == 0) continue;
            int issued = 0;                                     // lane 0: KV tiles of the item on their way
            bool q_free = true;
            if (lane == 0 && qn > 0) q_free = mbar_wait_call(q_empty, (qn - 1) & 1, abort_flag, kp.status);   // previous item's S MMAs done
            if (lane == 0 && q_free) {
                item_info[(qn & 1) * 2] = sub[1].n_tiles;
                item_info[(qn & 1) * 2 + 1] = sub[0].n_tiles;
                mbar_expect_tx(q_full, !kHalves && sub[0].n_tiles > 0 ? 2 * kTileBytes : kTileBytes);
#pragma unroll
                for (int t = kHalves ? 1 : 0; t < 2; ++t)       // (halves share sub-tile 1's Q)
                    if (sub[t].n_tiles > 0) {
                        tma_load_3d(sQ + t * kTileBytes, &map_q, q_full, 0, sub[t].head, sub[t].q_row0);
                        if (kBoxes == 2) tma_load_3d(sQ + t * kTileBytes + kHalfBytes, &map_q, q_full, 64, sub[t].head, sub[t].q_row0);
                    }
                const bool listed = general && it.b < 0;
                for (int j = 0; j < n_tiles; ++j) {
                    const int gt = git + j, st = gt & 1, use = gt >> 1;
                    int tile = kSpecial ? tile_of(it, j) : j;
                    if (listed) tile = walk[j] & 0x7fff;
                    const int row = it.kv_begin + tile * kKeys;
                    const int c1 = p.kv_head_major ? row : it.kvh, c2 = p.kv_head_major ? it.kvh : row;
                    if (gt >= 2 && !mbar_wait_call(k_empty + st, (use - 1) & 1, abort_flag, kp.status)) break;
                    issued = j + 1;
                    TRACE(j, 7);
                    mbar_expect_tx(k_full + st, kKvBytes);
                    tma_load_3d(sK + st * kKvBytes, &map_k, k_full + st, 0, c1, c2);
                    if (kBoxes == 2) tma_load_3d(sK + st * kKvBytes + kKvBox, &map_k, k_full + st, 64, c1, c2);
                    if (gt >= 2 && !mbar_wait_call(v_empty + st, (use - 1) & 1, abort_flag, kp.status)) break;
                    mbar_expect_tx(v_full + st, kKvBytes);
                    tma_load_3d(sV + st * kKvBytes, &map_v, v_full + st, 0, c1, c2);
                    if (kBoxes == 2) tma_load_3d(sV + st * kKvBytes + kKvBox, &map_v, v_full + st, 64, c1, c2);
                }
            }
            issued = __shfl_sync(0xffffffffu, issued, 0);
            git += issued;
            qn += __shfl_sync(0xffffffffu, (int)q_free, 0);
            if (issued < n_tiles) break;
        }
        if (lane == 0) {
            // end marker for the MMA issuer, in the slot and phase the next item would have used
            if (qn > 0) mbar_wait_call(q_empty, (qn - 1) & 1, abort_flag, kp.status);
            item_info[(qn & 1) * 2] = -1;
            mbar_arrive(q_full);
            if (*abort_flag) {
                // give the copies still in flight a bounded chance to land before the CTA retires
                for (int gt = max(0, git - 2); gt < git; ++gt) {
                    for (uint32_t w = 0; w < 4096 && !mbar_try_wait(k_full + (gt & 1), (gt >> 1) & 1); ++w) {}
                    for (uint32_t w = 0; w < 4096 && !mbar_try_wait(v_full + (gt & 1), (gt >> 1) & 1); ++w) {}
                }
                if (qn > 0)
                    for (uint32_t w = 0; w < 4096 && !mbar_try_wait(q_full, (qn - 1) & 1); ++w) {}
            }
        }
    } else if (warp == kMmaWarp) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kOtherRegs));
        // ================= MMA issuer =================
        // Issue order per item  S0(0) S1(0) | PV0(0) S0(1) | PV1(0) S1(1) | PV0(1) S0(2) | ...  : while one
        // sub-tile's softmax runs, the tensor pipe works on the other sub-tile.
        // The whole warp walks the loop (waits included) so that control flow and operand descriptors
        // stay warp-uniform; one elected lane issues the tcgen05 instructions.  Issued from inside a
        // single-lane branch the same instructions sustain only ~83 cycles per MMA instead of 64.
        const bool leader = elect_one();
        const uint32_t idesc_pv = make_idesc((uint32_t)(d + 15) & ~15u) | (1u << 16);     // exact instances: N = head_dim
        const uint32_t aQ = smem_u32(sQ), aK = smem_u32(sK), aV = smem_u32(sV);
        const uint64_t dQ = make_desc(aQ, 16, 1024), dK = make_desc(aK, 16, 1024), dV = make_desc(aV, kKvBox, 1024);
        auto issue_s = [&](int t, int st) {
            if (leader) {
#pragma unroll
                for (int ks = 0; ks < kBoxes * kBoxCols / 16; ++ks) {
                    const uint32_t off_q = ((ks >> 2) * kHalfBytes + (ks & 3) * 32) >> 4, off_k = ((ks >> 2) * kKvBox + (ks & 3) * 32) >> 4;
                    if (!kExact || 16 * ks < d)                  // columns beyond head_dim are zero in both tiles
                    umma_ss(tmem_base + kColS + t * 128, dQ + (uint64_t)((kHalves ? 1 : t) * (kTileBytes >> 4) + off_q),
                            dK + (uint64_t)(st * (kKvBytes >> 4) + off_k), make_idesc(kKeys), ks > 0);
                }
            }
        };
        auto commit = [&](uint64_t *bar) { if (leader) tc_commit(bar); };
        // ring counts the KV tiles; git / qn the KV tiles / items of sub-tile 1, git0 / qn0 those of sub-tile 0, which
        // may be missing or end earlier.
        int ring = 0, git = 0, qn = 0, git0 = 0, qn0 = 0;
        for (;;) {
            // the producer decodes the work items; this warp only learns their shape (decoding them here as
            // well does not fit into this role's 64 registers)
            if (!mbar_wait_call(q_full, qn & 1, abort_flag, kp.status)) break;
            const int n1 = item_info[(qn & 1) * 2];
            if (n1 < 0) break;
            const int n0 = item_info[(qn & 1) * 2 + 1];
            const int n = kHalves ? n0 + n1 : n1;                // KV tiles of the item
            // halves take the sub-tiles in the order of their tiles: 1 (tile 0) first
            for (int i = kHalves || n0 > 0 ? 0 : 1; i < 2; ++i) {
                const int t = kHalves ? 1 - i : i, tile = kHalves ? i : 0, st = (ring + tile) & 1;
                if (kHalves && tile >= n) break;
                mbar_wait_call(k_full + st, ((ring + tile) >> 1) & 1, abort_flag, kp.status);
                tc_fence_after();
                issue_s(t, st);
                commit(s_full + t);
                if (kHalves || t == 1) {
                    commit(k_empty + st);
                    if (tile == n - 1) commit(q_empty);          // last S of this item issued
                }
            }
            for (int j = 0; j < n1; ++j) {
                for (int i = kHalves || j < n0 ? 0 : 1; i < 2; ++i) {
                    const int t = kHalves ? 1 - i : i;
                    if (kHalves && t == 0 && j >= n0) break;
                    const int tile = kHalves ? 2 * j + i : j;
                    const int gt = ring + tile, st = gt & 1, ph = (gt >> 1) & 1;
                    const int gsub = (t ? git : git0) + j, qsub = t ? qn : qn0;
                    // (sub-tile 1 of a shared tile: sub-tile 0 has waited for it)
                    if (kHalves || t == 0 || j >= n0) mbar_wait_call(v_full + st, ph, abort_flag, kp.status);
                    if (j == 0 && qsub > 0) mbar_wait_call(o_free + t, (qsub - 1) & 1, abort_flag, kp.status);
#pragma unroll
                    for (int q = 0; q < kSplit; ++q) {
                        mbar_wait_call(p_full + kSplit * t + q, gsub & 1, abort_flag, kp.status);
                        if (lane == 0 && q == 0) TRACE(j, 2 + t);
                        tc_fence_after();
                        if (leader) {
#pragma unroll
                            for (int kk = 0; kk < kPartKeys / 16; ++kk) {
                                const int ks = q * (kPartKeys / 16) + kk;
                                const uint64_t desc = dV + (uint64_t)(st * (kKvBytes >> 4) + ks * (2048 >> 4));
                                if (kExact) {                    // chunk of 32 keys: 16 columns each of the first, second, third parts
                                    const uint32_t a = tmem_base + kColS + t * 128 + 32 * (ks >> 1) + 8 * (ks & 1);
                                    const uint32_t a3 = tmem_base + kColP3 + t * 128 + 16 * (ks >> 1) + 8 * (ks & 1);
                                    umma_ts(tmem_base + kColO + t * 128, a, desc, idesc_pv, (j > 0 || ks > 0));
                                    umma_ts(tmem_base + kColO + t * 128, a + 16, desc, idesc_pv, 1);
                                    umma_ts(tmem_base + kColO + t * 128, a3, desc, idesc_pv, 1);
                                } else {
                                    umma_ts(tmem_base + kColO + t * 128, tmem_base + kColS + t * 128 + q * kPartKeys + kk * 8, desc,
                                            kIdescPV, (j > 0 || ks > 0));
                                }
                            }
                        }
                    }
                    commit(o_done + t);
                    if (kHalves || t == 1) commit(v_empty + st);
                    if (j + 1 < (t ? n1 : n0)) {
                        const int next = tile + (kHalves ? 2 : 1), st1 = (ring + next) & 1;
                        if (kHalves || t == 0 || j + 1 >= n0)
                            mbar_wait_call(k_full + st1, ((ring + next) >> 1) & 1, abort_flag, kp.status);
                        issue_s(t, st1);
                        commit(s_full + t);
                        if (kHalves || t == 1) {
                            commit(k_empty + st1);
                            if (next == n - 1) commit(q_empty);
                        }
                    }
                    if (t == 1 && lane == 0) TRACE(j, 4);
                }
            }
            ring += n;
            git += n1;
            ++qn;
            if (n0 > 0) { git0 += n0; ++qn0; }
        }
    } else if (warp >= 4 * kSplit) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kOtherRegs));      // the two idle warps of that warpgroup
        // One of them checks what the prefix-count mask relies on: key positions that never decrease
        // along the aggregated rows of a head.  The CTAs share the pairs (i, i + 1) among them.
        if (!kExact && warp == kMmaWarp + 1 && p.kv_pos && !p.general && p.sync && (p.causal || p.remote_only) && p.total_kv > 1) {
            const int64_t per = p.total_kv - 1, total = per * (p.kv_head_major ? p.hkv : 1);
            bool bad = false;
            for (int64_t i = (int64_t)blockIdx.x * 32 + lane; i < total; i += (int64_t)gridDim.x * 32) {
                const int64_t a = i / per, e = a * p.total_kv + (i - a * per);
                bad |= ld_int(p.kv_pos + e) > ld_int(p.kv_pos + e + 1);
            }
            if (bad) atomicMax(kp.status, (int32_t)FEDATTN_ERR_ORDER);
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kSoftmaxRegs));
        // ================= softmax + epilogue =================
        // Warpgroup t serves sub-tile t (one query head of one query tile) on its own: thread = query row r = TMEM lane,
        // all key columns of the S tile, the whole row of O.  During the walk the two warpgroups never meet (those of a
        // halved item do in the epilogue): no row maximum or row sum has to be exchanged, and while one is in the
        // serial part of its visit (wait, TMEM load, maximum) the other computes.  A thread reads its row of S from TMEM once and keeps
        // its values in registers for both walks (maximum, then exponentials).
        const int t = warp >> 2;                                // sub-tile of this warpgroup
        const int r = tid & 127;                                // query row = TMEM lane
        const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t tS = tmem_base + lane_base + kColS + t * 128;   // fp32 S; bf16 P of keys 64q.. at column 64q
        const uint32_t tO = tmem_base + lane_base + kColO + t * 128;
        const float sl2 = kExact ? kp.sl2 : p.scale * 1.4426950408889634f;
        const uint64_t sl2_2 = pack_f32x2(sl2, sl2);
        int gsub = 0;                                           // KV tiles this sub-tile has been through
        auto below32 = [](int n) -> uint32_t { return n <= 0 ? 0u : (n >= 32 ? 0xffffffffu : (1u << n) - 1u); };

        // One visit = the softmax of one S tile.  kPartial: some row of the tile has masked columns; bit i of
        // vm[c] says whether column 32 c + i is visible to this thread's row.  Masked columns become -inf and
        // every exponential goes through ex2.approx, which maps -inf to 0; in unmasked tiles a fixed subset of
        // the columns takes the polynomial so that the ex2 unit is not the bottleneck.
        // kAnyFirst: the tile in which a row sees its first key may be any of the walk (explicit positions).
        constexpr bool kAnyFirst = kSpecial || kExact;
        auto visit = [&](auto partial_tag, int j, int gt, const uint32_t (&vm)[4], float &m_used, float &l) {
            constexpr bool kPartial = decltype(partial_tag)::value;
            mbar_wait(s_full + t, gt & 1, abort_flag, kp.status);
            if (tid == 0) TRACE(j, t ? 5 : 0);
            tc_fence_after();
            // the whole row of S in registers: read from TMEM once, used for the maximum and the exponentials
            uint32_t s0[32], s1[32], s2[32], s3[32];
            float mx[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) mx[i] = -INFINITY;
            FEDATTN_TMEM_LD32(tS, s0);
            FEDATTN_TMEM_LD32(tS + 32, s1);
            tmem_wait_ld();
            if (kChunks == 4) {
                FEDATTN_TMEM_LD32(tS + 64, s2);
                FEDATTN_TMEM_LD32(tS + 96, s3);
            }
#pragma unroll
            for (int c = 0; c < kChunks; ++c) {
                uint32_t *cur = c == 0 ? s0 : (c == 1 ? s1 : (c == 2 ? s2 : s3));
                if (c == 2) tmem_wait_ld();
                if (kPartial) {
#pragma unroll
                    for (int i = 0; i < 32; ++i)
                        if (!((vm[c] >> i) & 1u)) cur[i] = 0xff800000u;          // -inf
                }
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    mx[i] = max3(mx[i], __uint_as_float(cur[2 * i]), __uint_as_float(cur[2 * i + 1]));
                    mx[i] = max3(mx[i], __uint_as_float(cur[16 + 2 * i]), __uint_as_float(cur[16 + 2 * i + 1]));
                }
            }
            const float rm = fmaxf(max3(mx[0], mx[1], mx[2]), fmaxf(max3(mx[3], mx[4], mx[5]), fmaxf(mx[6], mx[7])));
            const float t_max = rm * sl2;
            if (j == 0) {
                // (a row of a prefix mask that sees nothing of its first tile sees nothing at all)
                m_used = (!kAnyFirst && t_max == -INFINITY) ? 0.f : t_max;
            } else {
                // The exponent reference moves only when the maximum grew by more than 2^8; then what
                // this row has accumulated so far (O in TMEM, l) is rescaled to the new reference.
                const bool need = t_max > m_used + kRescaleThreshold;
                if (__any_sync(0xffffffffu, need)) {
                    const float alpha = need ? ex2(m_used - t_max) : 1.f;
                    mbar_wait(o_done + t, (gt - 1) & 1, abort_flag, kp.status);   // O holds tiles 0..j-1
                    tc_fence_after();
#pragma unroll 1
                    for (int oc = 0; oc < 2 * kBoxes; ++oc) {
                        uint32_t o[32];
                        FEDATTN_TMEM_LD32(tO + oc * 32, o);
                        tmem_wait_ld();
#pragma unroll
                        for (int c = 0; c < 32; ++c) o[c] = __float_as_uint(__uint_as_float(o[c]) * alpha);
                        FEDATTN_TMEM_ST32(tO + oc * 32, o);
                    }
                    if (need) { l *= alpha; m_used = t_max; }
                }
            }
            // ---- pass 2: exponentials, row sum, P ----
            // (a row that has seen no key yet keeps the reference -inf, all its weights are 0)
            const float m_ref = kAnyFirst && m_used == -INFINITY ? 0.f : m_used;
            const uint64_t negm2 = pack_f32x2(-m_ref, -m_ref);
            uint64_t sum2[4] = {0, 0, 0, 0};
#pragma unroll
            for (int c = 0; c < kChunks; ++c) {
                uint32_t *cur = c == 0 ? s0 : (c == 1 ? s1 : (c == 2 ? s2 : s3));
                uint32_t pk[16];
                // Exact instances: the leading 8 bits of the values in cur as bf16 pairs; what is left stays in cur.  Three
                // times that is a weight's 24 bits.
                auto take_part = [&](bool last) {
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        pk[i] = __byte_perm(cur[2 * i], cur[2 * i + 1], 0x7632);
                        if (last) continue;
                        const uint64_t top = pack_f32x2(__uint_as_float(cur[2 * i] & 0xffff0000u), __uint_as_float(cur[2 * i + 1] & 0xffff0000u));
                        float r0, r1;
                        unpack_f32x2(fma_f32x2(top, pack_f32x2(-1.f, -1.f), pack_f32x2(__uint_as_float(cur[2 * i]), __uint_as_float(cur[2 * i + 1]))), r0, r1);
                        cur[2 * i] = __float_as_uint(r0);
                        cur[2 * i + 1] = __float_as_uint(r1);
                    }
                };
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    const uint64_t x2 = fma_f32x2(pack_f32x2(__uint_as_float(cur[2 * i]), __uint_as_float(cur[2 * i + 1])), sl2_2, negm2);
                    float p0, p1;
                    if (!kExact && !kPartial && ((kPolyMask >> (i & 7)) & 1)) {
                        exp2_poly_x2(x2, p0, p1);
                    } else {
                        float x0, x1;
                        unpack_f32x2(x2, x0, x1);
                        p0 = ex2(x0); p1 = ex2(x1);
                    }
                    sum2[i & 3] = add_f32x2(sum2[i & 3], pack_f32x2(p0, p1));
                    if (kExact) { cur[2 * i] = __float_as_uint(p0); cur[2 * i + 1] = __float_as_uint(p1); }
                    else pk[i] = pack_bf16(p0, p1);
                }
                // keys 32 c .. 32 c + 31 as bf16 pairs: columns 64 (c / 2) + 16 (c % 2) .., all inside S columns
                // that this thread has already read
                if (kExact) {
                    take_part(false);
                    FEDATTN_TMEM_ST16(tS + 32 * c, pk);
                    take_part(false);
                    FEDATTN_TMEM_ST16(tS + 32 * c + 16, pk);
                    take_part(true);
                    FEDATTN_TMEM_ST16(tmem_base + lane_base + kColP3 + t * 128 + 16 * c, pk);
                } else {
                    FEDATTN_TMEM_ST16(tS + 64 * (c >> 1) + 16 * (c & 1), pk);
                }
                if ((32 * c + 32) % kPartKeys == 0) {           // a half of P is complete: PV may start on it
                    tmem_wait_st();
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(p_full + kSplit * t + 32 * c / kPartKeys);       // one arrival per warp
                }
            }
            float r0, r1;
            unpack_f32x2(add_f32x2(add_f32x2(sum2[0], sum2[1]), add_f32x2(sum2[2], sum2[3])), r0, r1);
            l += r0 + r1;
            if (tid == 0) TRACE(j, t ? 6 : 1);
        };

        int pn = 0;                                             // items read from the producer's slots
        int n_met = 0;                                          // halves: items merged so far
        for (int k = 0; k < n_rounds; ++k) {
            const int item = item_of(k);
            if (item >= n_items) continue;
            Item it;
            Sub sub;
            bool listed = false;                                // the walk is a list of tiles, not a prefix
            bool halved = false;                                // the other warpgroup walks the other KV tiles of these rows
            {
                const bool ok = mbar_wait(item_full + (pn & 1), (pn >> 1) & 1, abort_flag, kp.status);
                if (!__all_sync(0xffffffffu, ok)) break;        // nothing is published any more
                const volatile int *slot = item_pub + (pn & 1) * 16;
                it.kvh = slot[0]; it.seg = slot[1]; it.kv_begin = slot[2]; it.n_a = slot[3]; it.t_b0 = slot[4];
                it.a = slot[5]; it.b = slot[6];
                sub.head = slot[8 + 4 * t]; sub.q_row0 = slot[9 + 4 * t]; sub.n_valid = slot[10 + 4 * t];
                sub.n_tiles = slot[11 + 4 * t];
                halved = kHalves && slot[11] > 0;
                it.kvp = p.kv_pos ? p.kv_pos + (p.kv_head_major ? (int64_t)it.kvh * p.total_kv : 0) : nullptr;
                __syncwarp();
                // (a listed walk is read as it goes: the slot is given back behind it)
                listed = kSpecial && !kExact && p.general && it.b < 0;
                if (lane == 0 && !listed) mbar_arrive(item_empty + (pn & 1));
                ++pn;
            }
            const int n_tiles = sub.n_tiles;
            const bool valid = r < sub.n_valid;
            __nv_bfloat16 *orow = reinterpret_cast<__nv_bfloat16 *>(p.o) + ((int64_t)(sub.q_row0 + r) * p.hq + sub.head) * d;
            float *lse_p = p.lse ? p.lse + (int64_t)(sub.q_row0 + r) * p.hq + sub.head : nullptr;
            const bool general = kSpecial && !kExact && p.general;
            if (n_tiles == 0 && listed && lane == 0) mbar_arrive(item_empty + ((pn - 1) & 1));
            if (n_tiles == 0) {                                 // nothing visible to any row of the tile, or no rows
                if (valid) {
                    for (int c = 0; c < d; c += 8) *reinterpret_cast<uint4 *>(orow + c) = make_uint4(0, 0, 0, 0);
                    if (lse_p) *lse_p = -INFINITY;
                }
                continue;
            }
            const bool two_range = kSpecial && p.sync && p.remote_only && !p.causal;      // (pairs comes first)
            const bool pairs = kExact && kp.pairs;
            int c_row = 0, n_full = 0, p_row = 0;
            PairRule mine{0, 0, false}, all{0, 0, false};       // pairs: this row's rule, and what every row of the warp sees
            int kpos[4] = {0, 0, 0, 0};                         // pairs: positions of keys 32 c + lane of the tile at hand
            auto load_pos = [&](int j) {
                const int T = (int)p.total_kv;
#pragma unroll
                for (int c = 0; c < kChunks; ++c) {
                    const int key = j * kKeys + 32 * c + lane;
                    kpos[c] = it.kvp ? ld_int(it.kvp + min(key, T - 1)) : key;
                }
            };
            if (pairs) {
                mine = pair_rule(p, it, sub, r);
                all = mine;
                all.lo = __reduce_min_sync(0xffffffffu, mine.lo);
                load_pos(kHalves ? 1 - t : 0);
            } else if (general) {
                // every (query, key) pair on its own positions
                n_full = it.b;
                const int row = sub.q_row0 + min(r, sub.n_valid - 1);
                p_row = p.q_pos ? ld_int(p.q_pos + row) : row;
            } else {
                if (p.sync && p.remote_only) {
                    c_row = it.a;                               // the same for every row of the segment
                } else if (p.sync && p.causal && it.kvp) {
                    // Sparse aggregate, row position = row index.  One cooperative search gives the keys
                    // visible to all of the warp's 32 consecutive rows; the next 32 keys are the only ones
                    // that can tell these rows apart (more only if positions repeat: then each lane searches).
                    const int T = (int)p.total_kv, p0 = sub.q_row0 + (r & ~31);
                    const int cw = count_le_warp(it.kvp, T, p0 - 1, lane);
                    const int wv = cw + lane < T ? ld_int(it.kvp + cw + lane) : INT32_MAX;
                    int cnt = 0;
#pragma unroll
                    for (int jj = 0; jj < 32; ++jj) cnt += __shfl_sync(0xffffffffu, wv, jj) <= p0 + lane;
                    c_row = cw + cnt;
                    if (__shfl_sync(0xffffffffu, wv, 31) <= p0 + 31) c_row = count_le(it.kvp, T, p0 + lane);
                } else {
                    c_row = prefix_len(p, it, sub, r, lane);   // arithmetic only
                }
                // prefix lengths do not decrease with the row, so KV tiles below the prefix of the warp's first
                // row are unmasked for the whole warp (the choice of code path only has to be warp-uniform)
                n_full = __shfl_sync(0xffffffffu, c_row, 0) / kKeys;
            }
            const int T = (int)p.total_kv;
            float m_run = 0.f, l_run = 0.f;
            for (int j = 0; j < n_tiles; ++j) {
                const int gt = gsub + j;
                int tile = kHalves ? 2 * j + 1 - t : j, entry = 0;
                if (listed) {
                    entry = reinterpret_cast<const volatile uint16_t *>(walks)[((pn - 1) & 1) * kWalkMost + tile];
                    tile = entry & 0x7fff;
                }
                // which columns of this tile the thread's row sees: everything (warp-uniform), or a mask per chunk
                bool full;
                uint32_t vm[4] = {0, 0, 0, 0};
                if (pairs) {
                    // column 32 c + i of the tile is its key 32 c + i, whose position lane i holds
                    const int k0 = tile * kKeys;
                    bool see_all = true;
#pragma unroll
                    for (int c = 0; c < kChunks; ++c) see_all = see_all && k0 + 32 * c + lane < T && all.sees(kpos[c]);
                    full = __all_sync(0xffffffffu, see_all);
                    if (!full) {
#pragma unroll
                        for (int c = 0; c < kChunks; ++c) {
                            uint32_t m = 0;
#pragma unroll 4
                            for (int i = 0; i < 32; ++i)
                                if (mine.sees(__shfl_sync(0xffffffffu, kpos[c], i))) m |= 1u << i;
                            vm[c] = m & below32(T - k0 - 32 * c);
                        }
                    }
                    if (j + 1 < n_tiles) load_pos(tile + (kHalves ? 2 : 1));        // lands during this tile's visit
                } else if (two_range) {                         // keys [0, a) and [b, T)
                    const int k0 = tile_of(it, tile) * kKeys;   // first key of the tile
                    full = k0 + kKeys <= it.a || (k0 >= it.b && k0 + kKeys <= T);
                    if (!full) {
#pragma unroll
                        for (int c = 0; c < kChunks; ++c) {
                            const int cb = k0 + 32 * c;
                            vm[c] = below32(it.a - cb) | (below32(T - cb) & ~below32(it.b - cb));
                        }
                    }
                } else {
                    full = listed ? (entry >> 15) != 0 : tile < n_full;
                    if (!full && general) {
                        // column i of chunk c is key cb + i: visible iff it exists and its position is not above
                        // the row's.  The address is the same in every lane: broadcast loads.
#pragma unroll
                        for (int c = 0; c < kChunks; ++c) {
                            const int cb = tile * kKeys + 32 * c;
                            uint32_t m = 0;
#pragma unroll 4
                            for (int i = 0; i < 32; ++i) {
                                const int key = cb + i;
                                const int kpos = it.kvp ? ld_int(it.kvp + min(key, T - 1)) : key;
                                if (key < T && kpos <= p_row) m |= 1u << i;
                            }
                            vm[c] = m;
                        }
                    } else if (!full) {
#pragma unroll
                        for (int c = 0; c < kChunks; ++c) vm[c] = below32(c_row - tile * kKeys - 32 * c);
                    }
                }
                if (full) visit(std::false_type{}, j, gt, vm, m_run, l_run);
                else visit(std::true_type{}, j, gt, vm, m_run, l_run);
            }

            if (listed) {
                __syncwarp();
                if (lane == 0) mbar_arrive(item_empty + ((pn - 1) & 1));
            }

            // The first key a row sees weighs 1 but for the rounding of its reference.  Where a unit of the reference is
            // worth more than its weight (logits beyond 2^24) the row is one for the routine below.
            if (kExact && m_run != -INFINITY && !(l_run >= 0.25f)) l_run = __int_as_float(0x7fc00000);       // NaN

            // ---- epilogue: drain this row of O from TMEM (frees it for the next item), O / l -> bf16 -> global
            mbar_wait(o_done + t, (gsub + n_tiles - 1) & 1, abort_flag, kp.status);
            tc_fence_after();
            // Halves: this thread and the one with the same row in the other warpgroup hold the two partials of the row.
            // Both read both accumulators (each half of the columns; one box: sub-tile 1's warps all of them) and
            // weigh them by w0 and w1; otherwise w = 1 / l weighs the own accumulator.
            float w0 = 0.f, w1 = 0.f;
            if (kHalves && halved) {
                // (sub-tile 0's Q buffer is not used; two slots: a warp that is an item ahead finds the other one, and it
                // gets no further before every warp has arrived there, behind its reads of this one)
                float2 *xch = reinterpret_cast<float2 *>(sQ) + (n_met & 1) * 256;
                const float m_mine = l_run == 0.f ? -INFINITY : m_run;
                xch[t * 128 + r] = make_float2(m_mine, l_run);
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(halves_met);
                mbar_wait(halves_met, n_met & 1, abort_flag, kp.status);
                tc_fence_after();
                ++n_met;
                // both warpgroups add in the same order: they hold the same row sum to the last bit
                const float2 ml0 = xch[r], ml1 = xch[128 + r];
                m_run = fmaxf(ml0.x, ml1.x);
                const float ref = m_run == -INFINITY ? 0.f : m_run, f0 = ex2(ml0.x - ref), f1 = ex2(ml1.x - ref);
                l_run = ml0.y * f0 + ml1.y * f1;
                const float inv_l = l_run > 0.f ? 1.f / l_run : 0.f;
                w0 = f0 * inv_l;
                w1 = f1 * inv_l;
            }
            const float inv = l_run > 0.f ? 1.f / l_run : 0.f;
            const int c_lo = kHalves && halved && kBoxes == 2 ? 2 * t : 0;                  // 32-column chunks of this thread
            const int c_hi = kHalves && halved ? (kBoxes == 2 ? c_lo + 2 : 2 * t) : 2 * kBoxes;
            // chunk c of the row, normalised
            auto load_o = [&](int c, uint32_t (&o)[32]) {
                if (kHalves && halved) {
                    uint32_t x[32];
                    FEDATTN_TMEM_LD32(tmem_base + lane_base + kColO + 32 * c, o);
                    FEDATTN_TMEM_LD32(tmem_base + lane_base + kColO + 128 + 32 * c, x);
                    tmem_wait_ld();
#pragma unroll
                    for (int i = 0; i < 32; ++i)
                        o[i] = __float_as_uint(fmaf(__uint_as_float(x[i]), w1, __uint_as_float(o[i]) * w0));
                } else {
                    FEDATTN_TMEM_LD32(tO + 32 * c, o);
                    tmem_wait_ld();
#pragma unroll
                    for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * inv);
                }
            };
            // this warp has read what it needs of O: one arrival per warp lets the accumulator be overwritten (halves: of
            // both, or, where the other warpgroup has no part in the item, its share too)
            auto release_o = [&]() {
                tc_fence_before();
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(o_free + t);
                    if (kHalves) mbar_arrive(o_free + (halved ? 1 - t : t));
                }
            };
            // Full warps of rows leave through shared memory and TMA stores (a warp's 32 rows x 64 columns at a
            // time); a warp with rows beyond the segment writes its valid rows directly.
            bool by_tma = kp.o_tma && (r | 31) < sub.n_valid;
            uint32_t bad = 0;                                   // exact instances: rows of the warp with a non-finite channel
            if (kExact) {
                float probe = l_run * 0.f;                      // 0 unless something is Inf or NaN
                // (halves: all columns, so that both warpgroups find the same rows)
#pragma unroll 1
                for (int c = 0; c < 2 * kBoxes && 32 * c < d; ++c) {
                    uint32_t o[32];
                    load_o(c, o);
#pragma unroll
                    for (int i = 0; i < 32; ++i)
                        if (32 * c + (i & ~7) < d) probe = fmaf(__uint_as_float(o[i]), 0.f, probe);
                }
                bad = __ballot_sync(0xffffffffu, valid && !(probe == 0.f));
                by_tma = by_tma && bad == 0;
            }
            uint8_t *my_stage = stage + (size_t)warp * kStageBytes;
            if (kHalves && by_tma) {
                // one box of 64 columns per warp at a time; short items, so the code stays short
                if (lane == 0) tma_store_wait_read();
                __syncwarp();
#pragma unroll 1
                for (int c = c_lo; c < c_hi; ++c) {
                    uint32_t o[32];
                    load_o(c, o);
                    if (c == c_hi - 1) release_o();
                    if (c == c_lo + 2) {                        // the first box's store has read the staging rows
                        if (lane == 0) tma_store_wait_read();
                        __syncwarp();
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        uint32_t w[4];
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            w[i] = pack_bf16(__uint_as_float(o[8 * u + 2 * i]), __uint_as_float(o[8 * u + 2 * i + 1]));
                        const int unit = 4 * (c & 1) + u;
                        *reinterpret_cast<uint4 *>(my_stage + lane * 128 + ((unit ^ (lane & 7)) << 4)) = make_uint4(w[0], w[1], w[2], w[3]);
                    }
                    if (c & 1) {
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                        __syncwarp();
                        if (lane == 0) tma_store_3d(&map_o, my_stage, 64 * (c >> 1), sub.head, sub.q_row0 + (r & ~31));
                    }
                }
                if (c_lo == c_hi) release_o();
            } else if (by_tma) {
                if (lane == 0) tma_store_wait_read();           // the previous item's last store has read the staging rows
                __syncwarp();
                uint32_t oa[32], ob[32];
                FEDATTN_TMEM_LD32(tO, oa);
#pragma unroll
                for (int c = 0; c < 2 * kBoxes; ++c) {
                    uint32_t *cur = (c & 1) ? ob : oa, *nxt = (c & 1) ? oa : ob;
                    tmem_wait_ld();
                    if (c < 2 * kBoxes - 1) {
                        FEDATTN_TMEM_LD32(tO + 32 * (c + 1), nxt);
                    } else {
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(o_free + t); // one arrival per warp: O_t may be overwritten
                    }
                    if (c == 2) {                               // the first half's store has read the staging rows
                        if (lane == 0) tma_store_wait_read();
                        __syncwarp();
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u) {               // 16-byte unit 4 (c & 1) + u of the row's 128 staged bytes
                        uint32_t w[4];
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            w[i] = pack_bf16(__uint_as_float(cur[8 * u + 2 * i]) * inv, __uint_as_float(cur[8 * u + 2 * i + 1]) * inv);
                        const int unit = 4 * (c & 1) + u;
                        *reinterpret_cast<uint4 *>(my_stage + lane * 128 + ((unit ^ (lane & 7)) << 4)) = make_uint4(w[0], w[1], w[2], w[3]);
                    }
                    if (c & 1) {
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                        __syncwarp();
                        if (lane == 0) tma_store_3d(&map_o, my_stage, 64 * (c >> 1), sub.head, sub.q_row0 + (r & ~31));
                    }
                }
            } else {
                // the rare path (a warp with rows beyond the segment) is kept short rather than fast
#pragma unroll 1
                for (int c = c_lo; c < c_hi; ++c) {
                    uint32_t o[32];
                    load_o(c, o);
                    if (c == c_hi - 1) release_o();
                    if (valid && !((bad >> lane) & 1u)) {
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            if (kExact && 32 * c + 8 * u >= d) break;
                            uint32_t w[4];
#pragma unroll
                            for (int i = 0; i < 4; ++i)
                                w[i] = pack_bf16(__uint_as_float(o[8 * u + 2 * i]), __uint_as_float(o[8 * u + 2 * i + 1]));
                            *reinterpret_cast<uint4 *>(orow + 32 * c + 8 * u) = make_uint4(w[0], w[1], w[2], w[3]);
                        }
                    }
                }
                if (kHalves && c_lo == c_hi) release_o();
            }
            // (halves: sub-tile 1's warpgroup, which has a part in every item, writes it)
            if (valid && lse_p && !(kHalves && halved && t == 0) && !((bad >> lane) & 1u))
                *lse_p = !(l_run > 0.f) ? -INFINITY : kExact ? lse_exact(m_run, l_run) : (m_run + log2f(l_run)) * 0.6931471805599453f;
            if (kExact && bad && !(kHalves && halved && t == 0)) {      // (one warpgroup redoes them, neither stores them)
                if (lane == 0) tma_store_wait_read();           // the staging rows are free again: the routine's row of Q
                __syncwarp();
#pragma unroll 1
                for (uint32_t left = bad; left; left &= left - 1) {
                    attn_row_warp<__nv_bfloat16>(kp.row, sub.q_row0 + (r & ~31) + __ffs(left) - 1, sub.head,
                                                 reinterpret_cast<float *>(my_stage));
                    __syncwarp();
                }
            }
            gsub += n_tiles;
        }
        if (lane == 0) tma_store_wait_read();                   // the staging rows stay alive until they are read
    }

    // ---- teardown -----------------------------------------------------------------------------------
    tc_fence_before();
    __syncthreads();
    if (warp == kProducerWarp) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols) : "memory");
    }
}

// ---- position tables of a general-position call -------------------------------------------------------
// grid: one block per KV position array (n_arrays of them), then one block for the query positions.
// A warp reduces one 128-entry tile at a time.
constexpr int kTabThreads = 1024;

__device__ __forceinline__ void tile_min_max(const int32_t *pos, int64_t n, int64_t tile, int lane, int &mn, int &mx)
{
    mn = INT32_MAX; mx = INT32_MIN;
    const int64_t i0 = tile * kTileN + lane * 4;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int64_t i = i0 + e;
        if (i < n) {
            const int v = pos ? ld_int(pos + i) : (int)i;
            mn = min(mn, v); mx = max(mx, v);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        mn = min(mn, __shfl_xor_sync(0xffffffffu, mn, o));
        mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
}

__global__ void __launch_bounds__(kTabThreads)
position_tables_kernel(const int32_t *q_pos, int64_t n_q, const int32_t *kv_pos, int64_t total_kv, int n_arrays,
                       int n_qtiles, int n_kt, int32_t *tab)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, n_warps = kTabThreads / 32;
    const PosTables pt = pos_tables(tab, n_qtiles, n_arrays, n_kt);
    if ((int)blockIdx.x == n_arrays) {
        int32_t *q_min = tab, *q_max = tab + n_qtiles;
        for (int64_t t = warp; t < n_qtiles; t += n_warps) {
            int mn, mx;
            tile_min_max(q_pos, n_q, t, lane, mn, mx);
            if (lane == 0) { q_min[t] = mn; q_max[t] = mx; }
        }
        return;
    }
    const int a = blockIdx.x;
    const int32_t *pos = kv_pos ? kv_pos + (size_t)a * total_kv : nullptr;
    int32_t *kv_min = const_cast<int32_t *>(pt.kv_min) + (size_t)a * n_kt, *kv_max = const_cast<int32_t *>(pt.kv_max) + (size_t)a * n_kt;
    for (int64_t t = warp; t < n_kt; t += n_warps) {
        int mn, mx;
        tile_min_max(pos, total_kv, t, lane, mn, mx);
        if ((t + 1) * kTileN > total_kv) mx = INT32_MAX;      // ragged tile: never fully visible
        if (lane == 0) { kv_min[t] = mn; kv_max[t] = mx; }
    }
}

// ---- self-test of the bounded wait ---------------------------------------------------------------------
// Waits with mbar_wait, the routine every role above waits with, on a barrier that nothing signals.
__global__ void wait_selftest_kernel(int32_t *status, uint32_t max_polls)
{
    __shared__ uint64_t bar;
    __shared__ int abort_flag;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    mbar_wait(&bar, 0, &abort_flag, status, max_polls);        // phase 0 never completes: runs out, flags the status
}

// ---- host ---------------------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

#ifdef FEDATTN_TRACE
extern "C" int fedattn_debug_read_trace(long long *host, int n)
{
    return (int)cudaMemcpyFromSymbol(host, g_trace, sizeof(long long) * n);
}
#endif

bool prefill_sm100_supported(const Context *ctx) { return ctx->encode_tiled != nullptr; }

// The range of fast_div: calls outside it run on the SIMT kernel where that served them before (head_dim < 128).
bool prefill_sm100_takes(const Context *ctx, const PrefillParams &p)
{
    if (!prefill_sm100_supported(ctx)) return false;
    if (p.d == 128) return true;
    const int64_t per_tile = (int64_t)p.hkv * ((p.hq / p.hkv + 1) / 2);
    const int64_t n_qtiles = p.n_q_rows / kTileM + p.n_seg;          // at most
    return per_tile <= 4096 && n_qtiles * per_tile < (1LL << 28) && p.n_q_rows < 0x7fffff00LL && p.total_kv < 0x7fffff00LL;
}

// [rows, heads, d] bf16 (token-major) or [heads, rows, d] (head-major); boxes of 64 columns x 128 rows.  Columns
// beyond d read as zero and are not written.
static bool encode_map(const Context *ctx, CUtensorMap *map, const void *base, int64_t rows, int heads, int d, bool head_major,
                       int box_rows = kTileN)
{
    EncodeTiledFn fn = reinterpret_cast<EncodeTiledFn>(ctx->encode_tiled);
    cuuint64_t dims[3], strides[2];
    cuuint32_t box[3], estr[3] = {1, 1, 1};
    dims[0] = (cuuint64_t)d;
    if (head_major) {
        dims[1] = (cuuint64_t)rows; dims[2] = (cuuint64_t)heads;
        strides[0] = (cuuint64_t)d * 2; strides[1] = (cuuint64_t)rows * d * 2;
        box[0] = kBoxCols; box[1] = (cuuint32_t)box_rows; box[2] = 1;
    } else {
        dims[1] = (cuuint64_t)heads; dims[2] = (cuuint64_t)rows;
        strides[0] = (cuuint64_t)d * 2; strides[1] = (cuuint64_t)heads * d * 2;
        box[0] = kBoxCols; box[1] = 1; box[2] = (cuuint32_t)box_rows;
    }
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

size_t position_table_bytes(int hkv, int64_t n_q_rows, int64_t total_kv)
{
    const int64_t n_qt = (n_q_rows + kTileM - 1) / kTileM, n_kt = (total_kv + kTileN - 1) / kTileN;
    return (size_t)(2 * n_qt + 2 * (int64_t)hkv * n_kt) * sizeof(int32_t);
}

cudaError_t launch_wait_selftest(Context *ctx, int max_polls, cudaStream_t s)
{
    wait_selftest_kernel<<<1, 32, 0, s>>>(ctx->status, (uint32_t)max_polls);
    ++ctx->launches;
    return cudaGetLastError();
}

// How the query heads of a group and the query tiles form work items.
enum ItemForm {
    kPairs,       // two heads of a query tile; an odd group's last head stays alone
    kStraddle,    // odd groups: the last head of two neighbouring query tiles forms an item too
    kHalvesForm,  // one head, its KV tiles shared by the two sub-tiles (kernel instances kHalves)
};
// The form that is estimated to end first.  Unit: a lone sub-tile's time per KV tile, 1.6 us; a pair takes 1.14 times as
// long (8 / 8 heads, 17 query tiles: lone 32.7 us, pairs 37.4), halves 0.6 per KV tile of their head, and every item costs
// about 2 on top (its Q, its epilogue, the restart of the chain; halves 2.6, they merge).  With exact weights, and an item
// per CTA, the unit is 3.2 us per 128 keys, a pair takes 1.05, halves 0.65 and an item 1 on top (halves 1.4): 4 / 4 heads
// of 64, two segments of 500 rows: 16.6 -> 14.5 and 31.1 -> 24.7 us (halves for pairs).  Several items per CTA gain less,
// halves 0.9: 16 / 4 heads of 64, six segments of 2160 rows, sync 55.5 -> 51.5 us in a loop, but a round that runs its local
// call as pairs fetches the other instance's code for it, and takes 85.3 us with pairs and 87.4 with halves.
// Calls of a few items per CTA are dealt out on paper as the kernel deals them; for more items the mean load of a CTA
// decides, and halves never pay (twice the items and twice the K and V traffic).  Measured against the estimate's second
// choice, us: 16 / 4 heads, 700 + 500 rows: local 18.4 -> 13.9, sync 25.8 -> 18.5 (halves for pairs); 32 / 8 heads there:
// 18.9 and 26.3 with pairs, 22.6 and 30.8 with halves; 14 / 2 heads, 2160 rows, sync: 37.9 -> 29.1 (halves for straddling
// pairs); 24 / 8 heads, 1000 + 2000 + 3000 rows: local 120 -> 100, sync 241 -> 198 (straddling pairs for lone last heads).
static ItemForm item_form(const PrefillParams &p, int64_t n_qtiles, int sm_count)
{
    constexpr int kMostSms = 256;
    const int g = p.hq / p.hkv;
    if ((int64_t)p.hkv * g > 4096 || n_qtiles * p.hkv * g >= (1LL << 28) || sm_count > kMostSms) return kPairs;      // fast_div range
    const bool alone = n_qtiles * p.hq <= sm_count;             // an item per CTA in every form
    const bool narrow = p.d < 128 && alone;
    const float pair = narrow ? 1.05f : 1.14f, half = narrow ? 0.65f : (p.d < 128 ? 0.9f : 0.6f);
    const float start = narrow ? 1.0f : 2.0f, merge = narrow ? 0.4f : 0.6f, n_kt = (float)((p.total_kv + kTileN - 1) / kTileN);
    const bool grows = p.causal && !p.remote_only && !(p.sync && p.q_pos);
    // KV tiles of query tile `tile` (1 ..) of a segment with `tiles` of them
    auto walk = [&](int seg, int tile, int tiles) -> float {
        if (p.remote_only) return p.causal ? n_kt * p.cu[seg] / p.n_q_rows : n_kt;
        const float most = p.sync ? n_kt : (float)tiles;
        return grows ? most * tile / tiles : most;
    };
    auto tiles_of = [&](int seg) { return (p.cu[seg + 1] - p.cu[seg] + kTileM - 1) / kTileM; };
    if (n_qtiles * p.hkv * ((g + 1) / 2) > 3 * sm_count) {
        // Many items: straddling pairs save 0.43 of a unit per two lone KV tiles and hardly change the end.
        return (g & 1) ? kStraddle : kPairs;
    }
    float load[kMostSms];
    int longest = 0;
    for (int n = 0; n < p.n_seg; ++n) longest = tiles_of(n) > longest ? tiles_of(n) : longest;
    if (alone) {                                                // the longest item decides
        float w = 0.f;
        for (int n = 0; n < p.n_seg; ++n)
            if (tiles_of(n) > 0) w = walk(n, tiles_of(n), tiles_of(n)) > w ? walk(n, tiles_of(n), tiles_of(n)) : w;
        return w > 1.f && half * w + merge + start < 0.95f * ((g > 1 ? pair : 1.f) * w + start) ? kHalvesForm : kPairs;
    }
    auto ends = [&](ItemForm form) -> float {
        const int rows = form == kStraddle ? 2 : 1;             // query tiles per ranked tile
        for (int c = 0; c < sm_count; ++c) load[c] = 0.f;
        int c = 0, step = 1;
        auto deal = [&](float cost) {
            load[c] += cost;
            c += step;
            if (c == sm_count || c < 0) { step = -step; c += step; }
        };
        for (int level = (longest + rows - 1) / rows; level >= 1; --level)
            for (int n = 0; n < p.n_seg; ++n) {
                const int tiles = tiles_of(n), first = rows * (level - 1) + 1;
                if (tiles < first) continue;
                const float w = walk(n, first, tiles), w2 = rows == 2 && first < tiles ? walk(n, first + 1, tiles) : 0.f;
                for (int h = 0; h < p.hkv; ++h) {
                    if (form == kHalvesForm) {
                        for (int u = 0; u < g; ++u) deal((w > 1.f ? half * w + merge : w) + start);
                    } else {
                        for (int u = 0; u < g / 2; ++u) deal(pair * w + start);
                        if (rows == 2)
                            for (int u = 0; u < g / 2; ++u) deal(w2 > 0.f ? pair * w2 + start : 0.f);
                        if (g & 1) deal((w2 > 0.f ? pair * (w2 > w ? w2 : w) : w) + start);
                    }
                }
            }
        float most = 0.f;
        for (int i = 0; i < sm_count; ++i) most = load[i] > most ? load[i] : most;
        return most;
    };
    ItemForm best = kPairs;
    float t = ends(kPairs);
    if (g & 1) {
        const float u = ends(kStraddle);
        if (u < 0.97f * t) { t = u; best = kStraddle; }
    }
    if (n_qtiles * p.hq <= 3 * sm_count && ends(kHalvesForm) < 0.95f * t) best = kHalvesForm;
    return best;
}

cudaError_t launch_prefill_sm100(Context *ctx, const PrefillParams &p, cudaStream_t s)
{
    static_assert(sizeof(KernelParams) + 4 * sizeof(CUtensorMap) <= 4096, "kernel parameter block too large");
    KernelParams kp;
    kp.p = p;
    kp.status = ctx->status;
    kp.pairs = 0;
    if (p.d < 128) {
        // positions in any order, as the row routine takes them, and no tables: those calls keep off the scratch
        kp.pairs = p.sync && (p.kv_pos || p.q_pos) && (p.causal || p.remote_only);
        kp.row = generic_params(p);
        // The tensor core cuts off what a sum has below its last place, after each step of 16 channels: a logit comes out
        // smaller by kCutOff of itself for the last step and proportionally less for the ones before.  (lse of N(0, 1)
        // inputs, error against fp64, mean and rms in 1e-7: head_dim 64 -1.0 and 1.9 without the factor, -0.3 and 1.6
        // with it; 96: -1.5 and 2.3, -0.5 and 1.8; 120: -1.8 and 2.5, 0.3 and 1.6; fp32 FMA chains: rms 1.8.)
        constexpr double kCutOff = 3e-8;
        const int steps = (p.d + 15) / 16;
        kp.sl2 = (float)((double)p.scale * 1.4426950408889634 * (1.0 + kCutOff * (steps + 1) / 2));
    }
    kp.n_kt = (int32_t)((p.total_kv + kTileN - 1) / kTileN);
    const int g = p.hq / p.hkv;
    int64_t n_qtiles = 0, n_ranked = 0;
    for (int n = 0; n < p.n_seg; ++n) n_qtiles += (p.cu[n + 1] - p.cu[n] + kTileM - 1) / kTileM;
    if (n_qtiles > 0x7fffffffLL) return cudaErrorInvalidValue;
    kp.n_qtiles = (int32_t)n_qtiles;
    const ItemForm item = item_form(p, n_qtiles, ctx->sm_count);
    const bool halves = item == kHalvesForm;
    kp.straddle = item == kStraddle ? 1 : 0;
    const int rank_rows = kp.straddle ? 2 * kTileM : kTileM, ppk = halves || kp.straddle ? g : (g + 1) / 2;
    for (int n = 0; n < p.n_seg; ++n) {
        kp.ord_seg[n] = n;
        kp.ord_nt[n] = (p.cu[n + 1] - p.cu[n] + rank_rows - 1) / rank_rows;
        n_ranked += kp.ord_nt[n];
    }
    for (int a = 1; a < p.n_seg; ++a)          // insertion sort by tile count, descending (stable)
        for (int b = a; b > 0 && kp.ord_nt[b] > kp.ord_nt[b - 1]; --b) {
            const int32_t tn = kp.ord_nt[b], ts = kp.ord_seg[b];
            kp.ord_nt[b] = kp.ord_nt[b - 1]; kp.ord_seg[b] = kp.ord_seg[b - 1];
            kp.ord_nt[b - 1] = tn; kp.ord_seg[b - 1] = ts;
        }
    kp.band_rank[0] = 0;
    for (int b = 0; b < p.n_seg; ++b) {
        const int64_t next = b + 1 < p.n_seg ? kp.ord_nt[b + 1] : 0;
        kp.band_rank[b + 1] = kp.band_rank[b] + (int32_t)((kp.ord_nt[b] - next) * (b + 1));
    }
    const int64_t items = n_ranked * p.hkv * ppk;
    if (items == 0) return cudaSuccess;
    if (items >= (1LL << 28) || (int64_t)p.hkv * ppk > 4096) return cudaErrorInvalidValue;   // fast_div range
    kp.n_items = (int32_t)items;
    auto magic = [](int64_t d) { return (uint64_t)(((1ULL << 40) + (uint64_t)d - 1) / (uint64_t)d); };
    kp.group = g;
    kp.magic_per_tile = magic((int64_t)p.hkv * ppk);
    kp.magic_ppk = magic(ppk);
    for (int i = 0; i < kMaxP; ++i) kp.magic_small[i] = magic(i + 1);
    const int64_t blocks = items < ctx->sm_count ? items : ctx->sm_count;     // persistent: one CTA per SM
    const int boxes = p.d <= kBoxCols ? 1 : 2;
    CUtensorMap mq, mk, mv, mo;
    if (!encode_map(ctx, &mq, p.q, p.n_q_rows, p.hq, p.d, false) ||
        !encode_map(ctx, &mk, p.k, p.total_kv, p.hkv, p.d, p.kv_head_major != 0, tile_keys(p.d < 128, boxes)) ||
        !encode_map(ctx, &mv, p.v, p.total_kv, p.hkv, p.d, p.kv_head_major != 0, tile_keys(p.d < 128, boxes)))
        return cudaErrorInvalidValue;
    // the output as [rows, heads, head_dim] in boxes of 32 rows x 64 columns; a base the encoder refuses (alignment)
    // leaves the kernel on its direct stores
    kp.o_tma = encode_map(ctx, &mo, p.o, p.n_q_rows, p.hq, p.d, false, 32) ? 1 : 0;
    if (!kp.o_tma) mo = mq;
    // the plain instance serves local attention and sync attention under the prefix mask; explicit positions
    // and bidirectional remote-only attention run the instance that carries their extra state; head dims below
    // 128 run the exact instances
    typedef void (*Kernel)(const CUtensorMap, const CUtensorMap, const CUtensorMap, const CUtensorMap, const KernelParams);
    static const Kernel kernels[8] = {
        prefill_sm100_kernel<false, 2, false, false>, prefill_sm100_kernel<true, 2, false, false>,
        prefill_sm100_kernel<true, 1, true, false>,   prefill_sm100_kernel<true, 2, true, false>,
        prefill_sm100_kernel<false, 2, false, true>,  prefill_sm100_kernel<true, 2, false, true>,
        prefill_sm100_kernel<true, 1, true, true>,    prefill_sm100_kernel<true, 2, true, true>};
    const int form = p.d < 128 ? 1 + boxes : (p.general || (p.remote_only && !p.causal)) ? 1 : 0;
    const int which = form + (halves ? 4 : 0);
    const uint32_t smem = smem_bytes(boxes);
    static bool attr_set[64][8] = {};
    if (!attr_set[ctx->device & 63][which]) {
        cudaError_t e = cudaFuncSetAttribute(kernels[which], cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        // the register split inside the kernel has to fit into what the launch allocates: an increase that
        // the CTA's pool cannot serve would wait for ever, so such a build is refused here
        cudaFuncAttributes fa;
        if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, kernels[which]);
        if (e == cudaSuccess && 3 * fa.numRegs < 2 * kSoftmaxRegs + kOtherRegs) e = cudaErrorLaunchOutOfResources;
        if (e != cudaSuccess) {
            if (getenv("FEDATTN_DEBUG")) fprintf(stderr, "prefill_sm100_kernel attribute: %s\n", cudaGetErrorString(e));
            return e;
        }
        attr_set[ctx->device & 63][which] = true;
    }
    if (p.general) {
        // the per-tile position tables first (same stream): the walk and the unmasked fast path read them
        const int n_arrays = p.kv_head_major ? p.hkv : 1;
        position_tables_kernel<<<n_arrays + 1, kTabThreads, 0, s>>>(p.q_pos, p.n_q_rows, p.kv_pos, p.total_kv, n_arrays,
                                                                    kp.n_qtiles, kp.n_kt, p.tab);
        ++ctx->launches;
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    // Set up while the preceding grid ends, but behind a kernel that releases its dependents early launched as usual: there
    // the CTAs would take whatever SMs that grid leaves one by one (sparse sync behind its selection 569 us, 577 set up
    // early; bidirectional local + remote behind theirs 115.5, 117.0).  Elsewhere the early set-up gains where calls are short
    // (ragged round with 64 channels 84.3 -> 80.2) and costs nothing where they are long.  (The barriers and the TMEM set up
    // before the wait: 79.5, local of 4 x 2048 152.5 -> 155.7, dense sync 518.5 -> 533.7.)  In front of a call with explicit
    // query positions stands the kernel of its tables.
    WaitFirstLaunch l(dim3((unsigned)blocks), dim3(kThreads), smem, s);
    if (!p.general && front_releases(ctx->device, s)) l.cfg.numAttrs = 0;
    cudaError_t e = cudaLaunchKernelEx(&l.cfg, kernels[which], mq, mk, mv, mo, kp);
    ++ctx->launches;
    ++ctx->tc_launches;
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e == cudaSuccess) front_note(ctx->device, s, false);
    if (e != cudaSuccess && getenv("FEDATTN_DEBUG")) fprintf(stderr, "prefill_sm100_kernel launch: %s\n", cudaGetErrorString(e));
    return e;
}

}  // namespace fedattn
