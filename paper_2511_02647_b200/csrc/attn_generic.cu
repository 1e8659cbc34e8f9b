// Tiled fp32 attention on the FMA pipes: fp32 or bf16 storage, fp32 arithmetic, head_dim <= 128.  Serves fp32
// storage (the tensor cores have no fp32 kind and TF32 would miss the fp32 error bound), decode at the head dims
// and types the tensor-core decode does not cover, and calls over an empty aggregate.
//
// The query rows that share a KV head are stacked (g grouped heads of a token are neighbours), so that a K/V tile
// is read once for all of them.  A CTA owns M stacked rows and walks tiles of 64 or 128 keys; a cluster of up to 8
// CTAs shares the tiles of one row tile when the row tiles alone leave SMs idle.  Both products work on packed
// pairs (fma.rn.f32x2): S pairs neighbouring channels, so both operands come as they lie in shared memory; O pairs
// neighbouring rows, whose weights lie side by side in the transposed P tile, and duplicates the value instead.
//
// Two warp arrangements.  kKeyWarps = 1: 4 warps, a warp owns 2 kR rows and all 64 keys of a tile.  kKeyWarps = 4, 8:
// every warp owns all M = 2 kR rows and 16 of a tile's 64 or 128 keys, with softmax state of its own: K and V are then
// read once per tile from shared memory instead of once per warp, which is what bounds a tile with few rows.
//
// Bound by the latency of LDS and FMA chains rather than by the FMA pipes: 52 % of their rate on 2048 causal rows of
// 16 heads of 64 channels (280 us), a few us per call on the smallest (two segments of
// 128 rows, 4 heads: one warp per row 60 and 111 us, tiles 7 and 11 us; decode of 8 x 512 fp32 keys, 32 / 8 heads: 11 us).
//
// Every partial (one per warp or CTA) is merged through (distributed) shared memory at the end.  Rows that come
// out non-finite are redone by the row routine, which does not touch excluded keys.
#include <cooperative_groups.h>
#include <limits.h>
#include <string.h>

#include "attn_row.cuh"

namespace fedattn {

namespace {

constexpr int kMaxCluster = 8;           // portable cluster size
constexpr int kMaxStages = 3;            // K/V tile pairs of the ring

struct TiledPlan {
    int32_t n_tiles;                     // row tiles over all segments
    int32_t splits;                      // CTAs of the cluster that shares a row tile
    int32_t stages;                      // K/V tile pairs in flight per CTA
    int32_t n_seg;
    int32_t tile0[kMaxP + 1];            // first row tile of a segment
    int32_t row0[kMaxP + 1];             // first query row (token, participant) of a segment
};

__device__ __forceinline__ uint64_t pack2(float lo, float hi)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ float2 unpack2(uint64_t v)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b)
{
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// four consecutive channels from shared memory
__device__ __forceinline__ float4 lds4(const float *p) { return *reinterpret_cast<const float4 *>(p); }
__device__ __forceinline__ float4 lds4(const __nv_bfloat16 *p)
{
    const uint2 w = *reinterpret_cast<const uint2 *>(p);
    return make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xffff0000u), __uint_as_float(w.y << 16),
                       __uint_as_float(w.y & 0xffff0000u));
}
__device__ __forceinline__ void stg4(float *p, float4 v) { *reinterpret_cast<float4 *>(p) = v; }
__device__ __forceinline__ void stg4(__nv_bfloat16 *p, float4 v)
{
    const __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y), hi = __floats2bfloat162_rn(v.z, v.w);
    *reinterpret_cast<uint2 *>(p) = make_uint2(*reinterpret_cast<const uint32_t *>(&lo), *reinterpret_cast<const uint32_t *>(&hi));
}

// Shared memory, in floats unless said otherwise.  Row pitches are padded by 16 bytes: 16 lanes that read the same
// 16-byte column of 16 consecutive rows then meet every bank group twice, which is the least a 256-byte read takes.
template <typename T, int kR, int kDP, int kKeyWarps> struct Layout {
    static constexpr int kM = kKeyWarps > 1 ? 2 * kR : 8 * kR;               // stacked rows of a CTA
    static constexpr int kThreads = kKeyWarps > 1 ? 32 * kKeyWarps : 128;
    static constexpr int kKeys = kKeyWarps > 1 ? 16 * kKeyWarps : 64;        // keys per tile
    static constexpr int kQPitch = kDP + 4;
    static constexpr int kPPitch = kM + 4;
    static constexpr int kKvPitch = kDP + 16 / (int)sizeof(T);               // elements
    static constexpr int kKvBytes = kKeys * kKvPitch * (int)sizeof(T);       // K or V tile
    static constexpr int kQBytes = kM * kQPitch * 4, kPBytes = kKeys * kPPitch * 4;
    static constexpr int kOffP = kQBytes, kOffKv = kOffP + kPBytes;
    static constexpr int bytes(int stages) { return kOffKv + stages * 2 * kKvBytes; }
    static_assert(kKeyWarps * kM * kQPitch * 4 <= 2 * kKvBytes, "the partials take the place of the K and V tiles");
};

template <typename T, int kR, int kDP, int kKeyWarps>
__global__ void __launch_bounds__(Layout<T, kR, kDP, kKeyWarps>::kThreads)
attn_tiled_kernel(const __grid_constant__ GenericParams p, const __grid_constant__ TiledPlan plan)
{
    using L = Layout<T, kR, kDP, kKeyWarps>;
    constexpr int kM = L::kM, kThreads = L::kThreads, kKeys = L::kKeys;
    constexpr int kJ = kKeyWarps > 1 ? 1 : 4;                                // keys of a tile per thread
    constexpr int kC = kDP / 16;                                             // output columns per thread: 4 tk + 64 cc + 0..3
    // Keys, rows and positions are ints up to 2^31 - 1: no sum below passes the last key.
    extern __shared__ __align__(16) uint8_t smem[];
    float *sQ = reinterpret_cast<float *>(smem), *sP = reinterpret_cast<float *>(smem + L::kOffP);
    T *sKV = reinterpret_cast<T *>(smem + L::kOffKv);                        // [stage][K, V]
    float *part = reinterpret_cast<float *>(smem + L::kOffKv);               // [warp group][row][kQPitch], after the walk
    __shared__ float2 s_ml[kKeyWarps][kM];
    __shared__ int s_bad[kM], s_last, s_lo[kM];
    __shared__ int64_t s_out[kM];                                            // stacked row -> row * hq + head

    namespace cg = cooperative_groups;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, tk = lane & 15, half = lane >> 4;
    const int rank = (int)(blockIdx.x % (unsigned)plan.splits);
    const unsigned unit = blockIdx.x / (unsigned)plan.splits;
    const int kvh = (int)(unit % (unsigned)p.hkv);
    const int tile = plan.n_tiles - 1 - (int)(unit / (unsigned)p.hkv);       // late, heavy tiles of a causal call first
    int seg = 0;
    while (seg + 1 < plan.n_seg && tile >= plan.tile0[seg + 1]) ++seg;
    const int g = p.hq / p.hkv, d = p.d;
    const int64_t stacked0 = (int64_t)(tile - plan.tile0[seg]) * kM;         // first stacked row, within the segment
    const int64_t stacked_n = (int64_t)(plan.row0[seg + 1] - plan.row0[seg]) * g;
    const int n_rows = (int)min((int64_t)kM, stacked_n - stacked0);
    const int token0 = (int)(stacked0 / g), sub0 = (int)(stacked0 - (int64_t)token0 * g);
    auto token_of = [&](int r) -> int { return token0 + (int)((unsigned)(sub0 + r) / (unsigned)g); };   // within the segment

    // Visibility: key x of [kv_lo, kv_hi) is seen by a row iff pos(x) <= lo of the row, or, two_sided, pos(x) >= hi.
    const bool decode = p.mode == kDecodeLocal || p.mode == kDecodeSync;
    const bool by_pos = p.mode == kSync && (p.causal || p.remote_only);
    const bool two_sided = by_pos && p.remote_only && !p.causal;
    const int hi = two_sided ? p.cu[seg + 1] : 0;
    int kv_lo = 0, kv_hi;
    grid_wait();                                                             // nothing is read or written before
    if (p.mode == kLocal) {
        kv_lo = p.cu[seg];
        kv_hi = p.causal ? kv_lo + token_of(n_rows - 1) + 1 : p.cu[seg + 1];
    } else if (decode) {
        kv_hi = p.kv_len[p.mode == kDecodeLocal ? seg : 0];
    } else {
        kv_hi = (int)p.total_kv;
    }
    const int64_t kv_base = (int64_t)kvh * p.kv_head_stride + (p.mode == kDecodeLocal ? (int64_t)seg * p.cache_stride : 0);
    const T *K = reinterpret_cast<const T *>(p.k) + kv_base, *V = reinterpret_cast<const T *>(p.v) + kv_base;
    const int32_t *kvp = p.kv_pos ? p.kv_pos + (int64_t)kvh * p.kv_pos_head_stride : nullptr;

    // A tile copy: thread = one 16-byte column of every kStep-th row.  Rolled: the kernel's code is fetched cold by
    // most calls, and a straight line of copies costs more than the loop.
    constexpr int kVec = 16 / (int)sizeof(T), kRowVecs = kDP / kVec, kStep = kThreads / kRowVecs;
    const int ld_r = tid / kRowVecs, ld_c = (tid % kRowVecs) * kVec;
    auto load_tile = [&](T *dst, const T *src, int t) {
        const int left = kv_hi - kv_lo - t * kKeys - ld_r;                   // this thread's rows: ld_r + kStep i, while below `left`
        if (ld_c < d) {                                                      // head_dim is a multiple of 8
            const T *from = src + ((int64_t)kv_lo + (int64_t)t * kKeys + ld_r) * p.kv_tok_stride + ld_c;
            uint32_t to = (uint32_t)__cvta_generic_to_shared(dst + ld_r * L::kKvPitch + ld_c);
            const int64_t step = (int64_t)kStep * p.kv_tok_stride;
#pragma unroll 4
            for (int i = 0; i < kKeys / kStep; ++i, from += step, to += kStep * L::kKvPitch * (int)sizeof(T)) {
                const bool ok = i * kStep < left;                            // rows past the end read as zero
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(to), "l"(ok ? from : src), "r"(ok ? 16 : 0) : "memory");
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    // the first K and V tile are on their way while Q and the rows' bounds are set up (a walk that turns out shorter
    // does not use them)
    const int n_kt_most = kv_hi > kv_lo ? (kv_hi - kv_lo - 1) / kKeys + 1 : 0;
    constexpr int kKvElts = L::kKvBytes / (int)sizeof(T);
    const int stages = plan.stages;
#pragma unroll 1
    for (int x = 0; x < 2 * stages; ++x) {
        const int t = rank + (x >> 1) * plan.splits;
        if (t < n_kt_most) load_tile(sKV + x * kKvElts, (x & 1) ? V : K, t);
        else asm volatile("cp.async.commit_group;" ::: "memory");
    }

    // every row's place and lo, then Q as fp32
    for (int r = tid; r < kM; r += kThreads) {
        const int tok = token_of(r), row = plan.row0[seg] + tok;
        s_out[r] = (int64_t)row * p.hq + kvh * g + (sub0 + r - (tok - token0) * g);
        int lo = INT_MAX;
        if (r >= n_rows) lo = INT_MIN;                                       // no such row
        else if (p.mode == kLocal && p.causal) lo = row;
        else if (by_pos) lo = p.remote_only ? p.cu[seg] - 1 : (p.q_pos ? ld_int(p.q_pos + row) : row);
        s_lo[r] = lo;
        s_bad[r] = 0;
    }
    if (tid == 0) s_last = -1;
    __syncthreads();
#pragma unroll 1
    for (int i = tid; i < kM * (kDP / 4); i += kThreads) {
        const int r = i / (kDP / 4), c = (i % (kDP / 4)) * 4;
        if (c >= d) continue;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (r < n_rows) v = lds4(reinterpret_cast<const T *>(p.q) + s_out[r] * d + c);
        *reinterpret_cast<float4 *>(sQ + r * L::kQPitch + c) = v;
    }
    int lo[kR], lo_max = INT_MIN, lo_min = INT_MAX;
    const int my_row0 = ((kKeyWarps > 1 ? 0 : 2 * warp) + half) * kR;
#pragma unroll
    for (int i = 0; i < kR; ++i) lo[i] = s_lo[my_row0 + i];
    for (int r = lane; r < n_rows; r += 32) { lo_max = max(lo_max, s_lo[r]); lo_min = min(lo_min, s_lo[r]); }
    lo_max = __reduce_max_sync(0xffffffffu, lo_max);
    lo_min = __reduce_min_sync(0xffffffffu, lo_min);
    if (by_pos) {
        // the walk ends behind the last key that some row sees: positions backwards, 1024 at a time
        if (!kvp && !two_sided) kv_hi = min(kv_hi, lo_max < 0 ? 0 : (lo_max == INT_MAX ? INT_MAX : lo_max + 1));
        else if (kvp && n_kt_most > 2 * plan.splits) {                       // (a shorter walk is not worth the search)
#pragma unroll 1
            for (int base = kv_hi > 0 ? ((kv_hi - 1) / 1024) * 1024 : -1; base >= 0; base -= 1024) {
                int last = -1;
#pragma unroll
                for (int i = 0; i < 1024 / kThreads; ++i) {
                    if (i * kThreads + tid < kv_hi - base) {
                        const int key = base + i * kThreads + tid;
                        const int pos = ld_int(kvp + key);
                        if (pos <= lo_max || (two_sided && pos >= hi)) last = key;
                    }
                }
                if (__syncthreads_or(last >= 0)) {
                    last = __reduce_max_sync(0xffffffffu, last);
                    if (lane == 0) atomicMax(&s_last, last);
                    break;
                }
            }
            __syncthreads();
            kv_hi = s_last + 1;
        }
    }

    const int n_kt = kv_hi > kv_lo ? (kv_hi - kv_lo - 1) / kKeys + 1 : 0;
    float m[kR], l[kR];
    uint64_t acc[kR / 2][kC];                                                // rows (2 i, 2 i + 1)
#pragma unroll
    for (int i = 0; i < kR; ++i) { m[i] = -INFINITY; l[i] = 0.f; }
#pragma unroll
    for (int i = 0; i < kR / 2; ++i)
#pragma unroll
        for (int c = 0; c < kC; ++c) acc[i][c] = 0;

    const int key_l = kKeyWarps > 1 ? 16 * warp + tk : tk;                  // this thread's keys of a tile: key_l + 16 j
    // the copies of the tiles behind the one needed may still be in flight: 2 stages - 1 groups
    auto wait_copy = [&]() {
        if (stages == 1) asm volatile("cp.async.wait_group 1;" ::: "memory");
        else if (stages == 2) asm volatile("cp.async.wait_group 3;" ::: "memory");
        else asm volatile("cp.async.wait_group 5;" ::: "memory");
        __syncthreads();
    };
    int pos[kJ], slot = 0;
    auto load_pos = [&](int t) {
#pragma unroll
        for (int j = 0; j < kJ; ++j) {
            const int key = min(key_l + 16 * j, kv_hi - 1 - kv_lo - t * kKeys) + kv_lo + t * kKeys;     // (past the end: the last one)
            pos[j] = kvp && by_pos ? ld_int(kvp + key) : key;
        }
    };
    if (rank < n_kt) load_pos(rank);
#pragma unroll 1
    for (int t = rank; t < n_kt; t += plan.splits) {
        const int k0 = kv_lo + t * kKeys, left = kv_hi - k0;                 // keys from the tile's first to the last
        const int next = t + stages * plan.splits;                           // the tile that takes this one's place
        T *sK = sKV + 2 * slot * kKvElts, *sV = sK + kKvElts;
        slot = slot + 1 == stages ? 0 : slot + 1;
        wait_copy();                                                         // K
        // ---- S = Q K^T: even and odd channels in the two halves of a pair ----
        uint64_t s2[kR][kJ];
#pragma unroll
        for (int i = 0; i < kR; ++i)
#pragma unroll
            for (int j = 0; j < kJ; ++j) s2[i][j] = 0;
        const float *q0 = sQ + my_row0 * L::kQPitch;
        const T *k_s = sK + key_l * L::kKvPitch;
#pragma unroll (kKeyWarps > 1 ? 4 : 2)
        for (int c = 0; c < d; c += 4) {
            uint64_t kk[kJ][2];
#pragma unroll
            for (int j = 0; j < kJ; ++j) {
                const float4 v = lds4(k_s + 16 * j * L::kKvPitch + c);
                kk[j][0] = pack2(v.x, v.y); kk[j][1] = pack2(v.z, v.w);
            }
#pragma unroll
            for (int i = 0; i < kR; ++i) {
                const float4 v = lds4(q0 + i * L::kQPitch + c);
                const uint64_t qa = pack2(v.x, v.y), qb = pack2(v.z, v.w);
#pragma unroll
                for (int j = 0; j < kJ; ++j) s2[i][j] = fma2(qb, kk[j][1], fma2(qa, kk[j][0], s2[i][j]));
            }
        }
        __syncthreads();                                                     // every warp is done with K
        if (next < n_kt) load_tile(sK, K, next);
        else asm volatile("cp.async.commit_group;" ::: "memory");
        // ---- mask, online softmax (16 lanes share a row), P transposed to shared memory ----
        const bool all_seen = !(kvp && by_pos) && !two_sided && kKeys <= left && k0 + kKeys - 1 <= lo_min;
        float al[kR];
#pragma unroll
        for (int i = 0; i < kR; ++i) {
            float s[kJ], mx = -INFINITY;
#pragma unroll
            for (int j = 0; j < kJ; ++j) {
                const float2 v = unpack2(s2[i][j]);
                s[j] = (v.x + v.y) * p.scale;
                if (!all_seen && !(key_l + 16 * j < left && (pos[j] <= lo[i] || (two_sided && pos[j] >= hi && my_row0 + i < n_rows))))
                    s[j] = -INFINITY;
                mx = fmaxf(mx, s[j]);
            }
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            const float mn = fmaxf(m[i], mx), ref = mn == -INFINITY ? 0.f : mn;
            al[i] = expf(m[i] - ref);                                        // 0 while nothing has been seen
            m[i] = mn;
            float sum = 0.f;
#pragma unroll
            for (int j = 0; j < kJ; ++j) {
                s[j] = expf(s[j] - ref);
                sum += s[j];
                s2[i][j] = __float_as_uint(s[j]);
            }
            l[i] = l[i] * al[i] + sum;
        }
#pragma unroll
        for (int j = 0; j < kJ; ++j) {
            float *dst = sP + (key_l + 16 * j) * L::kPPitch + my_row0;
#pragma unroll
            for (int i = 0; i < kR; i += 4)
                *reinterpret_cast<float4 *>(dst + i) =
                    make_float4(__uint_as_float((uint32_t)s2[i][j]), __uint_as_float((uint32_t)s2[i + 1][j]),
                                __uint_as_float((uint32_t)s2[i + 2][j]), __uint_as_float((uint32_t)s2[i + 3][j]));
        }
#pragma unroll
        for (int i = 0; i < kR / 2; ++i) {
            const uint64_t a2 = pack2(al[2 * i], al[2 * i + 1]);
#pragma unroll
            for (int c = 0; c < kC; ++c) acc[i][c] = mul2(acc[i][c], a2);
        }
        if (t + plan.splits < n_kt) load_pos(t + plan.splits);
        wait_copy();                                                         // V
        // ---- O += P V ----
        const int kb = kKeyWarps > 1 ? 16 * warp : 0;
#pragma unroll 4
        for (int key = kb; key < kb + (kKeyWarps > 1 ? 16 : kKeys); ++key) {
            uint64_t pp[kR / 2];
#pragma unroll
            for (int i = 0; i < kR / 4; ++i) {
                const float4 v = lds4(sP + key * L::kPPitch + my_row0 + 4 * i);
                pp[2 * i] = pack2(v.x, v.y); pp[2 * i + 1] = pack2(v.z, v.w);
            }
#pragma unroll
            for (int cc = 0; cc < kC / 4; ++cc) {
                const float4 v = lds4(sV + key * L::kKvPitch + 4 * tk + 64 * cc);
                const uint64_t vv[4] = {pack2(v.x, v.x), pack2(v.y, v.y), pack2(v.z, v.z), pack2(v.w, v.w)};
#pragma unroll
                for (int i = 0; i < kR / 2; ++i)
#pragma unroll
                    for (int e = 0; e < 4; ++e) acc[i][4 * cc + e] = fma2(pp[i], vv[e], acc[i][4 * cc + e]);
            }
        }
        __syncthreads();                                                     // every warp is done with V (and P)
        if (next < n_kt) load_tile(sV, V, next);
        else asm volatile("cp.async.commit_group;" ::: "memory");
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");

    // ---- partials to shared memory (where K and V were), then the merge over warps and CTAs ----
#pragma unroll
    for (int i = 0; i < kR; ++i)
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) l[i] += __shfl_xor_sync(0xffffffffu, l[i], o);
    __syncthreads();
    const int group = kKeyWarps > 1 ? warp : 0;
#pragma unroll
    for (int i = 0; i < kR / 2; ++i)
#pragma unroll
        for (int cc = 0; cc < kC / 4; ++cc) {
            float2 v[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) v[e] = unpack2(acc[i][4 * cc + e]);
            float *dst = part + (group * kM + my_row0 + 2 * i) * L::kQPitch + 4 * tk + 64 * cc;
            *reinterpret_cast<float4 *>(dst) = make_float4(v[0].x, v[1].x, v[2].x, v[3].x);
            *reinterpret_cast<float4 *>(dst + L::kQPitch) = make_float4(v[0].y, v[1].y, v[2].y, v[3].y);
        }
    if (tk == 0)
#pragma unroll
        for (int i = 0; i < kR; ++i) s_ml[group][my_row0 + i] = make_float2(m[i], l[i]);
    cg::cluster_group cluster = cg::this_cluster();
    if (plan.splits > 1) cluster.sync(); else __syncthreads();
    // rank r of the cluster finishes rows r, r + splits, ...; a thread four channels of one row
    const int n_mine = n_rows > rank ? (n_rows - rank + plan.splits - 1) / plan.splits : 0;
#pragma unroll 1
    for (int i = tid; i < n_mine * (kDP / 4); i += kThreads) {
        const int c = (i % (kDP / 4)) * 4, r = rank + i / (kDP / 4) * plan.splits;
        if (c >= d) continue;
        float mx = -INFINITY;
#pragma unroll 1
        for (int q = 0; q < plan.splits; ++q) {
            const float2 *ml = plan.splits > 1 ? cluster.map_shared_rank(&s_ml[0][0], q) : &s_ml[0][0];
#pragma unroll
            for (int w = 0; w < kKeyWarps; ++w) mx = fmaxf(mx, ml[w * kM + r].x);
        }
        const float ref = mx == -INFINITY ? 0.f : mx;
        float z = 0.f;
        float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
        for (int q = 0; q < plan.splits; ++q) {
            const float2 *ml = plan.splits > 1 ? cluster.map_shared_rank(&s_ml[0][0], q) : &s_ml[0][0];
            const float *src = plan.splits > 1 ? cluster.map_shared_rank(part, q) : part;
#pragma unroll
            for (int w = 0; w < kKeyWarps; ++w) {
                const float2 e = ml[w * kM + r];
                const float4 v = *reinterpret_cast<const float4 *>(src + (w * kM + r) * L::kQPitch + c);
                const float f = expf(e.x - ref);
                z = fmaf(e.y, f, z);
                o.x = fmaf(v.x, f, o.x); o.y = fmaf(v.y, f, o.y); o.z = fmaf(v.z, f, o.z); o.w = fmaf(v.w, f, o.w);
            }
        }
        const float inv = z > 0.f ? 1.f / z : 0.f;
        o.x *= inv; o.y *= inv; o.z *= inv; o.w *= inv;
        const float probe = (o.x + o.y + o.z + o.w + z) * 0.f;               // 0 unless something is Inf or NaN
        if (!(probe == 0.f)) s_bad[r] = 1;
        const int64_t out = s_out[r];
        stg4(reinterpret_cast<T *>(p.o) + out * d + c, o);
        if (c == 0 && p.lse) p.lse[out] = z > 0.f ? mx + logf(z) : -INFINITY;
    }
    __syncthreads();
#pragma unroll 1
    for (int r = rank; r < n_rows; r += plan.splits)
        if (s_bad[r] && (r / plan.splits) % (kThreads / 32) == warp)
            attn_row_warp<T, true>(p, s_out[r] / p.hq, (int)(s_out[r] % p.hq), sQ + r * L::kQPitch);
    if (plan.splits > 1) cluster.sync();                                     // peers may still be reading this CTA's partials
}

template <typename T, int kR, int kDP, int kKeyWarps>
cudaError_t launch_variant(const GenericParams &p, TiledPlan plan, int sm_count, int64_t max_kv, cudaStream_t s)
{
    using L = Layout<T, kR, kDP, kKeyWarps>;
    constexpr int kMost = 110 * 1024;                                        // two CTAs per SM (a cluster of 8 finds few places among
                                                                             // SMs that hold one); static shared memory comes on top
    // Clusters share the keys as long as every CTA finds an SM.  A walk of several tiles keeps as many tile pairs in
    // flight as two CTAs per SM leave room for; four CTAs per SM hide latency better where there are many row tiles
    // (kKeyWarps = 1: 93 and 280 us with one pair against 107 and 341 with two, local and sync of 2048 rows x 16 heads).
    const int64_t key_tiles = (max_kv + L::kKeys - 1) / L::kKeys, units = (int64_t)plan.n_tiles * p.hkv;
    plan.splits = 1;
    while (plan.splits < kMaxCluster && units * plan.splits <= sm_count && plan.splits * 2 <= key_tiles) plan.splits *= 2;
    const int64_t per_cta = (key_tiles + plan.splits - 1) / plan.splits;     // tiles of a CTA, at most
    plan.stages = 1;
    while (kKeyWarps > 1 && plan.stages < kMaxStages && plan.stages < per_cta && L::bytes(plan.stages + 1) <= kMost) ++plan.stages;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    static bool attr_set[64] = {};                                           // the attribute is per device
    if (e == cudaSuccess && !attr_set[dev & 63]) {
        e = cudaFuncSetAttribute(attn_tiled_kernel<T, kR, kDP, kKeyWarps>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMost);
        attr_set[dev & 63] = e == cudaSuccess;
    }
    if (e != cudaSuccess) return e;
    WaitFirstLaunch l(dim3((unsigned)((int64_t)plan.n_tiles * p.hkv * plan.splits)), dim3(L::kThreads), L::bytes(plan.stages), s);
    l.attr[1].id = cudaLaunchAttributeClusterDimension;
    l.attr[1].val.clusterDim.x = plan.splits; l.attr[1].val.clusterDim.y = 1; l.attr[1].val.clusterDim.z = 1;
    l.cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&l.cfg, attn_tiled_kernel<T, kR, kDP, kKeyWarps>, p, plan);
}

// M = 8, 16 (keys over warps), 32 (rows over warps; four CTAs of 64 channels share an SM.  64 rows at 8 per thread
// need 208 registers: two CTAs, and 308 instead of 280 us for 2048 causal rows of 16 heads of 64 channels)
template <typename T>
cudaError_t launch_rows(int rows, const GenericParams &p, const TiledPlan &plan, int sm_count, int64_t max_kv, cudaStream_t s)
{
    if (p.d <= 64) {
        switch (rows) {
        case 8: return launch_variant<T, 4, 64, 8>(p, plan, sm_count, max_kv, s);
        case 16: return launch_variant<T, 8, 64, 8>(p, plan, sm_count, max_kv, s);
        default: return launch_variant<T, 4, 64, 1>(p, plan, sm_count, max_kv, s);
        }
    }
    constexpr int kWide = sizeof(T) == 4 ? 4 : 8;                            // 128 fp32 keys of 128 channels: one CTA per SM
    switch (rows) {
    case 8: return launch_variant<T, 4, 128, kWide>(p, plan, sm_count, max_kv, s);
    case 16: return launch_variant<T, 8, 128, kWide>(p, plan, sm_count, max_kv, s);
    default: return launch_variant<T, 4, 128, 1>(p, plan, sm_count, max_kv, s);
    }
}

}  // namespace

cudaError_t launch_attn_generic(const GenericParams &p, int dtype, int max_kv, int sm_count, cudaStream_t s, int64_t *launches)
{
    if (p.n_rows == 0) return cudaSuccess;
    const int g = p.hq / p.hkv;
    // Segments of stacked rows: participants (local, remote-only), one participant each (decode local), or all rows.
    TiledPlan plan;
    int64_t longest = 0;
    plan.n_seg = 1;
    plan.row0[0] = 0; plan.row0[1] = (int32_t)p.n_rows;
    if (p.mode == kDecodeLocal) {
        plan.n_seg = (int32_t)p.n_rows;
        for (int i = 0; i <= plan.n_seg; ++i) plan.row0[i] = i;
    } else if (p.mode == kLocal || (p.mode == kSync && p.remote_only)) {
        plan.n_seg = p.n_seg;
        for (int i = 0; i <= plan.n_seg; ++i) plan.row0[i] = p.cu[i];
    }
    for (int i = 0; i < plan.n_seg; ++i) longest = max(longest, (int64_t)(plan.row0[i + 1] - plan.row0[i]) * g);
    auto tiles_of = [&](int rows) {
        int64_t n = 0;
        for (int i = 0; i < plan.n_seg; ++i) n += ((int64_t)(plan.row0[i + 1] - plan.row0[i]) * g + rows - 1) / rows;
        return n;
    };
    // The most rows per tile that still give every SM a tile (more rows read K and V less often), but no more than
    // the longest segment fills; 8 when none does, and clusters share the keys.
    int rows = 32;
    while (rows > 8 && (tiles_of(rows) * p.hkv < sm_count || rows >= 2 * longest)) rows /= 2;
    const int64_t tiles = tiles_of(rows);
    if (tiles * p.hkv > 0x7fffffffLL / kMaxCluster) return cudaErrorInvalidValue;
    plan.n_tiles = (int32_t)tiles;
    plan.tile0[0] = 0;
    for (int i = 0; i < plan.n_seg; ++i)
        plan.tile0[i + 1] = plan.tile0[i] + (int32_t)(((int64_t)(plan.row0[i + 1] - plan.row0[i]) * g + rows - 1) / rows);
    const cudaError_t e = dtype == FEDATTN_F32 ? launch_rows<float>(rows, p, plan, sm_count, max_kv, s)
                                             : launch_rows<__nv_bfloat16>(rows, p, plan, sm_count, max_kv, s);
    ++*launches;
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace fedattn
