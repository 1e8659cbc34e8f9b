// Shared declarations of the FedAttn CUDA library (host dispatch <-> kernel launchers).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include "fedattn.h"

namespace fedattn {

// Workspace layout: [0, 256) status area (word 0: the status word; bytes 64..71: the sequence number of the
// latest sparse aggregation known to be complete), then the scratch region.
constexpr size_t kStatusBytes = 256;
constexpr size_t kDoneSeqOffset = 64;
constexpr int kMaxP = FEDATTN_MAX_PARTICIPANTS;
// Upper bound on spin iterations of any in-kernel wait before it gives up.
constexpr uint32_t kSpinLimit = 1u << 22;

// m2 ln 2 + ln l with one rounding beside the logarithm's: the product and the sum keep what they round off
__device__ __forceinline__ float lse_exact(float m2, float l)
{
    const float ln2 = 0.6931471805599453f, ln2_rest = (float)(0.69314718055994530942 - (double)0.6931471805599453f);
    const float prod = m2 * ln2, prod_rest = fmaf(m2, ln2, -prod) + m2 * ln2_rest;
    const float lg = logf(l), sum = prod + lg, back = sum - prod;
    return sum + (((prod - (sum - back)) + (lg - back)) + prod_rest);
}

// How an entry point answers a runtime call.  The runtime keeps a failed call's error until it is taken; left there, the
// next call's own check would report it although its work was enqueued.
inline fedattn_status status_of(cudaError_t e)
{
    if (e == cudaSuccess) return FEDATTN_OK;
    cudaGetLastError();
    return FEDATTN_ERR_CUDA;
}

struct Context {
    int device;
    int sm_count;
    char *workspace;       // dev
    size_t workspace_bytes;
    int32_t *status;       // dev, == workspace
    char *scratch;         // dev, workspace + kStatusBytes
    size_t scratch_bytes;
    int64_t launches;
    int64_t tc_launches;   // launches of the tcgen05 attention kernel among them
    int64_t agg_seq;       // sequence number of the latest sparse aggregation call
    uint64_t agg_key;      // key of the stream that call ran on (early-start bookkeeping)
    void *encode_tiled;    // cuTensorMapEncodeTiled entry point (driver), or nullptr
};

// ---- early-start bookkeeping (programmatic dependent launch) ------------------------------------
struct MemRange {
    const void *p;
    size_t bytes;
};
struct EarlyStart {
    bool early;          // the inputs may be read before the preceding grid of the stream is complete
    int64_t seq;         // this call's sequence number in its context (0: none, publish nothing)
    int64_t need_seq;    // the context's latest recorded call that reads or writes one of `out` (0: none;
                         // INT64_MAX: one that cannot be named, wait before the first write)
    int device;
    cudaStream_t stream;
    bool capturing;
};
// Records `in` (read) and `out` (written) as buffers that grids of this call may still be using when
// later grids of `stream` start, and decides how the call may start.  writes_before_wait: the call's
// kernel writes `out` before its griddepcontrol.wait when need_seq allows it (otherwise overlaps of
// `out` with recorded buffers do not matter).  owner / seq_counter / owner_key: the context's done
// word, its sequence counter and the key of the stream its numbered calls last ran on (all null for
// calls without sequence numbers).
EarlyStart early_start(int device, cudaStream_t stream, const MemRange *in, int n_in, const MemRange *out, int n_out,
                       bool writes_before_wait = false, const void *owner = nullptr, int64_t *seq_counter = nullptr,
                       uint64_t *owner_key = nullptr);
// Behind the call's last launch, or where it ends without one; returns e.  A call that was not launched leaves no record of
// the grids before it behind.  While the stream is being captured, notes the node that the last launch became.
cudaError_t early_start_end(const EarlyStart &r, cudaError_t e);
// Whether the latest kernel that this library put on the stream, by any context or none, releases its dependents early
// (selection, gather, bf16 decode: early_start_end notes them; the others note themselves).  A hint for the form of a
// launch, kept for a few streams; no order rests on it.
bool front_releases(int device, cudaStream_t stream);
void front_note(int device, cudaStream_t stream, bool releases);
// The owner's sequence numbers are about to lose their meaning (its context is being destroyed).
void early_start_forget(int device, const void *owner);

// Launch configuration of a kernel that calls grid_wait() before it reads or writes anything: its CTAs are set up while the
// preceding grid of the stream ends, instead of behind its end, and it completes behind that grid like an ordinary launch.
// It releases nothing early, so it needs no record below.  Bound by launches and the gaps between them, the fp32 round of
// two 128-token participants (local, concatenation, sync) takes 24.6 us with ordinary launches and 19.7-20.6 with these; the
// round of six ragged bf16 segments, 16 / 4 heads of 64, 84.4 -> 82.4; local + remote + merge of 2160 tokens 120.1 -> 117.7.
// (Dependents released at the kernel's start: 21.9, 82.4, 116.8, and every output would need a record.)
// Concatenation, merge and SIMT attention are launched so behind kernels that release early too: us a pass in a loop,
// ordinary -> this, fp32 4 x 128 tokens, 8 / 2 heads of 64: selection, sync 24.7 -> 22.3; gather, sync 20.5 -> 18.3;
// selection, local, remote, merge 43.6 -> 37.1; selection, concatenation 12.8 -> 11.3.  4 x 512, 128 channels: 113.1 -> 112.6,
// 104.6 -> 102.5, 224.6 -> 218.5, 18.5 -> 16.9.  8 x 1024, 8 / 8 heads of 64: 535.7 -> 534.2, 527.1 -> 520.1, 804.5 -> 791.9,
// 26.7 -> 25.2.  bf16 decode of 8 x 4096, local, shared and their merge 59.7 -> 58.8.  (As graphs: 0 to 7 us less; 0.4 us more
// in one, selection, sync at 4 x 512, where the runs differ by 0.2.)
struct WaitFirstLaunch {
    cudaLaunchAttribute attr[2];
    cudaLaunchConfig_t cfg;
    WaitFirstLaunch(dim3 grid, dim3 block, size_t smem, cudaStream_t s)
    {
        memset(&cfg, 0, sizeof(cfg));
        cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = s;
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
    }
    WaitFirstLaunch(const WaitFirstLaunch &) = delete;
};
// Every kernel of this library may be resident while earlier grids still write what it reads behind its wait.  So none reads
// through ld.global.nc or __ldg, which want data that nobody writes during the kernel's life and which the compiler need not
// keep behind the wait: plain loads, or volatile ones.  (Positions by ld_int: a plain load through a pointer from a parameter
// block is a generic one and takes the SIMT attention other registers: fp32 round of 2 x 128 tokens 19.3 -> 19.5 us.)
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ int ld_int(const int32_t *p)
{
    int v;
    asm volatile("ld.global.s32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}

// ---- tiled SIMT attention (fp32 or bf16 storage, any head_dim <= 128) -----------------------
enum GenericMode { kLocal = 0, kSync = 1, kDecodeLocal = 2, kDecodeSync = 3 };

struct GenericParams {
    const void *q, *k, *v;
    void *o;
    float *lse;
    int64_t n_rows;               // query rows (tokens, or participants for decode)
    int32_t hq, hkv, d;
    float scale;
    int32_t causal;
    int32_t mode;                 // GenericMode
    int32_t remote_only;          // kSync: a row sees the keys positioned before its segment (cu) and, when
                                  // causal == 0, those positioned after it
    int64_t kv_tok_stride;        // elements between consecutive KV rows of one head
    int64_t kv_head_stride;       // elements between KV heads
    int64_t kv_pos_head_stride;   // ints between heads in kv_pos (0 = shared)
    int64_t total_kv;             // sync: rows of the aggregated KV
    const int32_t *q_pos;         // nullable
    const int32_t *kv_pos;        // nullable
    const int32_t *kv_len;        // decode: dev lengths
    int64_t cache_stride;         // decode local: elements between participants' caches
    int32_t n_seg;
    int32_t cu[kMaxP + 1];        // local: segment offsets
};

// max_kv: an upper bound (decode: the caller's) on the keys of one row, which only sets how many CTAs share them
cudaError_t launch_attn_generic(const GenericParams &p, int dtype, int max_kv, int sm_count, cudaStream_t s, int64_t *launches);

// ---- aggregation -----------------------------------------------------------------------------
struct PartsParams {
    const void *k[kMaxP];
    const void *v[kMaxP];
    int32_t n;
    int32_t off[kMaxP + 1];       // prefix sum of L_n  (rows)
    int32_t cu_kv[kMaxP + 1];     // prefix sum of k_sel (rows), sparse modes
};

cudaError_t launch_concat(const PartsParams &pp, int hkv, int d, int elt_bytes, void *k_agg, void *v_agg,
                          int32_t *kv_pos, int32_t *cu_kv, cudaStream_t s, int sm_count, int64_t *launches);

cudaError_t launch_topk_fused(const PartsParams &pp, int hkv, int d, int dtype, void *k_agg, void *v_agg,
                              int32_t *kv_pos, int32_t *cu_kv, int32_t *sel_idx_out, Context *ctx, cudaStream_t s);
cudaError_t launch_gather(const PartsParams &pp, int hkv, int d, int elt_bytes, const int32_t *sel_idx,
                          void *k_agg, void *v_agg, int32_t *kv_pos, int32_t *cu_kv, int32_t *sel_idx_out,
                          int32_t *status, int device, int sm_count, cudaStream_t s, int64_t *launches);

// ---- prefill calls (local, sync, remote-only sync); bf16 runs on tensor cores (tcgen05 + TMEM + TMA) --------
struct PrefillParams {
    const void *q, *k, *v;
    void *o;
    float *lse;
    int64_t n_q_rows;
    int64_t total_kv;             // rows of K/V (== n_q_rows for local)
    int32_t hq, hkv, d;
    float scale;
    int32_t causal;
    int32_t sync;                 // 0 local, 1 sync
    int32_t remote_only;          // sync: a row sees the aggregated rows positioned before its segment (and, when
                                  // causal == 0, those positioned after it)
    int32_t kv_head_major;
    const int32_t *kv_pos;        // nullable
    int32_t general;              // sync, causal: every (query, key) pair is tested on explicit positions
    const int32_t *q_pos;         // general: nullable (= row index)
    int32_t *tab;                 // general: scratch for the position tables (position_table_bytes)
    int32_t n_seg;
    int32_t cu[kMaxP + 1];        // query segments (local: also the KV segments)
};
// the same call for the SIMT kernels
inline GenericParams generic_params(const PrefillParams &p)
{
    GenericParams g = {};
    g.q = p.q; g.k = p.k; g.v = p.v; g.o = p.o; g.lse = p.lse;
    g.n_rows = p.n_q_rows; g.hq = p.hq; g.hkv = p.hkv; g.d = p.d;
    g.scale = p.scale; g.causal = p.causal; g.mode = p.sync ? kSync : kLocal; g.remote_only = p.remote_only;
    g.kv_tok_stride = p.kv_head_major ? p.d : (int64_t)p.hkv * p.d;
    g.kv_head_stride = p.kv_head_major ? p.total_kv * p.d : p.d;
    g.kv_pos_head_stride = p.kv_head_major ? p.total_kv : 0;
    g.total_kv = p.total_kv; g.q_pos = p.q_pos; g.kv_pos = p.kv_pos;
    g.n_seg = p.n_seg;
    for (int i = 0; i <= p.n_seg; ++i) g.cu[i] = p.cu[i];
    return g;
}
bool prefill_sm100_supported(const Context *ctx);
// whether the tensor-core kernel takes a bf16 call (its work-item arithmetic has a limited range)
bool prefill_sm100_takes(const Context *ctx, const PrefillParams &p);
// scratch bytes of the per-tile position tables of a general-position sync call
size_t position_table_bytes(int hkv, int64_t n_q_rows, int64_t total_kv);
cudaError_t launch_prefill_sm100(Context *ctx, const PrefillParams &p, cudaStream_t s);
// one small kernel whose bounded wait runs out after max_polls polls (raises FEDATTN_ERR_TIMEOUT)
cudaError_t launch_wait_selftest(Context *ctx, int max_polls, cudaStream_t s);

// ---- merge of two partial attention results through their log-sum-exps ----------------------
cudaError_t launch_merge(int dtype, int64_t n_rows, int hq, int d, const void *o_a, const float *lse_a, const void *o_b,
                         const float *lse_b, void *o, float *lse, int sm_count, cudaStream_t s, int64_t *launches);

// ---- bf16 split-KV decode (tensor-core scores, warp-shuffle softmax) ---------------------------
struct DecodeParams {
    const void *q, *k, *v;
    void *o;
    float *lse;
    int32_t n_part, hq, hkv, d;
    float scale;
    int32_t sync;
    int64_t cache_stride;
    const int32_t *kv_len;
    int32_t max_kv_len;
    float *partial;               // scratch: per-split partial results
    size_t partial_bytes;
    int32_t g_shift;              // log2(hq / hkv) when that is a power of two, else -1 (set by the launcher)
    int32_t early;                // inputs may be read before the preceding grid is complete (set by the launcher)
};
size_t decode_scratch_bytes(int n_part, int hq, int d, int sm_count);
cudaError_t launch_decode_bf16(const Context *ctx, const DecodeParams &p, cudaStream_t s, int64_t *launches);

}  // namespace fedattn
