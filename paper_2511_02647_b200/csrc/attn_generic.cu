// Generic SIMT attention kernel: fp32 or bf16 storage, fp32 arithmetic, head_dim <= 128.
// Serves the fp32 configuration (tensor cores have no fp32 kind and TF32 would miss the 1e-4
// bound) and decode at the types and head dims that the tensor-core decode does not cover.  One warp owns one (query row, query head): lanes split the keys of a
// 32-key block for the logits, and split the head dimension for the weighted value sum.
#include "attn_row.cuh"

namespace fedattn {

constexpr int kWarpsPerBlock = 4;

template <typename T>
__global__ void __launch_bounds__(kWarpsPerBlock * 32)
attn_generic_kernel(const __grid_constant__ GenericParams p)
{
    __shared__ float q_s[kWarpsPerBlock][FEDATTN_MAX_HEAD_DIM];
    const int warp = threadIdx.x >> 5;
    const int64_t item = (int64_t)blockIdx.x * kWarpsPerBlock + warp;
    if (item >= p.n_rows * p.hq) return;            // whole warp leaves together
    attn_row_warp<T>(p, item / p.hq, (int)(item % p.hq), q_s[warp]);
}

cudaError_t launch_attn_generic(const GenericParams &p, int dtype, cudaStream_t s, int64_t *launches)
{
    const int64_t items = p.n_rows * p.hq;
    if (items == 0) return cudaSuccess;
    const int64_t blocks = (items + kWarpsPerBlock - 1) / kWarpsPerBlock;
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
    if (dtype == FEDATTN_F32)
        attn_generic_kernel<float><<<(unsigned)blocks, kWarpsPerBlock * 32, 0, s>>>(p);
    else
        attn_generic_kernel<__nv_bfloat16><<<(unsigned)blocks, kWarpsPerBlock * 32, 0, s>>>(p);
    ++*launches;
    return cudaGetLastError();
}

}  // namespace fedattn
