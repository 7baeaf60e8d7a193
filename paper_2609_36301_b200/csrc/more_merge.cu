// Hierarchical top-k for a router whose expert dimension is sharded (the paper leaves "local top-k per device, then
// global top-k" to future work; the combination of the per-shard softmax statistics is Eq. app_online applied to whole
// shards).  Every shard has routed the same T tokens over its own experts with more_route_ex and reports its k best
// (id, logit) pairs per token and its log-sum-exp; once the shards' reports sit side by side in this GPU's memory
// (an all-gather of k pairs per token and shard -- nothing of size M crosses a link), one warp per token keeps the k
// best of the S k pairs under the full order (value descending, id ascending), then gates, ids and the expert histogram as
// in the router's own finish.
//
// Bound by reading the reports (S (8 k + 4) bytes per token) and, for few tokens, by the two launches.  A warp reads a
// token's rows of 4 k bytes each, all at once; what it does with them is ~350 instructions.  (One thread per token, which
// inserts S k pairs into a list in registers one after the other, took 92 us for 8 shards, 8192 tokens, k = 16.)
#include "more_internal.h"

#include "more_topk.cuh"

namespace more {

namespace {

constexpr int kMergeWarps = 8;                    // tokens per CTA

struct MergeParams {
    const int32_t* idx;      // [S][T][k]
    const float* val;        // [S][T][k]
    const float* lse;        // [S][T] or nullptr
    int S, T, k, M, gate_mode;
    uint32_t inv_k;          // ceil(2^32 / k); 0 for k = 1
    int base[MORE_MERGE_MAX_SHARDS];   // added to the ids of each shard
    int32_t* out_idx;
    float* out_gate;
    float* out_val;          // nullable
    float* out_lse;          // nullable
    int32_t* out_counts;
};

// out_counts = 0, in a kernel of its own so that the merge can be launched behind it before it has finished.
__global__ void __launch_bounds__(256) merge_clear_kernel(int32_t* counts, int M)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    for (int e = blockIdx.x * 256 + threadIdx.x; e < M; e += gridDim.x * 256) counts[e] = 0;
}

__global__ void __launch_bounds__(kMergeWarps * 32) merge_shards_kernel(const __grid_constant__ MergeParams p)
{
    constexpr unsigned kAll = 0xffffffffu;
    constexpr float kLog2e = 1.4426950408889634f, kLn2 = 0.6931471805599453f;
    __shared__ Cand buf[kMergeWarps][64];
    __shared__ int base[MORE_MERGE_MAX_SHARDS];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x < MORE_MERGE_MAX_SHARDS) base[threadIdx.x] = p.base[threadIdx.x];
    __syncthreads();
    const int t = blockIdx.x * kMergeWarps + warp;
    if (t < p.T) {
        const int k = p.k;
        auto get = [&](int f) {
            const int sh = p.inv_k ? (int)__umulhi((uint32_t)f, p.inv_k) : f;       // f / k
            const size_t at = ((size_t)sh * (size_t)p.T + (size_t)t) * (size_t)k + (size_t)(f - sh * k);
            const int raw = __ldg(p.idx + at);
            const float x = __ldg(p.val + at);
            const int e = raw + base[sh];
            return (raw < 0 || e >= p.M || !(x > -INFINITY)) ? no_cand() : Cand{x, e};      // (an unused slot)
        };
        float lse2 = 0.f;                                     // log2-domain log-sum-exp over all shards
        if (p.lse) {
            const float a = lane < p.S ? p.lse[(size_t)lane * p.T + t] : -INFINITY;
            const float b = lane + 32 < p.S ? p.lse[(size_t)(lane + 32) * p.T + t] : -INFINITY;
            float m = fmaxf(a, b);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(kAll, m, o));
            float z = (lane < p.S ? exp2f((a - m) * kLog2e) : 0.f) + (lane + 32 < p.S ? exp2f((b - m) * kLog2e) : 0.f);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) z += __shfl_xor_sync(kAll, z, o);
            lse2 = m * kLog2e + log2f(z);
        }
        const Cand c = warp_topk<4>(p.S * k, k, get, buf[warp], lane);
        const bool used = lane < k && c.id != INT_MAX;
        float inv = 1.f, ref2 = lse2;
        if (p.gate_mode == MORE_GATE_TOPK_SOFTMAX) {
            const float v0 = __shfl_sync(kAll, c.v, 0);
            float sum = used ? exp2f((c.v - v0) * kLog2e) : 0.f;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(kAll, sum, o);
            inv = 1.f / sum;
            ref2 = v0 * kLog2e;
        }
        asm volatile("griddepcontrol.wait;" ::: "memory");    // the counts are clear (and what ran before is complete)
        if (lane < k) {
            const size_t o = (size_t)t * (size_t)k + (size_t)lane;
            p.out_idx[o] = used ? c.id : -1;
            p.out_gate[o] = used ? exp2f(c.v * kLog2e - ref2) * inv : 0.f;
            if (p.out_val) p.out_val[o] = c.v;
            if (used) atomicAdd(p.out_counts + c.id, 1);
        }
        if (lane == 0 && p.lse && p.out_lse) p.out_lse[t] = lse2 * kLn2;
    }
}

}  // namespace

}  // namespace more

using namespace more;

extern "C" int more_merge_shards(const int32_t* idx, const float* topval, const float* lse, const int32_t* shard_base,
                                 int S, int T, int k, int M, int gate_mode, int32_t* out_idx, float* out_gate,
                                 float* out_topval, float* out_lse, int32_t* out_counts, void* stream)
{
    if (S < 1 || S > MORE_MERGE_MAX_SHARDS || T < 0 || k < 1 || k > MORE_K_MAX || M < 1) return MORE_ERR_SHAPE;
    if (gate_mode != MORE_GATE_TOPK_SOFTMAX && gate_mode != MORE_GATE_FULL_SOFTMAX) return MORE_ERR_MODE;
    if (!out_counts) return MORE_ERR_NULL;
    if (T > 0 && (!idx || !topval || !out_idx || !out_gate)) return MORE_ERR_NULL;
    if (gate_mode == MORE_GATE_FULL_SOFTMAX && !lse) return MORE_ERR_NULL;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int clear_blocks = M < 148 * 1024 ? (M + 1023) / 1024 : 148;
    merge_clear_kernel<<<clear_blocks, 256, 0, st>>>(out_counts, M);
    count_launch(1);
    if (T == 0) return cudaGetLastError() == cudaSuccess ? MORE_OK : MORE_ERR_CUDA;
    MergeParams p;
    p.idx = idx; p.val = topval; p.lse = lse;
    p.S = S; p.T = T; p.k = k; p.M = M; p.gate_mode = gate_mode;
    p.inv_k = k > 1 ? (uint32_t)(((1ull << 32) + (unsigned)k - 1) / (unsigned)k) : 0u;
    for (int s = 0; s < MORE_MERGE_MAX_SHARDS; ++s) p.base[s] = (shard_base && s < S) ? shard_base[s] : 0;
    p.out_idx = out_idx; p.out_gate = out_gate; p.out_val = out_topval; p.out_lse = out_lse; p.out_counts = out_counts;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)((T + kMergeWarps - 1) / kMergeWarps));
    cfg.blockDim = dim3(kMergeWarps * 32);
    cfg.stream = st;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, merge_shards_kernel, p) != cudaSuccess) return MORE_ERR_CUDA;
    count_launch(1);
    return cudaGetLastError() == cudaSuccess ? MORE_OK : MORE_ERR_CUDA;
}
