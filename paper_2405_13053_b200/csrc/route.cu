// Token -> adapter grouping (Sec. 3.3): histogram, exclusive prefix sum and the stable
// permutation of the T*k (token, pick) slots by adapter index.  Integer work only.
//
// One CTA of 32 warps, each over a contiguous share of the slots, 32 at a time.  First pass: every warp counts its share by
// key (__match_any_sync finds the equal keys among 32 slots).  Then the counts are summed over keys and, per key, over the
// warps before.  Second pass: the rank of a slot is that sum + the warp's running count of the key + the equal keys in
// lower lanes.  All terms count slots with a smaller slot number, so equal keys keep ascending slot order.  Latency-bound
// (one CTA): three block barriers in all, where a walk in tiles of 1024 slots took three per tile (8192 slots: 14.0 us).
#include "common.cuh"

namespace meteora {

constexpr int kRouteThreads = 1024;
constexpr int kRouteWarps = kRouteThreads / 32;
constexpr int kRouteHeld = 8;      // steps whose keys a warp keeps in registers between the passes

__global__ void __launch_bounds__(kRouteThreads)
k_route(const int32_t* __restrict__ topk_idx, int S, int N, int32_t* __restrict__ counts,
        int32_t* __restrict__ offsets, int32_t* __restrict__ perm) {
    __shared__ int warp_cnt[kRouteWarps][METEORA_MAX_N];  // counts, then the next free position, per (warp, key)
    __shared__ int total[METEORA_MAX_N];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned below = (1u << lane) - 1u;
    const long long steps_all = ((long long)S + 31) / 32;
    const long long s_lo = steps_all * warp / kRouteWarps * 32, s_hi = steps_all * (warp + 1) / kRouteWarps * 32;
    for (int e = lane; e < N; e += 32) warp_cnt[warp][e] = 0;
    asm volatile("griddepcontrol.wait;" ::: "memory");               // (launched dependent: set-up under the kernel ahead)
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    auto key_of = [&](long long s) { return s < S ? min(max(__ldg(topk_idx + s), 0), N - 1) : -1 - lane; };   // dead lanes match nobody
    int held[kRouteHeld];
#pragma unroll
    for (int i = 0; i < kRouteHeld; ++i) held[i] = s_lo + 32 * i < s_hi ? key_of(s_lo + 32 * i + lane) : -1 - lane;
    __syncwarp();
    auto count = [&](int key) {
        const unsigned peers = __match_any_sync(0xFFFFFFFFu, key);
        if (key >= 0 && (peers & below) == 0) warp_cnt[warp][key] += __popc(peers);
        __syncwarp();
    };
#pragma unroll
    for (int i = 0; i < kRouteHeld; ++i)
        if (s_lo + 32 * i < s_hi) count(held[i]);
    for (long long s = s_lo + 32 * kRouteHeld; s < s_hi; s += 32) count(key_of(s + lane));
    __syncthreads();
    if (tid < N) {
        int acc = 0;
#pragma unroll
        for (int w = 0; w < kRouteWarps; ++w) {
            const int c = warp_cnt[w][tid];
            warp_cnt[w][tid] = acc;
            acc += c;
        }
        total[tid] = acc;
        counts[tid] = acc;
    }
    __syncthreads();
    if (tid < N) {                                                   // first position of the key's group
        int first = 0;
        for (int e = 0; e < tid; ++e) first += total[e];
        offsets[tid] = first;
        if (tid == N - 1) offsets[N] = first + total[tid];
#pragma unroll
        for (int w = 0; w < kRouteWarps; ++w) warp_cnt[w][tid] += first;
    }
    __syncthreads();
    auto place = [&](int key, long long s) {
        const unsigned peers = __match_any_sync(0xFFFFFFFFu, key);
        int at = 0;
        if (key >= 0) at = warp_cnt[warp][key];
        __syncwarp();
        if (key >= 0) {
            if ((peers & below) == 0) warp_cnt[warp][key] = at + __popc(peers);
            perm[at + __popc(peers & below)] = (int)s;
        }
        __syncwarp();
    };
#pragma unroll
    for (int i = 0; i < kRouteHeld; ++i)
        if (s_lo + 32 * i < s_hi) place(held[i], s_lo + 32 * i + lane);
    for (long long s = s_lo + 32 * kRouteHeld; s < s_hi; s += 32) place(key_of(s + lane), s + lane);
}

int launch_route(const int32_t* topk_idx, int T, int k, int N, int32_t* counts, int32_t* offsets, int32_t* perm,
                 cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(1);
    cfg.blockDim = dim3(kRouteThreads);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = tuning().pdl ? 1 : 0;
    return cuda_status(cudaLaunchKernelEx(&cfg, k_route, topk_idx, T * k, N, counts, offsets, perm));
}

}  // namespace meteora
