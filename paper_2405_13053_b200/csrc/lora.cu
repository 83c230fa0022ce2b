// Low-rank shrink (x A_i) and expand ((x A_i) B_i, weighted and summed over the picks) of Eq. 2
// on CUDA cores.  The shrink goes adapter by adapter over the grouped slots (Sec. 3.3 grouping from meteora_route): a CTA
// takes up to kSegSlots slots of ONE adapter, stages that adapter's A_i in shared memory chunk by chunk and reuses it
// for all its slots.  The expand is token-major and sums the k picks in pick order, so it needs no atomics.
#include "common.cuh"

#include <algorithm>
#include <atomic>

namespace meteora {

constexpr int kSegSlots = 32;    // slots of one adapter per CTA
constexpr int kSegWarps = 8;
constexpr int kSegSlotsPerWarp = kSegSlots / kSegWarps;
constexpr int kSegRows = 8;      // adapter rows (rank entries) staged at a time
constexpr int kSegChunkBytes = 32 * 1024;

template <typename TI>
__global__ void __launch_bounds__(kSegWarps * 32)
k_shrink_segments(const TI* __restrict__ x, const TI* __restrict__ A, const int32_t* __restrict__ offsets,
                  const int32_t* __restrict__ perm, int d_in, int N, int r, int k, float* __restrict__ u) {
    constexpr int DC = kSegChunkBytes / (kSegRows * (int)sizeof(TI));  // elements of d_in per staged chunk
    __shared__ __align__(16) TI sA[kSegRows][DC];
    __shared__ int s_tile[3];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    if (tid == 0) {  // which (adapter, tile of its group) is this CTA?
        int b = blockIdx.x, e = 0;
        for (; e < N; ++e) {
            const int c = offsets[e + 1] - offsets[e];
            const int nt = (c + kSegSlots - 1) / kSegSlots;
            if (b < nt) break;
            b -= nt;
        }
        s_tile[0] = e < N ? e : -1;
        if (e < N) {
            s_tile[1] = offsets[e] + b * kSegSlots;
            s_tile[2] = min(offsets[e + 1], s_tile[1] + kSegSlots);
        }
    }
    __syncthreads();
    const int e = s_tile[0];
    if (e < 0) return;
    const int p_begin = s_tile[1], p_end = s_tile[2];
    const bool vec = (d_in % 8) == 0;

    int slot[kSegSlotsPerWarp];
#pragma unroll
    for (int i = 0; i < kSegSlotsPerWarp; ++i) {
        const int p = p_begin + warp + i * kSegWarps;
        slot[i] = p < p_end ? perm[p] : -1;
    }

    for (int r0 = 0; r0 < r; r0 += kSegRows) {
        const int rows = min(kSegRows, r - r0);
        float acc[kSegSlotsPerWarp][kSegRows];
#pragma unroll
        for (int i = 0; i < kSegSlotsPerWarp; ++i)
#pragma unroll
            for (int q = 0; q < kSegRows; ++q) acc[i][q] = 0.f;

        for (int d0 = 0; d0 < d_in; d0 += DC) {
            const int len = min(DC, d_in - d0);
            __syncthreads();  // previous chunk fully consumed
            const TI* src = A + ((size_t)e * r + r0) * d_in + d0;
            if (vec) {
                const int vec_per_row = len / 8;
                for (int v = tid; v < rows * vec_per_row; v += kSegWarps * 32) {
                    const int q = v / vec_per_row, c = v - q * vec_per_row;
                    if (sizeof(TI) == 2) {
                        *reinterpret_cast<uint4*>(&sA[q][c * 8]) =
                            *reinterpret_cast<const uint4*>(src + (size_t)q * d_in + c * 8);
                    } else {
                        *reinterpret_cast<float4*>(&sA[q][c * 8]) =
                            *reinterpret_cast<const float4*>(src + (size_t)q * d_in + c * 8);
                        *reinterpret_cast<float4*>(&sA[q][c * 8 + 4]) =
                            *reinterpret_cast<const float4*>(src + (size_t)q * d_in + c * 8 + 4);
                    }
                }
            } else {
                for (int v = tid; v < rows * len; v += kSegWarps * 32) {
                    const int q = v / len, c = v - q * len;
                    sA[q][c] = src[(size_t)q * d_in + c];
                }
            }
            __syncthreads();
#pragma unroll
            for (int i = 0; i < kSegSlotsPerWarp; ++i) {
                if (slot[i] < 0) continue;
                const TI* xt = x + (size_t)(slot[i] / k) * d_in + d0;
                if (vec) {
                    // all of the slot's x values of this chunk first (one round trip to memory instead of one
                    // per 256 columns), then the products against the staged rows
                    constexpr int NV = DC / 256;
                    float xv[NV][8];
#pragma unroll
                    for (int v = 0; v < NV; ++v) {
                        const int d = lane * 8 + v * 256;
                        if (d < len) {
                            load8(xt + d, xv[v]);
                        } else {
#pragma unroll
                            for (int c = 0; c < 8; ++c) xv[v][c] = 0.f;
                        }
                    }
#pragma unroll
                    for (int v = 0; v < NV; ++v) {
                        const int d = lane * 8 + v * 256;
                        if (d < len) {
#pragma unroll
                            for (int q = 0; q < kSegRows; ++q) {
                                if (q < rows) {
                                    float av[8];
                                    load8(&sA[q][d], av);
#pragma unroll
                                    for (int c = 0; c < 8; ++c) acc[i][q] = fmaf(av[c], xv[v][c], acc[i][q]);
                                }
                            }
                        }
                    }
                } else {
                    for (int d = lane; d < len; d += 32) {
                        const float xv = to_f32(xt[d]);
#pragma unroll
                        for (int q = 0; q < kSegRows; ++q)
                            if (q < rows) acc[i][q] = fmaf(to_f32(sA[q][d]), xv, acc[i][q]);
                    }
                }
            }
        }
#pragma unroll
        for (int i = 0; i < kSegSlotsPerWarp; ++i) {
#pragma unroll
            for (int q = 0; q < kSegRows; ++q) {
                const float v = warp_sum(acc[i][q]);
                if (lane == 0 && slot[i] >= 0 && q < rows) u[(size_t)slot[i] * r + r0 + q] = v;
            }
        }
    }
}

// delta[t,o] = sum_j w[t,j] * sum_p B[idx[t,j], o, p] * u[t*k + j, p].   One thread per output row o,
// kExpTokens tokens per CTA so that the B rows of an adapter picked by several of them stay in L1.
constexpr int kExpTokens = 8;
constexpr int kExpThreads = 256;

template <typename TI>
__global__ void __launch_bounds__(kExpThreads)
k_expand(const TI* __restrict__ B, const int32_t* __restrict__ topk_idx, const float* __restrict__ topk_w,
         const float* __restrict__ u, int T, int d_out, int N, int r, int k, float* __restrict__ delta) {
    __shared__ int s_idx[kExpTokens * METEORA_MAX_K];
    __shared__ float s_w[kExpTokens * METEORA_MAX_K];
    __shared__ float s_u[kExpTokens * METEORA_MAX_K * METEORA_MAX_R];
    const int t0 = blockIdx.x * kExpTokens;
    const int nt = min(kExpTokens, T - t0);
    for (int i = threadIdx.x; i < nt * k; i += kExpThreads) {
        s_idx[i] = min(max(topk_idx[(size_t)t0 * k + i], 0), N - 1);
        s_w[i] = topk_w[(size_t)t0 * k + i];
    }
    for (int i = threadIdx.x; i < nt * k * r; i += kExpThreads) s_u[i] = u[(size_t)t0 * k * r + i];
    __syncthreads();
    const int o = blockIdx.y * kExpThreads + threadIdx.x;
    if (o >= d_out) return;
    const bool vec = (r % 8) == 0;
    for (int tt = 0; tt < nt; ++tt) {
        float out = 0.f;
        for (int j = 0; j < k; ++j) {
            const TI* brow = B + ((size_t)s_idx[tt * k + j] * d_out + o) * r;
            const float* uj = &s_u[(tt * k + j) * r];
            float acc = 0.f;
            if (vec) {
                for (int p = 0; p < r; p += 8) {
                    float bv[8];
                    load8(brow + p, bv);
#pragma unroll
                    for (int c = 0; c < 8; ++c) acc = fmaf(bv[c], uj[p + c], acc);
                }
            } else {
                for (int p = 0; p < r; ++p) acc = fmaf(to_f32(brow[p]), uj[p], acc);
            }
            out = fmaf(s_w[tt * k + j], acc, out);
        }
        delta[(size_t)(t0 + tt) * d_out + o] = out;
    }
}

// The same for bf16 adapters of a rank that is a multiple of 8, with the B rows of 128 outputs and ALL adapters staged in
// shared memory once per CTA: lane l of a warp owns outputs 4 l .. 4 l + 3 of the CTA's 128 and a warp walks groups of 4
// consecutive tokens, so B is read from shared memory without bank conflicts (slab[e][8 rank entries][i][lane] holds
// output 4 lane + i) and delta leaves 512 bytes per warp and token.  Bound by the issue of unpacking and FMAs (per pick and
// output: one 16-byte read, 8 unpacks, 4 packed FMAs) and by writing delta once; four tokens side by side hide the
// latency of the reads.  The kernel above gathers 16 bytes of B per (token, pick, output) through L1 / L2.
constexpr int kSlabTokens = 4;
constexpr size_t kSlabSmem = 200 * 1024;

template <int R8>
__global__ void __launch_bounds__(256)
k_expand_slab(const __nv_bfloat16* __restrict__ B, const int32_t* __restrict__ topk_idx, const float* __restrict__ topk_w,
              const float* __restrict__ u, int T, int d_out, int N, int k, float* __restrict__ delta) {
    constexpr int R = R8 * 8, TT = kSlabTokens;
    extern __shared__ __align__(16) uint4 slab[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int o0 = blockIdx.x * 128, n = k * R;
    float* s_u = reinterpret_cast<float*>(slab + (size_t)N * R8 * 128) + warp * TT * n;            // [token][pick][R]
    int* s_e = reinterpret_cast<int*>(reinterpret_cast<float*>(slab + (size_t)N * R8 * 128) + 8 * TT * n) + warp * TT * k;
    const uint4* Bv = reinterpret_cast<const uint4*>(B);
    for (int v = threadIdx.x; v < N * R8 * 128; v += 256) {         // [e][output][c]: as B lies in memory
        const int c = v % R8, row = (v / R8) & 127, e = v / (R8 * 128);
        const bool in = o0 + row < d_out;
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(slab + ((e * R8 + c) * 4 + (row & 3)) * 32 + (row >> 2));
        const uint4* src = Bv + ((size_t)e * d_out + (in ? o0 + row : 0)) * R8 + c;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(in ? 16 : 0) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");               // u comes from the grid before, the weights do not
    const int g_all = (T + TT - 1) / TT;
    const int g_lo = (int)((long long)g_all * blockIdx.y / gridDim.y), g_hi = (int)((long long)g_all * (blockIdx.y + 1) / gridDim.y);
    // the next group's routing and its first 64 shrink values are on their way while this one is expanded
    int e_n = 0;
    float w_n = 0.f, u_n[2] = {0.f, 0.f};
    auto fetch = [&](int g) {
        if (g >= g_hi) return;
        const int slots = min(TT, T - g * TT) * k;
        const size_t s0 = (size_t)g * TT * k;
        e_n = lane < slots ? min(max(__ldg(topk_idx + s0 + lane), 0), N - 1) : 0;
        w_n = lane < slots ? __ldg(topk_w + s0 + lane) : 0.f;
#pragma unroll
        for (int h = 0; h < 2; ++h) u_n[h] = lane + 32 * h < slots * R ? __ldg(u + s0 * R + lane + 32 * h) : 0.f;
    };
    fetch(g_lo + warp);
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    for (int g = g_lo + warp; g < g_hi; g += 8) {
        const int nt = min(TT, T - g * TT), slots = nt * k;
        const size_t s0 = (size_t)g * TT * k;
        const float w = w_n;
        if (lane < TT * k) s_e[lane] = e_n;
        for (int c0 = 0; c0 < TT * n; c0 += 32) {
            const int c = c0 + lane;
            const float wj = __shfl_sync(0xFFFFFFFFu, w, min(c / R, TT * k - 1));
            const float uv = c0 == 0 ? u_n[0] : c0 == 32 ? u_n[1] : c < slots * R ? __ldg(u + s0 * R + c) : 0.f;
            if (c < TT * n) s_u[c] = wj * uv;
        }
        fetch(g + 8);
        __syncwarp();
        unsigned long long acc[TT][4];
#pragma unroll
        for (int tt = 0; tt < TT; ++tt)
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[tt][i] = 0ull;
        for (int j = 0; j < k; ++j) {
#pragma unroll
            for (int tt = 0; tt < TT; ++tt) {
                const uint4* rows = slab + (size_t)s_e[tt * k + j] * (R8 * 128) + lane;
                const float* up = s_u + (tt * k + j) * R;
#pragma unroll
                for (int c = 0; c < R8; ++c) {
                    const ulonglong2 ua = *reinterpret_cast<const ulonglong2*>(up + c * 8);
                    const ulonglong2 ub = *reinterpret_cast<const ulonglong2*>(up + c * 8 + 4);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const uint4 b = rows[(c * 4 + i) * 32];
                        fma2(acc[tt][i], bf16x2_to_f32x2(b.x), ua.x);
                        fma2(acc[tt][i], bf16x2_to_f32x2(b.y), ua.y);
                        fma2(acc[tt][i], bf16x2_to_f32x2(b.z), ub.x);
                        fma2(acc[tt][i], bf16x2_to_f32x2(b.w), ub.y);
                    }
                }
            }
        }
#pragma unroll
        for (int tt = 0; tt < TT; ++tt) {
            if (tt >= nt) break;
            float out[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) out[i] = __uint_as_float((uint32_t)acc[tt][i]) + __uint_as_float((uint32_t)(acc[tt][i] >> 32));
            float* dst = delta + ((size_t)g * TT + tt) * d_out + o0 + lane * 4;
            if (d_out % 4 == 0) {
                if (o0 + lane * 4 < d_out) *reinterpret_cast<float4*>(dst) = make_float4(out[0], out[1], out[2], out[3]);
            } else {
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (o0 + lane * 4 + i < d_out) dst[i] = out[i];
            }
        }
        __syncwarp();
    }
}

// Where the tensor cores take the layer, the picks' shrink comes from token tiles (all adapters as one dense product, the
// picks gathered on the chip); else adapter by adapter over the bucketed slots.
int launch_shrink(const void* x, const void* A, const int32_t* topk_idx, const int32_t* offsets, const int32_t* perm,
                  const meteora_shape_t& s, float* u, int32_t* status, cudaStream_t st) {
    if (token_shrink_supported(s)) return launch_token_shrink(x, A, topk_idx, s, u, status, false, false, expand_tile_supported(s), st);
    return launch_shrink_segments(x, A, offsets, perm, s, u, st);
}

int launch_shrink_segments(const void* x, const void* A, const int32_t* offsets, const int32_t* perm,
                           const meteora_shape_t& s, float* u, cudaStream_t st) {
    if (s.T == 0) return METEORA_OK;
    const int S = s.T * s.k;
    const int blocks = (S + kSegSlots - 1) / kSegSlots + s.N;  // upper bound of sum_e ceil(count_e / kSegSlots)
    if (s.dtype == METEORA_BF16)
        k_shrink_segments<__nv_bfloat16><<<blocks, kSegWarps * 32, 0, st>>>(
            (const __nv_bfloat16*)x, (const __nv_bfloat16*)A, offsets, perm, s.d_in, s.N, s.r, s.k, u);
    else
        k_shrink_segments<float><<<blocks, kSegWarps * 32, 0, st>>>((const float*)x, (const float*)A, offsets, perm,
                                                                    s.d_in, s.N, s.r, s.k, u);
    return last_launch_status();
}

int launch_expand(const void* B, const int32_t* topk_idx, const float* topk_w, const float* u,
                  const meteora_shape_t& s, float* delta, int32_t* status, cudaStream_t st) {
    if (s.T == 0) return METEORA_OK;
    if (expand_tile_supported(s)) return launch_expand_tile(B, topk_idx, topk_w, u, s, delta, status, st);
    // the staged rows of all adapters for 128 outputs have to fit, next to 8 warps' values of 4 tokens
    const size_t slab_smem = (size_t)s.N * s.r * 256 + (size_t)8 * kSlabTokens * s.k * (s.r + 1) * 4;
    const int r8 = s.r / 8;
    if (s.dtype == METEORA_BF16 && s.r % 8 == 0 && (r8 == 1 || r8 == 2 || r8 == 4 || r8 == 8) && slab_smem <= kSlabSmem) {
        const auto kernel = r8 == 1 ? k_expand_slab<1> : r8 == 2 ? k_expand_slab<2> : r8 == 4 ? k_expand_slab<4> : k_expand_slab<8>;
        static std::atomic<bool> attr_set[64];
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess) return METEORA_ERR_CUDA;
        if (dev < 0 || dev >= 64) return METEORA_ERR_UNSUPPORTED_SHAPE;
        if (!attr_set[dev].load(std::memory_order_relaxed)) {
            for (auto f : {k_expand_slab<1>, k_expand_slab<2>, k_expand_slab<4>, k_expand_slab<8>})
                if (cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSlabSmem) != cudaSuccess) return METEORA_ERR_CUDA;
            attr_set[dev].store(true, std::memory_order_relaxed);
        }
        // one wave: as many shares of the tokens as CTAs fit, a group of 4 tokens per warp at the least
        const int per_sm = std::max(1, std::min(3, (int)(220 * 1024 / (slab_smem + 1024)))), row_blocks = (s.d_out + 127) / 128;
        const int shares = std::max(1, std::min(148 * per_sm / row_blocks, (s.T + 8 * kSlabTokens - 1) / (8 * kSlabTokens)));
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(row_blocks, shares);
        cfg.blockDim = dim3(256);
        cfg.dynamicSmemBytes = slab_smem;
        cfg.stream = st;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = tuning().pdl ? 1 : 0;
        return cuda_status(cudaLaunchKernelEx(&cfg, kernel, (const __nv_bfloat16*)B, topk_idx, topk_w, u, s.T, s.d_out, s.N, s.k, delta));
    }
    dim3 grid((s.T + kExpTokens - 1) / kExpTokens, (s.d_out + kExpThreads - 1) / kExpThreads);
    if (s.dtype == METEORA_BF16)
        k_expand<__nv_bfloat16><<<grid, kExpThreads, 0, st>>>((const __nv_bfloat16*)B, topk_idx, topk_w, u, s.T,
                                                               s.d_out, s.N, s.r, s.k, delta);
    else
        k_expand<float><<<grid, kExpThreads, 0, st>>>((const float*)B, topk_idx, topk_w, u, s.T, s.d_out, s.N, s.r,
                                                       s.k, delta);
    return last_launch_status();
}

}  // namespace meteora
