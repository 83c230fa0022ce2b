// Plain CUDA-core path of the layer (Eq. 2 with Eq. 3): fp32 layers (the tensor cores would round fp32 inputs to tf32)
// and every shape the TMA/tcgen05 path does not take.  fp32 FMA throughout, one rounding of y.  Two launches:
//   k_simt_partial  every product that reads x in ONE pass: the rows of W0, of all A_i and of Wg are one stacked matrix,
//                   cut into tiles and slices of the contraction axis; slice z writes its own fp32 copy of the result;
//   k_simt_finish   adds the slices in order, selects and weighs (Eq. 3), expands (Eq. 2), rounds once and stores y.
//
// What bounds it: large problems instruction issue (12 warps per SM, packed FMAs), small ones the chain of launches and load
// latencies, so a small problem is cut along the contraction axis until its tiles fill the SMs.  Measured per call (graph replay; before: a gate
// kernel, a shrink kernel and a 64 x 64 GEMM with scalar loads and the whole axis per CTA): 256 -> 256, 4 adapters, 64
// tokens 77 -> 7.9 us; 2048 -> 2048, 28 adapters: one token 258 -> 15.6 us, 512 tokens 495 -> 132 us (42 TFLOP/s of the
// first launch, of 74 that the FMA pipes hold).
#include "common.cuh"
#include "select.cuh"

#include <algorithm>
#include <cmath>

namespace meteora {

constexpr int kSimtK = 16;              // contraction elements per staged chunk
constexpr int kSimtMaxSlices = 16;      // what the selection reads in one round trip

__device__ __forceinline__ void store_out(float* p, float v) { *p = v; }
__device__ __forceinline__ void store_out(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }

// Elements d .. d + 3 of a row (nullptr: a padding row), zero beyond n.  `vec`: rows are 4-element aligned and n % 4 == 0.
__device__ __forceinline__ float4 load_quad(const float* row, int d, int n, bool vec) {
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (!row || d >= n) return v;
    if (vec) return __ldg(reinterpret_cast<const float4*>(row + d));
    v.x = row[d];
    if (d + 1 < n) v.y = row[d + 1];
    if (d + 2 < n) v.z = row[d + 2];
    if (d + 3 < n) v.w = row[d + 3];
    return v;
}
__device__ __forceinline__ float4 load_quad(const __nv_bfloat16* row, int d, int n, bool vec) {
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (!row || d >= n) return v;
    if (vec) {
        const uint2 q = __ldg(reinterpret_cast<const uint2*>(row + d));
        return make_float4(__uint_as_float(q.x << 16), __uint_as_float(q.x & 0xFFFF0000u), __uint_as_float(q.y << 16),
                           __uint_as_float(q.y & 0xFFFF0000u));
    }
    v.x = to_f32(row[d]);
    if (d + 1 < n) v.y = to_f32(row[d + 1]);
    if (d + 2 < n) v.z = to_f32(row[d + 2]);
    if (d + 3 < n) v.w = to_f32(row[d + 3]);
    return v;
}

struct SimtParams {
    int T, d_in, d_out, a_rows, N, ldp;   // stacked rows: d_out of W0, a_rows = N * r of A, N of Wg; ldp = row pitch of a copy
    size_t zstride;                       // floats between the copies
    float* part;                          // part[z][t][row]
};

// A CTA multiplies BM stacked rows with BN tokens over its slice of the contraction axis; a thread owns TM rows x TN tokens
// (rows in groups of 4, the groups BM / (TM / 4) apart, so that a warp's 16-byte reads of the staged rows touch
// different banks).  Chunks of 16 elements are double-buffered: the next chunk's loads are in registers while this one
// is multiplied.
template <typename TI, int BM, int BN, int TM, int TN>
__global__ void __launch_bounds__((BM / TM) * (BN / TN))
k_simt_partial(const TI* __restrict__ x, const TI* __restrict__ W0, const TI* __restrict__ A, const TI* __restrict__ Wg,
               const SimtParams p) {
    constexpr int NT = (BM / TM) * (BN / TN), TX = BM / TM, G = TM / 4;
    constexpr int QW = (BM * 4 + NT - 1) / NT, QX = (BN * 4 + NT - 1) / NT;   // 4-element loads per thread and chunk
    __shared__ __align__(16) float sw[2][kSimtK][BM + 4];
    __shared__ __align__(16) float sx[2][kSimtK][BN + 4];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // k_simt_finish waits for this grid before it reads
    const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
    const int row0 = blockIdx.y * BM, tok0 = blockIdx.x * BN;
    const int rows = p.d_out + p.a_rows + p.N;
    const bool vec = p.d_in % 4 == 0;
    const int chunks = (p.d_in + kSimtK - 1) / kSimtK;
    const int c0 = (int)((long long)chunks * blockIdx.z / gridDim.z), c1 = (int)((long long)chunks * (blockIdx.z + 1) / gridDim.z);
    const int kq = (tid % 4) * 4;                                   // this thread's 4 elements of a chunk
    const TI *wrow[QW], *xrow[QX];
#pragma unroll
    for (int i = 0; i < QW; ++i) {
        const int r = tid / 4 + i * (NT / 4), R = row0 + r;
        wrow[i] = r >= BM || R >= rows ? nullptr
                  : R < p.d_out ? W0 + (size_t)R * p.d_in
                  : R < p.d_out + p.a_rows ? A + (size_t)(R - p.d_out) * p.d_in
                                           : Wg + (size_t)(R - p.d_out - p.a_rows) * p.d_in;
    }
#pragma unroll
    for (int i = 0; i < QX; ++i) {
        const int r = tid / 4 + i * (NT / 4);
        xrow[i] = r >= BN || tok0 + r >= p.T ? nullptr : x + (size_t)(tok0 + r) * p.d_in;
    }
    float4 wq[QW], xq[QX];
    auto fetch = [&](int c) {
#pragma unroll
        for (int i = 0; i < QW; ++i) wq[i] = load_quad(wrow[i], c * kSimtK + kq, p.d_in, vec);
#pragma unroll
        for (int i = 0; i < QX; ++i) xq[i] = load_quad(xrow[i], c * kSimtK + kq, p.d_in, vec);
    };
    auto stage = [&](int b) {
#pragma unroll
        for (int i = 0; i < QW; ++i) {
            const int r = tid / 4 + i * (NT / 4);
            if (BM % (NT / 4) == 0 || r < BM) {
                sw[b][kq][r] = wq[i].x;
                sw[b][kq + 1][r] = wq[i].y;
                sw[b][kq + 2][r] = wq[i].z;
                sw[b][kq + 3][r] = wq[i].w;
            }
        }
#pragma unroll
        for (int i = 0; i < QX; ++i) {
            const int r = tid / 4 + i * (NT / 4);
            if (BN % (NT / 4) == 0 || r < BN) {
                sx[b][kq][r] = xq[i].x;
                sx[b][kq + 1][r] = xq[i].y;
                sx[b][kq + 2][r] = xq[i].z;
                sx[b][kq + 3][r] = xq[i].w;
            }
        }
    };
    unsigned long long acc[TM / 2][TN];
#pragma unroll
    for (int i = 0; i < TM / 2; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = 0ull;
    if (c0 < c1) {
        fetch(c0);
        stage(0);
    }
    __syncthreads();
    for (int c = c0; c < c1; ++c) {
        const int b = (c - c0) & 1;
        if (c + 1 < c1) fetch(c + 1);
#pragma unroll
        for (int kk = 0; kk < kSimtK; ++kk) {
            unsigned long long wv[TM / 2], xv[TN];
#pragma unroll
            for (int g = 0; g < G; ++g) {
                const ulonglong2 q = *reinterpret_cast<const ulonglong2*>(&sw[b][kk][g * (BM / G) + tx * 4]);
                wv[2 * g] = q.x;
                wv[2 * g + 1] = q.y;
            }
            float xs[TN];
            if (TN % 4 == 0) {
#pragma unroll
                for (int j = 0; j < TN; j += 4) *reinterpret_cast<float4*>(xs + j) = *reinterpret_cast<const float4*>(&sx[b][kk][ty * TN + j]);
            } else {
#pragma unroll
                for (int j = 0; j < TN; j += 2) *reinterpret_cast<float2*>(xs + j) = *reinterpret_cast<const float2*>(&sx[b][kk][ty * TN + j]);
            }
#pragma unroll
            for (int j = 0; j < TN; ++j) xv[j] = twice(xs[j]);
#pragma unroll
            for (int i = 0; i < TM / 2; ++i)
#pragma unroll
                for (int j = 0; j < TN; ++j) fma2(acc[i][j], wv[i], xv[j]);
        }
        if (c + 1 < c1) stage(b ^ 1);
        __syncthreads();
    }
    float* out = p.part + (size_t)blockIdx.z * p.zstride;
#pragma unroll
    for (int j = 0; j < TN; ++j) {
        const int t = tok0 + ty * TN + j;
        if (t >= p.T) continue;
#pragma unroll
        for (int g = 0; g < G; ++g) {
            const int R = row0 + g * (BM / G) + tx * 4;             // the pitch is a multiple of 4: whole quads or nothing
            ulonglong2 q;
            q.x = acc[2 * g][j];
            q.y = acc[2 * g + 1][j];
            if (R < p.ldp) *reinterpret_cast<ulonglong2*>(out + (size_t)t * p.ldp + R) = q;
        }
    }
}

// A CTA finishes TT tokens x 256 outputs: the slices of its outputs are requested first, a warp per token selects
// from the summed logits while they arrive (each CTA of a token repeats that: it is cheaper than a third launch), then
// each thread expands its output.  Bound by round trips to L2 (slices, logits, the picks' shrink, the picks' rows of B),
// so the loads of all TT tokens of a step go out together.
template <typename TI, int TT>
__global__ void __launch_bounds__(256)
k_simt_finish(const TI* __restrict__ B, const SimtParams p, int zsplits, int r, int k, float inv_tau, TI* __restrict__ y,
              int32_t* __restrict__ topk_idx, float* __restrict__ topk_w) {
    __shared__ int32_t s_idx[TT * METEORA_MAX_K];
    __shared__ float s_w[TT * METEORA_MAX_K];
    __shared__ __align__(16) float s_uw[TT * METEORA_MAX_K * METEORA_MAX_R];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int t0 = blockIdx.x * TT, nt = min(TT, p.T - t0);
    const int o = blockIdx.y * 256 + threadIdx.x;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    float acc[TT];
#pragma unroll
    for (int tt = 0; tt < TT; ++tt) acc[tt] = 0.f;
    if (o < p.d_out) {
#pragma unroll 4
        for (int z = 0; z < zsplits; ++z) {
            const float* src = p.part + (size_t)z * p.zstride + (size_t)t0 * p.ldp + o;
#pragma unroll
            for (int tt = 0; tt < TT; ++tt) acc[tt] += src[(size_t)min(tt, nt - 1) * p.ldp];
        }
    }
    if (warp < nt)
        select_token_few<false, kSimtMaxSlices>(p.part + (size_t)(t0 + warp) * p.ldp + p.d_out, p.a_rows, zsplits, p.zstride, warp,
                                                p.N, r, k, inv_tau, lane, s_idx, s_w, s_uw);
    __syncthreads();
    if (blockIdx.y == 0 && threadIdx.x < nt * k) {
        topk_idx[(size_t)t0 * k + threadIdx.x] = s_idx[threadIdx.x];
        topk_w[(size_t)t0 * k + threadIdx.x] = s_w[threadIdx.x];
    }
    if (o >= p.d_out) return;
    const bool vec = r % 4 == 0;
    float lora[TT];
#pragma unroll
    for (int tt = 0; tt < TT; ++tt) lora[tt] = 0.f;
    const int quads = (r + 3) / 4, steps = k * quads;               // (pick, 4 rank entries)
#pragma unroll 2
    for (int i = 0; i < steps; ++i) {
        const int j = i / quads, q = (i - j * quads) * 4;
#pragma unroll
        for (int tt = 0; tt < TT; ++tt) {
            const int slot = min(tt, nt - 1) * k + j;
            const float4 b = load_quad(B + ((size_t)s_idx[slot] * p.d_out + o) * r, q, r, vec);
            const float* uq = s_uw + slot * r + q;
            lora[tt] = fmaf(b.x, uq[0], lora[tt]);
            if (q + 1 < r) lora[tt] = fmaf(b.y, uq[1], lora[tt]);
            if (q + 2 < r) lora[tt] = fmaf(b.z, uq[2], lora[tt]);
            if (q + 3 < r) lora[tt] = fmaf(b.w, uq[3], lora[tt]);
        }
    }
#pragma unroll
    for (int tt = 0; tt < TT; ++tt)
        if (tt < nt) store_out(&y[(size_t)(t0 + tt) * p.d_out + o], acc[tt] + lora[tt]);
}

// Tile of the first launch and how often the contraction axis is cut.  Few tokens: 64 rows x 16 tokens (the weights are
// what is read); else 128 x 64 (fewer shared-memory reads per FMA: 114 against 131 us at 2048 -> 2048, 512 tokens) where
// those tiles, cut into slices of 128 elements, fill the SMs, and 64 x 64 below that.  Slices until there are three CTAs
// per SM (2048 -> 2048, partial products at 1 / 512 tokens with one, two, three, four CTAs per SM: 17.6 / 12.5 / 11.2 / 10.5
// and 142 / 120 / 114 / 114 us), each of two chunks at the least, and no more than 8 of a short axis: the second launch
// adds them (512 -> 2000, 33 tokens: 11.4 us with 8, 13.0 with 13).
// A large batch goes in blocks of tokens that share the scratch of one (a copy for all of 8192 tokens x 14336 outputs would be 478
// MB): up to 128 MB and at least two waves of three CTAs per SM, the block whose last wave is fullest.  There is one slice then,
// so the sums are the same.
struct SimtPlan {
    int bm, bn, z, ldp, tokens;                                     // tokens per block
};
static SimtPlan simt_plan(const meteora_shape_t& s) {
    SimtPlan sp;
    const int rows = s.d_out + s.N * s.r + s.N;
    auto tiles = [&](int bm, int bn) { return (long long)((rows + bm - 1) / bm) * ((s.T + bn - 1) / bn); };
    sp.bn = s.T <= 16 ? 16 : 64;
    sp.bm = s.T > 16 && tiles(128, 64) * std::max(1, s.d_in / 128) >= 148 ? 128 : 64;
    const int chunks = (s.d_in + kSimtK - 1) / kSimtK;
    const int cap = std::min(std::min(kSimtMaxSlices, chunks / 2), std::max(8, chunks / 8));
    sp.z = (int)std::max<long long>(1, std::min<long long>(cap, 444 / tiles(sp.bm, sp.bn)));
    sp.ldp = (int)align_up((size_t)rows, 4);
    sp.tokens = s.T;
    const long long row_tiles = (rows + sp.bm - 1) / sp.bm, least = (888 + row_tiles - 1) / row_tiles;
    const long long most = std::max(least, ((long long)128 << 20) / (4LL * sp.ldp) / 64);   // tiles of 64 tokens
    if (s.T > 64 * most) {
        double fullest = 0.0;
        for (long long n = least; n <= std::min(most, least + 64); ++n) {
            const double waves = (double)(row_tiles * n) / 444, full = waves / std::ceil(waves);
            if (full >= fullest) {
                fullest = full;
                sp.tokens = (int)(64 * n);
            }
        }
    }
    return sp;
}

size_t simt_part_floats(const meteora_shape_t& s) {
    const SimtPlan sp = simt_plan(s);
    return (size_t)sp.z * sp.tokens * sp.ldp;
}

// Tokens [t0, t0 + n) of the batch.
template <typename TI>
static int launch_simt_block(const SimtPlan& sp, const TI* x, const TI* W0, const TI* A, const TI* B, const TI* Wg, const meteora_shape_t& s,
                             const Workspace& ws, TI* y, int t0, int n, cudaStream_t st) {
    SimtParams p = {};
    p.T = n;
    p.d_in = s.d_in;
    p.d_out = s.d_out;
    p.a_rows = s.N * s.r;
    p.N = s.N;
    p.ldp = sp.ldp;
    p.zstride = (size_t)n * sp.ldp;
    p.part = ws.simt_part;
    x += (size_t)t0 * s.d_in;
    const dim3 grid((n + sp.bn - 1) / sp.bn, (s.d_out + p.a_rows + s.N + sp.bm - 1) / sp.bm, sp.z);
    // (no dependent launch: the block before has been finished when this one's products overwrite the scratch)
    if (sp.bn == 16)
        k_simt_partial<TI, 64, 16, 4, 2><<<grid, 128, 0, st>>>(x, W0, A, Wg, p);
    else if (sp.bm == 64)
        k_simt_partial<TI, 64, 64, 8, 4><<<grid, 128, 0, st>>>(x, W0, A, Wg, p);
    else
        k_simt_partial<TI, 128, 64, 8, 8><<<grid, 128, 0, st>>>(x, W0, A, Wg, p);
    const int rc = last_launch_status();
    if (rc != METEORA_OK) return rc;
    cudaLaunchConfig_t cfg = {};
    // one token per CTA while that leaves at most four CTAs of 256 threads per SM, else four
    const int row_blocks = (s.d_out + 255) / 256;
    const bool one = (long long)n * row_blocks <= 592;
    cfg.gridDim = dim3(one ? n : (n + 3) / 4, row_blocks);
    cfg.blockDim = dim3(256);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = tuning().pdl ? 1 : 0;
    return cuda_status(cudaLaunchKernelEx(&cfg, one ? k_simt_finish<TI, 1> : k_simt_finish<TI, 4>, B, (const SimtParams)p, sp.z, s.r, s.k,
                                          1.0f / s.temperature, y + (size_t)t0 * s.d_out, ws.topk_idx + (size_t)t0 * s.k,
                                          ws.topk_w + (size_t)t0 * s.k));
}

template <typename TI>
static int launch_simt(const void* x, const void* W0, const void* A, const void* B, const void* Wg, const meteora_shape_t& s,
                       const Workspace& ws, void* y, cudaStream_t st) {
    const SimtPlan sp = simt_plan(s);
    int rc = METEORA_OK;
    for (int t0 = 0; t0 < s.T && rc == METEORA_OK; t0 += sp.tokens)
        rc = launch_simt_block<TI>(sp, (const TI*)x, (const TI*)W0, (const TI*)A, (const TI*)B, (const TI*)Wg, s, ws, (TI*)y, t0,
                                   std::min(sp.tokens, s.T - t0), st);
    return rc;
}

int launch_forward_simt(const void* x, const void* W0, const void* A, const void* B, const void* Wg, const meteora_shape_t& s,
                        const Workspace& ws, void* y, cudaStream_t st) {
    if (s.T == 0) return METEORA_OK;
    if (s.dtype == METEORA_BF16) return launch_simt<__nv_bfloat16>(x, W0, A, B, Wg, s, ws, y, st);
    return launch_simt<float>(x, W0, A, B, Wg, s, ws, y, st);
}

}  // namespace meteora
