// The gate's gradient behind the two shrinks (Sec. 3.2): g[t,j] = <u[t,j], z[t,j]> with u = A_e x_t and z = B_e^T dy_t per slot,
// dlogit = w_j (g_j - sum_m w_m g_m) / tau, and dWg = sum over the slots of dlogit[slot] * x[token(slot)] as a
// tensor-core product.  Every CTA works out the dlogit of its own tokens (a few KB of u and z from L2); the first column
// tile's CTAs write it.
// Included by wgemm_tcgen05.cu after the device helpers it uses.
//
// The sum is D[adapter, column] = sum over tokens of L[adapter, token] x[token, column] with L holding k values per
// token.  L would lose precision as bf16, so each dlogit is split into three bf16 parts whose sum has all 24 bits of
// it, and the parts are separate rows of the MMA's M axis: up to 42 adapters make 126 of its 128 rows, so the split
// costs nothing.  x is read as it lies: columns contiguous, i.e. the MN-major form of the B operand.  A CTA takes 256
// columns and a share of the tokens and writes its result; with more than one share a second kernel adds them in
// order, so every run gives the same bits.  Slots of one token that name the same adapter share an element of L: their sum.
// The product multiplies the zeros of L too, and 0 times an infinity or a NaN in x is NaN: a column with a NaN is summed again
// from the slots alone, so that such a token reaches the rows of its own picks only.
//
// Bound by reading x once (16.8 MB at 2048 tokens x 4096) and the latency of building L and of the second launch.
#pragma once

namespace meteora {

constexpr int kDwgCols = 256;                       // columns per CTA: four operand tiles of 64
constexpr int kDwgTok = 64;                         // tokens per stage
constexpr int kDwgXBytes = kDwgTok * kDwgCols * 2;
constexpr int kDwgStages = 4;
constexpr int kDwgLBytes = kBM * kDwgTok * 2;       // L tile: 128 rows x 64 tokens of bf16, K-major, 128-byte swizzle
constexpr int kDwgMaxN = kBM / 3;
constexpr int kDwgSlots = 4096;                     // slots whose dlogit a CTA holds at a time (whole blocks of 64 tokens)
constexpr uint32_t kDwgTaken = 0x7FE0ED0Eu;         // (a NaN that no sum gives) the token's adapter is with an earlier slot
constexpr int kDwgMaxShares = 16;                   // shares of the tokens: bounds the scratch

struct GateDwgParams {
    int T, N, k, d_in;         // (grid: column tiles x shares of the tokens)
    int r;
    float inv_tau;
    const int32_t* topk_idx;
    const float* topk_w;
    const float* u;            // [slot][r]
    const float* z;
    const __nv_bfloat16* x;    // (for the columns that are summed again)
    float* dlogit;             // optional out
    float* out;                // [share][N][d_in]
    int32_t* status;
};

__global__ void __launch_bounds__(kThreads)
k_gate_dwg_tc(const __grid_constant__ CUtensorMap tmX, const GateDwgParams p) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ int s_odd;                               // 1: some result is NaN, 2: a wait has expired
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t ring = (raw + 1023u) & ~1023u;
    uint8_t* ring_ptr = smem_raw + (ring - raw);
    constexpr uint32_t kStage = kDwgXBytes + kDwgLBytes;
    const uint32_t bar_x = ring + kDwgStages * kStage, bar_l = bar_x + kDwgStages * 8, bar_free = bar_l + kDwgStages * 8;
    const uint32_t bar_acc = bar_free + kDwgStages * 8;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(ring_ptr + kDwgStages * kStage + (3 * kDwgStages + 1) * 8);

    const int warp = warp_id(), lane = threadIdx.x & 31;
    const int col0 = blockIdx.x * kDwgCols;
    const int blocks = (p.T + kDwgTok - 1) / kDwgTok;
    const int b0 = (int)((long long)blocks * blockIdx.y / gridDim.y), nb = (int)((long long)blocks * (blockIdx.y + 1) / gridDim.y) - b0;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kDwgStages; ++s) {
            mbar_init(bar_x + s * 8, 1);
            mbar_init(bar_l + s * 8, 1);
            mbar_init(bar_free + s * 8, 1);
        }
        mbar_init(bar_acc, 1);
        s_odd = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(kDwgCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *reinterpret_cast<volatile uint32_t*>(tmem_slot);

    bool acc_ok = true;
    if (warp == 0) {
        {
            bool ok = true;
            for (int i = 0; i < nb; ++i) {
                const int s = i % kDwgStages, round = i / kDwgStages;
                if (round > 0) ok = mbar_wait_warp(bar_free + s * 8, (round & 1) ^ 1);
                if (!ok) break;
                if (elect_one()) {
                    mbar_expect_tx(bar_x + s * 8, kDwgXBytes);
#pragma unroll
                    for (int c = 0; c < kDwgCols / 64; ++c)              // (columns beyond d_in and tokens beyond T read as zero)
                        tma_load_2d(ring + s * kStage + c * (kDwgTok * 128), &tmX, col0 + c * 64, (b0 + i) * kDwgTok, bar_x + s * 8);
                }
                __syncwarp();
            }
            if (!ok && lane == 0) {
                atomicExch(p.status, 1);
                atomicExch(p.status + 1, 4100);
            }
        }
    } else if (warp == 1) {
        {
            // A = L (K-major), B = x (MN-major: instruction descriptor bit 16), N = 64 columns
            const uint32_t idesc = instr_desc_bf16(64) | (1u << 16);
            bool ok = true;
            for (int i = 0; i < nb; ++i) {
                const int s = i % kDwgStages, round = i / kDwgStages;
                ok = mbar_wait_warp(bar_x + s * 8, round & 1) && mbar_wait_warp(bar_l + s * 8, round & 1);
                if (!ok) break;
                tc_fence_after();
                const uint32_t xa = ring + s * kStage, la = xa + kDwgXBytes;
                const uint64_t da = smem_desc_sw128(la);
                if (elect_one()) {
#pragma unroll
                    for (int kk = 0; kk < kDwgTok / kUmmaK; ++kk)
#pragma unroll
                        for (int c = 0; c < kDwgCols / 64; ++c) {
                            // 16 tokens = two groups of 8 rows of 128 bytes, 1024 bytes apart
                            const uint64_t db = (smem_desc_sw128(xa + c * (kDwgTok * 128) + kk * 2048) & ~((uint64_t)0x3FFF << 16)) |
                                                ((uint64_t)(1024 >> 4) << 16);
                            umma_bf16(tmem_base + c * 64, da + (uint64_t)(kk * 2), db, idesc, (i | kk) != 0);
                        }
                    umma_commit(bar_free + s * 8);
                }
                __syncwarp();
            }
            if (elect_one()) umma_commit(bar_acc);
            __syncwarp();
            if (!ok && lane == 0) {
                atomicExch(p.status, 1);
                atomicExch(p.status + 2, 4200);
            }
        }
    } else {
        const int etid = threadIdx.x - 64;
        asm volatile("griddepcontrol.wait;" ::: "memory");           // u and z come from the grids before (x and the routing do not)
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        bool ok = true;
        float* s_g = reinterpret_cast<float*>(ring_ptr + kDwgStages * kStage + 256);
        float* s_dl = s_g + kDwgSlots;
        const int chunk = kDwgSlots / (kDwgTok * p.k);               // blocks per pass over u and z (k <= 8: 8 at the least)
        auto dlogits = [&](int i) {                                  // of the chunk whose first block is i, to s_dl
            const size_t s0 = (size_t)(b0 + i) * kDwgTok * p.k;
            const int slots = min(min(chunk, nb - i) * kDwgTok, p.T - (b0 + i) * kDwgTok) * p.k;
            for (int q = etid; q < slots; q += kEpiThreads) {
                const float4 *up = reinterpret_cast<const float4*>(p.u + (s0 + q) * p.r), *zp = reinterpret_cast<const float4*>(p.z + (s0 + q) * p.r);
                float g = 0.f;
#pragma unroll 2
                for (int c = 0; c < p.r / 4; ++c) {
                    const float4 a = up[c], b = zp[c];
                    g = fmaf(a.x, b.x, fmaf(a.y, b.y, fmaf(a.z, b.z, fmaf(a.w, b.w, g))));
                }
                s_g[q] = g;
            }
            __syncwarp();
            epi_barrier();
            for (int q = etid; q < slots; q += kEpiThreads) {
                const int first = q / p.k * p.k, e = min(max(p.topk_idx[s0 + q], 0), p.N - 1);
                uint32_t same = 0;                                   // picks of the token that name this slot's adapter
                float mean = 0.f;
                for (int m = 0; m < p.k; ++m) {
                    mean = fmaf(p.topk_w[s0 + first + m], s_g[first + m], mean);
                    if (min(max(p.topk_idx[s0 + first + m], 0), p.N - 1) == e) same |= 1u << m;
                }
                const float v = p.topk_w[s0 + q] * (s_g[q] - mean) * p.inv_tau;
                if (p.dlogit && blockIdx.x == 0) p.dlogit[s0 + q] = v;
                float sum = v;
                if (same & (same - 1u)) {                            // more than one: the first has their sum
                    sum = 0.f;
                    for (int m = 0; m < p.k; ++m)
                        if (same >> m & 1u) sum += p.topk_w[s0 + first + m] * (s_g[first + m] - mean) * p.inv_tau;
                    if (same & ((1u << (q - first)) - 1u)) sum = __uint_as_float(kDwgTaken);
                }
                s_dl[q] = sum;
            }
            __syncwarp();
            epi_barrier();
        };
        for (int i = 0; i < nb; ++i) {
            if (i % chunk == 0) dlogits(i);
            const int s = i % kDwgStages, round = i / kDwgStages;
            if (round > 0) ok = ok && mbar_wait(bar_free + s * 8, (round & 1) ^ 1);
            uint8_t* L = ring_ptr + s * kStage + kDwgXBytes;
#pragma unroll
            for (int v = 0; v < kDwgLBytes / 16; v += kEpiThreads) reinterpret_cast<uint4*>(L)[v + etid] = make_uint4(0u, 0u, 0u, 0u);
            const int t0 = (b0 + i) * kDwgTok, slots = min(kDwgTok, p.T - t0) * p.k;
            int e_i[2];                                              // (k <= 8: two slots per thread)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int q = etid + h * kEpiThreads;
                e_i[h] = q < slots ? min(max(p.topk_idx[(size_t)t0 * p.k + q], 0), p.N - 1) : -1;
            }
            epi_barrier();
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (e_i[h] < 0) continue;
                const int q = etid + h * kEpiThreads, tok = q / p.k;
                float v = s_dl[(i % chunk) * kDwgTok * p.k + q];
                if (__float_as_uint(v) == kDwgTaken) continue;
#pragma unroll
                for (int part = 0; part < 3; ++part) {
                    const __nv_bfloat16 b = __float2bfloat16_rn(v);
                    v -= __bfloat162float(b);
                    const int row = part * p.N + e_i[h];
                    *reinterpret_cast<__nv_bfloat16*>(L + row * 128 + (((tok >> 3) ^ (row & 7)) << 4) + (tok & 7) * 2) = b;
                }
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic writes -> tensor-core reads
            __syncwarp();
            epi_barrier();
            if (etid == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar_l + s * 8) : "memory");
        }
        acc_ok = mbar_wait(bar_acc, 0) && ok;
        if (!acc_ok && lane == 0) {
            atomicExch(p.status, 1);
            atomicExch(p.status + 3, 4300);
        }
        acc_ok = __all_sync(0xFFFFFFFFu, acc_ok);
        tc_fence_after();
        // accumulator rows (part, adapter) to shared memory, [column][row] (the stages are idle); then a thread per column adds
        // the three parts of every adapter and writes them, 1 KB per adapter and CTA
        float* acc = reinterpret_cast<float*>(ring_ptr);
        constexpr int pitch = kBM + 1;
        const int quad = warp & 3, row = quad * 32 + lane;
        const int c_begin = warp < 6 ? 0 : kDwgCols / 2;
        for (int c0 = c_begin; c0 < c_begin + kDwgCols / 2; c0 += 16) {
            float v[16];
            if (acc_ok && nb > 0) {
                tmem_ld16(tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)c0, v);
            } else {
#pragma unroll
                for (int i = 0; i < 16; ++i) v[i] = nb > 0 ? CUDART_NAN_F : 0.f;   // an expired wait must not pass for a result
            }
#pragma unroll
            for (int i = 0; i < 16; ++i) acc[(c0 + i) * pitch + row] = v[i];
        }
        if (!acc_ok && lane == 0) atomicOr(&s_odd, 2);
        __syncwarp();
        epi_barrier();
        float* a = acc + etid * pitch;
        float* dst = p.out + (size_t)blockIdx.y * p.N * p.d_in + col0 + etid;
        bool nan = false;
        if (col0 + etid < p.d_in) {
#pragma unroll 4
            for (int e = 0; e < p.N; ++e) {
                const float v = a[e] + (a[p.N + e] + a[2 * p.N + e]);
                nan |= v != v;
                dst[(size_t)e * p.d_in] = v;
            }
        }
        if (nan) atomicOr(&s_odd, 1);
        __syncwarp();
        epi_barrier();
        if (s_odd == 1) {                                            // (with an expired wait the NaNs stay)
            for (int e = 0; e < p.N; ++e) a[e] = 0.f;                // this thread's column
            for (int i = 0; i < nb; i += chunk) {
                dlogits(i);
                const int t0 = (b0 + i) * kDwgTok, slots = min(min(chunk, nb - i) * kDwgTok, p.T - t0) * p.k;
                for (int q = 0; nan && q < slots; ++q) {
                    const int e = min(max(p.topk_idx[(size_t)t0 * p.k + q], 0), p.N - 1);
                    if (__float_as_uint(s_dl[q]) != kDwgTaken) a[e] = fmaf(s_dl[q], to_f32(p.x[(size_t)(t0 + q / p.k) * p.d_in + col0 + etid]), a[e]);
                }
                __syncwarp();
                epi_barrier();                                       // s_dl is read before the next chunk's is written
            }
            for (int e = 0; nan && e < p.N; ++e) dst[(size_t)e * p.d_in] = a[e];
        }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kDwgCols) : "memory");
}

// dWg[i] = sum of the shares' partial sums in order.
__global__ void __launch_bounds__(256)
k_gate_dwg_sum(const float* __restrict__ part, int shares, size_t n, float* __restrict__ dWg) {
    const size_t i = ((size_t)blockIdx.x * 256 + threadIdx.x);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (i >= n) return;
    float v[kDwgMaxShares], sum = 0.f;
#pragma unroll
    for (int q = 0; q < kDwgMaxShares; ++q) v[q] = q < shares ? part[q * n + i] : 0.f;
#pragma unroll
    for (int q = 0; q < kDwgMaxShares; ++q) sum += v[q];
    dWg[i] = sum;
}

}  // namespace meteora
