// Everything the layer derives from a token through the adapters and the gate, for tiles of 128 TOKENS on the MMA's M
// axis: gate logits, top-k and softmax (Eq. 3), and the picks' shrink A_i x (Eq. 2).
// Included by wgemm_tcgen05.cu after the device helpers it uses.
//
// Tokens on M (128 TMEM lanes) and the rows of [Wg; A_0..A_{N-1}] on N (TMEM columns): one pass over x gives every
// logit and every A_i x of a tile.  A cluster of S CTAs shares a tile, each over its slice of the contraction axis; the
// partial accumulators go to the CTAs' own shared memory and the CTA that owns a token reads that token's few values
// (N logits, then the k r shrink values of its picks) from all S of them through distributed shared memory.  Nothing but
// the results reaches global memory: the stacked kernels this replaces wrote every slice's fp32 [T][N r + N] copy
// (19 MB at 2048 tokens, rank 8, 28 adapters) for a second kernel to add.
//
//   mode        product                 per token
//   GATE        [Wg] x                  top-k, softmax (standalone gate)
//   FORWARD     [Wg; A] x               top-k, softmax, uw = w_j (A_j x)
//   SHRINK      [A] x, picks given      u = A_j x (also B_j^T dy of the gate's gradient)
//
// What bounds it: the intake of the tiles (48 KB per 64-element k-step and CTA at 252 rows) and, around it, set-up and
// two cluster exchanges of about a microsecond each; so S is as large as the SMs allow.
#pragma once

namespace meteora {

enum { TOKEN_GATE = 0, TOKEN_FORWARD = 1, TOKEN_SHRINK = 2 };
constexpr int kTokTile = 128;               // tokens per tile (UMMA M)
constexpr int kTokXBytes = kTokTile * 128;  // token operand of one k-step
constexpr int kTokCols = 256;               // accumulator columns per round (UMMA N at the most)
constexpr int kTokMaxSplit = 16;            // CTAs per tile: 1 - 8 or 16

struct TokenTileParams {
    int T, mode, N, r, k;
    int ksteps;
    int gate_box, a_box, a_copies;   // rows per copy: Wg (N rounded up to 8; 0: none), A (a_copies copies of a_box rows)
    int a_group;               // adapters per grid row (SHRINK: the adapters may be dealt to several clusters per tile)
    int stages, stage_bytes, tmem_cols, pitch;   // pitch: floats per token of the shared-memory copy of a round
    int rounds, cols[2];       // accumulators of up to 256 columns
    int acc2;                  // DUAL: first column of the second one
    float inv_tau;
    int32_t* topk_idx;         // out (GATE, FORWARD) or in
    float* topk_w;             // (not read by SHRINK)
    float* logits;             // GATE: optional out
    float* u;                  // out: [slot][r], FORWARD weighted by w
    __nv_bfloat16* us;         // FORWARD, optional out: the same values as [T][us_parts][us_cols] with zeros elsewhere
    int us_cols, us_parts;
    int32_t* status;           // error flag of expired waits (may be null)
    int clear_status;          // CTA 0 zeroes the status words first
    int late_wait;             // nothing here depends on the kernel ahead: only leave after it
};

__device__ __forceinline__ float ld_cluster_f32(uint32_t cluster_addr) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(cluster_addr));
    return v;
}

// Sum over the cluster's CTAs, in rank order, of the float at this offset of their shared memory.
template <int S>
__device__ __forceinline__ float cluster_sum(const uint32_t (&base)[S], uint32_t off) {
    float part[S], sum = 0.f;
#pragma unroll
    for (int q = 0; q < S; ++q) part[q] = ld_cluster_f32(base[q] + off);
#pragma unroll
    for (int q = 0; q < S; ++q) sum += part[q];
    return sum;
}

// One round's part of the tokens this CTA owns, in passes over (token, value) elements spread over all epilogue threads, so
// that every exchange through distributed shared memory has all its reads in flight at once; the selection, from local
// shared memory then, is a warp per token.  (A warp per token for all of it, token after token, was a chain of 2.5 us per
// token: two reads through the cluster around the top-k.)
template <int S>
__device__ __forceinline__ void token_round(const TokenTileParams& p, uint32_t part, float* s_logits, int round, int rank, int tok0,
                                            int etid, bool valid) {
    uint32_t base[S];
#pragma unroll
    for (int q = 0; q < S; ++q) base[q] = map_to_cta(part, q);
    const int own0 = kTokTile * rank / S, own = min(kTokTile * (rank + 1) / S, p.T - tok0) - own0;   // (may be <= 0)
    const int t0 = tok0 + own0, n = p.k * p.r;
    const uint32_t pitch4 = (uint32_t)p.pitch * 4u;
    if (p.mode <= TOKEN_FORWARD && round == 0) {
        const int ld = p.N | 1;
        if (p.us) {
            const int ld_us = p.us_cols * p.us_parts;
            uint4* rows = reinterpret_cast<uint4*>(p.us + (size_t)t0 * ld_us);
            for (int i = etid; i < own * (ld_us / 8); i += kEpiThreads) rows[i] = make_uint4(0u, 0u, 0u, 0u);
        }
#pragma unroll 2
        for (int i = etid; i < own * p.N; i += kEpiThreads) {
            const int tt = i / p.N, c = i - tt * p.N;
            const float v = cluster_sum<S>(base, (uint32_t)(own0 + tt) * pitch4 + 4u * c);
            s_logits[tt * ld + c] = v;
            if (p.logits) p.logits[(size_t)t0 * p.N + i] = v;
        }
        __syncwarp();
        epi_barrier();
        const int lane = etid & 31;
        for (int tt = etid >> 5; tt < own; tt += kEpiThreads / 32) {
            float v[kSelVals], w;
            int idx;
#pragma unroll
            for (int i = 0; i < kSelVals; ++i) v[i] = lane + 32 * i < p.N ? s_logits[tt * ld + lane + 32 * i] : 0.f;
            warp_topk_softmax(v, p.N, p.k, p.inv_tau, lane, idx, w);
            if (lane < p.k) {
                p.topk_idx[(size_t)(t0 + tt) * p.k + lane] = idx;
                // an expired wait must not pass for a result
                p.topk_w[(size_t)(t0 + tt) * p.k + lane] = valid ? w : CUDART_NAN_F;
            }
        }
        if (p.mode == TOKEN_GATE) return;
        __syncwarp();
        epi_barrier();                                                // (the picks are read back below by other threads)
    }
    // the picks' shrink values whose columns are in this round
    const int c_lo = round * kTokCols, c_hi = c_lo + p.cols[round], e0 = (int)blockIdx.y * p.a_group;
#pragma unroll 2
    for (int i = etid; i < own * n; i += kEpiThreads) {
        const int slot = i / p.r, q = i - slot * p.r;
        const size_t g = (size_t)t0 * p.k + slot;
        const int e = min(max(p.topk_idx[g], 0), p.N - 1) - e0, col = p.gate_box + e * p.r + q;
        if (e >= 0 && e < p.a_group && col >= c_lo && col < c_hi) {
            const float v = cluster_sum<S>(base, (uint32_t)(own0 + slot / p.k) * pitch4 + 4u * (col - c_lo));
            p.u[(size_t)t0 * n + i] = p.mode == TOKEN_FORWARD ? p.topk_w[g] * v : v;
        }
    }
    // (a loop of its own, from what this thread has just written: in the loop above its stores hold back the next value's loads, and
    // the kernel is short enough that the size of its code shows: 4096 -> 1024 at 512 tokens 18.2 -> 18.5 - 19.3 us for the call)
    if (p.us) {
#pragma unroll 1
        for (int i = etid; i < own * n; i += kEpiThreads) {
            const int slot = i / p.r;
            store_us(p.us + (size_t)(t0 + slot / p.k) * p.us_cols * p.us_parts, p.topk_idx[(size_t)t0 * p.k + slot] * p.r + i - slot * p.r, p.us_cols,
                     p.us_parts, p.u[(size_t)t0 * n + i]);
        }
    }
}

// S: CTAs of the cluster that shares a tile.  DUAL (one round of columns): the MMAs go to two accumulators in turn, added in fp32.
// The tensor cores cut what they add to an accumulator off instead of rounding it, so an error grows with the steps into one: LoRA
// term over 4096 products 7.0e-7 with one, 4.3e-7 with two.  (A kernel of its own: as a branch it took 0.3 us where it was not used)
template <int S, bool DUAL>
__global__ void __launch_bounds__(kThreads)
k_token_tile(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmG, const __grid_constant__ CUtensorMap tmA,
             const TokenTileParams p) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t ring = (raw + 1023u) & ~1023u;
    // barriers first: full[stages], empty[stages], acc; then the ring
    const uint32_t bar_base = ring, bar_acc = bar_base + 2 * p.stages * 8;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem_raw + (ring - raw) + (2 * p.stages + 1) * 8);
    const uint32_t data = ring + 1024u;

    const int warp = warp_id(), lane = threadIdx.x & 31;
    const int rank = __shfl_sync(0xFFFFFFFFu, (int)cluster_rank(), 0);
    const int tok0 = (blockIdx.x / S) * kTokTile;
    const int a_row0 = (int)blockIdx.y * p.a_group * p.r;
    const int k0 = p.ksteps * rank / S, niter = p.ksteps * (rank + 1) / S - k0;

    if (threadIdx.x == 0) {
        for (int s = 0; s < 2 * p.stages + 1; ++s) mbar_init(bar_base + s * 8, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"((uint32_t)p.tmem_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *reinterpret_cast<volatile uint32_t*>(tmem_slot);

    bool acc_ok = true;
    if (warp == 0) {
        // Set-up ran under the kernel ahead; nothing is read or written before it has completed.  The kernel behind may
        // become resident only then, so that it can read what came before this one without a wait of its own.
        if (!p.late_wait) asm volatile("griddepcontrol.wait;" ::: "memory");
        if (lane == 0) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        if (p.clear_status && blockIdx.x == 0) p.status[lane] = p.status[lane + 32] = 0;
        {
            bool ok = true;
            for (int i = 0, s = 0, round = 0; i < niter; ++i) {
                if (round > 0) ok = mbar_wait_warp(bar_base + (p.stages + s) * 8, (round & 1) ^ 1);
                if (!ok) break;
                const uint32_t full = bar_base + s * 8, dst = data + s * p.stage_bytes;
                const int c0 = (k0 + i) * kBK;
                if (elect_one()) {
                    mbar_expect_tx(full, kTokXBytes + (uint32_t)(p.gate_box + p.a_copies * p.a_box) * 128u);
                    tma_load_2d(dst, &tmX, c0, tok0, full);
                    if (p.gate_box) tma_load_2d(dst + kTokXBytes, &tmG, c0, 0, full);
                    for (int q = 0; q < p.a_copies; ++q)
                        tma_load_2d(dst + kTokXBytes + (uint32_t)(p.gate_box + q * p.a_box) * 128u, &tmA, c0, a_row0 + q * p.a_box, full);
                }
                __syncwarp();
                if (++s == p.stages) s = 0, ++round;
            }
            if (!ok && lane == 0 && p.status) {
                atomicExch(p.status, 1);
                atomicExch(p.status + 1, 3100);
            }
        }
    } else if (warp == 1) {
        {
            bool ok = true;
            for (int i = 0, s = 0, round = 0; i < niter; ++i) {
                ok = mbar_wait_warp(bar_base + s * 8, round & 1);
                if (!ok) break;
                tc_fence_after();
                const uint32_t xa = data + s * p.stage_bytes, wa = xa + kTokXBytes;
                const uint64_t da = smem_desc_sw128(xa);
                if (elect_one()) {
                    for (int tile = 0; tile < p.rounds; ++tile) {
                        const uint64_t db = smem_desc_sw128(wa + (uint32_t)tile * kTokCols * 128u);
                        const uint32_t idesc = instr_desc_bf16(p.cols[tile]);
#pragma unroll
                        for (int kk = 0; kk < kBK / kUmmaK; ++kk)
                            umma_bf16(tmem_base + (DUAL ? (kk & 1) * p.acc2 : tile * kTokCols), da + (uint64_t)(kk * 2), db + (uint64_t)(kk * 2), idesc,
                                      DUAL ? i > 0 || kk > 1 : (i | kk) != 0);
                    }
                    umma_commit(bar_base + (p.stages + s) * 8);
                }
                __syncwarp();
                if (++s == p.stages) s = 0, ++round;
            }
            if (elect_one()) umma_commit(bar_acc);
            __syncwarp();
            if (!ok && lane == 0 && p.status) {
                atomicExch(p.status, 1);
                atomicExch(p.status + 2, 3200);
            }
        }
    } else {
        acc_ok = mbar_wait(bar_acc, 0);
        if (!acc_ok && lane == 0 && p.status) {
            atomicExch(p.status, 1);
            atomicExch(p.status + 3, 3300);
        }
        acc_ok = __all_sync(0xFFFFFFFFu, acc_ok);
        tc_fence_after();
    }
    for (int round = 0; round < p.rounds; ++round) {
        if (warp >= 2) {
            // this round's accumulators to shared memory, [token][columns] (the ring is idle: every load has been consumed)
            const int quad = warp & 3, cols = p.cols[round];
            const int half = (cols / 16 + 1) / 2 * 16;
            const int c_begin = warp < 6 ? 0 : half, c_end = warp < 6 ? half : cols;
            const uint32_t dst = data + (uint32_t)((quad * 32 + lane) * p.pitch) * 4u;
            const uint32_t src = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(round * kTokCols);
            for (int c0 = c_begin; c0 < c_end; c0 += 64) {
                uint32_t v[4][16];
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (c0 + 16 * q < c_end) tmem_ld16_issue(src + (uint32_t)(c0 + 16 * q), v[q]);
                if (DUAL) {                                          // (both accumulators behind one wait)
                    uint32_t v2[4][16];
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (c0 + 16 * q < c_end) tmem_ld16_issue(src + (uint32_t)(p.acc2 + c0 + 16 * q), v2[q]);
                    tmem_ld_wait();
#pragma unroll
                    for (int q = 0; q < 4; ++q)
#pragma unroll
                        for (int i = 0; i < 16; ++i) v[q][i] = __float_as_uint(__uint_as_float(v[q][i]) + __uint_as_float(v2[q][i]));
                } else {
                    tmem_ld_wait();
                }
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (c0 + 16 * q < c_end) {
#pragma unroll
                        for (int i = 0; i < 16; i += 4)
                            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst + (uint32_t)(c0 + 16 * q + i) * 4u), "r"(v[q][i]),
                                         "r"(v[q][i + 1]), "r"(v[q][i + 2]), "r"(v[q][i + 3])
                                         : "memory");
                    }
            }
        }
        __syncwarp();
        if (S > 1) cluster_sync(); else __syncthreads();
        if (warp >= 2) {
            float* s_logits = reinterpret_cast<float*>(smem_raw + (data - raw) + (uint32_t)(kTokTile * p.pitch) * 4u);
            token_round<S>(p, data, s_logits, round, rank, tok0, threadIdx.x - 64, acc_ok);
        }
        __syncwarp();
        if (S > 1) cluster_sync(); else __syncthreads();   // nobody overwrites or leaves while a peer may still read
    }
    if (p.late_wait) asm volatile("griddepcontrol.wait;" ::: "memory");
    tc_fence_before();
    __syncthreads();
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)p.tmem_cols) : "memory");
}

}  // namespace meteora
