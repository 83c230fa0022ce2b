// The LoRA term's expand on its own (Eq. 2): delta[t] = sum_j w_j B_{e_j} u_j in fp32, u_j = A_{e_j} x_t from the shrink before.
// Included by wgemm_tcgen05.cu after the device helpers it uses.
//
// A dense product of B's rows (128 outputs on the MMA's M axis, all adapters along K) and the masked w_j u_j of 32 tokens, the
// latter as three bf16 parts that add up to fp32's value exactly.  The parts are separate columns of the accumulator (3 x 32),
// so B is read from shared memory once for all three; the epilogue adds them.  A CTA keeps the B rows of its 128 outputs (16
// bytes per row, adapter and 8 rank entries: a core matrix's row, as it lies in memory) and walks over its share of the tokens
// with four operands and four accumulators in turn: while the MMAs of one tile run, two warps per operand clear and scatter the
// next ones (k x 48 bytes per token) and two groups of four warps store those before.
// Bound by writing delta and, beside it, by the MMAs (14 per tile at 224 columns of K, about 50 cycles each, for 16 KB of delta)
// and by the loop of an operand: its product (850 cycles), then clearing and scattering (2000 - 2600 beside the others); hence four of
// 32 tokens (two of 64, in the same memory: 4096 -> 14336 at 4096 tokens 186 us for the LoRA term, now 123).  k_expand_slab on
// CUDA cores, bound by unpacking B and by shared-memory reads, has the shorter start: us for the LoRA term with that kernel / with
// this one, by T k d_out: 0.8 M (200 tokens, 4096, k 1) 24.1 / 27.5; 1.6 M (200, 4096, k 2) 19.8 / 22.5; 2.5 M (300, 4096, k 2)
// 24.3 / 24.6; 4.2 M (512, 4096, k 2) 26.5 / 25.2; 14.7 M (512, 14336, k 2) 41.4 / 34.7; 16.8 M (2048, 4096, k 2) 48.6 / 43.0; 60 M
// (3000, 5000, k 4) 89.5 / 64.7; 117 M (4096, 14336, k 2) 174 / 123: this one from 3 M on (kExtMinWork).
// The product multiplies the zeros of adapters that a token did not pick, and 0 times an infinity or a NaN is NaN: an element
// that is NaN is computed again from the picks alone.
#pragma once

namespace meteora {

constexpr int kExtStages = 4;                       // token operands and accumulators
constexpr int kExtTok = 32;                         // tokens per tile
constexpr int kExtCols = 3 * kExtTok;               // accumulator columns: three parts
constexpr int kExtABlock = kBM * 16, kExtBBlock = kExtCols * 16;   // bytes per 8 columns of K
constexpr long long kExtMinWork = 3 << 20;          // T k d_out
constexpr int kExtMaxBlocks = 28;                   // what fits beside B's rows
constexpr int kExtBuilders = 64;                    // threads per token operand
constexpr int kExtEpilogue = 128;                   // threads per tile; two such groups take turns
constexpr int kExtFirstEpi = 2 + kExtStages * kExtBuilders / 32, kExtThreads = kExtFirstEpi * 32 + 2 * kExtEpilogue;
constexpr int kExtHead = 2048;                      // barriers and, per token operand, the picks that are written
constexpr size_t kExtMaxSmem = 1024 + kExtHead + (size_t)kExtMaxBlocks * (kExtABlock + kExtStages * kExtBBlock);
static_assert(kExtMaxSmem <= 227 * 1024, "shared memory of an SM");
static_assert(128 + kExtStages * kExtTok * METEORA_MAX_K <= kExtHead, "head of the shared memory");

struct ExpandTileParams {
    int T, d_out, N, r, k;
    int nblk;                  // N r / 8, rounded up to an even number
    const __nv_bfloat16* B;
    const int32_t* topk_idx;
    const float* topk_w;
    const float* u;            // [slot][r], 16-byte aligned
    float* delta;
    int32_t* status;           // error flag of expired waits (may be null)
};

// One element from the picks alone.
__device__ __noinline__ float expand_element(const ExpandTileParams& p, int t, int o) {
    float out = 0.f;
    for (int j = 0; j < p.k; ++j) {
        const size_t slot = (size_t)t * p.k + j;
        const int e = min(max(p.topk_idx[slot], 0), p.N - 1);
        float acc = 0.f;
        for (int q = 0; q < p.r; ++q) acc = fmaf(to_f32(p.B[((size_t)e * p.d_out + o) * p.r + q]), p.u[slot * p.r + q], acc);
        out = fmaf(p.topk_w[slot], acc, out);
    }
    return out;
}

__global__ void __launch_bounds__(kExtThreads, 1) k_expand_tile(const ExpandTileParams p) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t head = (raw + 1023u) & ~1023u;
    uint8_t* const head_ptr = smem_raw + (head - raw);
    // per stage: full (the builders' threads), done (the MMAs' commit), free (the epilogue's threads)
    const uint32_t bar_full = head, bar_done = bar_full + kExtStages * 8, bar_free = bar_done + kExtStages * 8;
    uint32_t* const tmem_slot = reinterpret_cast<uint32_t*>(head_ptr + 120);
    volatile int* const s_late = reinterpret_cast<volatile int*>(head_ptr + 124);   // a builder's wait ran out: no tile from there on is a result
    uint8_t* const s_pick = head_ptr + 128;                          // [stage][token][pick]: the adapter that holds the pick's values; 0xFF: none
    const uint32_t rows_at = head + kExtHead, toks_at = rows_at + (uint32_t)p.nblk * kExtABlock;
    const uint32_t tok_bytes = (uint32_t)p.nblk * kExtBBlock;
    uint8_t* const rows_ptr = head_ptr + kExtHead;
    uint8_t* const toks_ptr = rows_ptr + p.nblk * kExtABlock;

    const int warp = warp_id(), lane = threadIdx.x & 31;
    const int o0 = blockIdx.x * kBM, r8 = p.r / 8;
    const int blocks = (p.T + kExtTok - 1) / kExtTok;
    const int b0 = (int)((long long)blocks * blockIdx.y / gridDim.y), nb = (int)((long long)blocks * (blockIdx.y + 1) / gridDim.y) - b0;

    // B's rows (weights: they do not depend on the grid before) and the zeros of the token operands
    const uint4* Bv = reinterpret_cast<const uint4*>(p.B);
    for (int v = threadIdx.x; v < p.N * r8 * kBM; v += kExtThreads) {  // [e][output][c]: as B lies in memory
        const int c = v % r8, row = (v / r8) & (kBM - 1), e = v / (r8 * kBM);
        const bool in = o0 + row < p.d_out;
        const uint4* src = Bv + ((size_t)e * p.d_out + (in ? o0 + row : 0)) * r8 + c;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(rows_at + (uint32_t)((e * r8 + c) * kExtABlock + row * 16)), "l"(src),
                     "r"(in ? 16 : 0)
                     : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    for (int v = p.N * r8 * kBM + threadIdx.x; v < p.nblk * kBM; v += kExtThreads) reinterpret_cast<uint4*>(rows_ptr)[v] = make_uint4(0u, 0u, 0u, 0u);
    for (int v = threadIdx.x; v < min(nb, kExtStages) * (int)tok_bytes / 16; v += kExtThreads) reinterpret_cast<uint4*>(toks_ptr)[v] = make_uint4(0u, 0u, 0u, 0u);
    if (threadIdx.x == 0) {
        *s_late = 0;
        for (int s = 0; s < kExtStages; ++s) {
            mbar_init(bar_full + s * 8, kExtBuilders);
            mbar_init(bar_done + s * 8, 1);
            mbar_init(bar_free + s * 8, kExtEpilogue);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");               // u comes from the grid before, and delta may be read by it
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    // Item (token, pick, 8 rank entries) of tile i: its values, a round ahead for the first two items of a builder
    struct Item {
        bool live;                                                   // (not beyond the batch)
        int e;
        float w;
        float4 a, b;
    };
    struct Place {
        int it, slot, tok, j, c;
    };
    const int group = (warp - 2) / (kExtBuilders / 32), tid = (int)threadIdx.x - 64 - group * kExtBuilders, items = kExtTok * p.k * r8;
    auto place = [&](int it) {
        Place a;
        a.it = it;
        a.slot = it / r8;
        a.c = it - a.slot * r8;
        a.tok = a.slot / p.k;
        a.j = a.slot - a.tok * p.k;
        return a;
    };
    const Place mine[2] = {place(tid & (kExtBuilders - 1)), place((tid & (kExtBuilders - 1)) + kExtBuilders)};   // (divisions: 1500 cycles per tile where each step made its own)
    auto load = [&](int i, const Place& a, Item& q) {
        const int t0 = (b0 + i) * kExtTok;
        q.live = i < nb && a.it < items && t0 + a.tok < p.T;
        if (!q.live) return;
        const size_t at = (size_t)t0 * p.k + a.slot;
        const float4* src = reinterpret_cast<const float4*>(p.u + at * p.r + a.c * 8);
        // (volatile: a load that the compiler may move goes to its use, a round later, and is waited for there)
        asm volatile("ld.global.cg.b32 %0, [%1];" : "=r"(q.e) : "l"(p.topk_idx + at));
        asm volatile("ld.global.cg.f32 %0, [%1];" : "=f"(q.w) : "l"(p.topk_w + at));
        asm volatile("ld.global.cg.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(q.a.x), "=f"(q.a.y), "=f"(q.a.z), "=f"(q.a.w) : "l"(src));
        asm volatile("ld.global.cg.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(q.b.x), "=f"(q.b.y), "=f"(q.b.z), "=f"(q.b.w) : "l"(src + 1));
    };
    Item held[2];
    if (warp >= 2 && warp < kExtFirstEpi) {
        load(group, mine[0], held[0]);
        load(group, mine[1], held[1]);
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");     // generic writes -> tensor-core reads
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *reinterpret_cast<volatile uint32_t*>(tmem_slot);

    bool ok = true;
    int where = 0;
    if (warp == 0) {
        const uint32_t idesc = instr_desc_bf16(kExtCols);
        for (int i = 0; i < nb; ++i) {
            const int s = i % kExtStages, round = i / kExtStages;
            ok = mbar_wait_warp(bar_full + s * 8, round & 1) && (round == 0 || mbar_wait_warp(bar_free + s * 8, (round & 1) ^ 1));
            if (!ok) break;
            tc_fence_after();
            const uint64_t da = smem_desc_plain(rows_at, kExtABlock, 128), db = smem_desc_plain(toks_at + s * tok_bytes, kExtBBlock, 128);
            if (elect_one()) {
                for (int m = 0; m < p.nblk / 2; ++m)
                    umma_bf16(tmem_base + s * 128, da + (uint64_t)(m * (2 * kExtABlock >> 4)), db + (uint64_t)(m * (2 * kExtBBlock >> 4)), idesc, m != 0);
                umma_commit(bar_done + s * 8);
            }
            __syncwarp();
        }
        where = 1;
    } else if (warp >= 2 && warp < kExtFirstEpi) {
        // w_j u_j of the item in three parts; of several picks of a token that name one adapter the first takes their sum
        auto store = [&](int i, int s, const Place& a, Item& q) {
            if (!q.live) return;
            const int e = min(max(q.e, 0), p.N - 1);
            const uint8_t* const pick = s_pick + s * (kExtTok * METEORA_MAX_K) + a.tok * p.k;
            float v[8] = {q.w * q.a.x, q.w * q.a.y, q.w * q.a.z, q.w * q.a.w, q.w * q.b.x, q.w * q.b.y, q.w * q.b.z, q.w * q.b.w};
            for (int m = 0; m < p.k; ++m) {
                if (m == a.j || pick[m] != e) continue;
                if (m < a.j) return;
                const size_t at = (size_t)((b0 + i) * kExtTok + a.tok) * p.k + m;
                const float w = __ldcg(p.topk_w + at);
#pragma unroll
                for (int n = 0; n < 8; ++n) v[n] += w * __ldcg(p.u + at * p.r + a.c * 8 + n);
            }
            uint8_t* dst = toks_ptr + s * tok_bytes + (e * r8 + a.c) * kExtBBlock + a.tok * 16;
            float finite = 0.f;
#pragma unroll
            for (int n = 0; n < 8; ++n) finite = fmaf(v[n], 0.f, finite);
            if (finite == 0.f) {                                     // (cut off 16 bits at a time: see take_bf16_part)
#pragma unroll
                for (int part = 0; part < 3; ++part) {
                    uint32_t b[4];
#pragma unroll
                    for (int n = 0; n < 4; ++n) b[n] = __byte_perm(__float_as_uint(v[2 * n]), __float_as_uint(v[2 * n + 1]), 0x7632);
#pragma unroll
                    for (int n = 0; n < 8; ++n) v[n] -= __uint_as_float(__float_as_uint(v[n]) & 0xFFFF0000u);
                    *reinterpret_cast<uint4*>(dst + part * (kExtTok * 16)) = make_uint4(b[0], b[1], b[2], b[3]);
                }
            } else {
                for (int n = 0; n < 8; ++n)
                    for (int part = 0; part < 3; ++part)
                        reinterpret_cast<__nv_bfloat16*>(dst + part * (kExtTok * 16))[n] = take_bf16_part(v[n]);
            }
        };
        auto clear = [&](int s, const Place& a) {                    // what the tile before last left at the item
            const int e = a.it < items ? s_pick[s * (kExtTok * METEORA_MAX_K) + a.slot] : 0xFF;
            if (e == 0xFF) return;
            uint8_t* dst = toks_ptr + s * tok_bytes + (e * r8 + a.c) * kExtBBlock + a.tok * 16;
#pragma unroll
            for (int part = 0; part < 3; ++part) *reinterpret_cast<uint4*>(dst + part * (kExtTok * 16)) = make_uint4(0u, 0u, 0u, 0u);
        };
        auto note = [&](int s, const Place& a, const Item& q) {      // the tile's picks
            if (a.c == 0 && a.it < items) s_pick[s * (kExtTok * METEORA_MAX_K) + a.slot] = q.live ? (uint8_t)min(max(q.e, 0), p.N - 1) : 0xFF;
        };
        for (int i = group; i < nb; i += kExtStages) {
            const int s = group, round = i / kExtStages;
            if (round > 0) {
                // (each thread by itself; one whose wait ran out goes on all the same: the others count on it at the barriers below)
                ok = ok && mbar_wait(bar_done + s * 8, (round & 1) ^ 1);
                if (!ok) *s_late = 1;
                clear(s, mine[0]);
                clear(s, mine[1]);
                for (int it = tid + 2 * kExtBuilders; it < items; it += kExtBuilders) clear(s, place(it));
            }
            __syncwarp();
            asm volatile("bar.sync %0, %1;" ::"r"(2 + group), "n"(kExtBuilders) : "memory");
            note(s, mine[0], held[0]);
            note(s, mine[1], held[1]);
            for (int it = tid + 2 * kExtBuilders; it < items; it += kExtBuilders) {
                const Place a = place(it);
                Item more;
                load(i, a, more);
                note(s, a, more);
            }
            __syncwarp();
            asm volatile("bar.sync %0, %1;" ::"r"(2 + group), "n"(kExtBuilders) : "memory");
            store(i, s, mine[0], held[0]);
            store(i, s, mine[1], held[1]);
            for (int it = tid + 2 * kExtBuilders; it < items; it += kExtBuilders) {
                const Place a = place(it);
                Item more;
                load(i, a, more);
                store(i, s, a, more);
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar_full + s * 8) : "memory");
            load(i + kExtStages, mine[0], held[0]);
            load(i + kExtStages, mine[1], held[1]);
        }
        where = 2;
    } else if (warp >= kExtFirstEpi) {
        const int quad = warp & 3, o = o0 + quad * 32 + lane;
        for (int i = (warp - kExtFirstEpi) / 4; i < nb; i += 2) {
            const int s = i % kExtStages, t0 = (b0 + i) * kExtTok;
            ok = ok && mbar_wait(bar_done + s * 8, (i / kExtStages) & 1);
            ok = __all_sync(0xFFFFFFFFu, ok && *s_late == 0);         // (written ahead of the arrivals that this tile's product waited for)
            tc_fence_after();
            const uint32_t src = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(s * 128);
            uint32_t v[3][kExtTok];
#pragma unroll
            for (int part = 0; part < 3; ++part)
#pragma unroll
                for (int c = 0; c < kExtTok; c += 16)
                    tmem_ld16_issue(src + (uint32_t)(part * kExtTok + c), reinterpret_cast<uint32_t(&)[16]>(v[part][c]));
            tmem_ld_wait();
            tc_fence_before();
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar_free + s * 8) : "memory");
            float out[kExtTok];
            bool odd = false;
#pragma unroll
            for (int n = 0; n < kExtTok; ++n) {
                out[n] = ok ? __uint_as_float(v[0][n]) + (__uint_as_float(v[1][n]) + __uint_as_float(v[2][n])) : CUDART_NAN_F;
                odd |= out[n] != out[n];
            }
            if (o < p.d_out) {
                const int nt = min(kExtTok, p.T - t0);
                float* dst = p.delta + (size_t)t0 * p.d_out + o;
                const size_t pitch = p.d_out;
                if (nt == kExtTok) {
#pragma unroll
                    for (int n = 0; n < kExtTok; ++n) dst[n * pitch] = out[n];
                } else {
#pragma unroll
                    for (int n = 0; n < kExtTok; ++n)
                        if (n < nt) dst[n * pitch] = out[n];
                }
                if (odd && ok)                                       // (with an expired wait the NaNs stay)
                    for (int n = 0; n < nt; ++n)
                        if (dst[n * pitch] != dst[n * pitch]) dst[n * pitch] = expand_element(p, t0 + n, o);
            }
            __syncwarp();
        }
        where = 3;
    }
    if (__any_sync(0xFFFFFFFFu, !ok) && lane == 0 && p.status) {
        atomicExch(p.status, 1);
        atomicExch(p.status + where, 5000 + where);
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
}

}  // namespace meteora
