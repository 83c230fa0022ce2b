// Whole MeteoRA linears (Eq. 2 with Eq. 3) for a prefill batch as ONE launch: persistent pairs of SMs, a tile's epilogue under
// the next tile's main loop, gate and selection as the first tiles.
// Included by wgemm_tcgen05.cu after wgemm_pair.cuh, whose device helpers it uses.
//
// A pair (cluster of two CTAs) computes tiles of 256 rows x BN tokens with tcgen05.mma.cta_group::2, as k_wgemm_pair
// does (each CTA loads its own 128 rows and its own half of the tokens; no load is multicast), but
//   - the pairs stay and walk over the tiles: two accumulators in TMEM (256 columns each), so the MMAs of tile i + 1 run
//     while the epilogue warps round, stage and store tile i;
//   - the first tiles are those of the stacked matrix [Wg; A_0..A_{N-1}]: the CTA with Wg's rows selects from its accumulators
//     (top-k, softmax: a thread per token), then every CTA writes its rows' share of us[t][e r + q] = bf16(w_j (A_e x_t)_q)
//     where token t picked e, else 0, from its accumulators through shared memory and TMA (stores from
//     registers queue behind the tiles' loads: 60 - 75 ns each, 15 us in all);
//   - the LoRA expand is a few more k-steps of the same ring: the contraction goes on over the N r columns of us against
//     the B rows of the tile, both by TMA.  A tile's expand is issued near the end of the NEXT tile's main loop, by
//     which time the selection is ready: nothing waits for the routing;
//   - where the kernels otherwise taken expand in fp32 (decode batches, few tiles of large ranks: persist_us_parts) us is
//     three bf16 parts whose sum is w_j (A_e x_t)_q exactly: a k-step of the expand is then two stages, (B, part 0) and
//     (part 1, part 2), so that B is read once; the routing kernels ahead write the parts.  Such a token's y depends on its
//     own picks alone, also where an adapter that it did not pick holds an infinity or a NaN: 0 times those is NaN, and a
//     NaN of such a row is computed again from the picks.  Measured against rounded parts: 4096 -> 2 x 14336 at 64 tokens
//     49.9 -> 52.2 us, 5120 -> 13824 at 200 tokens 37.3 -> 39.4 (four stages more per tile);
//   - modules that share x (q/k/v, gate/up) are one walk: their tiles fill rounds of pairs together.
// Where the stacked matrix has more than 512 rows, the batch more token tiles than pairs, one round of tiles would become two, or
// us is three parts, the routing kernels ahead write us and only the base product runs here (stacked_pairs = 0).
// What bounds it: the tensor cores under the board's power limit (514 cycles per 64-element k-step and 256 x 256 tile, of
// the 512 that its four MMAs take).  All pairs walk the contraction axis in step, so a line of W0 or x is fetched once for the pairs
// that share it: dealing the last rounds as equal ranges of k-steps instead (partial tiles through L2) took 428 against 415 us
// at 4096 -> 14336, 517 against 477 at 14336 -> 4096 (4096 tokens, sustained load).  The issuing warps stay together and elect a
// lane per k-step: a loop entered by one lane moved every operand to uniform registers by itself, 450 - 530 cycles per step
// (4096 -> 4096 at 64 tokens 29.4 -> 18.7 us, 4096 -> 14336 at 2048 tokens 188 -> 178 us for the walk).
//   warp 0 (both CTAs)  TMA producer; every copy signals the leader's full barrier, which expects both CTAs' bytes.
//   warp 1 (leader)     MMA issue; stages are released and accumulators announced by commits that arrive in both CTAs.
//   warps 2-9 (both)    epilogue: two groups of four warps take turns at chunks of CT tokens, each with a staging buffer of
//                       its own: TMEM -> bf16 -> shared memory -> TMA store.
// Pairs wait for one another's selection, so with stacked tiles the launch is cooperative (all pairs resident).  Every wait
// is bounded; the pair leaves together.
#pragma once

namespace meteora {

constexpr int kPersistStageBufs = 2;                              // one per epilogue group
constexpr int kPersistStoreBytes = 64 * kBM * 2;                  // a staging buffer: up to 64 tokens x 128 rows of bf16
constexpr int kPersistMaxPairs = 74;
constexpr int kPersistMaxN = 64;                                  // adapters the selection here takes

struct PersistMaps {                                              // per module, then the shared tokens
    CUtensorMap W0[kMaxGroupModules], B[kMaxGroupModules], U[kMaxGroupModules], Y[kMaxGroupModules];
    CUtensorMap S[kMaxGroupModules];                              // us as the stacked tiles store it: 32 columns x 32 tokens
    CUtensorMap A[kMaxGroupModules], A0[kMaxGroupModules], G[kMaxGroupModules];   // A, its rows behind Wg in the first tile, Wg
    CUtensorMap X;
};
struct PersistModule {
    int tile0;                    // its first tile
    int row_tiles, row_pairs, group_pairs;   // group_pairs: row pairs per scheduling group
    const __nv_bfloat16* us;      // [T][parts][64 esteps]
    int32_t* topk_idx;
    float* topk_w;
    const __nv_bfloat16 *W0, *B;  // for the elements that are computed again
    int d_out;
};
struct PersistParams {
    int T, BN, CT;                // tokens per tile, tokens per epilogue chunk (divides BN)
    int ksteps, esteps;           // main k-steps; expand k-steps (8 blocks of 8 columns each)
    int N, r, k, nblk, cpa;       // N r / 8 blocks, r / 8 blocks per adapter
    int stages, stage_bytes;
    int n_mod, tok_tiles, tiles;
    int stacked_pairs;            // pairs of 128-row tiles of [Wg; A] (0: us comes from the kernel ahead)
    int gate_rows, us_cols;       // Wg's rows padded to whole 32s; columns of a part of us that are read
    int parts;                    // of us: 1 or 3
    float inv_tau;
    int32_t* flags;               // [module][token tile][2]: picks written, us written; zero between calls
    int32_t* leave_ctr;           // CTAs that are done with the flags
    int32_t* status;
    int pdl;
    const __nv_bfloat16* x;
    int d_in;
    PersistModule mod[kMaxGroupModules];
};

// 3-D and 4-D tile loads of a pair: the completion bytes go to a barrier that may live in the pair's other CTA.
__device__ __forceinline__ void tma_load_3d_grp(uint32_t dst, const CUtensorMap* tm, int c0, int c1, int c2, uint32_t cluster_bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(dst), "l"((uint64_t)tm), "r"(c0), "r"(c1), "r"(c2), "r"(cluster_bar)
        : "memory");
}
__device__ __forceinline__ void tma_load_4d_grp(uint32_t dst, const CUtensorMap* tm, int c0, int c1, int c2, int c3, uint32_t cluster_bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
        ::"r"(dst), "l"((uint64_t)tm), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(cluster_bar)
        : "memory");
}
__device__ __forceinline__ uint32_t instr_desc_bf16_pair_n(int bn) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(bn >> 3) << 17) | ((uint32_t)(256 >> 4) << 24);
}

// Tile number -> module, kind and place.  Stacked tiles of all modules come first; then module by module, groups of row
// pairs running over all token tiles before the next group starts, so that the tiles in flight share a few row pairs of W0.
struct PersistTile {
    int mod, row_pair, tok_tile;
    bool stacked;
    __device__ __forceinline__ PersistTile(const PersistParams& p, int lin) {
        const int per_mod = p.stacked_pairs * p.tok_tiles;
        stacked = lin < p.n_mod * per_mod;
        if (stacked) {
            mod = lin / per_mod;
            const int rem = lin - mod * per_mod;
            tok_tile = rem / p.stacked_pairs;
            row_pair = rem - tok_tile * p.stacked_pairs;
        } else {
            mod = 0;
#pragma unroll
            for (int m = 1; m < kMaxGroupModules; ++m)
                if (m < p.n_mod && lin >= p.mod[m].tile0) mod = m;
            const PersistModule& mo = p.mod[mod];
            lin -= mo.tile0;
            const int per_group = mo.group_pairs * p.tok_tiles, g = lin / per_group, rem = lin - g * per_group;
            const int n = min(mo.group_pairs, mo.row_pairs - g * mo.group_pairs);
            tok_tile = rem / n;
            row_pair = g * mo.group_pairs + rem - tok_tile * n;
        }
    }
};

// The token's k highest logits, descending, equal ones by ascending index, and their softmax (Eq. 3), by two adjacent lanes that
// hold half of the logits each as keys in registers.  Logit j of the token in column `tok` lies at s[j * 64 + (tok ^ (j & 31))]:
// neither the writers (a lane per logit) nor the readers meet in a bank.  NV: N padded to 32 or 64.  Returns the picks, a
// byte each.  Bound by the latency of its chain of compares (a thread per token: 2.8 us for 64 tokens).
template <int NV>
__device__ __forceinline__ unsigned long long persist_topk(const float* s, int tok, int half, int N, int k, float inv_tau, float& first,
                                                           float& sum) {
    uint32_t key[NV / 2];                                         // order-preserving; 0: none or taken
#pragma unroll
    for (int i = 0; i < NV / 2; ++i) {
        const int j = half * (NV / 2) + i;
        float v = s[j * 64 + (tok ^ (j & 31))];
        if (!(v > -CUDART_INF_F)) v = -CUDART_INF_F;              // NaN never wins
        const uint32_t bits = __float_as_uint(v + 0.f);           // -0 becomes +0
        key[i] = j >= N ? 0u : (bits & 0x80000000u) ? ~bits : (bits | 0x80000000u);
    }
    unsigned long long picks = 0;
    first = sum = 0.f;
#pragma unroll 1
    for (int n = 0; n < k; ++n) {
        uint32_t best = key[0];
        int at = 0;
#pragma unroll
        for (int i = 1; i < NV / 2; ++i)
            if (key[i] > best) {
                best = key[i];
                at = i;
            }
        at += half * (NV / 2);
        const uint32_t other = __shfl_xor_sync(0xFFFFFFFFu, best, 1);
        const int other_at = __shfl_xor_sync(0xFFFFFFFFu, at, 1);
        if (other > best || (other == best && half == 1)) {
            best = other;
            at = other_at;
        }
#pragma unroll
        for (int i = 0; i < NV / 2; ++i)
            if (half * (NV / 2) + i == at) key[i] = 0u;
        picks |= (unsigned long long)at << (8 * n);
        const float v = __uint_as_float((best & 0x80000000u) ? (best & 0x7FFFFFFFu) : ~best);
        if (n == 0) first = v;
        sum += expf((v - first) * inv_tau);
    }
    return picks;
}
// Weight of an adapter picked above.
__device__ __forceinline__ float persist_weight(const float* s, int tok, int j, float inv_tau, float first, float sum) {
    const float v = s[j * 64 + (tok ^ (j & 31))];
    return expf(((v > -CUDART_INF_F ? v : -CUDART_INF_F) + 0.f - first) * inv_tau) / sum;
}
// Whether 8 packed bf16 hold an infinity or a NaN.
__device__ __forceinline__ bool any_nonfinite(const uint4& v) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
    bool any = false;
#pragma unroll
    for (int i = 0; i < 4; ++i) any |= (w[i] & 0x7F80u) == 0x7F80u || (w[i] & 0x7F800000u) == 0x7F800000u;
    return any;
}

// A warp's 32 rows x `nt` tokens of a staged chunk of y ([token][128 rows]) in which some element is NaN: those of rows where some
// adapter's B is not finite are computed again as W0 x + the picks' terms.  (A NaN of any other row is the row's own.)  Never
// taken on finite weights; a row with such an entry costs a dot product per token.
__device__ __noinline__ void persist_repair(const PersistParams& p, const PersistModule& mo, __nv_bfloat16* ystage, int tile_row0, int quad,
                                            int tok0, int nt) {
    const int lane = threadIdx.x & 31, row0 = tile_row0 + quad * 32, row = row0 + lane;
    asm volatile("griddepcontrol.wait;" ::: "memory");               // (the producer has waited: this thread may read what it waited for)
    bool odd = false;
    if (row < mo.d_out)
        for (int e = 0; e < p.N; ++e)
            for (int c = 0; c < p.r; c += 8) odd |= any_nonfinite(*reinterpret_cast<const uint4*>(mo.B + ((size_t)e * mo.d_out + row) * p.r + c));
    const int cols = 64 * p.esteps;
    for (int i = 0; i < nt; ++i) {
        unsigned todo = __ballot_sync(0xFFFFFFFFu, odd && __hisnan(ystage[i * kBM + quad * 32 + lane]));
        const int t = tok0 + i;
        while (todo) {
            const int src = __ffs(todo) - 1;
            todo &= todo - 1;
            const float base = warp_dot(mo.W0 + (size_t)(row0 + src) * p.d_in, p.x + (size_t)t * p.d_in, p.d_in, lane, true);
            float lora = 0.f;
            for (int s = lane; s < p.k * p.r; s += 32) {
                const int j = s / p.r, q = s - j * p.r, e = min(max(__ldcg(mo.topk_idx + (size_t)t * p.k + j), 0), p.N - 1);
                const unsigned short* u = reinterpret_cast<const unsigned short*>(mo.us) + (size_t)t * 3 * cols + e * p.r + q;
                const float rest = __uint_as_float((uint32_t)__ldcg(u + cols) << 16) + __uint_as_float((uint32_t)__ldcg(u + 2 * cols) << 16);
                const float uw = __uint_as_float((uint32_t)__ldcg(u) << 16) + rest;
                lora = fmaf(to_f32(mo.B[((size_t)e * mo.d_out + row0 + src) * p.r + q]), uw, lora);
            }
            lora = warp_sum(lora);
            if (lane == src) ystage[i * kBM + quad * 32 + lane] = __float2bfloat16_rn(base + lora);
        }
    }
}

__device__ __forceinline__ void st_cluster_v2(uint32_t cluster_addr, int2 v) {
    asm volatile("st.shared::cluster.v2.b32 [%0], {%1, %2};" ::"r"(cluster_addr), "r"(v.x), "r"(v.y) : "memory");
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads)
k_wgemm_persist(const __grid_constant__ PersistMaps maps, const __grid_constant__ PersistParams p) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t ring = (raw + 1023u) & ~1023u;
    const uint32_t store = ring + p.stages * p.stage_bytes;       // staging buffers
    uint8_t* store_ptr = smem_raw + (store - raw);
    // full[stages], empty[stages], acc_full[2], acc_empty[2], picks[2]
    const uint32_t bar_base = store + kPersistStageBufs * kPersistStoreBytes;
    const uint32_t bar_accf = bar_base + 2 * p.stages * 8, bar_acce = bar_accf + 16, bar_pick = bar_accf + 32;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem_raw + (bar_base - raw) + (2 * p.stages + 6) * 8);

    const int warp = warp_id(), lane = threadIdx.x & 31;
    const uint32_t rank = __shfl_sync(0xFFFFFFFFu, cluster_rank(), 0);
    const bool leader = rank == 0;
    const int pair0 = (int)blockIdx.x >> 1, npairs = (int)gridDim.x >> 1;
    // where the tile before gets its expand: late, so that the selection is ready for the first tiles, and early enough for
    // that tile's epilogue to end under the rest (12 k-steps: 4 us)
    const int mid = max(p.ksteps / 2, p.ksteps - 12);

    if (threadIdx.x == 0) {
        for (int s = 0; s < p.stages; ++s) {
            mbar_init(bar_base + s * 8, 1);                       // the leader's expect-tx arrival
            mbar_init(bar_base + (p.stages + s) * 8, 1);          // one multicast commit
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(bar_accf + b * 8, 1);                       // one multicast commit
            mbar_init(bar_acce + b * 8, 4);                       // (leader's) two epilogue groups of each CTA, once per tile
            mbar_init(bar_pick + b * 8, 1);                       // the peer's group with the logits
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncwarp();
    cluster_sync();                                               // both CTAs' barriers exist before anyone signals
    tc_fence_after();
    const uint32_t tmem_base = *reinterpret_cast<volatile uint32_t*>(tmem_slot);
    // (the next call's first kernel waits for this one: its CTAs set up as this one's leave)
    if (p.pdl && threadIdx.x == 0) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer (both CTAs)
        {
            int s = 0, round = 0;                                 // ring slot, how often the ring has been filled
            bool waited = !p.pdl;
            // with stacked tiles x comes from the kernel ahead; else the kernel ahead is this call's routing, which read x
            if (p.stacked_pairs > 0 && !waited) {
                asm volatile("griddepcontrol.wait;" ::: "memory");
                waited = true;
            }
            auto slot = [&](uint32_t& full, uint32_t& full_leader, uint32_t& dst) {   // the next free stage
                if (round > 0 && !mbar_wait_warp(bar_base + (p.stages + s) * 8, (round & 1) ^ 1)) return false;
                full = bar_base + s * 8;
                full_leader = map_to_cta(full, 0);
                dst = ring + s * p.stage_bytes;
                if (++s == p.stages) {
                    s = 0;
                    ++round;
                }
                return true;
            };
            auto expand = [&](const PersistTile& t) {
                if (p.stacked_pairs > 0) {                        // the selection of these tokens
                    const bool there = lane != 0 || wait_counter_slow(p.flags + (t.mod * p.tok_tiles + t.tok_tile) * 2 + 1, 4 * p.stacked_pairs, 100);
                    if (!__all_sync(0xFFFFFFFFu, there)) return false;
                    asm volatile("fence.proxy.async;" ::: "memory");
                } else if (!waited) {
                    asm volatile("griddepcontrol.wait;" ::: "memory");
                    waited = true;
                }
                const int row0 = (t.row_pair * 2 + (int)rank) * kBM, tokh = t.tok_tile * p.BN + (int)rank * (p.BN / 2);
                uint32_t own, full, dst;
                for (int i = 0; i < p.esteps; ++i) {
                    if (!slot(own, full, dst)) return false;
                    const int q0 = i * 8;                         // first of the 8 blocks
                    if (elect_one()) {
                        if (leader) mbar_expect_tx(own, 2 * (uint32_t)p.stage_bytes);
                        if (p.cpa == 1)
                            tma_load_3d_grp(dst, &maps.B[t.mod], 0, row0 / 8, q0, full);
                        else
                            tma_load_4d_grp(dst, &maps.B[t.mod], 0, row0, q0 % p.cpa, q0 / p.cpa, full);
                        tma_load_2d_pair(dst + kWTileBytes, &maps.U[t.mod], q0 * 8, tokh, full);
                    }
                    __syncwarp();
                    if (p.parts == 1) continue;
                    if (!slot(own, full, dst)) return false;
                    if (elect_one()) {                            // the other two parts: one where W0's rows would lie
                        if (leader) mbar_expect_tx(own, 2 * (uint32_t)p.BN * 128u);
                        tma_load_2d_pair(dst, &maps.U[t.mod], (p.esteps + i) * kBK, tokh, full);
                        tma_load_2d_pair(dst + kWTileBytes, &maps.U[t.mod], (2 * p.esteps + i) * kBK, tokh, full);
                    }
                    __syncwarp();
                }
                return true;
            };
            bool ok = true;
            PersistTile before(p, 0);
            bool pending = false;
            for (int lin = pair0; lin < p.tiles && ok; lin += npairs) {
                const PersistTile t(p, lin);
                const int row_tile = t.row_pair * 2 + (int)rank, tokh = t.tok_tile * p.BN + (int)rank * (p.BN / 2);
                // own 128 rows of the stacked matrix: Wg and the first rows of A behind it, or 128 rows of A (zeros past the end)
                const bool gate = t.stacked && row_tile == 0;
                const CUtensorMap* mW = !t.stacked ? &maps.W0[t.mod] : gate ? &maps.A0[t.mod] : &maps.A[t.mod];
                const int w_row = !t.stacked ? row_tile * kBM : gate ? 0 : row_tile * kBM - p.gate_rows;
                const uint32_t w_off = gate ? (uint32_t)p.gate_rows * 128u : 0u;
                uint32_t own, full, dst;
                for (int i = 0; i < p.ksteps && ok; ++i) {
                    if (i == mid && pending) ok = expand(before);
                    if (!ok || !(ok = slot(own, full, dst))) break;
                    if (elect_one()) {
                        if (leader) mbar_expect_tx(own, 2 * (uint32_t)p.stage_bytes);
                        tma_load_2d_pair(dst + w_off, mW, i * kBK, w_row, full);
                        if (gate) tma_load_2d_pair(dst, &maps.G[t.mod], i * kBK, 0, full);
                        tma_load_2d_pair(dst + kWTileBytes, &maps.X, i * kBK, tokh, full);
                    }
                    __syncwarp();
                }
                pending = !t.stacked;
                before = t;
            }
            if (ok && pending) ok = expand(before);
            if (!ok && lane == 0) {
                atomicExch(p.status, 1);
                atomicExch(p.status + 1, 5100);
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer (leader only)
        if (leader) {
            const uint32_t idesc = instr_desc_bf16_pair_n(p.BN);
            bool ok = true, pending = false;
            int s = 0, phase = 0, n = 0;
            auto next = [&](uint32_t& wa) {                       // the next filled stage
                if (!mbar_wait_warp(bar_base + s * 8, phase)) return false;
                tc_fence_after();
                wa = ring + s * p.stage_bytes;
                return true;
            };
            auto release = [&]() {
                if (++s == p.stages) {
                    s = 0;
                    phase ^= 1;
                }
            };
            auto expand = [&](int b) {
                uint32_t wa, ua;
                for (int i = 0; i < p.esteps; ++i) {
                    if (!next(wa)) return false;
                    const int first = s;                          // stage with the B rows: released with the parts behind it
                    uint64_t db[3] = {smem_desc_sw128(wa + kWTileBytes), 0, 0};
                    if (p.parts > 1) {
                        release();
                        if (!next(ua)) return false;
                        db[1] = smem_desc_sw128(ua);
                        db[2] = smem_desc_sw128(ua + kWTileBytes);
                    }
                    const int nm = min(4, (p.nblk - i * 8 + 1) / 2);   // two blocks per MMA: 8-row x 16-byte core matrices, 2 KB per block
                    if (elect_one()) {
#pragma unroll
                        for (int h = 0; h < 3; ++h)
                            if (h < p.parts)
                                for (int kk = 0; kk < nm; ++kk)
                                    umma_bf16_pair(tmem_base + b * kPairTokens, smem_desc_plain(wa + kk * 2 * kBM * 16, kBM * 16, 128),
                                                   db[h] + (uint64_t)(kk * 2), idesc, 1);
                        umma_commit_pair(bar_base + (p.stages + first) * 8);
                        if (p.parts > 1) umma_commit_pair(bar_base + (p.stages + s) * 8);
                    }
                    __syncwarp();
                    release();
                }
                if (elect_one()) umma_commit_pair(bar_accf + b * 8);
                __syncwarp();
                return true;
            };
            for (int lin = pair0; lin < p.tiles && ok; lin += npairs, ++n) {
                const int b = n & 1;
                const uint32_t acc = tmem_base + b * kPairTokens;
                if (n >= 2) {                                     // the epilogue of tile n - 2 has read this accumulator
                    ok = __all_sync(0xFFFFFFFFu, mbar_wait_cluster(bar_acce + b * 8, ((n >> 1) & 1) ^ 1));
                    if (!ok) break;
                    tc_fence_after();
                }
                uint32_t wa;
                for (int i = 0; i < p.ksteps; ++i) {
                    if (i == mid && pending && !(ok = expand(b ^ 1))) break;
                    if (!(ok = next(wa))) break;
                    const uint64_t da = smem_desc_sw128(wa), db = smem_desc_sw128(wa + kWTileBytes);
                    if (elect_one()) {
#pragma unroll
                        for (int kk = 0; kk < kBK / kUmmaK; ++kk)
                            umma_bf16_pair(acc, da + (uint64_t)(kk * 2), db + (uint64_t)(kk * 2), idesc, (i | kk) != 0);
                        umma_commit_pair(bar_base + (p.stages + s) * 8);
                    }
                    __syncwarp();
                    release();
                }
                if (!ok) break;
                pending = lin >= p.mod[0].tile0;
                if (!pending && elect_one()) umma_commit_pair(bar_accf + b * 8);
                __syncwarp();
            }
            if (ok && pending) ok = expand((n & 1) ^ 1);
            if (!ok && lane == 0) {
                atomicExch(p.status, 1);
                atomicExch(p.status + 2, 5200);
            }
        }
    } else {
        // ------------------------------------------------------------------ epilogue (both CTAs)
        const int quad = warp & 3, grp = warp < 6 ? 0 : 1;        // TMEM lanes 32 quad ..; group of four warps
        const int row_in_tile = quad * 32 + lane;
        const bool elected = (warp == 2 || warp == 6) && lane == 0;
        const int chunks = p.BN / p.CT;
        __nv_bfloat16* ystage = reinterpret_cast<__nv_bfloat16*>(store_ptr + grp * kPersistStoreBytes);
        const uint32_t ysmem = store + grp * kPersistStoreBytes;
        bool acc_ok = true;
        int n = 0;
        for (int lin = pair0; lin < p.tiles; lin += npairs, ++n) {
            const PersistTile t(p, lin);
            const int tile_m = t.row_pair * 2 + (int)rank, tok0 = t.tok_tile * p.BN, b = n & 1;
            const PersistModule& mo = p.mod[t.mod];
            // (after an expired wait the rest of the walk only keeps the barriers going)
            acc_ok = __all_sync(0xFFFFFFFFu, acc_ok && mbar_wait(bar_accf + b * 8, (n >> 1) & 1));
            if (!acc_ok && lane == 0) {
                atomicExch(p.status, 1);
                atomicExch(p.status + 3, 5300);
            }
            tc_fence_after();
            const uint32_t taddr = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(b * kPairTokens);
            if (t.stacked) {
                int32_t* flag = p.flags + (t.mod * p.tok_tiles + t.tok_tile) * 2;
                float* s_lg = reinterpret_cast<float*>(ystage);
                // [own chunk][pick][token]: adapter, weight.  One pair of stacked tiles: behind the logits (N <= 32), handed to the
                // peer through distributed shared memory; two: through the routing arrays
                const bool one = p.stacked_pairs == 1;
                int2* s_pick = reinterpret_cast<int2*>(reinterpret_cast<uint8_t*>(ystage) + kPersistStoreBytes / 2);
                const uint32_t peer_pick = map_to_cta(ysmem + kPersistStoreBytes / 2, rank ^ 1u);
                const int gtid = quad * 32 + lane;                // thread of the group
                if (tile_m == 0) {
#pragma unroll 1
                    for (int c = grp; c < chunks; c += 2) {
                        if (quad * 32 < p.gate_rows) {            // warp-uniform: lane = logit
#pragma unroll 1
                            for (int q = 0; q < p.CT; q += 32) {
                                uint32_t v[2][16];
                                tmem_ld16_issue(taddr + (uint32_t)(c * p.CT + q), v[0]);
                                tmem_ld16_issue(taddr + (uint32_t)(c * p.CT + q + 16), v[1]);
                                tmem_ld_wait();
#pragma unroll
                                for (int i = 0; i < 32; ++i) s_lg[row_in_tile * 64 + ((q + i) ^ lane)] = __uint_as_float(v[i >> 4][i & 15]);
                            }
                        }
                        asm volatile("bar.sync %0, 128;" ::"r"(2 + grp) : "memory");
                        const int col = gtid >> 1, half = gtid & 1, tk = tok0 + c * p.CT + col;   // two lanes per token
                        if (col < p.CT) {                         // warp-uniform
                            float first, sum;
                            const unsigned long long picks = p.gate_rows <= 32
                                                                 ? persist_topk<32>(s_lg, col, half, p.N, p.k, p.inv_tau, first, sum)
                                                                 : persist_topk<64>(s_lg, col, half, p.N, p.k, p.inv_tau, first, sum);
#pragma unroll 1
                            for (int j = half; j < p.k; j += 2) {
                                const int e = (int)(picks >> (8 * j)) & 0xFF;
                                const float w = persist_weight(s_lg, col, e, p.inv_tau, first, sum);
                                const int at = ((c >> 1) * p.k + j) * p.CT + col;
                                const int2 pick = make_int2(tk < p.T ? e : -1, __float_as_int(w));
                                if (one) {
                                    s_pick[at] = pick;
                                    st_cluster_v2(peer_pick + (uint32_t)at * 8u, pick);
                                } else if (tk < p.T) {
                                    mo.topk_idx[(size_t)tk * p.k + j] = e;
                                    mo.topk_w[(size_t)tk * p.k + j] = w;
                                }
                            }
                        }
                        __syncwarp();
                        asm volatile("bar.sync %0, 128;" ::"r"(2 + grp) : "memory");
                    }
                    if (!one) {
                        __threadfence();
                        asm volatile("bar.sync %0, 128;" ::"r"(2 + grp) : "memory");
                    }
                    if (elected) {
                        if (one) mbar_arrive_cluster(map_to_cta(bar_pick + grp * 8, 1));
                        else atomicAdd(flag, 1);
                    }
                }
                bool have = true;
                if (one) {
                    if (tile_m != 0) have = mbar_wait_cluster(bar_pick + grp * 8, 0);
                } else {
                    if (elected) have = wait_counter(flag, 2);
                    __syncwarp();
                    asm volatile("bar.sync %0, 128;" ::"r"(2 + grp) : "memory");
                    __threadfence();
#pragma unroll 1
                    for (int c = grp; c < chunks; c += 2)
#pragma unroll 1
                        for (int i = gtid; i < p.CT * p.k; i += 128) {
                            const int j = i / p.CT, tk = i - j * p.CT;
                            const size_t src = (size_t)(tok0 + c * p.CT + tk) * p.k + j;
                            s_pick[(c >> 1) * p.k * p.CT + i] =
                                tok0 + c * p.CT + tk < p.T ? make_int2(__ldcg(mo.topk_idx + src), __float_as_int(__ldcg(mo.topk_w + src))) : make_int2(-1, 0);
                        }
                    __syncwarp();
                    asm volatile("bar.sync %0, 128;" ::"r"(2 + grp) : "memory");
                }
                if (!have && lane == 0) {
                    atomicExch(p.status, 1);
                    atomicExch(p.status + 4, 5400);
                }
                // a warp's 32 columns of us for 32 tokens at a time, in the lower half of the staging buffer
                const int a0 = tile_m * kBM + quad * 32 - p.gate_rows, e = (a0 + lane) / p.r;
                if (a0 >= 0 && a0 < p.us_cols) {
                    const uint32_t us_smem = ysmem + (uint32_t)quad * 2048u;
                    __nv_bfloat16* s_us = ystage + quad * 1024;   // [token][32 columns]
#pragma unroll 1
                    for (int c = grp; c < chunks; c += 2)
#pragma unroll 1
                        for (int h = 0; h < p.CT; h += 32) {
                            const int2* pk = s_pick + (c >> 1) * p.k * p.CT + h;
                            bool any = false;
                            for (int j = 0; j < p.k; ++j) {
                                const int x = pk[j * p.CT + lane].x;
                                any |= x >= 0 && x * p.r < a0 + 32 && (x + 1) * p.r > a0;
                            }
                            any = __any_sync(0xFFFFFFFFu, any);
                            if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");   // the store before
                            __syncwarp();
                            if (any) {
                                uint32_t v[2][16];
                                tmem_ld16_issue(taddr + (uint32_t)(c * p.CT + h), v[0]);
                                tmem_ld16_issue(taddr + (uint32_t)(c * p.CT + h + 16), v[1]);
                                float w[32];
#pragma unroll
                                for (int i = 0; i < 32; ++i) w[i] = -1.f;   // not picked (no weight is negative)
#pragma unroll 1
                                for (int j = 0; j < p.k; ++j)
#pragma unroll
                                    for (int i = 0; i < 32; ++i) {
                                        const int2 pick = pk[j * p.CT + i];
                                        w[i] = pick.x == e ? __int_as_float(pick.y) : w[i];
                                    }
                                tmem_ld_wait();
#pragma unroll
                                for (int i = 0; i < 32; ++i)
                                    s_us[i * 32 + lane] = __float2bfloat16_rn(w[i] < 0.f ? 0.f : w[i] * __uint_as_float(v[i >> 4][i & 15]));
                            } else {
#pragma unroll
                                for (int i = 0; i < 4; ++i) reinterpret_cast<uint4*>(s_us)[i * 32 + lane] = make_uint4(0u, 0u, 0u, 0u);
                            }
                            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic writes -> TMA read
                            __syncwarp();
                            if (lane == 0 && tok0 + c * p.CT + h < p.T) {
                                asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];"
                                             ::"l"((uint64_t)&maps.S[t.mod]), "r"(us_smem), "r"(a0), "r"(tok0 + c * p.CT + h)
                                             : "memory");
                                asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                            }
                        }
                    if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");   // written, not only read out
                }
                tc_fence_before();
                __threadfence();
                __syncwarp();
                asm volatile("bar.sync %0, 128;" ::"r"(2 + grp) : "memory");
                if (elected) {
                    mbar_arrive_cluster(map_to_cta(bar_acce + b * 8, 0));
                    atomicAdd(flag + 1, 1);
                }
                if (one && tile_m == 0) {                         // the routing for the caller
#pragma unroll 1
                    for (int c = grp; c < chunks; c += 2)
#pragma unroll 1
                        for (int i = gtid; i < p.CT * p.k; i += 128) {
                            const int j = i / p.CT, tk = i - j * p.CT;
                            const int2 pick = s_pick[(c >> 1) * p.k * p.CT + i];
                            if (pick.x >= 0) {
                                mo.topk_idx[(size_t)(tok0 + c * p.CT + tk) * p.k + j] = pick.x;
                                mo.topk_w[(size_t)(tok0 + c * p.CT + tk) * p.k + j] = __int_as_float(pick.y);
                            }
                        }
                }
                continue;
            }
            // a tile of one chunk (64 tokens at the most) is read by the first group alone: the other one owes its arrival all the same
            if (grp >= chunks && elected) mbar_arrive_cluster(map_to_cta(bar_acce + b * 8, 0));
            for (int c = grp; c < chunks; c += 2) {
                uint32_t v[4][16];
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (16 * q < p.CT) tmem_ld16_issue(taddr + (uint32_t)(c * p.CT + 16 * q), v[q]);
                tmem_ld_wait();
                const bool last = c + 2 >= chunks;
                if (last) tc_fence_before();                      // this group's last read of the accumulator
                // the staging buffer's last store has been read out
                if (elected) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
                asm volatile("bar.sync %0, 128;" ::"r"(2 + grp) : "memory");
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (16 * q < p.CT) {
#pragma unroll
                        for (int i = 0; i < 16; ++i)
                            ystage[(16 * q + i) * kBM + row_in_tile] = __float2bfloat16_rn(__uint_as_float(v[q][i]));
                    }
                if (p.parts > 1) {
                    bool nan = false;
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (16 * q < p.CT) {
#pragma unroll
                            for (int i = 0; i < 16; ++i) nan |= __uint_as_float(v[q][i]) != __uint_as_float(v[q][i]);
                        }
                    if (__any_sync(0xFFFFFFFFu, nan)) persist_repair(p, mo, ystage, tile_m * kBM, quad, tok0 + c * p.CT, min(p.CT, p.T - tok0 - c * p.CT));
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic writes -> TMA read
                asm volatile("bar.sync %0, 128;" ::"r"(2 + grp) : "memory");
                if (elected) {
                    if (last) mbar_arrive_cluster(map_to_cta(bar_acce + b * 8, 0));
                    if (tile_m < mo.row_tiles && tok0 + c * p.CT < p.T) {   // rows beyond d_out and tokens beyond T are clipped by the map
                        asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];"
                                     ::"l"((uint64_t)&maps.Y[t.mod]), "r"(ysmem), "r"(tile_m * kBM), "r"(tok0 + c * p.CT)
                                     : "memory");
                        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                    }
                }
            }
        }
        if (elected) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    }
    tc_fence_before();
    __syncwarp();
    cluster_sync();                                               // nobody leaves while the peer may still signal it
    if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
    if (p.stacked_pairs > 0 && threadIdx.x == 0) {                // the last CTA to leave readies the flags for the next call
        if (atomicAdd(p.leave_ctr, 1) == (int)gridDim.x - 1) {
            for (int i = 0; i < 2 * p.n_mod * p.tok_tiles; ++i) p.flags[i] = 0;
            *p.leave_ctr = 0;
        }
    }
}

}  // namespace meteora
