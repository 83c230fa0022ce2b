// Base product W0 x with the LoRA expand (Eq. 2) for prefill batches: persistent pairs of SMs, a tile's epilogue under the
// next tile's main loop.
// Included by wgemm_tcgen05.cu after wgemm_pair.cuh, whose device helpers it uses.
//
// A pair (cluster of two CTAs) computes tiles of 256 rows of W0 x BN tokens with tcgen05.mma.cta_group::2, as
// k_wgemm_pair does (each CTA loads its own 128 rows and its own half of the tokens; no load is multicast), but
//   - the pairs stay and walk over the tiles: two accumulators in TMEM (256 columns each), so the MMAs of tile i + 1 run
//     while the epilogue warps round, stage and store tile i;
//   - the LoRA expand is a few more k-steps of the same ring: the contraction goes on over the N r columns of a masked,
//     gate-weighted copy of the shrink, us[t][e r + q] = bf16(w_j (A_e x_t)_q) where token t picked e, else 0 (written by
//     the routing kernel), against the B rows of the tile, both by TMA; nothing waits for an idle ring.
// What bounds it: the tensor cores under the board's power limit (0.43 us per 64-element k-step and 256 x 256 tile, 1460
// TFLOP/s over 74 pairs).  All pairs walk the contraction axis in step, so a line of W0 or x is fetched once for the pairs
// that share it: dealing the last rounds as equal ranges of k-steps instead (partial tiles through L2) took 428 against 415 us
// at 4096 -> 14336, 517 against 477 at 14336 -> 4096 (4096 tokens, sustained load).  Tiles narrower than 192 tokens gain nothing more per k-step (0.37 us: an SM's intake).
//   warp 0 (both CTAs)  TMA producer; every copy signals the leader's full barrier, which expects both CTAs' bytes.
//   warp 1 (leader)     MMA issue; stages are released and accumulators announced by commits that arrive in both CTAs.
//   warps 2-9 (both)    epilogue: two groups of four warps take turns at chunks of CT tokens, each with a staging buffer of
//                       its own: TMEM -> bf16 -> shared memory -> TMA store.
// Every wait is bounded; the pair leaves together.
#pragma once

namespace meteora {

constexpr int kPersistStageBufs = 2;                              // one per epilogue group
constexpr int kPersistStoreBytes = 64 * kBM * 2;                  // a staging buffer: up to 64 tokens x 128 rows of bf16
constexpr int kPersistMaxPairs = 74;

struct PersistParams {
    int T, BN, CT;                // tokens per tile, tokens per epilogue chunk (divides BN)
    int ksteps, iters;            // main k-steps; with the expand's (8 blocks of 8 columns each)
    int nblk;                     // N r / 8
    int stages, stage_bytes;
    int row_tiles, row_pairs, tok_tiles;
    int group_pairs;              // row pairs per scheduling group
    int tiles;
    int cpa;                      // blocks of 8 rank entries per adapter
    int32_t* status;
    int pdl_wait;
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

// Tile number -> (row pair, token tile): groups of row pairs run over all token tiles before the next group starts, so that
// the tiles in flight share a few row pairs of W0.
__device__ __forceinline__ void persist_tile(const PersistParams& p, int lin, int& row_pair, int& tok_tile) {
    const int per_group = p.group_pairs * p.tok_tiles, g = lin / per_group, rem = lin - g * per_group;
    const int n = min(p.group_pairs, p.row_pairs - g * p.group_pairs);
    tok_tile = rem / n;
    row_pair = g * p.group_pairs + rem - tok_tile * n;
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads)
k_wgemm_persist(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmB,
                const __grid_constant__ CUtensorMap tmU, const __grid_constant__ CUtensorMap tmY, const PersistParams p) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t ring = (raw + 1023u) & ~1023u;
    const uint32_t store = ring + p.stages * p.stage_bytes;       // staging buffers
    uint8_t* store_ptr = smem_raw + (store - raw);
    // full[stages], empty[stages], acc_full[2], acc_empty[2]
    const uint32_t bar_base = store + kPersistStageBufs * kPersistStoreBytes;
    const uint32_t bar_accf = bar_base + 2 * p.stages * 8, bar_acce = bar_accf + 16;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem_raw + (bar_base - raw) + (2 * p.stages + 4) * 8);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank();
    const bool leader = rank == 0;
    const int pair0 = (int)blockIdx.x >> 1, npairs = (int)gridDim.x >> 1;

    if (threadIdx.x == 0) {
        for (int s = 0; s < p.stages; ++s) {
            mbar_init(bar_base + s * 8, 1);                       // the leader's expect-tx arrival
            mbar_init(bar_base + (p.stages + s) * 8, 1);          // one multicast commit
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(bar_accf + b * 8, 1);                       // one multicast commit
            mbar_init(bar_acce + b * 8, 4);                       // (leader's) two epilogue groups of each CTA
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
    if (p.pdl_wait && threadIdx.x == 0) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer (both CTAs)
        if (lane == 0) {
            bool ok = true, waited = !p.pdl_wait;
            int s = 0, round = 0;                                 // ring slot, how often the ring has been filled
            for (int lin = pair0; lin < p.tiles && ok; lin += npairs) {
                int row_pair, tok_tile;
                persist_tile(p, lin, row_pair, tok_tile);
                const int row0 = (row_pair * 2 + (int)rank) * kBM, tokh = tok_tile * p.BN + (int)rank * (p.BN / 2);
                for (int i = 0; i < p.iters; ++i) {
                    if (round > 0) ok = mbar_wait(bar_base + (p.stages + s) * 8, (round & 1) ^ 1);
                    if (!ok) break;
                    const uint32_t full = bar_base + s * 8, full_leader = map_to_cta(full, 0), dst = ring + s * p.stage_bytes;
                    if (leader) mbar_expect_tx(full, 2 * (uint32_t)p.stage_bytes);
                    if (i < p.ksteps) {
                        tma_load_2d_pair(dst, &tmW, i * kBK, row0, full_leader);
                        tma_load_2d_pair(dst + kWTileBytes, &tmX, i * kBK, tokh, full_leader);
                    } else {
                        if (!waited) asm volatile("griddepcontrol.wait;" ::: "memory");   // us comes from the kernel ahead
                        waited = true;
                        const int q0 = (i - p.ksteps) * 8;        // first of the 8 blocks
                        if (p.cpa == 1)
                            tma_load_3d_grp(dst, &tmB, 0, row0 / 8, q0, full_leader);
                        else
                            tma_load_4d_grp(dst, &tmB, 0, row0, q0 % p.cpa, q0 / p.cpa, full_leader);
                        tma_load_2d_pair(dst + kWTileBytes, &tmU, q0 * 8, tokh, full_leader);
                    }
                    if (++s == p.stages) {
                        s = 0;
                        ++round;
                    }
                }
            }
            if (!ok) {
                atomicExch(p.status, 1);
                atomicExch(p.status + 1, 5100);
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer (leader only)
        if (lane == 0 && leader) {
            const uint32_t idesc = instr_desc_bf16_pair_n(p.BN);
            bool ok = true;
            int s = 0, phase = 0, n = 0;
            for (int lin = pair0; lin < p.tiles && ok; lin += npairs, ++n) {
                const int b = n & 1;
                const uint32_t acc = tmem_base + b * kPairTokens;
                if (n >= 2) {                                     // the epilogue of tile n - 2 has read this accumulator
                    ok = mbar_wait_cluster(bar_acce + b * 8, ((n >> 1) & 1) ^ 1);
                    if (!ok) break;
                    tc_fence_after();
                }
                for (int i = 0; i < p.iters; ++i) {
                    ok = mbar_wait(bar_base + s * 8, phase);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t wa = ring + s * p.stage_bytes;
                    const uint64_t db = smem_desc_sw128(wa + kWTileBytes);
                    if (i < p.ksteps) {
                        const uint64_t da = smem_desc_sw128(wa);
#pragma unroll
                        for (int kk = 0; kk < kBK / kUmmaK; ++kk)
                            umma_bf16_pair(acc, da + (uint64_t)(kk * 2), db + (uint64_t)(kk * 2), idesc, (i | kk) != 0);
                    } else {                                      // two blocks per MMA: 8-row x 16-byte core matrices, 2 KB per block
                        const int nm = min(4, (p.nblk - (i - p.ksteps) * 8 + 1) / 2);
                        for (int kk = 0; kk < nm; ++kk)
                            umma_bf16_pair(acc, smem_desc_plain(wa + kk * 2 * kBM * 16, kBM * 16, 128), db + (uint64_t)(kk * 2), idesc, 1);
                    }
                    umma_commit_pair(bar_base + (p.stages + s) * 8);
                    if (++s == p.stages) {
                        s = 0;
                        phase ^= 1;
                    }
                }
                umma_commit_pair(bar_accf + b * 8);
            }
            if (!ok) {
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
            int row_pair, tok_tile;
            persist_tile(p, lin, row_pair, tok_tile);
            const int tile_m = row_pair * 2 + (int)rank, tok0 = tok_tile * p.BN, b = n & 1;
            // (after an expired wait the rest of the walk only keeps the barriers going)
            acc_ok = __all_sync(0xFFFFFFFFu, acc_ok && mbar_wait(bar_accf + b * 8, (n >> 1) & 1));
            if (!acc_ok && lane == 0) {
                atomicExch(p.status, 1);
                atomicExch(p.status + 3, 5300);
            }
            tc_fence_after();
            const uint32_t taddr = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(b * kPairTokens);
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
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic writes -> TMA read
                asm volatile("bar.sync %0, 128;" ::"r"(2 + grp) : "memory");
                if (elected) {
                    if (last) mbar_arrive_cluster(map_to_cta(bar_acce + b * 8, 0));
                    if (tile_m < p.row_tiles && tok0 + c * p.CT < p.T) {   // rows beyond d_out and tokens beyond T are clipped by the map
                        asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];"
                                     ::"l"((uint64_t)&tmY), "r"(ysmem), "r"(tile_m * kBM), "r"(tok0 + c * p.CT)
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
}

}  // namespace meteora
