// Whole MeteoRA linears (Eq. 2 with Eq. 3) for a prefill batch as ONE launch: persistent pairs of SMs, a tile's epilogue under
// the next tile's main loop, gate and selection as the first tiles.
// Included by wgemm_tcgen05.cu after wgemm_pair.cuh, whose device helpers it uses.
//
// A pair (cluster of two CTAs) computes tiles of 256 rows x BN tokens with tcgen05.mma.cta_group::2, as k_wgemm_pair
// does (each CTA loads its own 128 rows and its own half of the tokens; no load is multicast), but
//   - the pairs stay and walk over the tiles: two accumulators in TMEM (256 columns each), so the MMAs of tile i + 1 run
//     while the epilogue warps round, stage and store tile i;
//   - the first tiles are those of the stacked matrix: pairs of [Wg; a share of A_0..A_{N-1}].  The CTA with Wg's rows selects from
//     its accumulators (top-k, softmax: a thread per token) and hands the routing to its peer, then both write their rows' share of
//     us[t][e r + q] = bf16(w_j (A_e x_t)_q) where token t picked e, else 0, from their accumulators through shared memory
//     and TMA (stores from registers queue behind the tiles' loads: 60 - 75 ns each, 15 us in all).  11 us from the last MMA to the
//     flag at 256 tokens and k = 2, 12 at k = 4, under the next tile's main loop; with compares in a chain and a lane per column of us
//     it was 20 and 29, and the other pairs waited for it;
//   - the LoRA expand is a few more k-steps of the same ring: the contraction goes on over the N r columns of us against
//     the B rows of the tile, both by TMA.  A tile's expand is issued near the end of the NEXT tile's main loop, by
//     which time the selection is ready: nothing waits for the routing (its own
//     main loop's where the routing kernels ran ahead);
//   - where the kernels otherwise taken expand in fp32 (decode batches, few tiles of large ranks: persist_us_parts) us is
//     three bf16 parts whose sum is w_j (A_e x_t)_q exactly: a k-step of the expand is then two stages, (B, part 0) and
//     (part 1, part 2), or on narrow tiles one with all of them, so that B is read once; the routing kernels ahead write the parts.  Such a token's y depends on its
//     own picks alone, also where an adapter that it did not pick holds an infinity or a NaN: 0 times those is NaN, and a
//     NaN of such a row is computed again from the picks.  Against a rounded operand this cost, when a
//     tile's four k-steps took two stages each, 2.1 - 2.3 us (5120 -> 13824 at 200 tokens, where they still do, 37.3 -> 39.4);
//   - modules that share x (q/k/v, gate/up) are one walk: their tiles fill rounds of pairs together.
// Where [Wg; A] has more than 512 rows, or where it saves a round, a launch of gate tiles ahead selects, and the stacked tiles are A's rows alone.
// Where A has more than four pairs take, the batch more stacked tiles than pairs, one round of tiles would become two, or
// us is three parts, the routing kernels ahead write us and only the base product runs here (stacked_pairs = 0).
// What bounds it: the tensor cores under the board's power limit (514 cycles per 64-element k-step and 256 x 256 tile, of
// the 512 that its four MMAs take).  All pairs walk the contraction axis in step, so a line of W0 or x is fetched once for the pairs
// that share it: dealing the last rounds as equal ranges of k-steps instead (partial tiles through L2) took 428 against 415 us
// at 4096 -> 14336, 517 against 477 at 14336 -> 4096 (4096 tokens, sustained load).  The issuing warps stay together and elect a
// lane per k-step: a loop entered by one lane moved every operand to uniform registers by itself, 450 - 530 cycles per step
// (4096 -> 4096 at 64 tokens 29.4 -> 18.7 us, 4096 -> 14336 at 2048 tokens 188 -> 178 us for the walk).
//   warp 0 (both CTAs)  TMA producer; every copy signals the leader's full barrier, which expects both CTAs' bytes.
//   warp 1 (leader)     MMA issue; stages are released and accumulators announced by commits that arrive in both CTAs.
//   warps 2-9 (both)    epilogue: two groups of four warps take turns at chunks of 32 tokens, each with two staging buffers of
//                       its own: TMEM -> bf16 -> shared memory -> TMA store.
// Pairs wait for one another's selection, so with stacked tiles the launch is cooperative (all pairs resident).  Every wait
// is bounded; the pair leaves together.
#pragma once

namespace meteora {

constexpr int kPersistStageBufs = 2;                              // epilogue groups, each with staging buffers of its own
constexpr int kPersistChunk = 32;                                 // tokens an epilogue group takes at a time
constexpr int kPersistBufBytes = kPersistChunk * kBM * 2;         // as rows of bf16
constexpr int kPersistStoreBytes = 2 * kPersistBufBytes;          // a group's staging buffers
constexpr int kPersistAcc2 = 128;                                 // kWalkNarrow: column of a tile's second accumulator
constexpr int kPersistMaxPairs = 74;
constexpr int kPersistMaxN = 64;                                  // adapters the selection here takes
constexpr int kPersistMaxStacked = 4;                             // pairs of stacked tiles per token tile

struct PersistMaps {                                              // per module, then the shared tokens
    CUtensorMap W0[kMaxGroupModules], B[kMaxGroupModules], U[kMaxGroupModules], Y[kMaxGroupModules];
    CUtensorMap S[kMaxGroupModules];                              // us as the stacked tiles store it: 32 columns x 32 tokens
    CUtensorMap A[kMaxGroupModules], A0[kMaxGroupModules], G[kMaxGroupModules];   // A, its rows behind Wg in the first tile, Wg
    CUtensorMap X;
};
struct PersistModule {
    int tile0;                    // its first tile
    int row_pairs, group_pairs;   // group_pairs: row pairs per scheduling group
    const __nv_bfloat16* us;      // [T][parts][64 esteps]
    int32_t* topk_idx;
    float* topk_w;
    const __nv_bfloat16 *W0, *B;  // for the elements that are computed again
    int d_out;
};
struct PersistParams {
    int T, BN;                    // tokens per tile
    int ksteps, esteps;           // main k-steps; expand k-steps (8 blocks of 8 columns each)
    int N, r, k, nblk, cpa;       // N r / 8 blocks, r / 8 blocks per adapter
    int stages, stage_bytes;
    int tr;                       // kWalkNarrow: rows of W0 per CTA and tile, 128 or fewer (whole 8s from 64 up), which spreads a batch over the pairs
    int n_mod, tok_tiles, tiles;
    int stacked_pairs;            // pairs of 128-row tiles, [Wg; a share of A] each (0: us comes from the kernel ahead)
    int gate_rows, us_cols;       // Wg's rows padded to whole 32s (0: the kernel ahead selects); columns of a part of us that are read
    int parts;                    // of us: 1 or 3
    float inv_tau;
    int32_t* flags;               // [module][token tile]: warps whose part of us is written; zero between calls
    int32_t* leave_ctr;           // CTAs that are done with the flags
    int32_t* status;
    int pdl;
    const __nv_bfloat16* x;
    int d_in;
    PersistModule mod[kMaxGroupModules];
};

// 3-D tile load of a pair: the completion bytes go to a barrier that may live in the pair's other CTA.
__device__ __forceinline__ void tma_load_3d_grp(uint32_t dst, const CUtensorMap* tm, int c0, int c1, int c2, uint32_t cluster_bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(dst), "l"((uint64_t)tm), "r"(c0), "r"(c1), "r"(c2), "r"(cluster_bar)
        : "memory");
}
__device__ __forceinline__ uint32_t instr_desc_bf16_pair_n(int bn) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(bn >> 3) << 17) | ((uint32_t)(256 >> 4) << 24);
}

// First row of A in a stacked tile: each pair of tiles has Wg in front, the rest is A's rows in order.  (For the CTA with Wg the
// number counts from the tile's first row: A begins gate_rows behind it.)
__device__ __forceinline__ int persist_first_row(const PersistParams& p, int row_pair, int rank) {
    return row_pair * (2 * kBM - p.gate_rows) + rank * kBM - p.gate_rows;
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

// ---- selection from the logits in shared memory: logit j of the token in slot `tok` of a span of SPAN slots lies at
// s[j * SPAN + (tok ^ (j & 31))], where neither the writers (a lane per logit) nor the readers (a lane per token) meet in a bank.
// A logit as it competes: NaN never wins, -0 is +0.
__device__ __forceinline__ float persist_logit(const float* s, int at) { return fmaxf(s[at], -CUDART_INF_F) + 0.f; }
__device__ __forceinline__ uint32_t persist_key(float v) {        // order-preserving, never 0
    const int bits = __float_as_int(v);
    return (uint32_t)(bits ^ ((bits >> 31) | (int)0x80000000));
}

// The KP largest of 32 distinct keys, descending, in key[0..KP): lists of KP are sorted and merged (bitonic), minima and maxima
// only.  A tree of compares that carries the place along is three instructions per step and again two per key to strike out
// each pick: 5200 cycles for k = 2 and 9000 for k = 4 under a main loop.
template <int KP>
__device__ __forceinline__ void persist_merge(uint32_t (&a)[KP]) {  // bitonic -> descending
#pragma unroll
    for (int d = KP / 2; d > 0; d /= 2)
#pragma unroll
        for (int i = 0; i < KP; ++i)
            if ((i & d) == 0) {
                const uint32_t hi = max(a[i], a[i + d]), lo = min(a[i], a[i + d]);
                a[i] = hi;
                a[i + d] = lo;
            }
}
template <int KP>
__device__ __forceinline__ void persist_largest(uint32_t (&key)[32], uint32_t (&best)[KP]) {
#pragma unroll
    for (int l = 0; l < 32; l += KP) {
        uint32_t a[KP];
#pragma unroll
        for (int i = 0; i < KP; ++i) a[i] = key[l + i];
#pragma unroll
        for (int w = 2; w <= KP; w *= 2)                          // blocks of w, alternately descending and ascending
#pragma unroll
            for (int d = w / 2; d > 0; d /= 2)
#pragma unroll
                for (int i = 0; i < KP; ++i)
                    if ((i & d) == 0) {
                        const uint32_t hi = max(a[i], a[i + d]), lo = min(a[i], a[i + d]);
                        const bool down = w == KP || (i & w) == 0;
                        a[i] = down ? hi : lo;
                        a[i + d] = down ? lo : hi;
                    }
        if (l == 0) {
#pragma unroll
            for (int i = 0; i < KP; ++i) best[i] = a[i];
        } else {
#pragma unroll
            for (int i = 0; i < KP; ++i) best[i] = max(best[i], a[KP - 1 - i]);
            persist_merge<KP>(best);
        }
    }
}

// The picks (a byte each) of one token by LPT adjacent lanes that take 32 logits each, from keys whose low bits are replaced by the
// adapter (inverted: the lower one is the larger key).  `close`: two of the k + 1 largest differ in those bits alone.
template <int LPT, int KP>
__device__ __forceinline__ unsigned long long persist_picks(const float* s, int tok, int half, int N, int k, bool& close) {
    constexpr int SPAN = 128 / LPT;
    constexpr uint32_t low = 32 * LPT - 1;
    uint32_t key[32], best[KP];
#pragma unroll
    for (int i = 0; i < 32; ++i) {
        const int j = half * 32 + i;
        const uint32_t full = persist_key(persist_logit(s, j * SPAN + (tok ^ i)));
        key[i] = j < N ? (full & ~low) | (low - (uint32_t)j) : 0u;
    }
    persist_largest<KP>(key, best);
    if (LPT == 2) {
        uint32_t other[KP];
#pragma unroll
        for (int i = 0; i < KP; ++i) other[i] = __shfl_xor_sync(0xFFFFFFFFu, best[i], 1);
#pragma unroll
        for (int i = 0; i < KP; ++i) best[i] = max(best[i], other[KP - 1 - i]);
        persist_merge<KP>(best);
    }
    unsigned long long picks = 0;
#pragma unroll
    for (int i = 0; i + 1 < KP; ++i)
        if (i < k) {
            picks |= (unsigned long long)(low - (best[i] & low)) << (8 * i);
            close |= ((best[i] ^ best[i + 1]) & ~low) == 0;
        }
    return picks;
}
// The same from whole keys, one compare after the other: ties (the lower adapter first), and k = 8.
template <int LPT>
__device__ __noinline__ unsigned long long persist_picks_exact(const float* s, int tok, int N, int k) {
    unsigned long long picks = 0, taken = 0;
    for (int n = 0; n < k; ++n) {
        uint32_t best = 0;
        int at = 0;
#pragma unroll 1
        for (int j = 0; j < N; ++j) {
            const uint32_t key = (taken >> j) & 1 ? 0u : persist_key(persist_logit(s, j * (128 / LPT) + (tok ^ (j & 31))));
            if (key > best) {
                best = key;
                at = j;
            }
        }
        taken |= 1ull << at;
        picks |= (unsigned long long)at << (8 * n);
    }
    return picks;
}

// Whether 8 packed bf16 hold an infinity or a NaN.
__device__ __forceinline__ bool any_nonfinite(const uint4& v) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
    bool any = false;
#pragma unroll
    for (int i = 0; i < 4; ++i) any |= (w[i] & 0x7F80u) == 0x7F80u || (w[i] & 0x7F800000u) == 0x7F800000u;
    return any;
}

// Element (token, row) of a staged chunk of y: two blocks of [token][64 rows], 128-byte swizzle, or [token][tr rows].
__device__ __forceinline__ int persist_y_at(int tr, int tok, int row) {
    return tr < kBM ? tok * tr + row : ((row >> 6) * kPersistChunk + tok) * 64 + ((((row >> 3) & 7) ^ (tok & 7)) << 3) + (row & 7);
}

// A warp's 32 rows x `nt` tokens of a staged chunk of y in which some element is NaN: those of rows where some
// adapter's B is not finite are computed again as W0 x + the picks' terms.  (A NaN of any other row is the row's own.)  Never
// taken on finite weights; a row with such an entry costs a dot product per token.
__device__ __noinline__ void persist_repair(const PersistParams& p, const PersistModule& mo, __nv_bfloat16* ystage, int tile_row0, int quad,
                                            int tok0, int nt) {
    const int lane = threadIdx.x & 31, row0 = tile_row0 + quad * 32, row = row0 + lane;
    asm volatile("griddepcontrol.wait;" ::: "memory");               // (the producer has waited: this thread may read what it waited for)
    bool odd = false;
    if (quad * 32 + lane < p.tr && row < mo.d_out)
        for (int e = 0; e < p.N; ++e)
            for (int c = 0; c < p.r; c += 8) odd |= any_nonfinite(*reinterpret_cast<const uint4*>(mo.B + ((size_t)e * mo.d_out + row) * p.r + c));
    const int cols = 64 * p.esteps;
    for (int i = 0; i < nt; ++i) {
        unsigned todo = __ballot_sync(0xFFFFFFFFu, odd && __hisnan(ystage[persist_y_at(p.tr, i, quad * 32 + lane)]));
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
            if (lane == src) ystage[persist_y_at(p.tr, i, quad * 32 + lane)] = __float2bfloat16_rn(base + lora);
        }
    }
}

__device__ __forceinline__ void st_cluster_v2(uint32_t cluster_addr, int2 v) {
    asm volatile("st.shared::cluster.v2.b32 [%0], {%1, %2};" ::"r"(cluster_addr), "r"(v.x), "r"(v.y) : "memory");
}
__device__ __forceinline__ void st_cluster_f32(uint32_t cluster_addr, float v) {
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(cluster_addr), "f"(v) : "memory");
}

// 16 lanes x 32 columns of TMEM as accumulator fragments: register 4 b + 2 h + c of lane l holds row l / 4 + 8 h, column
// 8 b + 2 (l % 4) + c.
__device__ __forceinline__ void tmem_ld_frag_issue(uint32_t taddr, uint32_t (&v)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x4.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]), "=r"(v[9]),
          "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr));
}
// Four 8 x 8 blocks of such fragments (bf16, two columns per register), transposed: lane 8 i + j gives where column j of block i goes.
__device__ __forceinline__ void stmatrix_x4_trans(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d)
                 : "memory");
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&v);
}

// Tokens of an epilogue group (chunks grp, grp + 2, ... of 32 tokens) are its slots 0, 1, ...: the tile's column of a slot.
__device__ __forceinline__ int persist_column(const PersistParams& p, int grp, int slot) {
    const int c = slot / kPersistChunk;
    return (grp + 2 * c) * kPersistChunk + slot - c * kPersistChunk;
}

// What a group knows about its 128 slots, in the upper half of its staging buffer (both CTAs of the pair hold the same)
struct PersistRouting {
    unsigned long long picks[128];                                // adapters of a slot's token, a byte each; 0xFF: none, or no such token
    float w[8][128];                                              // [pick][slot]
    float4 spread[4][32];                                         // per warp: weights of 32 tokens for the warp's 4 x 8 columns (< 0: not picked)
};
static_assert(sizeof(PersistRouting) <= kPersistStoreBytes / 2, "routing must fit behind us");

// Selection by the group of four warps whose accumulator has the logits in its first 32 LPT rows, for itself and the pair's peer.
// The k largest logits, descending, equal ones by ascending adapter, and their softmax (Eq. 3).
template <int LPT>
__device__ __forceinline__ void persist_select(const PersistParams& p, float* s_lg, PersistRouting* rt, uint32_t peer_rt, uint32_t taddr,
                                               int grp, int quad, int nslots, int tok0) {
    constexpr int SPAN = 128 / LPT;
    const int lane = threadIdx.x & 31, gtid = quad * 32 + lane, tok = gtid / LPT, half = gtid % LPT;
    unsigned long long picks[LPT];
    float w[LPT][8 / LPT];
#pragma unroll
    for (int sp = 0; sp < LPT; ++sp) {
        const int slot0 = sp * SPAN;
        if (sp > 0) asm volatile("bar.sync %0, 128;" ::"r"(2 + grp) : "memory");
        if (quad < LPT) {                                         // warp-uniform: lane = logit
#pragma unroll 1
            for (int q = 0; q < SPAN && slot0 + q < nslots; q += 32) {
                const uint32_t col = (uint32_t)persist_column(p, grp, slot0 + q);
                uint32_t v[2][16];
                tmem_ld16_issue(taddr + col, v[0]);
                tmem_ld16_issue(taddr + col + 16, v[1]);
                tmem_ld_wait();
#pragma unroll
                for (int i = 0; i < 32; ++i) s_lg[gtid * SPAN + ((q + i) ^ lane)] = __uint_as_float(v[i >> 4][i & 15]);
            }
        }
        asm volatile("bar.sync %0, 128;" ::"r"(2 + grp) : "memory");
        if (slot0 + tok < nslots) {                               // warp-uniform
            bool close = p.k == 8;
            unsigned long long got = 0;
            if (p.k < 4) got = persist_picks<LPT, 4>(s_lg, tok, half, p.N, p.k, close);
            else if (p.k < 8) got = persist_picks<LPT, 8>(s_lg, tok, half, p.N, p.k, close);
            if (__any_sync(0xFFFFFFFFu, close)) got = persist_picks_exact<LPT>(s_lg, tok, p.N, p.k);
            float first = 0.f, sum = 0.f;
#pragma unroll 1
            for (int j = 0; j < p.k; ++j) {
                const int e = (int)(got >> (8 * j)) & 0xFF;
                const float v = persist_logit(s_lg, e * SPAN + (tok ^ (e & 31)));
                if (j == 0) first = v;
                sum += expf((v - first) * p.inv_tau);
            }
#pragma unroll
            for (int i = 0; i < 8 / LPT; ++i)
                if (half + LPT * i < p.k) {
                    const int e = (int)(got >> (8 * (half + LPT * i))) & 0xFF;
                    w[sp][i] = expf((persist_logit(s_lg, e * SPAN + (tok ^ (e & 31))) - first) * p.inv_tau) / sum;
                }
            if (tok0 + persist_column(p, grp, slot0 + tok) >= p.T) got = ~0ull;
            else if (p.k < 8) got |= ~0ull << (8 * p.k);
            picks[sp] = got;
        }
    }
    asm volatile("bar.sync %0, 128;" ::"r"(2 + grp) : "memory");   // all logits read: the routing takes their place
#pragma unroll
    for (int sp = 0; sp < LPT; ++sp) {
        const int slot = sp * SPAN + tok;
        if (slot >= nslots) continue;
        if (half == 0) {
            rt->picks[slot] = picks[sp];
            st_cluster_v2(peer_rt + (uint32_t)(offsetof(PersistRouting, picks) + slot * 8), make_int2((int)(uint32_t)picks[sp], (int)(uint32_t)(picks[sp] >> 32)));
        }
#pragma unroll
        for (int i = 0; i < 8 / LPT; ++i) {
            const int j = half + LPT * i;
            if (j >= p.k) continue;
            rt->w[j][slot] = w[sp][i];
            st_cluster_f32(peer_rt + (uint32_t)(offsetof(PersistRouting, w) + (j * 128 + slot) * 4), w[sp][i]);
        }
    }
    asm volatile("bar.sync %0, 128;" ::"r"(2 + grp) : "memory");
}

// The same from what the kernel ahead selected, by a group of four warps for itself.
__device__ __forceinline__ void persist_load_routing(const PersistParams& p, const PersistModule& mo, PersistRouting* rt, int grp, int quad,
                                                     int nslots, int tok0) {
    const int slot = quad * 32 + (threadIdx.x & 31);
    if (slot < nslots) {
        const int t = tok0 + persist_column(p, grp, slot);
        unsigned long long picks = ~0ull;
        if (t < p.T) {
            picks = p.k < 8 ? ~0ull << (8 * p.k) : 0ull;
#pragma unroll 1
            for (int j = 0; j < p.k; ++j) {
                picks |= (unsigned long long)(__ldcg(mo.topk_idx + (size_t)t * p.k + j) & 0xFF) << (8 * j);
                rt->w[j][slot] = __ldcg(mo.topk_w + (size_t)t * p.k + j);
            }
        }
        rt->picks[slot] = picks;
    }
    asm volatile("bar.sync %0, 128;" ::"r"(2 + grp) : "memory");
}

// What the issuing loops need to know at compile time: read from the parameters in the loops, the rows and k-steps of a stage cost
// 0.4 - 0.8 us of 29 (4096 -> 4096 at 512 tokens).
//   kWalkStacked  the routing in the walk, us rounded        k-steps one by one, 128 rows per CTA
//   kWalkBase     base product behind routing kernels        the same, us in 1 or 3 parts
//   kWalkNarrow   the same, tiles of up to 128 tokens        two k-steps per stage, tr rows per CTA
enum { kWalkStacked = 0, kWalkBase = 1, kWalkNarrow = 2 };

template <int kWalk>
// (one CTA per SM: for more the compiler keeps to 48 or 64 registers, and with the second accumulator the issuing loops spill: + 3 us)
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
k_wgemm_persist(const __grid_constant__ PersistMaps maps, const __grid_constant__ PersistParams p) {
    constexpr bool own = kWalk != kWalkStacked;                   // a tile's expand is in its own main loop
    constexpr int kc = kWalk == kWalkNarrow ? 2 : 1;              // k-steps per stage
    const int tr = kWalk == kWalkNarrow ? p.tr : kBM, parts = kWalk == kWalkStacked ? 1 : p.parts;
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
    // that tile's epilogue to end under the rest (12 k-steps: 4 us).  With the routing ahead a tile gets its own there: at the end
    // its loads and MMAs (3 - 3.5 us for three parts) had nothing to hide under; but not ahead of its main product's first step, which
    // clears the accumulator: behind the loop (mid == iters) where that has one iteration
    const int iters = (p.ksteps + kc - 1) / kc, mid = max(max(iters / 2, iters - 12 / kc), own ? 1 : 0);
    // A short axis reaches that point before the routing is ready, and the loads behind it would wait with it: a pair's first tile then
    // gets its own behind the loop (us, in the loop / behind it: 1024 -> 4096 at 300 tokens 13.9 / 12.6, 2048 -> 2560 at 2048 32.0 / 28.9, 2048 -> 9216 at
    // 64 14.3 / 12.9, 2560 -> 14336 at 128 17.1 / 16.2; from 48 k-steps on it hides less than it waits: 3072 -> 14336 at 64 16.9 / 17.1, 4096 27.0 / 27.8)
    const int mid0 = own && p.ksteps <= 40 ? iters : mid;

    // kWalkNarrow sums the two k-steps of a stage, and every other MMA of the expand, into an accumulator of their own each, 128 columns
    // apart: the tensor cores cut off what they add instead of rounding it, so the error grows with the MMAs into one.  An expand in three
    // parts of a prefill batch, which other kernels did in fp32, has the other two accumulators of the pair, whose only tile this is, to
    // itself.  Error of the fp32 sums against 64 bits (rms over the size of y, which a last few columns make cancel), with the split tiles
    // that short prompts took before / one accumulator / now: 4096 -> 1024 at 512 tokens 2.06e-6 / 4.42e-6 / 2.10e-6, with an expand of rank 16
    // 2.05e-6 / 4.57e-6 / 2.09e-6; 14336 -> 1024 7.85e-6 / 16.2e-6 / 7.84e-6; 1024 -> 1024 4.46e-7 / 9.60e-7 / 4.44e-7.  4096 -> 1024 at 512 tokens
    // takes 14.5 / 14.4 us with one accumulator / two, rank 32 with the expand apart 29.5 / 29.9.
    const bool apart = kc == 2 && parts > 1 && p.tok_tiles > 1 && p.tiles <= npairs;
    const uint32_t expand_odd = kc == 2 && p.nblk > 2 ? kPersistAcc2 : 0;

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
            const uint32_t leader_bars = map_to_cta(bar_base, 0);
            bool waited = !p.pdl;
            // with the selection in the walk x comes from the kernel ahead; else the kernel ahead is this call's routing, which read x
            if (!own && p.gate_rows > 0 && !waited) {
                asm volatile("griddepcontrol.wait;" ::: "memory");
                waited = true;
            }
            auto slot = [&](uint32_t& bar, uint32_t& full, uint32_t& dst) {   // the next free stage; its barrier here and in the leader
                if (round > 0 && !mbar_wait_warp(bar_base + (p.stages + s) * 8, (round & 1) ^ 1)) return false;
                bar = bar_base + s * 8;
                full = leader_bars + s * 8;
                dst = ring + s * p.stage_bytes;
                if (++s == p.stages) {
                    s = 0;
                    ++round;
                }
                return true;
            };
            const uint32_t part = (uint32_t)p.BN / 2 * 128u;      // bytes of half a tile's tokens: of x, of a part of us
            auto expand = [&](const PersistTile& t) {
                if (!own) {                                       // the selection of these tokens
                    const bool there = lane != 0 || wait_counter_slow(p.flags + t.mod * p.tok_tiles + t.tok_tile, 16 * p.stacked_pairs, 100);
                    if (!__all_sync(0xFFFFFFFFu, there)) return false;
                    asm volatile("fence.proxy.async;" ::: "memory");
                } else if (!waited) {
                    asm volatile("griddepcontrol.wait;" ::: "memory");
                    waited = true;
                }
                const int row0 = (t.row_pair * 2 + (int)rank) * tr, tokh = t.tok_tile * p.BN + (int)rank * (p.BN / 2);
                const int here = kc == 1 ? 1 : parts;             // a stage of two k-steps has room for all parts
                uint32_t bar, full, dst;
                for (int i = 0; i < p.esteps; ++i) {
                    if (!slot(bar, full, dst)) return false;
                    const int q0 = i * 8;                         // first of the 8 blocks
                    if (elect_one()) {
                        if (leader) mbar_expect_tx(bar, 2 * ((uint32_t)tr * 128u + (uint32_t)here * part));
                        tma_load_3d_grp(dst, &maps.B[t.mod], 0, p.cpa == 1 ? row0 / 8 : row0, q0 / p.cpa, full);
                        tma_load_2d_pair(dst + kWTileBytes, &maps.U[t.mod], q0 * 8, tokh, full);
                        for (int h = 1; h < here; ++h)
                            tma_load_2d_pair(dst + 2 * kWTileBytes + (uint32_t)(h - 1) * part, &maps.U[t.mod], (h * p.esteps + i) * kBK, tokh, full);
                    }
                    __syncwarp();
                    if (here == parts) continue;
                    if (!slot(bar, full, dst)) return false;
                    if (elect_one()) {                            // the other two parts: one where W0's rows would lie
                        if (leader) mbar_expect_tx(bar, 4 * part);
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
                const uint32_t tx = 2u * kc * ((uint32_t)(t.stacked ? kBM : tr) * 128u + part);
                uint32_t bar, full, dst;
                if (kWalk == kWalkStacked && t.stacked) {
                    // own 128 rows of the stacked matrix: Wg and rows of A behind it, or 128 rows of A (zeros past the end)
                    const CUtensorMap* mW = leader ? &maps.A0[t.mod] : &maps.A[t.mod];
                    const int w_row = persist_first_row(p, t.row_pair, (int)rank) + (leader ? p.gate_rows : 0);
                    const uint32_t w_off = leader ? (uint32_t)p.gate_rows * 128u : 0u;
                    for (int i = 0; i < iters && (ok = slot(bar, full, dst)); ++i) {   // (a pair's first tile: nothing is pending)
                        if (elect_one()) {
                            if (leader) mbar_expect_tx(bar, tx);
                            tma_load_2d_pair(dst + w_off, mW, i * kBK, w_row, full);
                            if (leader && p.gate_rows > 0) tma_load_2d_pair(dst, &maps.G[t.mod], i * kBK, 0, full);
                            tma_load_2d_pair(dst + kWTileBytes, &maps.X, i * kBK, tokh, full);
                        }
                        __syncwarp();
                    }
                } else {
                    const CUtensorMap* mW = &maps.W0[t.mod];
                    const int w_row = row_tile * tr;
                    for (int i = 0; i <= iters; ++i) {
                        if (i == (lin == pair0 ? mid0 : mid) && (pending || own) && !(ok = expand(own ? t : before))) break;
                        if (i == iters || !(ok = slot(bar, full, dst))) break;
                        if (elect_one()) {
                            if (leader) mbar_expect_tx(bar, tx);
                            if (kc == 1) {
                                tma_load_2d_pair(dst, mW, i * kBK, w_row, full);
                                tma_load_2d_pair(dst + kWTileBytes, &maps.X, i * kBK, tokh, full);
                            } else {                              // two k-steps per copy (zeros past the end of the axis)
                                tma_load_3d_grp(dst, mW, 0, w_row, 2 * i, full);
                                tma_load_3d_grp(dst + 2 * kWTileBytes, &maps.X, 0, tokh, 2 * i, full);
                            }
                        }
                        __syncwarp();
                    }
                }
                pending = !t.stacked && !own;
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
            // B's rows in a stage: 16 columns (an MMA) of the CTA's rows every 32 tr bytes, or 2 or 4 such side by side in rows of 64 or
            // 128.  (The MMAs take 128 rows; with fewer the rest is whatever lies behind, in rows of the accumulator that nobody reads)
            const uint64_t b_desc = p.cpa == 1 ? smem_desc_plain(0, tr * 16, 128) : smem_desc_rows(0, 16u * p.cpa);
            const int b_side = p.cpa <= 2 ? 0 : p.cpa == 4 ? 1 : 2;   // log2 of the MMAs side by side
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
                    if (parts > 1 && kc == 2) {
                        db[1] = smem_desc_sw128(wa + 2 * kWTileBytes);
                        db[2] = smem_desc_sw128(wa + 2 * kWTileBytes + (uint32_t)p.BN / 2 * 128u);
                    } else if (parts > 1) {
                        release();
                        if (!next(ua)) return false;
                        db[1] = smem_desc_sw128(ua);
                        db[2] = smem_desc_sw128(ua + kWTileBytes);
                    }
                    const int nm = min(4, (p.nblk - i * 8 + 1) / 2);   // two blocks per MMA: 8-row x 16-byte core matrices, 2 KB per block
                    if (elect_one()) {
#pragma unroll
                        for (int h = 0; h < 3; ++h)
                            if (h < parts)
                                for (int kk = 0; kk < nm; ++kk)
                                    umma_bf16_pair(tmem_base + (apart ? kPairTokens : b * kPairTokens) + (kk & 1) * expand_odd,
                                                   b_desc + ((wa + ((kk >> b_side) * (tr * 32 << b_side)) + (kk & ((1 << b_side) - 1)) * 32) >> 4),
                                                   db[h] + (uint64_t)(kk * 2), idesc, !apart || (i | h | (expand_odd ? kk >> 1 : kk)) != 0);
                        umma_commit_pair(bar_base + (p.stages + first) * 8);
                        if (parts > 1 && kc == 1) umma_commit_pair(bar_base + (p.stages + s) * 8);
                    }
                    __syncwarp();
                    release();
                }
                if (!own && elect_one()) umma_commit_pair(bar_accf + b * 8);
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
                for (int i = 0; i <= iters; ++i) {
                    if (i == (n == 0 ? mid0 : mid) && (pending || own) && !(ok = expand(own ? b : b ^ 1))) break;
                    if (i == iters || !(ok = next(wa))) break;
                    const uint64_t da = smem_desc_sw128(wa), db = smem_desc_sw128(wa + kc * kWTileBytes);
                    if (elect_one()) {
#pragma unroll
                        for (int kk = 0; kk < kBK / kUmmaK; ++kk)
                            umma_bf16_pair(acc, da + (uint64_t)(kk * 2), db + (uint64_t)(kk * 2), idesc, (i | kk) != 0);
                        if (kc == 2) {
                            const uint64_t da2 = da + (uint64_t)(tr * 8), db2 = db + (uint64_t)(p.BN * 4);   // (descriptors count 16 bytes)
#pragma unroll
                            for (int kk = 0; kk < kBK / kUmmaK; ++kk)
                                umma_bf16_pair(acc + kPersistAcc2, da2 + (uint64_t)(kk * 2), db2 + (uint64_t)(kk * 2), idesc, (i | kk) != 0);
                        }
                        umma_commit_pair(bar_base + (p.stages + s) * 8);
                    }
                    __syncwarp();
                    release();
                }
                if (!ok) break;
                pending = lin >= p.mod[0].tile0 && !own;
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
        const int chunks = (p.BN + kPersistChunk - 1) / kPersistChunk;
        __nv_bfloat16* ystage = reinterpret_cast<__nv_bfloat16*>(store_ptr + grp * kPersistStoreBytes);
        const uint32_t ysmem = store + grp * kPersistStoreBytes;
        bool acc_ok = true;
        // A first pass through the chunk code on whatever TMEM holds, results dropped: where a pair has a single tile its epilogue would
        // otherwise fetch the code at the end of the launch, from L2 behind the other pairs' loads (4096 -> 4096 at 512 tokens
        // 29.4 -> 28.7 us, 5120 -> 13824 at 200 42.9 -> 42.4)
        bool dry = own;
        int n = 0;
        for (int lin = dry ? pair0 - npairs : pair0; lin < p.tiles; lin += npairs, n += dry ? 0 : 1, dry = false) {
            const PersistTile t(p, max(lin, 0));
            const int tile_m = t.row_pair * 2 + (int)rank, tok0 = t.tok_tile * p.BN, b = n & 1;
            const PersistModule& mo = p.mod[t.mod];
            // (after an expired wait the rest of the walk only keeps the barriers going)
            if (!dry) acc_ok = __all_sync(0xFFFFFFFFu, acc_ok && mbar_wait(bar_accf + b * 8, (n >> 1) & 1));
            if (!acc_ok && lane == 0) {
                atomicExch(p.status, 1);
                atomicExch(p.status + 3, 5300);
            }
            tc_fence_after();
            const uint32_t taddr = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(b * kPairTokens);
            if (kWalk == kWalkStacked && t.stacked) {
                int32_t* flag = p.flags + t.mod * p.tok_tiles + t.tok_tile;
                // routing of the group's slots in the upper half of the staging buffer, us on its way out in the lower half
                PersistRouting* rt = reinterpret_cast<PersistRouting*>(reinterpret_cast<uint8_t*>(ystage) + kPersistStoreBytes / 2);
                const int nslots = grp < chunks ? (chunks - grp + 1) / 2 * kPersistChunk : 0;
                bool have = true;
                if (p.gate_rows == 0) {
                    asm volatile("griddepcontrol.wait;" ::: "memory");
                    persist_load_routing(p, mo, rt, grp, quad, nslots, tok0);
                } else if (rank == 0) {
                    const uint32_t peer_rt = map_to_cta(ysmem + kPersistStoreBytes / 2, 1);
                    if (p.gate_rows <= 32)
                        persist_select<1>(p, reinterpret_cast<float*>(ystage), rt, peer_rt, taddr, grp, quad, nslots, tok0);
                    else
                        persist_select<2>(p, reinterpret_cast<float*>(ystage), rt, peer_rt, taddr, grp, quad, nslots, tok0);
                    if (elected) mbar_arrive_cluster(map_to_cta(bar_pick + grp * 8, 1));
                } else {
                    have = mbar_wait_cluster(bar_pick + grp * 8, 0);
                }
                if (!have && lane == 0) {
                    atomicExch(p.status, 1);
                    atomicExch(p.status + 4, 5400);
                }
                // the warp's 32 columns of us for 32 tokens at a time: a lane per token spreads its weights over the warp's adapters, a
                // thread takes those of its fragments' 8 tokens, and the block leaves in four transposing stores.  As a lane per column
                // (32 k broadcast loads with two compares each, 32 stores of 2 bytes) a block took 2.0 us for k = 2, 3.0 for k = 4
                const int a0 = persist_first_row(p, t.row_pair, (int)rank) + quad * 32;
                if ((rank == 1 || quad * 32 >= p.gate_rows) && a0 < p.us_cols) {
                    const uint32_t us_smem = ysmem + (uint32_t)quad * 2048u;
                    const int e0 = a0 / p.r, e1 = (a0 + 8) / p.r, e2 = (a0 + 16) / p.r, e3 = (a0 + 24) / p.r;
                    // [token][32 columns], 64-byte swizzle
                    const uint32_t st_addr = us_smem + (uint32_t)(lane & 7) * 64u + (uint32_t)(((lane >> 3) ^ ((lane >> 1) & 3)) * 16);
#pragma unroll 1
                    for (int slot = 0; slot < nslots; slot += 32) {
                        const int col = persist_column(p, grp, slot);
                        const unsigned long long picks = rt->picks[slot + lane];
                        float4 spread = make_float4(-1.f, -1.f, -1.f, -1.f);   // (no weight is negative)
                        bool any = false;
#pragma unroll 1
                        for (int j = 0; j < p.k; ++j) {
                            const int e = (int)(picks >> (8 * j)) & 0xFF;
                            const float w = rt->w[j][slot + lane];
                            if (e == e0) spread.x = w;
                            if (e == e1) spread.y = w;
                            if (e == e2) spread.z = w;
                            if (e == e3) spread.w = w;
                            any |= e >= e0 && e <= e3;
                        }
                        any = __any_sync(0xFFFFFFFFu, any);
                        uint32_t v[2][16];
                        if (any) {
                            tmem_ld_frag_issue(taddr + (uint32_t)col, v[0]);
                            tmem_ld_frag_issue(taddr + (16u << 16) + (uint32_t)col, v[1]);
                            rt->spread[quad][lane] = spread;
                        }
                        if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");   // the store before
                        __syncwarp();
                        if (any) {
                            tmem_ld_wait();
                            auto scaled = [&](float w, int g, int b, int c) {
                                return w < 0.f ? 0.f : w * __uint_as_float(v[g >> 1][4 * b + 2 * (g & 1) + c]);
                            };
#pragma unroll
                            for (int b = 0; b < 4; ++b) {
                                const float4 w0 = rt->spread[quad][8 * b + 2 * (lane & 3)], w1 = rt->spread[quad][8 * b + 2 * (lane & 3) + 1];
                                stmatrix_x4_trans(st_addr + b * 512, pack_bf16(scaled(w0.x, 0, b, 0), scaled(w1.x, 0, b, 1)),
                                                  pack_bf16(scaled(w0.y, 1, b, 0), scaled(w1.y, 1, b, 1)),
                                                  pack_bf16(scaled(w0.z, 2, b, 0), scaled(w1.z, 2, b, 1)),
                                                  pack_bf16(scaled(w0.w, 3, b, 0), scaled(w1.w, 3, b, 1)));
                            }
                        } else {
#pragma unroll
                            for (int i = 0; i < 4; ++i)
                                reinterpret_cast<uint4*>(ystage + quad * 1024)[i * 32 + lane] = make_uint4(0u, 0u, 0u, 0u);
                        }
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic writes -> TMA read
                        __syncwarp();
                        if (lane == 0 && tok0 + col < p.T) {
                            asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];"
                                         ::"l"((uint64_t)&maps.S[t.mod]), "r"(us_smem), "r"(a0), "r"(tok0 + col)
                                         : "memory");
                            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                        }
                    }
                    if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");   // written, not only read out
                }
                if (lane == 0) {                                  // a count per warp
                    __threadfence();
                    atomicAdd(flag, 1);
                }
                tc_fence_before();
                __syncwarp();
                asm volatile("bar.sync %0, 128;" ::"r"(2 + grp) : "memory");
                if (elected) mbar_arrive_cluster(map_to_cta(bar_acce + b * 8, 0));
                if (rank == 0 && t.row_pair == 0 && p.gate_rows > 0) {   // the routing for the caller
#pragma unroll 1
                    for (int i = quad * 32 + lane; i < nslots * p.k; i += 128) {
                        const int j = i / nslots, slot = i - j * nslots, e = (int)(rt->picks[slot] >> (8 * j)) & 0xFF;
                        const size_t dst = (size_t)(tok0 + persist_column(p, grp, slot)) * p.k + j;
                        if (e != 0xFF) {
                            mo.topk_idx[dst] = e;
                            mo.topk_w[dst] = rt->w[j][slot];
                        }
                    }
                }
                continue;
            }
            // a tile of one chunk (32 tokens at the most) is read by the first group alone: the other one owes its arrival all the same
            if (grp >= chunks && elected && !dry) mbar_arrive_cluster(map_to_cta(bar_acce + b * 8, 0));
            // A chunk of y as fragments of 32 tokens x 16 rows, rounded, in two blocks of [token][64 rows] with 128-byte swizzle, or (fewer
            // rows than 128) in rows of tr: four transposing stores per thread instead of 32 of 2 bytes.  Two buffers per group, so that
            // a chunk is made while the one before is read out (4.2 us for 208 tokens as stores of 2 bytes, 3.5 for 256 now)
            const int y_row = quad * 32 + (lane >> 3) * 8;
            const bool y_there = y_row < tr;                    // (rows past tr go to the end of the buffer, which no store reads)
            const uint32_t y_lane = ysmem + (y_there ? (uint32_t)persist_y_at(tr, lane & 7, y_row) * 2u : (uint32_t)(kPersistBufBytes - 128 + (lane & 7) * 16));
            const uint32_t y_step = !y_there ? 0u : tr == kBM ? 1024u : (uint32_t)tr * 16u;   // to the next 8 tokens
            for (int c = grp, half = 0; c < (dry ? min(chunks, 2) : chunks); c += 2, half ^= 1) {
                const int cols = min(kPersistChunk, p.BN - c * kPersistChunk);   // (the last one of a single token tile may be short)
                const uint32_t buf = (uint32_t)half * kPersistBufBytes;
                uint32_t v[2][16];                                // 32 tokens of 16 rows each
                tmem_ld_frag_issue(taddr + (uint32_t)(c * kPersistChunk), v[0]);
                tmem_ld_frag_issue(taddr + (16u << 16) + (uint32_t)(c * kPersistChunk), v[1]);
                uint32_t v2[2][16];                               // the second accumulator's
                if (kc == 2) {
                    tmem_ld_frag_issue(taddr + (uint32_t)(kPersistAcc2 + c * kPersistChunk), v2[0]);
                    tmem_ld_frag_issue(taddr + (16u << 16) + (uint32_t)(kPersistAcc2 + c * kPersistChunk), v2[1]);
                }
                // this buffer's last store has been read out (of the one in between nobody knows)
                if (elected) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
                tmem_ld_wait();
                if (kc == 2) {
#pragma unroll
                    for (int h = 0; h < 2; ++h)
#pragma unroll
                        for (int i = 0; i < 16; ++i) v[h][i] = __float_as_uint(__uint_as_float(v[h][i]) + __uint_as_float(v2[h][i]));
                    if (apart) {
                        uint32_t e[2][2][16];
#pragma unroll
                        for (int q = 0; q < 2; ++q) {
                            tmem_ld_frag_issue(taddr + (uint32_t)(kPairTokens + q * (int)expand_odd + c * kPersistChunk), e[q][0]);
                            tmem_ld_frag_issue(taddr + (16u << 16) + (uint32_t)(kPairTokens + q * (int)expand_odd + c * kPersistChunk), e[q][1]);
                        }
                        tmem_ld_wait();
#pragma unroll
                        for (int h = 0; h < 2; ++h)
#pragma unroll
                            for (int i = 0; i < 16; ++i)
                                v[h][i] = __float_as_uint(__uint_as_float(v[h][i]) +
                                                          (__uint_as_float(e[0][h][i]) + (expand_odd ? __uint_as_float(e[1][h][i]) : 0.f)));
                    }
                }
                const bool last = c + 2 >= chunks;
                if (last) tc_fence_before();                      // this group's last read of the accumulator
                asm volatile("bar.sync %0, 128;" ::"r"(2 + grp) : "memory");
                bool nan = false;
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (8 * i < cols) {
                        float a[8];                               // [8 rows][2 tokens]
#pragma unroll
                        for (int g = 0; g < 8; ++g) {
                            a[g] = __uint_as_float(v[g >> 2][4 * i + (g & 3)]);
                            nan |= a[g] != a[g] && quad * 32 + (g >> 1) * 8 < tr;
                        }
                        stmatrix_x4_trans(y_lane + buf + (uint32_t)i * y_step, pack_bf16(a[0], a[1]), pack_bf16(a[2], a[3]), pack_bf16(a[4], a[5]),
                                          pack_bf16(a[6], a[7]));
                    }
                const int tok = tok0 + c * kPersistChunk;
                if (parts > 1 && __any_sync(0xFFFFFFFFu, nan) && !dry) {
                    __syncwarp();
                    persist_repair(p, mo, ystage + buf / 2, tile_m * tr, quad, tok, min(cols, p.T - tok));
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic writes -> TMA read
                asm volatile("bar.sync %0, 128;" ::"r"(2 + grp) : "memory");
                if (elected && !dry) {
                    if (last) mbar_arrive_cluster(map_to_cta(bar_acce + b * 8, 0));
                    // rows beyond d_out and tokens beyond T are clipped by the map; a group per chunk, also an empty one
                    for (int h = 0; h < (tr == kBM ? 2 : 1) && tok < p.T && tile_m * tr + 64 * h < mo.d_out; ++h)
                        asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];"
                                     ::"l"((uint64_t)&maps.Y[t.mod]), "r"(ysmem + buf + (uint32_t)(h * kPersistChunk * 128)), "r"(tile_m * tr + 64 * h), "r"(tok)
                                     : "memory");
                    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                }
            }
            // (an odd number of chunks: the next tile begins with the same buffer again, so both stores have to be out)
            if (((chunks - grp + 1) / 2) % 2 != 0 && elected) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
        }
        if (elected) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    }
    tc_fence_before();
    __syncwarp();
    cluster_sync();                                               // nobody leaves while the peer may still signal it
    if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
    if (kWalk == kWalkStacked && threadIdx.x == 0) {                // the last CTA to leave readies the flags for the next call
        if (atomicAdd(p.leave_ctr, 1) == (int)gridDim.x - 1) {
            for (int i = 0; i < p.n_mod * p.tok_tiles; ++i) p.flags[i] = 0;
            *p.leave_ctr = 0;
        }
    }
}

}  // namespace meteora
