// Forward kernel for head dimension 64 and dense masks: four query tiles per CTA, 64 keys at a time.
//   The exponentials are the floor at D = 64: a tile pair has as many as at D = 128 for half the MMA work (2048 cycles of the
// special-function unit for two query tiles x 128 keys, 1.3 k of MMAs).  With two query tiles (fwd_kernel.cuh) that unit idles
// a third of the time, since each tile is a chain scores -> TMEM load -> row maximum -> exponentials -> P V -> next scores
// and two chains do not fill it.  Scores and outputs of four query tiles fit in tensor memory when a step takes 64 keys
// (4 x (64 + 64) columns), and four softmax warps per SM sub-partition keep the unit busy.  K and V are read (and K tiles
// rotated) half as often, too.
//   Sustained, two -> four query tiles: 194 -> 185 us (B = 4, 12 heads, S = 4096, keys rotated on chip), 170 -> 157 us (rotated
// before), 86 -> 75 us (the same with window 256 and ALiBi), 45 -> 37 us (B = 8, S = 1024); all before the reference moved in
// masked blocks (softmax_block64), which costs 1.4 to 1.9 %.  With one issuing warp for all four
// tiles the issuer was the bound (3200 cycles per 64-key step, 188 us); with one per tile the rest of a step is MMAs of 64
// columns, which read their whole A operand for half the work, and the special-function unit.
// Warp roles: warps 0-3 issue the MMAs of a query tile each (warp 0 also all TMA loads), (kRotAll) warps 4-7 rotate the key
// tiles, then one softmax warpgroup per query tile, which first rotates it and in the end writes it out.
#pragma once
#include "fwd_kernel.cuh"

namespace af {

struct Fwd64Smem {
    static constexpr int NQ = 4, KS = 3, VS = 3;
    static constexpr int TILE = 128 * 64 * 2;
    static constexpr int OFF_Q = 0;
    static constexpr int OFF_K = OFF_Q + NQ * TILE;
    static constexpr int OFF_V = OFF_K + KS * TILE;
    static constexpr int OFF_BAR = OFF_V + VS * TILE;
    static constexpr int B_QFULL = 0, B_QROT = B_QFULL + NQ, B_KFULL = B_QROT + NQ, B_KROT = B_KFULL + KS, B_KEMPTY = B_KROT + KS,
                         B_VFULL = B_KEMPTY + KS, B_VEMPTY = B_VFULL + VS, B_SFULL = B_VEMPTY + VS, B_PREADY = B_SFULL + NQ,
                         B_ODONE = B_PREADY + NQ, N_BARS = B_ODONE + NQ;
    static constexpr int OFF_MISC = OFF_BAR + N_BARS * 8;
    static constexpr int BYTES = OFF_MISC + 16 + 1024;   // + alignment slack
};
__host__ __device__ constexpr int fwd64_threads(int rope) { return 128 * (rope == kRotAll ? 6 : 5); }

// 64 keys of the online softmax for one query row (this thread's TMEM lane); see softmax_tile_halves.
// The reference of a row moves when its maximum grows by more than kRescaleThreshold; in masked blocks whenever it grows.  A row's largest
// probability is exact in bf16 where the reference is its own score, and with steps of 64 keys that happened less often than
// with 128: the outputs' error against fp64 was 0.8 % (causal, no mask, window) to 3.2 % (slopes) above that of the kernel for two.
// The masked blocks are the last ones of a causal row, where slopes put the maximum: -0.2 % and -5 % now.  It costs 1.4 % of
// the time (167.7 -> 170.0 us, B = 4, 12 heads, S = 4096) to 1.9 % (B = 8, S = 1024), and gains 2 % with window and slopes.
template <bool MASKED, bool ALIBI>
__device__ __forceinline__ bool softmax_block64(uint32_t tS, uint32_t tO, bool first, float scale_log2, float kb, float bias0, int mlo,
                                                uint32_t mn, uint64_t* s_full, uint64_t* p_ready, uint32_t parity,
                                                volatile uint32_t* abort_flag, int lane, float& m_run, float& l_run) {
    uint32_t v[64];
    if (!mbar_wait_warp_quick(s_full, parity, abort_flag, 80)) return false;
    tc_fence_after_sync();
    tmem_ld32(tS, v);
    tmem_ld32(tS + 32, v + 32);
    tmem_wait_ld();
    float mx4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
    for (int e = 0; e < 64; e += 2) {
        float sv[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            sv[u] = __uint_as_float(v[e + u]);
            if (ALIBI) sv[u] = fmaf(kb, static_cast<float>(e + u), sv[u]);
            if (MASKED) sv[u] = (static_cast<uint32_t>(e + u - mlo) < mn) ? sv[u] : -INFINITY;
            if (ALIBI || MASKED) v[e + u] = __float_as_uint(sv[u]);
        }
        mx4[(e >> 1) & 3] = fmax3(mx4[(e >> 1) & 3], sv[0], sv[1]);
    }
    const float mx = fmaf(fmax3(fmaxf(mx4[0], mx4[1]), mx4[2], mx4[3]), scale_log2, bias0);
    const bool upd = mx > m_run + (MASKED ? 0.f : kRescaleThreshold);
    float alpha = 1.f;
    if (upd) {
        alpha = ex2(m_run - mx);  // m_run = -inf -> 0
        m_run = mx;
    }
    const float sub = bias0 - ((m_run == -INFINITY) ? 0.f : m_run);
    const float2 sc2 = make_float2(scale_log2, scale_log2), sub2 = make_float2(sub, sub);
    float2 ps2[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        uint32_t pk[16];
#pragma unroll
        for (int e = 0; e < 32; e += 2) {
            const float2 t = __ffma2_rn(make_float2(__uint_as_float(v[c * 32 + e]), __uint_as_float(v[c * 32 + e + 1])), sc2, sub2);
            const float2 pe = make_float2(ex2(t.x), ex2(t.y));
            ps2[(e >> 1) & 1] = __fadd2_rn(ps2[(e >> 1) & 1], pe);
            pk[e >> 1] = pack_bf16x2(pe.x, pe.y);
        }
        tmem_st16(tS + c * 16, pk);
    }
    if (!first && __any_sync(0xffffffffu, upd)) {
        // the accumulator must be rescaled before P V is added to it
#pragma unroll 1
        for (int c = 0; c < 2; ++c) {
            uint32_t o[32];
            tmem_ld32(tO + c * 32, o);
            tmem_wait_ld();
#pragma unroll
            for (int e = 0; e < 32; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * alpha);
            tmem_st32(tO + c * 32, o);
        }
    }
    tmem_wait_st();
    tc_fence_before_sync();
    __syncwarp();
    if (lane == 0) mbar_arrive(p_ready);
    l_run = l_run * alpha + ((ps2[0].x + ps2[0].y) + (ps2[1].x + ps2[1].y));
    return true;
}

// heads_per_cta (4, 2 or 1, a divisor of the GQA group): the four query tiles are 4 / heads_per_cta consecutive row blocks of
// that many adjacent heads.
template <int ROPE>
__global__ void __launch_bounds__(fwd64_threads(ROPE), 1)
attn_fwd64_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                  const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_o, const FwdParams p,
                  int heads_per_cta) {
    using L = Fwd64Smem;
    constexpr int D = 64, NQ = L::NQ, TILE = L::TILE, KS = L::KS, VS = L::VS;
    static_assert(KS == VS, "K and V of a key tile share a stage index");
    constexpr bool KROT = ROPE == kRotAll, hybrid = ROPE == kRotQueries;
    constexpr int kSoftmaxWarp = KROT ? 8 : 4;
    constexpr uint32_t TMEM_COLS = 512;
    constexpr uint32_t IDESC_S = idesc_bf16_f32(BM, 64, 0, 0), IDESC_O = idesc_bf16_f32(BM, D, 0, 1);

    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t *sQ = smem + L::OFF_Q, *sK = smem + L::OFF_K, *sV = smem + L::OFF_V;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + L::OFF_BAR);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + L::OFF_MISC);
    volatile uint32_t* abort_flag = reinterpret_cast<volatile uint32_t*>(smem + L::OFF_MISC + 4);

    const int warp = warp_uniform(static_cast<int>(threadIdx.x >> 5)), lane = threadIdx.x & 31;
    if (warp == 0 && elect_one()) {
        prefetch_tmap(&tm_q);
        prefetch_tmap(&tm_k);
        prefetch_tmap(&tm_v);
    }
    const int upb = p.Hq / heads_per_cta;   // units per batch
    const int b = static_cast<int>(blockIdx.x) / upb, h0 = (static_cast<int>(blockIdx.x) - b * upb) * heads_per_cta;
    const int hk = h0 / p.group;
    const int rb0 = (p.n_row_blocks - 1 - static_cast<int>(blockIdx.y)) * (NQ / heads_per_cta);   // heaviest first
    // query tile q: its head, first row, and the 64-key blocks that it sees
    auto head_of = [&](int q) { return h0 + q % heads_per_cta; };
    auto row0_of = [&](int q) { return (rb0 + q / heads_per_cta) * BM; };
    auto block_range = [&](int q, int& lo, int& hi) {
        const int i0 = row0_of(q), ilast = min(i0 + BM - 1, p.S - 1);
        const int hi_row = p.causal ? ilast : (p.window >= 0 ? min(ilast + p.window, p.S - 1) : p.S - 1);
        lo = i0 < p.S ? (p.window >= 0 ? max(0, i0 - p.window) : 0) / 64 : 1;
        hi = i0 < p.S ? hi_row / 64 : 0;   // (no rows: an empty range)
    };
    int n_first, n_last;   // of the CTA: its first query tile has rows, the later ones see later keys
    block_range(0, n_first, n_last);
#pragma unroll
    for (int q = 1; q < NQ; ++q) {
        int lo, hi;
        block_range(q, lo, hi);
        if (hi >= lo) n_last = max(n_last, hi);
    }
    const int j_first = n_first >> 1, n_tiles = (n_last >> 1) - j_first + 1;   // key tiles of 128

    if (warp == 0) {
        for (int i = lane; i < L::N_BARS; i += 32) {
            const bool by_warps = (i >= L::B_QROT && i < L::B_QROT + NQ) || (i >= L::B_KROT && i < L::B_KROT + KS) ||
                                  (i >= L::B_PREADY && i < L::B_PREADY + NQ);
            const bool by_issuers = (i >= L::B_KEMPTY && i < L::B_KEMPTY + KS) || (i >= L::B_VEMPTY && i < L::B_VEMPTY + VS);
            mbar_init(&bars[i], by_warps || by_issuers ? 4 : 1);   // an elected arrive per warp of the warpgroup; a commit per issuer
        }
        if (lane == 0) *abort_flag = 0;
        fence_mbar_init();
        __syncwarp();
        // (the hybrid arm waits for the pass that rotates the keys before its first key tile; its Q, table and outputs are settled
        // before that pass starts)
        if (!hybrid) grid_dep_wait();
        if (elect_one()) {
#pragma unroll
            for (int q = 0; q < NQ; ++q)
                if (row0_of(q) < p.S) {
                    mbar_arrive_expect_tx(&bars[L::B_QFULL + q], TILE);
                    tma_load_4d(sQ + q * TILE, &tm_q, &bars[L::B_QFULL + q], 0, row0_of(q), head_of(q), b);
                }
        }
    }
    if (warp == 1) {
        tmem_alloc(tmem_slot, TMEM_COLS);
        tmem_relinquish();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    constexpr uint32_t tmem_base = 0;   // all of tensor memory
    grid_dep_launch();
    if (!hybrid) grid_dep_wait();

    // 4 x 104 + 64 of 5 x 96 registers per thread slot; with the rotation warpgroup 4 x 88 + 80 + 48 of 6 x 80, which spills (140 bytes
    // per thread stored, 180 loaded): that kernel is left to windows, slopes and callers without scratch memory
    constexpr int kSoftmaxRegs = KROT ? 88 : 104, kLightRegs = KROT ? 48 : 64;
    if (warp < 4) setmaxnreg_dec<kLightRegs>();
    if (warp < NQ) {
        // ------------------------------------------------------------ MMA issuer of query tile `warp`; warp 0 is the TMA producer, too
        // One issuer per query tile: a tile's chain (P ready -> P V, next scores) then waits for nobody else's, the four
        // SM sub-partitions carry a share each, and the warps fetch the same short loop.
        constexpr int B_KREADY = KROT ? L::B_KROT : L::B_KFULL;
        constexpr int B_QREADY = ROPE != kRotNone ? L::B_QROT : L::B_QFULL;
        const int q = warp;
        int lo, hi;
        block_range(q, lo, hi);
        const uint32_t dhi = desc_hi(1024), bar0 = smem_u32(bars);
        const uint32_t q_lo = desc_lo(smem_u32(sQ) + q * TILE, 16), k_lo0 = desc_lo(smem_u32(sK), 16), v_lo0 = desc_lo(smem_u32(sV), BOX_BYTES);
        const uint32_t tS = tmem_base + q * 64, tO = tmem_base + 256 + q * 64;
        auto load = [&](int it) {   // key tile `it` into its stages, which the issuers have handed back
            const int st = it % KS, par = ((it / KS) & 1) ^ 1, j0 = (j_first + it) * 128;
            if (!mbar_wait_warp_quick(&bars[L::B_KEMPTY + st], par, abort_flag, 81)) return false;
            if (elect_one()) {
                mbar_arrive_expect_tx(&bars[L::B_KFULL + st], TILE);
                tma_load_4d(sK + st * TILE, &tm_k, &bars[L::B_KFULL + st], 0, j0, hk, b);
            }
            if (!mbar_wait_warp_quick(&bars[L::B_VEMPTY + st], par, abort_flag, 82)) return false;
            if (elect_one()) {
                mbar_arrive_expect_tx(&bars[L::B_VFULL + st], TILE);
                tma_load_4d(sV + st * TILE, &tm_v, &bars[L::B_VFULL + st], 0, j0, hk, b);
            }
            return true;
        };
        auto run = [&] {   // (returns early when a wait gave up)
            if (warp == 0) {
                if (hybrid) grid_dep_wait();
                for (int it = 0; it < min(KS, n_tiles); ++it) load(it);
            }
            auto issue_S = [&](int n, uint32_t k_lo) {   // 64 keys are 8 KB of a K or V tile
                tc_fence_after_sync();
                mma_scores<D>(tS, q_lo, k_lo + (n & 1) * 512, dhi, IDESC_S);
                commit_elected(bar0 + 8 * (L::B_SFULL + q));
            };
            if (hi >= lo && !mbar_wait_warp_quick(&bars[B_QREADY + q], 0, abort_flag, 84)) return;
            if (!mbar_wait_warp_quick(&bars[B_KREADY], 0, abort_flag, 83)) return;
            if (lo == n_first && hi >= lo) issue_S(n_first, k_lo0);
            if ((n_first & 1) || n_first == n_last) commit_elected(bar0 + 8 * L::B_KEMPTY);
            int st = 0;   // stage of block n's key tile, and the parity of its full barriers
            uint32_t par = 0;
            if (!mbar_wait_warp_quick(&bars[L::B_VFULL], 0, abort_flag, 85)) return;
            for (int n = n_first; n <= n_last; ++n) {
                const bool next = n < n_last, last_half = (n & 1) || !next;
                int st1 = st;
                uint32_t par1 = par;
                if (n & 1) {
                    if (++st1 == KS) st1 = 0, par1 ^= 1;
                    if (next && !mbar_wait_warp_quick(&bars[B_KREADY + st1], par1, abort_flag, 86)) return;
                }
                if (n >= lo && n <= hi) {
                    if (!mbar_wait_warp_quick(&bars[L::B_PREADY + q], (n - lo) & 1, abort_flag, 87)) return;
                    tc_fence_after_sync();
                    mma_pv4(tO, tS, v_lo0 + st * (TILE >> 4) + (n & 1) * 512, dhi, IDESC_O, n > lo ? 1u : 0u);
                }
                if (n + 1 >= lo && n + 1 <= hi) issue_S(n + 1, k_lo0 + st1 * (TILE >> 4));
                if (n == hi) commit_elected(bar0 + 8 * (L::B_ODONE + q));
                if (next && (!(n & 1) || n + 1 == n_last)) commit_elected(bar0 + 8 * (L::B_KEMPTY + st1));
                if (last_half) {
                    commit_elected(bar0 + 8 * (L::B_VEMPTY + st));
                    const int it = (n >> 1) - j_first;
                    // (the stage of the tile before this one)
                    if (warp == 0 && it > 0 && it + KS - 1 < n_tiles && !load(it + KS - 1)) return;
                    if (next && !mbar_wait_warp_quick(&bars[L::B_VFULL + st1], par1, abort_flag, 85)) return;
                }
                st = st1;
                par = par1;
            }
        };
        run();
    } else if (KROT && warp >= 4 && warp < 8) {
        // ------------------------------------------------------------ rotation warpgroup (Section 4.1)
        if constexpr (KROT) {
            const int t = threadIdx.x - 128;
            auto run = [&](auto cp_tag) {
                constexpr int CP = decltype(cp_tag)::value, CPT = CP > 0 ? CP : 1;   // 0: generic path (table read per row)
                bool ok = true;
                RotStep step;
                RotState<CPT> st;
                if (CP > 0) rotate_load_step<CPT>(p.table, p.S, p.R, t, step);
                for (int it = 0; ok && it < n_tiles; ++it) {
                    const int ks = it % KS;
                    if (CP > 0 && (it % kKeyRun) == 0) rotate_prefetch(st, p.table, (j_first + it) * 128, p.S, p.R, t);
                    ok = mbar_wait_warp_quick(&bars[L::B_KFULL + ks], (it / KS) & 1, abort_flag, 88);
                    if (!ok) break;
                    if (CP > 0) rotate_tile_fast(sK + ks * TILE, st, step, t);
                    else rotate_tile_smem(sK + ks * TILE, (j_first + it) * 128, p.S, p.R, p.table, t, 128);
                    fence_proxy_async_smem();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&bars[L::B_KROT + ks]);
                }
            };
            if (p.R == 64) run(std::integral_constant<int, 4>{});
            else if (p.R == 32) run(std::integral_constant<int, 2>{});
            else if (p.R == 16) run(std::integral_constant<int, 1>{});
            else run(std::integral_constant<int, 0>{});
        }
    } else if (warp >= kSoftmaxWarp) {
        // ------------------------------------------------------------ softmax warpgroups (one query row per thread)
        setmaxnreg_inc<kSoftmaxRegs>();
        const int q = (warp - kSoftmaxWarp) >> 2;
        const int row = threadIdx.x - kSoftmaxWarp * 32 - q * 128;   // == TMEM lane
        const int my_h = head_of(q), my_i0 = row0_of(q);
        int my_lo, my_hi;
        block_range(q, my_lo, my_hi);
        const uint32_t lane_addr = static_cast<uint32_t>((warp & 3) * 32) << 16;
        const uint32_t tS = tmem_base + lane_addr + q * 64, tO = tmem_base + lane_addr + 256 + q * 64;
        const int i = my_i0 + row;
        uint8_t* tile = sQ + q * TILE;
        bool ok = true;
        if (ROPE != kRotNone && my_hi >= my_lo) {
            // Section 4.1: the query tile is rotated once, before the key loop
            auto rot_q = [&](auto cp_tag) {
                constexpr int CP = decltype(cp_tag)::value, CPT = CP > 0 ? CP : 1;
                RotStep step;
                RotState<CPT> st;
                if (CP > 0) {
                    rotate_load_step<CPT>(p.table, p.S, p.R, row, step);
                    rotate_prefetch(st, p.table, my_i0, p.S, p.R, row);
                }
                ok = mbar_wait_warp_quick(&bars[L::B_QFULL + q], 0, abort_flag, 89);
                if (!ok) return;
                if (CP > 0) rotate_tile_fast(tile, st, step, row);
                else rotate_tile_smem(tile, my_i0, p.S, p.R, p.table, row, 128);
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) mbar_arrive(&bars[L::B_QROT + q]);
            };
            if (p.R == 64) rot_q(std::integral_constant<int, 4>{});
            else if (p.R == 32) rot_q(std::integral_constant<int, 2>{});
            else if (p.R == 16) rot_q(std::integral_constant<int, 1>{});
            else rot_q(std::integral_constant<int, 0>{});
        }
        const MaskSpec ms{p.S, p.causal, p.window};
        const bool alibi = p.slopes != nullptr;
        const float slope2 = alibi ? p.slopes[my_h] * 1.4426950408889634f : 0.f, kb = slope2 / p.scale_log2;
        float m_run = -INFINITY, l_run = 0.f;
        for (int n = my_lo; ok && n <= my_hi; ++n) {
            const int j0 = n * 64;
            const bool need_mask = j0 + 64 > p.S || (p.causal && j0 + 63 > my_i0) ||
                                   (p.window >= 0 && (my_i0 + BM - 1 - j0 > p.window || (!p.causal && j0 + 63 - my_i0 > p.window))) ||
                                   (!p.causal && n == my_lo + 1);   // (as if masked: for rows without masked blocks, see softmax_block64)
            const float bias0 = slope2 * static_cast<float>(j0 - i);
            int mlo = 0;
            uint32_t mn = 64;
            if (need_mask) kept_keys_of_query(ms, i, j0, mlo, mn);
            uint64_t *sf = &bars[L::B_SFULL + q], *pr = &bars[L::B_PREADY + q];
            const uint32_t parity = (n - my_lo) & 1;
            const bool first = n == my_lo;
            if (alibi) {
                if (need_mask) ok = softmax_block64<true, true>(tS, tO, first, p.scale_log2, kb, bias0, mlo, mn, sf, pr, parity, abort_flag, lane, m_run, l_run);
                else ok = softmax_block64<false, true>(tS, tO, first, p.scale_log2, kb, bias0, mlo, mn, sf, pr, parity, abort_flag, lane, m_run, l_run);
            } else {
                if (need_mask) ok = softmax_block64<true, false>(tS, tO, first, p.scale_log2, kb, bias0, mlo, mn, sf, pr, parity, abort_flag, lane, m_run, l_run);
                else ok = softmax_block64<false, false>(tS, tO, first, p.scale_log2, kb, bias0, mlo, mn, sf, pr, parity, abort_flag, lane, m_run, l_run);
            }
        }
        // epilogue (Section 4.4: save L = m + ln l, while the last product runs)
        const int bh = b * p.Hq + my_h;
        if (ok && my_hi >= my_lo && p.lse && i < p.S)
            p.lse[static_cast<size_t>(bh) * p.S + i] = l_run > 0.f ? (m_run + log2f(l_run)) * 0.6931471805599453f : -INFINITY;
        if (ok && my_hi >= my_lo) ok = mbar_wait_warp_quick(&bars[L::B_ODONE + q], 0, abort_flag, 90);
        if (my_hi >= my_lo) {
            tc_fence_after_sync();
            const float inv = l_run > 0.f ? 1.f / l_run : 0.f;
            if (!p.o_f32) {
                // bf16 output through the query tile's own buffer, which no MMA reads any more, and TMA (rows past S are clipped)
                // (a warp whose wait gave up takes the barrier all the same: the others must not be left alone there)
                if (ok) {
#pragma unroll 1
                    for (int c = 0; c < 2; ++c) {
                        uint32_t v[32];
                        tmem_ld32(tO + c * 32, v);
                        tmem_wait_ld();
#pragma unroll
                        for (int e = 0; e < 32; e += 8)
                            *reinterpret_cast<uint4*>(tile + swz_chunk_offset(row, c * 4 + (e >> 3))) = make_uint4(
                                pack_bf16x2(__uint_as_float(v[e]) * inv, __uint_as_float(v[e + 1]) * inv),
                                pack_bf16x2(__uint_as_float(v[e + 2]) * inv, __uint_as_float(v[e + 3]) * inv),
                                pack_bf16x2(__uint_as_float(v[e + 4]) * inv, __uint_as_float(v[e + 5]) * inv),
                                pack_bf16x2(__uint_as_float(v[e + 6]) * inv, __uint_as_float(v[e + 7]) * inv));
                    }
                    fence_proxy_async_smem();
                }
                asm volatile("bar.sync %0, 128;" ::"r"(4 + q) : "memory");   // this warpgroup only
                if (ok && row == 0) {
                    tma_store_4d(&tm_o, tile, 0, my_i0, my_h, b);
                    tma_store_commit();
                    tma_store_wait_read();   // the buffer must stay in place until it has been read
                }
            } else if (ok) {
                const size_t orow = (static_cast<size_t>(bh) * p.S + i) * D;
#pragma unroll 1
                for (int c = 0; c < 2; ++c) {
                    uint32_t v[32];
                    tmem_ld32(tO + c * 32, v);
                    tmem_wait_ld();
                    if (i < p.S) {
                        float4* dst = reinterpret_cast<float4*>(static_cast<float*>(p.o) + orow + c * 32);
#pragma unroll
                        for (int e = 0; e < 32; e += 4)
                            dst[e >> 2] = make_float4(__uint_as_float(v[e]) * inv, __uint_as_float(v[e + 1]) * inv,
                                                      __uint_as_float(v[e + 2]) * inv, __uint_as_float(v[e + 3]) * inv);
                    }
                }
            }
        }
    }
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 1) {
        __syncwarp();
        tmem_dealloc(tmem_base, TMEM_COLS);
    }
}

}  // namespace af
