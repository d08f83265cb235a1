// Flash Decoding (Section 4.2 of the paper): one query position per head against a long KV cache.
//
// Phase 1 (decode_split_kernel): the cache is cut into splits; a CTA takes one split of one kv head
// and computes, for the g query heads of that kv head, a partial (m, l, acc) triple with the online
// softmax.  The g heads are the columns of 8-wide MMA tiles, so K and V are read exactly once per CTA.  Phase 2 merges
// the partials with a log-sum-exp; it runs in the same launch, in the CTA that finishes last for its kv head (a ticket
// counter tells which).
//
// The path is bound by HBM (every K and V byte is read once and used for 4 g flops), so the kernel is
// built around the memory system: each of the 4 warps of a CTA streams its own 32-key tiles through
// its own ring of shared-memory stages with TMA (128-byte swizzle, an mbarrier per stage, no
// CTA-wide synchronisation in the loop), 192 KB in flight per SM.  The two small contractions per
// tile run on the warp-level tensor-core path (mma.sync m16n8k16 with ldmatrix fragments): with at most 16 heads a
// tcgen05 tile of 128 rows would be 7/8 padding, and the arithmetic is far from the bound.
// Timeline of a call at 8 kv heads, 4096 keys, D = 128 (18 splits, L2-cold caches): first tile 1.0 us after the start, two tiles
// per warp 1.2 us, the CTA's partial 0.6 us, fence and ticket 0.9 us, the last CTA's merge 1.6 us.  For short caches
// the parts behind the loop are what matters, so they are written as few dependent memory accesses and little code
// (it runs once per launch, so every instruction is fetched cold).  Replayed graph, before and after the merges were
// rewritten and the heads became the N dimension: 8.5 -> 6.5 us (4096 keys, 32 / 8 heads), 31.1 -> 27.3 us (32768 keys,
// 64 / 8 heads: 4.9 TB/s; the loop alone runs at 7), 26.9 -> 23.2 us (B = 16, 2048 keys), 22.6 -> 14.3 us (64 / 4 heads, 5000).
#pragma once
#include "common.cuh"
#include "ptx.cuh"

namespace af {

struct DecodeParams {
    int B, Hq, Hkv, N, group;   // N: keys in the cache; the query sits at position N - 1
    int window;                 // < 0: none; else keys j >= N - 1 - window are kept
    float scale_log2;           // softmax scale * log2(e)
    const float* slopes;        // Hq ALiBi slopes (bias m_h (j - (N - 1))) or nullptr
    const __nv_bfloat16* q;     // [B, Hq, D]
    float* part_o;              // [B * Hq, n_splits, D]   unnormalised partial outputs
    float* part_ml;             // [B * Hq, n_splits, 2]   running max (log2 units) and sum of each partial
    int n_splits;               // CTAs per (batch, kv head); the kept 32-key tiles are dealt out evenly among them
    // Merge in the same launch: one counter per (batch, kv head), zero before the launch.  The CTA that finishes
    // last for its kv head (it draws the last ticket) merges the partials of the g query heads, in split order,
    // writes o / lse and sets the counter back to zero.
    unsigned int* tickets;
    __nv_bfloat16* o;           // [B, Hq, D]
    float* lse;                 // [B, Hq] or nullptr
};

constexpr int kCombineMaxSplits = 256;
constexpr int kDecBatch = 20;   // partial rows the merging CTA requests at once (one CTA per SM: 18 splits at 8 kv heads)
constexpr int kDecTile = 32;    // keys per warp tile
constexpr int kDecWarps = 4;
constexpr int kDecStages = 3;   // tiles in flight per warp

// Up to here one CTA takes all keys of a kv head: a tile of each warp takes 0.6 us, publishing partials and merging them
// 2.8 us (5.1 us against 5.4 us with four splits and 6.1 us with two at 512 keys).
constexpr int kDecOneSplitKeys = 640;

template <int D>
struct DecodeSmem {
    static constexpr int TILE_BYTES = kDecTile * D * 2;                      // one K or V tile
    static constexpr int WARP_BYTES = kDecStages * 2 * TILE_BYTES;           // [stage][K | V]
    static constexpr int OFF_BAR = kDecWarps * WARP_BYTES;
    static constexpr int OFF_MISC = OFF_BAR + kDecWarps * kDecStages * 8;
    static constexpr int BYTES = OFF_MISC + 16 + 1024;
    static constexpr int PART_STRIDE = D + 4;                                // floats per partial row: acc[D], m, l, padding
    static_assert(16 * PART_STRIDE * 4 <= WARP_BYTES, "the partials of a warp must fit in its stages");
};

// 16-byte chunk `chunk` of key row r in a tile of D/64 boxes [32 rows][64 cols], 128-byte swizzle
__device__ __forceinline__ uint32_t dec_chunk_offset(int r, int chunk) {
    return static_cast<uint32_t>((chunk >> 3) * (kDecTile * 128) + r * 128 + (((chunk & 7) ^ (r & 7)) << 4));
}
__device__ __forceinline__ void ldmatrix_x4(uint32_t addr, uint32_t* r) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t addr, uint32_t* r) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}
// 8x8 matrix of bf16 (a word = two adjacent columns of row lane / 4) -> its transpose in the same layout
__device__ __forceinline__ uint32_t movmatrix_trans(uint32_t v) {
    uint32_t r;
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(r) : "r"(v));
    return r;
}
// D (16x8, fp32) += A (16x16, bf16, row) * B (16x8, bf16, col)
__device__ __forceinline__ void mma_16816(float* d, const uint32_t* a, uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ void dec_accumulate(float4& acc, float& lsum, float4 v, float l, float f) {
    acc.x = fmaf(v.x, f, acc.x);
    acc.y = fmaf(v.y, f, acc.y);
    acc.z = fmaf(v.z, f, acc.z);
    acc.w = fmaf(v.w, f, acc.w);
    lsum = fmaf(l, f, lsum);
}
// four head dims of row `bh` of the output, and its log-sum-exp
template <int D>
__device__ __forceinline__ void dec_store(const DecodeParams& p, size_t bh, int d4, float4 acc, float M, float lsum) {
    const float inv = lsum > 0.f ? 1.f / lsum : 0.f;
    *reinterpret_cast<uint2*>(p.o + bh * D + d4 * 4) =
        make_uint2(pack_bf16x2(acc.x * inv, acc.y * inv), pack_bf16x2(acc.z * inv, acc.w * inv));
    if (d4 == 0 && p.lse) p.lse[bh] = lsum > 0.f ? (M + log2f(lsum)) * 0.6931471805599453f : -INFINITY;
}

// NT: 8-head column tiles, ceil(g / 8).
template <int D, int NT>
__global__ void __launch_bounds__(kDecWarps * 32)
decode_split_kernel(const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v,
                    const DecodeParams p) {
    using L = DecodeSmem<D>;
    constexpr int TILE_BYTES = L::TILE_BYTES;
    constexpr int NBOX = D / 64, KSTEPS = D / 16, MT = kDecTile / 16, DT = D / 16;

    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + L::OFF_BAR);
    volatile uint32_t* abort_flag = reinterpret_cast<volatile uint32_t*>(smem + L::OFF_MISC);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int split = blockIdx.x;
    const int b = static_cast<int>(blockIdx.y) / p.Hkv, hk = static_cast<int>(blockIdx.y) - b * p.Hkv;
    const int qpos = p.N - 1;
    const int jmin = p.window >= 0 ? max(0, qpos - p.window) : 0;   // first kept key
    // tiles wholly before the window are skipped; the others are dealt out evenly (to within one tile)
    const int tile0 = jmin / kDecTile, tiles_all = (p.N + kDecTile - 1) / kDecTile - tile0;
    const int t_lo = static_cast<int>(static_cast<long long>(split) * tiles_all / p.n_splits);
    const int t_hi = static_cast<int>(static_cast<long long>(split + 1) * tiles_all / p.n_splits);
    const int k_lo = (tile0 + t_lo) * kDecTile;
    const int n_tiles = t_hi - t_lo;
    const int nt_tiles = n_tiles > warp ? (n_tiles - warp + kDecWarps - 1) / kDecWarps : 0;   // this warp's tiles

    if (threadIdx.x == 0) {
        for (int i = 0; i < kDecWarps * kDecStages; ++i) mbar_init(&bars[i], 1);
        *abort_flag = 0;
        fence_mbar_init();
    }
    if (lane == 0) {
        prefetch_tmap(&tm_k);
        prefetch_tmap(&tm_v);
    }
    __syncthreads();
    // Programmatic dependent launch: the set-up above overlaps with the end of the previous kernel.  The wait comes before the
    // signal, so that whatever is launched behind this kernel also finds the kernels before it complete.
    grid_dep_wait();
    grid_dep_launch();

    uint8_t* wbase = smem + warp * L::WARP_BYTES;
    uint64_t* wbar = bars + warp * kDecStages;
    auto issue = [&](int i) {   // the i-th tile of this warp into stage i % kDecStages
        if (lane == 0) {
            const int st = i % kDecStages;
            const int key0 = k_lo + kDecTile * (warp + kDecWarps * i);
            uint8_t* dk = wbase + st * 2 * TILE_BYTES;
            mbar_arrive_expect_tx(&wbar[st], 2 * TILE_BYTES);
#pragma unroll
            for (int bx = 0; bx < NBOX; ++bx) {
                tma_load_4d(dk + bx * (kDecTile * 128), &tm_k, &wbar[st], bx * 64, key0, hk, b);
                tma_load_4d(dk + TILE_BYTES + bx * (kDecTile * 128), &tm_v, &wbar[st], bx * 64, key0, hk, b);
            }
        }
    };
#pragma unroll
    for (int i = 0; i < kDecStages; ++i)
        if (nt_tiles > i) issue(i);

    // The heads are the N dimension of both products, S^T = K Q^T and O^T = V^T P^T (keys and head dims are M): 8 heads
    // fill an MMA, where with the heads as rows half of a 16-row tile would be copies for g <= 8.
    // Column c of tile nt of a result belongs to head hk * g + 8 nt + c (columns beyond g repeat heads and are dropped).
    uint32_t qb[NT][KSTEPS][2];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
        const int h = hk * p.group + (nt * 8 + (lane >> 2)) % p.group;
        const uint32_t* qr = reinterpret_cast<const uint32_t*>(p.q + (static_cast<size_t>(b) * p.Hq + h) * D) + (lane & 3);
#pragma unroll
        for (int ks = 0; ks < KSTEPS; ++ks) {
            qb[nt][ks][0] = ld_global(qr + ks * 8);
            qb[nt][ks][1] = ld_global(qr + ks * 8 + 4);
        }
    }
    // this lane's result columns: heads 8 nt + 2 (lane % 4) + {0, 1}
    float slope[NT][2], m[NT][2], l[NT][2];
    float o[NT][DT][4];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            slope[nt][e] = p.slopes ? p.slopes[hk * p.group + (nt * 8 + 2 * (lane & 3) + e) % p.group] * 1.4426950408889634f : 0.f;
            m[nt][e] = -INFINITY;
            l[nt][e] = 0.f;
        }
#pragma unroll
        for (int dt = 0; dt < DT; ++dt) o[nt][dt][0] = o[nt][dt][1] = o[nt][dt][2] = o[nt][dt][3] = 0.f;
    }

    bool ok = true;
    for (int i = 0; i < nt_tiles; ++i) {
        const int st = i % kDecStages;
        const int key0 = k_lo + kDecTile * (warp + kDecWarps * i);
        ok = mbar_wait_warp(&wbar[st], (i / kDecStages) & 1, abort_flag, 40);
        if (!ok) break;
        const uint32_t sk = smem_u32(wbase + st * 2 * TILE_BYTES), sv = sk + TILE_BYTES;
        const int mi = lane >> 3;

        // scores: A = K (16 keys x 16 dims per load), the loads of the next step issued before the MMAs of this one (the
        // asm statements keep their order, so the overlap is written out); two accumulators per tile, for even and odd
        // steps, halve the chain of dependent MMAs
        float s[NT][MT][4], s2[NT][MT][4];
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int mt = 0; mt < MT; ++mt) {
                s[nt][mt][0] = s[nt][mt][1] = s[nt][mt][2] = s[nt][mt][3] = 0.f;
                s2[nt][mt][0] = s2[nt][mt][1] = s2[nt][mt][2] = s2[nt][mt][3] = 0.f;
            }
        uint32_t kf[2][2][MT][4];   // [buffer][even / odd step][16 keys]
        auto load_k = [&](int k2, uint32_t (*dst)[MT][4]) {
#pragma unroll
            for (int u = 0; u < 2; ++u)
#pragma unroll
                for (int mt = 0; mt < MT; ++mt)
                    ldmatrix_x4(sk + dec_chunk_offset(mt * 16 + (mi & 1) * 8 + (lane & 7), (2 * k2 + u) * 2 + (mi >> 1)), dst[u][mt]);
        };
        load_k(0, kf[0]);
#pragma unroll
        for (int k2 = 0; k2 < KSTEPS / 2; ++k2) {
            if (k2 + 1 < KSTEPS / 2) load_k(k2 + 1, kf[(k2 + 1) & 1]);
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                for (int mt = 0; mt < MT; ++mt) {
                    mma_16816(s[nt][mt], kf[k2 & 1][0][mt], qb[nt][2 * k2][0], qb[nt][2 * k2][1]);
                    mma_16816(s2[nt][mt], kf[k2 & 1][1][mt], qb[nt][2 * k2 + 1][0], qb[nt][2 * k2 + 1][1]);
                }
        }
        uint32_t pb[NT][MT][2];   // P^T as B operands
        bool grown = false;
        float f[NT][2];
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            // log2-domain scores with bias and mask: rows = keys lane / 4 (e = 0, 1) and + 8 (e = 2, 3), columns = heads
            float mx[2] = {-INFINITY, -INFINITY};
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int j = key0 + mt * 16 + (lane >> 2) + (e >> 1) * 8;
                    float t = fmaf(s[nt][mt][e] + s2[nt][mt][e], p.scale_log2, slope[nt][e & 1] * static_cast<float>(j - qpos));
                    t = (j < p.N && j >= jmin) ? t : -INFINITY;
                    s[nt][mt][e] = t;
                    mx[e & 1] = fmaxf(mx[e & 1], t);
                }
            float ref[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
#pragma unroll
                for (int off = 4; off < 32; off <<= 1) mx[e] = fmaxf(mx[e], __shfl_xor_sync(0xffffffffu, mx[e], off));
                const float mn = fmaxf(m[nt][e], mx[e]);
                ref[e] = mn == -INFINITY ? 0.f : mn;
                f[nt][e] = ex2(m[nt][e] - ref[e]);   // m = -inf -> 0
                grown = grown || f[nt][e] != 1.f;
                m[nt][e] = mn;
                l[nt][e] *= f[nt][e];
            }
#pragma unroll
            for (int mt = 0; mt < MT; ++mt) {
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    s[nt][mt][e] = ex2(s[nt][mt][e] - ref[e & 1]);
                    l[nt][e & 1] += s[nt][mt][e];   // per-lane partial sums; reduced over the key lanes at the end
                }
                // (keys x heads) -> (heads x keys): the B operand wants a head's adjacent keys in one word
                pb[nt][mt][0] = movmatrix_trans(pack_bf16x2(s[nt][mt][0], s[nt][mt][1]));
                pb[nt][mt][1] = movmatrix_trans(pack_bf16x2(s[nt][mt][2], s[nt][mt][3]));
            }
        }
        if (i > 0 && __any_sync(0xffffffffu, grown)) {   // a new maximum somewhere in the warp
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                for (int dt = 0; dt < DT; ++dt) {
                    o[nt][dt][0] *= f[nt][0];
                    o[nt][dt][1] *= f[nt][1];
                    o[nt][dt][2] *= f[nt][0];
                    o[nt][dt][3] *= f[nt][1];
                }
        }
        // O^T += V^T P^T: A = V^T (16 dims x 16 keys per load, transposed on the way), again one step ahead
        uint32_t vf[2][MT][4];
        auto load_v = [&](int dt, uint32_t (*dst)[4]) {
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
                ldmatrix_x4_trans(sv + dec_chunk_offset(mt * 16 + (mi >> 1) * 8 + (lane & 7), dt * 2 + (mi & 1)), dst[mt]);
        };
        load_v(0, vf[0]);
#pragma unroll
        for (int dt = 0; dt < DT; ++dt) {
            if (dt + 1 < DT) load_v(dt + 1, vf[(dt + 1) & 1]);
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                for (int nt = 0; nt < NT; ++nt) mma_16816(o[nt][dt], vf[dt & 1][mt], pb[nt][mt][0], pb[nt][mt][1]);
        }
        __syncwarp();
        if (i + kDecStages < nt_tiles) {
            fence_proxy_async_smem();   // the stage was read through the generic proxy; TMA writes it next
            issue(i + kDecStages);
        }
    }

    // Merge the four warps' partials and write one partial per head.  A warp's partials go to its own stages (idle now):
    // row h = (acc[D], m, l) of query head h.
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
#pragma unroll
            for (int off = 4; off < 32; off <<= 1) l[nt][e] += __shfl_xor_sync(0xffffffffu, l[nt][e], off);
            const int h = nt * 8 + 2 * (lane & 3) + e;
            if (h < p.group) {
                float* row = reinterpret_cast<float*>(wbase) + h * L::PART_STRIDE;
#pragma unroll
                for (int dt = 0; dt < DT; ++dt) {
                    row[dt * 16 + (lane >> 2)] = o[nt][dt][e];
                    row[dt * 16 + (lane >> 2) + 8] = o[nt][dt][e + 2];
                }
                if (lane < 4) *reinterpret_cast<float2*>(row + D) = make_float2(m[nt][e], l[nt][e]);
            }
        }
    __syncthreads();
    if (*abort_flag) return;
    // one thread per (head, four head dims): every load is independent of the others
    constexpr int D4 = D / 4;
    const size_t bh0 = static_cast<size_t>(b) * p.Hq + hk * p.group;
    for (int idx = threadIdx.x; idx < p.group * D4; idx += kDecWarps * 32) {
        const int h = idx / D4, d4 = idx - h * D4;
        const float* row = reinterpret_cast<const float*>(smem) + h * L::PART_STRIDE;
        float2 ml[kDecWarps];
        float4 v[kDecWarps];
#pragma unroll
        for (int w = 0; w < kDecWarps; ++w) {
            ml[w] = *reinterpret_cast<const float2*>(row + w * (L::WARP_BYTES / 4) + D);
            v[w] = *reinterpret_cast<const float4*>(row + w * (L::WARP_BYTES / 4) + d4 * 4);
        }
        const float M = fmaxf(fmaxf(ml[0].x, ml[1].x), fmaxf(ml[2].x, ml[3].x));
        const float ref = M == -INFINITY ? 0.f : M;
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        float lsum = 0.f;
#pragma unroll
        for (int w = 0; w < kDecWarps; ++w) dec_accumulate(acc, lsum, v[w], ml[w].y, ex2(ml[w].x - ref));   // m = -inf -> 0
        if (p.n_splits == 1) {
            dec_store<D>(p, bh0 + h, d4, acc, M, lsum);
        } else {
            const size_t at = (bh0 + h) * p.n_splits + split;
            *reinterpret_cast<float4*>(p.part_o + at * D + d4 * 4) = acc;
            if (d4 == 0) *reinterpret_cast<float2*>(p.part_ml + at * 2) = make_float2(M, lsum);
        }
    }
    if (p.n_splits == 1) return;

    // ---- phase 2 in the same launch (Section 4.2: log-sum-exp combine of the partials).  Every CTA publishes its
    // partials (fence), then draws a ticket; the CTA with the last ticket of its kv head sees all of them.  The sums
    // run over the splits in index order whichever CTA is last, so the result is run-to-run deterministic.
    __shared__ int s_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned int t = atomicAdd(p.tickets + blockIdx.y, 1u);
        s_last = (t == static_cast<unsigned int>(p.n_splits) - 1u) ? 1 : 0;
        if (s_last) p.tickets[blockIdx.y] = 0u;   // ready for the next call on this workspace
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    // The last CTA is a chain of memory latencies, so it makes as few of them as it can: a group of D / 4 lanes (one per
    // four head dims) takes a head, requests up to kDecBatch partial rows at once beside the statistics of all splits
    // (one lane per split), and only then forms the weights, which it hands round by shuffles.
    constexpr int GROUPS = 32 / D4 > 0 ? 32 / D4 : 1, LANES = D4;   // heads per warp, lanes per head
    static_assert(LANES == 32 || LANES == 16, "a head's four-dim columns are a warp or half of one");
    const int n = p.n_splits, gl = lane % LANES, gbase = lane - gl;
    for (int h0w = warp * GROUPS; h0w < p.group; h0w += kDecWarps * GROUPS) {   // (uniform over the warp)
        const int h = min(h0w + lane / LANES, p.group - 1);
        const float4* po = reinterpret_cast<const float4*>(p.part_o + (bh0 + h) * n * D) + gl;
        const float2* pm = reinterpret_cast<const float2*>(p.part_ml) + (bh0 + h) * n;
        constexpr int ROUNDS = (kDecBatch + LANES - 1) / LANES;   // statistics per lane and batch
        float4 v[kDecBatch];
        float2 ml[ROUNDS];
        auto load_batch = [&](int s0) {   // (short straight code: every instruction of this part is fetched cold)
#pragma unroll
            for (int r = 0; r < ROUNDS; ++r)
                ml[r] = (r * LANES + gl < kDecBatch && s0 + r * LANES + gl < n) ? ld_global_cg(pm + s0 + r * LANES + gl) : make_float2(-INFINITY, 0.f);
#pragma unroll
            for (int u = 0; u < kDecBatch; ++u)   // (no row beyond the last: zero, since its weight of zero does not cancel an infinity)
                v[u] = s0 + u < n ? ld_global_cg(po + static_cast<size_t>(s0 + u) * D4) : make_float4(0.f, 0.f, 0.f, 0.f);
        };
        load_batch(0);
        float M = ml[0].x;
#pragma unroll
        for (int r = 1; r < ROUNDS; ++r) M = fmaxf(M, ml[r].x);
        for (int s = kDecBatch + gl; s < n; s += LANES) M = fmaxf(M, ld_global_cg(pm + s).x);
#pragma unroll
        for (int off = LANES / 2; off > 0; off >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, off));
        const float ref = M == -INFINITY ? 0.f : M;
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        float lsum = 0.f;
        for (int s0 = 0; s0 < n; s0 += kDecBatch) {
            if (s0 > 0) load_batch(s0);
            float f[ROUNDS];
#pragma unroll
            for (int r = 0; r < ROUNDS; ++r) f[r] = ex2(ml[r].x - ref);   // m = -inf, or no such split -> 0
#pragma unroll
            for (int u = 0; u < kDecBatch; ++u)
                dec_accumulate(acc, lsum, v[u], __shfl_sync(0xffffffffu, ml[u / LANES].y, gbase + u % LANES),
                               __shfl_sync(0xffffffffu, f[u / LANES], gbase + u % LANES));
        }
        if (h0w + lane / LANES < p.group) dec_store<D>(p, bh0 + h, gl, acc, M, lsum);
    }
}

}  // namespace af
