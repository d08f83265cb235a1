// Bandwidth-class kernels: the cos/sin table (set-up of Section 4.1) and the separate RoPE pass
// (the pre-rotation arm of Section 5.3).
#pragma once
#include "common.cuh"

namespace af {

// table[s][i] = {cos, sin}((p0 + s) * theta^(-2i/R)); the angle is formed in fp64 so that large
// positions do not lose the fraction of a turn, then rounded to fp32.  One trailer row [S][i] holds
// {cos, sin}(stride * theta^(-2i/R)), the constant the fused kernels use to walk from row to row.
__global__ void rope_table_kernel(float2* __restrict__ table, __nv_bfloat16* __restrict__ table_bf16, int S, int R,
                                  double theta, int p0) {
    const int half = R >> 1;
    const long long idx = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
    if (idx >= static_cast<long long>(S + 1) * half) return;
    const int s = static_cast<int>(idx / half), i = static_cast<int>(idx - static_cast<long long>(s) * half);
    const double freq = pow(theta, -2.0 * static_cast<double>(i) / static_cast<double>(R));
    const double pos = s < S ? static_cast<double>(p0 + s) : static_cast<double>(rope_fast_stride(R));
    double sn, cs;
    sincos(pos * freq, &sn, &cs);
    table[idx] = make_float2(static_cast<float>(cs), static_cast<float>(sn));
    if (s < S) {   // bf16 copy, row layout [R/2 cos | R/2 sin]
        table_bf16[static_cast<size_t>(s) * R + i] = __float2bfloat16_rn(static_cast<float>(cs));
        table_bf16[static_cast<size_t>(s) * R + half + i] = __float2bfloat16_rn(static_cast<float>(sn));
    }
}

// x [B, H, S, D] (element strides xb, xh, xs; D contiguous) -> y [B*H, S, D] contiguous, rows rotated by their position; NH = B * H.  One thread owns the 16-byte chunk pair
// (columns 8cp.., R/2+8cp..) of sequence row s for HPT consecutive heads, so the table entry is
// read once and reused; consecutive threads touch consecutive 16-byte chunks (coalesced).
// Chunks past R are copied when y != x.  sgn = -1 applies the transpose rotation.
// idx: (row, chunk) of this thread, h0: its first head
template <int HPT>
__device__ __forceinline__ void rope_apply_heads(long long idx, int h0, const uint4* x, uint4* y, const float2* __restrict__ table,
                                                 int NH, int H, int S, int D, int R, float sgn, long long xb, long long xh,
                                                 long long xs) {
    const int CP = R >> 4;                 // rotated chunk pairs per row
    const int PT = (D - R) >> 3;           // pass-through chunks per row
    const int per_row = CP + PT;
    if (idx >= static_cast<long long>(S) * per_row) return;
    const int s = static_cast<int>(idx / per_row), c = static_cast<int>(idx - static_cast<long long>(s) * per_row);
    const int row_chunks = D >> 3;
    // 16-byte chunk index of row s of flattened head h in the (possibly strided) input
    auto in_base = [&](int h) {
        return static_cast<size_t>(((h / H) * xb + (h % H) * xh + static_cast<long long>(s) * xs) >> 3);
    };
    if (c < CP) {
        const float4* tb = reinterpret_cast<const float4*>(table + static_cast<size_t>(s) * (R >> 1) + c * 8);
        float4 t0 = ld_global(tb), t1 = ld_global(tb + 1), t2 = ld_global(tb + 2), t3 = ld_global(tb + 3);
        t0.y *= sgn; t0.w *= sgn; t1.y *= sgn; t1.w *= sgn;
        t2.y *= sgn; t2.w *= sgn; t3.y *= sgn; t3.w *= sgn;
        uint4 lo[HPT], hi[HPT];
#pragma unroll
        for (int u = 0; u < HPT; ++u) {
            if (h0 + u < NH) {
                const size_t base = in_base(h0 + u);
                lo[u] = ld_global_cs(x + base + c);
                hi[u] = ld_global_cs(x + base + c + CP);
            }
        }
#pragma unroll
        for (int u = 0; u < HPT; ++u) {
            if (h0 + u < NH) {
                const size_t base = (static_cast<size_t>(h0 + u) * S + s) * row_chunks;
                rotate_word(lo[u].x, hi[u].x, t0.x, t0.y, t0.z, t0.w);
                rotate_word(lo[u].y, hi[u].y, t1.x, t1.y, t1.z, t1.w);
                rotate_word(lo[u].z, hi[u].z, t2.x, t2.y, t2.z, t2.w);
                rotate_word(lo[u].w, hi[u].w, t3.x, t3.y, t3.z, t3.w);
                y[base + c] = lo[u];
                y[base + c + CP] = hi[u];
            }
        }
    } else if (x != y) {
        const int cc = 2 * CP + (c - CP);
#pragma unroll
        for (int u = 0; u < HPT; ++u) {
            if (h0 + u < NH) {
                const size_t base = (static_cast<size_t>(h0 + u) * S + s) * row_chunks;
                y[base + cc] = ld_global_cs(x + in_base(h0 + u) + cc);
            }
        }
    }
}

template <int HPT>
__global__ void __launch_bounds__(256)
rope_apply_kernel(const uint4* x, uint4* y, const float2* __restrict__ table, int NH, int H, int S,
                  int D, int R, float sgn, long long xb, long long xh, long long xs) {
    // programmatic dependent launch, both ways: as a dependent (inside this library's sequences) wait for the
    // predecessor before touching memory; as a predecessor (of the hybrid forward) let the next grid be scheduled
    // and run its set-up while this pass runs
    grid_dep_wait();
    grid_dep_launch();
    rope_apply_heads<HPT>(blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x, blockIdx.y * HPT, x, y, table, NH, H, S, D,
                          R, sgn, xb, xh, xs);
}

// K' = RoPE(K) for the forward kernel, with the bits that its on-chip rotation of a key tile gives (rotate_tile_fast on tiles
// that start at key 0): the cos/sin state of a thread's rows is read from the table at the first tile of a run of kKeyRun
// and walked from there by the same angle-addition steps.  A block takes one key tile of one head; its 128 threads own
// the same chunk pairs and rows as the rotation warpgroup.  The walk to the block's own tile (at most 24 steps of two
// dependent multiply-adds) runs while the loads of the tile's rows are in flight.  R = 16 CP; columns past R are copied.
template <int CP>
__global__ void __launch_bounds__(128)
rope_key_tiles_kernel(const uint4* __restrict__ x, uint4* __restrict__ y, const float2* __restrict__ table, int H, int S, int D,
                      long long xb, long long xh, long long xs) {
    grid_dep_wait();
    grid_dep_launch();   // (the forward kernel may be scheduled; it waits for this grid before its first key tile)
    constexpr int RP = 128 / CP;
    const int t = threadIdx.x, rg = t / CP, cp = t % CP;
    const int tile = blockIdx.x, row0 = tile * BN;
    const int h = blockIdx.y % H;
    const size_t in0 = static_cast<size_t>((blockIdx.y / H * xb + h * xh) >> 3), step_in = static_cast<size_t>(xs >> 3);
    const int chunks = D >> 3;
    const size_t out0 = static_cast<size_t>(blockIdx.y) * S * chunks;
    uint4 lo[CP], hi[CP];
#pragma unroll
    for (int k = 0; k < CP; ++k) {
        const int r = row0 + rg + RP * k;
        if (r < S) {
            lo[k] = ld_global_cs(x + in0 + r * step_in + cp);
            hi[k] = ld_global_cs(x + in0 + r * step_in + cp + CP);
        }
    }
    RotStep step;
    RotState<CP> st;
    rotate_load_step<CP>(table, S, 16 * CP, t, step);
    rotate_prefetch(st, table, tile / kKeyRun * kKeyRun * BN, S, 16 * CP, t);
    auto advance = [&] {
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            const float2 nc = __ffma2_rn(st.s[w], step.ns[w], __fmul2_rn(st.c[w], step.c[w]));
            const float2 nsn = __ffma2_rn(st.c[w], step.s[w], __fmul2_rn(st.s[w], step.c[w]));
            st.c[w] = nc;
            st.s[w] = nsn;
        }
    };
    for (int n = (tile % kKeyRun) * CP; n > 0; --n) advance();
#pragma unroll
    for (int k = 0; k < CP; ++k) {
        const int r = row0 + rg + RP * k;
        rotate_word2(lo[k].x, hi[k].x, st.c[0], st.s[0]);
        rotate_word2(lo[k].y, hi[k].y, st.c[1], st.s[1]);
        rotate_word2(lo[k].z, hi[k].z, st.c[2], st.s[2]);
        rotate_word2(lo[k].w, hi[k].w, st.c[3], st.s[3]);
        advance();
        if (r < S) {
            y[out0 + static_cast<size_t>(r) * chunks + cp] = lo[k];
            y[out0 + static_cast<size_t>(r) * chunks + cp + CP] = hi[k];
        }
    }
    const int rest = chunks - 2 * CP;
    for (int i = t; i < 128 * rest; i += 128) {
        const int r = row0 + i / rest, c = 2 * CP + i % rest;
        if (r < S) y[out0 + static_cast<size_t>(r) * chunks + c] = ld_global_cs(x + in0 + r * step_in + c);
    }
}

}  // namespace af
