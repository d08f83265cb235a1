// Thin inline-PTX wrappers for sm_100a: mbarrier, TMA (cp.async.bulk.tensor), tcgen05 (MMA, TMEM).
// Every wait is bounded: a wait that runs out records an error code in a global status word
// and in a shared abort flag that all other waits observe, so a protocol bug ends the kernel
// with an error status instead of hanging the GPU.
#pragma once
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>

namespace af {

// Device-global status word: 0 = ok, otherwise (code << 16 | detail) of the first bounded wait that gave up.
// (this library is a single translation unit, so the definition lives here)
static __device__ unsigned int g_device_status = 0;

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// ---------------------------------------------------------------- mbarrier
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Upper bound for any single wait, in SM clock cycles (about one second).
constexpr long long kWaitLimitCycles = 2000000000LL;

// Bounded wait.  Returns false if it gave up (limit reached, or another thread already aborted).
// `abort_flag` lives in shared memory; `code` identifies the wait site.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, volatile uint32_t* abort_flag,
                                          uint32_t code, long long limit_cycles = kWaitLimitCycles) {
    if (mbar_try_wait(bar, parity)) return true;
    long long t0 = clock64();
    uint32_t spins = 0;
    while (true) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((++spins & 63u) == 0u) {
            if (*abort_flag) return false;
            if (clock64() - t0 > limit_cycles) {
                *abort_flag = 1u;
                atomicCAS(&g_device_status, 0u, (code << 16) | (blockIdx.x & 0xffffu));
                return false;
            }
        }
    }
}

// Warp-uniform variant for roles whose warps synchronise internally (__syncwarp, elected arrives,
// warp-collective tcgen05.ld/st): all 32 lanes wait, and all of them give up if any of them did.
// (Letting only lane 0 poll was measured slower: the warp woke up later.)
__device__ __forceinline__ bool mbar_wait_warp(uint64_t* bar, uint32_t parity, volatile uint32_t* abort_flag,
                                               uint32_t code, long long limit_cycles = kWaitLimitCycles) {
    return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag, code, limit_cycles));
}
// The same with one test and one vote in front: a barrier that is complete already costs no per-lane control flow, every other
// one a little more, and every wait some code.  Pays in kernels of several tiles whose chains hide each other's waits
// (one-pass backward at D = 64 702 -> 687 us, B = 16, 8 heads, S = 2213), costs where one chain is all there is: 13.9 -> 14.5 us
// (forward, one query tile, B = 2, 6 / 2 heads, S = 777, window and slopes), 35.2 -> 35.5 us (backward at D = 128 of the same call),
// 390.7 -> 392.1 us (8-bit operands, 8 heads, S = 16384).
template <bool QUICK = true>
__device__ __forceinline__ bool mbar_wait_warp_quick(uint64_t* bar, uint32_t parity, volatile uint32_t* abort_flag, uint32_t code) {
    if (QUICK && __all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
    return mbar_wait_warp(bar, parity, abort_flag, code);
}

// Self-test of the time-out path: one CTA, one barrier that nothing ever arrives on.  Warp 1 waits on it with
// the given (short) limit, gives up, records wait-site code kSelfTestWaitCode and raises the abort flag; warp 0
// waits on the same barrier with the full limit and must be released by the flag.  The kernel then returns
// normally: no trap, no fault, the context stays usable.
constexpr uint32_t kSelfTestWaitCode = 0x7e;
__global__ void wait_timeout_selftest_kernel(long long limit_cycles) {
    __shared__ uint64_t bar;
    __shared__ volatile uint32_t abort_flag;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        abort_flag = 0;
        fence_mbar_init();
    }
    __syncthreads();
    if (threadIdx.x >= 32) mbar_wait_warp(&bar, 0, &abort_flag, kSelfTestWaitCode, limit_cycles);
    else mbar_wait_warp(&bar, 0, &abort_flag, kSelfTestWaitCode + 1);
    __syncthreads();
}

// One lane of a converged warp.  The roles that issue MMAs and TMA copies run with all 32 lanes and guard only the issuing
// instructions with this: control flow and operands then stay warp-uniform, which is what those instructions need
// (their descriptors and addresses live in uniform registers).  A role run by lane 0 alone pays for every operand of
// every MMA: forward without rotation at 32 q / 8 kv heads, S = 16384, D = 128: 2142 -> 1923 us, S = 4096 with rotation
// 169.6 -> 164.0 us, hybrid 188.7 -> 175.6 us (B = 4, S = 2048); one-pass backward 525 -> 508 us (B = 4, 12 heads,
// S = 4096, D = 64), two-kernel backward 653 -> 641 us (B = 4, 32 / 8 heads, S = 2048).
__device__ __forceinline__ bool elect_one() {
    uint32_t r;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(r));
    return r != 0;
}
// A value that is the same in all lanes, in a form the compiler can keep in a uniform register.
template <typename T>
__device__ __forceinline__ T warp_uniform(T v) { return __shfl_sync(0xffffffffu, v, 0); }

// ---------------------------------------------------------------- proxies and fences
__device__ __forceinline__ void fence_proxy_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_before_sync() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after_sync() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// ---------------------------------------------------------------- TMA
// 4-D tiled load: coordinates (c0 innermost .. c3 outermost); completion counted in bytes on `bar`.
__device__ __forceinline__ void tma_load_4d(void* smem_dst, const void* tmap, uint64_t* bar, int c0, int c1,
                                            int c2, int c3) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], "
        "[%2];" ::"r"(smem_u32(smem_dst)),
        "l"(reinterpret_cast<uint64_t>(tmap)), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
        : "memory");
}
// 2-D tiled load (c0 innermost)
__device__ __forceinline__ void tma_load_2d(void* smem_dst, const void* tmap, uint64_t* bar, int c0, int c1) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];" ::"r"(
            smem_u32(smem_dst)),
        "l"(reinterpret_cast<uint64_t>(tmap)), "r"(smem_u32(bar)), "r"(c0), "r"(c1)
        : "memory");
}
__device__ __forceinline__ void tma_store_4d(const void* tmap, const void* smem_src, int c0, int c1, int c2,
                                             int c3) {
    asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%2, %3, %4, %5}], [%1];" ::"l"(
                     reinterpret_cast<uint64_t>(tmap)),
                 "r"(smem_u32(smem_src)), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
                 : "memory");
}
__device__ __forceinline__ void tma_store_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void tma_store_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void tma_store_wait_read() {
    asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}
__device__ __forceinline__ void prefetch_tmap(const void* tmap) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(tmap)) : "memory");
}

// ---------------------------------------------------------------- programmatic dependent launch
// grid_dep_wait: returns once the grids this one depends on have completed and their writes are visible (a
// no-op when the grid was launched without the programmatic-serialization attribute).  grid_dep_launch: lets a
// dependent grid that was launched with that attribute start before this grid has finished.
__device__ __forceinline__ void grid_dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_dep_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// Loads from global memory that stay behind grid_dep_wait.  __ldg (and a const __restrict__ pointer) promises that nothing writes
// the data while the kernel runs, which gives the compiler leave to move the load to the front of the kernel, before
// the wait; and that is where it was seen to move the lists of the block-sparse forward.  Everything that the kernels
// before this one in the stream may have written is therefore read with these: volatile, in the order written.
template <typename T>
__device__ __forceinline__ T ld_words(const uint32_t* w) {
    T v;
    memcpy(&v, w, sizeof(T));
    return v;
}
#define AF_LD_GLOBAL(name, op)                                                                                                    \
    template <typename T>                                                                                                         \
    __device__ __forceinline__ T name(const T* at) {                                                                              \
        static_assert(sizeof(T) == 4 || sizeof(T) == 8 || sizeof(T) == 16, "one load");                                           \
        uint32_t w[sizeof(T) / 4];                                                                                                \
        if constexpr (sizeof(T) == 4) asm volatile("ld.global" op ".b32 %0, [%1];" : "=r"(w[0]) : "l"(at));                       \
        else if constexpr (sizeof(T) == 8) asm volatile("ld.global" op ".v2.b32 {%0, %1}, [%2];" : "=r"(w[0]), "=r"(w[1]) : "l"(at)); \
        else asm volatile("ld.global" op ".v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]) : "l"(at)); \
        return ld_words<T>(w);                                                                                                    \
    }
AF_LD_GLOBAL(ld_global, "")
AF_LD_GLOBAL(ld_global_cs, ".cs")   // read once
AF_LD_GLOBAL(ld_global_cg, ".cg")   // L2 only: written by other CTAs of this grid
#undef AF_LD_GLOBAL
// For data that a loop reads again and again (block lists): `settled` ties a pointer to this point of the program, and
// ld_settled of such a pointer may be moved and shared by the compiler, but not to before it.  (Block-sparse forward with
// its lists read by volatile loads: 395 -> 402 us at B = 4, 12 heads, S = 4096, D = 64, all blocks active.)
template <typename T>
__device__ __forceinline__ const T* settled(const T* p) {
    asm volatile("" : "+l"(p)::"memory");
    return p;
}
__device__ __forceinline__ int ld_settled(const int* at) {
    int v;
    asm("ld.global.b32 %0, [%1];" : "=r"(v) : "l"(at));
    return v;
}

// ---------------------------------------------------------------- TMEM allocation (one warp, converged)
__device__ __forceinline__ void tmem_alloc(uint32_t* smem_result, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(smem_result)),
                 "r"(ncols)
                 : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

// ---------------------------------------------------------------- descriptors
// Instruction descriptor for kind::f16 with bf16 operands and fp32 accumulation.
// a_mn / b_mn: 1 if that operand is MN-major in shared memory (0: K-major).
__host__ __device__ constexpr uint32_t idesc_bf16_f32(int M, int N, int a_mn, int b_mn) {
    return (1u << 4) | (1u << 7) | (1u << 10) | (static_cast<uint32_t>(a_mn) << 15) |
           (static_cast<uint32_t>(b_mn) << 16) | (static_cast<uint32_t>(N >> 3) << 17) |
           (static_cast<uint32_t>(M >> 4) << 24);
}

// Lean forms for the issue loops: the descriptors differ only in their low word (the address field),
// so the caller keeps one high word and adds a constant to the low word per step; ACC is a
// compile-time accumulate flag.  Fewer instructions per MMA matter because the single issuing thread
// competes for issue slots with busy warps on its SM sub-partition.
template <bool ACC>
__device__ __forceinline__ void mma_ss_lo(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t desc_hi, uint32_t idesc) {
    if (ACC)
        asm volatile(
            "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\tmov.b64 da, {%1, %3};\n\tmov.b64 db, {%2, %3};\n\t"
            "setp.eq.b32 p, 0, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p;\n\t}" ::"r"(d_tmem),
            "r"(a_lo), "r"(b_lo), "r"(desc_hi), "r"(idesc)
            : "memory");
    else
        asm volatile(
            "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\tmov.b64 da, {%1, %3};\n\tmov.b64 db, {%2, %3};\n\t"
            "setp.ne.b32 p, 0, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p;\n\t}" ::"r"(d_tmem),
            "r"(a_lo), "r"(b_lo), "r"(desc_hi), "r"(idesc)
            : "memory");
}
// run-time accumulate flag
__device__ __forceinline__ void mma_ss_lo_rt(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t desc_hi, uint32_t idesc,
                                             uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\tmov.b64 da, {%1, %3};\n\tmov.b64 db, {%2, %3};\n\t"
        "setp.ne.b32 p, %5, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p;\n\t}" ::"r"(d_tmem),
        "r"(a_lo), "r"(b_lo), "r"(desc_hi), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void mma_ts_lo(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_lo, uint32_t desc_hi, uint32_t idesc,
                                          uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 db;\n\tmov.b64 db, {%2, %3};\n\tsetp.ne.b32 p, %5, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], db, %4, p;\n\t}" ::"r"(d_tmem),
        "r"(a_tmem), "r"(b_lo), "r"(desc_hi), "r"(idesc), "r"(accumulate)
        : "memory");
}
// Low and high words of a shared-memory matrix descriptor with the 128-byte swizzle (rows of 128 bytes, 8-row atoms of 1024 bytes; the
// tile base must be 1024-byte aligned): address and leading-dimension offset; stride offset, descriptor version 1, swizzle mode 2.
__device__ __forceinline__ uint32_t desc_lo(uint32_t saddr, uint32_t lbo_bytes) {
    return ((saddr & 0x3FFFFu) >> 4) | (((lbo_bytes >> 4) & 0x3FFFu) << 16);
}
__device__ __forceinline__ uint32_t desc_hi(uint32_t sbo_bytes) {
    return ((sbo_bytes >> 4) & 0x3FFFu) | (1u << 14) | (2u << 29);
}
// the same for an operand without swizzle (layout type 0: core matrices of 8 rows x 16 bytes, stored contiguously)
__device__ __forceinline__ uint32_t desc_hi_noswizzle(uint32_t sbo_bytes) {
    return ((sbo_bytes >> 4) & 0x3FFFu) | (1u << 14);
}

// Arrive on `bar` once every MMA issued so far by this thread has completed.
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

// The same from a converged warp.  (elect.sync picks the same lane every time, so the commit sees that lane's MMAs.)
__device__ __forceinline__ void elect_commit(uint64_t* bar) {
    if (elect_one()) mma_commit(bar);
}


// Groups of MMAs issued by one elected lane of a converged warp, each instruction predicated with the election instead of
// standing in a branch.  The offsets between the MMAs of a group are immediates, so that what changes from group to group
// is one add per operand.  A branch around a group cost the forward's issuer 170 cycles from the election to the first MMA
// (re-forming its operands) and 80 for the way out of it, several times per tile.  Together with the waits for K and V in
// front of those for P (see the issuer): 202 -> 195 us (B = 4, 12 heads, S = 4096, D = 64, rotation on chip), 179 -> 171
// us (the same with rotated keys), 1972 -> 1932 us (32 / 8 heads, S = 16384, D = 128, no rotation; under the power cap).
// Scores of one tile pair: D / 16 K steps, both operands K-major with the 128-byte swizzle, 64 columns (16 KB) per box.
#define AF_MMA_SS_STEP(off, acc) \
    "add.u32 a, %1, " #off ";\n\tadd.u32 b, %2, " #off ";\n\tmov.b64 da, {a, %3};\n\tmov.b64 db, {b, %3};\n\t" \
    "@e tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, " acc ";\n\t"
template <int D>
__device__ __forceinline__ void mma_scores(uint32_t d, uint32_t a_lo, uint32_t b_lo, uint32_t hi, uint32_t idesc) {
    if constexpr (D == 128)
        asm volatile("{\n\t.reg .pred e, t, f;\n\t.reg .b64 da, db;\n\t.reg .b32 a, b;\n\telect.sync _|e, 0xffffffff;\n\tsetp.eq.b32 t, 0, 0;\n\tsetp.ne.b32 f, 0, 0;\n\t"
            AF_MMA_SS_STEP(0, "f") AF_MMA_SS_STEP(2, "t") AF_MMA_SS_STEP(4, "t") AF_MMA_SS_STEP(6, "t")
            AF_MMA_SS_STEP(1024, "t") AF_MMA_SS_STEP(1026, "t") AF_MMA_SS_STEP(1028, "t") AF_MMA_SS_STEP(1030, "t") "}"
            ::"r"(d), "r"(a_lo), "r"(b_lo), "r"(hi), "r"(idesc) : "memory");
    else
        asm volatile("{\n\t.reg .pred e, t, f;\n\t.reg .b64 da, db;\n\t.reg .b32 a, b;\n\telect.sync _|e, 0xffffffff;\n\tsetp.eq.b32 t, 0, 0;\n\tsetp.ne.b32 f, 0, 0;\n\t"
            AF_MMA_SS_STEP(0, "f") AF_MMA_SS_STEP(2, "t") AF_MMA_SS_STEP(4, "t") AF_MMA_SS_STEP(6, "t") "}"
            ::"r"(d), "r"(a_lo), "r"(b_lo), "r"(hi), "r"(idesc) : "memory");
}
#define AF_MMA_TS_STEP(aoff, boff, acc) \
    "add.u32 a, %1, " #aoff ";\n\tadd.u32 b, %2, " #boff ";\n\tmov.b64 db, {b, %3};\n\t" \
    "@e tcgen05.mma.cta_group::1.kind::f16 [%0], [a], db, %4, " acc ";\n\t"
// Four K steps (64 keys) of O += P V: P from TMEM (8 columns of bf16 pairs per step), V MN-major (2 KB per step).
__device__ __forceinline__ void mma_pv4(uint32_t d, uint32_t a_tmem, uint32_t b_lo, uint32_t hi, uint32_t idesc, uint32_t acc) {
    asm volatile("{\n\t.reg .pred e, t, f;\n\t.reg .b64 db;\n\t.reg .b32 a, b;\n\telect.sync _|e, 0xffffffff;\n\tsetp.eq.b32 t, 0, 0;\n\tsetp.ne.b32 f, %5, 0;\n\t"
            AF_MMA_TS_STEP(0, 0, "f") AF_MMA_TS_STEP(8, 128, "t") AF_MMA_TS_STEP(16, 256, "t") AF_MMA_TS_STEP(24, 384, "t") "}"
            ::"r"(d), "r"(a_tmem), "r"(b_lo), "r"(hi), "r"(idesc), "r"(acc) : "memory");
}
#undef AF_MMA_SS_STEP
#undef AF_MMA_TS_STEP
// elect_commit without a branch; `bar`: shared-memory address.
__device__ __forceinline__ void commit_elected(uint32_t bar) {
    asm volatile("{\n\t.reg .pred e;\n\telect.sync _|e, 0xffffffff;\n\t@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(bar) : "memory");
}

// ---------------------------------------------------------------- TMEM <-> registers (32 lanes x 32-bit, one row per thread)
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t* r) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,"
        "%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t* r) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t* r) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
        "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,"
        "%29,%30,%31,%32};" ::"r"(taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
        "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]),
        "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]),
        "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
        : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t* r) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
        "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
        "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
        : "memory");
}
// Register budget per warpgroup (all warps of a warpgroup execute the same one).
template <int N>
__device__ __forceinline__ void setmaxnreg_inc() {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N));
}
template <int N>
__device__ __forceinline__ void setmaxnreg_dec() {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N));
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// ---------------------------------------------------------------- thread-block clusters
// All threads of the cluster that have not exited; writes to shared memory before it are visible to the cluster after it.
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// four floats at the same offset of CTA `rank`'s shared memory
__device__ __forceinline__ float4 ld_cluster4(uint32_t saddr, int rank) {
    uint32_t a;
    float4 v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(saddr), "r"(rank));
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a) : "memory");
    return v;
}

__device__ __forceinline__ float2 ld_cluster2(uint32_t saddr, int rank) {
    uint32_t a;
    float2 v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(saddr), "r"(rank));
    asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a) : "memory");
    return v;
}

// four fp32 values added to global memory (16-byte aligned)
__device__ __forceinline__ void red_add4(float* at, float4 v) {
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(at), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}

// ---------------------------------------------------------------- small math helpers
__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// max of three in one instruction (sm_100)
__device__ __forceinline__ float fmax3(float a, float b, float c) {
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}
__device__ __forceinline__ float bf16lo_to_f32(uint32_t u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float bf16hi_to_f32(uint32_t u) { return __uint_as_float(u & 0xffff0000u); }

}  // namespace af
