// Device-side building blocks of the tensor-core convolutions: mbarriers, TMA loads, tcgen05 MMA and tensor memory,
// clusters.  Used by dc_conv_bf16.cu and dc_conv_cluster.cu.
#pragma once
#include <cuda.h>

#include "dc_common.cuh"

namespace {

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// One lane of a converged warp, chosen by the hardware.  The producer and MMA roles run inside `if (elect_one())`: behind
// elect.sync the compiler knows that a single lane of a converged warp is active and issues TMA, MMA and commit
// instructions directly; behind `lane == 0` it does not, and a step of a role's loop (64 channels) took up to twice as long.
__device__ __forceinline__ bool elect_one()
{
    uint32_t p;
    asm volatile("{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\tselp.u32 %0, 1, 0, q;\n\t}" : "=r"(p));
    return p != 0;
}
__device__ __forceinline__ void mbar_init(void* bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(void* bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// Arrival that orders nothing but the barrier itself: used to hand a TMEM accumulator back (its reads are
// ordered by tcgen05.wait::ld + tcgen05.fence), so the arrival need not wait for the epilogue's global stores.
__device__ __forceinline__ void mbar_arrive_relaxed(void* bar)
{
    asm volatile("mbarrier.arrive.relaxed.cta.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// Arrival on a barrier in the other CTA of a pair (addr: shared::cluster address from mapa).
__device__ __forceinline__ void mbar_arrive_remote(uint32_t addr)
{
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(addr) : "memory");
}
__device__ __forceinline__ unsigned long long now_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}
// Barriers and destinations of loads as 32-bit shared-memory addresses: what bounds a role's loop is the instructions that
// one lane can issue, so the loops keep addresses in registers and advance them (RingPos).
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
// Bounded wait: false (with the abort flag and the status word set) when `limit` nanoseconds have passed or another role
// has given up.
__device__ __forceinline__ bool mbar_wait_at(uint32_t bar, uint32_t parity, volatile int* abort_flag, const unsigned long long* limit, int32_t* status)
{
    if (mbar_try(bar, parity)) return true;
    const unsigned long long t0 = now_ns();
    for (uint32_t spin = 1;; ++spin) {
        if (mbar_try(bar, parity)) return true;
        if ((spin & 255u) == 0) {
            if (*abort_flag) return false;
            if (now_ns() - t0 > *limit) {
                *abort_flag = 1;
                atomicExch(status, (int)DC_ERR_TIMEOUT);
                return false;
            }
        }
    }
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* tm, int c0, int c1, int c2, int c3, uint32_t bar)
{
    asm volatile("cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
                 ::"r"(dst), "l"(tm), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3) : "memory");
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* tm, int c0, int c1, uint32_t bar)
{
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
                 ::"r"(dst), "l"(tm), "r"(bar), "r"(c0), "r"(c1) : "memory");
}
__device__ __forceinline__ void bulk_copy(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ void umma_commit_at(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// n (1 to 4) MMAs of K = 16 along a chunk; descriptors as constant upper and running lower halves, astep / bstep per MMA;
// accumulate = 0: the first one overwrites the accumulator.
#define DC_UMMA_CHUNK(name, group)                                                                                                              \
    __device__ __forceinline__ void name(uint32_t d, uint32_t a_lo, uint32_t a_hi, uint32_t a_step, uint32_t b_lo, uint32_t b_hi, uint32_t b_step, \
                                         uint32_t idesc, uint32_t accumulate, int n)                                                            \
    {                                                                                                                                           \
        _Pragma("unroll") for (int k = 0; k < 4; ++k)                                                                                           \
            if (k < n)                                                                                                                          \
                asm volatile("{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\tsetp.ne.b32 p, %6, 0;\n\tmov.b64 da, {%1, %2};\n\tmov.b64 db, {%3, %4};\n\t" \
                             "tcgen05.mma." group ".kind::f16 [%0], da, db, %5, p;\n\t}"                                                        \
                             ::"r"(d), "r"(a_lo + k * a_step), "r"(a_hi), "r"(b_lo + k * b_step), "r"(b_hi), "r"(idesc),                        \
                               "r"(k == 0 ? accumulate : 1u) : "memory");                                                                       \
    }
DC_UMMA_CHUNK(umma_chunk, "cta_group::1")
DC_UMMA_CHUNK(umma_chunk_pair, "cta_group::2")
#undef DC_UMMA_CHUNK
// A ring's running slot: its barrier and its data, advanced by fixed strides and wrapped with the phase.
struct RingPos {
    uint32_t off, data, left, phase;      // barrier offset (8 bytes a slot), data position, slots until the wrap, phase parity
    __device__ __forceinline__ void start(uint32_t data0, uint32_t slots) { off = 0; data = data0; left = slots; phase = 0; }
    __device__ __forceinline__ void next(uint32_t data0, uint32_t slots, uint32_t stride)
    {
        off += 8; data += stride;
        if (--left == 0) { off = 0; data = data0; left = slots; phase ^= 1u; }
    }
};

// K-major operand tile in shared memory.  Swizzled layouts: rows of BK bf16, 8-row groups `sbo`
// bytes apart (lbo unused, 16).  Unswizzled layout (layout_type 0): 8-row x 16-byte core matrices,
// `sbo` bytes apart along M/N and `lbo` bytes apart along K.
__device__ __forceinline__ uint64_t umma_desc(uint32_t saddr, uint32_t sbo, uint32_t layout_type, uint32_t lbo = 16)
{
    uint32_t lo = ((saddr >> 4) & 0x3FFFu) | (((lbo >> 4) & 0x3FFFu) << 16);   // start address, LBO
    uint32_t hi = ((sbo >> 4) & 0x3FFFu) | (1u << 14) | (layout_type << 29);   // SBO, descriptor version 1, swizzle
    return ((uint64_t)hi << 32) | lo;
}
__device__ __forceinline__ void umma_f16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                 ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void umma_commit(void* bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t* r)
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 "
                 "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
                 "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
                   "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
                   "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
                 : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// 16-byte accesses to the epilogue's staging by shared-space address: through a generic pointer they would be
// generic loads and stores, which resolve the address space first and wait on the long-latency scoreboard.
__device__ __forceinline__ void sts128(uint32_t addr, uint32_t x, uint32_t y, uint32_t z, uint32_t w)
{
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(x), "r"(y), "r"(z), "r"(w) : "memory");
}
__device__ __forceinline__ uint4 lds128(uint32_t addr)
{
    uint4 v;
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
    return v;
}
// (acc0 + b0, acc1 + b1) in fp32 (one packed add), then round to nearest even into two bf16; RELU clamps negative
// results to zero in the same conversion (rounding is monotonic, so clamping before or after it gives the same value).
template <bool RELU>
__device__ __forceinline__ uint32_t bias_pack_bf16(uint32_t acc0, uint32_t acc1, float b0, float b1)
{
    uint32_t out;
    if (RELU)
        asm("{\n\t.reg .b64 a, b, d;\n\t.reg .f32 x, y;\n\tmov.b64 a, {%1, %2};\n\tmov.b64 b, {%3, %4};\n\t"
            "add.rn.f32x2 d, a, b;\n\tmov.b64 {x, y}, d;\n\tcvt.rn.relu.bf16x2.f32 %0, y, x;\n\t}"
            : "=r"(out) : "r"(acc0), "r"(acc1), "f"(b0), "f"(b1));
    else
        asm("{\n\t.reg .b64 a, b, d;\n\t.reg .f32 x, y;\n\tmov.b64 a, {%1, %2};\n\tmov.b64 b, {%3, %4};\n\t"
            "add.rn.f32x2 d, a, b;\n\tmov.b64 {x, y}, d;\n\tcvt.rn.bf16x2.f32 %0, y, x;\n\t}"
            : "=r"(out) : "r"(acc0), "r"(acc1), "f"(b0), "f"(b1));
    return out;
}

// a + b (+ ReLU) of eight bf16: fp32 sums, each rounded once (as the add layer's own kernel)
__device__ __forceinline__ uint4 add_bf16x8(uint4 a, uint4 b, int relu)
{
    const uint32_t x[4] = {a.x, a.y, a.z, a.w}, z[4] = {b.x, b.y, b.z, b.w};
    uint32_t r[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        float lo = __uint_as_float(x[k] << 16) + __uint_as_float(z[k] << 16);
        float hi = __uint_as_float(x[k] & 0xffff0000u) + __uint_as_float(z[k] & 0xffff0000u);
        if (relu) { lo = fmaxf(lo, 0.f); hi = fmaxf(hi, 0.f); }
        const __nv_bfloat162 t = __floats2bfloat162_rn(lo, hi);
        r[k] = *(const uint32_t*)&t;
    }
    return make_uint4(r[0], r[1], r[2], r[3]);
}

__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t map_to_cta(const void* p, uint32_t rank)      // shared::cluster address of p in CTA `rank`
{
    uint32_t out;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(out) : "r"(smem_u32(p)), "r"(rank));
    return out;
}
__device__ __forceinline__ void cluster_sync_all()
{
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
}  // namespace
