// Device-side helpers shared by the kernels of libqnn: inline PTX for mbarriers,
// bulk copies and the 5th-generation tensor cores (tcgen05), plus the library's
// device status word.  sm_103a only.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "qnn.h"

namespace qnn {

// A bounded wait gives up after this many SM clock cycles (about two seconds at
// GB300 clocks).  Each mbarrier try_wait may park the thread for a bounded,
// system-defined time, and the hardware wakes it as soon as the phase completes.
constexpr long long kWaitLimitCycles = 4000000000ll;

__device__ __forceinline__ void report(int *status, int code) { atomicCAS(status, 0, code); }

// Programmatic dependent launch: a primary grid lets the next kernel of the
// stream start early (pdl_trigger); that kernel calls pdl_wait before it
// touches the primary's results.  Both are no-ops without such a launch.
// A kernel launched that way releases its successor only after its own wait:
// whatever runs ahead of its wait then knows every launch but its direct
// predecessor to have ended, which is what a prepared image read that early
// relies on (with the release ahead of the wait a chain of short launches let
// the image be read while a launch two before was still writing).
// Nor does such a kernel use __ldg: that load is for data nobody writes while
// the kernel lives, and the direct predecessor may be writing its inputs then.
// It reads them with ld_global, or plainly.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Coherent loads from global memory, kept behind pdl_wait and in their order.
// (The window kernel's filters: with one generic load for both of their places the
// 56 x 56 x 64 layer at batch 256 took 68.3 us instead of 66.5.)
__device__ __forceinline__ uint2 ld_global(const uint2 *p)
{
    uint2 v;
    asm volatile("ld.global.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
    return v;
}
__device__ __forceinline__ uint32_t ld_global(const uint32_t *p)
{
    uint32_t v;
    asm volatile("ld.global.u32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ uint32_t ld_global(const uint16_t *p)
{
    uint16_t v;
    asm volatile("ld.global.u16 %0, [%1];" : "=h"(v) : "l"(p));
    return v;
}

// Launch with programmatic stream serialization: the kernel may start while
// its predecessor in the stream still runs, and calls pdl_wait, then
// pdl_trigger, before it touches global memory.
template <class... Params, class... Args>
cudaError_t launch_pdl(void (*kern)(Params...), unsigned grid, unsigned block, size_t smem, cudaStream_t st,
                       Args... args)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<Params>(args)...);
}

__device__ __forceinline__ uint32_t smem_addr(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// ------------------------------------------------------------------ mbarrier

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void fence_mbar_init()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

__device__ __forceinline__ bool mbar_try_wait_at(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// Warp-collective bounded wait: every lane of a converged warp calls it and
// every lane observes the phase completion itself (so each has the acquire
// ordering of the barrier).  All lanes poll with try_wait, which parks them in
// hardware until the phase completes: a hand-off between warps then takes on
// the order of a hundred cycles, where a single polling lane, a sleep between
// polls or a shuffle of the result each add more.  Returns false on every lane
// (and records QNN_ETIMEOUT in *status) once `limit_cycles` SM cycles pass.
__device__ __forceinline__ bool mbar_wait_warp_at(uint32_t bar, uint32_t parity, int *status,
                                                  long long limit_cycles = kWaitLimitCycles)
{
    // a phase that has completed already costs no clock read
    if (__all_sync(0xffffffffu, mbar_try_wait_at(bar, parity))) return true;
    const long long t0 = clock64();
    while (true) {
        const bool ok = mbar_try_wait_at(bar, parity);
        if (__all_sync(0xffffffffu, ok)) return true;
        if (__any_sync(0xffffffffu, clock64() - t0 > limit_cycles)) {
            if ((threadIdx.x & 31) == 0) report(status, QNN_ETIMEOUT);
            return false;
        }
    }
}

__device__ __forceinline__ bool mbar_wait_warp(uint64_t *bar, uint32_t parity, int *status,
                                               long long limit_cycles = kWaitLimitCycles)
{
    return mbar_wait_warp_at(smem_addr(bar), parity, status, limit_cycles);
}

// The same with the clock read ahead of the first poll, for the general
// tensor-core kernel: with the shortcut above its layers take up to 8 % longer
// (361 images of 10 x 40 x 8 -> 112, 1 x 1: 26.0 us, 24.0 this way; 64 of 14 x 14 x
// 256 -> 256, 3 x 3: 49.2 and 46.7).
__device__ __forceinline__ bool mbar_wait_warp_timed(uint64_t *bar, uint32_t parity, int *status,
                                                     long long limit_cycles = kWaitLimitCycles)
{
    const long long t0 = clock64();
    while (true) {
        const bool ok = mbar_try_wait(bar, parity);
        if (__all_sync(0xffffffffu, ok)) return true;
        if (__any_sync(0xffffffffu, clock64() - t0 > limit_cycles)) {
            if ((threadIdx.x & 31) == 0) report(status, QNN_ETIMEOUT);
            return false;
        }
    }
}

// ------------------------------------------------------------------ bulk copy (TMA, untiled)

// global -> shared copy of `bytes` (multiple of 16, both addresses 16-byte aligned),
// completing as transaction bytes on `bar`.
__device__ __forceinline__ void bulk_g2s(void *smem_dst, const void *gmem_src, uint32_t bytes, uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_addr(smem_dst)),
        "l"(gmem_src), "r"(bytes), "r"(smem_addr(bar))
        : "memory");
}

// Makes this thread's generic-proxy shared-memory writes visible to the async
// proxy (the tensor cores read operands through it).
__device__ __forceinline__ void fence_proxy_async_smem()
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// ------------------------------------------------------------------ tcgen05

__device__ __forceinline__ void tmem_alloc(uint32_t *smem_result, uint32_t ncols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(smem_result)),
                 "r"(ncols)
                 : "memory");
}

__device__ __forceinline__ void tmem_relinquish()
{
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// D[tmem] (+)= A[smem desc] * B[smem desc]^T, kind::f16 (fp16 operands, fp32
// accumulator), and a commit: an arrival on `bar` when every tcgen05 operation
// issued so far has completed.
// Warp-collective forms: every lane of a converged warp executes them and
// elect.sync (full mask, so always the same lane) issues the operation.  The
// loop around them then stays converged, its descriptor arithmetic stays
// warp-uniform, and single-thread issue runs at the shared-memory operand rate
// instead of paying for a divergent region per MMA.
__device__ __forceinline__ void mma_f16_ss_warp(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                                uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p, e;\n\t"
        "elect.sync _|e, 0xffffffff;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}

// As mma_f16_ss_warp with kind::f8f6f4: A and B e4m3 (instruction-descriptor
// format fields 0), K = 32 per MMA, fp32 accumulator.
__device__ __forceinline__ void mma_f8_ss_warp(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                               uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p, e;\n\t"
        "elect.sync _|e, 0xffffffff;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}

// The same two MMAs without a "memory" clobber, for issue loops that read their
// descriptors from shared memory: the compiler may then load the next entries
// while earlier MMAs are being issued.  The MMAs read their operands through
// the async proxy; the issuing warp writes no operand memory, and the volatile
// asm statements (MMAs, commits, barrier waits) keep their relative order.
__device__ __forceinline__ void mma_f16_ss_warp_nc(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                                   uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p, e;\n\t"
        "elect.sync _|e, 0xffffffff;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate));
}

__device__ __forceinline__ void mma_f8_ss_warp_nc(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                                  uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p, e;\n\t"
        "elect.sync _|e, 0xffffffff;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate));
}

__device__ __forceinline__ void mma_commit_warp_at(uint32_t bar)
{
    asm volatile(
        "{\n\t.reg .pred e;\n\t"
        "elect.sync _|e, 0xffffffff;\n\t"
        "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(bar)
        : "memory");
}

__device__ __forceinline__ void mma_commit_warp(uint64_t *bar)
{
    asm volatile(
        "{\n\t.reg .pred e;\n\t"
        "elect.sync _|e, 0xffffffff;\n\t"
        "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(
            smem_addr(bar))
        : "memory");
}

// 32 lanes x 32 bits, 16 consecutive columns per thread.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&v)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr)
        : "memory");
}

__device__ __forceinline__ uint32_t max_u16x2(uint32_t a, uint32_t b)
{
    uint32_t r;
    asm("max.u16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}

// Field-wise unsigned maximum of two words of packed Q-bit values (Q = 8, 4, 2).
// INT-8: the larger halfword has the larger high byte; the low bytes by themselves.
// INT-4: bit 3 of (a | 8) - (b & 7) says whether a's low three bits are not below
// b's (no borrow leaves the field); with the top bits it gives a >= b, spread to
// the field.  INT-2: the high bits' OR, and the low bit of whichever high bit is
// not the smaller one.  5, 8 and 7 operations; a byte-wise maximum (__vmaxu4) takes
// about 20, which made the fused INT-8 pool the slowest part of its layers, and
// INT-2 pooling (four of them on masked words) compute-bound.
template <int BITS>
__device__ __forceinline__ uint32_t max_fields(uint32_t a, uint32_t b)
{
    if (BITS == 8) {
        constexpr uint32_t kEven = 0x00FF00FFu;
        return (max_u16x2(a, b) & ~kEven) | max_u16x2(a & kEven, b & kEven);
    }
    if (BITS == 4) {
        constexpr uint32_t kTop = 0x88888888u;
        const uint32_t low = (a | kTop) - (b & ~kTop);
        const uint32_t ge = ((a & ~b) | (~(a ^ b) & low)) & kTop;
        const uint32_t mask = ge | (ge - (ge >> 3));
        return (a & mask) | (b & ~mask);
    }
    constexpr uint32_t kLow = 0x55555555u;
    const uint32_t ah = a >> 1, bh = b >> 1;
    const uint32_t low = (a & (ah | ~bh)) | (b & (bh | ~ah));
    return ((a | b) & ~kLow) | (low & kLow);
}

__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Writes the same 32-bit value into 16 consecutive columns of this thread's lane.
__device__ __forceinline__ void tmem_st16_fill(uint32_t taddr, uint32_t v)
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
        "{%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1};" ::"r"(taddr),
        "r"(v)
        : "memory");
}

// Writes 16 consecutive columns of this thread's lane.
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&v)[16])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
        "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(taddr),
        "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]),
        "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
        : "memory");
}

__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// 4-column load.
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t (&v)[4])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
                 : "r"(taddr)
                 : "memory");
}

// 8-column forms of the three operations above.
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&v)[8])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                 : "r"(taddr)
                 : "memory");
}

__device__ __forceinline__ void tmem_st8_fill(uint32_t taddr, uint32_t v)
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%1,%1,%1,%1,%1,%1,%1};" ::"r"(taddr), "r"(v)
                 : "memory");
}

__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t (&v)[8])
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(taddr), "r"(v[0]),
                 "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
                 : "memory");
}

// Shared-memory matrix descriptor, K-major, no swizzle.  Core matrices are 8
// rows x 16 bytes stored contiguously (128 B); `lbo` is the byte distance
// between core matrices adjacent in K, `sbo` between core matrices adjacent in
// M/N.  Bits 46-47 hold the descriptor version (1) used by sm_100-family MMAs.
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo)
{
    uint64_t d = 0;
    d |= static_cast<uint64_t>((saddr >> 4) & 0x3FFFu);
    d |= static_cast<uint64_t>((lbo >> 4) & 0x3FFFu) << 16;
    d |= static_cast<uint64_t>((sbo >> 4) & 0x3FFFu) << 32;
    d |= static_cast<uint64_t>(1) << 46;
    return d;  // base offset 0, relative LBO mode, layout type 0 = no swizzle
}

// Instruction descriptor for kind::f16: fp16 A and B, fp32 D, both K-major,
// N in bits 17-22 (N >> 3), M in bits 24-28 (M >> 4).
__host__ __device__ constexpr uint32_t idesc_f16_f32(uint32_t m, uint32_t n)
{
    return (1u << 4)            // D format: f32
           | (0u << 7)          // A format: f16
           | (0u << 10)         // B format: f16
           | ((n >> 3) << 17)   // N
           | ((m >> 4) << 24);  // M
}

}  // namespace qnn
