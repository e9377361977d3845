// Inline-PTX helpers shared by the kernels: mbarriers, bulk copies and the
// tcgen05 tensor-core instructions (TMEM allocation, MMA, commit, loads).
// Every wait on an mbarrier is bounded (kWaitLimitNs) so that a kernel whose
// pipeline stalls reports an error instead of hanging.
#pragma once

#include "common.cuh"

#include <cuda_runtime.h>
#include <stdint.h>

namespace gabp {

constexpr unsigned long long kWaitLimitNs = 2000000000ull;   // bounded waits: 2 s

// Kernels of a round are launched so that each may start while the one before
// it still runs (launch_chained): the next kernel may start from here on ...
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// ... and waits here until the one before it has ended and its writes are seen.
// Every thread of a chained kernel passes it before it reads what a kernel of
// the round writes, and before it leaves.
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ uint32_t smem_u32(const void* ptr)
{
    return (uint32_t)__cvta_generic_to_shared(ptr);
}

// Rounds a dynamic shared-memory pointer up to a multiple of `a` bytes (a
// power of two) by adding an offset to it: the result keeps the provenance of
// the __shared__ array, so the compiler emits shared-memory loads and stores
// through it (a round trip through an integer would leave it a generic
// pointer, and every access through it a generic one).
__device__ __forceinline__ unsigned char* align_smem(unsigned char* raw, uint32_t a)
{
    return raw + ((a - (smem_u32(raw) & (a - 1))) & (a - 1));
}

__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void mbar_init(unsigned long long* bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(unsigned long long* bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void mbar_arrive(unsigned long long* bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(unsigned long long* bar, uint32_t parity)
{
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

// Waits for the phase of `parity` to complete; false after limit_ns.
__device__ __forceinline__ bool mbar_wait(unsigned long long* bar, uint32_t parity,
                                          unsigned long long limit_ns = kWaitLimitNs)
{
    if (mbar_try_wait(bar, parity)) return true;
    const unsigned long long t0 = global_ns();
    while (!mbar_try_wait(bar, parity))
        if (global_ns() - t0 > limit_ns) return false;
    return true;
}

// Warp-uniform bounded wait (every lane takes the same branch afterwards, as
// .sync.aligned instructions and full-mask shuffles need): all lanes test the
// phase and the warp proceeds once every lane has seen it complete; the time
// limit is likewise decided by a vote.  No lane diverges on the fast path.
__device__ __forceinline__ bool mbar_wait_warp(unsigned long long* bar, uint32_t parity)
{
    if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
    const unsigned long long t0 = global_ns();
    for (;;) {
        if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
        if (__any_sync(0xffffffffu, global_ns() - t0 > kWaitLimitNs)) return false;
    }
}

__device__ __forceinline__ uint64_t l2_evict_first_policy()
{
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}

// For data read again by other CTAs of the same launch (node aggregates).
__device__ __forceinline__ uint64_t l2_evict_last_policy()
{
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}

// Bulk copy global -> shared (16-byte aligned addresses, size a multiple of
// 16) completing on `bar` with a transaction count of `bytes`.
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, unsigned long long* bar,
                                          uint64_t pol)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::
            "r"(smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar)), "l"(pol)
        : "memory");
}

// Parity of the last fill of stage s of a ring, `stage` being the one to fill next
// and `phase` the parity of this pass over the ring; of a stage that was never
// filled, the parity that a fresh mbarrier counts as done.
__host__ __device__ constexpr uint32_t last_fill_parity(int s, int stage, uint32_t phase)
{
    return s < stage ? phase : phase ^ 1u;
}
// A producer's last step: every copy that it has issued into its N stages has
// landed (bounded, as every wait), so that none is under way when the CTA's shared
// memory passes on, even where a role has given up and nobody reads them.
template <int N>
__device__ __forceinline__ void await_copies(unsigned long long* full, int stage, uint32_t phase)
{
#pragma unroll
    for (int s = 0; s < N; ++s) mbar_wait(&full[s], last_fill_parity(s, stage, phase));
}

// 1/d for the cavity precisions: the hardware approximate reciprocal
// refined by one Newton-Raphson step r <- r (2 - d r) (error within about one
// unit in the last place for normal positive d; checked against IEEE division
// by gabp_selftest_reciprocal).
__device__ __forceinline__ float rcp_nr(float d)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(d));
    return fmaf(r, fmaf(-d, r, 1.0f), r);
}

// Sums the eight values {x0 .. x7} over the warp in a fixed order:
// afterwards every lane of the group (lane / 4) % 8 = k holds the total of
// value k (nine shuffles).
__device__ __forceinline__ float reduce_scatter8x(const float (&x)[8], int lane)
{
    const bool hi = (lane & 16) != 0;
    float y[4];
#pragma unroll
    for (int k = 0; k < 4; ++k)
        y[k] = (hi ? x[k + 4] : x[k]) + __shfl_xor_sync(0xffffffffu, hi ? x[k] : x[k + 4], 16);
    const bool b8 = (lane & 8) != 0;
    float z[2];
#pragma unroll
    for (int k = 0; k < 2; ++k)
        z[k] = (b8 ? y[k + 2] : y[k]) + __shfl_xor_sync(0xffffffffu, b8 ? y[k] : y[k + 2], 8);
    const bool b4 = (lane & 4) != 0;
    float v = (b4 ? z[1] : z[0]) + __shfl_xor_sync(0xffffffffu, b4 ? z[0] : z[1], 4);
    v += __shfl_xor_sync(0xffffffffu, v, 2);
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    return v;
}

// First error of a kernel -> the instance's control block.
__device__ __forceinline__ void record_error(Ctrl* c, int code, long long where)
{
    if (atomicCAS(&c->status, 0, code) == 0) c->bad_index = where;
}

// ---- tcgen05 (5th-generation tensor cores, TMEM accumulators) -------------
// Allocates `ncols` TMEM columns (power of two >= 32); executed by one whole
// warp; the base address is written to *smem_dst.
__device__ __forceinline__ void tmem_alloc(uint32_t* smem_dst, uint32_t ncols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(smem_dst)),
                 "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Shared-memory matrix descriptor, no swizzle, K-major canonical layout:
// core matrices of 8 rows x 16 bytes stored as contiguous 128-byte blocks;
// lbo = byte distance between core matrices adjacent along K, sbo = along M/N.
__device__ __forceinline__ uint64_t smem_desc(const void* base, uint32_t lbo, uint32_t sbo)
{
    const uint32_t a = smem_u32(base);
    uint64_t d = 0;
    d |= (uint64_t)((a & 0x3FFFFu) >> 4);
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;        // descriptor version for tcgen05
    return d;                      // base offset 0, relative LBO, no swizzle
}

// Instruction descriptor of tcgen05.mma kind::f16: BF16 x BF16 -> FP32,
// both operands K-major, shape M x N.
__host__ __device__ constexpr uint32_t idesc_bf16_f32(int M, int N)
{
    return (1u << 4)                       // D format: F32
           | (1u << 7)                     // A format: BF16
           | (1u << 10)                    // B format: BF16
           | ((uint32_t)(N >> 3) << 17)    // N / 8
           | ((uint32_t)(M >> 4) << 24);   // M / 16
}

// D[tmem] (+)= A[smem] * B[smem]^T, issued by one thread.
__device__ __forceinline__ void tc_mma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                            uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

// Arrives once on `bar` when every tcgen05 operation issued so far by this
// thread has completed.
__device__ __forceinline__ void tc_commit(unsigned long long* bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

// 32 consecutive FP32 columns of one TMEM lane per thread (lanes 32*(warp%4)+t).
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32])
{
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int k = 0; k < 32; ++k) v[k] = __uint_as_float(r[k]);
}

// 16 consecutive FP32 columns of one TMEM lane per thread (lanes 32*(warp%4)+t).
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16])
{
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = __uint_as_float(r[k]);
}

}  // namespace gabp
