// Blackwell (sm_100 family) building blocks written as inline PTX:
// mbarriers with bounded waits, TMA tensor loads, tcgen05 MMA / TMEM access,
// and the shared-memory / instruction descriptors the MMA consumes.
//
// Shared-memory operand layout used throughout: 128-byte swizzle ("SW128").
// A tile of R rows x 64 bf16 (128 B per row) is stored as 8-row atoms of
// 1024 B; within an atom the 16-byte chunk c of row r sits at chunk
// c ^ (r & 7).  TMA writes exactly this layout when its tensor map uses
// CU_TENSOR_MAP_SWIZZLE_128B and the destination is 1024-byte aligned.
#pragma once

#include <cuda.h>
#include <stdint.h>

namespace rola {
namespace tc {

// ------------------------------------------------------------------ timers / status

__device__ __forceinline__ uint64_t globaltimer_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

// ------------------------------------------------------------------ mbarrier

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init()
{
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n.reg .pred p;\n"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        "selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// Waits for the phase with the given parity to complete.  Gives up after
// `limit_ns` (or at once when *abort is set by another warp), sets *abort and
// returns false; the caller then records a timeout and winds down.  Pass a
// private zero flag to wait on time alone (used to drain in-flight copies).
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort, uint64_t limit_ns)
{
    if (mbar_try_wait(bar, parity)) return true;
    const uint64_t t0 = globaltimer_ns();
    for (uint32_t i = 1;; ++i) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((i & 63) == 0) {
            if (*abort) return false;
            if (globaltimer_ns() - t0 > limit_ns) {
                *abort = 1;
                return false;
            }
        }
    }
}

// True in one thread of a converged warp.  The branch it guards is known to run
// with a single thread, so the operands of TMA and MMA instructions inside it
// go to uniform registers directly; under `lane == 0` each of them is wrapped
// in a loop over the active lanes (measured around one TMA load: 35 cycles
// here, 80 under `lane == 0`).
__device__ __forceinline__ bool elect_one()
{
    uint32_t r;
    asm volatile(
        "{\n.reg .pred p;\n"
        "elect.sync _|p, 0xffffffff;\n"
        "selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(r));
    return r != 0;
}

// ------------------------------------------------------------------ work items of a persistent CTA

// The items of a persistent, warp-specialised CTA: the first is the CTA's own index, the
// others come off a counter in global memory, so that SMs that run slower (they differ by
// some per cent) or meet longer items take fewer: dealt out evenly, the CTAs of the sparse
// kernels waited 2.6 % of their time for the last one at the 720p layer, 3-7 % at the
// 12-head 480p layer (forward 900 -> 880 us, training step 4.01 -> 3.94 ms).  One producer thread fetches them ahead
// and posts them in a ring of shared-memory slots; the other roles read them there, and a
// slot is written again once all of them have.  So a role that waits inside an item keeps
// the items kRing further on from everyone: what it waits for may depend on the item after
// its own (the producer posts that before it works on this one) and on no later one.
struct ItemRing {
    static constexpr int kRing = 16;
    static constexpr int kReaders = 11;      // the other producer, two more single-thread or one-warp roles, eight warps
    int32_t item[kRing];
    uint64_t full[kRing], empty[kRing];
    __device__ static uint32_t at(uint64_t* b) { return static_cast<uint32_t>(__cvta_generic_to_shared(b)); }
    __device__ void init()
    {
        for (int i = 0; i < kRing; ++i) {
            mbar_init(at(&full[i]), 1);
            mbar_init(at(&empty[i]), kReaders);
        }
    }
    // Makes x the CTA's i-th item (one thread).
    __device__ bool post(int i, int x, volatile int* abort, uint64_t limit_ns)
    {
        const int slot = i % kRing;
        if (i >= kRing && !mbar_wait(at(&empty[slot]), (i / kRing - 1) & 1, abort, limit_ns)) return false;
        item[slot] = x;
        mbar_arrive(at(&full[slot]));
        return true;
    }
    // The CTA's i-th item (a number past the last once there is none); ok goes false, and the
    // result past any item, if it does not come.  For a whole warp, or one thread (`single`).
    template <bool kSingle>
    __device__ int get(int i, bool& ok, volatile int* abort, uint64_t limit_ns)
    {
        const int slot = i % kRing;
        ok = mbar_wait(at(&full[slot]), (i / kRing) & 1, abort, limit_ns);
        const int x = ok ? *reinterpret_cast<volatile int32_t*>(&item[slot]) : 0x7fffffff;
        if constexpr (!kSingle) __syncwarp();
        if (kSingle || (threadIdx.x & 31) == 0) mbar_arrive(at(&empty[slot]));
        return x;
    }
};

// ------------------------------------------------------------------ TMA

__device__ __forceinline__ void tma_prefetch_desc(const void* map)
{
    asm volatile("prefetch.tensormap [%0];\n" ::"l"(map) : "memory");
}

// 3-D tiled load; coordinates (x innermost).  x * 2 bytes must be a multiple of 16.
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const void* map, uint32_t bar, int x, int y, int z)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], "
        "[%2];\n" ::"r"(dst),
        "l"(map), "r"(bar), "r"(x), "r"(y), "r"(z)
        : "memory");
}

// 4-D tiled load; coordinates (x innermost).
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const void* map, uint32_t bar, int x, int y, int z, int w)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], "
        "[%2];\n" ::"r"(dst),
        "l"(map), "r"(bar), "r"(x), "r"(y), "r"(z), "r"(w)
        : "memory");
}

// 4-D tiled store from shared memory (bulk-group completion); coordinates
// (x innermost), none negative.  Rows past the tensor's extent are not written.
__device__ __forceinline__ void tma_store_4d(const void* map, uint32_t src, int x, int y, int z, int w)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%2, %3, %4, %5}], [%1];\n" ::"l"(map),
        "r"(src), "r"(x), "r"(y), "r"(z), "r"(w)
        : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;\n" ::: "memory"); }
// Waits until this thread's committed bulk stores have finished reading shared memory.
__device__ __forceinline__ void bulk_wait_read_all() { asm volatile("cp.async.bulk.wait_group.read 0;\n" ::: "memory"); }
// Waits until this thread's committed bulk stores are complete.
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;\n" ::: "memory"); }

// Makes this thread's generic-proxy shared-memory writes visible to the async
// proxy (TMA, tensor core).
__device__ __forceinline__ void fence_proxy_async_smem()
{
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
}

// ------------------------------------------------------------------ descriptors

// Shared-memory matrix descriptor (sm_100 format): start address, leading and
// stride byte offsets (all >> 4), version 1, layout type in bits 61..63
// (2 = 128-byte swizzle).
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo, uint32_t layout = 2)
{
    uint64_t d = (uint64_t)((saddr >> 4) & 0x3FFFu);
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)(layout & 7u) << 61;
    return d;
}

// Instruction descriptor of kind::f16 with bf16 A/B and fp32 accumulation.
// a_mn / b_mn select MN-major operands; M, N are the MMA shape.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N, bool a_mn, bool b_mn)
{
    return (1u << 4)                        // D format: f32
           | (1u << 7)                      // A format: bf16
           | (1u << 10)                     // B format: bf16
           | ((a_mn ? 1u : 0u) << 15)       // A major-ness
           | ((b_mn ? 1u : 0u) << 16)       // B major-ness
           | ((uint32_t)(N >> 3) << 17)     // N / 8
           | ((uint32_t)(M >> 4) << 24);    // M / 16
}

// ------------------------------------------------------------------ tcgen05

__device__ __forceinline__ void tmem_alloc(uint32_t dst_smem, uint32_t ncols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(dst_smem), "r"(ncols)
                 : "memory");
}
__device__ __forceinline__ void tmem_relinquish()
{
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void fence_before_sync()
{
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
}
__device__ __forceinline__ void fence_after_sync()
{
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
}

// D[tmem] (+)= A[smem] * B[smem]; issued by one thread.  Each descriptor is passed as
// (lo, hi) 32-bit halves so that a K step only adds to lo (the start address field; no carry below 256 KB).
__device__ __forceinline__ void mma_ss_split(uint32_t d_tmem, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo,
                                             uint32_t b_hi, uint32_t idesc, uint32_t accum)
{
    asm volatile(
        "{\n.reg .pred p;\n.reg .b64 da, db;\n"
        "setp.ne.b32 p, %7, 0;\n"
        "mov.b64 da, {%1, %2};\n"
        "mov.b64 db, {%3, %4};\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %5, p;\n}\n" ::"r"(d_tmem),
        "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(0), "r"(accum)
        : "memory");
}

// Arrives once on the mbarrier when every MMA this thread issued so far is done.
__device__ __forceinline__ void mma_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(bar)
                 : "memory");
}

// 32 lanes x 32 bit, 16 consecutive columns per thread.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
        : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]),
          "=f"(v[8]), "=f"(v[9]), "=f"(v[10]), "=f"(v[11]), "=f"(v[12]), "=f"(v[13]), "=f"(v[14]), "=f"(v[15])
        : "r"(taddr));
}
// tcgen05.wait::ld, with the loaded registers tied to it so that no use is
// scheduled before the wait.
__device__ __forceinline__ void tmem_ld_wait(float (&v)[16])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;\n"
                 : "+f"(v[0]), "+f"(v[1]), "+f"(v[2]), "+f"(v[3]), "+f"(v[4]), "+f"(v[5]), "+f"(v[6]), "+f"(v[7]),
                   "+f"(v[8]), "+f"(v[9]), "+f"(v[10]), "+f"(v[11]), "+f"(v[12]), "+f"(v[13]), "+f"(v[14]),
                   "+f"(v[15])::"memory");
}
// Compiler-only barrier: later uses of v stay after the preceding wait.
__device__ __forceinline__ void reg_fence(float (&v)[16])
{
    asm volatile(""
                 : "+f"(v[0]), "+f"(v[1]), "+f"(v[2]), "+f"(v[3]), "+f"(v[4]), "+f"(v[5]), "+f"(v[6]), "+f"(v[7]),
                   "+f"(v[8]), "+f"(v[9]), "+f"(v[10]), "+f"(v[11]), "+f"(v[12]), "+f"(v[13]), "+f"(v[14]),
                   "+f"(v[15])::"memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const float (&v)[16])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};\n" ::"r"(
            taddr),
        "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]), "f"(v[8]), "f"(v[9]),
        "f"(v[10]), "f"(v[11]), "f"(v[12]), "f"(v[13]), "f"(v[14]), "f"(v[15])
        : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory"); }

// D[tmem] (+)= A[tmem] * B[smem]: A is M rows of K 16-bit values in TMEM,
// two per 32-bit column (the lower K index in the low half).
__device__ __forceinline__ void mma_ts_split(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_lo, uint32_t b_hi,
                                             uint32_t idesc, uint32_t accum)
{
    asm volatile(
        "{\n.reg .pred p;\n.reg .b64 db;\n"
        "setp.ne.b32 p, %5, 0;\n"
        "mov.b64 db, {%2, %3};\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], db, %4, p;\n}\n" ::"r"(d_tmem),
        "r"(a_tmem), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(accum)
        : "memory");
}

// 16x32bx2 accesses: over the 16 lanes from taddr's lane, threads 0-15 take
// lane `lane` at columns [c, c + 16), threads 16-31 lane `lane - 16` at
// columns [c + OFF, c + OFF + 16).
template <int OFF>
__device__ __forceinline__ void tmem_ld16_half(uint32_t taddr, float (&v)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.16x32bx2.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16], %17;\n"
        : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]),
          "=f"(v[8]), "=f"(v[9]), "=f"(v[10]), "=f"(v[11]), "=f"(v[12]), "=f"(v[13]), "=f"(v[14]), "=f"(v[15])
        : "r"(taddr), "n"(OFF));
}
template <int OFF>
__device__ __forceinline__ void tmem_st16_half(uint32_t taddr, const float (&v)[16])
{
    asm volatile(
        "tcgen05.st.sync.aligned.16x32bx2.x16.b32 [%0], %17, {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};\n" ::"r"(
            taddr),
        "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]), "f"(v[8]), "f"(v[9]),
        "f"(v[10]), "f"(v[11]), "f"(v[12]), "f"(v[13]), "f"(v[14]), "f"(v[15]), "n"(OFF)
        : "memory");
}

// (a, b) = (a * m + c, b * m + c), one packed f32x2 instruction (each element an IEEE fma)
__device__ __forceinline__ void ffma2(float& a, float& b, float m, float c)
{
    asm("{\n.reg .b64 ra, rm, rc;\nmov.b64 ra, {%0, %1};\nmov.b64 rm, {%2, %2};\nmov.b64 rc, {%3, %3};\n"
        "fma.rn.f32x2 ra, ra, rm, rc;\nmov.b64 {%0, %1}, ra;\n}\n"
        : "+f"(a), "+f"(b) : "f"(m), "f"(c));
}
__device__ __forceinline__ void fadd2(float& a, float& b, float p, float q)
{
    asm("{\n.reg .b64 ra, rp;\nmov.b64 ra, {%0, %1};\nmov.b64 rp, {%2, %3};\n"
        "add.rn.f32x2 ra, ra, rp;\nmov.b64 {%0, %1}, ra;\n}\n"
        : "+f"(a), "+f"(b) : "f"(p), "f"(q));
}

// (a, b) *= (p, q)
__device__ __forceinline__ void fmul2(float& a, float& b, float p, float q)
{
    asm("{\n.reg .b64 ra, rp;\nmov.b64 ra, {%0, %1};\nmov.b64 rp, {%2, %3};\n"
        "mul.rn.f32x2 ra, ra, rp;\nmov.b64 {%0, %1}, ra;\n}\n"
        : "+f"(a), "+f"(b) : "f"(p), "f"(q));
}

// barrier.cta.red.or over `count` threads on named barrier `id`.
__device__ __forceinline__ bool bar_red_or(int id, int count, bool pred)
{
    uint32_t out;
    asm volatile(
        "{\n.reg .pred p, q;\n"
        "setp.ne.u32 p, %1, 0;\n"
        "barrier.cta.red.or.pred q, %2, %3, p;\n"
        "selp.u32 %0, 1, 0, q;\n}\n"
        : "=r"(out)
        : "r"((uint32_t)pred), "r"(id), "r"(count)
        : "memory");
    return out != 0;
}
__device__ __forceinline__ void bar_sync(int id, int count)
{
    asm volatile("barrier.cta.sync %0, %1;\n" ::"r"(id), "r"(count) : "memory");
}

}  // namespace tc
}  // namespace rola
