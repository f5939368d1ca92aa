// Per-warp streams of per-step blocks, prefetched into shared memory by bulk
// asynchronous copies (cp.async.bulk, completion counted on an mbarrier).
//
// The handoff buffers are laid out [warp][step][component][32 lanes], so the
// data a warp needs at one step is one contiguous block. A stream keeps a few
// shared-memory stages per warp: while the warp consumes step s from one
// stage, the copies of the next steps land in the others. One lane issues the
// copies; every lane reads its own column of the stage.
//
// Bulk copies read global memory through the asynchronous proxy, the lanes write
// it through the generic one. A buffer that a kernel both writes and streams
// needs, between the two: in every writing lane, after its last store of the
// pass, stores_before_bulk_reads(); then a barrier (__syncwarp or __syncthreads)
// that the writing lanes share with the lane that issues the copies. What an
// earlier kernel wrote needs neither.
//
// Every wait is bounded: after about a second a wait gives up, sets
// ST_TIMEOUT in the status word and returns, so the kernel always ends.
#pragma once

#include "pes_model.cuh"

namespace pes {

PES_DEV uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

PES_DEV void mbar_init(uint64_t* bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

// Make initialised barriers visible to the asynchronous proxy.
PES_DEV void mbar_init_fence() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }

// Order earlier generic-proxy shared-memory accesses before later bulk copies.
PES_DEV void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// Order this thread's earlier stores to global memory before bulk copies that
// read them, issued by any thread of the block after a barrier with it.
PES_DEV void stores_before_bulk_reads() { asm volatile("fence.proxy.async.global;" ::: "memory"); }

// The one arrival of a phase of `bar`, which completes with `bytes` copied.
PES_DEV void bulk_expect(uint64_t* bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

// Bulk copy of `bytes` (multiple of 16, both addresses 16-byte aligned) from
// global to shared memory, counted on `bar`.
PES_DEV void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

PES_DEV bool mbar_try_wait(uint64_t* bar, uint32_t parity)
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

PES_DEV long long async_now_ns()
{
    long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Bounded wait for the phase of `bar` with the given parity to complete.
PES_DEV void mbar_wait(uint64_t* bar, uint32_t parity, int* status)
{
    if (mbar_try_wait(bar, parity)) return;
    const long long t0 = async_now_ns();
    for (unsigned polls = 0;; ++polls) {
        if (mbar_try_wait(bar, parity)) return;
        if (polls > (1u << 24) || async_now_ns() - t0 > 1000000000LL) {
            atomicOr(status, ST_TIMEOUT);
            return;
        }
    }
}

// Stream of one warp through blocks of NC * 32 scalars, ST stages deep.
template <typename T, int NC, int ST>
struct WarpStream {
    static_assert((32 * sizeof(T)) % 16 == 0, "bulk copies move multiples of 16 bytes");
    T* stage;        // shared: [ST][NC * 32]
    uint64_t* bar;   // shared: a barrier per stage
    uint32_t parity; // expected parity per stage (bit i)
    int lane;

    // `par` is the warp's barrier parity state, carried across streams that
    // reuse the same barriers.
    PES_DEV void init(T* stage_mem, uint64_t* bars, uint32_t par)
    {
        stage = stage_mem;
        bar = bars;
        parity = par;
        lane = threadIdx.x & 31;
    }
    // Start the copy of a block into stage i (all lanes call; lane 0 issues).
    // The stage must no longer be read (a __syncwarp since its last use).
    PES_DEV void issue(const T* src, int i)
    {
        if (lane == 0) {
            fence_proxy_async();
            bulk_expect(bar + i, NC * 32 * sizeof(T));
            bulk_g2s(stage + i * NC * 32, src, NC * 32 * sizeof(T), bar + i);
        }
    }
    // The same for a block in two parts of n1 and n2 components (n1 + n2 = NC).
    PES_DEV void issue2(const T* src1, int n1, const T* src2, int n2, int i)
    {
        if (lane == 0) {
            fence_proxy_async();
            bulk_expect(bar + i, NC * 32 * sizeof(T));
            bulk_g2s(stage + i * NC * 32, src1, n1 * 32 * sizeof(T), bar + i);
            bulk_g2s(stage + i * NC * 32 + n1 * 32, src2, n2 * 32 * sizeof(T), bar + i);
        }
    }
    PES_DEV void wait(int i, int* status)
    {
        mbar_wait(bar + i, (parity >> i) & 1u, status);
        parity ^= (1u << i);
    }
    PES_DEV T get(int i, int c) const { return stage[i * NC * 32 + c * 32 + lane]; }
};

}  // namespace pes
