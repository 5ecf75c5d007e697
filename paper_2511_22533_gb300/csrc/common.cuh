// common.cuh -- device helpers of libf3dc: inline-PTX wrappers for
// mbarriers, TMA (cp.async.bulk.tensor) and 5th-generation tensor cores
// (tcgen05 + TMEM) on sm_103a, bounded waits, and small numeric helpers.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#define F3DC_DEV __device__ __forceinline__

namespace f3dc {

// Device status word bits (mirrors F3DC_DEV_* in f3dc.h).
constexpr uint32_t kDevTimeout = 1u;
constexpr uint32_t kDevBadIndex = 2u;
constexpr uint32_t kDevBadPlan = 4u;

// Every spin on an mbarrier gives up after this long (ns of %globaltimer);
// the kernel then records kDevTimeout, stops issuing work and drains.
constexpr uint64_t kWaitLimitNs = 1000ull * 1000ull * 1000ull;  // 1 s

F3DC_DEV uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

F3DC_DEV uint64_t globaltimer()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

F3DC_DEV void raise_error(uint32_t *err, uint32_t bit)
{
    if (err) atomicOr(err, bit);
}

// ---------------------------------------------------------------- mbarrier
F3DC_DEV void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}

F3DC_DEV void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }

F3DC_DEV void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

F3DC_DEV void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

F3DC_DEV bool mbar_try_wait(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Non-blocking test of the phase with the given parity.
F3DC_DEV bool mbar_test(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// try_wait with a suspend-time hint: the thread sleeps until the phase
// completes or about `hint_ns` passes, instead of spinning on issue slots.
F3DC_DEV bool mbar_try_wait_sleep(uint64_t *bar, uint32_t parity, uint32_t hint_ns)
{
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity), "r"(hint_ns)
        : "memory");
    return ok != 0;
}

// Waits for the phase with the given parity to complete.  Gives up (returns
// false) when *abort is set by another thread or after kWaitLimitNs; in the
// latter case it sets *abort and records kDevTimeout.  The code is kept short:
// it is inlined at every wait of kernels whose warps share an instruction cache.
F3DC_DEV bool mbar_wait(uint64_t *bar, uint32_t parity, volatile int *abort, uint32_t *err)
{
    if (mbar_try_wait(bar, parity)) return true;
    const uint64_t end = globaltimer() + kWaitLimitNs;
#pragma unroll 1
    while (!mbar_try_wait_sleep(bar, parity, 100000u)) {
        if (*abort) return false;
        if (globaltimer() > end) {
            *abort = 1;
            raise_error(err, kDevTimeout);
            return false;
        }
    }
    return true;
}

// Spins (bounded) for ns nanoseconds; used to let in-flight TMA copies land
// before a CTA that aborted exits.
F3DC_DEV void spin_ns(uint64_t ns)
{
    const uint64_t t0 = globaltimer();
    while (globaltimer() - t0 < ns) {
    }
}

// ---------------------------------------------------------------- TMA
F3DC_DEV void tma_prefetch(const CUtensorMap *map)
{
    asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)map) : "memory");
}

F3DC_DEV void tma_load_2d(void *smem_dst, const CUtensorMap *map, int x, int y, uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3}], [%4];" ::"r"(smem_u32(smem_dst)),
        "l"((uint64_t)map), "r"(x), "r"(y), "r"(smem_u32(bar))
        : "memory");
}

// Pulls one box of a tiled tensor into L2 (no shared memory, no completion).
F3DC_DEV void tma_prefetch_l2_2d(const CUtensorMap *map, int x, int y)
{
    asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global.tile [%0, {%1, %2}];" ::"l"((uint64_t)map), "r"(x),
                 "r"(y)
                 : "memory");
}

F3DC_DEV void tma_prefetch_l2_3d(const CUtensorMap *map, int x, int y, int z)
{
    asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global.tile [%0, {%1, %2, %3}];" ::"l"((uint64_t)map), "r"(x),
                 "r"(y), "r"(z)
                 : "memory");
}

// Tiled TMA store of a shared-memory box to global memory (bulk-group
// completion), and the same as an element-wise fp32 add into global memory.
// Coordinates: x = innermost (column), y = row; the box is clipped at the
// tensor's extent.
F3DC_DEV void tma_store_2d(const CUtensorMap *map, const void *smem_src, int x, int y)
{
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];" ::"l"((uint64_t)map),
                 "r"(x), "r"(y), "r"(smem_u32(smem_src))
                 : "memory");
}
F3DC_DEV void tma_reduce_add_2d(const CUtensorMap *map, const void *smem_src, int x, int y)
{
    asm volatile("cp.reduce.async.bulk.tensor.2d.global.shared::cta.add.tile.bulk_group [%0, {%1, %2}], [%3];" ::"l"(
                     (uint64_t)map),
                 "r"(x), "r"(y), "r"(smem_u32(smem_src))
                 : "memory");
}
F3DC_DEV void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// at most N committed bulk groups may still be reading their shared-memory source
template <int N>
F3DC_DEV void bulk_wait_read()
{
    asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory");
}
// every committed bulk group complete (writes performed)
F3DC_DEV void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// Programmatic dependent launch.  A kernel launched with programmatic stream
// serialization may start (and run its prologue) while the previous kernel
// in the stream is still running.  griddep_wait() blocks until that kernel
// has completed and its memory operations are visible; without the launch
// attribute it returns at once.  Every kernel of this library calls it
// before its first global-memory access (read or write) but for what follows,
// which also keeps completion ordered along a chain of such kernels.
// griddep_launch() lets the next kernel be scheduled early; its CTAs still wait
// in griddep_wait().
//
// What may be read before the wait: weights, and in a step what was written
// before gather_embed -- the row plan and the modulation vectors.  That kernel
// lets the next one start only after its own wait, so whatever starts after it
// does so when the plan's and the modulation's writers have completed.  These
// reads go to L2 (ld_plan, __ldcg): a line left in L1 could be older.  The
// first loads of a kernel that wait for one another (row count, then rows) are
// then one round trip after the wait instead of two or three: a cached step of
// 24 blocks at 1229 tokens 2945 -> 2851 us, a sampling run of the 8^3 model of
// width 128 1000 -> 966, a 25-step one of width 1024 96.0 -> 93.9 ms.
F3DC_DEV void griddep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
F3DC_DEV void griddep_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
F3DC_DEV int32_t ld_plan(const int32_t *p)
{
    int32_t v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Register split between warpgroups (every warp of a warpgroup executes the
// same one).  The sum over the block must not exceed its registers at launch.
template <int N>
F3DC_DEV void reg_inc()
{
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N));
}
template <int N>
F3DC_DEV void reg_dec()
{
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N));
}

// Orders this thread's generic-proxy shared-memory writes before later
// async-proxy (tensor core / TMA) reads of the same memory.
F3DC_DEV void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// ---------------------------------------------------------------- tcgen05
F3DC_DEV void tmem_alloc(uint32_t *holder_smem, uint32_t ncols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(holder_smem)),
                 "r"(ncols));
}

F3DC_DEV void tmem_relinquish() { asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;"); }

F3DC_DEV void tmem_dealloc(uint32_t taddr, uint32_t ncols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols));
}

// ---- CTA-pair (cta_group::2) forms: a cluster of two CTAs shares one MMA
// of 256 rows; every tcgen05 instruction of such a kernel uses cta_group::2.
F3DC_DEV uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

// shared::cluster address of the variable at `smem_addr` in CTA `rank`
F3DC_DEV uint32_t mapa_shared(uint32_t smem_addr, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_addr), "r"(rank));
    return r;
}

// every thread of both CTAs of the cluster
F3DC_DEV void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

F3DC_DEV void mbar_arrive_cluster(uint32_t cluster_addr)
{
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}

// TMA load of a 3-D box into this CTA's shared memory whose completion is
// counted on an mbarrier of either CTA of the pair (shared::cluster address)
F3DC_DEV void tma_load_3d_pair(void *smem_dst, const CUtensorMap *map, int x, int y, int z, uint32_t bar_cluster)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(smem_u32(smem_dst)),
        "l"((uint64_t)map), "r"(x), "r"(y), "r"(z), "r"(bar_cluster)
        : "memory");
}

// one warp of each CTA of the pair, same ncols
F3DC_DEV void tmem_alloc_pair(uint32_t *holder_smem, uint32_t ncols)
{
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(holder_smem)),
                 "r"(ncols));
}

F3DC_DEV void tmem_relinquish_pair() { asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;"); }

F3DC_DEV void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols)
{
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols));
}

F3DC_DEV void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
F3DC_DEV void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// ---- tcgen05 issue from a converged warp.  Every lane of the issuing warp
// runs the issue loop (barrier outcomes taken as warp votes, warp_all) and
// elect.sync picks the issuing lane inside each instruction.  With the warp
// converged and the member mask full the same lane is elected every time, so
// a commit tracks the MMAs that lane issued.  Measured: a 12-MMA tile issued
// this way takes ~525 cycles against ~580 from a loop run by lane 0 alone,
// and ~945 against ~1500-2600 when two warps running FMA chains share the
// issuer's SM sub-partition.

// every lane's outcome, so a warp takes the same branch around its
// warp-collective instructions even when a bounded wait gives up in one lane
F3DC_DEV bool warp_all(bool v) { return __all_sync(0xffffffffu, v); }

// mbar_wait by a whole warp: true in every lane, or false in every lane.  The
// vote on the first look comes before any branch, so a wait that is already
// over costs one look, one vote and no divergence.
F3DC_DEV bool warp_wait(uint64_t *bar, uint32_t parity, volatile int *abort, uint32_t *err)
{
    if (warp_all(mbar_try_wait(bar, parity))) return true;
    return warp_all(mbar_wait(bar, parity, abort, err));
}

// D[tmem] (+)= A[smem desc] * B[smem desc]^T, bf16 inputs, fp32 accumulate.
F3DC_DEV void mma_bf16_elect(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n .reg .pred p, e;\n elect.sync _|e, 0xffffffff;\n setp.ne.b32 p, %4, 0;\n"
        " @e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
        "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}

// The same with A read from tensor memory (TMEM address a_tmem: row m of A
// in lane m, K elements along the columns, two bf16 per 32-bit column, the
// lower K index in the low half); B from shared memory.
F3DC_DEV void mma_bf16_ts_elect(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n .reg .pred p, e;\n elect.sync _|e, 0xffffffff;\n setp.ne.b32 p, %4, 0;\n"
        " @e tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(d_tmem),
        "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}

// Arrives once on *bar when every tcgen05.mma issued so far by the elected
// thread has completed.
F3DC_DEV void mma_commit_elect(uint64_t *bar)
{
    asm volatile(
        "{\n .reg .pred e;\n elect.sync _|e, 0xffffffff;\n"
        " @e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n" ::"r"(smem_u32(bar))
        : "memory");
}

// D (+)= A B^T over a CTA pair: A rows 0..127 from this CTA's shared memory
// and rows 128..255 from the peer's, at the same offsets; B's N rows split the
// same way; D rows 0..127 in this CTA's TMEM, 128..255 in the peer's.  The eight
// MMAs of 128 K (two 64-K regions of each operand, a_half and b_half apart in
// descriptor units; 16 K further is 2 units) under one election.
F3DC_DEV void mma_bf16_pair_128k(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint64_t a_half, uint64_t b_half,
                                 uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n .reg .pred p, e, t;\n .reg .b64 a, b;\n elect.sync _|e, 0xffffffff;\n setp.ne.b32 p, %6, 0;\n setp.eq.b32 t, 0, 0;\n"
        " @e tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %5, p;\n"
        " add.s64 a, %1, 2;\n add.s64 b, %2, 2;\n @e tcgen05.mma.cta_group::2.kind::f16 [%0], a, b, %5, t;\n"
        " add.s64 a, a, 2;\n add.s64 b, b, 2;\n @e tcgen05.mma.cta_group::2.kind::f16 [%0], a, b, %5, t;\n"
        " add.s64 a, a, 2;\n add.s64 b, b, 2;\n @e tcgen05.mma.cta_group::2.kind::f16 [%0], a, b, %5, t;\n"
        " add.s64 a, %1, %3;\n add.s64 b, %2, %4;\n @e tcgen05.mma.cta_group::2.kind::f16 [%0], a, b, %5, t;\n"
        " add.s64 a, a, 2;\n add.s64 b, b, 2;\n @e tcgen05.mma.cta_group::2.kind::f16 [%0], a, b, %5, t;\n"
        " add.s64 a, a, 2;\n add.s64 b, b, 2;\n @e tcgen05.mma.cta_group::2.kind::f16 [%0], a, b, %5, t;\n"
        " add.s64 a, a, 2;\n add.s64 b, b, 2;\n @e tcgen05.mma.cta_group::2.kind::f16 [%0], a, b, %5, t;\n"
        "}\n" ::"r"(d_tmem),
        "l"(a_desc), "l"(b_desc), "l"(a_half), "l"(b_half), "r"(idesc), "r"(accumulate)
        : "memory");
}

// completion of the elected thread's earlier pair MMAs, arriving once on the
// mbarrier at the same offset in every CTA of `cta_mask`
F3DC_DEV void mma_commit_pair_mc_elect(uint64_t *bar, uint16_t cta_mask)
{
    asm volatile(
        "{\n .reg .pred e;\n elect.sync _|e, 0xffffffff;\n"
        " @e tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;\n"
        "}\n" ::"r"(smem_u32(bar)),
        "h"(cta_mask)
        : "memory");
}

// the same, on this CTA's mbarrier only
F3DC_DEV void mma_commit_pair_elect(uint64_t *bar)
{
    asm volatile(
        "{\n .reg .pred e;\n elect.sync _|e, 0xffffffff;\n"
        " @e tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n" ::"r"(smem_u32(bar))
        : "memory");
}

// 32 TMEM lanes x 32 consecutive 32-bit columns: thread t of the warp gets
// lane (taddr.lane + t), columns taddr.col .. +31.
F3DC_DEV void tmem_ld32(uint32_t taddr, uint32_t (&r)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
          "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]),
          "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]),
          "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
}

F3DC_DEV void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Store 32 consecutive 32-bit columns of the warp's 32 TMEM lanes.
F3DC_DEV void tmem_st32(uint32_t taddr, const uint32_t (&r)[32])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
        "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};" ::"r"(taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
        "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]),
        "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]),
        "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
        : "memory");
}

// 32 TMEM lanes x 16 consecutive 32-bit columns (load / store).
F3DC_DEV void tmem_ld16(uint32_t taddr, uint32_t (&r)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}
F3DC_DEV void tmem_st16(uint32_t taddr, const uint32_t (&r)[16])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(
            taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
        "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
        : "memory");
}

F3DC_DEV void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Shared-memory matrix descriptor for tcgen05.mma (sm_100 family):
// start >> 4 in [0,14), leading-dimension byte offset >> 4 in [16,30),
// stride-dimension byte offset >> 4 in [32,46), the fixed version bit 46,
// base offset 0 (atoms 1024-byte aligned) and the swizzle mode in [61,64).
constexpr uint32_t kSwizzleNone = 0, kSwizzle128 = 2, kSwizzle64 = 4, kSwizzle32 = 6;

F3DC_DEV uint64_t make_sdesc(uint32_t saddr, uint32_t lbo, uint32_t sbo, uint32_t swz)
{
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)(swz & 7u) << 61;
    return d;
}

// Instruction descriptor, kind::f16: fp32 accumulator (bits 4-5 = 1), bf16 A
// and B (bits 7-9, 10-12 = 1), K-major (0) or MN-major (1) A / B in bits 15
// and 16, N >> 3 in bits 17-22, M >> 4 in bits 24-28.
__host__ __device__ constexpr uint32_t make_idesc_bf16(int M, int N, int a_mn_major, int b_mn_major)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)a_mn_major << 15) | ((uint32_t)b_mn_major << 16) |
           ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// ---------------------------------------------------------------- numerics
F3DC_DEV float bf16_bits_to_f32(uint32_t u16) { return __uint_as_float(u16 << 16); }

// Round to nearest even; NaN -> quiet NaN 0x7FC0.
F3DC_DEV uint32_t f32_to_bf16_bits(float f)
{
    uint32_t x = __float_as_uint(f);
    if ((x & 0x7FFFFFFFu) > 0x7F800000u) return 0x7FC0u;
    return (x + (((x >> 16) & 1u) + 0x7FFFu)) >> 16;
}

// Exact software round-to-nearest-even with NaN canonicalised (the velocity
// history, which must match the reference rounding bit for bit).
F3DC_DEV uint32_t pack_bf16x2_exact(float lo, float hi)
{
    return f32_to_bf16_bits(lo) | (f32_to_bf16_bits(hi) << 16);
}

// Hardware round-to-nearest-even pack of two floats (activations, P).
F3DC_DEV uint32_t pack_bf16x2(float lo, float hi)
{
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

F3DC_DEV float tanh_fast(float x)
{
    float y;
    asm("tanh.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

F3DC_DEV float exp2_fast(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// three-input maximum (one instruction on sm_100 and later)
F3DC_DEV float fmax3(float a, float b, float c)
{
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// packed pairs of fp32 for the paired FMA / add instructions of sm_100+
struct f32x2 {
    float x, y;
};
F3DC_DEV f32x2 ffma2(f32x2 a, f32x2 b, f32x2 c)
{
    uint64_t pa, pb, pc, d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(pa) : "f"(a.x), "f"(a.y));
    asm("mov.b64 %0, {%1, %2};" : "=l"(pb) : "f"(b.x), "f"(b.y));
    asm("mov.b64 %0, {%1, %2};" : "=l"(pc) : "f"(c.x), "f"(c.y));
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(pa), "l"(pb), "l"(pc));
    f32x2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(d));
    return r;
}
F3DC_DEV f32x2 fadd2(f32x2 a, f32x2 b)
{
    uint64_t pa, pb, d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(pa) : "f"(a.x), "f"(a.y));
    asm("mov.b64 %0, {%1, %2};" : "=l"(pb) : "f"(b.x), "f"(b.y));
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(pa), "l"(pb));
    f32x2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(d));
    return r;
}

F3DC_DEV f32x2 fmul2(f32x2 a, f32x2 b)
{
    uint64_t pa, pb, d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(pa) : "f"(a.x), "f"(a.y));
    asm("mov.b64 %0, {%1, %2};" : "=l"(pb) : "f"(b.x), "f"(b.y));
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(pa), "l"(pb));
    f32x2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(d));
    return r;
}

// A product that must round on its own before it is added: the compiler makes
// one FMA of mul.rn.f32x2 and add.rn.f32x2 (with -fmad=false too), unlike of the
// scalar __fmul_rn and __fadd_rn.  An FMA with an addend of -0.0 is the product
// alone, and the compiler cannot see the addend: it comes from a kernel argument.
F3DC_DEV f32x2 fmul2_alone(f32x2 a, f32x2 b, float neg_zero) { return ffma2(a, b, {neg_zero, neg_zero}); }

F3DC_DEV float gelu_tanh(float x)
{
    const float k0 = 0.7978845608028654f;  // sqrt(2/pi)
    float inner = k0 * (x + 0.044715f * x * x * x);
    return 0.5f * x * (1.0f + tanh_fast(inner));
}

F3DC_DEV float warp_sum(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// LayerNorm of one row held by a warp (Supp. Sec. F; eps 1e-6): lane l holds
// the float4 groups q * 32 + l (q < NV) of the row's W = 128 NV values.  The
// mean first, then the mean of squared deviations, each summed per lane in
// q order and then across the warp; both kernels that normalise rows (the
// LayerNorm kernel and the final layer) take them from here, so their outputs
// agree bit for bit.
template <int NV>
F3DC_DEV void ln_row_stats(const float4 (&v)[NV], int W, float &mean, float &rstd)
{
    float s = 0.f;
#pragma unroll
    for (int q = 0; q < NV; ++q) s += (v[q].x + v[q].y) + (v[q].z + v[q].w);
    mean = warp_sum(s) / (float)W;
    float ss = 0.f;
#pragma unroll
    for (int q = 0; q < NV; ++q) {
        const float a = v[q].x - mean, b = v[q].y - mean, c = v[q].z - mean, d = v[q].w - mean;
        ss += (a * a + b * b) + (c * c + d * d);
    }
    const float var = warp_sum(ss) / (float)W;
    rstd = rsqrtf(var + 1e-6f);
}

// (x - mean) rstd mul + add for four columns, packed to bf16 pairs.
F3DC_DEV uint2 ln_out4(float4 v, float mean, float rstd, float4 mu, float4 ad)
{
    const float y0 = (v.x - mean) * rstd * mu.x + ad.x;
    const float y1 = (v.y - mean) * rstd * mu.y + ad.y;
    const float y2 = (v.z - mean) * rstd * mu.z + ad.z;
    const float y3 = (v.w - mean) * rstd * mu.w + ad.w;
    uint2 pk;
    pk.x = pack_bf16x2(y0, y1);
    pk.y = pack_bf16x2(y2, y3);
    return pk;
}

}  // namespace f3dc
