// Device-side wrappers of the Blackwell (sm_100 family) PTX this library
// uses: mbarriers with bounded waits, TMA tile loads, tcgen05 MMA,
// commit, TMEM allocation and loads, and the shared-memory / instruction
// descriptors.  Host-side tensor-map encoding is declared at the end.
#pragma once

#include <cuda.h>
#include <stdint.h>

#include "pmpe_internal.cuh"

namespace pmpe {

// A bounded wait gives up after this long: far beyond any legitimate wait.
constexpr unsigned long long kWaitLimitNs = 4000000000ull;

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(bar) : "memory");
}
// `count` arrivals at once (a thread arriving on behalf of others).
__device__ __forceinline__ void mbar_arrive_count(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// The last arrival of a participant (address from dsmem_addr): it counts in the
// current phase, and later phases expect one arrival less.
__device__ __forceinline__ void mbar_arrive_drop(uint32_t remote_bar)
{
    asm volatile("mbarrier.arrive_drop.shared::cluster.b64 _, [%0];\n" ::"r"(remote_bar) : "memory");
}
// The phase's state now, without waiting.
__device__ __forceinline__ bool mbar_test_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ unsigned long long globaltimer_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// mbar_try_wait for a longer wait: the thread may sleep up to 20 us (it wakes
// when the phase completes), so that waiting roles poll less beside busy ones.
__device__ __forceinline__ bool mbar_try_wait_hint(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity), "r"(20000u)
        : "memory");
    return ok != 0;
}
// Wait for the phase of `bar` with parity `parity`, for at most limit_ns
// (kWaitLimitNs for the layer's kernels) or until another role raised the
// abort flag.  On expiry it raises the abort flag, records
// PMPE_STATUS_PIPELINE_TIMEOUT and returns false.
// The global timer is read only after kWaitTries failed tries: one read takes
// about 350 clocks, and a wait that read it whenever its first try failed cost
// every stage of every pipeline role one or two reads, 1,100 to 1,240 clocks a
// stage in the thread that issues the MMAs whatever the tile's size.
constexpr int kWaitTries = 32;
__device__ __noinline__ static bool mbar_wait_for(uint32_t bar, uint32_t parity, volatile int *abort_flag,
                                                  uint32_t *status, unsigned long long limit_ns)
{
    unsigned long long t0 = 0;
    for (;;) {
#pragma unroll 1
        for (int i = 0; i < kWaitTries; ++i)
            if (mbar_try_wait_hint(bar, parity)) return true;
        if (*abort_flag) return false;
        const unsigned long long now = globaltimer_ns();
        if (t0 == 0) {
            t0 = now;
        } else if (now - t0 > limit_ns) {
            *abort_flag = 1;
            if (status) atomicOr(status, PMPE_STATUS_PIPELINE_TIMEOUT);
            return false;
        }
    }
}
__device__ __forceinline__ static bool mbar_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag,
                                                 uint32_t *status)
{
    if (mbar_try_wait(bar, parity)) return true;
    return mbar_wait_for(bar, parity, abort_flag, status, kWaitLimitNs);
}

// Whether this is the elected lane of a converged warp (the same lane every
// time).  Tested directly before TMA and tcgen05 instructions, in a loop that
// the whole warp runs: with the loop inside the elected branch, or the result
// kept in a variable, the operands' broadcasts made a stage of four MMAs and a
// commit cost about 390 clocks instead of 60 to 190.
__device__ __forceinline__ bool elect_one()
{
    uint32_t pred;
    asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(pred));
    return pred != 0;
}

// Named CTA barriers of `threads` threads (whole warps): a plain one, and one
// that tells every thread whether all of them passed `pred`.
__device__ __forceinline__ void named_barrier_sync(int id, int threads)
{
    asm volatile("barrier.cta.sync.aligned %0, %1;\n" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ bool named_barrier_all(int id, int threads, int pred)
{
    uint32_t r;
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.b32 p, %3, 0;\n barrier.cta.red.and.aligned.pred q, %1, %2, p;\n selp.u32 %0, 1, "
        "0, q;\n}\n"
        : "=r"(r)
        : "r"(id), "r"(threads), "r"(pred)
        : "memory");
    return r != 0;
}

// Shared-memory accesses by 32-bit shared address.
__device__ __forceinline__ void st_shared_f32(uint32_t addr, float v)
{
    asm volatile("st.shared.f32 [%0], %1;\n" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ uint4 ld_shared_v4(uint32_t addr)
{
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];\n" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void st_shared_v4(uint32_t addr, const uint4 &v)
{
    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};\n" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ float2 ld_shared_f32x2(uint32_t addr)
{
    float2 v;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];\n" : "=f"(v.x), "=f"(v.y) : "r"(addr) : "memory");
    return v;
}
// Four 8 x 8 BF16 matrices in the mma fragment layout (thread i: row i / 4,
// columns 2 (i & 3), + 1), each stored transposed: thread 8 m + r gives the
// address of the 16-byte row r of (transposed) matrix m.
__device__ __forceinline__ void stmatrix_x4_trans(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d)
{
    asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1, %2, %3, %4};\n" ::"r"(addr), "r"(a), "r"(b),
                 "r"(c), "r"(d)
                 : "memory");
}
// The reverse: four 8 x 8 BF16 matrices read by 16-byte rows and transposed into
// the mma fragment layout.
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t &r0, uint32_t &r1, uint32_t &r2, uint32_t &r3, uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(addr)
                 : "memory");
}
// 16 bytes to global memory with an L2 cache policy.
__device__ __forceinline__ void st_global_hint(void *ptr, const uint4 &v, uint64_t policy)
{
    asm volatile("st.global.L2::cache_hint.v4.u32 [%0], {%1, %2, %3, %4}, %5;\n" ::"l"(ptr), "r"(v.x), "r"(v.y), "r"(v.z),
                 "r"(v.w), "l"(policy)
                 : "memory");
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, uint32_t bar, int x, int y)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];\n" ::
            "r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(x), "r"(y)
        : "memory");
}

// L2 eviction-priority policies for the cache-hinted copies below: data read
// once and streamed through L2 (evict_first), and data read again soon by
// other CTAs or phases of the same kernel (evict_last).
__device__ __forceinline__ uint64_t l2_policy_evict_first()
{
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;\n" : "=l"(p));
    return p;
}
__device__ __forceinline__ uint64_t l2_policy_evict_normal()
{
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;\n" : "=l"(p));
    return p;
}
__device__ __forceinline__ uint64_t l2_policy_evict_last()
{
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;\n" : "=l"(p));
    return p;
}

// Untiled bulk copy of `bytes` (a multiple of 16; both addresses 16-byte
// aligned) from global to this CTA's shared memory, completing on `bar`,
// with an L2 cache policy.
__device__ __forceinline__ void bulk_load_g2s(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar,
                                              uint64_t policy)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;\n" ::
            "r"(dst),
        "l"(src), "r"(bytes), "r"(bar), "l"(policy)
        : "memory");
}

// 16-byte async copy global -> shared with an explicit source size (0: the
// 16 bytes are zero-filled and nothing is read) and an L2 cache policy.
__device__ __forceinline__ void cp_async16_zfill(uint32_t dst, const void *src, uint32_t src_bytes, uint64_t policy)
{
    asm volatile("cp.async.cg.shared.global.L2::cache_hint [%0], [%1], 16, %2, %3;\n" ::"r"(dst), "l"(src),
                 "r"(src_bytes), "l"(policy)
                 : "memory");
}

// One arrival on `bar` once every cp.async this thread issued so far has
// completed; the barrier's expected count includes it (noinc).
__device__ __forceinline__ void cp_async_arrive_noinc(uint32_t bar)
{
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];\n" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory"); }

// Shared-memory matrix descriptor: K-major operand, 128-byte swizzle, rows of
// 128 bytes, 8-row groups 1024 bytes apart (SBO); LBO is unused for this
// layout; bits 46..48 hold the fixed value 0b001; swizzle mode 2 = 128 B.
__device__ __forceinline__ uint64_t sw128_desc(uint32_t saddr)
{
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

// Shared-memory matrix descriptor: MN-major operand, 128-byte swizzle.  The
// operand is stored as blocks of 64 MN-contiguous elements (one 128-byte row
// per K index, 8-row / 1024-byte swizzle atoms along K, SBO = 1024); LBO is the
// byte distance between consecutive 64-element MN blocks.
__device__ __forceinline__ uint64_t mn_sw128_desc(uint32_t saddr, uint32_t lbo_bytes)
{
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)((lbo_bytes >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)(1024 >> 4) << 32) | ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

__device__ __forceinline__ void tc_mma(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                       uint32_t accumulate)
{
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
        "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void tc_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(bar)
                 : "memory");
}

// 32 consecutive FP32 columns of this warp's 32 TMEM lanes: thread i gets
// lane (base lane + i), columns col .. col+31.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float *v)
{
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}
// 16 TMEM lanes x 32 FP32 columns in the mma fragment layout: v[4 j + q] is
// lane 8 (q / 2) + i / 4 (of the 16 from taddr's lane), column 8 j + 2 (i & 3) + (q & 1).
__device__ __forceinline__ void tmem_frag16(uint32_t taddr, float *v)
{
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x4.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory"); }

// Prefetch [ptr, ptr + bytes) into L2 (16-byte aligned, a multiple of 16 bytes).
__device__ __forceinline__ void bulk_prefetch_l2(const void *ptr, uint32_t bytes)
{
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;\n" ::"l"(ptr), "r"(bytes) : "memory");
}

// Fetch a tensor map (a kernel parameter) into the TMA unit's descriptor
// cache ahead of its first use.
__device__ __forceinline__ void prefetch_tmap(const void *map)
{
    asm volatile("prefetch.tensormap [%0];\n" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}
// Make this thread's completed generic-proxy shared-memory writes (e.g. from
// cp.async) visible to the async proxy that tcgen05.mma reads through.
__device__ __forceinline__ void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }

__device__ __forceinline__ void tmem_alloc(uint32_t slot_smem_addr, uint32_t ncols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(slot_smem_addr),
                 "r"(ncols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::);
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(taddr), "r"(ncols));
}

// ------------------------------------------------------------ CTA pairs
//
// A pair is a cluster of two CTAs on one TPC.  Its MMA (cta_group::2) is
// issued by the leader (rank 0) and multiplies M = 256 rows, 128 staged by
// each CTA, with N columns, N / 2 staged by each; each CTA's TMEM gets its own
// 128 rows of all N columns.  Per FLOP the pair stages and reads half of what
// a single CTA's 128 x 256 tile does: 128 x 256 x 16 MMAs of one CTA want 96
// bytes of operand reads and 96 bytes of fills a clock at the full rate,
// beyond the 128 bytes a clock of an SM's shared memory; the pair wants 64 + 64.

__device__ __forceinline__ uint32_t cluster_ctarank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync_all()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}
// The shared::cluster address of CTA `rank`'s copy of this CTA's shared address.
__device__ __forceinline__ uint32_t dsmem_addr(uint32_t local, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(local), "r"(rank));
    return r;
}
// One arrival on a barrier of another CTA of the cluster (address from
// dsmem_addr), with the default semantics of a local arrival: what it hands
// over is this CTA's own TMEM, whose reads tcgen05.wait has completed, a queue slot
// that has been read, or rows in this CTA's shared memory that have landed and are
// fenced for the pair's MMAs.  (A release at cluster
// scope waits for the thread's TMA stores in flight as well: about 3,000
// clocks a tile in the weight-gradient epilogue.)
__device__ __forceinline__ void mbar_arrive_remote(uint32_t remote_bar)
{
    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];\n" ::"r"(remote_bar) : "memory");
}

// 3-D tile load into this CTA's shared memory that completes on `bar`, a
// shared::cluster address: the pair leader's barrier.
__device__ __forceinline__ void tma_load_3d_pair(uint32_t dst, const CUtensorMap *map, uint32_t bar, int x, int y, int z)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, "
        "%5}], [%2];\n" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(x), "r"(y), "r"(z)
        : "memory");
}

// The same for a 2-D box with an L2 cache policy.
__device__ __forceinline__ void tma_load_2d_pair_hint(uint32_t dst, const CUtensorMap *map, uint32_t bar, int x, int y,
                                                      uint64_t policy)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], "
        "[%1, {%3, %4}], [%2], %5;\n" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(x), "r"(y), "l"(policy)
        : "memory");
}
// 32 bytes into another CTA's shared memory, handed over on that CTA's barrier
// `remote_bar` (addresses from dsmem_addr): one arrival and the bytes' transaction.
__device__ __forceinline__ void st_async_32(uint32_t remote_addr, const uint4 &x, const uint4 &y, uint32_t remote_bar)
{
    asm volatile(
        "mbarrier.arrive.expect_tx.shared::cluster.b64 _, [%1], 32;\n"
        "st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.u32 [%0], {%2, %3, %4, %5}, [%1];\n"
        "st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.u32 [%0 + 16], {%6, %7, %8, %9}, [%1];\n" ::"r"(remote_addr),
        "r"(remote_bar), "r"(x.x), "r"(x.y), "r"(x.z), "r"(x.w), "r"(y.x), "r"(y.y), "r"(y.z), "r"(y.w)
        : "memory");
}

__device__ __forceinline__ void tma_load_3d_pair_hint(uint32_t dst, const CUtensorMap *map, uint32_t bar, int x, int y,
                                                      int z, uint64_t policy)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], "
        "[%1, {%3, %4, %5}], [%2], %6;\n" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(x), "r"(y), "r"(z), "l"(policy)
        : "memory");
}

__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap *map, uint32_t bar, int x, int y)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], "
        "[%2];\n" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(x), "r"(y)
        : "memory");
}

// Four rows (y0 .. y3) of a 2-D tensor, 64 columns from x, into four consecutive
// 128-byte rows of this CTA's shared memory (a map with one-row boxes),
// completing on the leader's barrier.
__device__ __forceinline__ void tma_gather4_pair(uint32_t dst, const CUtensorMap *map, uint32_t bar, int x, int y0, int y1,
                                                 int y2, int y3, uint64_t policy)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile::gather4.mbarrier::complete_tx::bytes.cta_group::2.L2::"
        "cache_hint [%0], [%1, {%3, %4, %5, %6, %7}], [%2], %8;\n" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(x), "r"(y0), "r"(y1), "r"(y2), "r"(y3), "l"(policy)
        : "memory");
}

// One warp of each CTA of the pair executes the allocation and the release.
__device__ __forceinline__ void tmem_alloc_pair(uint32_t slot_smem_addr, uint32_t ncols)
{
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(slot_smem_addr),
                 "r"(ncols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;\n" ::);
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols)
{
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;\n" ::"r"(taddr), "r"(ncols));
}
// The pair's MMA, issued by one thread of the leader; descriptors and TMEM
// address name the same offsets in both CTAs.
__device__ __forceinline__ void tc_mma_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                            uint32_t accumulate)
{
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
        "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// Once the leader's MMAs issued so far are done: one arrival on the barrier
// at this offset in both CTAs.
__device__ __forceinline__ void tc_commit_pair(uint32_t bar)
{
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;\n" ::"r"(bar),
        "h"((uint16_t)3)
        : "memory");
}

// TMA store of a 2-D box from shared memory (bulk-group completion).
__device__ __forceinline__ void tma_store_2d(const CUtensorMap *map, uint32_t src, int x, int y)
{
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];\n" ::"l"(
                     reinterpret_cast<uint64_t>(map)),
                 "r"(src), "r"(x), "r"(y)
                 : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;\n" ::: "memory"); }
// Wait until at most N committed bulk groups still read their shared-memory source.
template <int N>
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read %0;\n" ::"n"(N) : "memory"); }
// Wait until all committed bulk groups have completed.
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;\n" ::: "memory"); }

// A counter another CTA releases (ld.acquire at GPU scope).
__device__ __forceinline__ uint32_t ld_acquire_gpu(const uint32_t *ptr)
{
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];\n" : "=r"(v) : "l"(ptr) : "memory");
    return v;
}

// ---------------------------------------------------------------- host side

// 2-D BF16 tensor map over a row-major [rows, cols] matrix with a 64-column x
// box_rows box, 128-byte swizzle, zero fill out of bounds.
bool encode_2d(CUtensorMap *m, const void *ptr, uint64_t cols, uint64_t rows, uint32_t box_rows);
// 2-D BF16 tensor map with a box_cols x box_rows box and the given swizzle.
bool encode_2d_box(CUtensorMap *m, const void *ptr, uint64_t cols, uint64_t rows, uint32_t box_cols,
                   uint32_t box_rows, CUtensorMapSwizzle swizzle);
// 2-D FP32 tensor map with a box_cols x box_rows box and the given swizzle.
bool encode_2d_f32(CUtensorMap *m, const void *ptr, uint64_t cols, uint64_t rows, uint32_t box_cols,
                   uint32_t box_rows, CUtensorMapSwizzle swizzle);
// 3-D BF16 tensor map over a row-major [rows, cols] matrix seen as
// [cols / 64 blocks][rows][64]: a box of box_rows rows x nblocks consecutive
// 64-column blocks lands in shared memory as nblocks 128-byte-swizzled
// [box_rows][64] tiles one after another (the layout of an MN-major operand
// whose MN blocks are box_rows * 128 bytes apart).
bool encode_3d_blocks(CUtensorMap *m, const void *ptr, uint64_t cols, uint64_t rows, uint32_t box_rows, uint32_t nblocks);
// 3-D BF16 tensor map over the gate and up weights, two row-major [rows, cols]
// matrices anywhere in memory (one dimension steps from the lower to the
// higher): a box of 64 columns x 64 rows of both, one after the other, 128-byte
// swizzle, the up rows first when *up_first.  False where a map cannot hold
// both (one tensor as both, or 2^40 bytes apart).
bool encode_gate_up(CUtensorMap *m, const bf16 *gate, const bf16 *up, uint64_t cols, uint64_t rows, bool *up_first);
// tcgen05 instruction descriptor: BF16 x BF16 -> FP32, both operands K-major.
uint32_t make_idesc(int M, int N);
// The same with either operand MN-major (transpose bits 15 for A, 16 for B).
uint32_t make_idesc_major(int M, int N, bool a_mn_major, bool b_mn_major);

}  // namespace pmpe
