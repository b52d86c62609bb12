// Split-KV pass of the verification mode on the sm_100a tensor path.
//
// One CTA per SM-sized work item (sequence, KV head, row group of 1 or 2 128-row blocks, piece of
// the key range).  A block packs the GQA group's g heads x p = 128 / g draft tokens (row r = (t % p) g + head;
// g = 7: 18 tokens, 2 rows of padding), so each K/V byte crosses HBM -> SM once per KV head and row group.
//
//   warp 8, one thread   TMA producer: the Q block(s) (two boxes of 64 dims x g heads x p tokens
//                        each, which land exactly in the K-major 128-byte-swizzled operand
//                        layout), then K and V tiles of 128 keys x 128 dims (4 boxes of 128 x 64)
//                        into a 2- or 3-stage shared-memory ring, mbarrier full / empty handshakes.
//   warp 9               tcgen05.mma issuer: the warp stays converged, an elected lane issues.  A job is one key tile against one row block:
//                        S = Q K^T (A, B from shared memory, K-major) into a 128 x 128 fp32 TMEM
//                        block; O += P V with P read from TMEM (bf16, aliasing the S block) and V
//                        from shared memory as an MN-major operand.  The scores of up to three
//                        jobs are kept ahead of the softmax.
//   warps 0-7            softmax, TMEM lane = query row: tcgen05.ld, ancestor / range / window
//                        masking, fp32 online softmax with a lazy maximum, P packed to bf16 and
//                        stored back with tcgen05.st.
//                        One row block (T <= 18): the two threads with the same lane (warps w and
//                        w + 4, one scheduler) share a row, warpgroup g taking key columns [64 g, 64 g + 64) of every
//                        tile, with its P over its own scores.  They use the same reference maximum and run apart from one
//                        another, by a tile at most: what one does besides its exponentials is filled by the
//                        exponentials of the other.  A reference only moves when a score exceeds it by more than
//                        2^8; the warp that finds one says so and goes on, and its partner follows
//                        before it hands over P of that tile (softmax_pair.cuh: no barrier but in the first tile and at the end).
//                        Each thread sums its own columns; the halves' sums meet once, in the epilogue.
//                        Cycles per tile (41 tiles a CTA, 20 CTAs): 1,985 with a barrier of all softmax warps in every tile, 1,880
//                        with one between the two of a pair, 1,520 to 1,550 without (0.77 to 0.79 us at 1,965 MHz, in step or half a
//                        tile apart); the exponentials alone are 1,024, the products 1,030 (a wait at a barrier that is complete costs
//                        the issuing warp 85 and the pipe holds about 100 cycles of work behind the issuing lane, so V is waited for
//                        together with P).  With all SMs at work the GPU is at its power cap, 1.55 to 1.7 GHz, and a cycle saved is a
//                        third of one in time.
//                        References that move, 16,384 keys, 64 nodes, us (a barrier of all in every tile in brackets): nothing
//                        moves 22.2 (25.2), one key in 700 stands out 23.9 (25.7), one half outgrows the reference in every
//                        second tile 27.2 (27.2), both halves of every row in every tile 32.2 (28.6: there P of a half is
//                        rescaled as well, and each waits for what the other posts).
//                        Two row blocks: warpgroup g owns block g, one thread per row and all 128
//                        keys of a tile, and works through its block's tiles on its own (no
//                        barrier between the warpgroups); per block the chain is scores -> softmax
//                        -> O += P V -> next scores, and the two chains interleave on the tensor
//                        pipe and the exponential unit.  P is handed over in two halves, the first
//                        half's product running beside the exponentials of the second.  3,200 cycles per tile: 2,030 of
//                        softmax and 1,100 until the next scores are there.
//                        What a score costs: packed fp32 multiply-add and addition (half an instruction each), 2^x, half a
//                        conversion to bf16, half a maximum; with single fp32 operations and bf16 packed by integer
//                        ones 8.5 cycles a score and scheduler instead of 8.1 (the unit for 2^x alone: 8.0).
//   warp 10              gatekeeper: fills the tables of ancestor words and window bounds, then one
//                        thread waits (overlapped mode), beside the main loop, for the counters that
//                        allow this CTA's first global write.
//
// With one row block there are three S blocks and one O accumulator, with two row blocks one S
// block and one accumulator per block.
//
// Ordering against neighbouring kernels in the stream (see SyncArgs).  Overlapped mode: the kernel
// is launched with programmatic stream serialisation and never waits for the previous grid as a
// whole.  All reads of q / k / v / parents are issued as soon as the CTA starts, so the K/V stream
// of this call overlaps the tail of the previous one; in front of its first global write a CTA
// waits on the finisher counters.  A CTA publishes its item after storing its partials, and the
// call's finisher CTAs wait for the arrivals, share the call's rows among them, merge each row's
// pieces by log-sum-exp and write out / lse.  Stream-ordered mode (a call captured into a graph, or
// with programmatic launch switched off): the kernel touches no counter, only stores partials and
// direct results, and the combine kernel follows.
//
// Every wait is bounded; a wait that gives up sets the timeout status bit and the CTA drains and
// exits.  TMEM is always released.
#pragma once
#include <cuda.h>
#include <cuda_fp16.h>

#include "combine.cuh"
#include "common.cuh"
#include "softmax_pair.cuh"

namespace sparrow {

struct TcArgs {
    const int32_t* parents;      // DEV [B][T_tree]
    const int32_t* first_visible;   // DEV [B][T] or nullptr: query t sees prefix key j only if j >= first_visible[b][t]
    int32_t n_q_heads;
    float scale_log2e;           // softmax_scale * log2(e)
    int32_t leave_l2;            // K and V tiles that are the first to leave L2: none, half (1), all (2)
    __half* o_part;              // [n_items][part_rows] partial rows: 128 fp16 outputs + fp32 LSE (kPartRowHalves)
    __nv_bfloat16* out;          // final output
    float* lse;
    unsigned* status;
};

namespace tc {

constexpr int kThreads = 352;                    // 8 softmax warps, producer, MMA issuer, gatekeeper
// Declared thread bound: caps the kernel at 65536 / 384 = 170 registers per thread.
constexpr int kBoundThreads = 384;
constexpr int kProducerWarp = 8, kMmaWarp = 9, kGateWarp = 10;
constexpr int kTile = 128;                       // keys per stage and per job
constexpr int kSubTileBytes = 128 * 64 * 2;      // one 128 x 64 bf16 box: 16 KB
constexpr int kQBlockBytes = 2 * kSubTileBytes;  // 128 rows x 128 dims: 32 KB
constexpr int kStageBytes = 4 * kSubTileBytes;   // K (32 KB) + V (32 KB)
constexpr int kRowBytes = kPartRowHalves * 2;    // a partial row: 272 bytes
constexpr int kMiscBytes = 2048;                 // barriers, flags, ancestor words, maxima exchange
constexpr uint32_t kSpinLimit = 1u << 22;        // polls before a wait gives up
constexpr uint32_t kPairLag = 512;               // cycles by which the second softmax warp of a pair lags: 64 exponentials of a warp
constexpr int kPrefetchTiles = 2;                // brought into L2 ahead of the wait for the predecessor
// Lazy-max threshold in log2 units.  A key that holds most of a row's weight should be the reference: its P is then 1, otherwise
// rounded to bf16 while the row is divided by the sum of unrounded ones (one key by 2^9 ... 2^15 above the rest, |v| < 4: out is 7.8e-3
// off at most with 8, 2.0e-2 with 16).  Where no reference moves the two are equally fast.
constexpr float kRescaleLog2 = 8.0f;

// Rows received from the CTAs of a cluster lie in one stage of the ring (see recv_stage).  One row block: behind the start of it, where in the
// first stage the end of the staged rows lies.  Two row blocks (up to 256 rows and rounded-up shares): in the last
// stage and a little more behind it.
constexpr int kMaxMergeCluster = 16;
constexpr int kRecvSkip = 4096;
static_assert(kBlockRows * kRowBytes - kQBlockBytes <= kRecvSkip && kRecvSkip + (kBlockRows + kMaxMergeCluster) * kRowBytes <= kStageBytes, "");
__host__ __device__ constexpr int recv_extra(int n_blocks)
{
    return n_blocks == 1 ? 0 : ((2 * kBlockRows + kMaxMergeCluster) * kRowBytes - kStageBytes + 1023) / 1024 * 1024;
}
__host__ __device__ constexpr int smem_bytes(int n_blocks, int n_stages)
{
    return 1024 /*alignment slack*/ + n_blocks * kQBlockBytes + n_stages * kStageBytes + recv_extra(n_blocks) + kMiscBytes;
}
// S blocks (score tiles in flight) for a given number of row blocks; TMEM: S blocks first, then
// one 128-column O accumulator per row block, 512 columns in all.
__host__ __device__ constexpr int s_blocks(int n_blocks) { return n_blocks == 1 ? 3 : 2; }

// ---- PTX wrappers ------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
// The same without being held up where the phase is not complete.
__device__ __forceinline__ bool mbar_test_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
// Bounded wait: false when the phase did not complete within kSpinLimit polls.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity)
{
    for (uint32_t i = 0; i < kSpinLimit; ++i)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}
// Bounded as well, as one piece of code for a warp whose next instruction should follow the phase at once: a wait at a
// complete barrier costs about 85 cycles, during which the tensor pipe runs out of work.
__device__ __forceinline__ bool mbar_wait_tight(uint32_t bar, uint32_t parity)
{
    uint32_t left;
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .u32 i;\n\tmov.u32 i, %3;\n\t"
        "WAIT:\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t@p bra DONE;\n\t"
        "sub.u32 i, i, 1;\n\tsetp.ne.u32 p, i, 0;\n\t@p bra WAIT;\n\t"
        "DONE:\n\tmov.u32 %0, i;\n\t}"
        : "=r"(left) : "r"(bar), "r"(parity), "n"(kSpinLimit) : "memory");
    return left != 0;
}
// Same for a whole warp.  Every lane polls, so that the warp stays converged and no shuffle stands
// between the phase flip and the next instruction: a wait-issue-commit round of eight tensor-core
// instructions takes 616 cycles like this, 672 with one lane polling and issuing, 815 with one lane
// polling, a shuffle, and an elected lane issuing.
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity) { return mbar_wait(bar, parity); }
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, int c0, int c1, int c2, int c3, uint32_t bar)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
        ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(bar) : "memory");
}
// the same with an L2 eviction policy
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, int c0, int c1, int c2, int c3, uint32_t bar, uint64_t policy)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, %3, %4, %5}], [%6], %7;"
        ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(bar), "l"(policy) : "memory");
}
// Brings a box into L2 only: a hint, which neither reads nor orders anything.
__device__ __forceinline__ void tma_prefetch_4d(const CUtensorMap* map, int c0, int c1, int c2, int c3, uint64_t policy)
{
    asm volatile("cp.async.bulk.prefetch.tensor.4d.L2.global.tile.L2::cache_hint [%0, {%1, %2, %3, %4}], %5;"
                 ::"l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "l"(policy) : "memory");
}
// 1-D bulk copy global -> shared (16-byte aligned, size a multiple of 16), completion on an mbarrier
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
// 1-D bulk copy shared -> global, and the wait until this thread's copies are complete (written, not only read)
__device__ __forceinline__ void bulk_store(void* dst, uint32_t src, uint32_t bytes)
{
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_store_wait()
{
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
    asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}
__device__ __forceinline__ void fence_barrier_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
// Orders this thread's accesses to global memory across the generic and the async proxy (bulk copies).
__device__ __forceinline__ void fence_proxy_async_global() { asm volatile("fence.proxy.async.global;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// barrier among the 256 softmax threads only (id 1; id 0 is __syncthreads)
__device__ __forceinline__ void softmax_bar_sync() { asm volatile("bar.sync 1, 256;" ::: "memory"); }
// The gatekeeper warp has filled the tables that the 256 softmax threads read (id 3).
__device__ __forceinline__ void tables_ready_arrive() { asm volatile("bar.arrive 3, 288;" ::: "memory"); }
__device__ __forceinline__ void tables_ready_sync() { asm volatile("bar.sync 3, 288;" ::: "memory"); }
// ---- thread-block clusters
// (relaxed: nothing but the barrier's own phase is ordered; a releasing arrive took 0.7 us of every set-up)
__device__ __forceinline__ void cluster_arrive_relaxed() { asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory"); }
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
// address of the same place in the shared memory of CTA `rank` of the cluster
__device__ __forceinline__ uint32_t map_to_rank(uint32_t addr, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
// 1-D bulk copy from this CTA's shared memory to a CTA of the cluster, counted on an mbarrier there
__device__ __forceinline__ void bulk_push(uint32_t dst_cluster, uint32_t src, uint32_t bytes, uint32_t bar_cluster)
{
    asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst_cluster), "r"(src), "r"(bytes), "r"(bar_cluster) : "memory");
}
// One lane of a converged warp.  The tensor-core instructions take their descriptors from uniform
// registers, which the compiler only uses behind elect.sync in a warp whose control flow stays
// converged.  Behind `if (lane == 0)` every tcgen05.mma first moves its operands over: 93 to 104
// cycles per 128 x 128 x 16 instruction, against the pipe's own 64 (one CTA per SM).
__device__ __forceinline__ bool elect_one()
{
    uint32_t r;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(r));
    return r != 0;
}
// D[tmem] (+)= A[smem] * B[smem]
__device__ __forceinline__ void mma_ss(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
// D[tmem] (+)= A[tmem] * B[smem]
__device__ __forceinline__ void mma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float* v)
{
    uint32_t* r = reinterpret_cast<uint32_t*>(v);
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v)
{
    uint32_t* r = reinterpret_cast<uint32_t*>(v);
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t* r)
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
        "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
        ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
          "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]),
          "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]),
          "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
        : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t* r)
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
        ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
          "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
        : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ float ex2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float lds_f32(uint32_t addr)
{
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ void lds_v4(uint32_t addr, uint32_t (&v)[4])
{
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]) : "r"(addr));
}
__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi)
{
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
__device__ __forceinline__ uint32_t pack_half2(float lo, float hi)
{
    const __half2 h2 = __floats2half2_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&h2);
}

// Shared-memory matrix descriptor, 128-byte swizzle, descriptor version 1 (sm_100).
// K-major operand: rows of 128 bytes, 8-row groups 1024 bytes apart (stride offset); the leading
// offset is unused.  MN-major operand: 64-element (128-byte) runs along MN, 8 K-rows per 1024-byte
// group (stride offset), next 64-element MN run `lbo` bytes away (leading offset).
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo_bytes, uint32_t sbo_bytes)
{
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3FFFFu) >> 4);
    d |= (uint64_t)((lbo_bytes >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo_bytes >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;          // descriptor version
    d |= (uint64_t)2 << 61;          // SWIZZLE_128B
    return d;
}
// Instruction descriptor, kind::f16: D fp32, A/B bf16, A K-major, M = 128, N = n (128 or 64).
__host__ __device__ constexpr uint32_t idesc_bf16(bool b_mn_major, uint32_t n = 128u)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((b_mn_major ? 1u : 0u) << 16) | ((n >> 3) << 17) | ((128u >> 4) << 24);
}

// ---- softmax helpers on a 32-column chunk of one score row ---------------------------------------
__device__ __forceinline__ float max3(float a, float b, float c)
{
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
__device__ __forceinline__ void mask_chunk(float (&x)[32], uint32_t visible)
{
    #pragma unroll
    for (int c = 0; c < 32; ++c)
        if (!((visible >> c) & 1u)) x[c] = -INFINITY;
}
__device__ __forceinline__ float chunk_max(const float (&x)[32])
{
    float a = max3(x[0], x[1], x[2]), b = max3(x[3], x[4], x[5]);
    #pragma unroll
    for (int c = 6; c < 30; c += 4) { a = max3(a, x[c], x[c + 1]); b = max3(b, x[c + 2], x[c + 3]); }
    return max3(a, b, fmaxf(x[30], x[31]));
}
// Two fp32 operations per instruction (a pair of registers each).
__device__ __forceinline__ uint64_t pair_of(float lo, float hi)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void pair_parts(uint64_t p, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(p)); }
__device__ __forceinline__ uint64_t fma_pair(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ uint64_t add_pair(uint64_t a, uint64_t b)
{
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
// p = 2^(x c2 - mc) for 32 scores (c2 and -mc twice each); adds the unrounded p to sum and stores the 16 packed bf16
// pairs to 16 TMEM columns at p_addr.
__device__ __forceinline__ void exp_chunk(const float (&x)[32], uint64_t c2, uint64_t neg_mc, uint64_t (&sum)[2], uint32_t p_addr)
{
    uint32_t p[16];
    #pragma unroll
    for (int c = 0; c < 16; ++c) {
        float p0, p1;
        pair_parts(fma_pair(pair_of(x[2 * c], x[2 * c + 1]), c2, neg_mc), p0, p1);
        p0 = ex2(p0);
        p1 = ex2(p1);
        sum[c & 1] = add_pair(sum[c & 1], pair_of(p0, p1));
        p[c] = pack_bf16x2(p0, p1);
    }
    tmem_st16(p_addr, p);
}
__device__ __forceinline__ float sum_of(const uint64_t (&sum)[2])
{
    float a, b;
    pair_parts(add_pair(sum[0], sum[1]), a, b);
    return a + b;
}

// Barriers between the two softmax warps that share a scheduler and 32 rows (ids 4 to 11).
__device__ __forceinline__ void pair_sync(uint32_t id) { asm volatile("bar.sync %0, 64;" ::"r"(id) : "memory"); }
// What is on reference m, brought to reference m_new >= m (raw scores; none yet: -inf).
__device__ __forceinline__ float rescale(float m, float m_new, float c2) { return m == m_new ? 1.f : m == -INFINITY ? 0.f : ex2((m - m_new) * c2); }

// The stage of the ring that a CTA of a cluster receives its rows in, for a piece of n tiles: with one row block the one whose last tile
// is furthest back (of a piece that does not fill the ring: an unused one), which is idle two tiles before the product of
// the last.  With two row blocks only the last stage has the room.
__host__ __device__ constexpr int recv_stage(int n_blocks, int n) { return n_blocks == 1 ? n % 3 : 1; }
// The last tile in that stage, of n >= the ring's depth.
__host__ __device__ constexpr int recv_last_tile(int n_blocks, int n) { return n_blocks == 1 ? n - 3 : (n & ~1) - 1; }

// Shared-memory addresses of the mbarriers (8-byte slots).  K and V tiles have their own empty
// barriers: a K tile is released as soon as its last S = Q K^T has been computed, a V tile
// only after its last O += P V, so the K stream runs ahead of the V stream.  They have their own full barriers as
// well, except that with one row block V counts on the barrier of its tile's P, the last tile's on its own.
struct Bars {
    uint32_t base;
    // slots of 8 bytes: 0-27 here and in o_done, 31 is p_full(3); 28 and 29 hold the TMEM address and flags, 30 is free.
    // With one row block 31 is free as well, and 24-27 (o_done of the second block) hold the words that the softmax pairs post.
    __device__ __forceinline__ uint32_t k_full(int i) const { return base + 8u * (uint32_t)i; }
    __device__ __forceinline__ uint32_t k_empty(int i) const { return base + 24u + 8u * (uint32_t)i; }
    __device__ __forceinline__ uint32_t v_full(int i) const { return base + 48u + 8u * (uint32_t)i; }
    __device__ __forceinline__ uint32_t v_empty(int i) const { return base + 72u + 8u * (uint32_t)i; }
    __device__ __forceinline__ uint32_t s_full(int i) const { return base + 96u + 8u * (uint32_t)i; }
    // (a fourth, with two row blocks: two halves of P for each)
    __device__ __forceinline__ uint32_t p_full(int i) const { return i < 3 ? base + 120u + 8u * (uint32_t)i : base + 248u; }
    __device__ __forceinline__ uint32_t q_full() const { return base + 144u; }
    __device__ __forceinline__ uint32_t fin() const { return base + 152u; }       // finishers' bulk copies
    // Completion of O += P V of key tile j on row block blk: a ring of four barriers per block,
    // tile j on barrier j % 4 with phase parity (j / 4) & 1.  The softmax only looks at it when a
    // row maximum moves and in the epilogue, asking for the last tile that this warp has handed over and its partner has
    // or will on its own.  A parity wait is only meaningful for the phase in progress or the one just completed; here the
    // barrier is in exactly that state: with tile t asked for, its previous use (tile t - 4) completed before the
    // scores of tile t, which the warp has seen (the tensor pipe completes in issue order and they
    // were issued after the product of tile t - 3), and its next use (tile t + 4) needs P that this warp
    // has yet to hand over.
    __device__ __forceinline__ uint32_t o_done(int blk, int j) const { return base + 160u + 32u * (uint32_t)blk + 8u * (uint32_t)(j & 3); }
};

constexpr uint32_t kBarrierBytes = 256;      // what the slots above and the words between them take of the barrier area
static_assert(kMiscBytes >= 1024 + 2 * 128 * 4 && kBarrierBytes + kMaxT * 8 == 768, "barriers, ancestor words, bounds, exchange");

struct MergeOut {
    __nv_bfloat16* out;
    float* lse;
    int T, n_q_heads, qg, inv_qg;
};
// The final bf16 row and LSE from a row's weighted sum, the sum of weights and the reference of the weights; 16
// threads of 8 dims each.
__device__ __forceinline__ void write_merged(const float (&acc)[8], float s, float m, int b, int t, int h, int c16, const MergeOut& mo)
{
    const float inv = s > 0.f ? __fdividef(1.f, s) : 0.f;
    uint4 pk;
    pk.x = pack_bf16x2(acc[0] * inv, acc[1] * inv); pk.y = pack_bf16x2(acc[2] * inv, acc[3] * inv);
    pk.z = pack_bf16x2(acc[4] * inv, acc[5] * inv); pk.w = pack_bf16x2(acc[6] * inv, acc[7] * inv);
    *reinterpret_cast<uint4*>(mo.out + (((size_t)b * mo.T + t) * mo.n_q_heads + h) * kD + c16 * 8) = pk;
    if (c16 == 0) mo.lse[((size_t)b * mo.n_q_heads + h) * mo.T + t] = s > 0.f ? m + __logf(s) : -INFINITY;
}
// One thread's share of a row: `count` pieces `hop` bytes apart from `row` on, 8 dims.  The largest LSE first, so
// that the pieces' weights do not depend on one another.
__device__ __forceinline__ void fold_pieces(uint32_t row, int count, uint32_t hop, int c16, float (&acc)[8], float& s, float& m)
{
    uint32_t at = row + 2 * kD;
    #pragma unroll 4
    for (int i = 0; i < count; ++i, at += hop) m = fmaxf(m, lds_f32(at));
    const float m_log2 = m == -INFINITY ? 0.f : m * 1.4426950408889634f;           // (all pieces empty: weights 0)
    at = row;
    #pragma unroll 2
    for (int i = 0; i < count; ++i, at += hop) {
        const float w = ex2(fmaf(lds_f32(at + 2 * kD), 1.4426950408889634f, -m_log2));
        uint32_t raw[4];
        lds_v4(at + c16 * 16, raw);
        s += w;
        #pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&raw[q]));
            acc[2 * q] = fmaf(w, f.x, acc[2 * q]); acc[2 * q + 1] = fmaf(w, f.y, acc[2 * q + 1]);
        }
    }
}
// Merges rows [0, n) of a run whose ns pieces lie in shared memory at `base` as [piece][row][272 bytes] and writes
// the results; row i is row r0 + i of its unit (token idx / g, head idx % g).  256 threads, no barrier: more than
// eight rows go two to a warp, 16 lanes of 8 dims each; of fewer a warp takes 128, 64, 32 or 16 dims, and the
// groups of lanes left over share the row's pieces and add up by shuffles.  What this costs is instructions one
// after the other (two warps per scheduler), divisions first: trip counts and shares go by shifts and by
// reciprocals from the host (verification of 2,048 keys, T = 8 8.3 -> 7.9 us).
__device__ __forceinline__ void merge_run(int tid, uint32_t base, int ns, int n, int r0, int b, int tok0, int head0, bool landed, const MergeOut& mo)
{
    const int warp = tid >> 5, lane = tid & 31;
    const uint32_t pstride = (uint32_t)n * kRowBytes;              // bytes between pieces
    const bool two_rows = n > 8;
    const int lg_lanes = n > 4 ? 4 : (n > 2 ? 3 : n);              // lanes of a group
    const int grp = lane >> lg_lanes, parts = 4 - lg_lanes;        // (two_rows: grp is the row)
    const int tasks = two_rows ? (n + 1) >> 1 : n << parts;
    // a group's pieces: first, first + 2^lg_step, ...
    const int first = two_rows ? 0 : grp, lg_step = two_rows ? 0 : 5 - lg_lanes;
    const int count = (ns - first + (1 << lg_step) - 1) >> lg_step;
    #pragma unroll 1
    for (int task = warp; task < tasks; task += 8) {
        const int r = two_rows ? 2 * task + grp : task >> parts;
        const int c16 = (lane & ((1 << lg_lanes) - 1)) + ((task & ((1 << parts) - 1)) << lg_lanes);
        float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, s = 0.f, m = -INFINITY;
        if (landed && r < n) fold_pieces(base + (uint32_t)r * kRowBytes + (uint32_t)first * pstride, count, pstride << lg_step, c16, acc, s, m);
        if (!two_rows) {
            float m_all = m;
            #pragma unroll 1
            for (int o = 1 << lg_lanes; o < 32; o <<= 1) m_all = fmaxf(m_all, __shfl_xor_sync(0xffffffffu, m_all, o));
            const float f = m == -INFINITY ? 0.f : ex2((m - m_all) * 1.4426950408889634f);
            m = m_all;
            s *= f;
            #pragma unroll
            for (int q = 0; q < 8; ++q) acc[q] *= f;
            #pragma unroll 1
            for (int o = 1 << lg_lanes; o < 32; o <<= 1) {
                s += __shfl_xor_sync(0xffffffffu, s, o);
                #pragma unroll
                for (int q = 0; q < 8; ++q) acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], o);
            }
        }
        if (landed && r < n && (two_rows || grp == 0)) {
            const int idx = r0 + r, tok = (idx * mo.inv_qg) >> 16;
            write_merged(acc, s, m, b, tok0 + tok, head0 + idx - tok * mo.qg, c16, mo);
        }
    }
}

// Rows of a unit that CTA `rank` of a cluster finishes: [begin, return value).  inv_cl: 2^16 / cluster size, rounded
// up (exact: for c CTAs and x = rows * rank <= 256 * 16, x (c inv_cl - 2^16) <= 4096 * 15 < 2^16).
__device__ __forceinline__ int merge_share(int unit_rows, int rank, int inv_cl, int* begin)
{
    *begin = (unit_rows * rank * inv_cl) >> 16;
    return (unit_rows * (rank + 1) * inv_cl) >> 16;
}

// What one pass of the merge takes: runs of rows of one unit (sequence, KV head, row group).
struct MergeSegment {
    int b, ns, n, split;             // sequence, pieces, rows, rows of them in the run's first block
    int src, src2;                   // workspace row of the first piece's first row; of the unit's second block
    int offset;                      // byte offset in the ring
    int r0, tok0, head0;             // first row inside the unit, the unit's first token and query head
};
constexpr int kMaxSegments = 8;
struct MergeList {
    MergeSegment seg[kMaxSegments];
    int n_seg, bytes, next_row;
};
static_assert(sizeof(MergeList) <= kMaxT * 8, "the list lies over the ancestor words");

// NB: row blocks of an item.  CL: the call's units are thread-block clusters, which merge their pieces in shared memory;
// otherwise a piece is final or goes through the workspace.  One kernel for both was 0.4 us slower where a call is
// short (2,048 keys, T = 8 7.20 -> 6.85 us, 300 keys 6.53 -> 6.29): code that is not there is not fetched.
//
// The kernels of one row block must not spill: the stack lies in L2 behind the stream of tiles (nearly all of L1 is shared memory), and
// 24 bytes of it between the last product and the partial rows took 0.5 us (26,112 keys, T = 16).  What an
// edge tile needs is therefore read from the tables when it comes and not kept over the loop.
template <int NB, bool CL>
__global__ void __launch_bounds__(kBoundThreads, 1)
verify_tc_kernel(const __grid_constant__ TcArgs args, const __grid_constant__ SyncArgs sync,
                 const __grid_constant__ SplitPlan plan, const __grid_constant__ CUtensorMap tmap_q,
                 const __grid_constant__ CUtensorMap tmap_k, const __grid_constant__ CUtensorMap tmap_v)
{
    constexpr int NSB = s_blocks(NB);                 // S blocks
    constexpr uint32_t kOCol = 512 - 128 * NB;        // first accumulator's TMEM column
    extern __shared__ unsigned char smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    unsigned char* sm = smem_raw + ((1024u - (raw & 1023u)) & 1023u);
    constexpr int NS = NB == 1 ? 3 : 2;               // K/V ring depth
    unsigned char* q_sm = sm;
    unsigned char* kv_sm = sm + NB * kQBlockBytes;
    unsigned char* misc = kv_sm + NS * kStageBytes + recv_extra(NB);
    uint64_t* bar_mem = reinterpret_cast<uint64_t*>(misc);                  // barriers in bytes 0-223 and 248-255 (see Bars)
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(misc + 224);
    volatile uint32_t* abort_flag = reinterpret_cast<volatile uint32_t*>(misc + 228);
    volatile uint32_t* write_ok = reinterpret_cast<volatile uint32_t*>(misc + 232);   // the counters allow global writes
    volatile int32_t* fin_go = reinterpret_cast<volatile int32_t*>(misc + 236);       // finishers: their waits succeeded
    // one row block, in the slots of barriers that only two blocks use: [8] what the softmax warps have posted (see pair_word)
    volatile int32_t* pair_s = reinterpret_cast<volatile int32_t*>(misc + 192);
    unsigned long long* anc_s = reinterpret_cast<unsigned long long*>(misc + kBarrierBytes);   // [64]
    int32_t* par_s = reinterpret_cast<int32_t*>(misc + 768);                          // [64]: parents in the prologue, then the rows' first visible keys
    float* xch = reinterpret_cast<float*>(misc + 1024);                               // [2][128] maxima that the halves of a row exchange (one row block)

    Bars B;
    SPARROW_TIMELINE_CALL(sync.call);
    if (threadIdx.x == 0) SPARROW_STAMP(0);                             // entry
    B.base = smem_u32(bar_mem);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const Item it = decode_item(plan, blockIdx.x);
    const int T = plan.T;
    const int qg = plan.group, tpb = plan.tok_per_block;   // query heads per KV head, tokens per 128-row block
    const int kv_len = plan.seq[it.b].kv_len;
    const int n_keys_seq = plan.seq[it.b].n_keys;
    const int n_tiles = (it.key_end - it.key_begin + kTile - 1) / kTile;
    const int n_jobs = n_tiles * NB;                        // key tile x row block
    const int block0 = it.group * NB;                       // first 128-row block of this item

    // K and V tiles of a lone call leave L2 before anything else does: a cache is streamed once per call, and would
    // otherwise push out the code, the queries and the partial rows, which then come back from DRAM behind the
    // stream of tiles.  All tiles of a call that takes more than half of L2, half of them of a shorter one,
    // whose next call on the same cache then finds as much as before (26,112 keys on one and the same cache: none
    // 15.9 us, half 16.0, all 17.3; caches out of L2: 18.6, 18.2, 17.9).  In batches it gave nothing.
    uint64_t stream_policy;
    if (args.leave_l2 == 0) asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(stream_policy));
    else if (args.leave_l2 == 1) asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 0.5;" : "=l"(stream_policy));
    else asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(stream_policy));
    auto issue_k = [&](int j) {                     // producer thread only
        const int st = j % NS;
        const uint32_t dst = smem_u32(kv_sm + st * kStageBytes);
        const int row = it.key_begin + j * kTile;
        mbar_expect_tx(B.k_full(st), 2 * kSubTileBytes);
        tma_load_4d(dst, &tmap_k, 0, row, it.kvh, it.b, B.k_full(st), stream_policy);
        tma_load_4d(dst + kSubTileBytes, &tmap_k, 64, row, it.kvh, it.b, B.k_full(st), stream_policy);
    };
    auto issue_v = [&](int j) {
        const int st = j % NS;
        const uint32_t dst = smem_u32(kv_sm + st * kStageBytes + 2 * kSubTileBytes);
        const int row = it.key_begin + j * kTile;
        uint32_t bar = B.v_full(st);
        // One row block: V counts on the barrier of its tile's P, so that the product waits once; the last tile's has its own
        // (its rows past the end are zeroed ahead of P).  The phase is the tile's: its stage is free, so P of the
        // tile before in it was complete.
        if (NB == 1) {
            if (j < n_tiles - 1) bar = B.p_full(st);
            else mbar_arrive(B.p_full(st));
        }
        mbar_expect_tx(bar, 2 * kSubTileBytes);
        tma_load_4d(dst, &tmap_v, 0, row, it.kvh, it.b, bar, stream_policy);
        tma_load_4d(dst + kSubTileBytes, &tmap_v, 64, row, it.kvh, it.b, bar, stream_policy);
    };

    // The first tiles are on their way into L2 while the kernel waits to be released behind its predecessor (1.7 us), which may
    // still write them: the loads behind the wait find what it wrote, in L2 like everything else.  Two tiles: 26,112 keys alone
    // 17.4 -> 16.9 us, three sequences of 9,001 21.6 -> 20.2, caches that L2 holds as before; one tile 16.9 and 21.1, three
    // 17.7 and 20.9, all of them 19.6 and 23.3 (the loads queue behind them).  Row groups share their tiles: the first one's items ask.
    if (warp == kGateWarp && lane == 0 && sync.wait_first == 1 && it.group == 0) {
        #pragma unroll 1
        for (int j = 0; j < n_tiles && j < kPrefetchTiles; ++j) {
            const int row = it.key_begin + j * kTile;
            tma_prefetch_4d(&tmap_k, 0, row, it.kvh, it.b, stream_policy);
            tma_prefetch_4d(&tmap_k, 64, row, it.kvh, it.b, stream_policy);
            tma_prefetch_4d(&tmap_v, 0, row, it.kvh, it.b, stream_policy);
            tma_prefetch_4d(&tmap_v, 64, row, it.kvh, it.b, stream_policy);
        }
    }

    // ---- setup: barriers, TMEM.  Nothing here waits for an earlier kernel: every warp runs on to its own first
    // wait before the loads start.  With the wait and the first loads in front of the CTA barrier the MMA
    // warp fetched its code behind the stream of tiles, up to 2 us late (26,112 keys, T = 16 18.3 -> 17.7 us).
    if (warp == kProducerWarp && lane == 0) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(&tmap_q) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&tmap_k) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&tmap_v) : "memory");
        for (int i = 0; i < 3; ++i) { mbar_init(B.k_full(i), 1); mbar_init(B.k_empty(i), 1); mbar_init(B.v_full(i), 1); mbar_init(B.v_empty(i), 1); }      // (a tile is read by every block)
        // one row block: a P block comes from all eight softmax warps and counts its tile's V; two: from the block's own four
        for (int i = 0; i < 3; ++i) { mbar_init(B.s_full(i), 1); mbar_init(B.p_full(i), NB == 1 ? 9 : 4); }
        for (int i = 0; i < 4; ++i) mbar_init(B.o_done(0, i), 1);
        if (NB == 2) {
            mbar_init(B.p_full(3), 4);
            for (int i = 0; i < 4; ++i) mbar_init(B.o_done(1, i), 1);
        } else {
            for (int i = 0; i < 8; ++i) pair_s[i] = 0;
        }
        mbar_init(B.q_full(), 1);
        mbar_init(B.fin(), 1);
        *abort_flag = 0;
        *write_ok = sync.enabled ? 0u : 1u;
        fence_barrier_init();
    }
    if (warp == kMmaWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // (waited for ahead of the first access to a peer.  The rows that peers send come to a stage of the ring: where this piece
    // uses it, the producer's warp arrives once it is idle.)
    if (CL && !(warp == kProducerWarp && n_tiles >= NS)) cluster_arrive_relaxed();
    const uint32_t tmem = *tmem_slot;
    if (threadIdx.x == 0) SPARROW_STAMP(1);                             // set-up done

    if (warp == kProducerWarp) {
        // ================= TMA producer =================
        if (lane == 0) {
            int j_first = 0;                                 // tiles requested ahead of the wait
            if (sync.wait_first) {
                if (sync.wait_first == 2)
                    for (; j_first < n_tiles && j_first < NS && it.key_begin + (j_first + 1) * kTile <= kv_len; ++j_first) { issue_k(j_first); issue_v(j_first); }
                wait_for_predecessors();
            }
            // Q first (the first S = Q K^T needs it and it is small), then K and V tiles in the order
            // they are consumed.
            mbar_expect_tx(B.q_full(), (uint32_t)(NB * 2 * 64 * qg * tpb * 2));   // two boxes of 64 dims x g heads x p tokens per block
            #pragma unroll
            for (int blk = 0; blk < NB; ++blk) {
                const uint32_t dst = smem_u32(q_sm + blk * kQBlockBytes);
                const int tok = (block0 + blk) * tpb;
                tma_load_4d(dst, &tmap_q, 0, it.kvh * qg, tok, it.b, B.q_full());
                tma_load_4d(dst + kSubTileBytes, &tmap_q, 64, it.kvh * qg, tok, it.b, B.q_full());
            }
            for (int j = j_first; j < n_tiles && j < NS; ++j) { issue_k(j); issue_v(j); }
            // refill whichever ring has a free slot; K slots free up ahead of V slots
            int jk = NS < n_tiles ? NS : n_tiles, jv = jk;
            uint32_t idle = 0;
            #pragma unroll 1
            while (jk < n_tiles || jv < n_tiles) {
                bool progress = false;
                if (jk < n_tiles && mbar_try_wait(B.k_empty(jk % NS), (jk / NS - 1) & 1)) { issue_k(jk); ++jk; progress = true; }
                if (jv < n_tiles && mbar_try_wait(B.v_empty(jv % NS), (jv / NS - 1) & 1)) { issue_v(jv); ++jv; progress = true; }
                if (progress) idle = 0;
                else if (++idle > kSpinLimit) { atomicOr(args.status, timeout_bits(kSiteProducer)); *abort_flag = 1; break; }
            }
            if (CL && n_tiles >= NS) {
                const int last = recv_last_tile(NB, n_tiles);           // (its phase is the one in progress or just completed: see issue_v)
                if (!mbar_wait(B.v_empty(recv_stage(NB, n_tiles)), (last / NS) & 1)) { atomicOr(args.status, timeout_bits(kSiteProducer)); *abort_flag = 1; }
            }
        }
        // Peers may write over the stage now.  What was written to it and read from it, by the loads, by zero_v_tail and by the
        // products, is ordered ahead of this by the products' barrier, and the arrival releases it.  The fence in a releasing
        // arrival takes 0.4 us: here it runs beside the last two tiles, behind the last product it took 8,000 keys, T = 8 from 9.2 to 9.6.
        if (CL && n_tiles >= NS) {
            __syncwarp();
            cluster_arrive();
        }
    } else if (warp == kMmaWarp) {
        // ================= MMA issuer =================
        // the whole warp walks the jobs, converged; one elected lane issues (see elect_one)
        {
            const uint32_t tmem_u = __shfl_sync(0xffffffffu, tmem, 0);
            // V rows past the end of the sequence may hold anything: they are zeroed in shared memory, so that
            // 0 * x stays 0, ahead of the last tile's first product and beside its softmax.
            auto zero_v_tail = [&](int j) {
                const int valid = n_keys_seq - (it.key_begin + j * kTile);
                if (valid >= kTile) return;
                unsigned char* v_tile = kv_sm + (j % NS) * kStageBytes + 2 * kSubTileBytes;
                #pragma unroll 1
                for (int i = valid * 8 + lane; i < kTile * 8; i += 32) {
                    *reinterpret_cast<uint4*>(v_tile + i * 16) = make_uint4(0, 0, 0, 0);
                    *reinterpret_cast<uint4*>(v_tile + kSubTileBytes + i * 16) = make_uint4(0, 0, 0, 0);
                }
                fence_proxy_async();
                __syncwarp();
            };
            // descriptors differ from job to job only in their 14-bit address field
            const uint64_t q_desc0 = smem_desc(smem_u32(q_sm), 16, 1024);
            const uint64_t k_desc0 = smem_desc(smem_u32(kv_sm), 16, 1024);
            const uint64_t v_desc0 = smem_desc(smem_u32(kv_sm) + 2 * kSubTileBytes, kSubTileBytes, 1024);
            // Rows that no box of Q covers are zeros, as are the tokens of a box past the last: scores and P of padding are zeros
            // as well, and products of zeros take less power, which is what long calls are short of (four sequences of
            // 20,000 keys, T = 20, 45 % of the rows padding, 41.2 -> 40.5 us; three of 9,001, T = 23 20.5 -> 20.0).
            #pragma unroll 1
            for (int i = lane + qg * tpb * 8; i < kBlockRows * 8; i += 32)
                #pragma unroll
                for (int sub = 0; sub < 2 * NB; ++sub) *reinterpret_cast<uint4*>(q_sm + sub * kSubTileBytes + i * 16) = make_uint4(0, 0, 0, 0);
            fence_proxy_async();
            __syncwarp();
            // (a bounded wait must not include what is left of the predecessor's time: kernels that let their
            // dependents start early may run on for longer than its polls)
            if (sync.wait_first) wait_for_predecessors();
            bool ok = mbar_wait_warp(B.q_full(), 0);
            if (lane == 0) SPARROW_STAMP(2);                                           // Q landed
            if constexpr (NB == 2) {
                // Two row blocks, each with its own softmax warpgroup.  Job n = (key tile j = n / 2,
                // block b = n % 2).  Block b owns TMEM columns [128 b, 128 b + 128) for its scores,
                // with its P (bf16, 64 columns) written over the upper half, and the accumulator at
                // 256 + 128 b.  Per block the chain is scores -> softmax -> O += P V -> next scores;
                // the two blocks' chains interleave, so the tensor pipe works for one block while
                // the other block's warpgroup is in its exponentials.
                constexpr uint32_t idesc_qk = idesc_bf16(false);
                constexpr uint32_t idesc_pv = idesc_bf16(true);
                auto issue_qk2 = [&](int m) -> bool {
                    const int j = m >> 1, b = m & 1, st = j % NS;
                    if (b == 0) {                                             // first use of this K tile
                        if (!mbar_wait_warp(B.k_full(st), (j / NS) & 1)) return false;
                        tc_fence_after();
                        if (j == 0 && lane == 0) SPARROW_STAMP(3);                   // first K tile landed
                    }
                    const uint64_t qd = q_desc0 + (uint64_t)((b * kQBlockBytes) >> 4);
                    const uint64_t kd = k_desc0 + (uint64_t)((st * kStageBytes) >> 4);
                    if (elect_one()) {
                        #pragma unroll
                        for (int ks = 0; ks < 8; ++ks) {
                            const uint32_t off = ((ks >> 2) * kSubTileBytes + (ks & 3) * 32) >> 4;
                            mma_ss(tmem_u + b * 128, qd + off, kd + off, idesc_qk, ks > 0);
                        }
                        tc_commit(B.s_full(b));
                        if (b == 1) tc_commit(B.k_empty(st));                 // last use of the tile
                    }
                    __syncwarp();
                    return true;
                };
                for (int m = 0; m < 2 && m < n_jobs && ok; ++m) ok = issue_qk2(m);
                #pragma unroll 1
                for (int n = 0; n < n_jobs && ok; ++n) {
                    const int j = n >> 1, b = n & 1, st = j % NS;
                    if (b == 0) {
                        if (!mbar_wait_warp(B.v_full(st), (j / NS) & 1)) { ok = false; break; }
                        if (j == n_tiles - 1) zero_v_tail(j);
                    }
                    if (!mbar_wait_warp(B.p_full(b), j & 1)) { ok = false; break; }
                    tc_fence_after();
                    const uint64_t vd = v_desc0 + (uint64_t)((st * kStageBytes) >> 4);
                    #pragma unroll
                    for (int half = 0; half < 2; ++half) {                    // keys 64-127, then 0-63, as their P arrives
                        if (half == 1) {
                            if (!mbar_wait_warp(B.p_full(2 + b), j & 1)) { ok = false; break; }
                            tc_fence_after();
                        }
                        if (elect_one()) {
                            #pragma unroll
                            for (int kk = 4 - half * 4; kk < 8 - half * 4; ++kk)
                                mma_ts(tmem_u + 256 + b * 128, tmem_u + b * 128 + 64 + kk * 8, vd + (uint64_t)((kk * 2048) >> 4),
                                       idesc_pv, (j > 0 || half > 0 || kk > 4) ? 1u : 0u);
                            if (half == 1) {
                                tc_commit(B.o_done(b, j));
                                if (b == 1) tc_commit(B.v_empty(st));
                            }
                        }
                        __syncwarp();
                    }
                    if (!ok) break;
                    if (n + 2 < n_jobs) ok = issue_qk2(n + 2);                // this block's next scores
                }
            } else {
                // One row block: a job is a key tile, the scores of tile j lie in S block j % NSB.
                constexpr uint32_t idesc_qk = idesc_bf16(false);
                constexpr uint32_t idesc_pv = idesc_bf16(true);
                auto issue_qk = [&](int ring) {                           // S = Q K^T of the tile in stage and S block `ring`
                    const uint64_t kd = k_desc0 + (uint64_t)((ring * kStageBytes) >> 4);
                    if (elect_one()) {
                        #pragma unroll
                        for (int ks = 0; ks < 8; ++ks) {
                            const uint32_t off = ((ks >> 2) * kSubTileBytes + (ks & 3) * 32) >> 4;
                            mma_ss(tmem_u + ring * 128, q_desc0 + off, kd + off, idesc_qk, ks > 0);
                        }
                        tc_commit(B.s_full(ring));
                        tc_commit(B.k_empty(ring));
                    }
                    __syncwarp();
                };
                static_assert(NB == 2 || NS == NSB, "one ring index for stages and S blocks");
                #pragma unroll 1
                for (int j = 0; j < NS && j < n_tiles && ok; ++j) {
                    ok = mbar_wait_warp(B.k_full(j), 0);
                    if (!ok) break;
                    tc_fence_after();
                    if (j == 0 && lane == 0) SPARROW_STAMP(3);                       // first K tile landed
                    issue_qk(j);
                }
                int ring = 0;                                             // tile modulo 3
                uint32_t parity = 0;
                #pragma unroll 1
                for (int j = 0; j < n_tiles && ok; ++j) {
                    if (j == n_tiles - 1) {
                        ok = mbar_wait_warp(B.v_full(ring), 0);
                        if (!ok) break;
                        zero_v_tail(j);
                    }
                    const uint64_t vd = v_desc0 + (uint64_t)((ring * kStageBytes) >> 4);
                    const uint32_t p_col = tmem_u + ring * 128, o_bar = B.o_done(0, j), v_bar = B.v_empty(ring), k_bar = B.k_full(ring);
                    const int this_ring = ring;
                    const uint32_t this_parity = parity;
                    if (++ring == NS) { ring = 0; parity ^= 1u; }
                    ok = mbar_wait_tight(B.p_full(this_ring), this_parity);
                    if (!ok) break;
                    tc_fence_after();
                    if (elect_one()) {
                        #pragma unroll
                        for (int kk = 0; kk < 8; ++kk)
                            mma_ts(tmem_u + kOCol, p_col + (kk >> 2) * 64 + (kk & 3) * 8, vd + (uint64_t)((kk * 2048) >> 4),
                                   idesc_pv, (j > 0 || kk > 0) ? 1u : 0u);
                        tc_commit(o_bar);
                        tc_commit(v_bar);
                    }
                    __syncwarp();
                    if (j + NS < n_tiles) {                               // the S block and the stage that have become free
                        ok = mbar_wait_tight(k_bar, this_parity ^ 1u);
                        if (!ok) break;
                        tc_fence_after();
                        issue_qk(this_ring);
                    }
                }
            }
            if (lane == 0) SPARROW_STAMP(4);                            // last product issued
            if (!ok && lane == 0) { atomicOr(args.status, timeout_bits(kSiteMma)); *abort_flag = 1; }
        }
    } else if (warp == kGateWarp) {
        // The tree and the window bounds, beside the first loads; the softmax warps wait for them at a barrier.
        {
            const int Tt = plan.T_tree;
            const bool needs_tree = it.key_end > kv_len;       // this piece reaches the draft block
            if (sync.wait_first) wait_for_predecessors();
            // (behind the wait: a dependent that starts early may rely on everything before this call; not
            // from the producer, whose refills it held up)
            if (sync.enabled) let_dependents_launch();
            int par[2] = {-1, -1}, lo[2] = {0, 0};
            #pragma unroll
            for (int k = 0; k < 2; ++k) {
                const int i = lane + 32 * k;
                if (needs_tree && i < Tt) par[k] = ld_behind(args.parents + (size_t)it.b * Tt + i);
                if (args.first_visible && i < T) lo[k] = ld_behind(args.first_visible + (size_t)it.b * T + i);
            }
            if (needs_tree) build_ancestor_words(par[0], par[1], anc_s, Tt, args.status);
            // Lower window bound of every query token, clamped to what this call streams: a bound
            // left of the first streamed key cannot be honoured (the keys in between were not planned)
            // and is reported.
            const int key0 = plan.seq[it.b].key0;
            #pragma unroll
            for (int k = 0; k < 2; ++k) {
                const int t = lane + 32 * k;
                if (t < T) {
                    if (lo[k] < key0) {
                        if (args.first_visible) atomicOr(args.status, kStatAnchor);
                        lo[k] = key0;
                    }
                    par_s[t] = lo[k] < kv_len ? lo[k] : kv_len;
                }
            }
            tables_ready_arrive();
        }
        if (lane == 0 && sync.enabled) {
            // Overlapped mode: whoever read this parity's partial buffer two calls ago must be done
            // before this CTA's first global write, and final results may only follow every earlier
            // call's.  Waiting here, beside the main loop, keeps the round trip to the counters off the
            // epilogue's critical path.  1 = go, 2 = a wait gave up.
            bool go = wait_counter(sync.fin_done + sync.parity, sync.fin_wait_same);
            if (!go) atomicOr(args.status, timeout_bits(kSiteWriteSame));
            if (go && (CL || plan.seq[it.b].n_splits == 1)) {
                go = wait_counter(sync.fin_done + (sync.parity ^ 1), sync.fin_wait_other);
                if (!go) atomicOr(args.status, timeout_bits(kSiteWriteOther));
            }
            __threadfence_block();
            *write_ok = go ? 1u : 2u;
        }
    } else if (warp < 8) {
        // ================= softmax =================
        tables_ready_sync();                             // ancestor words and window bounds are in shared memory
        const int wg = warp >> 2;                        // key-column half this thread takes
        const int row_local = (warp & 3) * 32 + lane;    // TMEM lane = row inside the 128-row block
        const uint32_t lane_addr = tmem + ((uint32_t)((warp & 3) * 32) << 16);
        const float c2 = args.scale_log2e;
        const float thr = kRescaleLog2 / c2;             // threshold in raw score units
        const uint64_t c22 = pair_of(c2, c2);
        const int g_row = row_local % qg;
        // A thread's row: of the one block, or of its warpgroup's own.
        const int blk = NB == 1 ? 0 : wg;
        const int t_row = (block0 + blk) * tpb + row_local / qg;
        const bool row_ok = row_local < tpb * qg && t_row < T;
        // (read from the tables where they are needed; the queries are the last T nodes of the tree)
        auto row_anc = [&]() { return (row_ok && it.key_end > kv_len) ? anc_s[plan.T_tree - T + t_row] : 0ull; };
        auto row_lo = [&]() { return row_ok ? par_s[t_row] : 0; };
        const int lo_first = row_lo();
        // tiles whose every key is visible to the warp's rows: [j_head, j_tail)
        const int j_tail = (min(it.key_end, kv_len) - it.key_begin) / kTile;
        const int j_head = __reduce_max_sync(0xffffffffu, lo_first > it.key_begin ? (lo_first - it.key_begin + kTile - 1) / kTile : 0);
        float m_ref = -INFINITY, l_run = 0.f;
        bool ok = true;

        // visibility word, for the 64 keys that start at key j0, of a row with ancestor word `anc_row` and lower
        // window bound `lo` (which never exceeds kv_len): the prefix columns, then the ancestor word shifted to the
        // draft block's column, cut at the end of the key range and left of the window
        auto vis_word = [&](int j0, unsigned long long anc_row, int lo) -> unsigned long long {
            const int d0 = kv_len - j0;                                 // column of draft token 0 (any sign)
            const int nval = it.key_end - j0;                           // valid columns (may be <= 0)
            unsigned long long vis;
            if (d0 >= 64) vis = ~0ull;
            else if (d0 > 0) vis = ((1ull << d0) - 1ull) | (anc_row << d0);
            else if (d0 > -64) vis = anc_row >> (-d0);
            else vis = 0ull;
            if (nval <= 0) vis = 0ull;
            else if (nval < 64) vis &= (1ull << nval) - 1ull;
            const int cut = lo - j0;
            if (cut >= 64) vis = 0ull;
            else if (cut > 0) vis &= ~((1ull << cut) - 1ull);
            return vis;
        };
        if constexpr (NB == 2) {
            // ---- two row blocks: warpgroup g owns block g, one thread per query row, and works
            // through the block's half-tile jobs on its own -- no exchange with the other warpgroup,
            // whose exponentials fill the gaps this one leaves while it waits for the tensor pipe.
            const uint32_t s_addr = lane_addr + blk * 128;
            #pragma unroll 1
            for (int j = 0; j < n_tiles; ++j) {
                const int tile0 = it.key_begin + j * kTile;
                if (!mbar_wait_warp(B.s_full(blk), j & 1)) { ok = false; break; }
                tc_fence_after();
                // First pass over the row's 128 scores, 64 at a time: the maximum.  In a tile that crosses a
                // visibility boundary of some row the scores are masked on the way; the lower 64, which are
                // fetched again for the second pass, go back to TMEM masked.
                const bool edge = j >= j_tail || j < j_head;
                float x0[32], x1[32];
                tmem_ld32(s_addr, x0);
                tmem_ld32(s_addr + 32, x1);
                tmem_wait_ld();
                if (edge) {
                    const unsigned long long vis = vis_word(tile0, row_anc(), row_lo());
                    mask_chunk(x0, (uint32_t)vis);
                    mask_chunk(x1, (uint32_t)(vis >> 32));
                    tmem_st32(s_addr, reinterpret_cast<uint32_t*>(x0));
                    tmem_st32(s_addr + 32, reinterpret_cast<uint32_t*>(x1));
                    tmem_wait_st();
                }
                float mx = chunk_max(x0);
                tmem_ld32(s_addr + 64, x0);
                mx = fmaxf(mx, chunk_max(x1));
                tmem_ld32(s_addr + 96, x1);
                tmem_wait_ld();
                if (edge) {
                    const unsigned long long vis = vis_word(tile0 + 64, row_anc(), row_lo());
                    mask_chunk(x0, (uint32_t)vis);
                    mask_chunk(x1, (uint32_t)(vis >> 32));
                }
                mx = fmaxf(mx, fmaxf(chunk_max(x0), chunk_max(x1)));
                // lazy reference maximum, per row; the accumulator is rescaled by the whole warp (the
                // TMEM accesses are warp-wide) whenever one of its rows moved
                const bool need = row_ok && (mx > m_ref + thr || (m_ref == -INFINITY && mx > -INFINITY));
                if (__any_sync(0xffffffffu, need)) {
                    float alpha = 1.f;
                    if (need) {
                        alpha = (m_ref == -INFINITY) ? 0.f : ex2((m_ref - mx) * c2);
                        m_ref = mx;
                        l_run *= alpha;
                    }
                    if (j > 0) {                                            // O holds earlier tiles
                        if (!mbar_wait_warp(B.o_done(blk, j - 1), ((j - 1) >> 2) & 1)) { ok = false; break; }
                        tc_fence_after();
                        const uint32_t o_addr = lane_addr + kOCol + blk * 128;
                        #pragma unroll 1
                        for (int ch = 0; ch < 8; ++ch) {
                            float o[16];
                            tmem_ld16(o_addr + ch * 16, o);
                            tmem_wait_ld();
                            #pragma unroll
                            for (int c = 0; c < 16; ++c) o[c] *= alpha;
                            tmem_st16(o_addr + ch * 16, reinterpret_cast<uint32_t*>(o));
                        }
                    }
                }
                // second pass: p = 2^(s c2 - m c2), row sum from the unrounded p, P (bf16) over the upper half
                // of the score block -- first the upper 64 keys (their scores are in registers and their
                // columns are the ones P overwrites), then the lower 64, fetched again.  The upper keys'
                // half of O += P V runs beside the exponentials of the lower ones.
                const float mc = m_ref > -INFINITY ? m_ref * c2 : row_ok ? 0.f : INFINITY;     // (padding: P is 0)
                const uint64_t neg_mc2 = pair_of(-mc, -mc);
                uint64_t sum[2] = {0ull, 0ull};
                exp_chunk(x0, c22, neg_mc2, sum, s_addr + 96);
                tmem_ld32(s_addr, x0);
                exp_chunk(x1, c22, neg_mc2, sum, s_addr + 112);
                tmem_ld32(s_addr + 32, x1);
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(B.p_full(blk));
                tmem_wait_ld();
                exp_chunk(x0, c22, neg_mc2, sum, s_addr + 64);
                exp_chunk(x1, c22, neg_mc2, sum, s_addr + 80);
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(B.p_full(2 + blk));
                l_run += sum_of(sum);
            }
        } else {
        // One row block: the two warpgroups split a tile's 128 keys; thread = one row, 64 keys.  The two warps that share
        // 32 rows run apart from one another, by a tile at most (softmax_pair.cuh).
        const int sb_wg = 64 * wg;
        const uint32_t pair_id = 4u + (uint32_t)(warp & 3);
        float x0[32], x1[32];
        // scores above this need a new reference (rows of padding never do)
        float limit = row_ok ? -INFINITY : INFINITY;
        float mc = row_ok ? 0.f : INFINITY;                                 // reference in log2 units, 0 as long as there is none (padding: P is 0)
        float m_acc = -INFINITY;                                            // what the accumulator is on; m_ref: what this tile's P is on
        int sb = 0;                                                         // the tile's S block
        uint32_t s_parity = 0, moved = 0;                                   // moved: bit 0 in the tile passed last, bit 1 in the one before
        bool have = false;                                                  // the tile's scores are requested
        uint32_t p_addr = 0, p_bar = 0;                                     // P of the tile before, which is not handed over, and its barrier
        int word = 0;                                                       // the partner's
        auto post = [&](float mine) {                                       // (the partner has read what was posted before)
            xch[wg * 128 + row_local] = mine;
            __threadfence_block();
            __syncwarp();
        };
        #pragma unroll 1
        for (int j = 0;; ++j) {
            float mx = -INFINITY;
            word = pair_s[warp ^ 4];                                        // (looked at below: the scores take longer)
            if (j < n_tiles) {
                if (__builtin_expect(!have, 0)) {                           // not there when the tile before looked for them
                    ok = __all_sync(0xffffffffu, mbar_wait_warp(B.s_full(sb), s_parity));
                    tc_fence_after();
                    if (!ok) {
                        if (j == 0) { post(-INFINITY); pair_sync(pair_id); }
                        break;
                    }
                    tmem_ld32(lane_addr + sb * 128 + sb_wg, x0);
                    tmem_ld32(lane_addr + sb * 128 + sb_wg + 32, x1);
                }
                tmem_wait_ld();
                if (j >= j_tail || j < j_head) {
                    const unsigned long long vis = vis_word(it.key_begin + j * kTile + sb_wg, row_anc(), row_lo());
                    mask_chunk(x0, (uint32_t)vis);
                    mask_chunk(x1, (uint32_t)(vis >> 32));
                }
                mx = fmaxf(chunk_max(x0), chunk_max(x1));
            }
            // settle the tile before, pass this one
            if (__builtin_expect(j == 0 || (moved & 1u) || __any_sync(0xffffffffu, mx > limit || !pair_quiet(word, j - 1)), 0)) {
                if (j > 0) {
                    #pragma unroll 1
                    for (uint32_t i = 0; ok; ++i) {
                        word = __shfl_sync(0xffffffffu, pair_s[warp ^ 4], 0);
                        if (pair_passed(word) >= j) break;
                        if (i >= 256) __nanosleep(100);
                        if (i >= kSpinLimit) ok = false;
                    }
                    if (!ok) break;
                    const bool other = pair_moved(word, j - 1);
                    if (other || (moved & 1u)) {
                        float m_new = m_ref;
                        if (other) {
                            __threadfence_block();
                            m_new = fmaxf(m_new, xch[(wg ^ 1) * 128 + row_local]);
                            __syncwarp();
                            if (lane == 0) pair_s[warp] = pair_word(j, true, moved);
                        }
                        const float of_p = rescale(m_ref, m_new, c2), of_acc = rescale(m_acc, m_new, c2);
                        tmem_wait_st();
                        if (__any_sync(0xffffffffu, of_p != 1.f)) {
                            #pragma unroll 1
                            for (int h = 0; h < 2; ++h) {
                                uint32_t p[16];
                                tmem_ld16(p_addr + 16 * h, reinterpret_cast<float*>(p));
                                tmem_wait_ld();
                                #pragma unroll
                                for (int c = 0; c < 16; ++c)
                                    p[c] = pack_bf16x2(__uint_as_float(p[c] << 16) * of_p, __uint_as_float(p[c] & 0xffff0000u) * of_p);
                                tmem_st16(p_addr + 16 * h, p);
                            }
                        }
                        if (j > 1 && __any_sync(0xffffffffu, of_acc != 1.f)) {  // (this half of it)
                            ok = __all_sync(0xffffffffu, mbar_wait_warp(B.o_done(0, j - 2), ((j - 2) >> 2) & 1));
                            if (!ok) break;
                            tc_fence_after();
                            #pragma unroll 1
                            for (int ch = 0; ch < 4; ++ch) {
                                const uint32_t o_addr = lane_addr + kOCol + sb_wg + ch * 16;
                                float o[16];
                                tmem_ld16(o_addr, o);
                                tmem_wait_ld();
                                #pragma unroll
                                for (int c = 0; c < 16; ++c) o[c] *= of_acc;
                                tmem_st16(o_addr, reinterpret_cast<uint32_t*>(o));
                            }
                        }
                        l_run *= of_p;
                        m_ref = m_acc = m_new;
                        if (m_new > -INFINITY) { limit = m_new + thr; mc = m_new * c2; }
                    }
                }
                moved <<= 1;
                const float mine = mx > limit ? mx : -INFINITY;
                if (j == 0) {
                    post(mine);
                    pair_sync(pair_id);
                    m_ref = m_acc = fmaxf(mine, xch[(wg ^ 1) * 128 + row_local]);
                    if (m_acc > -INFINITY) { limit = m_acc + thr; mc = m_acc * c2; }
                    // The second warp of the pair starts half a tile's exponentials late and stays so: what each does besides them
                    // falls into the other's; in step, both wait for the exponentials together.  Lone calls, caches in L2, in step
                    // -> like this, us: three tiles a CTA (4,089 keys, T = 8) 8.26 -> 8.00, four (8,000 keys, T = 8) 9.46 -> 9.05,
                    // (3,000 keys, T = 64) 10.63 -> 10.30, five or six (26,112 keys) 16.49 -> 16.28, 14 or 15 (64 nodes on
                    // 16,384 keys) 22.63 -> 22.32.  41 tiles a CTA on 20 CTAs, 0.77 to 0.79 us each: 42.4 and 42.4.  One and two
                    // tiles: alike (1,500 keys, T = 16 7.03 and 7.08, 4,000 keys, T = 8 7.88 and 7.86).
                    if (wg == 1 && n_tiles > 2) {
                        const uint32_t c0 = (uint32_t)clock();
                        while ((uint32_t)clock() - c0 < kPairLag) {}
                    }
                    __syncwarp();
                } else if (__any_sync(0xffffffffu, mine > -INFINITY)) {
                    if (moved & 2u) {                                       // what this warp posted for the tile before
                        #pragma unroll 1
                        for (uint32_t i = 0; ok && !pair_settled(__shfl_sync(0xffffffffu, pair_s[warp ^ 4], 0), j - 1); ++i) {
                            if (i >= 256) __nanosleep(100);
                            if (i >= kSpinLimit) ok = false;
                        }
                        if (!ok) break;
                    }
                    moved |= 1u;
                    post(mine);
                    if (mine > -INFINITY) {
                        l_run *= rescale(m_ref, mine, c2);
                        m_ref = mine;
                        mc = mine * c2;
                    }
                }
            } else {
                moved <<= 1;
            }
            // (the post first: the partner may be waiting for it.  The order and one vote for both questions: 41 tiles alone 44.3 -> 42.5 us,
            // a call of two tiles 7.04 -> 7.20, where P of the last tile is handed over a little later.)
            if (lane == 0 && j < n_tiles) pair_s[warp] = pair_word(j + 1, false, moved);
            if (j > 0) {                                                    // P of the tile before is in TMEM and settled
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(p_bar);
            }
            if (j == n_tiles) break;
            // p = 2^(s c2 - m c2), row sum from the unrounded p, P (bf16) over this thread's own scores
            const uint64_t neg_mc2 = pair_of(-mc, -mc);
            uint64_t sum[2] = {0ull, 0ull};
            p_addr = lane_addr + sb * 128 + sb_wg;                          // this thread's scores, then its P
            p_bar = B.p_full(sb);
            exp_chunk(x0, c22, neg_mc2, sum, p_addr);
            if (++sb == NSB) { sb = 0; s_parity ^= 1u; }
            const uint32_t s_next = lane_addr + sb * 128 + sb_wg;
            have = j + 1 < n_tiles && __all_sync(0xffffffffu, mbar_test_wait(B.s_full(sb), s_parity));
            tc_fence_after();
            if (have) tmem_ld32(s_next, x0);
            exp_chunk(x1, c22, neg_mc2, sum, p_addr + 16);
            if (have) tmem_ld32(s_next + 32, x1);
            l_run += sum_of(sum);
        }
        if (!ok && lane == 0) pair_s[warp] = pair_word(n_tiles, false, 0u);  // (the partner need not wait as well)
        // The sums meet, behind the row as it is staged below: every Q K^T is complete, Q's place is free.
        reinterpret_cast<float*>(q_sm + row_local * kRowBytes + kD * 2)[1 + wg] = l_run;
        pair_sync(pair_id + 4u);
        }
        // ---- epilogue: normalised partial output + natural-log LSE -------------------------------
        if (tid == 0) SPARROW_STAMP(5);                                 // softmax loop left
        const bool direct = !CL && plan.seq[it.b].n_splits == 1;                  // the only piece: write the final result
        constexpr bool clustered = CL;                           // the unit's pieces meet in the cluster's shared memory
        if (tid == 0) {
            // Global writes start below.  In overlapped mode a lane of the gate warp has been waiting,
            // since the kernel started, for the counters that allow them (see there).
            uint32_t w = *write_ok;
            for (uint32_t i = 0; w == 0u && i < (1u << 26); ++i) { __nanosleep(20); w = *write_ok; }
            __threadfence_block();
            if (w == 1u && sync.enabled && blockIdx.x == 0) sync.arrivals[(sync.slot + 2) & 3] = 0u;   // the call after next: unused by now
            *write_ok = w == 1u ? 1u : 2u;
        }
        // A thread finishes one row: its 64 output dims [64 wg, 64 wg + 64) of the one block, or all 128 of its
        // warpgroup's own block.
        const int dim0 = NB == 1 ? 64 * wg : 0;
        // Partial rows are staged as they lie in the workspace ([row][272 bytes]: an odd number of 16-byte
        // chunks, so a warp's rows do not share banks) and leave as one bulk copy per block: the copy's own
        // completion orders them ahead of the publication, where ordinary stores needed a second pass
        // and a proxy fence.  The staging area is the Q blocks and the start of the K ring: every Q K^T of the one block has
        // completed with its last scores; with two, the other block's may not have.
        unsigned char* stage = q_sm + blk * (kBlockRows * kRowBytes);
        float* tail = reinterpret_cast<float*>(stage + row_local * kRowBytes + kD * 2);
        if constexpr (NB == 2) softmax_bar_sync();
        // (one row block: the halves' sums met with the pair's last barrier; the maxima are the same)
        const float l_all = NB == 1 ? tail[1] + tail[2] : l_run;
        const float inv = l_all > 0.f ? 1.f / l_all : 0.f;
        const float lse_val = l_all > 0.f ? (m_ref * c2 + log2f(l_all)) * 0.6931471805599453f : -INFINITY;
        if (ok) ok = mbar_wait_warp(B.o_done(blk, n_tiles - 1), ((n_tiles - 1) >> 2) & 1);    // the last product is in
        tc_fence_after();
        if (tid == 0) SPARROW_STAMP(6);                                // last product complete
        const int h_row = it.kvh * qg + g_row;
        const bool has_lse = row_ok && (wg == 0 || NB == 2);
        if (ok && has_lse && !direct) *tail = lse_val;
        if (ok) {
            #pragma unroll 1
            for (int col = dim0; col < dim0 + (NB == 1 ? 64 : 128); col += 32) {
                float o[32];
                tmem_ld32(lane_addr + kOCol + blk * 128 + col, o);
                tmem_wait_ld();
                uint4 pk[4];
                uint32_t* w = reinterpret_cast<uint32_t*>(pk);
                if (direct) {
                    #pragma unroll
                    for (int c = 0; c < 16; ++c) w[c] = pack_bf16x2(o[2 * c] * inv, o[2 * c + 1] * inv);
                } else {
                    #pragma unroll
                    for (int c = 0; c < 16; ++c) w[c] = pack_half2(o[2 * c] * inv, o[2 * c + 1] * inv);
                }
                if (row_ok) {
                    uint4* dst = reinterpret_cast<uint4*>(stage + row_local * kRowBytes + col * 2);
                    #pragma unroll
                    for (int c = 0; c < 4; ++c) dst[c] = pk[c];
                }
            }
        }
        if (!direct) fence_proxy_async();                              // the staged rows, ahead of the bulk copies
        softmax_bar_sync();                                            // every row is staged
        ok = ok && *write_ok == 1u;                                    // (thread 0 settled it ahead of the barrier)
        if (direct) {
            if (ok && has_lse) args.lse[((size_t)it.b * args.n_q_heads + h_row) * T + t_row] = lse_val;
            // final rows: 16 threads write a row's 256 bytes (a row per thread took 2 us longer)
            #pragma unroll
            for (int bk = 0; bk < NB; ++bk) {
                const int t0 = (block0 + bk) * tpb, rows_here = ok ? min(tpb, max(0, T - t0)) * qg : 0;
                #pragma unroll 4
                for (int r = tid >> 4; r < rows_here; r += 16) {
                    const int tok = (r * plan.inv_group) >> 16, h = it.kvh * qg + r - tok * qg;
                    *reinterpret_cast<uint4*>(args.out + (((size_t)it.b * T + t0 + tok) * args.n_q_heads + h) * kD + (tid & 15) * 8) =
                        *reinterpret_cast<const uint4*>(q_sm + bk * (kBlockRows * kRowBytes) + r * kRowBytes + (tid & 15) * 16);
                }
            }
            softmax_bar_sync();                                        // every row is written
        } else if (tid == 0 && ok && !clustered) {
            #pragma unroll
            for (int bk = 0; bk < NB; ++bk) {
                const int rows_here = min(tpb, max(0, T - (block0 + bk) * tpb)) * qg;
                if (rows_here > 0)
                    bulk_store(args.o_part + ((size_t)blockIdx.x * plan.part_rows + bk * kBlockRows) * kPartRowHalves,
                               smem_u32(q_sm + bk * (kBlockRows * kRowBytes)), (uint32_t)(rows_here * kRowBytes));
            }
        }

        // ---- publish this item; the call's finisher CTAs merge its partials ---------------------------
        // (overlapped mode: arrival words and finisher counters as described at SyncArgs; a
        // stream-ordered call only stores its partials, and a combine kernel follows)
        const int fin_idx = CL ? -1 : (int)blockIdx.x - (plan.n_items - sync.n_fin);     // >= 0: this CTA is a finisher
        const int rows_per_block = tpb * qg;                            // 126 for 7 heads x 18 tokens
        const int seq_rows = plan.n_kv_heads * qg * T;                  // query rows of a sequence
        // The call's row list: the query rows of every sequence with several pieces, (KV head, row group,
        // row) in order.  Finisher f takes rows [f chunk, (f + 1) chunk).
        int total = 0, chunk = 0;
        if (sync.enabled && fin_idx >= 0) {                             // (in a lone call every CTA is one)
            for (int b = 0; b < plan.batch; ++b)
                if (plan.seq[b].n_splits > 1) total += seq_rows;
            chunk = (total + sync.n_fin - 1) / sync.n_fin;
        }
        const int my_begin = fin_idx >= 0 ? min(total, fin_idx * chunk) : 0;
        int share_end = fin_idx >= 0 ? min(total, my_begin + chunk) : 0;       // end of the share being merged
        const bool merges = !CL && my_begin < share_end;
        MergeList* list = reinterpret_cast<MergeList*>(anc_s);          // (the tables are no longer needed)
        // Fills the list with what one pass merges, from row `row` on: runs of rows of one unit, as many as
        // fit the K/V ring with all their pieces.
        auto list_rows = [&](int row) {
            int n_seg = 0, bytes = 0;
            #pragma unroll 1
            while (row < share_end && n_seg < kMaxSegments) {
                MergeSegment sg;
                int rest = row;
                sg.b = 0;
                while (plan.seq[sg.b].n_splits == 1 || rest >= seq_rows) {
                    if (plan.seq[sg.b].n_splits > 1) rest -= seq_rows;
                    ++sg.b;
                }
                sg.ns = plan.seq[sg.b].n_splits;
                const int kvh = rest / (qg * T);
                rest -= kvh * qg * T;
                const int grp = rest / (NB * rows_per_block);
                sg.r0 = rest - grp * NB * rows_per_block;
                sg.tok0 = grp * NB * tpb;
                sg.head0 = kvh * qg;
                const int unit_left = qg * min(NB * tpb, T - sg.tok0) - sg.r0;
                sg.n = min(min(unit_left, share_end - row), (NS * kStageBytes - bytes) / (sg.ns * kRowBytes));
                if (sg.n == 0) break;
                // the run may straddle the unit's two blocks: `split` rows in the first of them
                const int bk0 = sg.r0 / rows_per_block;
                sg.split = (bk0 == 0 && sg.r0 + sg.n > rows_per_block) ? rows_per_block - sg.r0 : sg.n;
                const int part_row0 = (plan.seq[sg.b].item_begin + (kvh * plan.n_groups + grp) * sg.ns) * plan.part_rows;
                sg.src = part_row0 + bk0 * kBlockRows + sg.r0 - bk0 * rows_per_block;
                sg.src2 = part_row0 + kBlockRows;
                sg.offset = bytes;
                list->seg[n_seg++] = sg;
                bytes += sg.n * sg.ns * kRowBytes;
                row += sg.n;
            }
            list->n_seg = n_seg;
            list->bytes = bytes;
            list->next_row = row;
        };
        const MergeOut merge_out = {args.out, args.lse, T, args.n_q_heads, qg, plan.inv_group};
        if (clustered) {
            // Every CTA of the cluster merges a share of the unit's rows: it is sent its rows of every piece, one
            // bulk copy from each peer, into a stage of the K/V ring.
            const int cl = plan.cluster;
            const int unit_rows = qg * min(NB * tpb, T - block0 * tpb);
            auto recv_at = [&](int tiles) { return smem_u32(kv_sm) + (uint32_t)(recv_stage(NB, tiles) * kStageBytes + (NB == 1 ? kRecvSkip : 0)); };
            const uint32_t recv = recv_at(n_tiles);
            int r_begin;
            const int n = merge_share(unit_rows, it.split, plan.inv_cluster, &r_begin) - r_begin;
            const int peer = warp + 8 * lane;                          // (spread over the warps: a warp's lanes issue one after the other)
            const uint32_t peer_recv = recv_at(piece_tiles((n_keys_seq - plan.seq[it.b].key0 + kTile - 1) / kTile, cl, peer).count);
            cluster_wait();                                            // every peer runs, its barriers are initialised, the stage is free
            if (tid == 0) mbar_expect_tx(B.fin(), (uint32_t)(n * cl * kRowBytes));
            if (peer < cl) {
                int r0;
                const int r1 = merge_share(unit_rows, peer, plan.inv_cluster, &r0);      // the peer's share
                const uint32_t dst = map_to_rank(peer_recv + (uint32_t)(it.split * (r1 - r0) * kRowBytes), (uint32_t)peer);
                const uint32_t bar = map_to_rank(B.fin(), (uint32_t)peer);
                // (staged block by block: the share may straddle the two)
                const int mid = min(max(rows_per_block, r0), r1);
                if (mid > r0) bulk_push(dst, smem_u32(q_sm) + (uint32_t)(r0 * kRowBytes), (uint32_t)((mid - r0) * kRowBytes), bar);
                if (r1 > mid)
                    bulk_push(dst + (uint32_t)((mid - r0) * kRowBytes),
                              smem_u32(q_sm) + (uint32_t)((kBlockRows + mid - rows_per_block) * kRowBytes), (uint32_t)((r1 - mid) * kRowBytes), bar);
            }
            if (tid == 0) SPARROW_STAMP(12);                           // pushes issued
            const bool landed = mbar_wait_warp(B.fin(), 0);
            cluster_arrive_relaxed();                                  // (all pushes to this CTA are through: its peers may leave)
            if (!landed && lane == 0) atomicOr(args.status, timeout_bits(kSiteFinCopies));
            if (tid == 0) SPARROW_STAMP(15);                           // every piece is here
            merge_run(tid, recv, cl, n, r_begin, it.b, block0 * tpb, it.kvh * qg, landed && ok, merge_out);
            if (tid == 0) SPARROW_STAMP(10);                           // merged rows written
            softmax_bar_sync();
        }
        // (thread 0, while its bulk copies are on their way)
        if (tid == 0 && merges) list_rows(my_begin);
        if (tid == 0 && ok && !direct && !clustered) {
            bulk_store_wait();
            fence_proxy_async_global();
        }
        if (sync.enabled) {
            unsigned* arrive_word = sync.arrivals + sync.slot;
            if (tid == 0) SPARROW_STAMP(7);                            // partial rows stored
            const bool arrives = !direct && !clustered;
            if (tid == 0 && arrives) publish_counter(arrive_word);
            if (!CL && (merges || (sync.lone && arrives))) {
                if (tid == 0) {
                    // every partial of the call in place, and the previous call's final results written
                    // (both words are polled in one loop: the second is usually there already, and a lone
                    // call's predecessors have ended as grids)
                    bool have_all = false, prev_done = sync.lone != 0;
                    uint32_t word = 0;
                    const uint32_t polls = !merges ? 1u : sync.lone ? kPatiencePolls : kCounterPolls;
                    #pragma unroll 1
                    for (uint32_t i = 0; i < polls && !(have_all && prev_done); ++i) {
                        if (!have_all) {
                            word = ld_acquire(arrive_word);
                            have_all = (word & kArrivedMask) == (unsigned)sync.n_arrive;
                        }
                        if (!prev_done) prev_done = (int32_t)(ld_acquire(sync.fin_done + (sync.parity ^ 1)) - sync.fin_wait_other) >= 0;
                        if (!(have_all && prev_done)) __nanosleep(i < 256 ? 20 : 200);
                    }
                    SPARROW_STAMP(8);                                   // all arrivals seen
                    bool adopts = false;
                    if (sync.lone) {
                        // (one that would leave but finds all arrivals counted stays: nobody needs to have noticed it)
                        if (merges && !have_all) have_all = (add_acquire_release(arrive_word, kOneLeft) & kArrivedMask) == (unsigned)sync.n_arrive;
                        else if (have_all && word >= kOneLeft) adopts = (atomicOr(arrive_word, kAdopted) & kAdopted) == 0u;
                    } else if (!have_all) {
                        atomicOr(args.status, timeout_bits(kSiteArrivals));
                    } else if (!prev_done) {
                        atomicOr(args.status, timeout_bits(kSiteFinOther));
                    }
                    SPARROW_STAMP(9);                                   // previous call's finishers seen
                    *fin_go = !(have_all && prev_done) ? 0 : adopts ? 2 : merges ? 1 : 0;
                }
                // The rows' pieces are first brought into the (idle) K/V ring by bulk copies, [piece][row]
                // [272 bytes], one copy per piece and block touched -- far fewer and larger requests than
                // per-thread loads (16-byte words that carry a tag, read by the threads as they arrive and without
                // any counter, were there 1.6 us earlier but took 2 us longer to collect).
                int adopted = 0;                                           // (thread 0) next finisher whose share is taken over
                if (tid == 0 && !merges) list->n_seg = list->bytes = list->next_row = 0;
                #pragma unroll 1
                for (int phase = 0;; phase ^= 1) {
                    if (tid == 0 && *fin_go) mbar_expect_tx(B.fin(), (uint32_t)list->bytes);
                    softmax_bar_sync();                                    // the list and the byte count are posted
                    const int go = *fin_go;
                    if (!go) break;
                    const int n_seg = list->n_seg;
                    #pragma unroll 1
                    for (int k = 0; k < n_seg; ++k) {
                        const MergeSegment& sg = list->seg[k];
                        const int ns = sg.ns, n = sg.n, split = sg.split;
                        const __half* src = args.o_part + (size_t)sg.src * kPartRowHalves;
                        const uint32_t dst = smem_u32(kv_sm) + (uint32_t)sg.offset;
                        const size_t pitch = (size_t)plan.part_rows * kPartRowHalves;      // halves between pieces
                        // one copy per thread, spread over the warps (a warp's lanes issue theirs one after the other)
                        for (int sp = warp + 8 * lane; sp < ns; sp += 256) {
                            bulk_load(dst + (uint32_t)(sp * n * kRowBytes), src + sp * pitch, (uint32_t)split * kRowBytes, B.fin());
                            if (split < n)
                                bulk_load(dst + (uint32_t)((sp * n + split) * kRowBytes),
                                          args.o_part + (size_t)sg.src2 * kPartRowHalves + sp * pitch, (uint32_t)(n - split) * kRowBytes, B.fin());
                        }
                    }
                    if (tid == 0) SPARROW_STAMP(12);                       // bulk copies issued
                    const bool landed = mbar_wait_warp(B.fin(), phase);
                    if (tid == 0) SPARROW_STAMP(15);                       // bulk copies landed
                    if (!landed && lane == 0) atomicOr(args.status, timeout_bits(kSiteFinCopies));
                    #pragma unroll 1
                    for (int k = 0; k < n_seg; ++k) {
                        const MergeSegment& sg = list->seg[k];
                        merge_run(tid, smem_u32(kv_sm) + (uint32_t)sg.offset, sg.ns, sg.n, sg.r0, sg.b, sg.tok0, sg.head0, landed, merge_out);
                    }
                    const int next = list->next_row;
                    if (!landed || (next >= share_end && go == 1)) break;
                    softmax_bar_sync();                                    // everybody is through with the ring and the list
                    if (tid == 0) {
                        int row = next;
                        while (row >= share_end && adopted < sync.n_fin) { // (only where go is 2)
                            row = adopted == fin_idx ? total : min(total, adopted * chunk);
                            share_end = min(total, row + chunk);
                            ++adopted;
                        }
                        if (row < share_end) list_rows(row);
                        else *fin_go = 0;
                    }
                }
                if (tid == 0) SPARROW_STAMP(10);                        // merged rows written
                softmax_bar_sync();
            }
            if (tid == 0) {
                const unsigned done = (direct || clustered ? 1u : 0u) + (fin_idx >= 0 ? 1u : 0u);
                if (done) {
                    if (sync.lone) atomicAdd(sync.fin_done + sync.parity, done);       // (relaxed: nobody reads this call's results before the grid has ended)
                    else publish_counter(sync.fin_done + sync.parity, done);
                }
            }
        }
        if (!ok) { atomicOr(args.status, timeout_bits(kSiteSoftmax)); *abort_flag = 1; }
    }

    // ---- teardown -------------------------------------------------------------------------------
    if (CL) {
        // Nobody leaves before its peers have received what it sends them.
        if (warp >= 8) { cluster_wait(); cluster_arrive_relaxed(); }    // (the softmax warps have done both)
        cluster_wait();
    }
    tc_fence_before();
    __syncthreads();
    if (*abort_flag) {
        // give copies that are still in flight time to land before the CTA's memory is released
        #pragma unroll 1
        for (int i = 0; i < 2000; ++i) __nanosleep(1000);
        __syncthreads();
    }
    // an early-started call must not complete before its predecessors (see wait_for_predecessors)
    if (sync.enabled && !sync.wait_first && blockIdx.x == 0 && threadIdx.x == 0) wait_for_predecessors();
    if (threadIdx.x == 0) SPARROW_STAMP(11);                            // leaving
    if (warp == kMmaWarp) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
    }
}

}  // namespace tc
}  // namespace sparrow
