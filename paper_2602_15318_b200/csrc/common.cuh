// Shared declarations of the CUDA path: the work decomposition handed to the kernels, the sticky
// device status bits, and the device-side ancestor-mask construction.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

// Timeline build (-DSPARROW_TIMELINE, made by `python -m paper_2602_15318_b200.timeline`; never
// the shipped library): SPARROW_STAMP(slot) records %globaltimer for (call, CTA, slot), and three
// extra exported calls read the table back.  A kernel names the call it belongs to once with
// SPARROW_TIMELINE_CALL(index) (kept modulo 32).  In the ordinary build both macros expand to nothing.
#ifdef SPARROW_TIMELINE
namespace sparrow {
constexpr int kTimelineCalls = 32, kTimelineCtas = 256, kTimelineSlots = 16;
__device__ unsigned long long g_timeline[kTimelineCalls * kTimelineCtas * kTimelineSlots];
__device__ __forceinline__ unsigned long long global_timer_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
}  // namespace sparrow
#define SPARROW_TIMELINE_CALL(index) const unsigned sparrow_tl_call = (unsigned)(index) % ::sparrow::kTimelineCalls
#define SPARROW_STAMP(slot)                                                                        \
    do {                                                                                           \
        if (blockIdx.x < ::sparrow::kTimelineCtas)                                                 \
            ::sparrow::g_timeline[((size_t)sparrow_tl_call * ::sparrow::kTimelineCtas + blockIdx.x) * ::sparrow::kTimelineSlots + (slot)] = \
                ::sparrow::global_timer_ns();                                                      \
    } while (0)
#else
#define SPARROW_TIMELINE_CALL(index) ((void)0)
#define SPARROW_STAMP(slot) ((void)0)
#endif

namespace sparrow {

constexpr int kD = 128;           // head_dim
constexpr int kMaxGroup = 16;      // query heads per KV head: 1 .. 16 (7 for the Qwen2-7B-shaped models of the paper)
constexpr int kMaxT = 64;
constexpr int kMaxBatch = 64;
// draft tokens per 128-row block for a group of g query heads: 18 for g = 7 (126 rows, 2 rows of padding)
__host__ __device__ constexpr int tokens_per_block(int g) { return 128 / g < 64 ? 128 / g : 64; }
constexpr int kBlockRows = 128;
constexpr int kKeyTile = 128;      // keys per tile of the tensor-core kernel; pieces of the key range are whole tiles

// device status bits (sticky, OR-ed into the first word of the workspace)
constexpr unsigned kStatTree = 1u;
constexpr unsigned kStatAnchor = 2u;
constexpr unsigned kStatTimeout = 4u;
// A wait that gives up also sets bit (8 + site) of the status word, so that the raw word tells which wait it was.
__host__ __device__ constexpr unsigned timeout_bits(int site) { return kStatTimeout | (1u << (8 + site)); }
enum WaitSite { kSiteProducer = 0, kSiteMma = 1, kSiteSoftmax = 2, kSiteWriteSame = 3, kSiteWriteOther = 4,
                kSiteArrivals = 5, kSiteFinOther = 6, kSiteFinCopies = 7, kSiteDebug = 8, kSiteSample = 9 };

// The GQA group's g query heads x T draft tokens are packed into 128-row blocks of p = 128 / g
// tokens: block i holds tokens [p i, p i + p), row r of a block is (token p i + r / g, head r % g),
// rows from g p on are padding (g = 7: 18 tokens, rows 126 and 127).  A row group is 1 or 2
// consecutive blocks, handled by one work item.
//
// One work item = (sequence b, KV head, row group, key-range piece).  Items of sequence b occupy
// [seq[b].item_begin, seq[b+1].item_begin); inside, the index runs (kv head, row group, piece) with the
// piece fastest.  Pieces are whole tiles, the longer ones first (decode_item).
struct SeqPlan {                  // per sequence
    int32_t item_begin;           // first work item of the sequence
    int32_t n_splits;             // key-range pieces per unit
    int32_t n_keys;               // kv_len + draft-tree nodes (verify) or n_anchor (anchored)
    int32_t kv_len;               // verify mode only
    int32_t key0;                 // first key that is streamed at all (a multiple of the tile; 0 unless a window cuts the prefix)
};
// Scalars first and the per-sequence entries as an array of structs: what a CTA reads of the plan
// then sits in one or two lines of the constant bank the kernel parameters live in.
struct SplitPlan {
    int32_t n_items;
    int32_t batch;
    int32_t T;                    // query tokens
    int32_t T_tree;               // nodes of the draft tree = rows of the draft block; the queries are its last T nodes
    int32_t group;                // g: query heads per KV head
    int32_t tok_per_block;        // p = tokens_per_block(g)
    int32_t M;                    // query rows per KV head = g*T
    int32_t blocks_per_group;     // 128-row blocks one work item handles (1 or 2)
    int32_t n_groups;             // ceil(T / (18 * blocks_per_group))
    int32_t n_kv_heads;
    int32_t part_rows;            // row pitch of one item's partial block in the workspace
    int32_t inv_group;            // 2^16 / group rounded up: x / group = x * inv_group >> 16 for x <= 512
    int32_t inv_cluster;          // the same of cluster
    int32_t cluster;              // > 1: every unit has this many pieces, in CTAs of one thread-block cluster that merge among themselves
    int32_t piece_tile;           // pieces of the key range are whole tiles of this many keys (128 or 64)
    SeqPlan seq[kMaxBatch];
};

constexpr int kFinisherCtas = 32;  // CTAs of a call that share its combine step
// An arrival word counts arrivals in its lower half and, in a lone call, finishers that have left above; the top bit is
// taken by the CTA that merges for them.
constexpr uint32_t kArrivedMask = 0xFFFFu, kOneLeft = 0x10000u, kAdopted = 0x80000000u;
// Polls after which a finisher of a lone call leaves its rows to the last CTA to arrive, some 200 us: the CTAs of one
// wave end within a few microseconds of one another, unless kernels of other streams hold SMs that some have yet to start on.
constexpr uint32_t kPatiencePolls = 256;
// A partial row in the workspace: 128 fp16 outputs, then the row's fp32 LSE, padded to 16 bytes,
// so that one bulk copy brings a run of rows with everything needed to merge them.
constexpr int kPartRowHalves = 136;

// Overlapped mode: ordering between the CTAs of one call and between consecutive calls.
//
// A call that starts early is launched with programmatic stream serialisation and does not wait for the
// previous grid as a whole (but for CTA 0, which does before it leaves), so the next call's CTAs start (and read their inputs) while the
// previous call is still finishing.  What must be ordered goes through counters in the workspace,
// released / acquired at GPU scope.  Partial buffers are double-buffered by the parity of the call
// number n, arrival words rotate over n modulo 4.
//   arrivals[n % 4]   items of call n that have published their partials
//   fin_done[n % 2]   final-result writers of calls with this parity that are done, cumulative
// An item whose unit (sequence, KV head, row group) has several key-range pieces stores a partial
// and arrives; an item that is its unit's only piece writes final results itself.  The last
// n_fin CTAs of the grid are the call's finishers (all of them where the call has the GPU to
// itself anyway) -- they are the last to start, so by the time
// they are through with their own items little is left to wait for: they wait until every
// partial of the call has arrived, then each merges a contiguous share of the call's rows by
// log-sum-exp and writes the final out / lse.  Every final-result writer (finisher or single
// piece) bumps fin_done once.
// Before its first global write an item of call n waits until the writers of call n-2 are done
// (fin_wait_same: the finishers among them read the partial buffer it is about to overwrite);
// whoever writes final results also waits for the writers of call n-1 (fin_wait_other), so
// results land in call order.  CTA 0 then clears the arrival word of slot (n + 2) % 4: its last
// user was call n-2, and the items of call n+2 cannot arrive before the finishers of call n are
// done, which in turn have seen CTA 0's arrival (or, if it had none, follow it in the stream).
// In a lone call every CTA is a finisher, and the grid may fill the GPU: waiting for all of it would need all of
// it resident at once, and two such calls of different contexts, each holding the SMs that the other's last CTAs
// need, would wait for each other.  There nobody waits without end: a finisher that has polled kPatiencePolls
// times adds kOneLeft to the arrival word and leaves.  The first CTA that finds all arrivals counted and somebody gone
// merges the rows of every finisher; there always is one, the last CTA to arrive, if no other.  It goes share by share, so
// that the results are the same bits (a finisher that has not left writes the same values into its own share).
// With enabled == 0 the kernels are ordered by the stream alone: they touch no counter, and a
// separate combine kernel follows the split-KV kernel.
struct SyncArgs {
    unsigned* arrivals;      // [4]
    unsigned* fin_done;      // [2]
    int32_t enabled;         // overlapped mode
    int32_t parity;          // n % 2
    int32_t slot;            // n % 4
    int32_t n_arrive;        // items of this call that store partials
    int32_t n_fin;           // finisher CTAs of this call (0 when no unit has several pieces)
    uint32_t fin_wait_same;
    uint32_t fin_wait_other;
    int32_t wait_first;      // launched with programmatic stream serialisation but ordered behind its predecessor: wait before the first global access (2: but for key tiles that lie in the prefix)
    int32_t lone;            // no later call can start before this grid has ended
    uint32_t call;           // running number of the context's fused calls (the timeline build files its stamps under it)
};

__device__ __forceinline__ unsigned ld_acquire(const unsigned* addr)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(addr) : "memory");
    return v;
}
// Polls of a counter wait before it gives up: with the pause between polls this is of the order of
// a second.  The bound counts polls rather than reading a timer, so it cannot misfire on a timer
// glitch and does not depend on the timer's resolution.
constexpr uint32_t kCounterPolls = 1u << 22;
// Bounded acquire-wait until a cumulative counter has reached `target` (wrap-safe compare).
__device__ __forceinline__ bool wait_counter(const unsigned* addr, uint32_t target)
{
    #pragma unroll 1
    for (uint32_t i = 0; i < kCounterPolls; ++i) {
        if ((int32_t)(ld_acquire(addr) - target) >= 0) return true;
        __nanosleep(i < 64 ? 40 : 200);
    }
    return false;
}
// Increment of a counter that also returns what it was; orders as publish_counter() and ld_acquire() do.
__device__ __forceinline__ unsigned add_acquire_release(unsigned* addr, unsigned n)
{
    unsigned v;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], %2;" : "=r"(v) : "l"(addr), "r"(n) : "memory");
    return v;
}
// Release-increment of a counter: orders every write this thread has observed (its own and, after
// a CTA barrier, its CTA's) before the increment.
__device__ __forceinline__ void publish_counter(unsigned* addr, unsigned n = 1u)
{
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(addr), "r"(n) : "memory");
}

// Launch overlap between kernels in stream order.  A kernel launched with programmatic stream
// serialisation starts while its predecessor is finishing, and wait_for_predecessors() holds it, in front
// of its first access to global memory, until the predecessor has completed with its writes visible.
// Every kernel of this library either waits like that or (early-started verification calls) does so
// before its grid ends, so completion of the predecessor implies completion of everything before it.
__device__ __forceinline__ void wait_for_predecessors() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void let_dependents_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Loads that stay behind that wait and see what the predecessor wrote: ordinary loads, neither through the
// non-coherent path nor open to reordering (which const __restrict__ parameters and __ldg would be).
__device__ __forceinline__ int32_t ld_behind(const int32_t* p)
{
    int32_t v;
    asm volatile("ld.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ uint4 ld_behind(const uint4* p)
{
    uint4 v;
    asm volatile("ld.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ float ld_behind(const float* p)
{
    float v;
    asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ __nv_bfloat16 ld_behind(const __nv_bfloat16* p)
{
    unsigned short v;
    asm volatile("ld.global.u16 %0, [%1];" : "=h"(v) : "l"(p) : "memory");
    return __ushort_as_bfloat16(v);
}

struct Item {
    int b, kvh, group, split, key_begin, key_end;
};

// Key range of piece `split` of `ns` over `n_keys` keys in whole tiles of `tile` keys, as even as whole tiles
// allow; the last piece takes the ragged end.  Needs ns <= number of tiles.  (What sparrow_plan_piece_range() reports: the
// sizes are the kernels', which take the longer pieces first, see piece_tiles.)
inline void piece_range(int n_keys, int ns, int split, int tile, int* begin, int* end)
{
    const long long n_tiles = (n_keys + tile - 1) / tile;
    const long long b = n_tiles * split / ns * tile, e = n_tiles * (split + 1) / ns * tile;
    *begin = (int)b;
    *end = (int)(e < n_keys ? e : n_keys);
}

// Tiles of piece `split` of `ns` over `tiles` tiles as the kernels take them: as even as whole tiles allow, the longer
// pieces first.  The last one holds the draft block, whose masks and tables already make it the latest (26,112 keys,
// T = 16: 0.7 us behind pieces of the same six tiles, about what one tile takes).
struct TileRun {
    int first, count;
};
__host__ __device__ __forceinline__ TileRun piece_tiles(int tiles, int ns, int split)
{
    const int least = tiles / ns, longer = tiles - least * ns;
    TileRun r;
    r.first = split * least + (split < longer ? split : longer);
    r.count = least + (split < longer ? 1 : 0);
    return r;
}

__device__ __forceinline__ Item decode_item(const SplitPlan& p, int item)
{
    int b = 0;
    while (b + 1 < p.batch && item >= p.seq[b + 1].item_begin) ++b;
    const int local = item - p.seq[b].item_begin;
    const int ns = p.seq[b].n_splits;
    Item it;
    it.b = b;
    it.split = local % ns;
    const int unit = local / ns;
    it.group = unit % p.n_groups;
    it.kvh = unit / p.n_groups;
    const int key0 = p.seq[b].key0, n_keys = p.seq[b].n_keys - key0;
    const TileRun run = piece_tiles((n_keys + p.piece_tile - 1) / p.piece_tile, ns, it.split);
    it.key_begin = key0 + run.first * p.piece_tile;
    it.key_end = key0 + min(n_keys, (run.first + run.count) * p.piece_tile);
    return it;
}

// Ancestor words of a draft tree of T <= 64 nodes, built by one warp: anc[i] (shared memory) gets bit a set iff
// a == i or a is an ancestor of i.  Lane l brings the parents of nodes l and l + 32.  A parent outside
// [-1, node) is treated as "root" and reported.  Pointer doubling in registers: after round r a word covers
// 2^r generations, so six rounds do for any tree.  The CTA that holds the draft block is the one a short
// call waits for: a walk from every node to its root, a chain of up to 64 dependent reads, made a 40-node
// chain 4.5 us late; doubling in shared memory took 0.13 us a round, shuffles take 0.03.
__device__ __forceinline__ void build_ancestor_words(int p0, int p1, unsigned long long* anc, int T, unsigned* status)
{
    const int lane = threadIdx.x & 31;
    int j0 = lane < T ? p0 : -1, j1 = lane + 32 < T ? p1 : -1;
    if (j0 < -1 || j0 >= lane || j1 < -1 || j1 >= lane + 32) {
        if (status) atomicOr(status, kStatTree);
        if (j0 < -1 || j0 >= lane) j0 = -1;
        if (j1 < -1 || j1 >= lane + 32) j1 = -1;
    }
    uint32_t lo0 = 1u << lane, lo1 = 0u, hi1 = 1u << lane;       // (a node below 32 has no ancestor above)
    while (__any_sync(0xffffffffu, j0 >= 0 || j1 >= 0)) {
        const uint32_t a0 = __shfl_sync(0xffffffffu, lo0, j0 & 31);
        const int n0 = __shfl_sync(0xffffffffu, j0, j0 & 31);
        if (T > 32) {
            const uint32_t l0 = __shfl_sync(0xffffffffu, lo0, j1 & 31), l1 = __shfl_sync(0xffffffffu, lo1, j1 & 31);
            const uint32_t h1 = __shfl_sync(0xffffffffu, hi1, j1 & 31);
            const int m0 = __shfl_sync(0xffffffffu, j0, j1 & 31), m1 = __shfl_sync(0xffffffffu, j1, j1 & 31);
            if (j1 >= 32) { lo1 |= l1; hi1 |= h1; j1 = m1; }
            else if (j1 >= 0) { lo1 |= l0; j1 = m0; }
        }
        if (j0 >= 0) { lo0 |= a0; j0 = n0; }
    }
    if (lane < T) anc[lane] = lo0;
    if (lane + 32 < T) anc[lane + 32] = (unsigned long long)hi1 << 32 | lo1;
    __syncwarp();
}

}  // namespace sparrow
