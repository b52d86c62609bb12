// Acceptance at temperature 1: multi-round rejection sampling over the draft tree (Appendix A: the
// verification keeps the target's output distribution exactly; the paper relies on the standard
// procedure).  At the current node, with target distribution p and draft distribution q, the
// children are tried in index order; a child with token x is accepted with probability
// min(1, p(x) / q(x)); after a rejection p becomes the normalised positive part of (p - q), and q
// loses x (the siblings were drawn without replacement); when no child is accepted the next token
// is drawn from what p has become.
//
// The results are integers (accepted path, bonus token), so the arithmetic is integer too:
// probabilities are rounded once to 30-bit fixed point, P = floor(p 2^30 + 1/2), and with A = sum P,
// B = sum Q and a 32-bit uniform r
//     accept x          iff  Q[x] > 0 and r Q[x] A < P[x] B 2^32               (128-bit products)
//     after a rejection      P <- max(B P - A Q, 0) >> 30 (unless B == 0), A <- sum P, B <- B - Q[x], Q[x] <- 0
//     bonus                  the smallest v with P[0] + ... + P[v] > (r A) >> 32, P being the row's
//                            original target row again if A == 0.
// Integer sums do not depend on the order of summation, so any parallel reduction gives the same
// bits.  Where a level's rows sum to about one and fit shared memory, the residual replaces the row
// there, one update per rejection; in every other case element v of the current P is recomputed from the
// two input rows and the level's short history of (A, B, x) triples.
//
// What bounds it: a chain of steps, each a sum over two vocabulary rows that the next decision
// waits for.  One thread-block cluster per sequence (up to 16 CTAs, each owning a contiguous slice
// of the vocabulary) walks the tree: a level's two rows are read from global memory once and kept in
// shared memory as fixed-point words for the passes after rejections and for the draw.  A step ends
// with every CTA pushing its partial sums into the other CTAs' shared memory (st.async on an mbarrier
// of the receiver: 0.9 us less per step than a cluster barrier), after which all CTAs take the same
// decision; while the sums travel, the rows of the child that is tested next are already on their way
// into registers.  The partial sums also tell which CTA holds the bonus token.
// Measured on a 32-node tree over 151,936 entries (back to back; the walk's length depends on the
// uniforms): 14 to 22 us with clusters of 16; one CTA per sequence, with the rows read again from L2 in
// every pass and the serial scan of the draw, took 145 to 420 us.  Stamps: a level 0.8 us to turn two rows into fixed point
// (1.0 a value at a time), 0.3 us to request the next (0.4 with 4-byte loads), 0.95 us for the cluster's sum and 0.4 for the
// decision; a rejection 0.15 to 0.5 us in front of the pass, 1.0 for it (1.25 with single entries), the sum, the decision; the draw 1.4.
#pragma once
#include "verify_tc.cuh"

namespace sparrow {
namespace sample {

constexpr int kThreads = 512;
constexpr int kWarps = kThreads / 32;
constexpr int kProbBits = 30;
constexpr int kMaxCluster = 16;
constexpr int kMinSlice = 4096;           // vocabulary entries per CTA below which sharing them out costs more than it saves
constexpr int kAhead = 20;                // row entries per thread fetched ahead (10,240 per CTA: vocabularies up to 163,840)
constexpr int kMaxResident = 25600;       // entries per CTA kept in shared memory (8 bytes each: 200 KB)

// floor(p 2^30 + 1/2) for p in [0, 1]; anything else (NaN, negative, > 1) is clamped into the range.
// Rounding p 2^30 + 1/2 down never crosses an integer, so the floor of the rounded value is the floor of
// the exact one (and from 2^23 on p 2^30 is an integer, to which the value rounds back).  Conversion
// instructions run at a quarter of the rate of an addition: below 2^23 the floor is read from the
// mantissa of a second addition instead.
__device__ __forceinline__ uint32_t fixed_prob(float p)
{
    const float y = __fmaf_rd(__saturatef(p), 1073741824.0f, 0.5f);      // (saturation maps NaN to 0)
    uint32_t r = __float_as_uint(__fadd_rd(y, 8388608.0f)) - 0x4B000000u;
    asm("{\n\t.reg .pred big;\n\tsetp.ge.f32 big, %1, 0f4B000000;\n\t@big cvt.rzi.u32.f32 %0, %1;\n\t}" : "+r"(r) : "f"(y));
    return r;
}

// The same for N values at once, in place (the bits of f become the weights); returns their sum.  y = p 2^30 + 1/2 keeps everything
// that matters of p: as unsigned words the y of ordinary small weights lie below 2^23's, and a negative p, a NaN or a
// weight of 2^-7 or more anywhere among them shows as a larger one; only then is each of them looked at.  Half the instructions
// a value of the function above.
template <int N>
__device__ __forceinline__ long long fixed_probs(float (&f)[N])
{
    static_assert(N <= 256, "N small weights fit 32 bits");
    uint32_t most = 0;
    #pragma unroll
    for (int k = 0; k < N; ++k) {
        f[k] = __fmaf_rd(f[k], 1073741824.0f, 0.5f);
        most = max(most, __float_as_uint(f[k]));
    }
    if (most < 0x4B000000u) {
        uint32_t sum = 0;
        #pragma unroll
        for (int k = 0; k < N; ++k) {
            const uint32_t r = __float_as_uint(__fadd_rd(f[k], 8388608.0f)) - 0x4B000000u;
            f[k] = __uint_as_float(r);
            sum += r;
        }
        return sum;
    }
    long long sum = 0;
    #pragma unroll
    for (int k = 0; k < N; ++k) {
        const float y = fminf(fmaxf(f[k], 0.f), 1073741824.0f);              // (NaN: 0)
        const uint32_t r = y < 8388608.0f ? __float_as_uint(__fadd_rd(y, 8388608.0f)) - 0x4B000000u : (uint32_t)y;
        f[k] = __uint_as_float(r);
        sum += r;
    }
    return sum;
}

// Rows whose sums stay below this (1 + 2^-7 in fixed point) keep every residual weight below 2^31, through
// up to 64 rejections: P' <= (B P) / 2^30 and A' <= (B A) / 2^30, and (1 + 2^-7)^64 < 1.7.
constexpr long long kPlainSum = (1ll << kProbBits) + (1ll << (kProbBits - 7));

struct Level {                      // history of the rejections at the current node
    long long A[kMaxT], B[kMaxT];
    int x[kMaxT];
};

// Current residual target weight and current draft weight of an entry with original weights P0, Q0
// at vocabulary index v, after the level's first n rejections.
__device__ __forceinline__ void weights_at(uint32_t P0, uint32_t Q0, int v, const Level& lv, int n, long long* P_out, long long* Q_out)
{
    long long P = P0;
    const long long q0 = Q0;
    bool gone = false;               // v was a rejected candidate: the draft distribution has lost it
    for (int s = 0; s < n; ++s) {
        const long long Q = gone ? 0ll : q0;
        if (lv.B[s] > 0) {
            const long long d = lv.B[s] * P - lv.A[s] * Q;
            P = d > 0 ? d >> kProbBits : 0ll;
        }
        if (v == lv.x[s]) gone = true;
    }
    *P_out = P;
    *Q_out = gone ? 0ll : q0;
}

// Entries of the vocabulary that a CTA of the cluster owns (the last ones fewer, or none): whole quads.
__host__ __device__ __forceinline__ int entries_per_cta(int V, int n_cta) { return ((V + n_cta - 1) / n_cta + 3) & ~3; }

__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
using tc::cluster_arrive;
using tc::cluster_wait;
// 16 bytes into the same place of CTA `rank`'s shared memory, counted on its mbarrier.
__device__ __forceinline__ void push_2x64(const void* local, const uint64_t* local_bar, uint32_t rank, long long a, long long b)
{
    uint32_t addr = tc::smem_u32(local), bar = tc::smem_u32(local_bar);
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(addr) : "r"(addr), "r"(rank));
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(bar) : "r"(bar), "r"(rank));
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.b64 [%0], {%1, %2}, [%3];"
                 ::"r"(addr), "l"(a), "l"(b), "r"(bar) : "memory");
}
struct Shared {
    Level lv;
    uint64_t bar[2];                                    // the cluster's pushes of even / odd steps have landed
    long long red[2][kWarps];
    alignas(16) long long part[2][kMaxCluster][2];      // per CTA of the cluster: its share of (A, B); two steps alternate
    long long row_part[kMaxCluster];                    // the CTAs' shares of the level's original A
    int32_t tok[kMaxT];
    uint32_t u_node[kMaxT], u_bonus[kMaxT + 1];
    unsigned long long kids[kMaxT + 1];                 // children of the committed prefix, then of the nodes
    uint32_t node_P[kMaxT], node_Q[kMaxT];              // original weights of the nodes' tokens in their parents' rows
};

// 64-bit sum (modulo 2^64) over a warp: three warp reductions of parts that cannot overflow 32 bits,
// a third of the instructions of a shuffle tree.
__device__ __forceinline__ long long warp_sum(long long v)
{
    const unsigned long long u = (unsigned long long)v;
    const unsigned long long lo = __reduce_add_sync(0xffffffffu, (uint32_t)u & 0x7FFFFFFu);
    const unsigned long long mid = __reduce_add_sync(0xffffffffu, (uint32_t)(u >> 27) & 0x7FFFFFFu);
    const unsigned long long hi = __reduce_add_sync(0xffffffffu, (uint32_t)(u >> 54));
    return (long long)(lo + (mid << 27) + (hi << 54));
}

// Sums (a, b), or a alone (b is 0), over the cluster; every thread gets the totals, sh.part[step & 1] the CTAs' shares.
// False when the peers' pushes did not arrive within the poll limit.
template <bool BOTH>
__device__ __forceinline__ bool sum_over_cluster(Shared& sh, long long& a, long long& b, int n_cta, uint32_t rank, uint32_t step)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    a = warp_sum(a);
    if (BOTH) b = warp_sum(b);
    if (lane == 0) { sh.red[0][warp] = a; if (BOTH) sh.red[1][warp] = b; }
    __syncthreads();
    if (warp == 0) {
        if (lane == 0) tc::mbar_expect_tx(tc::smem_u32(&sh.bar[step & 1]), 16u * (uint32_t)n_cta);
        a = warp_sum(lane < kWarps ? sh.red[0][lane] : 0ll);
        if (BOTH) b = warp_sum(lane < kWarps ? sh.red[1][lane] : 0ll);
        if (lane < n_cta) push_2x64(&sh.part[step & 1][rank][0], &sh.bar[step & 1], (uint32_t)lane, a, b);
    }
    // A slot is written again two steps later, by a CTA that has by then received this CTA's push of the
    // step in between, which this CTA sends after all its threads have read the slot.
    // (All threads of the CTA go on or give up together.)
    const bool ok = __syncthreads_and(tc::mbar_wait(tc::smem_u32(&sh.bar[step & 1]), (step >> 1) & 1u) ? 1 : 0) != 0;
    a = b = 0;
    #pragma unroll
    for (int r = 0; r < kMaxCluster; ++r) {                         // (slots past the cluster hold zeros)
        const longlong2 s = *reinterpret_cast<const longlong2*>(&sh.part[step & 1][r][0]);
        a += s.x;
        b += s.y;
    }
    return ok;
}

__device__ __forceinline__ bool cluster_sum(Shared& sh, long long& a, long long& b, int n_cta, uint32_t rank, uint32_t step)
{
    return sum_over_cluster<true>(sh, a, b, n_cta, rank, step);
}
__device__ __forceinline__ bool cluster_sum(Shared& sh, long long& a, int n_cta, uint32_t rank, uint32_t step)
{
    long long none = 0;
    return sum_over_cluster<false>(sh, a, none, n_cta, rank, step);
}

// VEC: a thread takes four neighbouring entries at a time, with 16-byte loads (rows that start on 16-byte boundaries: the vocabulary is
// a multiple of four); otherwise single ones, 512 apart.
template <bool VEC>
__global__ void __launch_bounds__(kThreads)
accept_sample_kernel(const int32_t* draft_tokens, const int32_t* parents,
                     const float* p_target, const float* p_draft,
                     const uint32_t* u_node, const uint32_t* u_bonus, int T, int V, int n_cta, int resident,
                     int32_t* path, int32_t* n_accept, int32_t* bonus, unsigned* status)
{
    let_dependents_launch();
    // the first `resident` entries of this CTA's slice, fixed point: all P, then all Q (VEC), or pairs
    extern __shared__ uint4 row_mem[];
    uint32_t* const P_s = reinterpret_cast<uint32_t*>(row_mem);
    uint32_t* const Q_s = P_s + resident;
    uint2* const PQ_s = reinterpret_cast<uint2*>(row_mem);
    auto put = [&](int i, uint32_t P, uint32_t Q) {
        if (VEC) { P_s[i] = P; Q_s[i] = Q; } else PQ_s[i] = make_uint2(P, Q);
    };
    auto held = [&](int i) -> uint2 { return VEC ? make_uint2(P_s[i], Q_s[i]) : PQ_s[i]; };
    __shared__ Shared sh;
    const int b = blockIdx.x / n_cta, tid = threadIdx.x;
    const uint32_t rank = n_cta > 1 ? cluster_rank() : 0u;
    const int per_cta = entries_per_cta(V, n_cta);
    const int v_begin = min(V, (int)rank * per_cta), n_mine = min(V, v_begin + per_cta) - v_begin;
    const int n_res = min(n_mine, resident);
    const float* p_seq = p_target + (size_t)b * (T + 1) * V;       // row r of this sequence: p_seq + r V
    const float* q_seq = p_draft + (size_t)b * (T + 1) * V;

    // the first kAhead entries per thread of a row pair, on their way
    float fp[kAhead], fq[kAhead];
    // entry of register k of those
    auto entry_of = [&](int k) -> int { return VEC ? ((k >> 2) * kThreads + tid) * 4 + (k & 3) : k * kThreads + tid; };
    auto fetch_row = [&](int r) {
        const float* pt = p_seq + (size_t)r * V + v_begin;
        const float* pq = q_seq + (size_t)r * V + v_begin;
        if (VEC) {
            #pragma unroll
            for (int k = 0; k < kAhead; k += 4) {
                const int i = entry_of(k);                          // (n_mine is a multiple of four)
                uint4 p4 = make_uint4(0u, 0u, 0u, 0u), q4 = p4;
                if (i < n_mine) { p4 = ld_behind(reinterpret_cast<const uint4*>(pt + i)); q4 = ld_behind(reinterpret_cast<const uint4*>(pq + i)); }
                fp[k] = __uint_as_float(p4.x); fp[k + 1] = __uint_as_float(p4.y); fp[k + 2] = __uint_as_float(p4.z); fp[k + 3] = __uint_as_float(p4.w);
                fq[k] = __uint_as_float(q4.x); fq[k + 1] = __uint_as_float(q4.y); fq[k + 2] = __uint_as_float(q4.z); fq[k + 3] = __uint_as_float(q4.w);
            }
        } else {
            #pragma unroll
            for (int k = 0; k < kAhead; ++k) {
                const int i = entry_of(k);
                fp[k] = i < n_mine ? ld_behind(pt + i) : 0.f;
                fq[k] = i < n_mine ? ld_behind(pq + i) : 0.f;
            }
        }
    };
    if (tid == 0) {
        tc::mbar_init(tc::smem_u32(&sh.bar[0]), 1);
        tc::mbar_init(tc::smem_u32(&sh.bar[1]), 1);
        tc::fence_barrier_init();
    }
    if (tid < 2 * kMaxCluster) sh.part[tid & 1][tid >> 1][0] = sh.part[tid & 1][tid >> 1][1] = 0;
    if (tid <= kMaxT) sh.kids[tid] = 0ull;
    __syncthreads();
    wait_for_predecessors();                           // (everything above needs nothing of them)
    fetch_row(0);
    if (tid <= T) sh.u_bonus[tid] = u_bonus[(size_t)b * (T + 1) + tid];
    float node_p = 0.f, node_q = 0.f;                  // the node's token in its parent's rows
    if (tid < T) {
        const int x = draft_tokens[(size_t)b * T + tid];
        int p = parents[(size_t)b * T + tid];
        sh.u_node[tid] = u_node[(size_t)b * T + tid];
        if (p < -1 || p >= tid) { if (rank == 0) atomicOr(status, kStatTree); p = -1; }
        sh.tok[tid] = x;
        atomicOr(&sh.kids[p + 1], 1ull << tid);
        if (x >= 0 && x < V) {
            node_p = ld_behind(p_seq + (size_t)(p + 1) * V + x);
            node_q = ld_behind(q_seq + (size_t)(p + 1) * V + x);
        }
    }
    cluster_arrive();
    cluster_wait();                                    // every CTA's barriers are initialised before anyone pushes
    auto next_child = [&](int of, int from) -> int {   // smallest child of node `of` with index >= from, or -1
        const unsigned long long m = from < 64 ? sh.kids[of + 1] >> from : 0ull;
        return m ? from + __ffsll((long long)m) - 1 : -1;
    };
    int cur = -1, n_acc = 0;
    uint32_t step = 0;
    bool ok = true, arrived = false;
    int32_t* out = path + (size_t)b * T;
    #pragma unroll 1
    for (int level = 0; level <= T && ok; ++level) {
        // (the row pair of node cur is in fp / fq, or on its way there)
        const float* pt = p_seq + (size_t)(cur + 1) * V + v_begin;
        const float* pq = q_seq + (size_t)(cur + 1) * V + v_begin;
        bool reread = false;                           // the row in shared memory is no longer what is asked for
        bool in_place = false;                         // it holds the current residual weights, not the original ones
        int n_rej = 0;                                 // rejections so far
        // entry i of this CTA's slice
        auto entry = [&](int i) -> uint2 {
            return i < n_res && !reread ? held(i) : make_uint2(fixed_prob(ld_behind(pt + i)), fixed_prob(ld_behind(pq + i)));
        };
        // weights of entry i now
        auto weights = [&](int i, long long* P, long long* Q) {
            const uint2 e = entry(i);
            if (in_place) { *P = e.x; *Q = e.y; }
            else weights_at(e.x, e.y, v_begin + i, sh.lv, n_rej, P, Q);
        };
        long long A = 0, Bq = 0;
        if (VEC) {
            A = fixed_probs(fp);
            Bq = fixed_probs(fq);                                  // (entries past the slice are zeros)
            #pragma unroll
            for (int k = 0; k < kAhead; k += 4) {
                const int i = entry_of(k);
                if (i < n_res) {                                   // (n_res is a multiple of four)
                    *reinterpret_cast<float4*>(P_s + i) = make_float4(fp[k], fp[k + 1], fp[k + 2], fp[k + 3]);
                    *reinterpret_cast<float4*>(Q_s + i) = make_float4(fq[k], fq[k + 1], fq[k + 2], fq[k + 3]);
                }
            }
        } else {
            #pragma unroll
            for (int k0 = 0; k0 < kAhead; k0 += 3) {               // (three weights fit 32 bits)
                uint32_t a3 = 0, b3 = 0;
                #pragma unroll
                for (int k = k0; k < k0 + 3 && k < kAhead; ++k) {
                    const int i = entry_of(k);
                    const uint2 e = make_uint2(fixed_prob(fp[k]), fixed_prob(fq[k]));
                    if (i < n_res) PQ_s[i] = e;
                    a3 += e.x;
                    b3 += e.y;
                }
                A += a3;
                Bq += b3;
            }
        }
        #pragma unroll 8
        for (int i = kAhead * kThreads + tid; i < n_mine; i += kThreads) {
            const uint2 e = make_uint2(fixed_prob(ld_behind(pt + i)), fixed_prob(ld_behind(pq + i)));
            if (i < n_res) put(i, e.x, e.y);
            A += e.x;
            Bq += e.y;
        }
        if (level == 0 && tid < T) { sh.node_P[tid] = fixed_prob(node_p); sh.node_Q[tid] = fixed_prob(node_q); }
        int c = next_child(cur, cur + 1);
        if (c >= 0) fetch_row(c + 1);
        ok = cluster_sum(sh, A, Bq, n_cta, rank, step++);
        if (tid < n_cta) sh.row_part[tid] = sh.part[(step - 1) & 1][tid][0];
        // The residual replaces the row where nothing can leave 32 bits.
        in_place = n_res == n_mine && A <= kPlainSum && Bq <= kPlainSum;
        // shares of the current A: those of the level's first sum until a rejection has a new one computed
        uint32_t a_step = step - 1;
        #pragma unroll 1
        while (c >= 0 && ok) {                                     // children of cur, in index order
            const int x = sh.tok[c];
            const bool in = x >= 0 && x < V;
            long long Px = 0, Qx = 0;
            if (in) weights_at(sh.node_P[c], sh.node_Q[c], x, sh.lv, n_rej, &Px, &Qx);
            else if (tid == 0 && rank == 0) atomicOr(status, kStatTree);        // a token outside the vocabulary is never accepted
            const unsigned __int128 lhs = (unsigned __int128)sh.u_node[c] * (unsigned long long)Qx * (unsigned long long)A;
            const unsigned __int128 rhs = ((unsigned __int128)(unsigned long long)Px * (unsigned long long)Bq) << 32;
            if (Qx > 0 && lhs < rhs) break;
            // rejected: the level's history grows by (A, B, x); the new A is the sum of the new residual
            const int sibling = next_child(cur, c + 1);
            if (sibling >= 0) fetch_row(sibling + 1);
            if (tid == 0) { sh.lv.A[n_rej] = A; sh.lv.B[n_rej] = Bq; sh.lv.x[n_rej] = in ? x : -1; }
            ++n_rej;
            // (read behind the barriers of the sum below, but where the pass itself reads it or there is none)
            if (!in_place || Bq <= 0) __syncthreads();
            if (Bq > 0) {
                long long s = 0;
                if (in_place) {
                    const uint32_t A0 = (uint32_t)A, B0 = (uint32_t)Bq;
                    auto residual = [&](uint32_t P, uint32_t Q) -> uint32_t {
                        const long long d = (long long)((unsigned long long)B0 * P) - (long long)((unsigned long long)A0 * Q);
                        return d > 0 ? (uint32_t)(d >> kProbBits) : 0u;
                    };
                    if (VEC) {
                        #pragma unroll 5
                        for (int i = 4 * tid; i < n_mine; i += 4 * kThreads) {
                            uint4 P = *reinterpret_cast<const uint4*>(P_s + i);
                            const uint4 Q = *reinterpret_cast<const uint4*>(Q_s + i);
                            P = make_uint4(residual(P.x, Q.x), residual(P.y, Q.y), residual(P.z, Q.z), residual(P.w, Q.w));
                            *reinterpret_cast<uint4*>(P_s + i) = P;
                            s += (long long)((unsigned long long)P.x + P.y) + (long long)((unsigned long long)P.z + P.w);
                        }
                        // the draft distribution loses x, by the thread that has just read it
                        const int at = x - v_begin;
                        if (in && at >= 0 && at < n_mine && (at >> 2) % kThreads == tid) Q_s[at] = 0u;
                    } else {
                        #pragma unroll 5
                        for (int i = tid; i < n_mine; i += kThreads) {
                            const uint2 e = PQ_s[i];
                            const uint32_t P = residual(e.x, e.y);
                            PQ_s[i] = make_uint2(P, v_begin + i == x ? 0u : e.y);
                            s += P;
                        }
                    }
                } else {
                    for (int i = tid; i < n_mine; i += kThreads) {
                        long long P, Q;
                        weights(i, &P, &Q);
                        s += P;
                    }
                }
                a_step = step;
                ok = cluster_sum(sh, s, n_cta, rank, step++);
                A = s;
            }
            Bq -= Qx;
            c = sibling;
        }
        if (c >= 0 && ok) {                                        // accepted
            if (tid == 0 && rank == 0) out[n_acc] = c;
            n_acc += 1;
            cur = c;
            __syncthreads();                                       // the history and the rows are replaced next
            continue;
        }
        if (!ok) break;
        cluster_arrive();                                          // this CTA pushes nothing more
        arrived = true;
        // nobody accepted: draw the next token from the residual (the original row if nothing is left of it)
        const bool original = A == 0;
        if (original) {
            __syncthreads();                                       // (row_part is there)
            n_rej = 0;
            reread = in_place;                                     // the residuals have replaced the row
            in_place = false;
            A = 0;
            for (int r = 0; r < n_cta; ++r) A += sh.row_part[r];
        }
        const unsigned long long t = (unsigned long long)(((unsigned __int128)sh.u_bonus[cur + 1] * (unsigned long long)A) >> 32);
        // the CTA whose slice holds the token: the shares of A in slice order
        long long before = 0;
        int owner = -1;
        for (int r = 0; r < n_cta; ++r) {
            const long long share = original ? sh.row_part[r] : sh.part[a_step & 1][r][0];
            if ((unsigned long long)(before + share) > t) { owner = r; break; }
            before += share;
        }
        if (owner < 0) {                                           // (A == 0 even for the original row)
            if (tid == 0 && rank == 0) bonus[b] = V - 1;
        } else if (owner == (int)rank) {
            // inside the slice: thread i owns entries [i per, (i + 1) per); its sum, a scan over the
            // threads, then a walk
            const int per = (n_mine + kThreads - 1) / kThreads;
            const int i0 = min(n_mine, tid * per), i1 = min(n_mine, i0 + per);
            long long mine = 0;
            for (int i = i0; i < i1; ++i) {
                long long P, Q;
                weights(i, &P, &Q);
                mine += P;
            }
            long long incl = mine;
            const int warp = tid >> 5, lane = tid & 31;
            #pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const long long n = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += n;
            }
            __syncthreads();
            if (lane == 31) sh.red[0][warp] = incl;
            __syncthreads();
            long long acc = before + incl - mine;
            for (int w = 0; w < warp; ++w) acc += sh.red[0][w];
            if ((unsigned long long)acc <= t && (unsigned long long)(acc + mine) > t) {      // exactly one thread
                int pick = i1 - 1;
                for (int i = i0; i < i1; ++i) {
                    long long P, Q;
                    weights(i, &P, &Q);
                    acc += P;
                    if ((unsigned long long)acc > t) { pick = i; break; }
                }
                bonus[b] = v_begin + pick;
            }
        }
        break;
    }
    if (rank == 0) {
        if (tid == 0) n_accept[b] = n_acc;
        for (int i = n_acc + tid; i < T; i += kThreads) out[i] = -1;
    }
    if (!ok && tid == 0) atomicOr(status, timeout_bits(kSiteSample));
    // No CTA leaves before its peers have sent their last push (they have, long since, unless a wait gave up).
    if (!arrived) cluster_arrive();
    cluster_wait();
}

}  // namespace sample
}  // namespace sparrow
