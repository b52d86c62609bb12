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
// Measured on a 32-node tree over 151,936 entries (kernel time; the walk's length depends on the
// uniforms): 16 to 35 us with clusters of 16; one CTA per sequence, with the rows read again from L2 in
// every pass and the serial scan of the draw, took 145 to 420 us.  Stamps of a level: 1.1 us to turn
// two rows into fixed point, 0.5 us to request the next, 0.9 us for the cluster's sum.
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

// Rows whose sums stay below this (1 + 2^-7 in fixed point) keep every residual weight below 2^31, through
// up to 64 rejections: P' <= (B P) / 2^30 and A' <= (B A) / 2^30, and (1 + 2^-7)^64 < 1.7.
constexpr long long kPlainSum = (1ll << kProbBits) + (1ll << (kProbBits - 7));

struct Level {                      // history of the rejections at the current node
    long long A[kMaxT], B[kMaxT];
    int x[kMaxT];
    int n;
};

// Current residual target weight and current draft weight of an entry with original weights P0, Q0
// at vocabulary index v.
__device__ __forceinline__ void weights_at(uint32_t P0, uint32_t Q0, int v, const Level& lv, long long* P_out, long long* Q_out)
{
    long long P = P0;
    const long long q0 = Q0;
    bool gone = false;               // v was a rejected candidate: the draft distribution has lost it
    for (int s = 0; s < lv.n; ++s) {
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

// Sums (a, b) over the cluster; every thread gets the totals, sh.part[step & 1] the CTAs' shares.
// False when the peers' pushes did not arrive within the poll limit.
__device__ __forceinline__ bool cluster_sum(Shared& sh, long long& a, long long& b, int n_cta, uint32_t rank, uint32_t step)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    a = warp_sum(a);
    b = warp_sum(b);
    if (lane == 0) { sh.red[0][warp] = a; sh.red[1][warp] = b; }
    __syncthreads();
    if (warp == 0) {
        if (lane == 0) tc::mbar_expect_tx(tc::smem_u32(&sh.bar[step & 1]), 16u * (uint32_t)n_cta);
        a = warp_sum(lane < kWarps ? sh.red[0][lane] : 0ll);
        b = warp_sum(lane < kWarps ? sh.red[1][lane] : 0ll);
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

__global__ void __launch_bounds__(kThreads)
accept_sample_kernel(const int32_t* draft_tokens, const int32_t* parents,
                     const float* p_target, const float* p_draft,
                     const uint32_t* u_node, const uint32_t* u_bonus, int T, int V, int n_cta, int resident,
                     int32_t* path, int32_t* n_accept, int32_t* bonus, unsigned* status)
{
    let_dependents_launch();
    extern __shared__ uint2 row_s[];                   // the first `resident` entries of this CTA's slice: (P, Q) fixed point
    __shared__ Shared sh;
    const int b = blockIdx.x / n_cta, tid = threadIdx.x;
    const uint32_t rank = n_cta > 1 ? cluster_rank() : 0u;
    const int per_cta = (V + n_cta - 1) / n_cta;
    const int v_begin = min(V, (int)rank * per_cta), n_mine = min(V, v_begin + per_cta) - v_begin;
    const int n_res = min(n_mine, resident);
    const float* p_seq = p_target + (size_t)b * (T + 1) * V;       // row r of this sequence: p_seq + r V
    const float* q_seq = p_draft + (size_t)b * (T + 1) * V;

    // the first kAhead entries per thread of a row pair, on their way
    float fp[kAhead], fq[kAhead];
    auto fetch_row = [&](int r) {
        const float* pt = p_seq + (size_t)r * V + v_begin;
        const float* pq = q_seq + (size_t)r * V + v_begin;
        #pragma unroll
        for (int k = 0; k < kAhead; ++k) {
            const int i = k * kThreads + tid;
            fp[k] = i < n_mine ? ld_behind(pt + i) : 0.f;
            fq[k] = i < n_mine ? ld_behind(pq + i) : 0.f;
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
        bool reread = false;                           // row_s no longer holds what is asked for
        bool in_place = false;                         // row_s holds the current residual weights, not the original ones
        // entry i of this CTA's slice
        auto entry = [&](int i) -> uint2 {
            return i < n_res && !reread ? row_s[i] : make_uint2(fixed_prob(ld_behind(pt + i)), fixed_prob(ld_behind(pq + i)));
        };
        // weights of entry i now
        auto weights = [&](int i, long long* P, long long* Q) {
            const uint2 e = entry(i);
            if (in_place) { *P = e.x; *Q = e.y; }
            else weights_at(e.x, e.y, v_begin + i, sh.lv, P, Q);
        };
        long long A = 0, Bq = 0;
        #pragma unroll
        for (int k0 = 0; k0 < kAhead; k0 += 3) {                   // (three weights fit 32 bits)
            uint32_t a3 = 0, b3 = 0;
            #pragma unroll
            for (int k = k0; k < k0 + 3 && k < kAhead; ++k) {
                const int i = k * kThreads + tid;
                const uint2 e = make_uint2(fixed_prob(fp[k]), fixed_prob(fq[k]));
                if (i < n_res) row_s[i] = e;
                a3 += e.x;
                b3 += e.y;
            }
            A += a3;
            Bq += b3;
        }
        #pragma unroll 8
        for (int i = kAhead * kThreads + tid; i < n_mine; i += kThreads) {
            const uint2 e = make_uint2(fixed_prob(ld_behind(pt + i)), fixed_prob(ld_behind(pq + i)));
            if (i < n_res) row_s[i] = e;
            A += e.x;
            Bq += e.y;
        }
        if (level == 0 && tid < T) { sh.node_P[tid] = fixed_prob(node_p); sh.node_Q[tid] = fixed_prob(node_q); }
        int c = next_child(cur, cur + 1);
        if (c >= 0) fetch_row(c + 1);
        if (tid == 0) sh.lv.n = 0;
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
            if (in) weights_at(sh.node_P[c], sh.node_Q[c], x, sh.lv, &Px, &Qx);
            else if (tid == 0 && rank == 0) atomicOr(status, kStatTree);        // a token outside the vocabulary is never accepted
            const unsigned __int128 lhs = (unsigned __int128)sh.u_node[c] * (unsigned long long)Qx * (unsigned long long)A;
            const unsigned __int128 rhs = ((unsigned __int128)(unsigned long long)Px * (unsigned long long)Bq) << 32;
            if (Qx > 0 && lhs < rhs) break;
            // rejected: the level's history grows by (A, B, x); the new A is the sum of the new residual
            const int sibling = next_child(cur, c + 1);
            if (sibling >= 0) fetch_row(sibling + 1);
            __syncthreads();                                       // everybody has read the history as it was
            if (tid == 0) { sh.lv.A[sh.lv.n] = A; sh.lv.B[sh.lv.n] = Bq; sh.lv.x[sh.lv.n] = in ? x : -1; sh.lv.n += 1; }
            __syncthreads();
            if (Bq > 0) {
                long long s = 0, none = 0;
                if (in_place) {
                    const uint32_t A0 = (uint32_t)A, B0 = (uint32_t)Bq;
                    #pragma unroll 5
                    for (int i = tid; i < n_mine; i += kThreads) {
                        const uint2 e = row_s[i];
                        const long long d = (long long)((unsigned long long)B0 * e.x) - (long long)((unsigned long long)A0 * e.y);
                        const uint32_t P = d > 0 ? (uint32_t)(d >> kProbBits) : 0u;
                        row_s[i] = make_uint2(P, v_begin + i == x ? 0u : e.y);
                        s += P;
                    }
                } else {
                    for (int i = tid; i < n_mine; i += kThreads) {
                        long long P, Q;
                        weights(i, &P, &Q);
                        s += P;
                    }
                }
                a_step = step;
                ok = cluster_sum(sh, s, none, n_cta, rank, step++);
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
            __syncthreads();
            if (tid == 0) sh.lv.n = 0;
            __syncthreads();
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
