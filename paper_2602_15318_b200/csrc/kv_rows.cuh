// Row movers around the two attention modes: appending the draft tokens' K/V rows to a cache,
// and compacting the text-anchored rows of a long cache into a short contiguous one (Section 3.1:
// the draft model keeps only the text-anchored states and discards the visual KV cache), after
// which the anchored mode is an ordinary contiguous stream for the tensor-core kernel.
//
// One thread moves 16 bytes; 16 consecutive threads move one 256-byte row of K and the same row
// of V.  Pure copies: results are bit-exact.
#pragma once
#include <cuda_bf16.h>

#include "common.cuh"

namespace sparrow {

// N: room for the sequences.  A launch with less than about 128 bytes of arguments costs the host 1.85 us, one
// with 440 bytes 2.1, and these launches are bound by it: commit of 28 layers, 57 launches, 183 -> 171 us.
template <int N>
struct RowMoveArgs {
    const __nv_bfloat16* k_src;
    const __nv_bfloat16* v_src;
    __nv_bfloat16* k_dst;
    __nv_bfloat16* v_dst;
    const int32_t* src_rows;         // DEV [batch][n_rows] source row of each moved row, or nullptr: rows 0 .. n_rows-1
    int32_t n_rows;                  // rows moved per (sequence, KV head)
    int32_t batch, n_kv_heads;
    int32_t src_capacity;            // valid source rows are [0, src_capacity)
    int64_t src_stride_batch, src_stride_head;      // in elements
    int64_t dst_stride_batch, dst_stride_head;
    unsigned* status;
    int32_t dst_row0[N];             // first destination row per sequence
};

// Where chunk i of the (sequence, KV head, row, 16-byte column) index space lies.  (Rows are counted in 32 bits: a
// 64-bit division is a hundred dependent instructions.)
struct RowChunk {
    int b, h, r, c;
    size_t src_head, dst;            // element offsets: the source's (sequence, KV head) with the column, the destination
};
template <int N>
__device__ __forceinline__ RowChunk find_row_chunk(const RowMoveArgs<N>& a, long long i)
{
    RowChunk x;
    x.c = (int)(i & 15);
    const unsigned row = (unsigned)(i >> 4), unit = row / (unsigned)a.n_rows;
    x.r = (int)(row - unit * (unsigned)a.n_rows);
    x.b = (int)(unit / (unsigned)a.n_kv_heads);
    x.h = (int)(unit - (unsigned)x.b * (unsigned)a.n_kv_heads);
    x.src_head = (size_t)x.b * a.src_stride_batch + (size_t)x.h * a.src_stride_head + x.c * 8;
    x.dst = (size_t)x.b * a.dst_stride_batch + (size_t)x.h * a.dst_stride_head + (size_t)(a.dst_row0[x.b] + x.r) * kD + x.c * 8;
    return x;
}
// Moves 16 bytes of K and of V.
template <int N>
__device__ __forceinline__ void move_row_chunk(const RowMoveArgs<N>& a, const RowChunk& x)
{
    const int src = a.src_rows ? ld_behind(a.src_rows + (size_t)x.b * a.n_rows + x.r) : x.r;
    const bool bad = src < 0 || src >= a.src_capacity;       // never read: the row is written as zeros
    if (bad && x.c == 0 && x.h == 0) atomicOr(a.status, kStatAnchor);
    const size_t s_off = x.src_head + (size_t)(bad ? 0 : src) * kD;
    uint4 kv = make_uint4(0, 0, 0, 0), vv = make_uint4(0, 0, 0, 0);
    if (!bad) {
        kv = *reinterpret_cast<const uint4*>(a.k_src + s_off);
        vv = *reinterpret_cast<const uint4*>(a.v_src + s_off);
    }
    *reinterpret_cast<uint4*>(a.k_dst + x.dst) = kv;
    *reinterpret_cast<uint4*>(a.v_dst + x.dst) = vv;
}

template <int N>
__global__ void __launch_bounds__(256)
move_rows_kernel(const __grid_constant__ RowMoveArgs<N> a)
{
    let_dependents_launch();
    const long long total = (long long)a.batch * a.n_kv_heads * a.n_rows * 16;
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    RowChunk x = find_row_chunk(a, i < total ? i : 0);       // (before the wait: the addresses need nothing of it)
    wait_for_predecessors();
    while (i < total) {
        move_row_chunk(a, x);
        i += (long long)gridDim.x * blockDim.x;
        if (i < total) x = find_row_chunk(a, i);
    }
}

// One step's inputs straight from host memory that the GPU can address (pinned or registered):
// the queries and the tree go to device staging (the attention kernel fetches the queries by TMA),
// the draft tokens' K/V rows go to their cache rows.  One 16-byte load per thread and buffer, all
// in flight together, so the launch costs about one round trip over the host link.
struct IngestArgs {
    RowMoveArgs<kMaxBatch> rows;     // k_src / v_src are host memory here
    const uint4* q_src;              // host view
    uint4* q_dst;
    const int32_t* parents_src;      // host view
    int32_t* parents_dst;
    int32_t q_chunks, n_parents;
};

__global__ void __launch_bounds__(256)
ingest_step_kernel(const __grid_constant__ IngestArgs a)
{
    // in this order: the attention call behind this kernel starts streaming the cache's prefix, which this
    // kernel does not write, as soon as it is launched, and relies on everything earlier being complete
    const long long row_chunks = (long long)a.rows.batch * a.rows.n_kv_heads * a.rows.n_rows * 16;
    const long long total = row_chunks + a.q_chunks + a.n_parents;
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    RowChunk x = find_row_chunk(a.rows, i < row_chunks ? i : 0);
    wait_for_predecessors();
    let_dependents_launch();
    for (; i < total; i += (long long)gridDim.x * blockDim.x) {
        if (i < row_chunks) {
            if (i >= (long long)gridDim.x * blockDim.x) x = find_row_chunk(a.rows, i);
            move_row_chunk(a.rows, x);
        }
        else if (i < row_chunks + a.q_chunks) a.q_dst[i - row_chunks] = a.q_src[i - row_chunks];
        else a.parents_dst[i - row_chunks - a.q_chunks] = a.parents_src[i - row_chunks - a.q_chunks];
    }
}

}  // namespace sparrow
