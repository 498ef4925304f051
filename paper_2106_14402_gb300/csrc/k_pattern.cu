// (or,and) products whose stored values are all true: every entry of C is
// true, so the values of C follow from its pattern, which the symbolic phase
// has already found.  Rows of the bitmap tier are then read out of their
// stored bitmaps, with no product formed a second time (numeric phase of
// R-MAT s18: 24.3 -> 6.9 ms; C is 15 GB, 2.2 ms of writes).  With a false
// value anywhere, or without stored bitmaps, the products decide (k_num_rank).
#include "cb_common.cuh"
#include "cb_kernels.h"

namespace cb {
namespace {

// counters[kFalse] > 0 when a stored value of M's rows is 0.  A whole matrix
// is one run of bytes, read 16 at a time (its ends byte by byte); a column
// window's rows are runs of their own, a warp per row.
__device__ __forceinline__ unsigned zero_bytes(unsigned x) { return (x - 0x01010101u) & ~x & 0x80808080u; }

__global__ void __launch_bounds__(256) k_any_false(DevCSR M, int64_t* counters) {
  const uint8_t* v = static_cast<const uint8_t*>(M.val);
  int bad = 0;
  if (!M.rpe) {
    const int64_t e0 = M.rp[0], e1 = M.rp[M.nrows];
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, n = (int64_t)gridDim.x * blockDim.x;
    const int64_t head = min(e1, e0 + (int64_t)((16 - (reinterpret_cast<uintptr_t>(v + e0) & 15)) & 15));
    const int64_t quads = (e1 - head) >> 4, tail = head + 16 * quads;
    for (int64_t q = e0 + t; q < head; q += n) bad |= v[q] == 0;
    const uint4* w = reinterpret_cast<const uint4*>(v + head);
    for (int64_t q = t; q < quads; q += n) {
      const uint4 x = __ldg(w + q);
      bad |= (zero_bytes(x.x) | zero_bytes(x.y) | zero_bytes(x.z) | zero_bytes(x.w)) != 0u;
    }
    for (int64_t q = tail + t; q < e1; q += n) bad |= v[q] == 0;
  } else {
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t r = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); r < M.nrows; r += nwarps) {
      const int64_t q1 = row_end(M, r);
      for (int64_t q = M.rp[r] + lane; q < q1; q += 32) bad |= v[q] == 0;
    }
  }
  bad = __syncthreads_or(bad);
  if (bad && threadIdx.x == 0) atomicAdd((unsigned long long*)&counters[kFalse], 1ull);
}

constexpr int kPatThreads = 256;
constexpr int kPatWarps = kPatThreads / 32;

// One CTA per (heavy row, span): its warps take equal runs of the span's
// words, count them, and read them out 32 words at a time: a lane walks its
// word's bits into the warp's shared buffer at their ranks and the warp copies
// the buffer out (a walk straight to C costs an L2 request per entry).  The
// words are read twice, the second time from L2.  Bound by issue (the walk:
// the fullest of 32 words) and by C's writes.
__global__ void __launch_bounds__(kPatThreads) k_pattern_rows(DevCSR A, DevCSR B, const int32_t* heavy_rows,
                                                              int64_t units, int64_t spans,
                                                              const int32_t* span_counts,
                                                              const unsigned* hbits, const int64_t* nnz,
                                                              const int64_t* Crp, int32_t* Ccol, uint8_t* Cval,
                                                              int64_t* err, int64_t* queue,
                                                              int64_t num_hash_max) {
  __shared__ int32_t stage[kPatWarps][1024];
  __shared__ int wsum[kPatWarps];
  __shared__ long long next;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  take_unit(queue, &next);
  __syncthreads();
  for (int64_t u = next; u < units; u = next) {
    const int64_t h = u / spans, sp = u - h * spans;
    const int i = heavy_rows[h];
    const int64_t lo = B.col_lo + sp * (int64_t)kSpanCols;
    const int64_t hi = min(lo + (int64_t)kSpanCols, B.col_lo + row_width(A, B, i));
    const int count = span_counts[u];
    const bool skip = nnz[i] <= num_hash_max || hi <= lo || count == 0;  // hash tiers own the small rows
    const int nw = skip ? 0 : (int)((hi - lo + 31) / 32);
    const int per = ((nw + kPatWarps * 32 - 1) / (kPatWarps * 32)) * 32;  // words of a warp
    const int w0 = min(nw, warp * per), w1 = min(nw, w0 + per);
    const unsigned* bits = hbits + (size_t)u * kSpanWords;
    int mine = 0;
    for (int w = w0 + lane; w < w1; w += 32) mine += __popc(bits[w]);
    mine = __reduce_add_sync(0xffffffffu, mine);
    if (lane == 0) wsum[warp] = mine;
    int64_t out = 0;  // C's entries before the span
    for (int64_t t = 0; t < sp; ++t) out += span_counts[h * spans + t];
    out += Crp[i];
    const int64_t row_end_c = Crp[i + 1];
    __syncthreads();
    take_unit(queue, &next);
    int before = 0, total = 0;
#pragma unroll
    for (int v = 0; v < kPatWarps; ++v) {
      before += v < warp ? wsum[v] : 0;
      total += wsum[v];
    }
    if (tid == 0 && !skip && total != count) atomicCAS((unsigned long long*)err, 0ull, 24ull);
    int64_t o = out + before;
    for (int g = w0; g < w1; g += 32) {
      unsigned word = g + lane < w1 ? bits[g + lane] : 0u;
      const int n = __popc(word);
      int incl = n;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += y;
      }
      const int all = __shfl_sync(0xffffffffu, incl, 31);
      int32_t* at = &stage[warp][incl - n];
      const int32_t c = (int32_t)(lo + 32 * (int64_t)(g + lane));
      while (word) {
        *at++ = c + __ffs(word) - 1;
        word &= word - 1;
      }
      __syncwarp();
      const int fit = (int)max((int64_t)0, min((int64_t)all, row_end_c - o));  // (all, unless a count is wrong)
      guard(fit == all, 39, o + all);
      for (int t = lane; t < fit; t += 32) st_out(Ccol + o + t, stage[warp][t]);
      o += all;
      __syncwarp();
    }
    // the span's values: 1, sixteen to a store between the 16-byte boundaries
    const int64_t v0 = skip ? 0 : out, v1 = skip ? 0 : max(v0, min(row_end_c, out + total));
    const int64_t h1 = min(v1, v0 + (int64_t)((16 - (reinterpret_cast<uintptr_t>(Cval + v0) & 15)) & 15));
    const int64_t quads = (v1 - h1) >> 4;
    if (v0 + tid < h1) Cval[v0 + tid] = 1;
    const uint4 ones = make_uint4(0x01010101u, 0x01010101u, 0x01010101u, 0x01010101u);
    for (int64_t q = tid; q < quads; q += kPatThreads) __stcs(reinterpret_cast<uint4*>(Cval + h1) + q, ones);
    if (h1 + 16 * quads + tid < v1) Cval[h1 + 16 * quads + tid] = 1;
    __syncthreads();
  }
}

}  // namespace

void launch_any_false(const DevCSR& M, int64_t* counters, cudaStream_t s, int sms) {
  if (M.nrows == 0) return;
  k_any_false<<<sms * 4, 256, 0, s>>>(M, counters);
}

void launch_pattern_rows(const DevCSR& A, const DevCSR& B, const int32_t* heavy_rows, int64_t n_heavy,
                         int64_t spans, const int32_t* span_counts, const unsigned* hbits, const int64_t* nnz,
                         const int64_t* Crp, int32_t* Ccol, void* Cval, int64_t* counters, cudaStream_t s,
                         int sms, int64_t num_hash_max) {
  const int64_t units = n_heavy * spans;
  if (units == 0) return;
  const int64_t most = (int64_t)sms * 6;
  k_pattern_rows<<<(unsigned)(units < most ? units : most), kPatThreads, 0, s>>>(
      A, B, heavy_rows, units, spans, span_counts, hbits, nnz, Crp, Ccol, static_cast<uint8_t*>(Cval),
      counters + kError, counters + kNumQueue, num_hash_max);
}

CB_CHECK_READER(pattern)

}  // namespace cb
