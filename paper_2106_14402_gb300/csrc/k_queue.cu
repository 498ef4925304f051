// One-pass SpGEMM for rows of bounded size and width, run by a persistent
// kernel that takes rows from a device work queue.  It serves the batched
// workloads of many independent products (paper Sec. 5 runs one library
// call per product; here the stacked rows of all products of a wave are one
// queue), where every output row holds at most kQueueAcc entries and lies in
// a column range of at most kQueueWidth columns.
//
// The three phases of Sec. 4.1 collapse per row, in one CTA:
//   1. flops bound and load balance: the row's A entries go through shared
//      memory, a warp takes four of their B rows at a time;
//   2. symbolic: the products' columns set bits of a dense bitmap of the
//      row's column range; popcounts, prefix-summed, give nnz(C_i) and every
//      column's rank;
//   3. numeric: each column's first product (the one that set its bit) is
//      stored, with the column, at the column's rank, the others are combined
//      into it with the semiring's atomic after a barrier; no accumulator is
//      initialised and the row comes out in column order with no sort.
// The rows' compression ratio is near 1 (uniform operands), so nearly every
// product is its column's first.  Semirings whose accumulator is C's value
// store it in C itself, the others in shared memory.
// A row is a chain of dependent latencies (queue, A's row, B's bounds, B's
// rows, look-back, B's rows again: about 13000 cycles), so the kernel lives
// from the rows an SM has in flight: small CTAs and no per-row accumulator
// (256-thread CTAs with a 4096-entry accumulator, four or five rows on an SM
// and an A entry per warp at a time, took 22.2 ms for 950000 rows of 1730
// fp64 products; an ER product of 65536 rows of 1600 fp64 products took 1.9 ms,
// now 1.02).
// Rows are dequeued in order with one atomic per row, and a row's output
// offset comes from a decoupled look-back over the rows before it, whose
// CTAs are all running (they dequeued earlier) and never wait on later rows:
// no cooperative launch is needed.  Row status words carry the launch epoch
// of the one-launch kernel (shared tile-status array and sync words), so no
// reset is needed between launches.  Waits are bounded: a row that gives up
// records CB_FUSED_STALLED and publishes anyway.  (spin_limit and silent_row
// serve fault injection: a row that never publishes.)
#include <algorithm>

#include "cb.h"
#include "cb_common.cuh"
#include "cb_kernels.h"

namespace cb {
namespace {

constexpr int kQThreads = 128;
constexpr int kQWarps = kQThreads / 32;
constexpr int kQWords = kQueueWidth / 32;   // bitmap words of the widest row
constexpr int kQRepeats = 256;              // repeated products kept in shared memory
constexpr unsigned kQFull = 0xFFFFFFFFu;

// Whether the accumulators live in C's values (of their size); where the bits
// differ (cb_wlabel's packed keys) they are converted when the row is complete.
template <int SR>
constexpr bool kQInPlace = sizeof(typename Sem<SR>::A) == sizeof(typename Sem<SR>::TC);
template <int SR>
constexpr bool kQConvert = SR == 6 || SR == 7;

// The sum that starts with product y: y, but +0.0 for -0.0, as 0.0 + y gives
// (on the bits: an addition, a second use of the FP64 pipe, took 1.3% of a
// batched call).
template <int SR>
__device__ __forceinline__ typename Sem<SR>::A started(typename Sem<SR>::A y) {
  if constexpr (SR == 2) return __double_as_longlong(y) == LLONG_MIN ? 0.0 : y;
  else return y;
}

// CTAs per SM: 64 registers a thread, 12 bytes of them spilled for int64 and
// fp64 (7 and 9 took 2% and 9% longer).
constexpr int kQCtas = 8;

// status words: [63:40] epoch, [39:38] kind, [37:0] value (as in k_fused.cu)
constexpr int kQEpochShift = 40;
constexpr unsigned kQEpochMask = (1u << 24) - 1;
constexpr unsigned long long kQAgg = 1ull << 38;
constexpr unsigned long long kQInc = 2ull << 38;
constexpr unsigned long long kQKind = 3ull << 38;
constexpr unsigned long long kQVal = (1ull << 38) - 1;

__device__ __forceinline__ unsigned long long ld_volatile64(const unsigned long long* p) {
  return *reinterpret_cast<const volatile unsigned long long*>(p);
}

template <int SR>
__global__ void __launch_bounds__(kQThreads, kQInPlace<SR> ? kQCtas : 5)
    k_queue_rows(DevCSR A, DevCSR B, int64_t m, int64_t* __restrict__ Crp, int32_t* Ccol,
                 typename Sem<SR>::TC* Cval, int64_t cap, unsigned long long* tstat, int64_t tstat_cap,
                 unsigned* sync, int* status, unsigned spin_limit, int64_t silent_row) {
  typedef Sem<SR> S;
  typedef typename S::A Acc;
  typedef typename S::TA TA;
  typedef typename S::TB TB;
  constexpr bool kInPlace = kQInPlace<SR>;
  __shared__ __align__(16) unsigned bits[kQWords];
  __shared__ __align__(16) unsigned short pre[kQWords];  // entries in the row's earlier words (< kQueueAcc)
  __shared__ unsigned short cols[kQueueAcc];             // the row's columns in order
  __shared__ Acc acc_s[kInPlace ? 1 : kQueueAcc];
  __shared__ long long s_q[kQThreads];  // A entries, kQThreads at a time: first B entry,
  __shared__ int s_len[kQThreads];      // B row length
  __shared__ TA s_a[kQThreads];         // and A's value
  __shared__ unsigned short rep_slot[kQRepeats];
  __shared__ Acc rep_val[kQRepeats];
  __shared__ int s_rep;
  __shared__ int s_wsum[kQWarps];
  __shared__ int s_min[kQWarps];
  __shared__ long long s_red[kQWarps];
  __shared__ long long s_row;
  __shared__ unsigned s_epoch, s_last;
  static_assert(kQueueWidth <= 65536 && kQueueAcc <= 65536, "columns and slots are kept in 16 bits");
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const TA* __restrict__ Aval = reinterpret_cast<const TA*>(A.val);
  const TB* __restrict__ Bval = reinterpret_cast<const TB*>(B.val);
  unsigned long long* queue = reinterpret_cast<unsigned long long*>(sync + 10);
  if (tid == 0) s_epoch = *reinterpret_cast<volatile unsigned*>(sync) & kQEpochMask;
  __syncthreads();
  const unsigned long long ep = (unsigned long long)s_epoch << kQEpochShift;

  for (;;) {
    if (tid == 0) {
      s_row = (long long)atomicAdd(queue, 1ull);
      s_rep = 0;
    }
    __syncthreads();
    const int64_t r = s_row;
    if (r >= m) break;
    const unsigned width = (unsigned)row_width(A, B, r);
    const int nw = (int)((width + 31) >> 5);
    const int64_t a0 = A.rp[r], a1 = A.rp[r + 1];
    const unsigned col_lo = (unsigned)B.col_lo;
    for (int w = tid; w < (nw + 3) / 4; w += kQThreads)
      reinterpret_cast<uint4*>(bits)[w] = make_uint4(0u, 0u, 0u, 0u);
    const auto stage = [&](int64_t c0) {
      const int64_t p = c0 + tid;
      int64_t len = 0;
      if (p < a1) {
        const int k = __ldg(A.col + p);
        const int64_t q0 = __ldg(B.rp + k);
        len = row_end(B, k) - q0;
        s_q[tid] = q0;
        if (S::kUsesA) s_a[tid] = ldg_val(Aval + p);
      }
      s_len[tid] = (int)min(len, (int64_t)(INT_MAX - 64));  // (a row of this kernel holds at most kQueueAcc products)
    };
    // A warp's share of the A entries from c0 on, four B rows at a time and up
    // to 64 entries of each per step: f(step, e0, x, most), x the lane's first
    // entry, most the longest of the four.
    const auto walk = [&](int64_t c0, int& step, auto&& f) {
      const int n = (int)min((int64_t)kQThreads, a1 - c0);
      for (int e0 = 4 * warp; e0 < n; e0 += 4 * kQWarps) {
        const int most = max(max(s_len[e0], s_len[e0 + 1]), max(s_len[e0 + 2], s_len[e0 + 3]));
        for (int x = 0; x < most; x += 64, ++step) f(step, e0, x + lane, most - x);
      }
    };
    // symbolic: the row's columns.  A lane keeps a bit for each product of the
    // warp's first 8 steps: set when the product is not its column's first.
    unsigned long long later = 0;
    int steps = 0;
    for (int64_t c0 = a0; c0 < a1; c0 += kQThreads) {
      if (c0 != a0) __syncthreads();
      stage(c0);
      __syncthreads();
      walk(c0, steps, [&](int step, int e0, int x, int most) {
        int c[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          if (u >= 4 && most <= 32) break;  // uniform
          const int e = e0 + (u & 3), y = x + 32 * (u >> 2);
          c[u] = y < s_len[e] ? __ldg(B.col + s_q[e] + y) : -1;
        }
        unsigned was = 0;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          if (u >= 4 && most <= 32) break;
          const unsigned d = (unsigned)c[u] - col_lo;
          if (c[u] >= 0 && guard(d < width, 42, d)) {
            const unsigned bit = 1u << (d & 31);
            if (atomicOr(&bits[d >> 5], bit) & bit) was |= 1u << u;
          }
        }
        later |= (unsigned long long)was << ((8 * step) & 63);
      });
    }
    // a warp with more steps (a few long B rows, many A entries) sends the row
    // through the atomic for every product
    const bool marked = !__syncthreads_or(steps > 8);

    // ranks: exclusive prefix of the word popcounts.  A thread reads a run of
    // WPT words at once and stores the counts before them; WPT (uniform) keeps
    // the threads at work in narrow rows.  (Words past the row's last one, in
    // its 16-byte vector, are clear.)
    int nnz = 0;
    const auto rank_words = [&](auto wpt) {
      constexpr int WPT = decltype(wpt)::value;
      unsigned w[WPT];
      const int w0 = tid * WPT;
      int mine = 0;
#pragma unroll
      for (int q = 0; q < WPT / 4; ++q) {
        const uint4 v = w0 + 4 * q < nw ? reinterpret_cast<const uint4*>(bits + w0)[q] : make_uint4(0u, 0u, 0u, 0u);
        w[4 * q] = v.x;
        w[4 * q + 1] = v.y;
        w[4 * q + 2] = v.z;
        w[4 * q + 3] = v.w;
        mine += __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w);
      }
      int incl = mine;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int y = __shfl_up_sync(kQFull, incl, d);
        if (lane >= d) incl += y;
      }
      if (lane == 31) s_wsum[warp] = incl;
      __syncthreads();
      int before = 0;
#pragma unroll
      for (int v = 0; v < kQWarps; ++v) {
        const int x = s_wsum[v];
        before += v < warp ? x : 0;
        nnz += x;
      }
      // publish the row's size
      if (tid == 0 && r != silent_row)  // (fault injection: a row that never publishes)
        atomicExch(&tstat[r], ep | (r == 0 ? kQInc : kQAgg) | (unsigned long long)(nnz <= kQueueAcc ? nnz : 0));
      if (nnz > kQueueAcc || w0 >= nw) return;  // (the row does not fit this kernel)
      int run = before + incl - mine;
#pragma unroll
      for (int q = 0; q < WPT / 4; ++q) {
        unsigned p[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const unsigned lo16 = (unsigned)run;
          run += __popc(w[4 * q + 2 * h]);
          p[h] = lo16 | ((unsigned)run << 16);
          run += __popc(w[4 * q + 2 * h + 1]);
        }
        if (w0 + 4 * q < nw) *reinterpret_cast<uint2*>(pre + w0 + 4 * q) = make_uint2(p[0], p[1]);
      }
    };
    if (nw > 8 * kQThreads) rank_words(std::integral_constant<int, 16>{});
    else if (nw > 4 * kQThreads) rank_words(std::integral_constant<int, 8>{});
    else rank_words(std::integral_constant<int, 4>{});
    const bool fits = nnz <= kQueueAcc;
    if (!fits) {  // the row does not fit this kernel (uniform)
      if (tid == 0) atomicOr(status, CB_FUSED_ROW_TOO_LARGE);
      nnz = 0;
    }

    // the row's offset from the rows before it, two of them per thread
    long long excl = 0;
    for (int64_t top = r - 1; top >= 0; top -= 2 * kQThreads) {
      unsigned long long wv[2] = {0, 0};
      int first = 2 * kQThreads;
#pragma unroll
      for (int h = 1; h >= 0; --h) {
        const int64_t j = top - 2 * tid - h;
        if (j < 0) continue;
        unsigned spins = 0;
        for (;;) {
          wv[h] = ld_volatile64(&tstat[j]);
          if ((wv[h] & ~((1ull << kQEpochShift) - 1)) == ep && (wv[h] & kQKind)) break;
          if (++spins >= spin_limit) {
            atomicOr(status, CB_FUSED_STALLED);
            wv[h] = ep | kQInc;
            break;
          }
          __nanosleep(32);
        }
        if ((wv[h] & kQKind) == kQInc) first = 2 * tid + h;
      }
      // the nearest inclusive prefix in this window (smallest index)
      first = __reduce_min_sync(kQFull, first);
      if (lane == 0) s_min[warp] = first;
      __syncthreads();
      int stop = 2 * kQThreads;
#pragma unroll
      for (int v = 0; v < kQWarps; ++v) stop = min(stop, s_min[v]);
      long long part = (2 * tid <= stop ? (long long)(wv[0] & kQVal) : 0) +
                       (2 * tid + 1 <= stop ? (long long)(wv[1] & kQVal) : 0);
#pragma unroll
      for (int d = 16; d >= 1; d >>= 1) part += __shfl_xor_sync(kQFull, part, d);
      if (lane == 0) s_red[warp] = part;
      __syncthreads();
#pragma unroll
      for (int v = 0; v < kQWarps; ++v) excl += s_red[v];
      __syncthreads();
      if (stop < 2 * kQThreads) break;
    }
    if (tid == 0) {
      if (r > 0 && r != silent_row) atomicExch(&tstat[r], ep | kQInc | (unsigned long long)(excl + nnz));
      Crp[r] = excl;
      if (r == m - 1) {
        Crp[m] = excl + nnz;
        __threadfence();  // before this CTA counts itself finished
      }
    }
    const long long base = excl;
    const int n = nnz;
    if (base + n > cap) {  // uniform
      if (tid == 0 && n > 0) atomicOr(status, CB_FUSED_CAPACITY);
      __syncthreads();
      continue;
    }
    Acc* acc = kInPlace ? reinterpret_cast<Acc*>(Cval + base) : acc_s;
    if (!marked)
      for (int t = tid; t < n; t += kQThreads) acc[t] = S::ident();
    __syncthreads();  // the ranks are complete, and the accumulators of an unmarked row

    // numeric: products at their column's rank
    enum { kFirst, kLater, kAll };
    const auto products = [&](auto which) {
      constexpr int W = decltype(which)::value;
      int step0 = 0;
      for (int64_t c0 = a0; c0 < a1; c0 += kQThreads) {
        if (a1 - a0 > kQThreads) {  // else the row's entries are still there
          __syncthreads();
          stage(c0);
          __syncthreads();
        }
        walk(c0, step0, [&](int step, int e0, int x, int most) {
          const unsigned m = W == kAll ? 0u : (unsigned)(later >> ((8 * step) & 63)) & 255u;
#pragma unroll
          for (int g = 0; g < 8; g += 4) {
            if (g && most <= 32) break;
            int c[4];
            TB v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const int e = e0 + u, y = x + 8 * g;
              c[u] = -1;
              if (y < s_len[e] && (W != kLater || ((m >> (g + u)) & 1u))) {
                const int64_t q = s_q[e] + y;
                c[u] = __ldg(B.col + q);
                v[u] = ldg_val(Bval + q);
              }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const unsigned d = (unsigned)c[u] - col_lo;
              if (c[u] < 0 || d >= width) continue;
              const int slot = (int)pre[d >> 5] + __popc(bits[d >> 5] << (~d & 31u)) - 1;
              if (!guard((unsigned)slot < (unsigned)n, 43, slot)) continue;
              const Acc y = S::mul(S::kUsesA ? s_a[e0 + u] : TA(), v[u]);
              if constexpr (W == kAll) cols[slot] = (unsigned short)d;
              if constexpr (W != kFirst) {
                S::atomic(&acc[slot], y);
              } else if (!((m >> (g + u)) & 1u)) {
                cols[slot] = (unsigned short)d;
                acc[slot] = started<SR>(y);
              } else {
                const int at = atomicAdd(&s_rep, 1);
                if (at < kQRepeats) {
                  rep_slot[at] = (unsigned short)slot;
                  rep_val[at] = y;
                }
              }
            }
          }
        });
      }
    };
    if (fits) {
      if (marked) products(std::integral_constant<int, kFirst>{});
      else products(std::integral_constant<int, kAll>{});
    }
    __syncthreads();
    for (int t = tid; t < n; t += kQThreads)
      if (chk(base + t < cap, 44, base + t)) st_out(Ccol + base + t, (int32_t)(col_lo + cols[t]));
    const int nrep = s_rep;  // (0 for an unmarked row)
    if (nrep > kQRepeats) {
      products(std::integral_constant<int, kLater>{});
    } else {
      for (int t = tid; t < nrep; t += kQThreads) S::atomic(&acc[rep_slot[t]], rep_val[t]);
    }
    if constexpr (!kInPlace || kQConvert<SR>) {
      __syncthreads();
      for (int t = tid; t < n; t += kQThreads) st_out(Cval + base + t, S::out(kInPlace ? __ldcg(acc + t) : acc[t]));
    }
    __syncthreads();
  }

  // the last CTA to finish records nnz(C), advances the epoch and resets
  // the queue (status words are cleared when the 24-bit epoch wraps)
  if (tid == 0) {
    __threadfence();
    s_last = atomicAdd(&sync[1], 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (s_last) {
    if (tid == 0) {
      __threadfence();
      unsigned long long* s64 = reinterpret_cast<unsigned long long*>(sync);
      s64[1] = m > 0 ? (unsigned long long)*reinterpret_cast<volatile int64_t*>(Crp + m) : 0ull;
    }
    const unsigned ne = (s_epoch + 1) & kQEpochMask;
    if (ne == 0)
      for (int64_t j = tid; j < tstat_cap; j += kQThreads) tstat[j] = 0;
    __syncthreads();
    if (tid == 0) {
      *queue = 0;
      sync[1] = 0;
      __threadfence();
      atomicExch(&sync[0], ne);
    }
  }
}

template <int SR>
cudaError_t launch_queue_sr(const DevCSR& A, const DevCSR& B, int64_t m, int64_t* Crp, int32_t* Ccol,
                            void* Cval, int64_t cap, unsigned long long* tstat, int64_t tstat_cap,
                            unsigned* sync, int* status, cudaStream_t s, int sms, unsigned spin_limit,
                            int64_t silent_row) {
  if (m > tstat_cap) return cudaErrorInvalidValue;
  static int per_sm = 0;  // resident CTAs per SM (same for every device of one kind)
  if (per_sm == 0) {
    const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_queue_rows<SR>, kQThreads, 0);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
  }
  const int64_t grid = std::min<int64_t>(m, (int64_t)per_sm * sms);
  k_queue_rows<SR><<<(unsigned)grid, kQThreads, 0, s>>>(A, B, m, Crp, Ccol,
                                                       static_cast<typename Sem<SR>::TC*>(Cval), cap,
                                                       tstat, tstat_cap, sync, status,
                                                       spin_limit < 1 ? 1u : spin_limit, silent_row);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_queue_rows(int sr, const DevCSR& A, const DevCSR& B, int64_t m, int64_t* Crp,
                              int32_t* Ccol, void* Cval, int64_t cap, unsigned long long* tstat,
                              int64_t tstat_cap, unsigned* sync, int* status, cudaStream_t s, int sms,
                              unsigned spin_limit, int64_t silent_row) {
  if (m <= 0) return cudaSuccess;
  switch (sr) {
#define CB_CASE(SRV) \
  case SRV: return launch_queue_sr<SRV>(A, B, m, Crp, Ccol, Cval, cap, tstat, tstat_cap, sync, status, s, sms, spin_limit, silent_row);
    CB_FOR_EACH_SEMIRING(CB_CASE)
#undef CB_CASE
  }
  return cudaErrorInvalidValue;
}

CB_CHECK_READER(queue)

}  // namespace cb
