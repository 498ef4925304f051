// Device-side building blocks shared by the SpGEMM kernels: semiring
// traits, the shared-memory hash probe, team synchronisation and the
// tier limits that the host dispatcher and the kernels agree on.
#pragma once

#include <cstdint>
#include <climits>
#include <type_traits>
#include <cuda_runtime.h>

#include "cb_kernels.h"

namespace cb {

// ---------------------------------------------------------------------------
// Semirings (paper Sec. 1: user-defined (+) and (x) over up to three value
// types, two for the inputs and one for the output).  A semiring is one
// specialisation of Sem<SR> with
//   TA, TB  value types of A's and B's CSR arrays, TC of C's;
//   A       accumulator type (shared memory or L2), with ident() the
//           (+)-identity, mul(TA, TB) -> A the (x), add and atomic the (+),
//           out(A) -> TC the conversion of a finished entry;
//   kUsesA  false when (x) ignores A's value (A's values are not read);
// plus one entry in CB_FOR_EACH_SEMIRING and the value sizes in cb_api.cu.
// Every (+) here is commutative and associative on A, so products may be
// combined in any order with atomics; for fp64 that changes rounding only.
// ---------------------------------------------------------------------------
#define CB_FOR_EACH_SEMIRING(X) X(1) X(2) X(3) X(4) X(5) X(6) X(7)

// ---------------------------------------------------------------------------
// Debug build (compiled with -DCB_CHECK, library libcb_check.so): the index
// of every CSR write and of every shared or global hash-table access is
// checked at run time.  A failed check records (code, index) in the check
// word of its translation unit (the first failure wins) and the access is
// skipped, so nothing is written out of bounds; the host reads the words
// after every call and fails it (CB_ERR_CUDA, "bounds check ...").  In the
// normal build chk() is constant true and guard() is the plain condition.
// ---------------------------------------------------------------------------
#ifdef CB_CHECK
constexpr bool kChecked = true;
#else
constexpr bool kChecked = false;
#endif

namespace {
__device__ unsigned long long g_check_word[2];  // (code, index), one per translation unit
}

__device__ __forceinline__ void check_record(int code, int64_t index) {
  if (atomicCAS(&g_check_word[0], 0ull, (unsigned long long)code) == 0ull)
    g_check_word[1] = (unsigned long long)index;
}

// A check that only the debug build makes: true in the normal build.
__device__ __forceinline__ bool chk(bool ok, int code, int64_t index) {
  if constexpr (kChecked) {
    if (!ok) check_record(code, index);
    return ok;
  } else {
    return true;
  }
}

// A bound every build keeps (the access is skipped when it fails); the
// debug build also records the failure.
__device__ __forceinline__ bool guard(bool ok, int code, int64_t index) {
  if constexpr (kChecked) {
    if (!ok) check_record(code, index);
  }
  return ok;
}

// Host side, one per translation unit that includes this header: reads and
// clears the unit's check word on stream s (synchronises).  Returns the
// code (0: no failure) and the index in *index.  Always 0 in the normal build.
#define CB_CHECK_READER(NAME)                                                              \
  int64_t check_take_##NAME(cudaStream_t s, int64_t* index) {                              \
    *index = 0;                                                                            \
    if constexpr (!kChecked) {                                                             \
      return 0;                                                                            \
    } else {                                                                               \
      unsigned long long w[2] = {0, 0};                                                    \
      if (cudaMemcpyFromSymbolAsync(w, g_check_word, sizeof w, 0, cudaMemcpyDeviceToHost,  \
                                    s) != cudaSuccess)                                     \
        return -1;                                                                         \
      const unsigned long long z[2] = {0, 0};                                              \
      if (cudaMemcpyToSymbolAsync(g_check_word, z, sizeof z, 0, cudaMemcpyHostToDevice,    \
                                  s) != cudaSuccess ||                                     \
          cudaStreamSynchronize(s) != cudaSuccess)                                         \
        return -1;                                                                         \
      *index = (int64_t)w[1];                                                              \
      return (int64_t)w[0];                                                                \
    }                                                                                      \
  }

template <int SR> struct Sem;

// Read-only cached load of a value of any semiring type: integer types
// directly; floating-point values and 8-byte records (cb_wlabel) as their
// bits (an unsigned word of the same size), so that every bit pattern, NaN
// payloads included, arrives unchanged (a float load through __ldg lost NaN
// weights of the heterogeneous semiring).
template <class T>
__device__ __forceinline__ T ldg_val(const T* p) {
  if constexpr (std::is_integral<T>::value) {
    return __ldg(p);
  } else {
    static_assert(sizeof(T) == 4 || sizeof(T) == 8, "values are 4 or 8 bytes");
    typedef typename std::conditional<sizeof(T) == 8, unsigned long long, unsigned>::type U;
    const U u = __ldg(reinterpret_cast<const U*>(p));
    T r;
    memcpy(&r, &u, sizeof r);
    return r;
  }
}

// Store of a value written once and not read again by the kernel (C's
// entries, stored bitmaps): with kStreamOut an evict-first store, so that the
// output streaming through L2 does not push out the operands being gathered.
constexpr bool kStreamOut = true;
template <class T>
__device__ __forceinline__ void st_out(T* p, T v) {
  if constexpr (!kStreamOut) {
    *p = v;
  } else if constexpr (sizeof(T) == 8) {
    unsigned long long u;
    memcpy(&u, &v, sizeof u);
    __stcs(reinterpret_cast<unsigned long long*>(p), u);
  } else if constexpr (sizeof(T) == 4) {
    unsigned u;
    memcpy(&u, &v, sizeof u);
    __stcs(reinterpret_cast<unsigned*>(p), u);
  } else {
    static_assert(sizeof(T) == 1, "values of 1, 4 or 8 bytes");
    unsigned char u;
    memcpy(&u, &v, sizeof u);
    __stcs(reinterpret_cast<unsigned char*>(p), u);
  }
}

template <> struct Sem<1> {  // (+,x) over int64, wrapping
  typedef int64_t TA, TB, TC;
  typedef unsigned long long A;
  static constexpr bool kUsesA = true;
  __device__ static __forceinline__ A ident() { return 0ull; }
  __device__ static __forceinline__ A mul(TA a, TB b) { return (A)a * (A)b; }
  __device__ static __forceinline__ A add(A x, A y) { return x + y; }
  __device__ static __forceinline__ void atomic(A* p, A v) { atomicAdd(p, v); }
  __device__ static __forceinline__ TC out(A x) { return (TC)x; }
};

template <> struct Sem<2> {  // (+,x) over fp64
  typedef double TA, TB, TC;
  typedef double A;
  static constexpr bool kUsesA = true;
  __device__ static __forceinline__ A ident() { return 0.0; }
  __device__ static __forceinline__ A mul(TA a, TB b) { return __dmul_rn(a, b); }
  __device__ static __forceinline__ A add(A x, A y) { return __dadd_rn(x, y); }
  __device__ static __forceinline__ void atomic(A* p, A v) { atomicAdd(p, v); }
  __device__ static __forceinline__ TC out(A x) { return x; }
};

template <> struct Sem<3> {  // (min,+) over uint32, + saturating at UINT32_MAX
  typedef uint32_t TA, TB, TC;
  typedef unsigned A;
  static constexpr bool kUsesA = true;
  __device__ static __forceinline__ A ident() { return 0xFFFFFFFFu; }
  __device__ static __forceinline__ A mul(TA a, TB b) {
    const unsigned room = ~a;  // what a + b may add without saturating
    return a + (b < room ? b : room);
  }
  __device__ static __forceinline__ A add(A x, A y) { return x < y ? x : y; }
  __device__ static __forceinline__ void atomic(A* p, A v) { atomicMin(p, v); }
  __device__ static __forceinline__ TC out(A x) { return x; }
};

template <> struct Sem<4> {  // (or,and) over bool (uint8 storage)
  typedef uint8_t TA, TB, TC;
  typedef unsigned A;
  static constexpr bool kUsesA = true;
  __device__ static __forceinline__ A ident() { return 0u; }
  __device__ static __forceinline__ A mul(TA a, TB b) { return (a != 0 && b != 0) ? 1u : 0u; }
  __device__ static __forceinline__ A add(A x, A y) { return x | y; }
  __device__ static __forceinline__ void atomic(A* p, A v) { if (v) atomicOr(p, v); }
  __device__ static __forceinline__ TC out(A x) { return x ? 1 : 0; }
};

template <> struct Sem<5> {  // (select2nd,min) over int32
  typedef int32_t TA, TB, TC;
  typedef int A;
  static constexpr bool kUsesA = false;
  __device__ static __forceinline__ A ident() { return INT_MAX; }
  __device__ static __forceinline__ A mul(TA, TB b) { return b; }
  __device__ static __forceinline__ A add(A x, A y) { return x < y ? x : y; }
  __device__ static __forceinline__ void atomic(A* p, A v) { atomicMin(p, v); }
  __device__ static __forceinline__ TC out(A x) { return x; }
};

// Heterogeneous (paper Sec. 1: three value types): A holds fp32 edge weights,
// B int32 labels, C (weight, label) pairs.  (x)(w, l) = (w, l); (+) keeps the
// pair with the larger weight in IEEE 754 totalOrder (-NaN < -inf < ... <
// -0 < +0 < ... < +inf < +NaN), and of equal weights the smaller label.  So
// C(i,j) is the label B(k,j) reached through the heaviest edge A(i,k).
// The accumulator packs both into one 64-bit key whose unsigned order is
// that order: high word = the weight's bits mapped monotonically (sign bit
// set: all bits flipped; clear: the sign bit flipped), low word =
// 0x7FFFFFFF - label (mod 2^32), which decreases with the label.
struct WLabel {
  float w;
  int32_t label;
};
template <> struct Sem<6> {
  typedef float TA;
  typedef int32_t TB;
  typedef WLabel TC;
  typedef unsigned long long A;
  static constexpr bool kUsesA = true;
  __device__ static __forceinline__ A ident() { return 0ull; }
  __device__ static __forceinline__ A mul(TA a, TB b) {
    const unsigned u = __float_as_uint(a);
    const unsigned hi = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
    const unsigned lo = 0x7FFFFFFFu - (unsigned)b;
    return ((A)hi << 32) | lo;
  }
  __device__ static __forceinline__ A add(A x, A y) { return x > y ? x : y; }
  __device__ static __forceinline__ void atomic(A* p, A v) { atomicMax(p, v); }
  __device__ static __forceinline__ TC out(A x) {
    const unsigned hi = (unsigned)(x >> 32), lo = (unsigned)x;
    TC r;
    r.w = __uint_as_float((hi & 0x80000000u) ? (hi & 0x7FFFFFFFu) : ~hi);
    r.label = (int32_t)(0x7FFFFFFFu - lo);
    return r;
  }
  // the accumulator of a finished entry (used by the merge form below)
  __device__ static __forceinline__ A in(TC v) { return mul(v.w, v.label); }
};

// Merge form of Sem<6> (internal, not an ABI semiring): the selector product
// that (+)-combines partial results of Sem<6> has B and C of Sem<6>'s C
// type; (x)(selector, c) = c and (+) is Sem<6>'s.
template <> struct Sem<7> {
  typedef uint8_t TA;
  typedef WLabel TB, TC;
  typedef unsigned long long A;
  static constexpr bool kUsesA = false;
  __device__ static __forceinline__ A ident() { return Sem<6>::ident(); }
  __device__ static __forceinline__ A mul(TA, TB b) { return Sem<6>::in(b); }
  __device__ static __forceinline__ A add(A x, A y) { return Sem<6>::add(x, y); }
  __device__ static __forceinline__ void atomic(A* p, A v) { Sem<6>::atomic(p, v); }
  __device__ static __forceinline__ TC out(A x) { return Sem<6>::out(x); }
};

// ---------------------------------------------------------------------------
// Tier limits.  Symbolic tiers are chosen by u_i = min(flops_i, ncols) (an
// upper bound of nnz(C_i)); numeric tiers by the exact nnz(C_i).
//   * u <= 512: counted with a shared-memory hash table (warp or 256-thread
//     team); u > 512: counted with a dense bitmap per span of kSpanCols
//     columns, which also cuts the row into rank windows (below).
//   * nnz <= 512: numeric in a shared-memory hash table + bitonic sort;
//     nnz > 512: numeric per rank window.  Every such row has u > 512, so its
//     windows exist.
// A rank window is a run of whole bitmap words of one span that fits the
// numeric kernel's shared memory (num_window_cut); inside it an output column's slot is
// its rank (popcount of the set bits before it), so a dense array of
// accumulators indexed by rank holds the window and reads out sorted.
// ---------------------------------------------------------------------------
constexpr int kEmptyKey = -1;

constexpr int kSymWarpMax = 128;     // warp team, table <= 256 slots
constexpr int kSymSmallMax = 512;    // 256-thread team, table <= 1024
constexpr int kSymHashMax = 512;     // default bound of the hash tiers (runtime-tunable)
constexpr int kSymLargeMax = 4096;   // largest bound the 512-thread hash tier supports
constexpr int kSpanCols = 1 << 18;   // columns per bitmap span
constexpr int kSpanWords = kSpanCols / 32;
constexpr int kMaxWindowsPerSpan = 64;

constexpr int kNumWarpMax = 64;      // warp team, table <= 128
constexpr int kNumSmallMax = 512;    // 256-thread team, table <= 1024
// Shared memory of a rank window with 4-byte accumulators: its bitmap words,
// their counts (6 bytes a word) and its accumulators (k_numeric.cu).
constexpr int kWinPool = 61440;
template <int SR> struct NumLimits {
  static constexpr int kHashMax = kNumSmallMax;  // default bound of the hash tiers
  // largest bound the large hash tier supports (512-thread team, table of 2x slots)
  static constexpr int kLargeMax = 4096;
  // entries per rank window
  static constexpr int kWcap = sizeof(typename Sem<SR>::A) == 8 ? 16384 : SR == 4 ? 32768 : kWinPool / 4;
  // learned sizing: rows predicted to hold at most this many entries skip the
  // symbolic phase and are computed in one pass in a hash table of
  // 2^ceil(log2(2 cap)) slots (1024-thread team at most)
  static constexpr int kLearnHashMax = kLargeMax;
  // rank windows of 8-byte accumulators reduce into a per-CTA slice in L2
  // instead of shared memory (measured faster for int64 and fp64; slower for
  // the 4-byte ones, whose shared-memory atomics are cheap)
  static constexpr bool kL2Acc = sizeof(typename Sem<SR>::A) == 8;
};

// One rank window of a heavy row: row index h into the heavy-row list, the
// span, the word range [w_lo, w_hi) inside the span, its entry count and the
// rank of its first entry within the span.
struct Window {
  int32_t h, span, w_lo, w_hi, count, rank;
};

// Popcounts of the WPT consecutive bitmap words first .. first + WPT - 1 of
// a shared-memory bitmap (first a multiple of WPT, bits 16-byte aligned),
// words at or past nw counted as 0.  A thread's words are consecutive, so a
// load of one word per thread would put a warp's lanes 4*WPT bytes apart on
// a few banks (a WPT-way bank conflict); 16-byte loads of 4 words each take
// a quarter of the shared-memory wavefronts.
template <int WPT>
__device__ __forceinline__ void popc_words(const unsigned* bits, int first, int nw, int (&c)[WPT]) {
  static_assert(WPT % 4 == 0, "whole 16-byte vectors per thread");
  const uint4* v = reinterpret_cast<const uint4*>(bits + first);
#pragma unroll
  for (int q = 0; q < WPT / 4; ++q) {
    const int w = first + 4 * q;
    const uint4 x = w < nw ? v[q] : make_uint4(0u, 0u, 0u, 0u);
    c[4 * q + 0] = __popc(x.x);
    c[4 * q + 1] = w + 1 < nw ? __popc(x.y) : 0;
    c[4 * q + 2] = w + 2 < nw ? __popc(x.z) : 0;
    c[4 * q + 3] = w + 3 < nw ? __popc(x.w) : 0;
  }
}

// The running counts before each of those words, as 16-bit values (a
// window holds fewer than 2^16 entries), stored 8 per 16-byte vector:
// pre[first + j] = run + c[0] + ... + c[j - 1].  Vectors wholly past nw are
// not stored; counts past nw inside a stored vector are never read.
template <int WPT>
__device__ __forceinline__ void store_counts(unsigned short* pre, int first, int nw, int run,
                                             const int (&c)[WPT]) {
  static_assert(WPT % 8 == 0, "whole 16-byte vectors per thread");
  uint4* v = reinterpret_cast<uint4*>(pre + first);
#pragma unroll
  for (int q = 0; q < WPT / 8; ++q) {
    unsigned p[4];
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      const unsigned lo16 = (unsigned)run & 0xFFFFu;
      run += c[8 * q + 2 * h];
      const unsigned hi16 = (unsigned)run & 0xFFFFu;
      run += c[8 * q + 2 * h + 1];
      p[h] = lo16 | (hi16 << 16);
    }
    if (first + 8 * q < nw) v[q] = make_uint4(p[0], p[1], p[2], p[3]);
  }
}

// The set bits of a column bitmap, read out in column order: word w covers
// columns 32w .. 32w + 31 of the range, pre[w] counts the set bits of the
// words before it, and emit(j, c) receives the j-th set bit overall (c its
// column offset in the range), every j once.  Two walks, picked by the
// average number of set bits per word:
//   * dense (at least DENSE per word, DENSE > 0): one word per warp step; lane
//     l takes bit l, at the word's offset plus the bits set below it, so the
//     entries of one store instruction are consecutive (one or two L2
//     requests for up to 32 entries);
//   * sparse: one word per thread, its bits in turn.  A lane's entries are
//     consecutive and the lanes' words start a few entries apart.
// Walking a dense bitmap a word per thread places the 32 lanes' entries of
// one store a word's count apart, one L2 request per entry.
// The dense walk pays for that only where the kernel is bound by its
// requests to L2 (rank windows reducing in L2: R-MAT s18 fp64 numeric 55.7 ->
// 54.5 ms); where shared-memory accumulators bound it, its extra
// instructions and broadcast loads cost as much as they save (u32 and bool
// numeric unchanged at a bound of 8, 2-4 ms slower at 4), so those kernels
// pass DENSE = 0.
#ifndef CB_DENSE_WORD_BITS
#define CB_DENSE_WORD_BITS 8
#endif
constexpr int kDenseWordBits = CB_DENSE_WORD_BITS;
template <int DENSE, int CTA, class F>
__device__ __forceinline__ void for_bitmap_columns(const unsigned* bits, const unsigned short* pre,
                                                   int nw, int cnt, F&& emit) {
  const int tid = threadIdx.x;
  if (DENSE > 0 && (int64_t)cnt >= (int64_t)DENSE * nw) {  // uniform over the CTA
    const int lane = tid & 31;
    const unsigned below = (1u << lane) - 1u;
    for (int w = tid >> 5; w < nw; w += CTA / 32) {
      const unsigned word = bits[w];
      if ((word >> lane) & 1u) emit((int)pre[w] + __popc(word & below), 32 * w + lane);
    }
  } else {
    for (int w = tid; w < nw; w += CTA) {
      unsigned word = bits[w];
      int j = pre[w];
      while (word) {
        const int b = __ffs(word) - 1;
        word &= word - 1;
        emit(j, 32 * w + b);
        ++j;
      }
    }
  }
}

// The columns of a window's cnt entries, col0 + offset, to out[0 .. lim)
// (lim <= cnt) through a shared buffer of cnt words: the bitmap is walked a word per
// thread into the buffer, and the buffer copied out coalesced.  All threads of
// the CTA call it, after a barrier.  (u32 numeric of R-MAT s18 35.6 -> 34.0 ms
// against one L2 request per entry.  Where no shared memory of that size is
// free, a smaller buffer filled part by part gained 1% in fp64 and lost 9% in
// (or,and): those windows use for_bitmap_columns.)
template <int CTA>
__device__ __forceinline__ void write_columns(const unsigned* bits, const unsigned short* pre, int nw, int cnt,
                                              int lim, int32_t col0, int32_t* buf, int32_t* out) {
  const int tid = threadIdx.x;
  for (int w = tid; w < nw; w += CTA) {
    unsigned word = bits[w];
    int j = pre[w];
    const int32_t c = col0 + 32 * w;
    while (word) {
      if (j < cnt) buf[j] = c + __ffs(word) - 1;
      word &= word - 1;
      ++j;
    }
  }
  __syncthreads();
#pragma unroll 4
  for (int t = tid; t < lim; t += CTA) st_out(out + t, buf[t]);
}

enum SymTier { kSymEmpty = 0, kSymWarp = 1, kSymSmall = 2, kSymLarge = 3, kSymHeavy = 4, kSymTiers = 5 };
enum NumTier { kNumEmpty = 0, kNumWarp = 1, kNumSmall = 2, kNumLarge = 3, kNumHeavy = 4, kNumTiers = 5 };

__device__ __forceinline__ int sym_tier(int64_t u, int64_t hash_max) {
  return u == 0 ? kSymEmpty : u <= kSymWarpMax ? kSymWarp : u <= kSymSmallMax ? kSymSmall
         : u <= hash_max ? kSymLarge : kSymHeavy;
}


// Smallest power of two >= x (x >= 1), as log2.
__host__ __device__ __forceinline__ int ceil_log2(int64_t x) {
  int l = 0;
  while ((int64_t(1) << l) < x) ++l;
  return l;
}

// Fibonacci hashing into a table of 2^bits slots (bits in [1, 31]).
__device__ __forceinline__ uint32_t hash_slot(int32_t c, int shift) {
  return ((uint32_t)c * 2654435769u) >> shift;
}

// Units of a persistent kernel, taken one after the other from a counter that
// starts at zero: thread 0 puts the CTA's next unit into the shared *slot.
// A barrier stands between the others' last read of the slot and this call,
// another between the call and their next read.
__device__ __forceinline__ void take_unit(int64_t* queue, long long* slot) {
  if (threadIdx.x == 0) *slot = (long long)atomicAdd((unsigned long long*)queue, 1ull);
}

// Find the slot of key c in an open-addressing (linear probing) table of
// mask+1 slots, inserting it if absent.  Returns the slot, or -1 if the
// table is full (never happens for tables sized >= 2x the row bound).
// `inserted` reports whether this call created the key.
__device__ __forceinline__ int probe_insert(int* keys, uint32_t mask, int shift, int c,
                                           bool& inserted) {
  uint32_t s = hash_slot(c, shift);
  inserted = false;
  for (uint32_t n = 0; n <= mask; ++n) {
    int k = *(volatile int*)&keys[s];
    if (k == c) return (int)s;
    if (k == kEmptyKey) {
      int old = atomicCAS(&keys[s], kEmptyKey, c);
      if (old == kEmptyKey) { inserted = true; return (int)s; }
      if (old == c) return (int)s;
    }
    s = (s + 1) & mask;
  }
  return -1;
}

template <int TEAM>
__device__ __forceinline__ void team_sync() {
  if (TEAM == 32) __syncwarp();
  else __syncthreads();
}

// Group size (lanes per stored A entry) for a row: the power of two nearest
// below the mean B-row length, clamped to [1, TEAM_MAX].
template <int TEAM_MAX>
__device__ __forceinline__ int group_log2(int64_t flops, int64_t nnz_a) {
  if (nnz_a <= 0) return 0;
  int64_t avg = flops / nnz_a;
  int g = 0;
  while (g < 5 && (int64_t(2) << g) <= avg) ++g;
  int lim = TEAM_MAX >= 32 ? 5 : ceil_log2(TEAM_MAX);
  return g < lim ? g : lim;
}

// End offset of row k of a (possibly windowed) operand.
__device__ __forceinline__ int64_t row_end(const DevCSR& M, int64_t k) {
  return M.rpe ? M.rpe[k] : M.rp[k + 1];
}

// Whether a validation queued before this kernel failed (uniform).
__device__ __forceinline__ bool gated(const int64_t* gate) {
  return gate && *reinterpret_cast<const volatile int64_t*>(gate) != 0;
}

// Output width of row i of A.B: A.rcols[i] when set (stacked batches, where
// each product keeps its own columns), else the width of B's view.
__device__ __forceinline__ int64_t row_width(const DevCSR& A, const DevCSR& B, int64_t i) {
  return A.rcols ? (int64_t)A.rcols[i] : B.ncols;
}

// Whether column c belongs to B's column window (always true unless filtering).
__device__ __forceinline__ bool in_window(const DevCSR& B, int c) {
  return !B.filter || (uint64_t)((int64_t)c - B.col_lo) < (uint64_t)B.ncols;
}

// Lane layout of a group of G = 2^gl lanes inside a warp (G <= 32).
struct Group {
  int G, gq, shift;
  unsigned mask;
  __device__ __forceinline__ Group(int gl, int thread) {
    G = 1 << gl;
    gq = thread & (G - 1);
    shift = (thread & 31) & ~(G - 1);
    mask = G == 32 ? 0xffffffffu : (((1u << G) - 1u) << shift);
  }
  // ballot of the group's lanes, as G low bits
  __device__ __forceinline__ unsigned ballot(bool pred) const {
    return (__ballot_sync(mask, pred) & mask) >> shift;
  }
};

// First index in the sorted run col[q0, q1) whose column is >= x, found
// cooperatively by a lane group: each round lane j probes the (j+1)-th of
// G+1 equal cut points, and the number of probes below x narrows the run by
// a factor of about G+1.  Every lane of the group must call it.
__device__ __forceinline__ int64_t group_lower_bound(const int32_t* col, int64_t q0, int64_t q1,
                                                     int64_t x, const Group& g) {
  int64_t lo = q0, hi = q1;  // the answer lies in [lo, hi]
  while (hi - lo > g.G) {
    const int64_t len = hi - lo;
    const int64_t pos = lo + (len * (g.gq + 1)) / (g.G + 1);
    const int t = __popc(g.ballot((int64_t)col[pos] < x));
    const int64_t nlo = t > 0 ? lo + (len * t) / (g.G + 1) + 1 : lo;
    const int64_t nhi = t < g.G ? lo + (len * (t + 1)) / (g.G + 1) : hi;
    lo = nlo;
    hi = nhi;
  }
  const int64_t pos = lo + g.gq;
  return lo + __popc(g.ballot(pos < hi && (int64_t)col[pos] < x));
}

// Visit every product A(i,p) * B(p,q) of row i whose column lies in
// [lo, hi) (absolute columns): f(p, q, c) is called by the lane that owns
// it.  Lanes form groups of 2^gl per stored A entry (a team of TEAM
// threads, `thread` in [0, TEAM)).  `whole` means every entry of B's rows
// lies in [lo, hi) (no filter); `sorted` means B's rows are non-decreasing
// in column, so each B row's slice in [lo, hi) is located by a group search
// and walked to its end; otherwise whole B rows are read and filtered.
// Uniform per team.
template <int TEAM, class F>
__device__ __forceinline__ void for_row_products(const DevCSR& A, const DevCSR& B, int64_t i,
                                                 int64_t lo, int64_t hi, bool whole, bool sorted,
                                                 int gl, int thread, F&& f) {
  const Group g(gl, thread);
  const int groups = TEAM >> gl;
  const int64_t a0 = A.rp[i], a1 = A.rp[i + 1];
  const unsigned width = (unsigned)(hi - lo);
  if (whole || !sorted) {
    for (int64_t p = a0 + (thread >> gl); p < a1; p += groups) {
      const int k = A.col[p];
      const int64_t q1 = row_end(B, k);
      for (int64_t q = B.rp[k] + g.gq; q < q1; q += g.G) {
        const int c = B.col[q];
        if (whole || (unsigned)((int64_t)c - lo) < width) f(p, q, c);
      }
    }
    return;
  }
  for (int64_t p = a0 + (thread >> gl); p < a1; p += groups) {
    const int k = A.col[p];
    const int64_t q1 = row_end(B, k);
    int64_t q = group_lower_bound(B.col, B.rp[k], q1, lo, g);
    while (true) {
      const int64_t qq = q + g.gq;
      const int c = qq < q1 ? B.col[qq] : INT_MAX;
      const bool in = (int64_t)c < hi;
      const int n = __popc(g.ballot(in));
      if (in) f(p, qq, c);
      if (n < g.G) break;
      q += g.G;
    }
  }
}

// Exclusive scan of one int per thread across a team of TEAM threads.
template <int TEAM>
__device__ __forceinline__ int team_exclusive_scan(int x, int* scratch /* >= 33 ints */, int& total) {
  const int lane = threadIdx.x & 31;
  int incl = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (TEAM == 32) {
    total = __shfl_sync(0xffffffffu, incl, 31);
    return incl - x;
  }
  const int w = threadIdx.x >> 5;
  constexpr int NW = TEAM / 32;
  if (lane == 31) scratch[w] = incl;
  __syncthreads();
  if (w == 0) {
    int v = lane < NW ? scratch[lane] : 0;
    int vi = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      int y = __shfl_up_sync(0xffffffffu, vi, o);
      if (lane >= o) vi += y;
    }
    if (lane < NW) scratch[lane] = vi - v;
    if (lane == NW - 1) scratch[32] = vi;
  }
  __syncthreads();
  total = scratch[32];
  const int r = scratch[w] + incl - x;
  __syncthreads();
  return r;
}

// Exclusive scan of one int or int64 per thread across a CTA (blockDim.x
// threads, a multiple of 32, at most 1024) with a single barrier: every warp
// scans the warps' totals itself.  scratch: 32 values, free again after the
// caller's next barrier.
template <class T>
__device__ __forceinline__ T cta_exclusive_scan(T x, T* scratch, T& total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int nw = blockDim.x >> 5;
  T incl = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const T y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) scratch[w] = incl;
  __syncthreads();
  T t = lane < nw ? scratch[lane] : T(0);
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const T y = __shfl_up_sync(0xffffffffu, t, o);
    if (lane >= o) t += y;
  }
  total = __shfl_sync(0xffffffffu, t, 31);
  const T before = __shfl_sync(0xffffffffu, t, (w + 31) & 31);  // the warps before this one
  return (w ? before : T(0)) + incl - x;
}

// First index in the sorted run col[q0, q1) whose column is >= x (one thread).
__device__ __forceinline__ int64_t seq_lower_bound(const int32_t* col, int64_t q0, int64_t q1,
                                                   int64_t x) {
  while (q0 < q1) {
    const int64_t mid = q0 + ((q1 - q0) >> 1);
    if ((int64_t)col[mid] < x) q0 = mid + 1;
    else q1 = mid;
  }
  return q0;
}

// The slice of B row k whose columns lie in [lo, hi): both ends searched at
// once, between the two boundaries of the split table around each (the whole
// row without a table).  B's rows are sorted; lo < col_lo + ncols.
__device__ __forceinline__ void row_slice(const DevCSR& B, const SplitTable& t, int64_t k, int64_t lo,
                                          int64_t hi, int64_t& s0, int64_t& s1) {
  const int64_t q0 = B.rp[k], q1 = row_end(B, k);
  int64_t a0 = q0, a1 = q1, b0 = q0, b1 = q1;
  if (t.pos) {
    const int32_t* p = t.pos + k * t.stride;
    const int64_t ga = (lo - B.col_lo) >> t.shift, gb = (hi - B.col_lo) >> t.shift;
    a0 = q0 + p[ga];
    a1 = q0 + p[ga + 1];
    if (gb < t.stride - 1) {
      b0 = q0 + p[gb];
      b1 = q0 + p[gb + 1];
    } else {
      b0 = q1;
    }
  }
  while (a0 < a1 || b0 < b1) {
    const int64_t am = a0 + ((a1 - a0) >> 1), bm = b0 + ((b1 - b0) >> 1);
    const bool ga = a0 < a1, gb = b0 < b1;
    const int32_t ca = ga ? __ldg(B.col + am) : 0, cb = gb ? __ldg(B.col + bm) : 0;
    if (ga) {
      if ((int64_t)ca < lo) a0 = am + 1;
      else a1 = am;
    }
    if (gb) {
      if ((int64_t)cb < hi) b0 = bm + 1;
      else b1 = bm;
    }
  }
  s0 = a0;
  s1 = b0;
}

// Marks a call of for_row_pieces that needs no values of A or B.
struct NoValue {};

// All products of row i whose columns lie in [lo, hi), for a whole CTA: the
// row's stored A entries are taken in chunks of blockDim.x; each entry's
// product range (its B row, or the B row's slice in [lo, hi) when `sorted` and
// not `whole`) is cut into pieces of 128 consecutive entries of B, the chunk's
// pieces are numbered by one CTA scan, and every warp takes an equal
// contiguous run of pieces.  Inside a piece the A entry is the same for the
// whole warp.
//   f(a, c, v):  one product: A's value (from Aval), column c and B's value
//                there (from Bval); of type NoValue they are not read.
// A's values come with the ranges, through shared memory: read by the warp that
// reaches a range they cost it a load's latency there.
// Lane l takes entries l, l + 32, l + 64, l + 96 of a piece: coalesced loads,
// all in flight before the callbacks, and neighbouring lanes meet neighbouring
// columns, whose accumulators often share an L2 sector (with four consecutive
// entries per lane, read in 16-byte loads, fp64 numeric took 55 instead of 46
// ms on R-MAT s18 and 21.7 instead of 14.9 on the block-clustered product).
// The loop is bound by the instructions it issues, so a range's pieces are
// walked in an inner loop on 32-bit offsets from its first entry.
// All threads of the CTA must call it; it ends with a barrier.
template <class T>  // A's value type, or NoValue
struct PieceSmem {
  static constexpr bool kA = !std::is_same<T, NoValue>::value;
  long long* q0;    // [blockDim.x] first B entry of the range
  T* a;             // [blockDim.x] A's value
  int* len;         // [blockDim.x] entries in the range
  int* poff;        // [blockDim.x] first piece of each nonempty range (chunk numbering)
  long long* scan;  // [32]
  static constexpr size_t kBytesPerThread = sizeof(long long) + 2 * sizeof(int) + (kA ? sizeof(T) < 4 ? 4 : sizeof(T) : 0);
  // carved from threads * kBytesPerThread bytes, 8-byte aligned
  __device__ PieceSmem(void* p, int threads, long long* scan_) : scan(scan_) {
    q0 = static_cast<long long*>(p);
    len = reinterpret_cast<int*>(q0 + threads);
    poff = len + threads;
    a = reinterpret_cast<T*>(poff + threads);
  }
};

template <class T, class V, class F>
__device__ __forceinline__ void for_row_pieces(const DevCSR& A, const DevCSR& B, const SplitTable& tab,
                                               int64_t i, int64_t lo, int64_t hi, bool whole, bool sorted,
                                               const PieceSmem<T>& sm, const T* Aval, const V* Bval, F&& f) {
  constexpr int P = 128;
  constexpr bool kVals = !std::is_same<V, NoValue>::value, kA = PieceSmem<T>::kA;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nthr = blockDim.x, nwarp = nthr >> 5;
  const int64_t a0 = A.rp[i], a1 = A.rp[i + 1];
  const bool filter = !whole && !sorted;
  const unsigned width = (unsigned)(hi - lo);
  const unsigned lo32 = (unsigned)lo;
  for (int64_t c0 = a0; c0 < a1; c0 += nthr) {
    const int nch = (int)min((int64_t)nthr, a1 - c0);
    int64_t q0 = 0, q1 = 0;
    T av{};
    if (tid < nch) {
      const int k = A.col[c0 + tid];
      if constexpr (kA) av = ldg_val(Aval + c0 + tid);
      if (!whole && sorted) {
        row_slice(B, tab, k, lo, hi, q0, q1);
      } else {
        q0 = B.rp[k];
        q1 = row_end(B, k);
      }
    }
    const long long np = q0 < q1 ? (q1 - q0 + P - 1) / P : 0;
    // one scan numbers the pieces (high bits) and the nonempty ranges (low 11 bits)
    long long packed_total;
    const long long packed = cta_exclusive_scan((np << 11) | (np > 0 ? 1 : 0), sm.scan, packed_total);
    const long long npieces = packed_total >> 11;
    const int ne = (int)(packed_total & 2047);
    if (npieces >= (1 << 24)) {  // 2^31 products or more: 32-bit offsets do not do; entry by entry
      for (int t = 0; t < nch; ++t) {
        if (tid == t) {
          sm.q0[0] = q0;
          sm.q0[1] = q1;
          if constexpr (kA) sm.a[0] = av;
        }
        __syncthreads();
        T tok{};
        if constexpr (kA) tok = sm.a[0];
        const int64_t end = sm.q0[1];
        for (int64_t q = sm.q0[0] + tid; q < end; q += nthr) {
          const int c = __ldg(B.col + q);
          V v{};
          if constexpr (kVals) v = ldg_val(Bval + q);
          if (!filter || (unsigned)c - lo32 < width) f(tok, c, v);
        }
        __syncthreads();
      }
      continue;
    }
    if (np > 0) {
      const int slot = (int)(packed & 2047);
      sm.poff[slot] = (int)(packed >> 11);
      if constexpr (kA) sm.a[slot] = av;
      sm.q0[slot] = q0;
      sm.len[slot] = (int)(q1 - q0);
    }
    __syncthreads();
    // equal runs of pieces per warp; nwarp is a power of two (512-thread
    // CTAs), so the split needs no 64-bit division
    const int lgw = 31 - __clz(nwarp);
    const int k_beg = (int)((npieces * warp) >> lgw), k_end = (int)((npieces * (warp + 1)) >> lgw);
    if (k_beg < k_end) {  // uniform over the warp
      int l = 0, r = ne - 1;  // range holding piece k_beg
      while (l < r) {
        const int mid = (l + r + 1) >> 1;
        if (sm.poff[mid] <= k_beg) l = mid;
        else r = mid - 1;
      }
      int s = (k_beg - sm.poff[l]) * P;  // first entry of the next piece
      for (int j = l, left = k_end - k_beg; left > 0; ++j, s = 0) {
        const int len = sm.len[j];
        const int32_t* cp = B.col + sm.q0[j] + lane;
        const V* vp = kVals ? Bval + sm.q0[j] + lane : nullptr;
        T tok{};
        if constexpr (kA) tok = sm.a[j];
        for (; left > 0 && s < len; --left, s += P) {
          int c[4];
          V v[4];
          if (s + P <= len && !filter) {  // a whole piece (uniform)
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              c[u] = __ldg(cp + s + 32 * u);
              if constexpr (kVals) v[u] = ldg_val(vp + s + 32 * u);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) f(tok, c[u], v[u]);
          } else {
            const int n = len - s - lane;  // the lane's entries: 32 * u < n
#pragma unroll
            for (int u = 0; u < 4; ++u)
              if (32 * u < n) {
                c[u] = __ldg(cp + s + 32 * u);
                if constexpr (kVals) v[u] = ldg_val(vp + s + 32 * u);
              }
#pragma unroll
            for (int u = 0; u < 4; ++u)
              if (32 * u < n && (!filter || (unsigned)c[u] - lo32 < width)) f(tok, c[u], v[u]);
          }
        }
      }
    }
    __syncthreads();
  }
}

}  // namespace cb
