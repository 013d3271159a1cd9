// Hash-bin rows: rows of at most 4096 products whose column range is wide.
//
// A row of C = A*B is the sum of the scaled rows A[i,k] * B[k,:] (Gustavson's
// algorithm, Sec. 5.1).  One thread team (one or more warps) owns the row (the
// shard pattern, Sec. 4) and keeps all its products in registers; shared
// memory holds the row's private workspace.
//
// Products.  The B rows of the row's stored A entries are laid end to end:
// product q belongs to the last entry that starts at or before q.  A bitmap
// marks the starts, so the owner of a product is a population count, every
// lane has a product whatever the lengths of the B rows, and the loads of all
// products of a lane are in flight together.
//
// Ranks (rank_row).  Every product column lies in [lo, hi].  The monotone
// hash
//     h(c) = floor((c - lo) * K / span),  span = hi - lo + 1
// (h(c) = c - lo when span <= K) sorts the products into K = cap buckets: a
// shared-memory counter per bucket gives every product its arrival number, a
// prefix sum over the counters gives the buckets' places, and the columns are
// staged there.  The buckets are in column order, so only the products of one
// bucket (less than one other on average) still have to be compared: a
// product's rank is the number of distinct columns before its bucket plus
// those below it inside.  A row with a bucket of more than `run_limit`
// products (a skewed column distribution) is sorted instead (bitonic, in the
// same shared memory).  This replaced an open-addressing table of (column,
// value) pairs that every product entered by compare-and-swap, a chain of
// dependent shared-memory operations per product.
//
// Symbolic pass: counts the distinct columns and stores every product's rank
// in the plan (uint16, bit 15 set when another product of the row comes first
// at its column).  Numeric pass: the first product of every column stores its
// column and value at its rank, the others add theirs (shared-memory atomics,
// the atomic level of Sec. 4), and the row leaves in order.  When the plan has
// no room for the ranks the numeric pass works them out again.
//
// Rows of at most 32 products (bin 0) hold one product per lane and compare
// it with the others by shuffles.
#include <climits>
#include <type_traits>

#include "ws_internal.cuh"

namespace wsk {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kDupBit = 0x8000;

// Shape of a bin: rows of at most kCap products, a team of W warps, kS
// products per thread.
template <int LOGC, int W>
struct Bin {
  static constexpr int kCap = 1 << LOGC;
  static constexpr int kNT = 32 * W;
  static constexpr int kS = kCap / kNT;
  static constexpr int kWords = kCap / 32;
  static_assert(kS >= 1 && kS * kNT == kCap, "whole products per thread");
  // Workspace of a team, in bytes.  `Work` holds in turn the entries (B
  // position and, in the numeric pass, A value), the bucket counters and the
  // staged columns (or the sort's keys, indices and ranks), and the staged row.
  static constexpr size_t kCountBytes = (static_cast<size_t>(kCap) + 8) * 2;  // counters and an end mark
  static_assert(kCountBytes % 16 == 0, "the staged columns start on a 16-byte boundary");
  static constexpr size_t kRankBytes =
      kCountBytes + 4 * static_cast<size_t>(kCap) > 8 * static_cast<size_t>(kCap) ? kCountBytes + 4 * static_cast<size_t>(kCap)
                                                                                  : 8 * static_cast<size_t>(kCap);
  static constexpr size_t kSymWork = kRankBytes;  // entries: 8 bytes per product at most
  static constexpr size_t num_work(size_t vs) {
    const size_t entries = (8 + vs) * static_cast<size_t>(kCap), row = (4 + vs) * static_cast<size_t>(kCap);
    const size_t m = entries > row ? entries : row;
    return m > kRankBytes ? m : kRankBytes;
  }
  static constexpr size_t kBits = 8 * static_cast<size_t>(kWords);  // start bits and their word prefixes
  static constexpr size_t bytes(size_t work) { return (work + kBits + 15) / 16 * 16; }
};

template <int W>
__device__ __forceinline__ void team_sync() {
  if constexpr (W == 1) {
    __syncwarp();
  } else {
    __syncthreads();
  }
}

// Exclusive sum over the team's threads; scratch holds 32 ints (W > 1).
template <int W>
__device__ __forceinline__ int team_scan(int x, int* scratch, int* total) {
  if constexpr (W == 1) {
    const int lane = threadIdx.x & 31;
    int incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(kFull, incl, o);
      if (lane >= o) incl += y;
    }
    *total = __shfl_sync(kFull, incl, 31);
    return incl - x;
  } else {
    return block_exclusive_scan(x, scratch, total);
  }
}

template <int W>
__device__ __forceinline__ bool team_any(bool x) {
  if constexpr (W == 1) {
    return __any_sync(kFull, x);
  } else {
    return __syncthreads_or(x);
  }
}

// pre[w] = set bits of the words before w; one warp of the team calls it.
template <int WORDS>
__device__ __forceinline__ void bit_prefix(const uint32_t* bits, int* pre, int lane) {
  constexpr int kPer = WORDS >= 32 ? WORDS / 32 : 1;
  int n[kPer], sum = 0;
#pragma unroll
  for (int j = 0; j < kPer; ++j) {
    const int w = lane * kPer + j;
    n[j] = w < WORDS ? __popc(bits[w]) : 0;
    sum += n[j];
  }
  int incl = sum;
#pragma unroll
  for (int o = 1; o < 32 && o * kPer < WORDS; o <<= 1) {
    const int y = __shfl_up_sync(kFull, incl, o);
    if (lane >= o) incl += y;
  }
  int at = incl - sum;
#pragma unroll
  for (int j = 0; j < kPer; ++j) {
    const int w = lane * kPer + j;
    if (w < WORDS) pre[w] = at;
    at += n[j];
  }
}

// One stored A entry: its B row and value.
template <typename T>
struct Entry {
  long long b0;
  int len;
  T a;
};

template <typename T, bool VALS>
__device__ __forceinline__ Entry<T> load_entry(const RowPlan<T>& p, int64_t at) {
  Entry<T> e;
  const int k = p.A.colidx[at];
  e.b0 = p.B.rowptr[k];
  const long long n = p.B.rowptr[k + 1] - e.b0;
  e.len = static_cast<int>(n < kMaxHashProducts + 1 ? n : kMaxHashProducts + 1);
  e.a = T(0);
  if constexpr (VALS) e.a = p.A.vals[at];
  return e;
}

// Lays the row's B rows end to end: entry idx (non-empty ones only) covers the
// products from the idx-th set start bit on, product q at B position
// q + delta[idx].  `first` is the entry of thread t (the first kNT entries).
// Returns the product count; *bad if it exceeds kCap (only if the input
// changed since the symbolic pass).
template <typename T, int LOGC, int W, bool VALS>
__device__ __forceinline__ int lay_entries(const RowPlan<T>& p, int64_t ra, int64_t na, const Entry<T>& first, int t,
                                           long long* delta, T* av, uint32_t* bits, int* pre, int* scratch, bool* bad) {
  using S = Bin<LOGC, W>;
  for (int i = t; i < S::kWords; i += S::kNT) bits[i] = 0u;
  team_sync<W>();
  constexpr int kCountShift = 21;  // lengths of a chunk (at most 256 * 4097) below, non-empty entries above
  int off0 = 0, idx0 = 0;
  Entry<T> e = first;
  for (int64_t c0 = 0; c0 < na && off0 <= S::kCap; c0 += S::kNT) {
    if (c0 > 0) {
      e.len = 0;
      if (c0 + t < na) e = load_entry<T, VALS>(p, ra + c0 + t);
    }
    int total;
    const int ex = team_scan<W>(e.len > 0 ? e.len + (1 << kCountShift) : 0, scratch, &total);
    const int off = off0 + (ex & ((1 << kCountShift) - 1));
    const int idx = idx0 + (ex >> kCountShift);
    if (e.len > 0 && off < S::kCap) {  // idx <= off
      delta[idx] = e.b0 - off;
      if constexpr (VALS) av[idx] = e.a;
      atomicOr(bits + (off >> 5), 1u << (off & 31));
    }
    off0 += total & ((1 << kCountShift) - 1);
    idx0 += total >> kCountShift;
  }
  if (off0 > S::kCap) {
    *bad = true;
    off0 = S::kCap;
  }
  team_sync<W>();
  if (W == 1 || t < 32) bit_prefix<S::kWords>(bits, pre, t & 31);
  team_sync<W>();
  return off0;
}

// Ranks of the row's products among its distinct columns: rk[s] = rank, with
// kDupBit set unless the product is the first at its column (products are
// q = s * kNT + t < ub, their columns col[s]).  Returns the number of distinct
// columns.  `work` (kRankBytes), `bits` and `pre` are free on entry; every
// thread of the team has read them before (the function starts with stores
// after a barrier).
template <int LOGC, int W>
__device__ __forceinline__ int rank_row(const int (&col)[Bin<LOGC, W>::kS], int ub, int lo, unsigned long long mul,
                                        int run_limit, int t, unsigned char* work, uint32_t* bits, int* pre, int* scratch,
                                        int (&rk)[Bin<LOGC, W>::kS], bool* sorted) {
  using S = Bin<LOGC, W>;
  constexpr int kS = S::kS, kNT = S::kNT, kCap = S::kCap;
  const int lane = threadIdx.x & 31;
  *sorted = false;
  team_sync<W>();
  if constexpr (kCap == 32) {
    // one product per lane
    const int c = col[0];
    const unsigned act = __ballot_sync(kFull, c >= 0);
    rk[0] = 0;
    const unsigned peers = __match_any_sync(kFull, c);
    const bool is_first = c >= 0 && lane == __ffs(peers) - 1;
    const unsigned firsts = __ballot_sync(kFull, is_first);
    const int key = is_first ? c : INT_MAX;
    int less = 0;
    const int n = __popc(act);  // the active lanes are 0..n-1
    for (int i = 0; i < n; ++i) less += __shfl_sync(kFull, key, i) < c;
    rk[0] = less | (is_first ? 0 : kDupBit);
    return __popc(firsts);
  } else {
    uint16_t* base = reinterpret_cast<uint16_t*>(work);         // bucket counters, then places; kCap + 1 used
    uint32_t* cnt = reinterpret_cast<uint32_t*>(work);          // two counters per word
    int* stage = reinterpret_cast<int*>(work + S::kCountBytes);
    static_assert(kS >= 2, "a thread owns whole words of the counters");
    constexpr int kOwn = kS / 2;
    for (int i = t; i < kCap / 2; i += kNT) cnt[i] = 0u;
    for (int i = t; i < S::kWords; i += kNT) bits[i] = 0u;
    team_sync<W>();
    uint32_t place[kS];  // bucket, arrival number in the high half
#pragma unroll
    for (int s = 0; s < kS; ++s) {
      place[s] = 0;
      if (col[s] >= 0) {
        const uint32_t d = static_cast<uint32_t>(col[s] - lo);
        uint32_t h = static_cast<uint32_t>((static_cast<unsigned long long>(d) * mul) >> 32);
        h = h < static_cast<uint32_t>(kCap) ? h : kCap - 1;  // only if the input changed
        const int sh = static_cast<int>(h & 1u) * 16;
        place[s] = h | (((atomicAdd(cnt + (h >> 1), 1u << sh) >> sh) & 0xffffu) << 16);
      }
    }
    team_sync<W>();
    // places of the buckets: thread t owns the words [t * kOwn, (t + 1) * kOwn)
    uint32_t own[kOwn];
    int sum = 0, most = 0;
#pragma unroll
    for (int j = 0; j < kOwn; ++j) {
      const uint32_t w = cnt[t * kOwn + j];
      const int a = static_cast<int>(w & 0xffffu), b = static_cast<int>(w >> 16);
      own[j] = static_cast<uint32_t>(sum) | (static_cast<uint32_t>(sum + a) << 16);
      sum += a + b;
      most = max(most, max(a, b));
    }
    int total;
    const uint32_t ex = static_cast<uint32_t>(team_scan<W>(sum, scratch, &total));
    most = __reduce_max_sync(kFull, most);  // the warp's fullest bucket
    if constexpr (W > 1) {
      if (lane == 0) scratch[t >> 5] = most;
      team_sync<W>();
#pragma unroll
      for (int w = 0; w < W; ++w) most = max(most, scratch[w]);
    }
    if (most <= run_limit && most <= kMaxHashBucket) {  // the second test is for the compiler: the loops below are short
#pragma unroll
      for (int j = 0; j < kOwn; ++j) cnt[t * kOwn + j] = own[j] + (ex | (ex << 16));
      if (t == 0) base[kCap] = static_cast<uint16_t>(ub);
      team_sync<W>();
      // place[s]: first place of the product's bucket (13 bits), the bucket's
      // products (6 bits; 0 for no product), the arrival number (6 bits)
#pragma unroll
      for (int s = 0; s < kS; ++s) {
        rk[s] = 0;
        if (col[s] >= 0) {
          const uint32_t h = place[s] & 0xffffu, arrival = place[s] >> 16;
          const uint32_t b = base[h], n = base[h + 1] - b;
          place[s] = b | (n << 13) | (arrival << 19);
          stage[b + arrival] = col[s];
        }
      }
      team_sync<W>();
      // Every product is compared with its bucket's, all products of a thread
      // side by side (a loop per product is a chain of shared-memory loads:
      // 483 us instead of 254 for 39,000 rows of 257-512 products).
      int dups = 0;
      if (most > 1) {
        for (int i = 0; i < most; ++i) {
#pragma unroll
          for (int s = 0; s < kS; ++s) {
            if (i < static_cast<int>((place[s] >> 13) & 63u)) {
              const int c = stage[(place[s] & 0x1fffu) + i];
              rk[s] += c < col[s];
              if (c == col[s] && i < static_cast<int>(place[s] >> 19)) rk[s] |= kDupBit;
            }
          }
        }
#pragma unroll
        for (int s = 0; s < kS; ++s) dups += (rk[s] & kDupBit) != 0;
      }
#pragma unroll
      for (int s = 0; s < kS; ++s) rk[s] += static_cast<int>(place[s] & 0x1fffu);
      int ndup;
      if constexpr (W == 1) {
        ndup = __reduce_add_sync(kFull, dups);
      } else {
        team_scan<W>(dups, scratch, &ndup);
      }
      if (ndup > 0) {
        // Ranks count distinct columns: mark the first products' places, drop
        // the others from the comparison.
#pragma unroll
        for (int s = 0; s < kS; ++s) {
          if (col[s] >= 0) {
            const int q = static_cast<int>((place[s] & 0x1fffu) + (place[s] >> 19));
            if (rk[s] & kDupBit) {
              stage[q] = INT_MAX;
            } else {
              atomicOr(bits + (q >> 5), 1u << (q & 31));
            }
          }
        }
        team_sync<W>();
        if (W == 1 || t < 32) bit_prefix<S::kWords>(bits, pre, lane);
        team_sync<W>();
#pragma unroll
        for (int s = 0; s < kS; ++s) {
          if (col[s] >= 0) {
            const int b = static_cast<int>(place[s] & 0x1fffu);
            rk[s] = (rk[s] & kDupBit) + pre[b >> 5] + __popc(bits[b >> 5] & ((1u << (b & 31)) - 1u));
          }
        }
        for (int i = 0; i < most; ++i) {
#pragma unroll
          for (int s = 0; s < kS; ++s) {
            if (i < static_cast<int>((place[s] >> 13) & 63u)) rk[s] += stage[(place[s] & 0x1fffu) + i] < col[s];
          }
        }
      }
      return ub - ndup;
    }
    // Skewed row: sort (column, product) pairs.
    *sorted = true;
    int* key = reinterpret_cast<int*>(work);
    uint16_t* idx = reinterpret_cast<uint16_t*>(work + 4 * static_cast<size_t>(kCap));
    uint16_t* rank = idx + kCap;
    team_sync<W>();
#pragma unroll
    for (int s = 0; s < kS; ++s) {
      const int q = s * kNT + t;
      key[q] = col[s] >= 0 ? col[s] : INT_MAX;
      idx[q] = static_cast<uint16_t>(q);
    }
    team_sync<W>();
    for (int k = 2; k <= kCap; k <<= 1) {
      for (int j = k >> 1; j > 0; j >>= 1) {
        for (int i = t; i < kCap / 2; i += kNT) {
          const int x = ((i & ~(j - 1)) << 1) | (i & (j - 1)), y = x | j;
          const int a = key[x], b = key[y];
          if ((a > b) == ((x & k) == 0) && a != b) {
            key[x] = b;
            key[y] = a;
            const uint16_t u = idx[x];
            idx[x] = idx[y];
            idx[y] = u;
          }
        }
        team_sync<W>();
      }
    }
    int firsts = 0;
#pragma unroll
    for (int s = 0; s < kS; ++s) {
      const int q = t * kS + s;
      firsts += q < ub && (q == 0 || key[q] != key[q - 1]);
    }
    int nnz;
    int at = team_scan<W>(firsts, scratch, &nnz) - 1;
#pragma unroll
    for (int s = 0; s < kS; ++s) {
      const int q = t * kS + s;
      const bool f = q < ub && (q == 0 || key[q] != key[q - 1]);
      at += f;
      if (q < ub) rank[idx[q]] = static_cast<uint16_t>(at | (f ? 0 : kDupBit));
    }
    team_sync<W>();
#pragma unroll
    for (int s = 0; s < kS; ++s) {
      const int q = s * kNT + t;
      rk[s] = q < ub ? rank[q] : 0;
    }
    return nnz;
  }
}

// RANKED (numeric pass): the ranks come from the plan; otherwise they are
// worked out in place.
template <typename T, int LOGC, int W, int RPC, bool NUMERIC, bool RANKED>
__global__ void __launch_bounds__(32 * W * RPC, NUMERIC ? (sizeof(T) == 8 ? 640 : 768) / (32 * W * RPC)
                                                        : 768 / (32 * W * RPC))
    hash_rows_kernel(const RowPlan<T> p) {
  using S = Bin<LOGC, W>;
  static_assert(W == 1 || RPC == 1, "multi-warp teams use the whole CTA");
  constexpr int kS = S::kS, kNT = S::kNT, kCap = S::kCap;
  constexpr bool kRanks = !NUMERIC || !RANKED;  // this pass works the ranks out
  constexpr size_t kWork = NUMERIC ? S::num_work(sizeof(T)) : S::kSymWork;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int scratch[32];
  __shared__ int s_firsts;
  const int sub = threadIdx.x / kNT, t = threadIdx.x % kNT;
  const int lane = threadIdx.x & 31;
  unsigned char* work = smem_raw + static_cast<size_t>(sub) * S::bytes(kWork);
  uint32_t* bits = reinterpret_cast<uint32_t*>(work + kWork);
  int* pre = reinterpret_cast<int*>(bits + S::kWords);
  long long* delta = reinterpret_cast<long long*>(work);
  T* av = reinterpret_cast<T*>(delta + kCap);
  const unsigned below_eq = 0xffffffffu >> (31 - lane);

  bool bad = false;
  const int64_t stride = static_cast<int64_t>(gridDim.x) * RPC;
  for (int64_t rb = static_cast<int64_t>(blockIdx.x) * RPC + sub; rb < p.seg_len; rb += 32 * stride) {
    // Headers of a batch of 32 rows: lane l of every warp of the team fetches
    // row rb + l * stride, so the chain perm -> row bounds is waited for once
    // per batch.
    int32_t b_row = 0;
    int b_lo = 0, b_cnt = 0;
    long long b_ra = 0, b_na = 0, b_cb = 0;
    unsigned long long b_mul = 0;
    if (rb + lane * stride < p.seg_len) {
      b_row = p.perm[p.seg_begin + rb + lane * stride];
      if constexpr (kRanks) {
        b_lo = p.lo[b_row];
        const uint32_t span = static_cast<uint32_t>(p.hi[b_row] - b_lo) + 1u;
        b_mul = span <= static_cast<uint32_t>(kCap) ? 1ull << 32 : (static_cast<unsigned long long>(kCap) << 32) / span;
      }
      b_ra = p.A.rowptr[b_row];
      b_na = p.A.rowptr[b_row + 1] - b_ra;
      if constexpr (NUMERIC) {
        b_cb = p.c_rowptr[b_row];
        const long long n = p.c_rowptr[b_row + 1] - b_cb;
        b_cnt = static_cast<int>(n < INT_MAX ? (n > 0 ? n : 0) : INT_MAX);  // a bad count fails the checks below
      }
    }
    const int64_t left = (p.seg_len - rb + stride - 1) / stride;
    const int nb = left < 32 ? static_cast<int>(left) : 32;
    // The first kNT stored A entries of a row are loaded while the row before
    // it is worked on: their columns first, their B rows after its products.
    auto entry_col = [&](int j) {
      const int64_t ra = __shfl_sync(kFull, b_ra, j), na = __shfl_sync(kFull, b_na, j);
      return t < na ? p.A.colidx[ra + t] : -1;
    };
    auto entry_row = [&](int k, int j) {
      Entry<T> e{0, 0, T(0)};
      const int64_t ra = __shfl_sync(kFull, b_ra, j);
      if (k >= 0) {
        e.b0 = p.B.rowptr[k];
        const long long n = p.B.rowptr[k + 1] - e.b0;
        e.len = static_cast<int>(n < kMaxHashProducts + 1 ? n : kMaxHashProducts + 1);
        if constexpr (NUMERIC) e.a = p.A.vals[ra + t];
      }
      return e;
    };
    Entry<T> next = entry_row(entry_col(0), 0);
    for (int jb = 0; jb < nb; ++jb) {
      const Entry<T> first = next;
      const int jn = jb + 1 < nb ? jb + 1 : jb;
      const int next_col = entry_col(jn);
      const int32_t row = __shfl_sync(kFull, b_row, jb);
      const int lo = __shfl_sync(kFull, b_lo, jb);
      const unsigned long long mul = __shfl_sync(kFull, b_mul, jb);
      const int64_t ra = __shfl_sync(kFull, b_ra, jb), na = __shfl_sync(kFull, b_na, jb);
      const int ub = lay_entries<T, LOGC, W, NUMERIC>(p, ra, na, first, t, delta, av, bits, pre, scratch, &bad);
      uint16_t* ranks = p.hash_ranks + (rb + jb * stride) * kCap;
      int col[kS], rk[kS];
      T val[NUMERIC ? kS : 1];
      // products: every load of the row is issued before the first use
#pragma unroll
      for (int s = 0; s < kS; ++s) {
        const int q = s * kNT + t;
        col[s] = -1;
        rk[s] = 0;
        if constexpr (NUMERIC) val[s] = T(0);
        if (q < ub) {
          const int w = q >> 5;
          const int i = pre[w] + __popc(bits[w] & below_eq) - 1;
          const long long at = delta[i] + q;
          col[s] = p.B.colidx[at];
          if constexpr (NUMERIC) val[s] = p.B.vals[at];
          if constexpr (NUMERIC && RANKED) rk[s] = ranks[q];
        }
      }
      next = entry_row(next_col, jn);
      if constexpr (NUMERIC) {
#pragma unroll
        for (int s = 0; s < kS; ++s) {
          const int q = s * kNT + t;
          if (q < ub) val[s] *= av[pre[q >> 5] + __popc(bits[q >> 5] & below_eq) - 1];
        }
      }
      if constexpr (!NUMERIC) {
        bool sorted;
        const int nnz = rank_row<LOGC, W>(col, ub, lo, mul, p.run_limit, t, work, bits, pre, scratch, rk, &sorted);
        if (p.hash_ranks) {
#pragma unroll
          for (int s = 0; s < kS; ++s) {
            if (s * kNT + t < ub) ranks[s * kNT + t] = static_cast<uint16_t>(rk[s]);
          }
        }
        if (t == 0) {
          p.c_rowptr[row + 1] = nnz;
          if (sorted) atomicAdd(&p.sum->n_sort, 1);
        }
        team_sync<W>();
      } else {
        if constexpr (!RANKED) {
          bool sorted;
          rank_row<LOGC, W>(col, ub, lo, mul, p.run_limit, t, work, bits, pre, scratch, rk, &sorted);
        }
        const int64_t cbase = __shfl_sync(kFull, b_cb, jb);
        const int want = __shfl_sync(kFull, b_cnt, jb);
        const int cnt = want < kCap ? want : kCap;  // staging bounds every access
        T* st_val = reinterpret_cast<T*>(work);
        int* st_col = reinterpret_cast<int*>(st_val + kCap);
        if (W > 1 && t == 0) s_firsts = 0;
        team_sync<W>();  // the entries have been read
        int firsts = 0;
        bool rest = false;
#pragma unroll
        for (int s = 0; s < kS; ++s) {
          if (col[s] >= 0) {
            if (rk[s] < cnt) {  // a first product (no kDupBit) in range
              st_col[rk[s]] = col[s];
              st_val[rk[s]] = val[s];
              ++firsts;
            } else {
              rest = true;
            }
          }
        }
        if (team_any<W>(rest)) {
          team_sync<W>();
#pragma unroll
          for (int s = 0; s < kS; ++s) {
            if (col[s] >= 0 && rk[s] >= cnt) {
              const int r = rk[s] & ~kDupBit;
              if ((rk[s] & kDupBit) && r < cnt) {
                atomicAdd(st_val + r, val[s]);
              } else {
                bad = true;
              }
            }
          }
        }
        firsts = __reduce_add_sync(kFull, firsts);
        if (W > 1 && lane == 0) atomicAdd(&s_firsts, firsts);
        team_sync<W>();
        if ((W > 1 ? s_firsts : firsts) != want) bad = true;
        for (int i = t; i < cnt; i += kNT) {
          p.c_colidx[cbase + i] = st_col[i];
          p.c_vals[cbase + i] = st_val[i];
        }
        team_sync<W>();
      }
    }
  }
  if (bad) atomicOr(p.status, kErrCount);
}

template <typename T, int LOGC, int W, int RPC, bool NUMERIC, bool RANKED>
void launch_pass(const RowPlan<T>& p, int num_sms, cudaStream_t s) {
  using S = Bin<LOGC, W>;
  constexpr size_t smem = RPC * S::bytes(NUMERIC ? S::num_work(sizeof(T)) : S::kSymWork);
  auto kern = hash_rows_kernel<T, LOGC, W, RPC, NUMERIC, RANKED>;
  static int per_sm = 0;
  if (per_sm == 0) {
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    int n = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, 32 * W * RPC, smem);
    per_sm = n > 0 ? n : 1;
  }
  int64_t grid = (p.seg_len + RPC - 1) / RPC;
  const int64_t cap = static_cast<int64_t>(num_sms) * per_sm;
  if (grid > cap) grid = cap;
  if (grid < 1) grid = 1;
  kern<<<static_cast<int>(grid), 32 * W * RPC, smem, s>>>(p);
}

// Teams: 16 products per thread in the numeric pass; in the symbolic pass 8 for
// rows of 257 to 1024 products (with 16 the kernel waits for instruction
// fetches: 254 against 186 us for 39,000 rows of 257-512 products), but 16 for
// the longer ones (8 or 16 warps that wait for one another: 125 against 120
// and 48 against 36 us).
template <typename T, int LOGC, int W, int RPC>
void launch_bin(const RowPlan<T>& p, bool numeric, int num_sms, cudaStream_t s) {
  if (!numeric) {
    constexpr int kW = LOGC == 9 || LOGC == 10 ? 2 * W : W;
    launch_pass<T, LOGC, kW, kW == 1 ? RPC : 1, false, false>(p, num_sms, s);
  } else if (p.hash_ranks) {
    launch_pass<T, LOGC, W, RPC, true, true>(p, num_sms, s);
  } else {
    launch_pass<T, LOGC, W, RPC, true, false>(p, num_sms, s);
  }
}

}  // namespace

template <typename T>
void launch_hash(const RowPlan<T>& p, int bin, bool numeric, int num_sms, cudaStream_t s, int* launches) {
  switch (bin) {
    case 0: launch_bin<T, 5, 1, 4>(p, numeric, num_sms, s); break;
    case 1: launch_bin<T, 6, 1, 4>(p, numeric, num_sms, s); break;
    case 2: launch_bin<T, 7, 1, 4>(p, numeric, num_sms, s); break;
    case 3: launch_bin<T, 8, 1, 4>(p, numeric, num_sms, s); break;
    case 4: launch_bin<T, 9, 1, 4>(p, numeric, num_sms, s); break;
    case 5: launch_bin<T, 10, 2, 1>(p, numeric, num_sms, s); break;
    case 6: launch_bin<T, 11, 4, 1>(p, numeric, num_sms, s); break;
    case 7: launch_bin<T, 12, 8, 1>(p, numeric, num_sms, s); break;
    default: return;
  }
  *launches += 1;
}

template void launch_hash<float>(const RowPlan<float>&, int, bool, int, cudaStream_t, int*);
template void launch_hash<double>(const RowPlan<double>&, int, bool, int, cudaStream_t, int*);

}  // namespace wsk
