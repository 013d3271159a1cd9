// Elementwise operations on CSR matrices of one shape (Sec. 5.2, "Sparse
// Linear Algebra": C = A op B with op in {+, elementwise product}):
//   SpAdd     C = A + B   pattern union, a sum of exactly 0.0 is kept;
//   Hadamard  C = A .* B  pattern intersection.
// Row i of C depends only on rows i of A and B, so distinct output positions
// go to distinct workers -- the sharded sparse list of Sec. 5.2 -- and no
// worker ever waits on another.
//
// Work units.  The two matrices are one sequence of items: for every row the
// merge of its two sorted column lists (an entry of A ahead of an equal entry
// of B), then a terminator.  Row r starts at item A.rowptr[r] + B.rowptr[r] + r,
// so the sequence is cut into tiles of kEwTileItems items without any per-row
// preparation, and neither long rows nor stretches of empty ones unbalance
// them.  A tile's first item is found by two binary searches (the row, then the
// split of its two lists); an equal pair is never cut.  A CTA copies its tile's
// two runs of columns into shared memory, and every entry finds its place in
// the other list by a binary search among the entries of its row there.
//
// Positions.  The entries of C before a point of the sequence are (A entries +
// B entries - pairs) for the union and (pairs) for the intersection, so only
// the equal pairs have to be counted: a bitmap over the tile's A entries marks
// those with an equal partner, and population counts give the pairs before any
// entry.
//
// Symbolic pass.  Tiles count their pairs and store C.rowptr as if no pair lay
// before the tile; a scan of the tiles' counts and a pass over the rows make
// that right.  Numeric pass.  Every entry (the B entry of a pair excepted)
// writes its column and value at its position; a tile's positions are one
// contiguous run of C.
//
// Measured on two R-MAT 2^20 graphs (16.3 million entries, fp64, A + B; 400 MB
// read and written by the numeric pass): 57 us for the count, 112 us for the
// numeric pass.  Bound by the instructions of the searches (55-63% of the issue
// slots) and their shared-memory latency.  The lane-per-chunk merges these
// kernels replaced took 65 and 171 us, plus 52 us for laying out the chunks;
// threads that merge 8 items each from the same tiles 68 and 204 us.  For rows
// of 256 merged entries (33 million, fp64) 121 and 281 us; the warp-per-chunk
// ranking of such rows took 134 and 292 us.
#include <climits>

#include "ws_internal.cuh"

namespace wsk {

namespace {

constexpr int kEwThreads = 256;
constexpr int kEwItems = 8;                        // entries per thread
constexpr int kSlots = kEwThreads * kEwItems;      // 2048
static_assert(kEwTileItems + 1 <= kSlots, "a tile, one item longer for an equal pair at its end, fits the CTA");

// Largest x in [lo, hi] with ok(x), given ok(lo) and that ok(x) stays false once
// it is; a 32-way search by one warp (every lane probes one point per level).
template <typename F>
__device__ __forceinline__ int64_t warp_last(int64_t lo, int64_t hi, int lane, F&& ok) {
  for (int level = 0; level < 16 && hi > lo; ++level) {
    const int64_t step = (hi - lo + 32) / 32;
    const int64_t x = lo + lane * step;
    const unsigned m = __ballot_sync(0xffffffffu, lane == 0 || (x <= hi && ok(x)));
    const int64_t end = lo + (32 - __clz(m)) * step - 1;
    lo += static_cast<int64_t>(31 - __clz(m)) * step;
    hi = hi < end ? hi : end;
  }
  return lo;
}

// First item of every tile, found by a warp: its row and positions in A's and
// B's arrays.  The tiles at and past the end of the sequence start at row m.
// (Binary searches by one thread per tile took 16 us: the chain
// of dependent loads is what counts.)
template <typename T>
__global__ void __launch_bounds__(kEwThreads) ew_tiles_kernel(const EwisePlan<T> p) {
  const int64_t* arp = p.A.rowptr;
  const int64_t* brp = p.B.rowptr;
  const int lane = threadIdx.x & 31;
  for (int64_t t = (static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5; t <= p.ntiles;
       t += (static_cast<int64_t>(gridDim.x) * blockDim.x) >> 5) {
    const int64_t d = t * kEwTileItems;
    // the last row that starts at or before item d
    const int64_t row = warp_last(0, p.m, lane, [&](int64_t r) { return arp[r] + brp[r] + r <= d; });
    const int64_t a0 = arp[row], b0 = brp[row];
    int64_t i = 0, j = 0;
    if (row < p.m) {
      // the first q merged positions of the row hold a[0..i) and b[0..q - i);
      // an equal pair at the cut goes to the tile before (j + 1)
      const int32_t* a = p.A.colidx + a0;
      const int32_t* b = p.B.colidx + b0;
      const int64_t na = arp[row + 1] - a0, nb = brp[row + 1] - b0, q = d - (a0 + b0 + row);
      i = warp_last(q - nb > 0 ? q - nb : 0, q < na ? q : na, lane, [&](int64_t x) { return q - x >= nb || a[x - 1] <= b[q - x]; });
      j = q - i;
      if (i > 0 && j < nb && a[i - 1] == b[j]) ++j;
    }
    if (lane == 0) {
      p.tile_row[t] = static_cast<int32_t>(row);
      p.tile_a[t] = a0 + i;
      p.tile_b[t] = b0 + j;
    }
  }
}

// A tile: local row k is row r0 + k (k = 0..terms; the last one has no
// terminator in this tile).
struct TileShape {
  int64_t ga, gb;  // first positions in A's and B's arrays
  int32_t r0;
  int na, nb, terms;
};

template <typename T>
__device__ __forceinline__ TileShape tile_shape(const EwisePlan<T>& p, int64_t t) {
  TileShape s;
  // A changed input could leave the stored starts outside the lists: clamp
  // them (the count check then reports the difference).
  const int64_t a_end = p.A.rowptr[p.m], b_end = p.B.rowptr[p.m];
  const int64_t a0 = p.tile_a[t], a1 = p.tile_a[t + 1], b0 = p.tile_b[t], b1 = p.tile_b[t + 1];
  s.ga = a0 < a_end ? a0 : a_end;
  s.gb = b0 < b_end ? b0 : b_end;
  // At most kEwTileItems + 1 items, whatever the arrays hold.
  auto some = [](int64_t n, int most) { return static_cast<int>(n < 0 ? 0 : (n < most ? n : most)); };
  s.na = some((a1 < a_end ? a1 : a_end) - s.ga, kEwTileItems + 1);
  s.nb = some((b1 < b_end ? b1 : b_end) - s.gb, kEwTileItems + 1 - s.na);
  s.r0 = p.tile_row[t];
  s.terms = some(p.tile_row[t + 1] - s.r0, kEwTileItems + 1 - s.na - s.nb);
  return s;
}

constexpr int kWords = kSlots / 32;  // 64: two words per lane of a warp

// Shared memory of a tile.  The A columns come first in col, the B columns from
// na on; an entry's position there is its tile position.
struct TileSmem {
  int32_t col[kSlots];
  uint32_t other[kSlots];  // at the first entry of a row's part of a list: the row's part of the other list
  uint32_t start[kWords];  // bit: a row's part of a list starts here
  int prev[kWords];        // last start before the word
  uint32_t pair[kWords];   // bit (A entries): has an equal partner
  int before[kWords];      // pairs before the word
  int pairs;
};

// Pairs among the tile's first i A entries.
__device__ __forceinline__ int pairs_before(const TileSmem& sm, int i) {
  return sm.before[i >> 5] + __popc(sm.pair[i >> 5] & ((1u << (i & 31)) - 1u));
}

// Position of entry e (column c, in word w) in the other list: the first entry
// of its row there with a column >= c, and whether that is c.
__device__ __forceinline__ int place(const TileSmem& sm, int w, int lane, int c, bool* equal) {
  const uint32_t m = sm.start[w] & (0xffffffffu >> (31 - lane));
  const int first = m ? (w << 5) + 31 - __clz(m) : sm.prev[w];
  const uint32_t seg = sm.other[first];
  int lo = min(static_cast<int>(seg & 0xffffu), kSlots);  // within col even for a broken row pointer
  const int end = min(static_cast<int>(seg >> 16), kSlots);
  int hi = end;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (sm.col[mid] < c) {
      lo = mid + 1;
    } else {
      hi = mid;
    }
  }
  *equal = lo < end && sm.col[lo] == c;
  return lo;
}

template <typename T, int OP, bool FILL>
__global__ void __launch_bounds__(kEwThreads, FILL ? 4 : 6) ew_tile_kernel(const EwisePlan<T> p) {
  __shared__ TileSmem sm;
  const int tid = static_cast<int>(threadIdx.x), lane = tid & 31, warp = tid >> 5;
  constexpr bool kVals = FILL && OP == kEwiseAdd;
  bool bad = false;
  for (int64_t t = blockIdx.x; t < p.ntiles; t += gridDim.x) {
    const TileShape s = tile_shape(p, t);
    const int n = s.na + s.nb;
    int c[kEwItems];
    T v[kVals ? kEwItems : 1];
#pragma unroll
    for (int u = 0; u < kEwItems; ++u) {
      const int e = u * kEwThreads + tid;
      c[u] = 0;
      if (e < n) {
        const bool a = e < s.na;
        c[u] = a ? p.A.colidx[s.ga + e] : p.B.colidx[s.gb + (e - s.na)];
        if constexpr (kVals) v[u] = a ? p.A.vals[s.ga + e] : p.B.vals[s.gb + (e - s.na)];
      }
    }
    if (tid < kWords) sm.start[tid] = 0u;
    __syncthreads();
    // Rows: where their parts start, and what the other list holds of them.
    auto local = [](int64_t x, int most) { return static_cast<int>(x < 0 ? 0 : (x < most ? x : most)); };
    for (int k = tid; k <= s.terms; k += kEwThreads) {
      const int64_t* ar = p.A.rowptr + s.r0 + k;
      const int64_t* br = p.B.rowptr + s.r0 + k;
      const int a0 = k == 0 ? 0 : local(ar[0] - s.ga, s.na), a1 = k == s.terms ? s.na : local(ar[1] - s.ga, s.na);
      const int b0 = s.na + (k == 0 ? 0 : local(br[0] - s.gb, s.nb)), b1 = s.na + (k == s.terms ? s.nb : local(br[1] - s.gb, s.nb));
      if (a0 < a1) {
        sm.other[a0] = static_cast<uint32_t>(b0) | (static_cast<uint32_t>(b1) << 16);
        atomicOr(&sm.start[a0 >> 5], 1u << (a0 & 31));
      }
      if (b0 < b1) {
        sm.other[b0] = static_cast<uint32_t>(a0) | (static_cast<uint32_t>(a1) << 16);
        atomicOr(&sm.start[b0 >> 5], 1u << (b0 & 31));
      }
    }
#pragma unroll
    for (int u = 0; u < kEwItems; ++u) sm.col[u * kEwThreads + tid] = c[u];
    __syncthreads();
    if (warp == 0) {
      const uint32_t w0 = sm.start[2 * lane], w1 = sm.start[2 * lane + 1];
      const int l0 = w0 ? (lane << 6) + 31 - __clz(w0) : 0;
      int last = w1 ? (lane << 6) + 63 - __clz(w1) : l0;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, last, o);
        if (lane >= o) last = max(last, y);
      }
      int excl = __shfl_up_sync(0xffffffffu, last, 1);
      if (lane == 0) excl = 0;
      sm.prev[2 * lane] = excl;
      sm.prev[2 * lane + 1] = max(excl, l0);
    }
    __syncthreads();
    // A entries: place among B's, equal pairs.
    int at[kEwItems];
    uint32_t eq = 0;  // bit u: entry u has an equal partner
#pragma unroll
    for (int u = 0; u < kEwItems; ++u) {
      const int e = u * kEwThreads + tid, w = u * (kEwThreads / 32) + warp;
      at[u] = 0;
      bool equal = false;
      if (e < s.na) at[u] = place(sm, w, lane, c[u], &equal);
      eq |= static_cast<uint32_t>(equal) << u;
      const uint32_t m = __ballot_sync(0xffffffffu, equal);
      if (lane == 0) sm.pair[w] = m;
      // columns increase inside a row's part of a list
      if constexpr (!FILL) bad |= e < n && e > 0 && !((sm.start[w] >> lane) & 1u) && sm.col[e - 1] >= c[u];
    }
    __syncthreads();
    if (warp == 0) {
      const int n0 = __popc(sm.pair[2 * lane]), n1 = __popc(sm.pair[2 * lane + 1]);
      int incl = n0 + n1;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      sm.before[2 * lane] = incl - n0 - n1;
      sm.before[2 * lane + 1] = incl - n1;
      if (lane == 31) sm.pairs = incl;
    }
    __syncthreads();
    if constexpr (!FILL) {
      if (tid == 0) p.tile_off[t + 1] = sm.pairs;
      for (int k = tid; k < s.terms; k += kEwThreads) {
        const int64_t ar = p.A.rowptr[s.r0 + k + 1], br = p.B.rowptr[s.r0 + k + 1];
        const int np = pairs_before(sm, local(ar - s.ga, s.na));
        p.c_rowptr[s.r0 + k + 1] = OP == kEwiseAdd ? ar + br - np : np;
      }
    } else {
      const int64_t p0 = p.tile_off[t], p1 = p.tile_off[t + 1];
      const int64_t out0 = OP == kEwiseAdd ? s.ga + s.gb - p0 : p0;
      const int64_t want = OP == kEwiseAdd ? n - (p1 - p0) : p1 - p0;
      bad |= sm.pairs != p1 - p0;
#pragma unroll
      for (int u = 0; u < kEwItems; ++u) {
        const int e = u * kEwThreads + tid, w = u * (kEwThreads / 32) + warp;
        int rank = -1;
        T x = T(0);
        if constexpr (OP == kEwiseAdd) {
          if (e < s.na) {
            rank = e + (at[u] - s.na) - pairs_before(sm, e);
            x = v[u];
            if ((eq >> u) & 1u) x += p.B.vals[s.gb + (at[u] - s.na)];
          } else if (e < n) {
            bool equal;
            const int i = place(sm, w, lane, c[u], &equal);
            if (!equal) rank = i + (e - s.na) - pairs_before(sm, i);
            x = v[u];
          }
        } else if ((eq >> u) & 1u) {
          rank = pairs_before(sm, e);
          x = p.A.vals[s.ga + e] * p.B.vals[s.gb + (at[u] - s.na)];
        }
        if (rank >= 0) {
          if (rank < want) {
            p.c_colidx[out0 + rank] = c[u];
            p.c_vals[out0 + rank] = x;
          } else {
            bad = true;
          }
        }
      }
    }
    __syncthreads();
  }
  if (bad) atomicOr(p.status, kErrCount);
}

// C.rowptr with the pairs of the tiles before each row's terminator; nnz for
// the host.
template <typename T, int OP>
__global__ void __launch_bounds__(kEwThreads) ew_rowptr_kernel(const EwisePlan<T> p) {
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i <= p.m;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    if (i == 0) {
      p.c_rowptr[0] = 0;
      continue;
    }
    const int64_t item = p.A.rowptr[i] + p.B.rowptr[i] + i - 1;  // the terminator of row i - 1
    int64_t t = item / kEwTileItems;
    t = t < p.ntiles ? t : p.ntiles - 1;
    const int64_t x = p.c_rowptr[i] + (OP == kEwiseAdd ? -p.tile_off[t] : p.tile_off[t]);
    p.c_rowptr[i] = x;
    if (i == p.m) *const_cast<volatile long long*>(&p.host->nnz) = x;
  }
}

int grid_for(int64_t work, int per_block, int num_sms, int per_sm) {
  const int64_t want = (work + per_block - 1) / per_block;
  const int64_t cap = static_cast<int64_t>(num_sms) * per_sm;
  return static_cast<int>(want < 1 ? 1 : (want > cap ? cap : want));
}

template <typename T, int OP>
void symbolic_op(const EwisePlan<T>& p, int num_sms, cudaStream_t s, int* launches) {
  ew_tiles_kernel<T><<<grid_for(p.ntiles + 1, kEwThreads / 32, num_sms, 8), kEwThreads, 0, s>>>(p);
  ew_tile_kernel<T, OP, false><<<grid_for(p.ntiles, 1, num_sms, 1 << 20), kEwThreads, 0, s>>>(p);
  launch_scan(p.tile_off, p.ntiles, p.partials, p.sum, s, launches);
  ew_rowptr_kernel<T, OP><<<grid_for(p.m + 1, kEwThreads, num_sms, 8), kEwThreads, 0, s>>>(p);
  *launches += 3;
}

template <typename T, int OP>
void numeric_op(const EwisePlan<T>& p, int num_sms, cudaStream_t s, int* launches) {
  ew_tile_kernel<T, OP, true><<<grid_for(p.ntiles, 1, num_sms, 1 << 20), kEwThreads, 0, s>>>(p);
  *launches += 1;
}

}  // namespace

template <typename T>
void launch_ewise_symbolic(const EwisePlan<T>& p, int num_sms, cudaStream_t s, int* launches) {
  if (p.op == kEwiseAdd) {
    symbolic_op<T, kEwiseAdd>(p, num_sms, s, launches);
  } else {
    symbolic_op<T, kEwiseMul>(p, num_sms, s, launches);
  }
}

template <typename T>
void launch_ewise_numeric(const EwisePlan<T>& p, int num_sms, cudaStream_t s, int* launches) {
  if (p.op == kEwiseAdd) {
    numeric_op<T, kEwiseAdd>(p, num_sms, s, launches);
  } else {
    numeric_op<T, kEwiseMul>(p, num_sms, s, launches);
  }
}

template void launch_ewise_symbolic<float>(const EwisePlan<float>&, int, cudaStream_t, int*);
template void launch_ewise_symbolic<double>(const EwisePlan<double>&, int, cudaStream_t, int*);
template void launch_ewise_numeric<float>(const EwisePlan<float>&, int, cudaStream_t, int*);
template void launch_ewise_numeric<double>(const EwisePlan<double>&, int, cudaStream_t, int*);

}  // namespace wsk
