// Plan-phase and scan kernels: CSR validation, the per-row product count, the
// class histogram scan, the class scatter that groups rows by work, and the row-offset
// scan of C after the symbolic pass.
//
// The count is the number of partial products Algorithm 1 forms for row i (Sec. III-A):
// P_i = sum over the stored columns k of row i of A of nnz(row k of B), i.e. only the B
// rows named by row i are "streamed" (Sec. III-A, selective streaming of B rows).
// Grouping rows by P_i on the device plays the role of the CPU-side scheduling of RIR
// bundles (Sec. II, "RIR includes scheduling"; Sec. III-A, long rows split into bundles):
// every row class gets a kernel shaped for its size.
#include "kernels.h"

namespace spg {

namespace {

// Row pointers of rows [r0, r0 + n1 - 1) of a CSR matrix, rebased to start at 0 (int64).
__global__ void k_rowptr_rebase(const void* __restrict__ in, int idx64, int64_t r0, int64_t n1, int64_t base,
                                int64_t* __restrict__ out) {
  for (int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; t < n1; t += int64_t(gridDim.x) * blockDim.x) {
    const int64_t v = idx64 ? static_cast<const int64_t*>(in)[r0 + t] : static_cast<const int32_t*>(in)[r0 + t];
    out[t] = v - base;
  }
}

// Small reads of device state: a grid of SMs stores the words into mapped page-locked host
// memory, so the read never queues on the copy engine behind bulk copies to the host.
__global__ void k_fetch(const uint32_t* __restrict__ src, uint32_t* __restrict__ dst, int64_t words) {
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < words; i += int64_t(gridDim.x) * blockDim.x)
    dst[i] = src[i];
}

__global__ void k_rowptr_to64(const int32_t* __restrict__ in, int64_t* __restrict__ out, int64_t n1) {
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n1;
       i += int64_t(gridDim.x) * blockDim.x)
    out[i] = in[i];
}

// Row pointer i of a CSR matrix as its caller stores them.
__device__ __forceinline__ int64_t rowptr_at(const void* rp, int rp64, int64_t i) {
  return rp64 ? static_cast<const int64_t*>(rp)[i] : static_cast<const int32_t*>(rp)[i];
}

// First row r in [0, rows] with rp[r] >= x (rows + 1 pointers, non-decreasing; of others the result is
// still a row): a warp narrows the range 32 times a step.
__device__ __forceinline__ int64_t warp_first_row(const void* rp, int rp64, int64_t rows, int64_t x) {
  const int lane = threadIdx.x & 31;
  int64_t lo = 0, n = rows + 1;   // the answer is in [lo, lo + n]
  while (n > 0) {
    const int64_t step = (n + 31) / 32;
    const int64_t at = lo + step * (lane + 1) - 1;
    const bool below = step * (lane + 1) - 1 < n && rowptr_at(rp, rp64, at) < x;
    const int full = __popc(__ballot_sync(0xffffffffu, below));   // probes below x (a prefix of the lanes)
    lo += step * full;
    const int64_t rest = n - step * full;
    n = rest >= step ? step - 1 : (rest > 0 ? rest : 0);   // the next probe, if there was one, is not below x
  }
  return lo < rows ? lo : rows;
}

// Canonical-CSR check: row pointers from 0 to nnz, non-decreasing; columns strictly increasing in
// [0, cols) within each row. Any violation sets kErrInvalidCsr. A block takes kCheckEntries consecutive
// entries at a time: it marks the rows that start among them in a bitmap in shared memory and compares
// every entry with the one before it unless it starts a row. A block's entries are consecutive, so it
// searches the row pointers once, for its first row. The rows' own checks, and the copy of the row
// pointers as int64 (rp_out, may be null), are spread over the grid.
//
// Most of the rows that start among 2,048 entries are empty where there are many of them, and there may be
// millions. A block looks at kCheckRowSteps rows per thread at most; past those it searches the row pointers
// for the entries that are not above their predecessor, all of a thread's in step (few beside a run of
// empty rows, half of them where rows of one entry lie among empty ones). A product with 10^7 empty rows of B
// beside 10^5 entries takes 0.19 ms; 14.8 ms when a block walked its empty rows.
//
// Bound by the latency of the search and of the first loads. It replaces a bitmap of the row starts in
// global memory, set by a kernel over the rows and read by one over the entries, after the conversion
// of the row pointers: 1024^2 five-point stencil (5.2e6 entries, 1.05e6 rows), three kernels of 31 us
// -> 24 us (cold caches).
constexpr int kCheckEntries = 2048;
constexpr int kCheckBlocks = 6;   // per SM
constexpr int kCheckRowSteps = 16;
__global__ void __launch_bounds__(256, kCheckBlocks) k_validate(const void* __restrict__ rp, int rp64, int64_t rows,
                                                                int64_t cols, int64_t nnz,
                                                                const int32_t* __restrict__ col, int64_t share,
                                                                int64_t* __restrict__ rp_out, uint32_t* err) {
  constexpr int kPer = kCheckEntries / 256;
  __shared__ uint32_t starts[kCheckEntries / 32];
  __shared__ int64_t s_row, s_next;
  __shared__ int s_found;
  const int lane = threadIdx.x & 31;
  const int64_t first = blockIdx.x * share;
  const int64_t last = first + share < nnz ? first + share : nnz;
  bool bad = false;
  // entries and, per warp, the one before its first
  int32_t c[kPer], p[kPer];
  auto load = [&](int64_t j0) {
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      const int64_t j = j0 + u * 256 + threadIdx.x;
      c[u] = j < last ? col[j] : 0;
      p[u] = lane == 0 && j < last && j > 0 ? col[j - 1] : -1;
    }
  };
  load(first);   // in flight while the rows are found
  if (threadIdx.x < kCheckEntries / 32) starts[threadIdx.x] = 0u;
  if (threadIdx.x < 32 && first < last) {
    const int64_t r = warp_first_row(rp, rp64, rows, first);
    if (lane == 0) {
      s_row = r;
      s_found = 0;
    }
  }
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i <= rows; i += int64_t(gridDim.x) * blockDim.x) {
    const int64_t s = rowptr_at(rp, rp64, i);
    if (rp_out) rp_out[i] = s;
    if (i == 0 && s != 0) bad = true;
    if (i == rows) {
      if (s != nnz) bad = true;
    } else {
      const int64_t e = rowptr_at(rp, rp64, i + 1);
      if (s < 0 || e < s || e > nnz) bad = true;
    }
  }
  __syncthreads();
  for (int64_t j0 = first; j0 < last; j0 += kCheckEntries) {
    // the rows that start among these entries (their pointers do not decrease; of others, some rows)
    const int64_t row = s_row;
    int found = 0;
    {
      int64_t r = row + threadIdx.x;
      for (; found < kCheckRowSteps && r < rows; r += blockDim.x) {
        const int64_t at = rowptr_at(rp, rp64, r) - j0;
        if (at >= kCheckEntries) break;
        if (at >= 0) atomicOr(&starts[at >> 5], 1u << (at & 31));
        ++found;
      }
    }
    const bool many = __syncthreads_or(found == kCheckRowSteps) != 0;   // perhaps more rows than were looked at
    int64_t next = 0;   // many: the first row past these entries
    if (many) {
      if (threadIdx.x < 32) {
        const int64_t r = warp_first_row(rp, rp64, rows, j0 + kCheckEntries);
        if (lane == 0) s_next = r < row ? row : r;   // (before `row` only if the pointers decrease)
      }
      __syncthreads();
      next = s_next;
    } else {
      found = warp_sum(found);
      if (lane == 0 && found) atomicAdd(&s_found, found);
    }
    unsigned low = 0;   // many: the thread's entries that are not above their predecessor
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      const int q = u * 256 + threadIdx.x;
      int32_t prev = __shfl_up_sync(0xffffffffu, c[u], 1);
      if (lane == 0) prev = p[u];
      if (j0 + q < last) {
        const bool start = (starts[q >> 5] >> lane) & 1u;
        bad |= c[u] < 0 || c[u] >= cols || (!many && !start && prev >= c[u]);
        if (many && !start && prev >= c[u]) low |= 1u << u;
      }
    }
    if (many && __any_sync(0xffffffffu, low != 0u)) {
      // rows of [row, next) that start before each of them, then whether the one after does with it
      const uint32_t range = static_cast<uint32_t>(next - row);   // (rows: below 2^31)
      uint32_t step = 1;
      while (2 * step <= range) step *= 2;
      uint32_t before[kPer];
#pragma unroll
      for (int u = 0; u < kPer; ++u) before[u] = 0;
      for (; step > 0; step >>= 1) {
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
          const uint32_t at = before[u] + step;
          if ((low >> u & 1u) && at <= range && rowptr_at(rp, rp64, row + at - 1) < j0 + u * 256 + threadIdx.x) before[u] = at;
        }
      }
#pragma unroll
      for (int u = 0; u < kPer; ++u)
        if (low >> u & 1u) bad |= rowptr_at(rp, rp64, row + before[u]) != j0 + u * 256 + threadIdx.x;
    }
    load(j0 + kCheckEntries);
    __syncthreads();
    if (threadIdx.x < kCheckEntries / 32) starts[threadIdx.x] = 0u;
    if (threadIdx.x == 0) {
      s_row = many ? next : row + s_found;
      s_found = 0;
    }
    __syncthreads();
  }
  if (__any_sync(0xffffffffu, bad) && lane == 0) set_error(err, kErrInvalidCsr);
}

// Warp-aggregated increment of a shared counter per class; returns this lane's slot.
__device__ __forceinline__ int32_t aggregated_slot(int32_t* counters, int cls, bool valid) {
  const unsigned lane = lane_id();
  const unsigned peers = __match_any_sync(0xffffffffu, valid ? cls : 1000 + static_cast<int>(lane));
  const int leader = __ffs(peers) - 1;
  const int rank = __popc(peers & ((1u << lane) - 1u));
  int32_t base = 0;
  if (valid && static_cast<int>(lane) == leader) base = atomicAdd(&counters[cls], __popc(peers));
  base = __shfl_sync(0xffffffffu, base, leader);
  return base + rank;
}

// Rows of a tile per thread of the kernels of 256 threads below: row r * 256 + threadIdx.x. The loads of all
// of them are under way before the first is ranked, and the tile's rows are ranked at once (2^20 rows,
// with a ranking of its own, and three barriers, for every 256 rows: k_scatter_num 19 us, now 16,
// k_scatter_sym 11, now 9).
constexpr int kRowsPer = kTileRows / 256;
constexpr int kGroups = kTileRows / 32;   // of 32 consecutive rows
static_assert(kGroups == 32, "a lane per group");

// Places of a tile's rows within their classes, in row order, from base[class]: neighbouring rows of a class
// stay neighbours in the permutation (the merge kernel writes a warp's rows as one run). cls < 0: no row.
// cnt: a counter per group and class. Contains __syncthreads.
__device__ __forceinline__ void ordered_slots(const int32_t* base, int32_t (*cnt)[kMaxClasses],
                                              const int (&cls)[kRowsPer], int32_t (&pos)[kRowsPer]) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int r = 0; r < kRowsPer; ++r) {
    int32_t* mine = cnt[r * 8 + wid];
    if (lane < kMaxClasses) mine[lane] = 0;
    __syncwarp();
    pos[r] = 0;
    for (unsigned todo = __ballot_sync(0xffffffffu, cls[r] >= 0); todo;) {
      const int lc = __shfl_sync(0xffffffffu, cls[r], __ffs(todo) - 1);
      const unsigned same = __ballot_sync(0xffffffffu, cls[r] == lc);
      if (cls[r] == lc) pos[r] = __popc(same & ((1u << lane) - 1u));
      if (lane == 0) mine[lc] = __popc(same);
      todo &= ~same;
    }
  }
  __syncthreads();
  for (int c = wid; c < kMaxClasses; c += 8) {
    const int32_t v = cnt[lane][c];
    cnt[lane][c] = base[c] + warp_incl_scan(v) - v;
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < kRowsPer; ++r)
    if (cls[r] >= 0) pos[r] += cnt[r * 8 + wid][cls[r]];
}

// Rows with more entries than this are counted by the whole block of k_count.
constexpr int64_t kCountBlockNa = 2048;

// Row `row` of A as [a0, a0 + na) clamped to the stored entries, so that an input that has not yet been
// rejected cannot send a read outside A's arrays.
__device__ __forceinline__ void clamp_row(int64_t nnz, int64_t s, int64_t e, int64_t& a0, int64_t& na) {
  s = s < 0 ? 0 : (s > nnz ? nnz : s);
  e = e < s ? s : (e > nnz ? nnz : e);
  a0 = s;
  na = e - s;
}
__device__ __forceinline__ void clamped_row(const DevCsr& A, int64_t row, int64_t& a0, int64_t& na) {
  clamp_row(A.nnz, A.rp[row], A.rp[row + 1], a0, na);
}

// P_i of every row, one row per thread; rows with more than 64 entries are left to the block's warps,
// one row at a time, rows with more than kCountBlockNa to the whole block. A block's warps take runs of
// `run` rows (32, fewer when the matrix has too few rows to fill the SMs with such blocks; a power of
// two) from distant parts of the matrix, so that neighbouring long rows (the first rows of an R-MAT
// matrix) are counted by different blocks. Class counts, sums and maxima of P_i go to the tiles'
// (zeroed) histograms, one atomic per warp and class.
//
// The pass reads every column of A, so it also checks that A is canonical (check; the rules of
// k_validate): C = A*A, whose B is the same matrix, needs no pass of its own for that. Both inputs' row
// pointers are read as the caller stores them, and A's are copied as int64 (a64, may be null) for the
// passes that follow. Conversions, checks and count together (C = A*A, stage times): 1024^2 five-point
// stencil 131 -> 57 us, R-MAT 2^17 367 -> 204 us (bound by the blocks with the longest rows), R-MAT
// 2^19 595 -> 478 us; 30,000^2 uniform (A and B apart) 145 -> 89 us.
__global__ void __launch_bounds__(256) k_count(CsrArrays A, CsrArrays B, int run, int check, int64_t* a64,
                                               ClassParams cp, int64_t* P, int32_t* nnz_row, int32_t* tile_hist,
                                               int64_t* tile_sum, int64_t* tile_max, uint32_t* err) {
  __shared__ int32_t s_nlong, s_nblock;
  __shared__ int64_t s_long[256], s_block[256];   // rows left to a warp, to the block
  __shared__ long long s_red[8];
  if (threadIdx.x == 0) { s_nlong = 0; s_nblock = 0; }
  __syncthreads();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t ntiles = (A.rows + kTileRows - 1) / kTileRows;
  bool bad = false;
  // an entry's share of P_i; an invalid column counts nothing (the counts of an invalid input are
  // meaningless, but every access stays inside the arrays)
  auto share = [&](int32_t k) -> int64_t {
    if (k < 0 || k >= B.rows) return 0;
    return rowptr_at(B.rp, B.rp64, k + int64_t(1)) - rowptr_at(B.rp, B.rp64, k);
  };
  // the warp's part of a long row: 128 consecutive entries from `first` on, every `step` entries, the
  // loads of four groups of 32 in flight together
  auto long_part = [&](int64_t a0, int64_t na, int64_t first, int64_t step) {
    long long acc = 0;
    for (int64_t j0 = first; j0 < na; j0 += step) {
      int32_t k[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) k[u] = j0 + 32 * u + lane < na ? A.col[a0 + j0 + 32 * u + lane] : 0x7fffffff;
      int32_t before = lane == 0 && j0 > 0 ? A.col[a0 + j0 - 1] : -1;   // lane 0: the entry before the group
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        int32_t prev = __shfl_up_sync(0xffffffffu, k[u], 1);
        if (lane == 0) prev = before;
        before = __shfl_sync(0xffffffffu, k[u], 31);
        if (j0 + 32 * u + lane < na) {
          bad |= k[u] <= prev || k[u] >= A.cols;
          acc += share(k[u]);
        }
      }
    }
    return warp_sum(acc);
  };
  auto row_range = [&](int64_t row, int64_t& a0, int64_t& na) {
    clamp_row(A.nnz, rowptr_at(A.rp, A.rp64, row), rowptr_at(A.rp, A.rp64, row + 1), a0, na);
  };
  // one long row's count, by one thread
  auto settle = [&](int64_t row, int64_t na, long long p) {
    const int cls = sym_class(p, na > 0x7fffffff ? 0x7fffffff : static_cast<int32_t>(na), row_params(cp, row));
    P[row] = p;
    if (cls == kSymZero) nnz_row[row] = 0;
    const int64_t t = row / kTileRows;
    atomicAdd(&tile_hist[cls * ntiles + t], 1);
    atomicAdd(reinterpret_cast<unsigned long long*>(&tile_sum[t]), static_cast<unsigned long long>(p));
    if (tile_max) atomicMax(reinterpret_cast<unsigned long long*>(&tile_max[t]), static_cast<unsigned long long>(p));
  };
  const int64_t row0 = (wid * int64_t(gridDim.x) + blockIdx.x) * run;
  if (row0 < A.rows) {
    const int64_t row = row0 + lane;
    const bool valid = lane < run && row < A.rows;
    int64_t a0 = 0, na = 0;
    if (valid) {
      const int64_t s = rowptr_at(A.rp, A.rp64, row), e = rowptr_at(A.rp, A.rp64, row + 1);
      if (s < 0 || e < s || e > A.nnz || (row == 0 && s != 0) || (row == A.rows - 1 && e != A.nnz)) bad = true;
      if (a64) {
        a64[row] = s;
        if (row == A.rows - 1) a64[A.rows] = e;
      }
      clamp_row(A.nnz, s, e, a0, na);
    }
    const bool mine = valid && na <= 64;
    if (valid && !mine) {
      if (na > kCountBlockNa) s_block[atomicAdd(&s_nblock, 1)] = row;
      else s_long[atomicAdd(&s_nlong, 1)] = row;
    }
    int64_t p = 0;
    int cls = kSymZero;
    if (mine) {
      int32_t prev = -1;
#pragma unroll 4
      for (int64_t j = 0; j < na; ++j) {
        const int32_t k = A.col[a0 + j];
        bad |= k <= prev || k >= A.cols;
        prev = k;
        p += share(k);
      }
      cls = sym_class(p, static_cast<int32_t>(na), row_params(cp, row));
      P[row] = p;
      if (cls == kSymZero) nnz_row[row] = 0;
    }
    // the warp's rows lie in one tile: one atomic per class among them (a stencil has one)
    const int64_t t = row0 / kTileRows;
    unsigned todo = __ballot_sync(0xffffffffu, mine);
    while (todo) {
      const int lc = __shfl_sync(0xffffffffu, cls, __ffs(todo) - 1);
      const unsigned same = __ballot_sync(0xffffffffu, mine && cls == lc);
      if (lane == 0) atomicAdd(&tile_hist[lc * ntiles + t], __popc(same));
      todo &= ~same;
    }
    const unsigned long long sum = warp_sum(static_cast<unsigned long long>(p));
    const unsigned long long most = ~warp_min(~static_cast<unsigned long long>(p));
    if (lane == 0 && sum > 0) {
      atomicAdd(reinterpret_cast<unsigned long long*>(&tile_sum[t]), sum);
      if (tile_max) atomicMax(reinterpret_cast<unsigned long long*>(&tile_max[t]), most);
    }
  }
  __syncthreads();
  for (int d = wid; d < s_nlong; d += 8) {
    int64_t a0, na;
    row_range(s_long[d], a0, na);
    const long long p = long_part(a0, na, 0, 128);
    if (lane == 0) settle(s_long[d], na, p);
  }
  for (int d = 0; d < s_nblock; ++d) {
    int64_t a0, na;
    row_range(s_block[d], a0, na);
    const long long acc = long_part(a0, na, 128 * wid, 1024);
    if (lane == 0) s_red[wid] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
      long long p = 0;
      for (int w = 0; w < 8; ++w) p += s_red[w];
      settle(s_block[d], na, p);
    }
    __syncthreads();
  }
  if (check && __any_sync(0xffffffffu, bad) && lane == 0) set_error(err, kErrInvalidCsr);
}

// Tile histograms are stored class by class: class c's count of tile t at c * ntiles + t.
//
// Block c < nclasses turns class c's per-tile counts into offsets within the class (in place) and writes
// the class's rows to the summary; the block after them scans the per-tile sums. The scatter kernels
// and the host add the classes before a class up from its rows. Bound by latency: one block for
// everything, a warp per class, took 18 us for 1,024 tiles, this 4.
constexpr int kScanThreads = 1024;
template <typename T, typename Ld, typename St>
__device__ __forceinline__ T scan_tiles(int64_t ntiles, T* scratch, Ld&& ld, St&& st) {
  T run = 0;
  T v = threadIdx.x < ntiles ? ld(threadIdx.x) : T(0);
  for (int64_t t0 = 0; t0 < ntiles; t0 += kScanThreads) {
    const int64_t t = t0 + threadIdx.x, after = t + kScanThreads;
    const T ahead = after < ntiles ? ld(after) : T(0);
    T total;
    const T at = run + block_excl_scan<T>(v, scratch, &total);
    if (t < ntiles) st(t, at);
    run += total;
    v = ahead;
  }
  return run;
}

__global__ void __launch_bounds__(kScanThreads) k_class_scan(int64_t ntiles, int nclasses, int32_t* tile_hist,
                                                             const int64_t* tile_sum, const int64_t* tile_max,
                                                             int64_t* tile_sum_off, Summary* summary) {
  __shared__ int32_t s_scan[33];
  __shared__ int64_t s_scan64[33];
  const int c = blockIdx.x;
  if (c < nclasses) {
    int32_t* hist = tile_hist + c * ntiles;
    const int32_t rows = scan_tiles<int32_t>(ntiles, s_scan, [&](int64_t t) { return hist[t]; },
                                             [&](int64_t t, int32_t at) { hist[t] = at; });   // rows: below 2^31
    if (threadIdx.x == 0) summary->class_rows[c] = rows;
    return;
  }
  if (threadIdx.x >= nclasses && threadIdx.x < kMaxClasses) summary->class_rows[threadIdx.x] = 0;
  const int64_t total = scan_tiles<int64_t>(ntiles, s_scan64, [&](int64_t t) { return tile_sum[t]; },
                                            [&](int64_t t, int64_t at) {
                                              if (tile_sum_off) tile_sum_off[t] = at;
                                            });
  int64_t mx = 0;
  if (tile_max) {
    for (int64_t t = threadIdx.x; t < ntiles; t += kScanThreads) mx = mx > tile_max[t] ? mx : tile_max[t];
    mx = ~warp_min(~mx);
    if ((threadIdx.x & 31) == 0) s_scan64[threadIdx.x >> 5] = mx;
    __syncthreads();
    if (threadIdx.x < 32) mx = ~warp_min(~s_scan64[threadIdx.x]);
  }
  if (threadIdx.x == 0) {
    summary->total = total;
    summary->max_row = mx;
  }
}

// base[c]: where tile t's rows of class c go (all threads of the block call it; ends with a barrier).
__device__ __forceinline__ void class_bases(const int32_t* tile_hist, int64_t ntiles, int64_t t,
                                            const Summary* summary, int32_t* base) {
  if (threadIdx.x < 32) {
    const int c = threadIdx.x;
    const int32_t rows = c < kMaxClasses ? static_cast<int32_t>(summary->class_rows[c]) : 0;
    const int32_t before = warp_incl_scan(rows) - rows;
    if (c < kMaxClasses) base[c] = before + tile_hist[c * ntiles + t];
  }
  __syncthreads();
}

__global__ void __launch_bounds__(256) k_scatter_sym(DevCsr A, ClassParams cp, const int64_t* P,
                                                     const int32_t* tile_hist, const Summary* summary,
                                                     int32_t* perm) {
  __shared__ int32_t base[kMaxClasses];
  __shared__ int32_t s_cnt[kGroups][kMaxClasses];
  const int64_t t = blockIdx.x;
  int cls[kRowsPer];
#pragma unroll
  for (int r = 0; r < kRowsPer; ++r) {
    const int64_t row = t * kTileRows + r * 256 + threadIdx.x;
    cls[r] = -1;
    if (row < A.rows) {
      int64_t a0, na;
      clamped_row(A, row, a0, na);   // the same row length k_count classified (before validation's verdict)
      cls[r] = sym_class(P[row], na > 0x7fffffff ? 0x7fffffff : static_cast<int32_t>(na), row_params(cp, row));
    }
  }
  class_bases(tile_hist, gridDim.x, t, summary, base);
  int32_t pos[kRowsPer];
  ordered_slots(base, s_cnt, cls, pos);
#pragma unroll
  for (int r = 0; r < kRowsPer; ++r)
    if (cls[r] >= 0) perm[pos[r]] = static_cast<int32_t>(t * kTileRows + r * 256 + threadIdx.x);
}

__global__ void __launch_bounds__(256) k_num_tiles(DevCsr A, ClassParams cp, const int64_t* P,
                                                   const int32_t* nnz_row, int32_t* tile_hist,
                                                   int64_t* tile_sum, unsigned long long* cls_sums) {
  __shared__ int32_t hist[kMaxClasses];
  __shared__ unsigned long long s_sum;
  __shared__ unsigned long long s_cls[kMaxClasses][3];
  if (threadIdx.x < kMaxClasses) hist[threadIdx.x] = 0;
  if (threadIdx.x < kMaxClasses * 3) (&s_cls[0][0])[threadIdx.x] = 0;
  if (threadIdx.x == 0) s_sum = 0;
  __syncthreads();
  const int64_t t = blockIdx.x;
  unsigned long long my = 0;
  for (int r = 0; r < kTileRows / 256; ++r) {
    const int64_t row = t * kTileRows + r * 256 + threadIdx.x;
    const bool valid = row < A.rows;
    int cls = 0;
    unsigned long long vp = 0, vn = 0, vz = 0;
    if (valid) {
      const int64_t na = A.rp[row + 1] - A.rp[row];
      const int32_t z = nnz_row[row];
      cls = num_class(P[row], na > 0x7fffffff ? 0x7fffffff : static_cast<int32_t>(na), z, cp);
      my += static_cast<unsigned long long>(z);
      vp = static_cast<unsigned long long>(P[row]);
      vn = static_cast<unsigned long long>(na);
      vz = static_cast<unsigned long long>(z);
    }
    // per-class sums: one warp reduction per distinct class of the warp (a stencil has one), so
    // the shared counters see one atomic per class and warp instead of one per row
    unsigned todo = __ballot_sync(0xffffffffu, valid);
    while (todo) {
      const int lc = __shfl_sync(0xffffffffu, cls, __ffs(todo) - 1);
      const bool mine = valid && cls == lc;
      const unsigned long long sp = warp_sum(mine ? vp : 0ull);
      const unsigned long long sn = warp_sum(mine ? vn : 0ull);
      const unsigned long long sz = warp_sum(mine ? vz : 0ull);
      if ((threadIdx.x & 31) == 0) {
        atomicAdd(&s_cls[lc][0], sp);
        atomicAdd(&s_cls[lc][1], sn);
        atomicAdd(&s_cls[lc][2], sz);
      }
      todo &= ~__ballot_sync(0xffffffffu, mine);
    }
    aggregated_slot(hist, cls, valid);
  }
  my = warp_sum(my);
  if ((threadIdx.x & 31) == 0) atomicAdd(&s_sum, my);
  __syncthreads();
  if (threadIdx.x < kMaxClasses) tile_hist[threadIdx.x * int64_t(gridDim.x) + t] = hist[threadIdx.x];
  if (threadIdx.x == 0) tile_sum[t] = static_cast<int64_t>(s_sum);
  if (threadIdx.x < kMaxClasses * 3) {
    const unsigned long long v = (&s_cls[0][0])[threadIdx.x];
    if (v) atomicAdd(&cls_sums[threadIdx.x], v);
  }
}

// Row offsets of C (exclusive scan of nnz(C_i), int64) and the numeric class scatter.
__global__ void __launch_bounds__(256) k_scatter_num(DevCsr A, ClassParams cp, const int64_t* P,
                                                     const int32_t* nnz_row, const int32_t* tile_hist,
                                                     const int64_t* tile_sum_off, const Summary* summary,
                                                     int32_t* perm, int64_t* c_off) {
  __shared__ int32_t base[kMaxClasses];
  __shared__ int32_t s_cnt[kGroups][kMaxClasses];
  __shared__ int64_t s_z[kGroups];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t t = blockIdx.x;
  int cls[kRowsPer];
  int32_t z[kRowsPer];
#pragma unroll
  for (int r = 0; r < kRowsPer; ++r) {
    const int64_t row = t * kTileRows + r * 256 + threadIdx.x;
    cls[r] = -1;
    z[r] = 0;
    if (row < A.rows) {
      const int64_t na = A.rp[row + 1] - A.rp[row];
      z[r] = nnz_row[row];
      cls[r] = num_class(P[row], na > 0x7fffffff ? 0x7fffffff : static_cast<int32_t>(na), z[r], cp);
    }
  }
  const int64_t carry = tile_sum_off[t];
  int64_t incl[kRowsPer];
#pragma unroll
  for (int r = 0; r < kRowsPer; ++r) {
    incl[r] = warp_incl_scan(static_cast<int64_t>(z[r]));
    if (lane == 31) s_z[r * 8 + wid] = incl[r];
  }
  class_bases(tile_hist, gridDim.x, t, summary, base);   // (ends with a barrier)
  const int64_t group = s_z[lane], before = warp_incl_scan(group) - group;
#pragma unroll
  for (int r = 0; r < kRowsPer; ++r) {
    const int64_t row = t * kTileRows + r * 256 + threadIdx.x;
    const int64_t end = carry + __shfl_sync(0xffffffffu, before, r * 8 + wid) + incl[r];
    if (row < A.rows) {
      c_off[row] = end - z[r];
      if (row == A.rows - 1) c_off[A.rows] = end;
    }
  }
  int32_t pos[kRowsPer];
  ordered_slots(base, s_cnt, cls, pos);
#pragma unroll
  for (int r = 0; r < kRowsPer; ++r)
    if (cls[r] >= 0) perm[pos[r]] = static_cast<int32_t>(t * kTileRows + r * 256 + threadIdx.x);
}

__global__ void __launch_bounds__(256) k_collect_flagged(const int32_t* __restrict__ perm, int64_t count,
                                                         const int32_t* __restrict__ row_flag, int all,
                                                         int32_t* __restrict__ list, int32_t* list_count) {
  for (int64_t r0 = blockIdx.x * int64_t(blockDim.x); r0 < count; r0 += int64_t(gridDim.x) * blockDim.x) {
    const int64_t r = r0 + threadIdx.x;
    int32_t row = 0;
    bool take = false;
    if (r < count) {
      row = perm[r];
      take = all || row_flag[row] != 0;
    }
    const unsigned m = __ballot_sync(0xffffffffu, take);
    int32_t base = 0;
    if (lane_id() == 0 && m) base = atomicAdd(list_count, __popc(m));
    base = __shfl_sync(0xffffffffu, base, 0);
    if (take) list[base + __popc(m & ((1u << lane_id()) - 1u))] = row;
  }
}

__global__ void k_write_rowptr(const int64_t* __restrict__ c_off, int64_t m1, void* out, int idx64) {
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < m1;
       i += int64_t(gridDim.x) * blockDim.x) {
    if (idx64) static_cast<int64_t*>(out)[i] = c_off[i];
    else static_cast<int32_t*>(out)[i] = static_cast<int32_t>(c_off[i]);
  }
}

inline unsigned grid_for(int64_t n, int threads, int64_t cap = 65535LL * 16) {
  int64_t g = (n + threads - 1) / threads;
  if (g < 1) g = 1;
  if (g > cap) g = cap;
  return static_cast<unsigned>(g);
}

}  // namespace

int launch_rowptr_rebase(const void* in, int idx64, int64_t r0, int64_t n1, int64_t base, int64_t* out,
                         cudaStream_t s) {
  if (n1 <= 0) return 0;
  k_rowptr_rebase<<<grid_for(n1, 256), 256, 0, s>>>(in, idx64, r0, n1, base, out);
  return 1;
}

int launch_fetch(const void* src, void* dst, int64_t bytes, cudaStream_t s) {
  const int64_t words = bytes / 4;
  if (words <= 0) return 0;
  k_fetch<<<grid_for(words, 256), 256, 0, s>>>(static_cast<const uint32_t*>(src), static_cast<uint32_t*>(dst), words);
  return 1;
}

int launch_rowptr_to64(const int32_t* in, int64_t* out, int64_t n1, cudaStream_t s) {
  k_rowptr_to64<<<grid_for(n1, 256), 256, 0, s>>>(in, out, n1);
  return 1;
}

int launch_validate(const void* rp, int rp64, int64_t rows, int64_t cols, int64_t nnz, const int32_t* col,
                    int64_t* rp_out, uint32_t* err, int num_sms, cudaStream_t s) {
  // every block the same number of kCheckEntries, one wave of them; few entries: the rows' share
  const int64_t pieces = (nnz + kCheckEntries - 1) / kCheckEntries, most = int64_t(num_sms) * kCheckBlocks;
  const int64_t per = pieces > most ? (pieces + most - 1) / most : 1;
  int64_t g = pieces > 0 ? (pieces + per - 1) / per : 1;
  const int64_t by_rows = (rows + 255) / 256 < most ? (rows + 255) / 256 : most;
  if (g < by_rows) g = by_rows;
  k_validate<<<static_cast<unsigned>(g), 256, 0, s>>>(rp, rp64, rows, cols, nnz, col, per * kCheckEntries, rp_out, err);
  return 1;
}

int launch_count(const CsrArrays& A, const CsrArrays& B, int check, int64_t* a64, ClassParams cp, int64_t* P,
                 int32_t* nnz_row, int32_t* tile_hist, int64_t* tile_sum, int64_t* tile_max, uint32_t* err,
                 int num_sms, cudaStream_t s) {
  const int64_t ntiles = (A.rows + kTileRows - 1) / kTileRows;
  if (ntiles == 0) return 0;
  cudaMemsetAsync(tile_hist, 0, sizeof(int32_t) * ntiles * kMaxClasses, s);
  cudaMemsetAsync(tile_sum, 0, sizeof(int64_t) * ntiles, s);
  if (tile_max) cudaMemsetAsync(tile_max, 0, sizeof(int64_t) * ntiles, s);
  int run = 32;
  while (run > 1 && A.rows < int64_t(run / 2) * 8 * num_sms * 8) run /= 2;   // eight blocks per SM or more
  const int64_t blocks = (A.rows + 8 * run - 1) / (8 * run);
  k_count<<<static_cast<unsigned>(blocks), 256, 0, s>>>(A, B, run, check, a64, cp, P, nnz_row, tile_hist, tile_sum, tile_max,
                                                       err);
  return 1;
}

int launch_class_scan(int64_t ntiles, int nclasses, int32_t* tile_hist, const int64_t* tile_sum,
                       const int64_t* tile_max, int64_t* tile_sum_off, Summary* summary,
                       cudaStream_t s) {
  k_class_scan<<<nclasses + 1, kScanThreads, 0, s>>>(ntiles, nclasses, tile_hist, tile_sum, tile_max, tile_sum_off,
                                 summary);
  return 1;
}

int launch_scatter_sym(const DevCsr& A, ClassParams cp, const int64_t* P, const int32_t* tile_hist,
                        const Summary* summary, int32_t* perm, cudaStream_t s) {
  const int64_t ntiles = (A.rows + kTileRows - 1) / kTileRows;
  if (ntiles == 0) return 0;
  k_scatter_sym<<<static_cast<unsigned>(ntiles), 256, 0, s>>>(A, cp, P, tile_hist, summary, perm);
  return 1;
}

int launch_num_tiles(const DevCsr& A, ClassParams cp, const int64_t* P, const int32_t* nnz_row,
                      int32_t* tile_hist, int64_t* tile_sum, unsigned long long* cls_sums,
                      cudaStream_t s) {
  const int64_t ntiles = (A.rows + kTileRows - 1) / kTileRows;
  if (ntiles == 0) return 0;
  k_num_tiles<<<static_cast<unsigned>(ntiles), 256, 0, s>>>(A, cp, P, nnz_row, tile_hist, tile_sum, cls_sums);
  return 1;
}

int launch_scatter_num(const DevCsr& A, ClassParams cp, const int64_t* P, const int32_t* nnz_row,
                        const int32_t* tile_hist, const int64_t* tile_sum_off, const Summary* summary,
                        int32_t* perm, int64_t* c_off, cudaStream_t s) {
  const int64_t ntiles = (A.rows + kTileRows - 1) / kTileRows;
  if (ntiles == 0) return 0;
  k_scatter_num<<<static_cast<unsigned>(ntiles), 256, 0, s>>>(A, cp, P, nnz_row, tile_hist,
                                                              tile_sum_off, summary, perm, c_off);
  return 1;
}

int launch_collect_flagged(const int32_t* perm, int64_t count, const int32_t* row_flag, int all,
                           int32_t* list, int32_t* list_count, cudaStream_t s) {
  if (count <= 0) return 0;
  k_collect_flagged<<<grid_for(count, 256, 152 * 16), 256, 0, s>>>(perm, count, row_flag, all, list, list_count);
  return 1;
}

int launch_write_rowptr(const int64_t* c_off, int64_t m1, void* out, int idx64, cudaStream_t s) {
  k_write_rowptr<<<grid_for(m1, 256), 256, 0, s>>>(c_off, m1, out, idx64);
  return 1;
}

}  // namespace spg
