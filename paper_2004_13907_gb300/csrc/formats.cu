// Format front-ends: COO to canonical CSR, and CSR transposition (a CSR matrix's CSC form is
// the CSR of its transpose), both on the device.
//
// The paper's CPU side turns the input matrices into its streamed row bundles (RIR, Sec. II)
// and back; here the host hands the library COO or CSC arrays and the conversion runs on the GPU.
// Both conversions are a stable sort of the entries by a key (the column for a transposition, the
// row and the column side by side for COO), done by a least-significant-digit radix sort of 32- or
// 64-bit keys in equal digits of at most kMaxDigit bits:
//   1. per tile of kSortTile keys, a histogram of the current digit (shared atomics);
//   2. per digit, an exclusive scan of its tile counts (one block per digit);
//   3. per tile, every key's place among the tile's keys in digit order (each warp takes 32 consecutive
//      keys at a time: a match mask gives the rank among the warp's 32, per-warp digit counters the
//      rest, so equal keys keep their order); the tile is put in that order in shared memory and
//      leaves as one run per digit, at the digit's base + the tile's offset in it.
// The first pass makes its keys from the input arrays and checks their range. The sort carries a
// 32-bit index; the values are gathered by it at the end, and the row pointers are found in the
// sorted keys by binary search, a thread per row.
//
// Bound by the passes over keys and indices (20 or 32 bytes per entry and pass) and by the runs of a
// tile's digits, written as a few sectors each. 9-bit digits sort 18-bit indices in two passes
// instead of three of 8 bits, one sort of 36-bit keys replaces two sorts and the gather between
// them, and runs written through shared memory take a scatter pass of 3.9e6 entries from 75 us (32-bit
// keys) to 46 us (64-bit). The search replaces an atomic count of the keys (116 us with R-MAT's hubs)
// and a one-block scan (272 us for 262,144 rows). R-MAT 2^18 edges (3.9e6, shuffled) to CSR 963 -> 342
// us; transposition of 1.05e6 entries 435 -> 86 us of kernel time.
#include <cstring>

#include "runtime.h"

namespace spg {

namespace {

constexpr int kSortThreads = 256;
constexpr int kSortItems = 16;                        // keys per thread of a tile
constexpr int kSortTile = kSortThreads * kSortItems;  // 4096 keys
constexpr int kMaxDigit = 9;                          // bits per pass
constexpr int kRadix = 1 << kMaxDigit;
constexpr int kSortWarps = kSortThreads / 32;
static_assert(kRadix == 2 * kSortThreads, "a thread takes two digits");

// Where a pass reads its keys: an array of the pass before, the columns of a CSR matrix, or the rows
// and columns of COO triples side by side (out-of-range indices set kErrInvalidCsr; the digits of such
// a key are taken as they are).
template <typename K>
struct KeyArray {
  const K* keys;
  __device__ __forceinline__ K at(int64_t i, bool&) const { return keys[i]; }
};
struct ColKeys {
  const int32_t* col;
  int64_t cols;
  __device__ __forceinline__ uint32_t at(int64_t i, bool& bad) const {
    const int32_t c = col[i];
    bad |= c < 0 || c >= cols;
    return static_cast<uint32_t>(c);
  }
};
template <typename K>
struct CooKeys {
  const int32_t* row;
  const int32_t* col;
  int64_t rows, cols;
  int col_bits;
  __device__ __forceinline__ K at(int64_t i, bool& bad) const {
    const int32_t r = row[i], c = col[i];
    bad |= r < 0 || r >= rows || c < 0 || c >= cols;
    // (col_bits is below 32, the width of K when K is 32 bits and a row index is needed at all)
    return static_cast<K>(static_cast<uint32_t>(r)) << col_bits | static_cast<uint32_t>(c);
  }
};

template <typename Src>
__global__ void __launch_bounds__(kSortThreads) k_rs_hist(Src src, int64_t n, int shift, int bits, int64_t ntiles,
                                                          uint32_t* __restrict__ hist, uint32_t* err) {
  __shared__ uint32_t h[kRadix];
  h[threadIdx.x] = h[threadIdx.x + kSortThreads] = 0;
  __syncthreads();
  const int64_t t = blockIdx.x;
  const int64_t base = t * kSortTile;
  const uint32_t mask = (1u << bits) - 1u;
  bool bad = false;
#pragma unroll 4
  for (int q = threadIdx.x; q < kSortTile; q += kSortThreads) {
    const int64_t i = base + q;
    if (i < n) atomicAdd(&h[static_cast<uint32_t>(src.at(i, bad) >> shift) & mask], 1u);
  }
  if (bad) atomicOr(err, kErrInvalidCsr);
  __syncthreads();
  for (uint32_t d = threadIdx.x; d <= mask; d += kSortThreads) hist[int64_t(d) * ntiles + t] = h[d];
}

// One block per digit: exclusive scan of the digit's tile counts (in place), total to tot[d].
__global__ void __launch_bounds__(1024) k_rs_scan_tiles(uint32_t* __restrict__ hist, int64_t ntiles,
                                                        uint32_t* __restrict__ tot) {
  __shared__ uint32_t s_scan[33];
  uint32_t* row = hist + int64_t(blockIdx.x) * ntiles;
  uint32_t carry = 0;
  for (int64_t b = 0; b < ntiles; b += 1024) {
    const int64_t i = b + threadIdx.x;
    const uint32_t v = i < ntiles ? row[i] : 0u;
    uint32_t total;
    const uint32_t ex = block_excl_scan<uint32_t>(v, s_scan, &total);
    if (i < ntiles) row[i] = carry + ex;
    carry += total;
  }
  if (threadIdx.x == 0) tot[blockIdx.x] = carry;
}

template <typename K>
struct ScatterSmem {
  K key[kSortTile];
  uint32_t idx[kSortTile];
  uint32_t out[kRadix];                  // place of a digit's first key of the tile in the output,
  uint32_t local[kRadix];                //   and in the tile's digit order
  uint16_t cnt[kSortWarps][kRadix];      // per warp: its keys of each digit, then those of the warps before
  uint32_t scan[33];
};

// The lanes among `valid` with the same digit: a vote per bit (__match_any_sync takes
// about 60 clocks per warp and SM, nine votes about 10).
__device__ __forceinline__ unsigned digit_peers(uint32_t dg, unsigned valid) {
  unsigned peers = valid;
#pragma unroll
  for (int b = 0; b < kMaxDigit; ++b) {
    const bool one = (dg >> b) & 1u;
    const unsigned ones = __ballot_sync(0xffffffffu, one);   // (bits past the digit's are zero everywhere)
    peers &= one ? ones : ~ones;
  }
  return peers;
}

template <typename K, typename Src>
__global__ void __launch_bounds__(kSortThreads, 2) k_rs_scatter(Src src, const uint32_t* __restrict__ idx, int64_t n,
                                                             int shift, int bits, int64_t ntiles,
                                                             const uint32_t* __restrict__ tile_off,
                                                             const uint32_t* __restrict__ tot,
                                                             K* __restrict__ keys_out, uint32_t* __restrict__ idx_out) {
  extern __shared__ __align__(16) unsigned char rs_smem[];
  ScatterSmem<K>& sm = *reinterpret_cast<ScatterSmem<K>*>(rs_smem);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t t = blockIdx.x;
  const int64_t base = t * kSortTile;
  const int count = static_cast<int>(n - base < kSortTile ? n - base : kSortTile);
  const uint32_t mask = (1u << bits) - 1u;
  for (int d = lane; d < kRadix; d += 32) sm.cnt[w][d] = 0;
  // the thread's two digits: their bases (an exclusive scan of the digit totals) + the tile's offsets
  const uint32_t d0 = 2 * threadIdx.x, d1 = d0 + 1;
  {
    const uint32_t t0 = d0 <= mask ? tot[d0] : 0u, t1 = d1 <= mask ? tot[d1] : 0u;
    uint32_t total;
    const uint32_t ex = block_excl_scan<uint32_t>(t0 + t1, sm.scan, &total);
    if (d0 <= mask) sm.out[d0] = ex + tile_off[int64_t(d0) * ntiles + t];
    if (d1 <= mask) sm.out[d1] = ex + t0 + tile_off[int64_t(d1) * ntiles + t];
  }
  // warp w takes the tile's keys [w * 512, (w + 1) * 512), 32 at a time, in order
  const int wbase = w * (kSortTile / kSortWarps);
  K key[kSortItems];
  uint16_t rank[kSortItems];
  bool unused = false;
#pragma unroll
  for (int r = 0; r < kSortItems; ++r) {
    const int q = wbase + r * 32 + lane;
    key[r] = q < count ? src.at(base + q, unused) : K(0);
  }
#pragma unroll
  for (int r = 0; r < kSortItems; ++r) {
    const bool ok = wbase + r * 32 + lane < count;
    const uint32_t dg = static_cast<uint32_t>(key[r] >> shift) & mask;
    const unsigned peers = digit_peers(dg, __ballot_sync(0xffffffffu, ok));
    uint32_t before = 0;
    if (ok) before = sm.cnt[w][dg];
    __syncwarp();
    if (ok && lane == __ffs(peers) - 1) sm.cnt[w][dg] = static_cast<uint16_t>(before + __popc(peers));
    __syncwarp();
    rank[r] = static_cast<uint16_t>(before + __popc(peers & ((1u << lane) - 1u)));
  }
  __syncthreads();
  // the thread's two digits: the warps' keys before each warp's, and the digits' places in the tile
  {
    uint32_t c0 = 0, c1 = 0;
#pragma unroll
    for (int ww = 0; ww < kSortWarps; ++ww) {
      uint32_t* both = reinterpret_cast<uint32_t*>(&sm.cnt[ww][d0]);
      const uint32_t v = *both;
      *both = c0 | c1 << 16;
      c0 += v & 0xffffu;
      c1 += v >> 16;
    }
    uint32_t total;
    const uint32_t ex = block_excl_scan<uint32_t>(c0 + c1, sm.scan, &total);
    sm.local[d0] = ex;
    sm.local[d1] = ex + c0;
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < kSortItems; ++r) {
    const int q = wbase + r * 32 + lane;
    if (q < count) {
      const uint32_t dg = static_cast<uint32_t>(key[r] >> shift) & mask;
      const uint32_t pos = sm.local[dg] + sm.cnt[w][dg] + rank[r];
      sm.key[pos] = key[r];
      sm.idx[pos] = idx ? idx[base + q] : static_cast<uint32_t>(base + q);
    }
  }
  __syncthreads();
  for (int q = threadIdx.x; q < count; q += kSortThreads) {
    const K k = sm.key[q];
    const uint32_t dg = static_cast<uint32_t>(k >> shift) & mask;
    const uint32_t pos = sm.out[dg] + (static_cast<uint32_t>(q) - sm.local[dg]);
    keys_out[pos] = k;
    idx_out[pos] = sm.idx[q];
  }
}

// Stable sort of n keys whose values lie below 2^key_bits, carrying the index of each: the first pass
// reads `src`, the others alternate between the two pairs. Returns which pair (0 or 1) holds the sorted
// keys and indices.
template <typename K, typename Src>
int stable_sort(Src src, K* const (&keys)[2], uint32_t* const (&idx)[2], int64_t n, int key_bits, uint32_t* hist,
                uint32_t* tot, uint32_t* err, cudaStream_t s) {
  const int64_t ntiles = (n + kSortTile - 1) / kSortTile;
  const unsigned grid = static_cast<unsigned>(ntiles);
  const int passes = key_bits > kMaxDigit ? (key_bits + kMaxDigit - 1) / kMaxDigit : 1;
  const int bits = key_bits > passes ? (key_bits + passes - 1) / passes : 1;
  constexpr int smem = static_cast<int>(sizeof(ScatterSmem<K>));
  for (int q = 0; q < passes; ++q) {
    const int shift = q * bits;
    auto pass = [&](auto from, const uint32_t* from_idx) {
      auto scatter = k_rs_scatter<K, decltype(from)>;
      cudaFuncSetAttribute(scatter, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
      k_rs_hist<<<grid, kSortThreads, 0, s>>>(from, n, shift, bits, ntiles, hist, err);
      k_rs_scan_tiles<<<1u << bits, 1024, 0, s>>>(hist, ntiles, tot);
      scatter<<<grid, kSortThreads, smem, s>>>(from, from_idx, n, shift, bits, ntiles, hist, tot, keys[q & 1], idx[q & 1]);
    };
    if (q == 0) pass(src, nullptr);
    else pass(KeyArray<K>{keys[(q - 1) & 1]}, idx[(q - 1) & 1]);
  }
  return (passes - 1) & 1;
}

int bits_for(int64_t v) {
  int b = 0;
  while (b < 32 && (int64_t(1) << b) < v) ++b;
  return b;
}

// Row index of every stored entry of M: a row of up to 8 entries by its thread, a longer one by the
// whole warp. Row pointers that decrease, lie outside [0, nnz] or leave an entry to no row are reported.
__global__ void __launch_bounds__(256) k_expand_rows(const void* __restrict__ rp, int rp64, int64_t m, int64_t nnz,
                                                     uint32_t* __restrict__ row_of, uint32_t* err) {
  const int lane = threadIdx.x & 31;
  auto at = [&](int64_t i) { return rp64 ? static_cast<const int64_t*>(rp)[i] : static_cast<const int32_t*>(rp)[i]; };
  for (int64_t i0 = blockIdx.x * int64_t(blockDim.x) + (threadIdx.x & ~31); i0 < m; i0 += int64_t(gridDim.x) * blockDim.x) {
    const int64_t i = i0 + lane;
    int64_t s = 0, e = 0;
    if (i < m) {
      s = at(i);
      e = at(i + 1);
      if ((i == 0 && s != 0) || (i == m - 1 && e != nnz)) atomicOr(err, kErrInvalidCsr);
      if (s < 0 || e < s || e > nnz) {
        atomicOr(err, kErrInvalidCsr);
        s = e = 0;
      }
    }
    const bool is_long = e - s > 8;
    if (!is_long)
      for (int64_t q = s; q < e; ++q) row_of[q] = static_cast<uint32_t>(i);
    for (unsigned lm = __ballot_sync(0xffffffffu, is_long); lm; lm &= lm - 1) {
      const int src = __ffs(lm) - 1;
      const int64_t ls = __shfl_sync(0xffffffffu, s, src), le = __shfl_sync(0xffffffffu, e, src);
      for (int64_t q = ls + lane; q < le; q += 32) row_of[q] = static_cast<uint32_t>(i0 + src);
    }
  }
}

// Row pointers (int32 or int64) of m rows from n sorted keys, the row in the bits from `shift` up:
// out[r] = the first key of row r or later, by binary search.
template <typename K>
__global__ void __launch_bounds__(256) k_search_rowptr(const K* __restrict__ keys, int64_t n, int shift, int64_t m,
                                                       void* __restrict__ out, int idx64) {
  for (int64_t r = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; r <= m; r += int64_t(gridDim.x) * blockDim.x) {
    int64_t lo = 0, hi = n;
    if (r == m) lo = n;
    while (lo < hi) {
      const int64_t mid = lo + ((hi - lo) >> 1);
      if (static_cast<int64_t>(static_cast<uint64_t>(keys[mid]) >> shift) < r) lo = mid + 1;
      else hi = mid;
    }
    if (idx64) static_cast<int64_t*>(out)[r] = lo;
    else static_cast<int32_t*>(out)[r] = static_cast<int32_t>(lo);
  }
}

// The entries in sorted order: out_col[q] = new_col[perm[q]], out_val[q] = val[perm[q]] (8 or 4
// bytes per value).
__global__ void k_gather_entries(const uint32_t* __restrict__ perm, int64_t n, const uint32_t* __restrict__ new_col,
                                 const void* __restrict__ val, int vbytes, int32_t* __restrict__ out_col,
                                 void* __restrict__ out_val) {
  for (int64_t q = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; q < n; q += int64_t(gridDim.x) * blockDim.x) {
    const uint32_t p = perm[q];
    out_col[q] = static_cast<int32_t>(new_col[p]);
    if (vbytes == 8) static_cast<double*>(out_val)[q] = static_cast<const double*>(val)[p];
    else static_cast<float*>(out_val)[q] = static_cast<const float*>(val)[p];
  }
}

// Sorted COO entries: columns from the keys, values through the order; a repeated (row, column) pair is
// an error (the output must be canonical).
template <typename K>
__global__ void __launch_bounds__(256) k_coo_entries(const K* __restrict__ keys, const uint32_t* __restrict__ perm,
                                                     int64_t n, int col_bits, const void* __restrict__ val, int vbytes,
                                                     int32_t* __restrict__ out_col, void* __restrict__ out_val,
                                                     uint32_t* err) {
  bool bad = false;
  for (int64_t q = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; q < n; q += int64_t(gridDim.x) * blockDim.x) {
    const K k = keys[q];
    bad |= q > 0 && keys[q - 1] == k;
    out_col[q] = static_cast<int32_t>(k & ((K(1) << col_bits) - 1));
    const uint32_t p = perm[q];
    if (vbytes == 8) static_cast<double*>(out_val)[q] = static_cast<const double*>(val)[p];
    else static_cast<float*>(out_val)[q] = static_cast<const float*>(val)[p];
  }
  if (bad) atomicOr(err, kErrInvalidCsr);
}

unsigned grid_for(int64_t n) {
  int64_t g = (n + 255) / 256;
  if (g > 152 * 32) g = 152 * 32;
  return static_cast<unsigned>(g < 1 ? 1 : g);
}

// Device scratch of one conversion, from the caller's allocator or the stream-ordered pool.
struct Scratch {
  Workspace ws;
  spgemm_status st = SPGEMM_OK;
  template <typename T>
  T* get(int64_t count) {
    if (st != SPGEMM_OK) return nullptr;
    void* p = ws.get(static_cast<size_t>(count < 1 ? 1 : count) * sizeof(T));
    if (!p) st = set_error_msg(SPGEMM_ERR_OOM, "conversion scratch of %lld bytes", (long long)(count * sizeof(T)));
    return static_cast<T*>(p);
  }
};

spgemm_status finish(Scratch& sc, uint32_t* err, cudaStream_t s, const char* what) {
  uint32_t h = 0;
  spgemm_status st = cuda_status(cudaGetLastError(), what);
  if (st == SPGEMM_OK) st = read_small(&h, err, sizeof(h), s, nullptr, what);
  sc.ws.release_all();
  if (st != SPGEMM_OK) return st;
  if (h & kErrInvalidCsr)
    return set_error_msg(SPGEMM_ERR_INVALID_CSR,
                         "%s: an index or row pointer is out of range or a (row, column) pair repeats", what);
  if (h) return set_error_msg(SPGEMM_ERR_INTERNAL, "%s: device check failed (0x%x)", what, h);
  return SPGEMM_OK;
}

void init_scratch(Scratch& sc, const spgemm_allocator* alloc, void* stream) {
  sc.ws.stream = stream;
  if (alloc && alloc->alloc && alloc->free) {
    sc.ws.alloc = *alloc;
    sc.ws.has_alloc = true;
  }
}

}  // namespace

}  // namespace spg

using namespace spg;

extern "C" spgemm_status spgemm_csr_transpose(const spgemm_csr_in* M, int32_t value_bytes, spgemm_csr_out* T,
                                              const spgemm_allocator* alloc, void* stream) {
  clear_error_msg();
  if (!M || !T) return set_error_msg(SPGEMM_ERR_INVALID_ARG, "NULL argument");
  if (value_bytes != 8 && value_bytes != 4) return set_error_msg(SPGEMM_ERR_INVALID_ARG, "value_bytes is 8 or 4");
  spgemm_status st = check_csr_in(M, "M", value_bytes == 8 ? SPGEMM_F64 : SPGEMM_F32_COMPENSATED);
  if (st != SPGEMM_OK) return st;
  const int vbytes = value_bytes;
  const int64_t m = M->rows, n = M->cols, nnz = M->nnz;
  if (nnz > 0xffffffffLL) return set_error_msg(SPGEMM_ERR_UNSUPPORTED, "transposition takes fewer than 2^32 entries");
  if (!T->row_ptr || (nnz > 0 && (!T->col || !T->val)))
    return set_error_msg(SPGEMM_ERR_INVALID_ARG, "T's arrays are NULL");
  if (!T->idx64_rowptr && nnz > 0x7fffffffLL) return set_error_msg(SPGEMM_ERR_INDEX_OVERFLOW, "T needs an int64 row_ptr");
  if (m == 0 && nnz > 0) return set_error_msg(SPGEMM_ERR_INVALID_CSR, "transposing: entries but no rows");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  Scratch sc;
  init_scratch(sc, alloc, stream);
  uint32_t* err = sc.get<uint32_t>(4);
  const int64_t ntiles = (nnz + kSortTile - 1) / kSortTile;
  uint32_t* const keys[2] = {sc.get<uint32_t>(nnz), sc.get<uint32_t>(nnz)};
  uint32_t* const idx[2] = {sc.get<uint32_t>(nnz), sc.get<uint32_t>(nnz)};
  uint32_t* row_of = sc.get<uint32_t>(nnz);
  uint32_t* hist = sc.get<uint32_t>(kRadix * (ntiles > 0 ? ntiles : 1));
  uint32_t* tot = sc.get<uint32_t>(kRadix);
  if (sc.st != SPGEMM_OK) {
    sc.ws.release_all();
    return sc.st;
  }
  cudaMemsetAsync(err, 0, sizeof(uint32_t), s);
  int sorted = 0;
  if (nnz > 0) {
    k_expand_rows<<<grid_for(m), 256, 0, s>>>(M->row_ptr, M->idx64_rowptr, m, nnz, row_of, err);
    sorted = stable_sort<uint32_t>(ColKeys{M->col, n}, keys, idx, nnz, bits_for(n), hist, tot, err, s);
    k_gather_entries<<<grid_for(nnz), 256, 0, s>>>(idx[sorted], nnz, row_of, M->val, vbytes, T->col, T->val);
  }
  k_search_rowptr<uint32_t><<<grid_for(n + 1), 256, 0, s>>>(keys[sorted], nnz, 0, n, T->row_ptr, T->idx64_rowptr);
  st = finish(sc, err, s, "transposing");
  if (st != SPGEMM_OK) return st;
  T->rows = n;
  T->cols = m;
  T->nnz = nnz;
  return SPGEMM_OK;
}

extern "C" spgemm_status spgemm_coo_to_csr(int64_t rows, int64_t cols, int64_t nnz, const int32_t* row,
                                           const int32_t* col, const void* val, int32_t value_bytes,
                                           spgemm_csr_out* C, const spgemm_allocator* alloc, void* stream) {
  clear_error_msg();
  if (rows < 0 || cols < 0 || nnz < 0) return set_error_msg(SPGEMM_ERR_INVALID_ARG, "negative size");
  if (rows > 0x7fffffffLL || cols > 0x7fffffffLL)
    return set_error_msg(SPGEMM_ERR_INVALID_ARG, "row and column indices are int32");
  if (value_bytes != 8 && value_bytes != 4) return set_error_msg(SPGEMM_ERR_INVALID_ARG, "value_bytes is 8 or 4");
  if (nnz > 0xffffffffLL) return set_error_msg(SPGEMM_ERR_UNSUPPORTED, "conversion takes fewer than 2^32 entries");
  if (!C || !C->row_ptr || (nnz > 0 && (!row || !col || !val || !C->col || !C->val)))
    return set_error_msg(SPGEMM_ERR_INVALID_ARG, "NULL array");
  if (!C->idx64_rowptr && nnz > 0x7fffffffLL) return set_error_msg(SPGEMM_ERR_INDEX_OVERFLOW, "C needs an int64 row_ptr");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  Scratch sc;
  init_scratch(sc, alloc, stream);
  uint32_t* err = sc.get<uint32_t>(4);
  const int64_t ntiles = (nnz + kSortTile - 1) / kSortTile;
  uint32_t* hist = sc.get<uint32_t>(kRadix * (ntiles > 0 ? ntiles : 1));
  uint32_t* tot = sc.get<uint32_t>(kRadix);
  uint32_t* const idx[2] = {sc.get<uint32_t>(nnz), sc.get<uint32_t>(nnz)};
  // one sort by row and column side by side: 32-bit keys when both fit
  const int col_bits = bits_for(cols), key_bits = bits_for(rows) + col_bits;
  auto convert = [&](auto zero) {
    using K = decltype(zero);
    K* const keys[2] = {sc.get<K>(nnz), sc.get<K>(nnz)};
    if (sc.st != SPGEMM_OK) return;
    cudaMemsetAsync(err, 0, sizeof(uint32_t), s);
    int sorted = 0;
    if (nnz > 0) {
      sorted = stable_sort<K>(CooKeys<K>{row, col, rows, cols, col_bits}, keys, idx, nnz, key_bits, hist, tot, err, s);
      k_coo_entries<K><<<grid_for(nnz), 256, 0, s>>>(keys[sorted], idx[sorted], nnz, col_bits, val, value_bytes, C->col,
                                                     C->val, err);
    }
    k_search_rowptr<K><<<grid_for(rows + 1), 256, 0, s>>>(keys[sorted], nnz, col_bits, rows, C->row_ptr, C->idx64_rowptr);
  };
  if (key_bits <= 31) convert(uint32_t(0));
  else convert(uint64_t(0));
  if (sc.st != SPGEMM_OK) {
    sc.ws.release_all();
    return sc.st;
  }
  spgemm_status st = finish(sc, err, s, "converting COO to CSR");
  if (st != SPGEMM_OK) return st;
  C->rows = rows;
  C->cols = cols;
  C->nnz = nnz;
  return SPGEMM_OK;
}
