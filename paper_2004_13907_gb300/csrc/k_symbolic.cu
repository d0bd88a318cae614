// Symbolic pass: nnz(C_i) = |union over the stored k of row i of A of cols(B_k)|,
// the size of the COLB set Algorithm 1 builds for row i (Sec. III-A).
//
// Row classes (chosen by the plan from P_i and min(P_i, n)):
//  * tiny  : P_i <= 32, one warp, each lane holds one column; duplicates are found with a
//            warp match, so no shared table is needed;
//  * warp  : one warp per row, a shared-memory hash table of 128 / 512 / 2048 keys;
//  * micro, merge : one thread per row of at most 8 entries of A, a merge of the B rows;
//  * block : one block per row, a bitmap of up to 2^18 columns, or a hash table of 8192 keys;
//  * window: persistent blocks, one row at a time, a shared-memory bitmap of up to 2^20 columns.
//            Besides nnz(C_i) it records how many columns of C_i fall in each block of
//            kBlockCols columns (or sub-block of kSubCols), which the numeric pass uses to plan its windows. When B has
//            more than 2^20 columns the bitmap slides over the columns in windows and a
//            per-entry cursor in global memory remembers where each B row stopped.
// Hash tables are sized to at least twice the row's upper bound min(P_i, n), so probing
// always ends; a probe count over the table size still reports kErrHashFull.
#include "enumerate.cuh"

namespace spg {

namespace {

__global__ void __launch_bounds__(256) k_sym_tiny(DevCsr A, DevCsr B, const int32_t* __restrict__ perm,
                                                  int64_t count, int32_t* __restrict__ nnz_row) {
  const int lane = threadIdx.x & 31;
  const int64_t gw = (blockIdx.x * int64_t(blockDim.x) + threadIdx.x) >> 5;
  const int64_t nw = (int64_t(gridDim.x) * blockDim.x) >> 5;
  for (int64_t r = gw; r < count; r += nw) {
    const int32_t i = perm[r];
    const int64_t a0 = A.rp[i];
    const int32_t na = static_cast<int32_t>(A.rp[i + 1] - a0);
    int32_t col = -2 - lane;
    int32_t total = 0;
    int32_t len = 0;
    int64_t bs = 0;
    if (lane < na) {
      const int32_t k = A.col[a0 + lane];
      bs = B.rp[k];
      len = static_cast<int32_t>(B.rp[k + 1] - bs);
    }
    const int32_t incl = warp_incl_scan(len);
    total = __shfl_sync(0xffffffffu, incl, 31);
    int o = 0;
#pragma unroll
    for (int step = 16; step > 0; step >>= 1) {
      const int32_t v = __shfl_sync(0xffffffffu, incl, o + step - 1);
      if (v <= lane) o += step;
    }
    const int32_t incl_o = __shfl_sync(0xffffffffu, incl, o & 31);
    const int32_t len_o = __shfl_sync(0xffffffffu, len, o & 31);
    const int64_t bs_o = __shfl_sync(0xffffffffu, bs, o & 31);
    if (lane < total) col = B.col[bs_o + (lane - (incl_o - len_o))];
    const unsigned peers = __match_any_sync(0xffffffffu, col);
    const bool lead = lane < total && (__ffs(peers) - 1) == lane;
    const int n = __popc(__ballot_sync(0xffffffffu, lead));
    if (lane == 0) nnz_row[i] = n;
  }
}

// Micro and merge rows (nnz(A_i) <= kMicroNa): one thread per row merges the row's sorted B rows head
// by head (the smallest head column is the next column of C; every head holding it advances) and
// counts the distinct columns. NA: the most A entries of a row of the warp.
template <int NA>
__device__ __forceinline__ int32_t merge_count(const DevCsr& A, const DevCsr& B, int64_t a0, int na) {
  constexpr int32_t kEnd = 0x7fffffff;   // column of an exhausted head (every column is smaller)
  int64_t pos[NA];
  int32_t left[NA], hc[NA];
#pragma unroll
  for (int h = 0; h < NA; ++h) {
    pos[h] = 0; left[h] = 0; hc[h] = kEnd;
    if (h < na) {
      const int32_t k = A.col[a0 + h];
      pos[h] = B.rp[k];
      left[h] = static_cast<int32_t>(B.rp[k + 1] - pos[h]);
    }
  }
#pragma unroll
  for (int h = 0; h < NA; ++h) if (left[h] > 0) hc[h] = B.col[pos[h]];
  int32_t n = 0;
  for (;;) {
    int32_t m = hc[0];
#pragma unroll
    for (int h = 1; h < NA; ++h) m = min(m, hc[h]);
    if (m == kEnd) break;
    ++n;
#pragma unroll
    for (int h = 0; h < NA; ++h) {
      if (hc[h] == m) {
        ++pos[h];
        --left[h];
        hc[h] = left[h] > 0 ? B.col[pos[h]] : kEnd;
      }
    }
  }
  return n;
}

__global__ void __launch_bounds__(256) k_sym_micro(DevCsr A, DevCsr B, const int32_t* __restrict__ perm,
                                                   int64_t count, int32_t* __restrict__ nnz_row) {
  const int64_t stride = int64_t(gridDim.x) * blockDim.x;
  for (int64_t r0 = blockIdx.x * int64_t(blockDim.x) + (threadIdx.x & ~31); r0 < count; r0 += stride) {
    const int64_t r = r0 + (threadIdx.x & 31);
    const bool mine = r < count;
    const int32_t i = perm[mine ? r : r0];
    const int64_t a0 = A.rp[i];
    const int na = mine ? static_cast<int>(A.rp[i + 1] - a0) : 0;
    const int most = __reduce_max_sync(0xffffffffu, na);
    int32_t n;
    if (most <= 5) n = merge_count<5>(A, B, a0, na);
    else if (most <= 7) n = merge_count<7>(A, B, a0, na);
    else n = merge_count<kMicroNa>(A, B, a0, na);
    if (mine) nnz_row[i] = n;
  }
}

// Insert `key` into an open-addressing table (linear probing). Returns 1 if it was new.
template <int LOG2S>
__device__ __forceinline__ int insert_key(int32_t* table, int32_t key, uint32_t* err) {
  constexpr int S = 1 << LOG2S;
  uint32_t h = hash_slot(key, LOG2S);
  for (int probe = 0; probe < S; ++probe) {
    const int32_t cur = *reinterpret_cast<volatile int32_t*>(&table[h]);
    if (cur == key) return 0;
    if (cur == kEmpty) {
      const int32_t old = atomicCAS(&table[h], kEmpty, key);
      if (old == kEmpty) return 1;
      if (old == key) return 0;
    }
    h = (h + 1) & (S - 1);
  }
  set_error(err, kErrHashFull);
  return 0;
}

template <int LOG2S>
__global__ void __launch_bounds__(256) k_sym_warp(DevCsr A, DevCsr B, const int32_t* __restrict__ perm,
                                                  int64_t count, int32_t* __restrict__ nnz_row,
                                                  uint32_t* err) {
  constexpr int S = 1 << LOG2S;
  extern __shared__ int32_t smem_i32[];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int32_t* table = smem_i32 + wid * S;
  const int64_t gw = (blockIdx.x * int64_t(blockDim.x) + threadIdx.x) >> 5;
  const int64_t nw = (int64_t(gridDim.x) * blockDim.x) >> 5;
  for (int64_t r = gw; r < count; r += nw) {
    const int32_t i = perm[r];
    const int64_t a0 = A.rp[i];
    const int64_t na = A.rp[i + 1] - a0;
    for (int s = lane; s < S; s += 32) table[s] = kEmpty;
    __syncwarp();
    int cnt = 0;
    warp_for_each_product(A, B, a0, na, [&](int64_t j, int64_t) {
      cnt += insert_key<LOG2S>(table, B.col[j], err);
    });
    cnt = warp_sum(cnt);
    if (lane == 0) nnz_row[i] = cnt;
    __syncwarp();
  }
}

template <int LOG2S, int NT>
__global__ void __launch_bounds__(NT) k_sym_block(DevCsr A, DevCsr B, const int32_t* __restrict__ perm,
                                                  int64_t count, int32_t* __restrict__ nnz_row,
                                                  uint32_t* err) {
  constexpr int S = 1 << LOG2S;
  extern __shared__ int32_t smem_i32[];
  int32_t* table = smem_i32;
  __shared__ int32_t s_excl[NT];
  __shared__ int64_t s_bs[NT];
  __shared__ int32_t s_scan[33];
  __shared__ int32_t s_cnt;
  for (int64_t r = blockIdx.x; r < count; r += gridDim.x) {
    const int32_t i = perm[r];
    const int64_t a0 = A.rp[i];
    const int64_t na = A.rp[i + 1] - a0;
    for (int s = threadIdx.x; s < S; s += NT) table[s] = kEmpty;
    if (threadIdx.x == 0) s_cnt = 0;
    __syncthreads();
    int cnt = 0;
    block_for_each_product<NT>(A, B, a0, na, s_excl, s_bs, s_scan, [&](int64_t j, int64_t) {
      cnt += insert_key<LOG2S>(table, B.col[j], err);
    });
    cnt = warp_sum(cnt);
    if ((threadIdx.x & 31) == 0 && cnt) atomicAdd(&s_cnt, cnt);
    __syncthreads();
    if (threadIdx.x == 0) nnz_row[i] = s_cnt;
    __syncthreads();
  }
}

// Bitmap words of the windowed pass with six and with three blocks on an SM.
constexpr int kSymWinWords6 = 1 << 13;
constexpr int kSymWinWords3 = 1 << 14;

// Block rows in a column space of at most kSymBitmapCols: one bit per column in shared memory. A product
// whose atomic finds its bit clear counts, so there is no counting pass; the products of a row of one
// step per warp (all of them, unless the width itself is below block_max) stay in registers and clear
// their words afterwards. The hash table it replaces cleared 8,192 slots a row and probed: 20,000^2
// uniform (d = 2e-3, 19,000 rows of 1,600 products) 231 -> 145 us.
//
// A row whose products do not stay in registers sets a byte per column with a plain store where the column
// space has at most kSymByteCols (its products reach few columns many times: 32 of a warp meet in a few
// bitmap words, and their atomics wait for one another), and counts the bytes. 30,000 rows of 100,000 products in
// 1,200 columns: hash table 6.19 ms, bits 6.87, bytes 5.39; 2,040 columns 9.54, 9.60, 7.10.
constexpr int kSymBitmapCols = kSymWinWords6 * 32;
constexpr int kSymByteCols = 4096;
template <int NT, int Blocks, bool Bytes>
__global__ void __launch_bounds__(NT, Blocks) k_sym_bitmap(DevCsr A, DevCsr B, int bitmap_words,
                                                           const int32_t* __restrict__ perm, int64_t count,
                                                           int32_t* __restrict__ nnz_row,
                                                           const int32_t* __restrict__ abase, uint32_t* err) {
  extern __shared__ uint32_t bm[];  // bitmap_words, and with Bytes a byte per column
  __shared__ int32_t s_excl[NT + 1];
  __shared__ int64_t s_bs[NT];
  __shared__ long long s_scan64[33];
  __shared__ int32_t s_ctl[2];
  __shared__ int32_t s_cnt[2];
  constexpr int kHold = 8;
  uint32_t* const bytes = bm + bitmap_words;
  const int byte_words = Bytes ? 8 * bitmap_words : 0;
  for (int t = threadIdx.x; t < bitmap_words + byte_words; t += NT) bm[t] = 0u;
  if (threadIdx.x < 2) s_cnt[threadIdx.x] = 0;
  __syncthreads();
  const uint32_t span = static_cast<uint32_t>(bitmap_words) * 32u;
  int turn = 0;
  for (int64_t r = blockIdx.x; r < count; r += gridDim.x) {
    const int32_t i = perm[r];
    const int64_t a0 = A.rp[i];
    const int64_t na = A.rp[i + 1] - a0;
    const int32_t cb = abase ? abase[i] : 0;
    uint32_t held[kHold];
    int cnt = 0, steps = 0;
    bool outside = false;
    block_range_for_each_product<NT, kHold>(A, B, a0, na, s_excl, s_bs, s_scan64, s_ctl, [&](const int64_t (&j)[kHold]) {
#pragma unroll
      for (int u = 0; u < kHold; ++u) held[u] = j[u] >= 0 ? static_cast<uint32_t>(B.col[j[u]] - cb) : 0xffffffffu;
      if (Bytes && (na > NT || s_ctl[1] > NT * kHold)) {
#pragma unroll
        for (int u = 0; u < kHold; ++u) {
          if (held[u] < span) reinterpret_cast<uint8_t*>(bytes)[held[u]] = 1;
          else outside |= j[u] >= 0;
        }
        return;
      }
#pragma unroll
      for (int u = 0; u < kHold; ++u) {
        if (held[u] < span) {
          const uint32_t bit = 1u << (held[u] & 31);
          cnt += (atomicOr(&bm[held[u] >> 5], bit) & bit) == 0u;
        } else {
          outside |= j[u] >= 0;
        }
      }
      ++steps;
    });
    if (outside) set_error(err, kErrCount);
    // (the enumeration ends with a barrier: every product of the row is marked)
    const bool few = na <= NT && s_ctl[1] <= NT * kHold;
    if (few) {
      if (steps > 0)
#pragma unroll
        for (int u = 0; u < kHold; ++u)
          if (held[u] < span) bm[held[u] >> 5] = 0u;
    } else if (Bytes) {
      for (int t = threadIdx.x; t < byte_words; t += NT) {
        cnt += __popc(bytes[t]);
        bytes[t] = 0u;
      }
    } else {
      for (int t = threadIdx.x; t < bitmap_words; t += NT) bm[t] = 0u;
    }
    cnt = warp_sum(cnt);
    if ((threadIdx.x & 31) == 0 && cnt) atomicAdd(&s_cnt[turn], cnt);
    __syncthreads();
    if (threadIdx.x == 0) {
      nnz_row[i] = s_cnt[turn];
      s_cnt[turn] = 0;
    }
    turn ^= 1;
  }
}

// Windowed symbolic pass, one row per block at a time (rows handed out by an atomic
// counter, heaviest class first).
template <int NT, int Blocks>
__global__ void __launch_bounds__(NT, Blocks) k_sym_window(DevCsr A, DevCsr B, int bitmap_words,
                                                               const int32_t* __restrict__ perm,
                                                               int64_t count, int32_t* counter,
                                                               int32_t* __restrict__ nnz_row,
                                                               int32_t* __restrict__ win_slot,
                                                               uint16_t* __restrict__ blockcnt,
                                                               int64_t nblocks, int sub, int32_t* cursor,
                                                               const int32_t* __restrict__ abase,
                                                               const int32_t* __restrict__ awidth,
                                                               int64_t width_all, uint32_t* __restrict__ wbits,
                                                               int64_t wcap, unsigned long long* wcur,
                                                               int64_t* __restrict__ woff, uint32_t* err) {
  extern __shared__ uint32_t bm[];  // bitmap_words
  __shared__ int32_t s_excl[NT + 1];
  __shared__ int64_t s_bs[NT];
  __shared__ long long s_scan64[33];
  __shared__ int32_t s_ctl[2];
  __shared__ int32_t s_idx;
  __shared__ unsigned long long s_total;
  __shared__ long long s_woff;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  constexpr int kWarps = NT / 32;
  // the bitmap is cleared once here; every window's counting pass leaves it clear again
  for (int t = threadIdx.x; t < bitmap_words; t += NT) bm[t] = 0u;
  if (threadIdx.x == 0) {
    s_idx = atomicAdd(counter, 1);
    s_total = 0;
  }
  for (;;) {
    __syncthreads();
    const int64_t idx = s_idx;
    if (idx >= count) break;
    const int32_t i = perm[idx];
    if (threadIdx.x == 0) win_slot[i] = static_cast<int32_t>(idx);
    const int64_t a0 = A.rp[i];
    const int64_t na = A.rp[i + 1] - a0;
    const int64_t cb = abase ? abase[i] : 0;   // the row's columns are [cb, cb + width)
    const int64_t width = awidth ? awidth[i] : width_all;
    uint16_t* cnts = blockcnt + idx * nblocks;
    // a row inside one window stores its bitmap (its blocks, 128 words each) for the numeric
    // pass when wbits has room
    const bool store = wbits != nullptr && width <= kSymWinBits;
    // thread 0 claims the next row and this row's stored-bitmap space now; both results are used
    // only after the marking, so the atomics' latency hides behind it
    int64_t next_idx = 0;
    const int64_t words = store ? (width + kBlockCols - 1) / kBlockCols * kBlockWords : 0;
    unsigned long long woff_at = 0;
    if (threadIdx.x == 0) {
      next_idx = atomicAdd(counter, 1);
      if (store) woff_at = atomicAdd(wcur, static_cast<unsigned long long>(words));
    }
    for (int64_t r0 = 0; r0 < width; r0 += kSymWinBits) {
      const int64_t w0 = cb + r0;
      const int64_t wend = cb + ((r0 + kSymWinBits < width) ? r0 + kSymWinBits : width);
      if (width <= kSymWinBits) {
        // one window covers every column: no cursors; each warp marks a contiguous range of the
        // row's products (eight groups of 32 loaded before they are marked)
        // columns and the window start are below 2^31, so the offset fits 32 bits; a negative one
        // wraps above span
        const uint32_t span = static_cast<uint32_t>(wend - w0);
        const int32_t w0i = static_cast<int32_t>(w0);
        bool outside = false;
        block_range_for_each_product<NT, 8>(
            A, B, a0, na, s_excl, s_bs, s_scan64, s_ctl, [&](const int64_t (&j)[8]) {
              int32_t c[8];
#pragma unroll
              for (int u = 0; u < 8; ++u) c[u] = j[u] >= 0 ? B.col[j[u]] : w0i;
#pragma unroll
              for (int u = 0; u < 8; ++u) {
                if (j[u] < 0) continue;
                const uint32_t rel = static_cast<uint32_t>(c[u] - w0i);
                if (rel < span) atomicOr(&bm[rel >> 5], 1u << (rel & 31));
                else outside = true;
              }
            });
        if (outside) set_error(err, kErrWindowPlan);
      } else {
        for (int64_t e = wid; e < na; e += kWarps) {
          const int32_t k = A.col[a0 + e];
          const int64_t bstart = B.rp[k], bend = B.rp[k + 1];
          int64_t cur = (r0 == 0) ? bstart : bstart + cursor[a0 + e];
          while (cur < bend) {
            const int64_t j = cur + lane;
            const int32_t c = j < bend ? B.col[j] : kNoCol;
            const bool ok = c < wend;
            if (ok && c >= w0) atomicOr(&bm[(c - w0) >> 5], 1u << ((c - w0) & 31));
            const int got = __popc(__ballot_sync(0xffffffffu, ok));
            cur += got;
            if (got < 32) break;
          }
          if (lane == 0) cursor[a0 + e] = static_cast<int32_t>(cur - bstart);
        }
        __syncthreads();
      }
      if (r0 == 0) {
        // the stored copy's place (a stored row has this one window), published for the pass below
        if (threadIdx.x == 0) {
          long long o = -1;
          if (store && woff_at + words <= static_cast<unsigned long long>(wcap)) o = static_cast<long long>(woff_at);
          s_woff = o;
          if (woff) woff[idx] = o;
        }
        __syncthreads();
      }
      const long long wo = s_woff;
      // per-block counts of this window, the stored copy and the clearing of the bitmap in one
      // pass: a warp per block of kBlockWords words (lane: 4), blocks counted from the row's first
      // column cb. A window ends on a block boundary (kSymWinBits is a multiple of kBlockCols), so
      // every block's words lie inside the bitmap; words past the row's width were never marked.
      const int64_t b0 = r0 / kBlockCols;
      const int64_t b1 = (wend - cb + kBlockCols - 1) / kBlockCols;
      for (int64_t b = b0 + wid; b < b1; b += kWarps) {
        uint4* p = reinterpret_cast<uint4*>(bm + (b * kBlockWords - (r0 >> 5))) + lane;
        const uint4 v = *p;
        int c = __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w);
        // 8 lanes hold a sub-block
        constexpr int kSubLanes = kSubCols / 128;
#pragma unroll
        for (int d = 1; d < kSubLanes; d <<= 1) c += __shfl_xor_sync(0xffffffffu, c, d);
        const int64_t sb = b * (kBlockCols / kSubCols) + lane / kSubLanes;
        if (sub && lane % kSubLanes == 0 && sb < nblocks) cnts[sb] = static_cast<uint16_t>(c);
#pragma unroll
        for (int d = kSubLanes; d < 32; d <<= 1) c += __shfl_xor_sync(0xffffffffu, c, d);
        if (lane == 0) {
          if (!sub) cnts[b] = static_cast<uint16_t>(c);
          if (c) atomicAdd(&s_total, static_cast<unsigned long long>(c));
        }
        // a stored row has one window, starting at block 0
        if (wo >= 0) reinterpret_cast<uint4*>(wbits + wo)[b * (kBlockWords / 4) + lane] = v;
        if (v.x | v.y | v.z | v.w) *p = make_uint4(0u, 0u, 0u, 0u);
      }
      __syncthreads();
    }
    // s_total is final (the counting pass ended with a barrier); thread 0 resets it and hands out
    // the next row, which every thread reads after the barrier at the top
    if (threadIdx.x == 0) {
      nnz_row[i] = static_cast<int32_t>(s_total);
      s_total = 0;
      s_idx = next_idx;
    }
  }
}

inline unsigned grid_rows(int64_t count, int rows_per_block, int max_blocks) {
  int64_t g = (count + rows_per_block - 1) / rows_per_block;
  if (g > max_blocks) g = max_blocks;
  if (g < 1) g = 1;
  return static_cast<unsigned>(g);
}

}  // namespace

int launch_sym_tiny(const DevCsr& A, const DevCsr& B, const int32_t* perm, int64_t count,
                     int32_t* nnz_row, int num_sms, cudaStream_t s) {
  if (count <= 0) return 0;
  k_sym_tiny<<<grid_rows(count, 8, num_sms * 64), 256, 0, s>>>(A, B, perm, count, nnz_row);
  return 1;
}

int launch_sym_micro(const DevCsr& A, const DevCsr& B, const int32_t* perm, int64_t count,
                     int32_t* nnz_row, int num_sms, cudaStream_t s) {
  if (count <= 0) return 0;
  k_sym_micro<<<grid_rows(count, 256, num_sms * 16), 256, 0, s>>>(A, B, perm, count, nnz_row);
  return 1;
}

int launch_sym_warp(int log2S, const DevCsr& A, const DevCsr& B, const int32_t* perm,
                     int64_t count, int32_t* nnz_row, uint32_t* err, int num_sms, cudaStream_t s) {
  if (count <= 0) return 0;
  const unsigned g = grid_rows(count, 8, num_sms * 32);
  const size_t sm = size_t(8) << log2S << 2;
  switch (log2S) {
    case 7: k_sym_warp<7><<<g, 256, sm, s>>>(A, B, perm, count, nnz_row, err); break;
    case 9: k_sym_warp<9><<<g, 256, sm, s>>>(A, B, perm, count, nnz_row, err); break;
    case 11:
      cudaFuncSetAttribute(k_sym_warp<11>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(sm));
      k_sym_warp<11><<<g, 256, sm, s>>>(A, B, perm, count, nnz_row, err);
      break;
    default: break;
  }
  return 1;
}

int launch_sym_block(const DevCsr& A, const DevCsr& B, const int32_t* perm, int64_t count, int32_t* nnz_row,
                     const int32_t* abase, int64_t width, uint32_t* err, int num_sms, cudaStream_t s) {
  if (count <= 0) return 0;
  if (width <= kSymBitmapCols) {
    const int words = static_cast<int>((width + 31) / 32);
    auto go = [&](auto kernel, int bytes) {
      kernel<<<grid_rows(count, 1, num_sms * 6), 256, 4 * words + bytes, s>>>(A, B, words, perm, count, nnz_row, abase, err);
    };
    if (width <= kSymByteCols) go(k_sym_bitmap<256, 6, true>, 32 * words);
    else go(k_sym_bitmap<256, 6, false>, 0);
  } else {
    constexpr int kLog2 = 13;
    k_sym_block<kLog2, 512><<<grid_rows(count, 1, num_sms * 8), 512, size_t(4) << kLog2, s>>>(A, B, perm, count,
                                                                                             nnz_row, err);
  }
  return 1;
}

int launch_sym_window(const DevCsr& A, const DevCsr& B, const int32_t* perm, int64_t count,
                       int32_t* counter, int32_t* nnz_row, int32_t* win_slot, uint16_t* blockcnt,
                       int64_t nblocks, int sub, int32_t* cursor, const int32_t* abase, const int32_t* awidth,
                       int64_t width, uint32_t* wbits, int64_t wcap, unsigned long long* wcur, int64_t* woff,
                       int64_t total_products, int64_t max_row_products, int num_sms, uint32_t* err,
                       cudaStream_t s) {
  if (count <= 0) return 0;
  cudaMemsetAsync(counter, 0, sizeof(int32_t), s);
  const int64_t cols = width < kSymWinBits ? width : kSymWinBits;
  const int words = static_cast<int>((cols + kBlockCols - 1) / kBlockCols * kBlockWords);
  // (the limit belongs to the kernel, not to the call: always the most any call needs, as another thread may
  // be about to launch the kernel with more than this call's share)
  auto go = [&](auto kernel, int threads, int blocks, int most_words) {
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 4 * most_words);
    const int64_t g = count < int64_t(num_sms) * blocks ? count : int64_t(num_sms) * blocks;
    kernel<<<static_cast<unsigned>(g), threads, 4 * words, s>>>(A, B, words, perm, count, counter, nnz_row, win_slot,
                                                                blockcnt, nblocks, sub, cursor, abase, awidth, width,
                                                                wbits, wcap, wcur, woff, err);
  };
  // The kernel waits for memory and at its barriers more than on anything else, so as many rows as the
  // bitmaps leave room for are under way per SM. Measured, ms (R-MAT 2^17 with bitmaps of 16 KB, 30,000^2
  // uniform, 4 KB; R-MAT 2^19, 64 KB): one block of 1,024 threads 2.82, 1.95; 19.7. Two of 512: 2.02,
  // 1.50; 13.9. Three of 512: 1.79, 1.43; 12.4. Six of 256: 1.58, 1.32. Eight of 256: 1.78, 1.28.
  // A single row that outweighs an SM's share of the products keeps the larger block, as its block
  // finishes last.
  const int64_t share = 2 * total_products / num_sms;
  if (words <= kSymWinWords6 && max_row_products * 6 <= share) go(k_sym_window<256, 6>, 256, 6, kSymWinWords6);
  else if (words <= kSymWinWords3 && max_row_products * 3 <= share) go(k_sym_window<512, 3>, 512, 3, kSymWinWords3);
  else go(k_sym_window<kSymWinThreads, 1>, kSymWinThreads, 1, kSymWinBits / 32);
  return 1;
}

}  // namespace spg
