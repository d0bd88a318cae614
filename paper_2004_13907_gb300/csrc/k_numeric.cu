// Numeric pass, FP64: forms every partial product a_ik*b_kj of row i (the match
// and multiply unit of Sec. III-A), merges the products of equal column (the merge unit)
// and writes row i of C sorted by column (the sort unit; Algorithm 1 sorts PP and emits
// one entry per column of COLB, including sums that cancel to zero).
//
// Row classes (chosen from nnz(C_i) after the symbolic pass):
//  * tiny  : P_i <= 32: one warp, one product per lane; equal columns are grouped with a
//            warp match and summed by the lowest lane of the group in product order; the
//            output position is the number of smaller columns in the row.
//  * micro, merge : one thread per row of at most 8 entries of A, a merge of the B rows.
//  * warp  : one warp per row, a shared hash table (column -> FP64 sum) of 64/256/1024
//            slots, then the occupied slots are compacted and bitonic-sorted by column.
//  * block : one block per row: bitmaps of the row's columns and a rank-indexed array (rows of at
//            most 2^22 columns), or a hash table of 2048 or 8192 slots, compaction, bitonic sort.
//  * window: rows with more entries than a block table (k_winteam.cu, k_window.cu).
// Sums are accumulated with shared-memory FP64 atomics, so their order (and the last bits of
// a value) can change from run to run; the pattern is always exact.
#include <type_traits>

#include "enumerate.cuh"

namespace spg {

namespace {

template <int Mode>
__global__ void __launch_bounds__(256) k_num_tiny(DevCsr A, DevCsr B, const int32_t* __restrict__ perm,
                                                  int64_t count, const int64_t* __restrict__ c_off,
                                                  int32_t* __restrict__ ccol, void* __restrict__ cval_,
                                                  int32_t* __restrict__ row_flag, const int32_t* __restrict__ abase,
                                                  uint32_t* err) {
  __shared__ int32_t s_col[8][32];
  __shared__ double s_val[8][32];   // FP64 product (kModeF64, kModeF32R) or the FP32 high part
  __shared__ float s_lo[8][32];     // kModeF32C: the FP32 low part of the product
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t gw = (blockIdx.x * int64_t(blockDim.x) + threadIdx.x) >> 5;
  const int64_t nw = (int64_t(gridDim.x) * blockDim.x) >> 5;
  for (int64_t r = gw; r < count; r += nw) {
    const int32_t i = perm[r];
    const int64_t a0 = A.rp[i];
    const int32_t na = static_cast<int32_t>(A.rp[i + 1] - a0);
    int32_t len = 0;
    int64_t bs = 0;
    double av = 0.0;
    if (lane < na) {
      const int32_t k = A.col[a0 + lane];
      av = Mode == kModeF64 ? static_cast<const double*>(A.val)[a0 + lane]
                            : static_cast<double>(static_cast<const float*>(A.val)[a0 + lane]);
      bs = B.rp[k];
      len = static_cast<int32_t>(B.rp[k + 1] - bs);
    }
    const int32_t incl = warp_incl_scan(len);
    const int32_t total = __shfl_sync(0xffffffffu, incl, 31);
    int o = 0;
#pragma unroll
    for (int step = 16; step > 0; step >>= 1) {
      const int32_t v = __shfl_sync(0xffffffffu, incl, o + step - 1);
      if (v <= lane) o += step;
    }
    const int32_t incl_o = __shfl_sync(0xffffffffu, incl, o & 31);
    const int32_t len_o = __shfl_sync(0xffffffffu, len, o & 31);
    const int64_t bs_o = __shfl_sync(0xffffffffu, bs, o & 31);
    const double av_o = __shfl_sync(0xffffffffu, av, o & 31);
    int32_t col = -2 - lane;
    double val = 0.0;
    float lo = 0.f;
    if (lane < total) {
      const int64_t j = bs_o + (lane - (incl_o - len_o));
      col = B.col[j];
      if constexpr (Mode == kModeF64) {
        val = av_o * static_cast<const double*>(B.val)[j];
      } else if constexpr (Mode == kModeF32R) {
        val = av_o * static_cast<double>(static_cast<const float*>(B.val)[j]);   // exact in FP64
      } else {
        const float a = static_cast<float>(av_o);
        const float b = static_cast<const float*>(B.val)[j];
        const float ph = a * b;
        val = ph;
        lo = fmaf(a, b, -ph);   // a*b = ph + lo exactly
      }
    }
    const unsigned peers = __match_any_sync(0xffffffffu, col);
    s_col[wid][lane] = col;
    s_val[wid][lane] = val;
    s_lo[wid][lane] = lo;
    __syncwarp();
    const bool lead = lane < total && (__ffs(peers) - 1) == lane;
    const unsigned leaders = __ballot_sync(0xffffffffu, lead);
    bool missed = false;
    if (lead) {
      int rank = 0;
      for (unsigned m = leaders; m; m &= m - 1) rank += s_col[wid][__ffs(m) - 1] < col;
      if (rank < c_off[i + 1] - c_off[i]) {   // a miscount raises kErrCount, never writes out of the row
        const int64_t out = c_off[i] + rank;
        ccol[out] = col - (abase ? abase[i] : 0);
        if constexpr (Mode == kModeF32C) {
          // compensated sum of the group's products in product order (Dot2)
          float sum = 0.f, comp = 0.f, mag = 0.f;
          int t = 0;
          for (unsigned m = peers; m; m &= m - 1) {
            const int q = __ffs(m) - 1;
            const float ph = static_cast<float>(s_val[wid][q]);
            const float nsum = sum + ph;
            const float bp = nsum - sum;
            comp += (sum - (nsum - bp)) + (ph - bp) + s_lo[wid][q];
            sum = nsum;
            mag += fabsf(ph);
            ++t;
          }
          const float res = sum + comp;
          static_cast<float*>(cval_)[out] = res;
          missed = !f32c_within_bound(res, mag, t);
        } else {
          double sum = 0.0;
          for (unsigned m = peers; m; m &= m - 1) sum += s_val[wid][__ffs(m) - 1];
          if constexpr (Mode == kModeF64) static_cast<double*>(cval_)[out] = sum;
          else static_cast<float*>(cval_)[out] = static_cast<float>(sum);
        }
      }
    }
    if constexpr (Mode == kModeF32C) {
      if (__any_sync(0xffffffffu, missed) && lane == 0) row_flag[i] = 1;
    }
    if (lane == 0 && c_off[i + 1] - c_off[i] != __popc(leaders)) set_error(err, kErrCount);
    __syncwarp();
  }
}

// Micro and merge rows (nnz(A_i) <= kMicroNa, P_i <= maxp <= kMergeMax), FP64: one thread per row merges
// the columns of the row's sorted B rows head by head: the smallest head column is the next column of
// C, and every head holding it advances. The output comes out sorted, with no hash table and no atomics;
// the products of a column are summed in A-entry order.
//
// When the warp's 32 rows follow one another in C and fit `cap` entries (neighbouring rows of a stencil
// do), the merge notes each product's place in its row and the columns are put together in shared memory
// and leave as one run; then each thread takes the values of its B rows one row after the other, adds
// their products at the noted places in shared memory, and the values leave as one run. Other rows
// store from the merge.
//
// Bound by the L1 accesses, each lane's a B row apart. A merge that also read the values went back to
// every B row's values after all the others', beyond what L1 holds for the warps of an SM, and stored
// each lane's entries a row of C apart. 1024^2 five-point stencil (13.6e6 entries) 152 -> 104 us;
// 97^3 seven-point stencil, whose 49 products a row took a 64-slot hash table and a bitonic sort, 1295
// -> 207 us (416 with a merge of columns and values).
constexpr int kMicroWarps = 4;
constexpr int kMicroStaged = 8;   // mean entries of a row from which they are staged
__host__ __device__ constexpr int micro_warp_bytes(int cap, int maxp) { return cap * 8 + maxp * 32; }
// Entries staged per warp for rows of `mean` entries (at most kMergeMax).
constexpr int micro_cap(int64_t mean) { return static_cast<int>((32 * mean + 2 * mean + 31) & ~int64_t(31)); }

// The first U products (of the `m` there are, possibly none) of one B row at bv, times av, added at
// their places in the row of `len` entries at dval. The places of one B row's products differ, so all
// are loaded before any is added.
template <int U>
__device__ __forceinline__ void add_head(const double* __restrict__ bv, int32_t m, double av, const uint8_t* place,
                                         double* dval, int len) {
  double v[U], x[U];
  int t[U];
#pragma unroll
  for (int u = 0; u < U; ++u) v[u] = u < m ? bv[u] : 0.0;
#pragma unroll
  for (int u = 0; u < U; ++u) {
    t[u] = u < m ? place[u * 32] : len;
    x[u] = t[u] < len ? dval[t[u]] : 0.0;
  }
#pragma unroll
  for (int u = 0; u < U; ++u)
    if (t[u] < len) dval[t[u]] = x[u] + av * v[u];
}

// The rows of a warp, at most `most` <= NA entries of A in any of them (na: this lane's row's).
template <int NA, bool Staged>
__device__ __forceinline__ void micro_rows(const DevCsr& A, const DevCsr& B, unsigned char* mem, int cap, int maxp,
                                           int64_t a0, int na, int most, int64_t off, int len, int32_t cb,
                                           bool mine,
                                           int32_t* __restrict__ ccol, double* __restrict__ cval, uint32_t* err) {
  constexpr int32_t kEnd = 0x7fffffff;
  const int lane = threadIdx.x & 31;
  double* sval = reinterpret_cast<double*>(mem);       // the warp's values, after
  int32_t* scol = reinterpret_cast<int32_t*>(mem);     //   its columns
  uint8_t* place = mem + cap * 8 + lane;               // [product * 32]: its place in the lane's row
  const double* av64 = static_cast<const double*>(A.val);
  const double* bv64 = static_cast<const double*>(B.val);
  // products numbered head by head: head h holds numbers [q[h], qe[h]), product q is entry q + at[h] of B
  int64_t at[NA];
  int32_t q[NA], qe[NA], hc[NA];
  int32_t products = 0;
#pragma unroll
  for (int h = 0; h < NA; ++h) {
    at[h] = 0;
    qe[h] = 0;
    if (h < na) {
      const int32_t k = A.col[a0 + h];
      at[h] = B.rp[k];
      qe[h] = static_cast<int32_t>(B.rp[k + 1] - at[h]);
    }
  }
#pragma unroll
  for (int h = 0; h < NA; ++h) {
    hc[h] = qe[h] > 0 ? B.col[at[h]] : kEnd;
    q[h] = products;
    at[h] -= products;
    products += qe[h];
    qe[h] = products;
  }
  const int incl = warp_incl_scan(len);
  const int total = __shfl_sync(0xffffffffu, incl, 31);
  const int64_t off0 = __shfl_sync(0xffffffffu, off, 0);
  const bool staged =
      Staged && total <= cap && __all_sync(0xffffffffu, products <= maxp && (!mine || off == off0 + (incl - len)));
  int n = 0;
  if (staged) {
    int32_t* dcol = scol + (incl - len);
    for (;;) {
      int32_t m = hc[0];
#pragma unroll
      for (int h = 1; h < NA; ++h) m = min(m, hc[h]);
      if (m == kEnd) break;
#pragma unroll
      for (int h = 0; h < NA; ++h) {
        if (hc[h] == m) {
          place[q[h] * 32] = static_cast<uint8_t>(n);
          ++q[h];
          hc[h] = q[h] < qe[h] ? B.col[at[h] + q[h]] : kEnd;
        }
      }
      if (n < len) dcol[n] = m - cb;   // a miscount raises kErrCount, never writes out of the row
      ++n;
    }
    __syncwarp();
    for (int t = lane; t < total; t += 32) ccol[off0 + t] = scol[t];
    __syncwarp();
    for (int t = lane; t < total; t += 32) sval[t] = 0.0;
    __syncwarp();
    double* dval = sval + (incl - len);
    // the heads one after the other; the longest of the warp's B rows sets how many values are loaded
    // together
    int32_t p = 0;
    int32_t k = na > 0 ? A.col[a0] : 0;
    for (int h = 0; h < most; ++h) {
      const bool has = h < na;
      const double av = has ? av64[a0 + h] : 0.0;
      const int64_t s = has ? B.rp[k] : 0;
      const int32_t m = has ? static_cast<int32_t>(B.rp[k + 1] - s) : 0;
      if (h + 1 < na) k = A.col[a0 + h + 1];
      const int longest = __reduce_max_sync(0xffffffffu, m);
      const uint8_t* pl = place + p * 32;
      if (longest <= 1) add_head<1>(bv64 + s, m, av, pl, dval, len);
      else if (longest <= 3) add_head<3>(bv64 + s, m, av, pl, dval, len);
      else if (longest <= 5) add_head<5>(bv64 + s, m, av, pl, dval, len);
      else
        for (int32_t t = 0; t < longest; t += 8) add_head<8>(bv64 + s + t, m - t, av, pl + t * 32, dval, len);
      p += m;
    }
    __syncwarp();
    for (int t = lane; t < total; t += 32) cval[off0 + t] = sval[t];
    __syncwarp();
  } else {
    double av[NA];
#pragma unroll
    for (int h = 0; h < NA; ++h) av[h] = h < na ? av64[a0 + h] : 0.0;
    for (;;) {
      int32_t m = hc[0];
#pragma unroll
      for (int h = 1; h < NA; ++h) m = min(m, hc[h]);
      if (m == kEnd) break;
      double sum = 0.0;
#pragma unroll
      for (int h = 0; h < NA; ++h) {
        if (hc[h] == m) {
          sum += av[h] * bv64[at[h] + q[h]];
          ++q[h];
          hc[h] = q[h] < qe[h] ? B.col[at[h] + q[h]] : kEnd;
        }
      }
      if (n < len) {
        ccol[off + n] = m - cb;
        cval[off + n] = sum;
      }
      ++n;
    }
  }
  if (n != len) set_error(err, kErrCount);
}

// Staged: with room for the warps' rows in shared memory; else every row is stored from the merge.
template <bool Staged>
__global__ void __launch_bounds__(kMicroWarps * 32, Staged ? 6 : 8) k_num_micro(DevCsr A, DevCsr B, const int32_t* __restrict__ perm,
                                                   int64_t count, int cap, int maxp, const int64_t* __restrict__ c_off,
                                                   int32_t* __restrict__ ccol, double* __restrict__ cval,
                                                   const int32_t* __restrict__ abase, uint32_t* err) {
  extern __shared__ double smem_f64[];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  unsigned char* mem = reinterpret_cast<unsigned char*>(smem_f64) + wid * micro_warp_bytes(cap, maxp);
  const int64_t stride = int64_t(gridDim.x) * blockDim.x;
  for (int64_t r0 = blockIdx.x * int64_t(blockDim.x) + wid * 32; r0 < count; r0 += stride) {
    const bool mine = r0 + lane < count;
    const int32_t i = perm[mine ? r0 + lane : r0];
    const int64_t a0 = A.rp[i];
    const int na = mine ? static_cast<int>(A.rp[i + 1] - a0) : 0;
    const int64_t off = c_off[i];
    const int len = mine ? static_cast<int>(c_off[i + 1] - off) : 0;
    const int32_t cb = abase ? abase[i] : 0;
    const int most = __reduce_max_sync(0xffffffffu, na);   // heads no row of the warp has are left out
    if (most <= 5) micro_rows<5, Staged>(A, B, mem, cap, maxp, a0, na, most, off, len, cb, mine, ccol, cval, err);
    else if (most <= 7) micro_rows<7, Staged>(A, B, mem, cap, maxp, a0, na, most, off, len, cb, mine, ccol, cval, err);
    else micro_rows<kMicroNa, Staged>(A, B, mem, cap, maxp, a0, na, most, off, len, cb, mine, ccol, cval, err);
  }
}

// Value q of an FP64 (kModeF64) or FP32 (kModeF32C) array, as a double (exact).
template <int Mode>
__device__ __forceinline__ double value_at(const void* v, int64_t q) {
  if constexpr (Mode == kModeF32C) return static_cast<double>(static_cast<const float*>(v)[q]);
  else return static_cast<const double*>(v)[q];
}

// The slot of `key` (linear probing; keys are columns, kEmpty = free), claimed if new; -1 when
// the table is full.
template <int LOG2S>
__device__ __forceinline__ int hash_claim(int32_t* keys, int32_t key) {
  constexpr int S = 1 << LOG2S;
  uint32_t h = hash_slot(key, LOG2S);
  for (int probe = 0; probe < S; ++probe) {
    const int32_t cur = *reinterpret_cast<volatile int32_t*>(&keys[h]);
    if (cur == key) return static_cast<int>(h);
    if (cur == kEmpty) {
      const int32_t old = atomicCAS(&keys[h], kEmpty, key);
      if (old == kEmpty || old == key) return static_cast<int>(h);
    }
    h = (h + 1) & (S - 1);
  }
  return -1;
}

// Adds fa*fb into an FP32 sum sc[0] and its compensation sc[1]: the error-free product fa*fb = ph
// + pl, and the sum's own rounding error (TwoSum) rebuilt from the value the atomic returns.
__device__ __forceinline__ void add_compensated(float* sc, float fa, float fb) {
  const float ph = fa * fb;
  const float pl = fmaf(fa, fb, -ph);
  const float old = atomicAdd(&sc[0], ph);
  const float nw = old + ph;
  const float bp = nw - old;
  const float q = (old - (nw - bp)) + (ph - bp);
  atomicAdd(&sc[1], q + pl);
}

// Adds the partial product a*b into the slot of `key`. kModeF64: one FP64 atomic. kModeF32C: the
// slot's 8 bytes hold an FP32 sum and its compensation; the error-free product a*b = ph + pl and
// the sum's own rounding error (TwoSum, rebuilt from the value the atomic returns) go to the
// compensation, as in the windowed kernel (Dot2 accumulated concurrently).
template <int LOG2S, int Mode>
__device__ __forceinline__ void hash_accumulate(int32_t* keys, double* vals, int32_t key, double a, double b,
                                                uint32_t* err) {
  const int h = hash_claim<LOG2S>(keys, key);
  if (h < 0) {
    set_error(err, kErrHashFull);
    return;
  }
  if constexpr (Mode == kModeF32C) {
    add_compensated(reinterpret_cast<float*>(&vals[h]), static_cast<float>(a), static_cast<float>(b));
  } else {
    atomicAdd(&vals[h], a * b);
  }
}

// Value of an entry of C from its slot's 8 bytes (an FP64 sum, or an FP32 sum and compensation).
template <int Mode>
__device__ __forceinline__ void store_value(void* cval, int64_t at, double slot) {
  if constexpr (Mode == kModeF32C) {
    const float2 sc = *reinterpret_cast<const float2*>(&slot);
    static_cast<float*>(cval)[at] = sc.x + sc.y;
  } else {
    static_cast<double*>(cval)[at] = slot;
  }
}

// kModeF32C rows of the hash kernels: every partial product must be non-negative (no negative value
// in A or B, *negflag == 0) and the row's A length must pass the term-count bound, so that no
// entry can exceed Dot2's bound; otherwise the row is listed for the FP64 recomputation.
__device__ __forceinline__ bool f32c_hash_row_ok(const int32_t* negflag, int64_t na) {
  return negflag != nullptr && *negflag == 0 &&
         f32c_within_count(na < (int64_t(1) << 30) ? static_cast<int>(na) : (1 << 30));
}

// In-warp bitonic sort of keys/vals[0, N), N a power of two.
__device__ __forceinline__ void warp_bitonic(int32_t* keys, double* vals, int N) {
  const int lane = threadIdx.x & 31;
  for (int k = 2; k <= N; k <<= 1) {
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int t = lane; t < (N >> 1); t += 32) {
        const int a = ((t / j) * 2 * j) + (t % j);
        const int b = a + j;
        const bool up = (a & k) == 0;
        const int32_t ka = keys[a], kb = keys[b];
        if ((ka > kb) == up) {
          keys[a] = kb; keys[b] = ka;
          const double va = vals[a]; vals[a] = vals[b]; vals[b] = va;
        }
      }
      __syncwarp();
    }
  }
}

template <int NT>
__device__ __forceinline__ void block_bitonic(int32_t* keys, double* vals, int N) {
  for (int k = 2; k <= N; k <<= 1) {
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int t = threadIdx.x; t < (N >> 1); t += NT) {
        const int a = ((t / j) * 2 * j) + (t % j);
        const int b = a + j;
        const bool up = (a & k) == 0;
        const int32_t ka = keys[a], kb = keys[b];
        if ((ka > kb) == up) {
          keys[a] = kb; keys[b] = ka;
          const double va = vals[a]; vals[a] = vals[b]; vals[b] = va;
        }
      }
      __syncthreads();
    }
  }
}

__device__ __forceinline__ int pow2_ceil(int x) {
  return x <= 1 ? 1 : 1 << (32 - __clz(x - 1));
}

template <int LOG2S, int Mode>
__global__ void __launch_bounds__(256) k_num_warp(DevCsr A, DevCsr B, const int32_t* __restrict__ perm,
                                                  int64_t count, const int64_t* __restrict__ c_off,
                                                  int32_t* __restrict__ ccol, void* __restrict__ cval,
                                                  const int32_t* __restrict__ abase, int32_t* __restrict__ row_flag,
                                                  const int32_t* __restrict__ negflag, uint32_t* err) {
  constexpr int S = 1 << LOG2S;
  extern __shared__ double smem_f64[];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  double* vals = smem_f64 + wid * S;
  int32_t* keys = reinterpret_cast<int32_t*>(smem_f64 + 8 * S) + wid * S;
  const int64_t gw = (blockIdx.x * int64_t(blockDim.x) + threadIdx.x) >> 5;
  const int64_t nw = (int64_t(gridDim.x) * blockDim.x) >> 5;
  for (int64_t r = gw; r < count; r += nw) {
    const int32_t i = perm[r];
    const int64_t a0 = A.rp[i];
    const int64_t na = A.rp[i + 1] - a0;
    if (Mode == kModeF32C && lane == 0 && !f32c_hash_row_ok(negflag, na)) row_flag[i] = 1;
    for (int s = lane; s < S; s += 32) { keys[s] = kEmpty; vals[s] = 0.0; }
    __syncwarp();
    warp_for_each_product(A, B, a0, na, [&](int64_t j, int64_t e) {
      hash_accumulate<LOG2S, Mode>(keys, vals, B.col[j], value_at<Mode>(A.val, a0 + e), value_at<Mode>(B.val, j),
                                   err);
    });
    __syncwarp();
    // compact in place (a write position never passes the slot being read)
    int cnt = 0;
    for (int base = 0; base < S; base += 32) {
      const int32_t k = keys[base + lane];
      const double v = vals[base + lane];
      const bool occ = k != kEmpty;
      const unsigned b = __ballot_sync(0xffffffffu, occ);
      const int pos = cnt + __popc(b & ((1u << lane) - 1u));
      __syncwarp();
      if (occ) { keys[pos] = k; vals[pos] = v; }
      cnt += __popc(b);
      __syncwarp();
    }
    const int64_t off = c_off[i];
    const int64_t len = c_off[i + 1] - off;
    if (lane == 0 && len != cnt) set_error(err, kErrCount);
    const int N = pow2_ceil(cnt);
    for (int t = cnt + lane; t < N; t += 32) keys[t] = kNoCol;
    __syncwarp();
    warp_bitonic(keys, vals, N);
    const int nw_out = cnt < len ? cnt : static_cast<int>(len);
    const int32_t cb = abase ? abase[i] : 0;
    for (int t = lane; t < nw_out; t += 32) {
      ccol[off + t] = keys[t] - cb;
      store_value<Mode>(cval, off + t, vals[t]);
    }
    __syncwarp();
  }
}

// Block rows of a column space of at most kBitmapMaxWidth columns: no hash table and no sort. The
// row's columns are kept as a bitmap of 32-column words, dense when all the row's words fit `cap`
// (its table of words), else in two levels: a coarse bit per word of the row, whose prefix count
// numbers the words that hold a column (at most one per entry of C, so they fit the table). The
// prefix count over the words gives every column its rank, the products are added into a
// rank-indexed array and the row leaves in rank order.
//
// A row whose products fit the block's registers (kHeld per thread, one chunk of A entries) reads
// B once: its columns and products stay in registers between the marking and the accumulation.
// Longer rows enumerate their products in each pass.
//
// Bound by the latency of the gathers and the barriers between the passes. 256 threads with 64
// registers, so that four rows are in flight on an SM; the hash table and bitonic sort of
// k_num_block are bound by the sort's shared-memory traffic instead. Both block classes, hash
// and bitonic sort -> bitmaps: 20,000^2 uniform (19,400 rows of 1,540 entries) 3.83 -> 0.36 ms,
// R-MAT 2^17 2.67 -> 0.46 ms, R-MAT 2^19 7.87 -> 1.19 ms. Columns stored by the products (Direct): 20,000^2
// 0.355 -> 0.30 ms.
//
// Rows of many products per entry are bound by the enumerations, two or three of them, where the hash table needs
// one. A class of such rows by its mean (kManyProducts) takes instances of its own (Many), whose rows find
// their first and last column, from the ends of their B rows. Within `span` columns a row adds each product
// at its column, in one enumeration, and a byte per column says which were reached; else its words are
// numbered from its first column on, so that a band of a wide column space needs one level only. Numeric
// pass, ms, hash table / ranks / this: 30,000 rows of 1,000 entries in bands of a 300,000 column space, 8
// products per entry 2.91, 3.13, 1.35, 124 per entry 18.3, 39.4, 16.3; 70,000 rows of all 1,000 columns, 85
// per entry 31.5, 36.1, 28.3. 20,000 rows of 900 scattered columns of 300,000, 35 per entry: 10.6, 5.7, 6.0 (two
// levels). In FP32 the table's scattered rows are as fast from about 32 per entry on (5.97, 5.88; 14.2 and 15.7
// with 100): two levels hash from there.
constexpr int kManyProducts = 4, kManyProductsF32 = 32;
constexpr int kSpan = 4096;
constexpr int kHeld = 8;   // products per thread held in registers
constexpr int kStep = 4;   // products per thread in one step (loads in flight)
constexpr int64_t kBitmapMaxWidth = int64_t(1) << 22;   // coarse words: 16 KB

// Coarse words a block keeps: none when every row's words fit the table of `cap` words.
__host__ __device__ constexpr int bitmap_coarse_words(int64_t width, int cap) {
  const int64_t words = (width + 31) >> 5;
  return words <= cap ? 0 : static_cast<int>((words + 31) >> 5);
}

// Shared bytes of a block with `cap` entries of C and word-table words: one level (the words of the column
// space, which fit), and two with `coarse` coarse words.
// With `span`, room for a sum and a byte per column of that many.
constexpr size_t bitmap_bytes_direct(int cap, int64_t width, int span) {
  return size_t(cap > span ? cap : span) * 8 + size_t(cap) * 2 + size_t((width + 31) / 32) * (4 + 2) + span;
}
constexpr size_t bitmap_bytes(int cap, int coarse, int span) {
  return size_t(2 * cap > span ? 2 * cap : span) * 8 + size_t(cap) * (4 + 2) + size_t(coarse) * 6 + span;
}

template <int NT>
struct BitmapChunk {
  int64_t bs[NT];        // per non-empty B row of the chunk: its start in B,
  double av[NT];         //   a_ik,
  int32_t excl[NT + 1];  //   its first product's number (and the total last)
  long long scan64[33];
  int32_t scan[33];
  int32_t ctl[2];        // segments, products
};

// The A entries [base, base + NT) of the row, their non-empty B rows compacted into ck.
template <int NT, int Mode>
__device__ __forceinline__ void bitmap_chunk(const DevCsr& A, const DevCsr& B, int64_t a0, int64_t na, int64_t base,
                                             BitmapChunk<NT>& ck) {
  const int64_t e = base + threadIdx.x;
  int64_t bs = 0;
  int32_t len = 0;
  double av = 0.0;
  if (e < na) {
    const int32_t k = A.col[a0 + e];
    av = value_at<Mode>(A.val, a0 + e);
    bs = B.rp[k];
    len = static_cast<int32_t>(B.rp[k + 1] - bs);
  }
  const long long packed = (static_cast<long long>(len > 0) << 32) | static_cast<long long>(len);
  long long tot;
  const long long ex = block_excl_scan<long long>(packed, ck.scan64, &tot);
  if (len > 0) {
    const int pos = static_cast<int>(ex >> 32);
    ck.bs[pos] = bs;
    ck.av[pos] = av;
    ck.excl[pos] = static_cast<int32_t>(ex & 0xffffffffLL);
  }
  if (threadIdx.x == 0) {
    ck.ctl[0] = static_cast<int32_t>(tot >> 32);
    ck.ctl[1] = static_cast<int32_t>(tot & 0xffffffffLL);
    ck.excl[ck.ctl[0]] = ck.ctl[1];
  }
  __syncthreads();
}

// The chunk's products, one contiguous range per warp, kStep groups of 32 per call: f(q, j, av)
// with kStep indices into B (-1: none) and their a_ik, q the call's number (of a chunk that fits the
// registers: below kHeld / kStep, and known at compile time; else 0).
template <int NT, typename F>
__device__ __forceinline__ void bitmap_for_each(const BitmapChunk<NT>& ck, bool fits, F&& f) {
  const int wid = threadIdx.x >> 5;
  const int nent = ck.ctl[0];
  const int32_t total = ck.ctl[1];
  int32_t per = (total + NT / 32 - 1) / (NT / 32);
  per = (per + 31) & ~31;
  const int32_t lo = wid * per;
  const int32_t hi = total < lo + per ? total : lo + per;
  if (lo >= hi) return;
  auto walk = make_walker<double>(ck.excl, ck.bs, nent, search_owner(ck.excl, nent, lo),
                                  [&](int sgm) { return ck.av[sgm]; });
  int64_t j[kStep];
  double av[kStep];
  if (fits) {
#pragma unroll
    for (int q = 0; q < kHeld / kStep; ++q) {
      const int32_t p0 = lo + q * 32 * kStep;
      if (p0 < hi) {
        walk.template step_many<kStep>(p0, hi, j, av);
        f(q, j, av);
      }
    }
  } else {
    for (int32_t p0 = lo; p0 < hi; p0 += 32 * kStep) {
      walk.template step_many<kStep>(p0, hi, j, av);
      f(0, j, av);
    }
  }
}

// pre[w] = bits set in words[0, w); returns the number of bits set in words[0, n). Each thread
// takes a run of consecutive words. Ends with a barrier.
template <int NT>
__device__ __forceinline__ int bitmap_prefix(const uint32_t* words, uint16_t* pre, int n, int32_t* scan) {
  const int k = (n + NT - 1) / NT;
  const int lo = min(n, static_cast<int>(threadIdx.x) * k), hi = min(n, lo + k);
  int c = 0;
  for (int w = lo; w < hi; ++w) c += __popc(words[w]);
  int32_t total;
  int run = block_excl_scan<int32_t>(c, scan, &total);
  for (int w = lo; w < hi; ++w) {
    pre[w] = static_cast<uint16_t>(min(run, 65535));
    run += __popc(words[w]);
  }
  __syncthreads();
  return total;
}

// One partial product in eight bytes: a*b (kModeF64) or the FP32 pair (a, b) (kModeF32C).
template <int Mode>
__device__ __forceinline__ double held_product(double a, double b) {
  if constexpr (Mode == kModeF32C) {
    const float2 ab = make_float2(static_cast<float>(a), static_cast<float>(b));
    return *reinterpret_cast<const double*>(&ab);
  } else {
    return a * b;
  }
}

// Adds a held product into an eight-byte slot (the modes of hash_accumulate).
template <int Mode>
__device__ __forceinline__ void add_held(double* slot, double held) {
  if constexpr (Mode == kModeF32C) {
    const float2 ab = *reinterpret_cast<const float2*>(&held);
    add_compensated(reinterpret_cast<float*>(slot), ab.x, ab.y);
  } else {
    atomicAdd(slot, held);
  }
}

// Direct: every word of the column space fits the table, and a column 16 bits, so that a product stores
// its column at its rank and no pass walks the bits. Many: rows of many products per entry look for their
// ends (span > 0).
template <int NT, int Mode, bool Direct, bool Many>
__global__ void __launch_bounds__(NT, 1024 / NT) k_num_bitmap(DevCsr A, DevCsr B, const int32_t* __restrict__ perm,
                                                     int64_t count, const int64_t* __restrict__ c_off,
                                                     int32_t* __restrict__ ccol, void* __restrict__ cval,
                                                     const int32_t* __restrict__ abase,
                                                     const int32_t* __restrict__ awidth, int64_t width_all, int cap,
                                                     int span, int32_t* __restrict__ row_flag,
                                                     const int32_t* __restrict__ negflag, uint32_t* err) {
  extern __shared__ double smem_f64[];
  __shared__ BitmapChunk<NT> ck;
  __shared__ uint32_t s_ends[2];                                    // a row's first and last column
  double* vals = smem_f64;                                          // [cap] by rank, or [span] by column
  const int table = Direct ? (static_cast<int>(width_all) + 31) >> 5 : cap;   // words of the word table
  const int coarse_all = Direct ? 0 : bitmap_coarse_words(width_all, cap);
  int32_t* gword = reinterpret_cast<int32_t*>(vals + cap);          // [cap], two levels: word number of a table word
  int32_t* colbuf = gword + cap;                                    // [cap], two levels: the columns by rank
  uint32_t* fine = reinterpret_cast<uint32_t*>(vals + max(Direct ? cap : 2 * cap, span));   // [table], the word
                                                                    //   table (zero between rows)
  uint32_t* coarse = fine + table;                                  // a bit per word (zero between rows)
  uint16_t* fpre = reinterpret_cast<uint16_t*>(coarse + coarse_all);   // [table]
  uint16_t* cpre = fpre + table;                                    // [coarse_all]
  uint16_t* cols = cpre;                                            // [cap], Direct: the columns by rank
  uint8_t* reached = reinterpret_cast<uint8_t*>(Direct ? cols + cap : cpre + coarse_all);   // [span], by column
  for (int t = threadIdx.x; t < table + coarse_all; t += NT) fine[t] = 0u;
  for (int64_t r = blockIdx.x; r < count; r += gridDim.x) {
    const int32_t i = perm[r];
    const int64_t a0 = A.rp[i];
    const int64_t na = A.rp[i + 1] - a0;
    const int64_t off = c_off[i];
    const int64_t len = c_off[i + 1] - off;
    int32_t cb = abase ? abase[i] : 0;   // the row's columns are [cb, cb + width)
    uint32_t width = static_cast<uint32_t>(awidth ? awidth[i] : width_all);
    int words = static_cast<int>((width + 31) >> 5);
    bool direct = Direct || words <= cap;   // (a narrower job of a batch may fit where the widest does not)
    int32_t first = 0;                      // the column of the row's space at cb
    bool by_column = false;
    if (Mode == kModeF32C && threadIdx.x == 0 && !f32c_hash_row_ok(negflag, na)) row_flag[i] = 1;
    if (Many && threadIdx.x == 0) {
      s_ends[0] = 0xffffffffu;
      s_ends[1] = 0u;
    }
    __syncthreads();   // (also: the previous row's clearing of the bitmaps)
    // the table word of column rel (two levels), -1 past the table (a row counted otherwise)
    auto table_word = [&](uint32_t rel) {
      const uint32_t cw = coarse[rel >> 10];
      const int g = cpre[rel >> 10] + __popc(cw & ((1u << ((rel >> 5) & 31)) - 1u));
      return g < cap ? g : -1;
    };
    // held: per product of the step its table word * 32 + bit, -1 for none; of a held row only
    int32_t held[kHeld];
    double pv[kHeld];
    bool bad = false, keep = false;
    // pass 1: the words (one level) or the coarse bits of the row's columns
    for (int64_t base = 0; base < na; base += NT) {
      bitmap_chunk<NT, Mode>(A, B, a0, na, base, ck);
      keep = na <= NT && ck.ctl[1] <= NT * kHeld;
      if (Many && base == 0 && !keep) {
        uint32_t lo = 0xffffffffu, hi = 0u;
        for (int64_t e = threadIdx.x; e < na; e += NT) {
          const int32_t k = A.col[a0 + e];
          const int64_t s = B.rp[k], t = B.rp[k + 1];
          if (s < t) {
            lo = min(lo, static_cast<uint32_t>(B.col[s] - cb));
            hi = max(hi, static_cast<uint32_t>(B.col[t - 1] - cb));
          }
        }
        lo = __reduce_min_sync(0xffffffffu, lo);
        hi = __reduce_max_sync(0xffffffffu, hi);
        if ((threadIdx.x & 31) == 0) {
          atomicMin(&s_ends[0], lo);
          atomicMax(&s_ends[1], hi);
        }
        __syncthreads();
        lo = s_ends[0] & ~31u;
        hi = s_ends[1];
        if (lo <= hi && hi < width) {   // (else a column outside the row's space: reported below)
          first = static_cast<int32_t>(lo);
          cb += first;
          width = hi - lo + 1;
          words = static_cast<int>((width + 31) >> 5);
          direct = Direct || words <= cap;
          by_column = width <= static_cast<uint32_t>(span);
        }
        if (by_column) {
          for (int t = threadIdx.x; t < words * 32; t += NT) {
            if (t < span) reached[t] = 0;
            if (t < static_cast<int>(width)) vals[t] = 0.0;
          }
          __syncthreads();
        }
      }
      if (Many && by_column) {
        bitmap_for_each<NT>(ck, false, [&](int, const int64_t (&j)[kStep], const double (&av)[kStep]) {
          int32_t c[kStep];
          double p[kStep];
#pragma unroll
          for (int u = 0; u < kStep; ++u) {
            c[u] = j[u] >= 0 ? B.col[j[u]] : 0;
            p[u] = j[u] >= 0 ? held_product<Mode>(av[u], value_at<Mode>(B.val, j[u])) : 0.0;
          }
#pragma unroll
          for (int u = 0; u < kStep; ++u) {
            if (j[u] < 0) continue;
            const uint32_t rel = static_cast<uint32_t>(c[u] - cb);
            if (rel >= width) { bad = true; continue; }
            reached[rel] = 1;
            add_held<Mode>(&vals[rel], p[u]);
          }
        });
        __syncthreads();
        continue;
      }
#pragma unroll
      for (int u = 0; u < kHeld; ++u) held[u] = -1;
      bitmap_for_each<NT>(ck, keep, [&](int q, const int64_t (&j)[kStep], const double (&av)[kStep]) {
        int32_t c[kStep];
#pragma unroll
        for (int u = 0; u < kStep; ++u) c[u] = j[u] >= 0 ? B.col[j[u]] : 0;
        if (keep) {
#pragma unroll
          for (int u = 0; u < kStep; ++u)
            pv[q * kStep + u] = j[u] >= 0 ? held_product<Mode>(av[u], value_at<Mode>(B.val, j[u])) : 0.0;
        }
#pragma unroll
        for (int u = 0; u < kStep; ++u) {
          if (j[u] < 0) continue;
          const uint32_t rel = static_cast<uint32_t>(c[u] - cb);
          if (rel >= width) { bad = true; continue; }
          if (direct) atomicOr(&fine[rel >> 5], 1u << (rel & 31));
          else atomicOr(&coarse[rel >> 10], 1u << ((rel >> 5) & 31));
          held[q * kStep + u] = static_cast<int32_t>(rel);
        }
      });
      __syncthreads();
    }
    if (Many && by_column) {
      const int lane = threadIdx.x & 31;
      for (int w = threadIdx.x >> 5; w < words; w += NT / 32) {
        const uint32_t t = w * 32 + lane;
        const unsigned bits = __ballot_sync(0xffffffffu, t < width && reached[t]);
        if (lane == 0) fine[w] = bits;
      }
      __syncthreads();
      const int cnt = bitmap_prefix<NT>(fine, fpre, words, ck.scan);
      if (cnt != len) bad = true;
      for (uint32_t t = threadIdx.x; t < width; t += NT) {
        const uint32_t bits = fine[t >> 5];
        const int rk = fpre[t >> 5] + __popc(bits & ((1u << (t & 31)) - 1u));
        if ((bits >> (t & 31) & 1u) && rk < len) {
          ccol[off + rk] = first + static_cast<int32_t>(t);
          store_value<Mode>(cval, off + rk, vals[t]);
        }
      }
      __syncthreads();
      for (int w = threadIdx.x; w < words; w += NT) fine[w] = 0u;
      if (bad) set_error(err, kErrCount);
      continue;
    }
    int nwords = words;
    const int cwords = (words + 31) >> 5;
    if (!direct) {
      const int groups = bitmap_prefix<NT>(coarse, cpre, cwords, ck.scan);
      nwords = groups < cap ? groups : cap;
      for (int w = threadIdx.x; w < cwords; w += NT) {
        int g = cpre[w];
        for (uint32_t m = coarse[w]; m; m &= m - 1, ++g)
          if (g < cap) gword[g] = w * 32 + __ffs(m) - 1;
      }
      // pass 2: the table words
      if (keep) {
#pragma unroll
        for (int u = 0; u < kHeld; ++u) {
          if (held[u] < 0) continue;
          const int g = table_word(held[u]);
          const int bit = held[u] & 31;
          if (g >= 0) atomicOr(&fine[g], 1u << bit);
          held[u] = g >= 0 ? g * 32 + bit : -1;
        }
      } else {
        for (int64_t base = 0; base < na; base += NT) {
          bitmap_chunk<NT, Mode>(A, B, a0, na, base, ck);
          bitmap_for_each<NT>(ck, false, [&](int, const int64_t (&j)[kStep], const double (&)[kStep]) {
            int32_t c[kStep];
#pragma unroll
            for (int u = 0; u < kStep; ++u) c[u] = j[u] >= 0 ? B.col[j[u]] : 0;
#pragma unroll
            for (int u = 0; u < kStep; ++u) {
              const uint32_t rel = static_cast<uint32_t>(c[u] - cb);
              if (j[u] < 0 || rel >= width) continue;
              const int g = table_word(rel);
              if (g >= 0) atomicOr(&fine[g], 1u << (rel & 31));
            }
          });
          __syncthreads();
        }
      }
      __syncthreads();
    }
    const int cnt = bitmap_prefix<NT>(fine, fpre, nwords, ck.scan);
    const int n_out = cnt < len ? min(cnt, cap) : static_cast<int>(min(len, static_cast<int64_t>(cap)));
    if (cnt != len) bad = true;
    for (int t = threadIdx.x; t < n_out; t += NT) vals[t] = 0.0;
    __syncthreads();
    // pass 3: the products by rank
    auto add = [&](int g, int bit, double p) {
      const int rk = fpre[g] + __popc(fine[g] & ((1u << bit) - 1u));
      if (rk < n_out) {
        if constexpr (Direct) cols[rk] = static_cast<uint16_t>(g * 32 + bit);   // every product of the column the same
        add_held<Mode>(&vals[rk], p);
      }
    };
    if (keep) {
#pragma unroll
      for (int u = 0; u < kHeld; ++u)
        if (held[u] >= 0) add(held[u] >> 5, held[u] & 31, pv[u]);
      __syncthreads();
    } else {
      for (int64_t base = 0; base < na; base += NT) {
        bitmap_chunk<NT, Mode>(A, B, a0, na, base, ck);
        bitmap_for_each<NT>(ck, false, [&](int, const int64_t (&j)[kStep], const double (&av)[kStep]) {
          int32_t c[kStep];
          double p[kStep];
#pragma unroll
          for (int u = 0; u < kStep; ++u) {
            c[u] = j[u] >= 0 ? B.col[j[u]] : 0;
            p[u] = j[u] >= 0 ? held_product<Mode>(av[u], value_at<Mode>(B.val, j[u])) : 0.0;
          }
#pragma unroll
          for (int u = 0; u < kStep; ++u) {
            const uint32_t rel = static_cast<uint32_t>(c[u] - cb);
            if (j[u] < 0 || rel >= width) continue;
            const int g = direct ? static_cast<int>(rel >> 5) : table_word(rel);
            if (g >= 0) add(g, rel & 31, p[u]);
          }
        });
        __syncthreads();
      }
    }
    // the columns by rank, and the bitmaps cleared for the next row
    if constexpr (Direct) {
      for (int w = threadIdx.x; w < nwords; w += NT) fine[w] = 0u;
    } else {
      for (int w = threadIdx.x; w < nwords; w += NT) {
        uint32_t m = fine[w];
        if (!m) continue;
        const int col0 = first + 32 * (direct ? w : gword[w]);
        for (int rk = fpre[w]; m; m &= m - 1, ++rk)
          if (rk < n_out) colbuf[rk] = col0 + __ffs(m) - 1;
        fine[w] = 0u;
      }
      if (!direct)
        for (int w = threadIdx.x; w < cwords; w += NT) coarse[w] = 0u;
      __syncthreads();
    }
    for (int t = threadIdx.x; t < n_out; t += NT) {
      ccol[off + t] = Direct ? first + static_cast<int32_t>(cols[t]) : colbuf[t];
      store_value<Mode>(cval, off + t, vals[t]);
    }
    if (bad) set_error(err, kErrCount);
  }
}

template <int LOG2S, int NT, int Mode>
__global__ void __launch_bounds__(NT) k_num_block(DevCsr A, DevCsr B, const int32_t* __restrict__ perm,
                                                  int64_t count, const int64_t* __restrict__ c_off,
                                                  int32_t* __restrict__ ccol, void* __restrict__ cval,
                                                  const int32_t* __restrict__ abase, int32_t* __restrict__ row_flag,
                                                  const int32_t* __restrict__ negflag, uint32_t* err) {
  constexpr int S = 1 << LOG2S;
  extern __shared__ double smem_f64[];
  double* vals = smem_f64;
  int32_t* keys = reinterpret_cast<int32_t*>(smem_f64 + S);
  __shared__ int32_t s_excl[NT];
  __shared__ int64_t s_bs[NT];
  __shared__ int32_t s_scan[33];
  for (int64_t r = blockIdx.x; r < count; r += gridDim.x) {
    const int32_t i = perm[r];
    const int64_t a0 = A.rp[i];
    const int64_t na = A.rp[i + 1] - a0;
    if (Mode == kModeF32C && threadIdx.x == 0 && !f32c_hash_row_ok(negflag, na)) row_flag[i] = 1;
    for (int s = threadIdx.x; s < S; s += NT) { keys[s] = kEmpty; vals[s] = 0.0; }
    __syncthreads();
    block_for_each_product<NT>(A, B, a0, na, s_excl, s_bs, s_scan, [&](int64_t j, int64_t e) {
      hash_accumulate<LOG2S, Mode>(keys, vals, B.col[j], value_at<Mode>(A.val, a0 + e), value_at<Mode>(B.val, j),
                                   err);
    });
    // compact in place, one block-wide chunk at a time
    int cnt = 0;
    for (int base = 0; base < S; base += NT) {
      const int32_t k = keys[base + threadIdx.x];
      const double v = vals[base + threadIdx.x];
      const int occ = k != kEmpty;
      int32_t tot;
      const int32_t pos = cnt + block_excl_scan<int32_t>(occ, s_scan, &tot);
      if (occ) { keys[pos] = k; vals[pos] = v; }
      cnt += tot;
      __syncthreads();
    }
    const int64_t off = c_off[i];
    const int64_t len = c_off[i + 1] - off;
    if (threadIdx.x == 0 && len != cnt) set_error(err, kErrCount);
    const int N = pow2_ceil(cnt);
    for (int t = cnt + threadIdx.x; t < N; t += NT) keys[t] = kNoCol;
    __syncthreads();
    block_bitonic<NT>(keys, vals, N);
    const int nb_out = cnt < len ? cnt : static_cast<int>(len);
    const int32_t cb = abase ? abase[i] : 0;
    for (int t = threadIdx.x; t < nb_out; t += NT) {
      ccol[off + t] = keys[t] - cb;
      store_value<Mode>(cval, off + t, vals[t]);
    }
    __syncthreads();
  }
}

inline unsigned grid_rows(int64_t count, int rows_per_block, int max_blocks) {
  int64_t g = (count + rows_per_block - 1) / rows_per_block;
  if (g > max_blocks) g = max_blocks;
  if (g < 1) g = 1;
  return static_cast<unsigned>(g);
}

}  // namespace

int launch_num_tiny(int mode, const DevCsr& A, const DevCsr& B, const int32_t* perm, int64_t count,
                    const int64_t* c_off, int32_t* ccol, void* cval, int32_t* row_flag, const int32_t* abase,
                    uint32_t* err, int num_sms, cudaStream_t s) {
  if (count <= 0) return 0;
  const unsigned g = grid_rows(count, 8, num_sms * 64);
  if (mode == kModeF32C) k_num_tiny<kModeF32C><<<g, 256, 0, s>>>(A, B, perm, count, c_off, ccol, cval, row_flag, abase, err);
  else if (mode == kModeF32R) k_num_tiny<kModeF32R><<<g, 256, 0, s>>>(A, B, perm, count, c_off, ccol, cval, row_flag, abase, err);
  else k_num_tiny<kModeF64><<<g, 256, 0, s>>>(A, B, perm, count, c_off, ccol, cval, row_flag, abase, err);
  return 1;
}

int launch_num_micro(const DevCsr& A, const DevCsr& B, const int32_t* perm, int64_t count, int64_t entries, int maxp,
                     const int64_t* c_off, int32_t* ccol, double* cval, const int32_t* abase, uint32_t* err, int num_sms,
                     cudaStream_t s) {
  if (count <= 0) return 0;
  // Room for 32 rows a sixteenth longer than the mean: regular rows fit, and an SM holds many warps.
  // Rows of fewer entries are stored from the merge, whose lanes are then close together (A*P of the
  // Galerkin set-up, 3 entries a row: 41 us against 59).
  const int64_t mean = (entries + count - 1) / count;
  const int cap = micro_cap(mean);
  const size_t sm = size_t(kMicroWarps) * micro_warp_bytes(cap, maxp);
  auto go = [&](auto kernel, size_t smem) {
    // (the limit belongs to the kernel: always the most any call needs, so that no thread lowers another's)
    constexpr int most = kMicroWarps * micro_warp_bytes(micro_cap(kMergeMax), kMergeMax);
    if (smem) cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    kernel<<<grid_rows(count, kMicroWarps * 32, num_sms * 32), kMicroWarps * 32, smem, s>>>(A, B, perm, count, cap, maxp,
                                                                                           c_off, ccol, cval, abase, err);
  };
  if (mean >= kMicroStaged) go(k_num_micro<true>, sm);
  else go(k_num_micro<false>, 0);
  return 1;
}

int launch_num_warp(int log2S, int mode, const DevCsr& A, const DevCsr& B, const int32_t* perm, int64_t count,
                    const int64_t* c_off, int32_t* ccol, void* cval, const int32_t* abase, int32_t* row_flag,
                    const int32_t* negflag, uint32_t* err, int num_sms, cudaStream_t s) {
  if (count <= 0) return 0;
  const unsigned g = grid_rows(count, 8, num_sms * 32);
  const size_t sm = size_t(8) * (size_t(1) << log2S) * 12;
  auto go = [&](auto kernel) {
    if (sm > 48 * 1024) cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(sm));
    kernel<<<g, 256, sm, s>>>(A, B, perm, count, c_off, ccol, cval, abase, row_flag, negflag, err);
  };
  const bool f32c = mode == kModeF32C;
  switch (log2S) {
    case 6: f32c ? go(k_num_warp<6, kModeF32C>) : go(k_num_warp<6, kModeF64>); break;
    case 8: f32c ? go(k_num_warp<8, kModeF32C>) : go(k_num_warp<8, kModeF64>); break;
    case 10: f32c ? go(k_num_warp<10, kModeF32C>) : go(k_num_warp<10, kModeF64>); break;
    default: break;
  }
  return 1;
}

int launch_num_block(int log2S, int mode, const DevCsr& A, const DevCsr& B, const int32_t* perm, int64_t count,
                     const int64_t* c_off, int32_t* ccol, void* cval, const int32_t* abase, const int32_t* awidth,
                     int64_t width, int max_nnz, int64_t products, int64_t entries, int32_t* row_flag,
                     const int32_t* negflag, uint32_t* err, int num_sms, cudaStream_t s) {
  if (count <= 0) return 0;
  const bool f32c = mode == kModeF32C;
  const int cap = log2S == 11 ? 1024 : (max_nnz <= 2048 ? 2048 : 4096);
  const int cw = bitmap_coarse_words(width, cap);
  // (two levels: as many columns as their tables by rank leave room for)
  const int span = products < kManyProducts * entries ? 0 : (cw == 0 ? kSpan : min(kSpan, 2 * cap));
  // the coarse bitmap of wider rows would not leave room for four rows on an SM: they hash. So do FP32
  // rows of two levels and many products
  if (width <= kBitmapMaxWidth && !(f32c && cw > 0 && products >= kManyProductsF32 * entries)) {
    const bool direct = cw == 0 && width <= 65536;
    const size_t sm = direct ? bitmap_bytes_direct(cap, width, span) : bitmap_bytes(cap, cw, span);
    auto go = [&](auto kernel) {
      // (the limit belongs to the kernel: always the most any call needs, so that no thread lowers another's)
      constexpr int kMost = 4096;
      constexpr size_t direct_most = bitmap_bytes_direct(kMost, 65536, kSpan);
      constexpr size_t most = bitmap_bytes(kMost, bitmap_coarse_words(kBitmapMaxWidth, 0), kSpan);
      if (sm > 40 * 1024)
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(direct ? direct_most : most));
      kernel<<<grid_rows(count, 1, num_sms * 16), 256, sm, s>>>(A, B, perm, count, c_off, ccol, cval, abase, awidth, width,
                                                               cap, span, row_flag, negflag, err);
    };
    auto instance = [&](auto many) {
      constexpr bool kMany = decltype(many)::value;
      if (direct) f32c ? go(k_num_bitmap<256, kModeF32C, true, kMany>) : go(k_num_bitmap<256, kModeF64, true, kMany>);
      else f32c ? go(k_num_bitmap<256, kModeF32C, false, kMany>) : go(k_num_bitmap<256, kModeF64, false, kMany>);
    };
    if (span > 0) instance(std::true_type{});
    else instance(std::false_type{});
    return 1;
  }
  const size_t sm = (size_t(1) << log2S) * 12;
  auto go = [&](auto kernel, int nt, int per_sm) {
    if (sm > 48 * 1024) cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(sm));
    kernel<<<grid_rows(count, 1, num_sms * per_sm), nt, sm, s>>>(A, B, perm, count, c_off, ccol, cval, abase, row_flag,
                                                                 negflag, err);
  };
  if (log2S == 11) {
    f32c ? go(k_num_block<11, 256, kModeF32C>, 256, 8) : go(k_num_block<11, 256, kModeF64>, 256, 8);
  } else if (log2S == 13) {
    f32c ? go(k_num_block<13, 512, kModeF32C>, 512, 4) : go(k_num_block<13, 512, kModeF64>, 512, 4);
  }
  return 1;
}

}  // namespace spg
