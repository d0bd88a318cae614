// Windowed numeric pass over a list of windows: rows with more entries of C than a block row holds, of
// plans whose windowed rows all have their column bitmap stored by the symbolic pass (k_window.cu
// takes the other plans).
//
// The columns of C are cut into sub-blocks of kSubCols columns; the symbolic pass counted every
// windowed row's entries per sub-block. k_win_plan groups each row's consecutive sub-blocks into
// windows of at most kWinCap entries and kWinSpan sub-blocks and lists them with everything the numeric
// kernel needs to start on one. A block of k_num_winteam takes one window after the other:
//  1. the window's stored bitmap gives every column its rank among the window's columns;
//  2. a_ik * b_kj is added into an array indexed by the rank of column j, kChunk entries of A at a
//     time: the split table (k_bsplit_sub) gives each entry's part of its B row in the window;
//  3. columns and values leave in rank order.
// The output is sorted by column without a sort, as Algorithm 1's sorted PP (Sec. III-A).
//
// Bound by shared memory (the rank lookups and the sums' compare-and-swaps: 70 % of the peak wavefronts),
// by the instructions of a product (about 94 per 32 products) and by the FP64 pipe (50 %). What it saves against
// a block per row with windows of the same size (k_num_window) and a pass of its own for the columns
// (k_expand_cols): the list lets the next window's data be fetched while one is worked on and spreads a
// long row over all blocks; a product stores its column at its rank on the way, so no pass extracts the
// columns from the bitmap; three blocks of eight warps on an SM wait less at a window's barriers than two
// of sixteen; whole groups of 32 products of one segment need no search per product, and the others'
// segment is a popcount of the bits where segments start. Both kernels and this one: 30,000^2 uniform
// (d = 5e-3, 6.7e8 products) 7.35 and 4.21 ms, R-MAT 2^17 (1.09e9) 9.92 and 5.68 ms, R-MAT 2^19 (7.85e9) 77.6
// and 51.8 ms; a single row of 90,000 entries of A (9e6 products) 126 and 2.8 ms, all passes.
//
// FP32-compensated plans take the same kernel with FP32 sums and compensations in the eight bytes of a
// slot (two FP32 atomics a product, separate arrays so that both spread over all banks): R-MAT 2^17
// 7.93 -> 5.45 ms. A slot that also needs the sum of |p| and the term count takes sixteen bytes and its
// windows half the entries; with mixed signs (R-MAT 2^17 of 8 edges a vertex) 4.51 -> 3.50 ms.
#include <type_traits>

#include "common.cuh"
#include "kernels.h"

namespace spg {

namespace {

// A window's size against the number of windows an SM works on at once (one per block; a block is idle
// while its window's ranks are made, at its barriers and while it writes out), and the products a warp
// has under way. Measured, ms of the numeric pass on the 30,000^2 uniform product (d = 5e-3), R-MAT 2^17,
// the same FP32-compensated, and R-MAT 2^19:
//   8 warps, 4096 entries, 64 sub-blocks, 3 blocks per SM, 3 groups a step: 4.21, 5.68, 5.45, 51.8 (taken)
//   the same with 2 groups: 4.17, 5.74, 5.68, 51.7;  3584 entries: 4.17, 5.93, 5.68, 53.3
//   8 warps, 4096 entries, 32 sub-blocks, 3 blocks: 3.97, 5.87, 5.90, 54.5;  3072, 4 blocks: 4.06, 5.83, 5.53, 55.8
//   8 warps, 2560 entries, 64 sub-blocks, 4 blocks: 4.45, 6.09, 5.69, 54.4
//   4 warps, 2048 entries, 32 sub-blocks, 6 blocks: 4.53, 5.69, 5.75, 54.8;  3 groups: 4.69, 5.66, 5.60, 55.2
//   16 warps, 4096 entries, 64 sub-blocks, 2 blocks: 4.78, 7.34, 6.35, 64.5
constexpr int kWinCap = 4096;      // entries of C per window (>= kSubCols)
constexpr int kWinSpan = 64;       // sub-blocks per window
constexpr int kTeam = 8;           // warps per block: one window at a time
constexpr int kTeamBlocks = 3;     // blocks per SM
constexpr int kChunk = kTeam * 32; // A entries per chunk, one per thread
constexpr int kRankStep = kWinSpan / 4 / kTeam;   // runs of four sub-blocks per warp
constexpr int kGroups = 3;         // groups of 32 products per step; a warp has two steps under way
constexpr int kSlots = 3;          // window records in shared memory: this one, the next, the one after
constexpr unsigned kFull = 0xffffffffu;
constexpr int kWideCap = kWinCap / 2;   // entries of C per window of wide slots
static_assert(kWideCap >= kSubCols, "a window holds any single sub-block");

// A window of a row, as k_win_plan lists it.
struct alignas(64) WinRecord {
  int64_t a0;      // the row's first entry of A,
  int64_t out;     // the window's first entry of C,
  int64_t bits;    // its first bitmap word,
  int64_t cnts;    // the counts of its first sub-block
  int32_t na;      // entries of A
  int32_t cnt;     // entries of C
  int32_t wb, we;  // sub-blocks [wb, we) of the row
  int32_t w0;      // first column (of a stacked batch: in the stacked product)
  int32_t row;
  int32_t wide;    // kModeF32C: the row's entries need their term counts (wide slots, at most kWideCap of them)
};
static_assert(sizeof(WinRecord) == 64, "a record is four 16-byte pieces");

// A chunk's segments (the parts of its A entries' B rows in the window), as lists of those with at
// least one whole group of 32 products and of those with a remainder of fewer than 32, numbered
// consecutively in each list.
template <typename V>
struct WholeList {
  V av[kChunk];           // a_ik
  uint32_t bs[kChunk];    // start in B less 32 times the number of the segment's first group
  int32_t end[kChunk];    // end of its numbers
};
template <typename V>
struct RestList {
  V av[kChunk];
  uint32_t bs[kChunk];         // start in B less the number of the segment's first product
  uint32_t start[2][kChunk];   // bit per product: a segment starts there (this chunk's, and zeros for the next)
  uint16_t first[kChunk];      // per 32 products: the first segment that starts among them. None has 32
};                             // products, so one does

template <typename V>
struct TeamSmem {
  // By rank. kModeF64: the sums. kModeF32C: arrays of kWinCap FP32 sums and compensations; wide: of
  // kWideCap sums, compensations, sums of |p| and term counts.
  double vals[kWinCap];
  uint32_t bits[2][kWinSpan * 32];      // bitmap words of this window and the next
  uint16_t pre[kWinSpan * 32];          // set bits before each word
  uint16_t col[kWinCap];                // columns by rank, from the window's first
  WholeList<V> whole;                   // the chunk's segments
  RestList<V> rest;
  WinRecord rec[kSlots];
  unsigned long long tot[kTeam];
  int32_t have[kSlots];                 // a record follows in this slot
};

__device__ __forceinline__ void copy16(void* shared, const void* global) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(shared))),
               "l"(global)
               : "memory");
}
__device__ __forceinline__ void copies_done() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// The windows of every row of perm[0, count): a warp per row takes the row's sub-blocks 64 at a time
// (two counts per lane) and cuts windows greedily; a window ends at merge_cap entries (one sub-block may
// have more), at kWinSpan sub-blocks, or with those 64. kModeF32C (negflag given: whether A or B has a
// negative value): an entry of a row whose products are all non-negative and few enough is within the
// bound without counting its terms (f32c_within_count); the other rows' windows have wide slots.
__global__ void __launch_bounds__(256) k_win_plan(DevCsr A, const int32_t* __restrict__ perm, int64_t count,
                                                  const int32_t* __restrict__ win_slot, int64_t nslots,
                                                  const uint16_t* __restrict__ subcnt, int64_t nsub, int32_t merge_cap,
                                                  const int64_t* __restrict__ c_off, const int64_t* __restrict__ woff,
                                                  const int32_t* __restrict__ abase,
                                                  const int32_t* __restrict__ awidth, int64_t width_all,
                                                  const int32_t* __restrict__ negflag,
                                                  WinRecord* __restrict__ wins, int64_t cap, int32_t* n_wins,
                                                  uint32_t* err) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = (int64_t(gridDim.x) * blockDim.x) >> 5;
  for (int64_t q = (blockIdx.x * int64_t(blockDim.x) + threadIdx.x) >> 5; q < count; q += nw) {
    const int32_t i = perm[q];
    const int32_t slot = win_slot[i];
    // the row was not counted by the windowed symbolic pass, or its bitmap was not stored
    if (slot < 0 || slot >= nslots || woff[slot] < 0) {
      if (lane == 0) set_error(err, kErrWindowPlan);
      continue;
    }
    const int32_t cb = abase ? abase[i] : 0;
    const int32_t row_sub = static_cast<int32_t>(((awidth ? awidth[i] : width_all) + kSubCols - 1) / kSubCols);
    const uint16_t* cnt = subcnt + int64_t(slot) * nsub;
    WinRecord w{};
    w.a0 = A.rp[i];
    w.na = static_cast<int32_t>(A.rp[i + 1] - w.a0);
    w.row = i;
    w.wide = negflag && (*negflag != 0 || !f32c_within_count(w.na < (1 << 30) ? w.na : (1 << 30)));
    const int32_t most = w.wide ? kWideCap : kWinCap, row_cap = merge_cap < most ? merge_cap : most;
    const int64_t out0 = c_off[i], room = c_off[i + 1] - out0, bits0 = woff[slot];
    int64_t at = 0;
    for (int pass = 0; pass < 2; ++pass) {
      int32_t carry = 0, n = 0;   // entries and windows before this run of 64
      for (int32_t run0 = 0; run0 < row_sub; run0 += 64) {
        const int32_t ca = run0 + lane < row_sub ? cnt[run0 + lane] : 0;
        const int32_t cc = run0 + lane + 32 < row_sub ? cnt[run0 + lane + 32] : 0;
        const int32_t sa = warp_incl_scan(ca);
        const int32_t sb = warp_incl_scan(cc) + __shfl_sync(kFull, sa, 31);
        auto both = [&](bool x, bool y) {
          return static_cast<uint64_t>(__ballot_sync(kFull, x)) | (static_cast<uint64_t>(__ballot_sync(kFull, y)) << 32);
        };
        uint64_t todo = both(ca > 0, cc > 0);
        while (todo) {
          const int s = __ffsll(static_cast<long long>(todo)) - 1;
          const int32_t base = s == 0 ? 0 : __shfl_sync(kFull, s <= 32 ? sa : sb, (s - 1) & 31);
          // the sub-blocks from s on that fit the window (the first always does)
          const uint64_t fit =
              both(lane == s || (sa - base <= row_cap && lane >= s && lane < s + kWinSpan),
                   lane + 32 == s || (sb - base <= row_cap && lane + 32 >= s && lane + 32 < s + kWinSpan)) & todo;
          const int e = 64 - __clzll(static_cast<long long>(fit));   // past the last non-empty one
          todo &= e == 64 ? 0ull : ~0ull << e;
          w.cnt = __shfl_sync(kFull, e <= 32 ? sa : sb, (e - 1) & 31) - base;
          if (pass == 1 && lane == 0 && at + n < cap) {
            w.wb = run0 + s;
            w.we = run0 + e;
            w.w0 = cb + w.wb * kSubCols;
            w.out = out0 + carry + base;
            w.bits = bits0 + int64_t(w.wb) * 32;
            w.cnts = int64_t(slot) * nsub + w.wb;
            if (w.cnt > most || carry + base + w.cnt > room) {   // never writes past the rank array or the row
              set_error(err, kErrWindowPlan);
              w.cnt = w.na = 0;
            }
            wins[at + n] = w;
          }
          ++n;
        }
        carry += __shfl_sync(kFull, sb, 31);
      }
      if (pass == 0) {
        int32_t o = 0;
        if (lane == 0) {
          o = atomicAdd(n_wins, n);
          if (o + int64_t(n) > cap || carry != room) set_error(err, kErrWindowPlan);
        }
        at = __shfl_sync(kFull, o, 0);
      }
    }
  }
}

// Split table of B by sub-blocks: split[k * nsub + b] = the index into B of row k's first entry
// with column >= b * kSubCols (from the row's column base), so row k's entries in sub-blocks [b, e)
// are [split[k * nsub + b], split[k * nsub + e]) (the entry after a row's last is the next row's
// first). A warp per row: the first entry of each sub-block is noted in shared memory, and a suffix
// minimum over the sub-blocks gives the empty ones their successor's.
constexpr int kSplitWarps = 8;
__global__ void __launch_bounds__(kSplitWarps * 32) k_bsplit_sub(DevCsr B, int64_t nsub,
                                                                 const int32_t* __restrict__ bbase,
                                                                 uint32_t* __restrict__ split) {
  __shared__ uint32_t s_first[kSplitWarps][kMaxSub];
  const int lane = threadIdx.x & 31;
  uint32_t* first = s_first[threadIdx.x >> 5];
  const int64_t nw = (int64_t(gridDim.x) * blockDim.x) >> 5;
  const int last32 = static_cast<int>((nsub + 31) / 32 * 32);
  for (int64_t k = (blockIdx.x * int64_t(blockDim.x) + threadIdx.x) >> 5; k < B.rows; k += nw) {
    const int64_t s = B.rp[k], e = B.rp[k + 1];
    const int32_t bb = bbase ? bbase[k] : 0;
    for (int b = lane; b < last32; b += 32) first[b] = 0xffffffffu;
    __syncwarp();
    for (int64_t t0 = s; t0 < e; t0 += 32) {
      const int64_t t = t0 + lane;
      if (t < e) {
        const int bc = (B.col[t] - bb) >> kSubShift;
        const int bp = t == s ? -1 : (B.col[t - 1] - bb) >> kSubShift;
        if (bc != bp && bc >= 0 && bc < nsub) first[bc] = static_cast<uint32_t>(t);
      }
    }
    __syncwarp();
    if (k == B.rows - 1 && lane == 0) split[B.rows * nsub] = static_cast<uint32_t>(e);
    uint32_t carry = static_cast<uint32_t>(e);
    for (int b0 = last32 - 32; b0 >= 0; b0 -= 32) {
      uint32_t v = first[b0 + lane];
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const uint32_t o = __shfl_down_sync(kFull, v, d);
        if (lane + d < 32) v = min(v, o);
      }
      v = min(v, carry);
      if (b0 + lane < nsub) split[k * nsub + b0 + lane] = v;
      carry = __shfl_sync(kFull, v, 0);
    }
    __syncwarp();
  }
}

// A window's columns and ranks.
struct Window {
  int32_t w0;      // first column (global)
  uint32_t span;   // columns
  const uint32_t* bits;
  const uint16_t* pre;
  double* vals;
  uint16_t* col;
  bool wide, neg;   // kModeF32C
};

// Segments of a list of n that end at or before x: the number of the one that owns x.
// A warp asks for ascending x: `from` (a multiple of 32, at first 0) is where its last answer was.
__device__ __forceinline__ int first_after(const int32_t* end, int n, int32_t x, int& from) {
  for (;;) {
    const int t = from + static_cast<int>(threadIdx.x & 31);
    const int o = __popc(__ballot_sync(kFull, t < n && end[t] <= x));
    if (o < 32) return from + o;
    from += 32;
  }
}

// kGroups products per lane: a * v at column c (want bit u: the lane's u-th takes part).
template <typename V>
struct Step {
  int32_t c[kGroups];
  V a[kGroups], v[kGroups];
  unsigned want;
};

// Adds the product a * b into the slot of rank r.
__device__ __forceinline__ void add_product(const Window& win, int r, double a, double b) {
  add_product_f64(win.vals + r, a, b);
}

// FP32: the error-free product ph + pl, and the sum's own rounding error (TwoSum) rebuilt from the value
// the atomic returns, as the other compensated kernels do (Dot2 accumulated concurrently).
__device__ __forceinline__ void add_product(const Window& win, int r, float a, float b) {
  float* slot = reinterpret_cast<float*>(win.vals) + r;
  const float ph = a * b;
  const float pl = fmaf(a, b, -ph);
  const float old = atomicAdd(slot, ph);
  const float nw = old + ph;
  const float bp = nw - old;
  const float q = (old - (nw - bp)) + (ph - bp);
  atomicAdd(slot + (win.wide ? kWideCap : kWinCap), q + pl);
  if (win.wide) {
    if (win.neg) atomicAdd(slot + 2 * kWideCap, fabsf(ph));
    atomicAdd(reinterpret_cast<int*>(slot) + 3 * kWideCap, 1);
  }
}

// A step's products into the window's sums. The ranks of all of them are looked up before the first is
// added.
template <typename V>
__device__ __forceinline__ void add_step(const Window& win, const Step<V>& st, bool& bad) {
  const auto& c = st.c;
  const auto& a = st.a;
  const auto& v = st.v;
  const unsigned want = st.want;
  uint32_t rel[kGroups], word[kGroups], before[kGroups];
#pragma unroll
  for (int u = 0; u < kGroups; ++u) {
    rel[u] = static_cast<uint32_t>(c[u] - win.w0);
    const uint32_t w = min(rel[u], win.span - 1u) >> 5;
    word[u] = win.bits[w];
    before[u] = win.pre[w];
  }
  int r[kGroups];
#pragma unroll
  for (int u = 0; u < kGroups; ++u) {
    const uint32_t bit = 1u << (rel[u] & 31);
    const bool in = rel[u] < win.span && (word[u] & bit) != 0u;
    r[u] = in && (want >> u & 1u) ? static_cast<int>(before[u]) + __popc(word[u] & (bit - 1u)) : -1;
    bad |= (want >> u & 1u) && !in;   // a product outside the stored columns
  }
#pragma unroll
  for (int u = 0; u < kGroups; ++u)
    if (r[u] >= 0) {
      win.col[r[u]] = static_cast<uint16_t>(rel[u]);   // every product of the column stores the same
      add_product(win, r[u], a[u], v[u]);
    }
}
static_assert(kWinSpan * kSubCols <= 65536, "a window's columns fit 16 bits");

// One step of the whole groups: groups [g, g + kGroups) of the list's `groups` in n segments.
template <typename V>
__device__ __forceinline__ void load_whole(const WholeList<V>& sl, int n, int32_t g, int32_t groups,
                                           const int32_t* __restrict__ bcol, const V* __restrict__ bval,
                                           Step<V>& st, int& from) {
  const int lane = threadIdx.x & 31;
  const int o = first_after(sl.end, n, g, from);
  // every segment has a group, so kGroups groups see at most kGroups segments
  const int32_t e = sl.end[min(o + lane, n - 1)];
  uint32_t j[kGroups];
#pragma unroll
  for (int u = 0; u < kGroups; ++u) {
    const int32_t x = min(g + u, groups - 1);
    const int k = o + __popc(__ballot_sync(kFull, e <= x) & ((1u << kGroups) - 1u));
    j[u] = sl.bs[k] + static_cast<uint32_t>(32 * x + lane);
    st.a[u] = sl.av[k];
  }
#pragma unroll
  for (int u = 0; u < kGroups; ++u) {
    st.c[u] = bcol[j[u]];
    st.v[u] = bval[j[u]];
  }
  st.want = g + kGroups <= groups ? (1u << kGroups) - 1u : (1u << (groups - g)) - 1u;
}

// One step of the remainders: products [p, p + 32 * kGroups) of the list's `total` (p a multiple of 32).
template <typename V>
__device__ __forceinline__ void load_rest(const RestList<V>& sl, const uint32_t* start, int32_t p, int32_t total,
                                          const int32_t* __restrict__ bcol, const V* __restrict__ bval,
                                          Step<V>& st) {
  const int lane = threadIdx.x & 31;
  uint32_t j[kGroups];
  st.want = 0;
#pragma unroll
  for (int u = 0; u < kGroups; ++u) {
    const int32_t x = p + 32 * u + lane;
    if (x < total) st.want |= 1u << u;
    const int32_t y = min(x, total - 1);   // a lane past the end takes the last product
    const int k = sl.first[y >> 5] + __popc(start[y >> 5] & (0xffffffffu >> (31 - (y & 31)))) - 1;
    j[u] = sl.bs[k] + static_cast<uint32_t>(y);
    st.a[u] = sl.av[k];
  }
#pragma unroll
  for (int u = 0; u < kGroups; ++u) {
    st.c[u] = bcol[j[u]];
    st.v[u] = bval[j[u]];
  }
}

// First index in col[s, e) with col >= x (col ascending); e when none.
__device__ __forceinline__ uint32_t lower_bound_at(const int32_t* __restrict__ col, uint32_t s, uint32_t e, int64_t x) {
  while (s < e) {
    const uint32_t mid = s + ((e - s) >> 1);
    if (col[mid] < x) s = mid + 1;
    else e = mid;
  }
  return s;
}

// V: double (kModeF64) or float (kModeF32C; row_flag takes the rows with an entry over the bound).
template <typename V>
__global__ void __launch_bounds__(kTeam * 32, kTeamBlocks) k_num_winteam(
    DevCsr A, DevCsr B, const WinRecord* __restrict__ wins, const int32_t* __restrict__ n_wins, int64_t wins_cap,
    int32_t* counter, const uint16_t* __restrict__ subcnt, int64_t nsub, const uint32_t* __restrict__ split,
    int32_t* __restrict__ ccol, V* __restrict__ cval, const uint32_t* __restrict__ wbits,
    const int32_t* __restrict__ negflag, int32_t* row_flag, uint32_t* err) {
  extern __shared__ __align__(64) unsigned char win_smem[];
  TeamSmem<V>& sw = *reinterpret_cast<TeamSmem<V>*>(win_smem);
  constexpr bool kF32 = sizeof(V) == 4;
  const bool neg = kF32 && *negflag != 0;
  constexpr int kThreads = kTeam * 32;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const V* aval = static_cast<const V*>(A.val);
  const V* bval = static_cast<const V*>(B.val);
  const int32_t n = static_cast<int32_t>(*n_wins < wins_cap ? *n_wins : wins_cap);
  bool bad = false;
  // What a window needs first is fetched while the one before is worked on: its record two windows
  // ahead, its bitmap words, counts and first chunk of A entries one ahead, the chunk's bounds in B
  // at the end of the one before.
  auto fetch_record = [&](int slot, int32_t idx) {   // warp 0
    if (lane < 4 && idx < n) copy16(reinterpret_cast<char*>(&sw.rec[slot]) + 16 * lane,
                                    reinterpret_cast<const char*>(wins + idx) + 16 * lane);
    if (lane == 0) sw.have[slot] = idx < n;
  };
  auto fetch_bits = [&](const WinRecord& r, int buf) {
    const int pieces = (r.we - r.wb) * 8;   // of 16 bytes
    for (int t = threadIdx.x; t < pieces; t += kThreads) copy16(&sw.bits[buf][4 * t], wbits + r.bits + 4 * t);
  };
  int32_t k1 = -1, ca = 0, cc = 0;
  V v1 = 0;
  auto fetch_entries = [&](const WinRecord& r) {
    const int ns = r.we - r.wb;
    ca = lane < ns ? subcnt[r.cnts + lane] : 0;
    cc = lane + 32 < ns ? subcnt[r.cnts + lane + 32] : 0;
    const bool mine = static_cast<int>(threadIdx.x) < r.na;
    k1 = mine ? A.col[r.a0 + threadIdx.x] : -1;
    v1 = mine ? aval[r.a0 + threadIdx.x] : V(0);
  };
  auto bound = [&](const WinRecord& r, int32_t k, int32_t b) -> uint32_t {
    if (split) return split[k * nsub + b];
    return lower_bound_at(B.col, static_cast<uint32_t>(B.rp[k]), static_cast<uint32_t>(B.rp[k + 1]),
                          int64_t(r.w0) + int64_t(b - r.wb) * kSubCols);
  };
  sw.rest.start[0][threadIdx.x] = 0u;
  int32_t next = 0;   // warp 0, lane 0: the index of the window after the next
  if (wid == 0) {
    fetch_record(0, blockIdx.x);
    int32_t second = 0;
    if (lane == 0) {
      // the first window of each block is the block's number, the others come from the counter
      second = gridDim.x + atomicAdd(counter, 1);
      next = gridDim.x + atomicAdd(counter, 1);
    }
    fetch_record(1, __shfl_sync(kFull, second, 0));
  }
  copies_done();
  __syncthreads();
  uint32_t bs = 0, be = 0;
  if (sw.have[0]) {
    fetch_bits(sw.rec[0], 0);
    fetch_entries(sw.rec[0]);
    if (k1 >= 0) {
      bs = bound(sw.rec[0], k1, sw.rec[0].wb);
      be = bound(sw.rec[0], k1, sw.rec[0].we);
    }
  }
  copies_done();
  __syncthreads();
  int slot = 0, buf = 0, list = 0;
  while (sw.have[slot]) {
    const WinRecord& r = sw.rec[slot];
    const int ns = r.we - r.wb;
    const int32_t cnt = r.cnt, na = r.na;
    const int slot1 = slot == kSlots - 1 ? 0 : slot + 1, slot2 = slot1 == kSlots - 1 ? 0 : slot1 + 1;
    // 1. ranks: a warp takes the runs of four sub-blocks wid, wid + kTeam, ... (lane: four consecutive
    // words); the bits before a run are its counts' sum
    {
      const int32_t sa = warp_incl_scan(ca);
      const int32_t sb = warp_incl_scan(cc) + __shfl_sync(kFull, sa, 31);
      uint4 w[kRankStep];
      int incl[kRankStep];
#pragma unroll
      for (int q = 0; q < kRankStep; ++q) {
        const int t = 4 * (wid + q * kTeam);
        w[q] = t + lane / 8 < ns ? *reinterpret_cast<const uint4*>(&sw.bits[buf][t * 32 + lane * 4]) : make_uint4(0u, 0u, 0u, 0u);
        incl[q] = __popc(w[q].x) + __popc(w[q].y) + __popc(w[q].z) + __popc(w[q].w);
      }
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
#pragma unroll
        for (int q = 0; q < kRankStep; ++q) {
          const int o = __shfl_up_sync(kFull, incl[q], d);
          if (lane >= d) incl[q] += o;
        }
      }
#pragma unroll
      for (int q = 0; q < kRankStep; ++q) {
        const int t = 4 * (wid + q * kTeam);
        const int32_t before = t == 0 ? 0 : __shfl_sync(kFull, t <= 32 ? sa : sb, (t - 1) & 31);
        const uint32_t p3 = before + incl[q] - __popc(w[q].w), p2 = p3 - __popc(w[q].z), p1 = p2 - __popc(w[q].y),
                       p0 = p1 - __popc(w[q].x);
        if (t + lane / 8 < ns)
          *reinterpret_cast<uint2*>(&sw.pre[t * 32 + lane * 4]) = make_uint2(p0 | p1 << 16, p2 | p3 << 16);
      }
    }
    const bool wide = kF32 && r.wide != 0;
    if constexpr (kF32) {
      const int arrays = wide ? 4 : 2, stride = (wide ? kWideCap : kWinCap) / 4;
      for (int q = threadIdx.x; q < (cnt + 3) / 4; q += kThreads)
        for (int w = 0; w < arrays; ++w)
          reinterpret_cast<float4*>(sw.vals)[w * stride + q] = make_float4(0.f, 0.f, 0.f, 0.f);
    } else {
      for (int q = threadIdx.x; q < (cnt + 1) / 2; q += kThreads)
        reinterpret_cast<double2*>(sw.vals)[q] = make_double2(0.0, 0.0);
    }
    // 2. products; inside a row of several chunks, the next chunk's entries and bounds are loaded ahead
    const Window win{r.w0, static_cast<uint32_t>(ns) * kSubCols, sw.bits[buf], sw.pre, sw.vals, sw.col, wide, neg};
    const int64_t a0 = r.a0;
    int32_t k2 = static_cast<int>(threadIdx.x) + kChunk < na ? A.col[a0 + threadIdx.x + kChunk] : -1;
    V v2 = static_cast<int>(threadIdx.x) + kChunk < na ? aval[a0 + threadIdx.x + kChunk] : V(0);
    for (int32_t c0 = 0; c0 == 0 || c0 < na; c0 += kChunk) {
      // one scan numbers the whole groups (20 bits), the remainders (16), and both lists' segments
      const uint32_t len = be - bs, nw = len >> 5, nr = len & 31;
      const unsigned long long mine = nw | static_cast<unsigned long long>(nr) << 20 |
                                      static_cast<unsigned long long>(nw > 0) << 36 |
                                      static_cast<unsigned long long>(nr > 0) << 48;
      const unsigned long long incl = warp_incl_scan(mine);
      if (lane == 31) sw.tot[wid] = incl;
      __syncthreads();   // (the first chunk's: the ranks and zeros; later ones': the lists are read)
      unsigned long long at = incl - mine, all = 0;
#pragma unroll
      for (int w = 0; w < kTeam; ++w) {
        if (w < wid) at += sw.tot[w];
        all += sw.tot[w];
      }
      if (nw > 0) {
        const int o = static_cast<int>(at >> 36) & 0xfff, g = static_cast<int>(at & 0xfffff);
        sw.whole.av[o] = v1;
        sw.whole.bs[o] = bs - 32u * g;
        sw.whole.end[o] = g + nw;
      }
      if (nr > 0) {
        const int o = static_cast<int>(at >> 48), p = static_cast<int>(at >> 20) & 0xffff;
        sw.rest.av[o] = v1;
        sw.rest.bs[o] = bs + 32u * nw - p;
        atomicOr(&sw.rest.start[list][p >> 5], 1u << (p & 31));
        if (p == 0) sw.rest.first[0] = 0;
        if ((p + nr) >> 5 != static_cast<uint32_t>(p) >> 5) sw.rest.first[(p + nr) >> 5] = static_cast<uint16_t>(o + 1);
      }
      if (c0 + kChunk < na) {
        bs = be = 0;
        if (k2 >= 0) {
          bs = bound(r, k2, r.wb);
          be = bound(r, k2, r.we);
        }
        v1 = v2;
        const int32_t q3 = c0 + 2 * kChunk + static_cast<int>(threadIdx.x);
        k2 = q3 < na ? A.col[a0 + q3] : -1;
        v2 = q3 < na ? aval[a0 + q3] : V(0);
      } else if (sw.have[slot1]) {
        fetch_bits(sw.rec[slot1], buf ^ 1);
        fetch_entries(sw.rec[slot1]);
      }
      __syncthreads();
      const int32_t groups = static_cast<int32_t>(all & 0xfffff), rest = static_cast<int32_t>(all >> 20) & 0xffff;
      sw.rest.start[list ^ 1][threadIdx.x] = 0u;   // (its last readers are before the barrier above the lists)
      const uint32_t* start = sw.rest.start[list];
      list ^= 1;
      // the warps take the steps of both lists in turn: at most one step of each list is short
      const int wsteps = (groups + kGroups - 1) / kGroups, steps = wsteps + (rest + 32 * kGroups - 1) / (32 * kGroups);
      int from = 0;
      auto load = [&](int q, Step<V>& st) {
        if (q < wsteps) load_whole(sw.whole, static_cast<int>(all >> 36) & 0xfff, kGroups * q, groups, B.col, bval, st, from);
        else load_rest(sw.rest, start, 32 * kGroups * (q - wsteps), rest, B.col, bval, st);
      };
      if (wid < steps) {
        Step<V> cur;
        load(wid, cur);
        for (int q = wid + kTeam; q < steps; q += kTeam) {   // a step's loads are under way while the last is added
          Step<V> ahead;
          load(q, ahead);
          add_step(win, cur, bad);
          cur = ahead;
        }
        add_step(win, cur, bad);
      }
    }
    // the next window's bounds, and the record of the one after it
    if (sw.have[slot1]) {
      const WinRecord& r1 = sw.rec[slot1];
      bs = be = 0;
      if (k1 >= 0) {
        bs = bound(r1, k1, r1.wb);
        be = bound(r1, k1, r1.we);
      }
    }
    if (wid == 0) {
      const int32_t idx = __shfl_sync(kFull, next, 0);
      fetch_record(slot2, idx);
      if (lane == 0) next = gridDim.x + atomicAdd(counter, 1);
    }
    __syncthreads();
    // 3. out, in rank order
    {
      const int64_t out = r.out;
      const int32_t first = r.wb * kSubCols;
      bool missed = false;
      for (int q = threadIdx.x; q < cnt; q += kThreads) {
        ccol[out + q] = first + sw.col[q];
        if constexpr (kF32) {
          const float* f = reinterpret_cast<const float*>(sw.vals) + q;
          const float res = f[0] + f[wide ? kWideCap : kWinCap];
          cval[out + q] = res;
          if (wide) {
            const int t = __float_as_int(f[3 * kWideCap]);
            missed |= neg ? !f32c_within_bound(res, f[2 * kWideCap], t) : !f32c_within_count(t);
          }
        } else {
          cval[out + q] = sw.vals[q];
        }
      }
      if (missed) row_flag[r.row] = 1;
    }
    copies_done();
    slot = slot1;
    buf ^= 1;
    __syncthreads();
  }
  if (__any_sync(kFull, bad) && lane == 0) set_error(err, kErrWindowPlan);
}

}  // namespace

int64_t win_list_bytes(int64_t rows, int64_t entries, int64_t nsub, int32_t merge_cap, int f32c, int64_t* cap) {
  // a window ends with its run of 64 sub-blocks, or it and the next of the run hold more than merge_cap
  // entries together (a run of e entries: at most 2 e / merge_cap + 1 windows); and it holds at least one
  // sub-block
  static_assert(kWinSpan >= 64, "the span of a window does not end it inside a run");
  const int64_t most = f32c ? kWideCap : kWinCap;
  const int64_t m = merge_cap < 1 ? 1 : (merge_cap < most ? merge_cap : most);
  const int64_t by_entries = 2 * (entries / m + 1) + rows * ((nsub + 63) / 64);
  *cap = by_entries < rows * nsub ? by_entries : rows * nsub;
  return *cap * static_cast<int64_t>(sizeof(WinRecord));
}

int launch_win_plan(const DevCsr& A, const int32_t* perm, int64_t count, const int32_t* win_slot, int64_t nslots,
                    const uint16_t* subcnt, int64_t nsub, int32_t merge_cap, const int64_t* c_off, const int64_t* woff,
                    const int32_t* abase, const int32_t* awidth, int64_t width, const int32_t* negflag, void* wins,
                    int64_t cap, int32_t* n_wins, int num_sms, uint32_t* err, cudaStream_t s) {
  if (count <= 0) return 0;
  cudaMemsetAsync(n_wins, 0, sizeof(int32_t), s);
  int64_t g = (count + 7) / 8;
  if (g > int64_t(num_sms) * 8) g = int64_t(num_sms) * 8;
  k_win_plan<<<static_cast<unsigned>(g), 256, 0, s>>>(A, perm, count, win_slot, nslots, subcnt, nsub,
                                                      merge_cap < kWinCap ? merge_cap : kWinCap, c_off, woff, abase,
                                                      awidth, width, negflag, static_cast<WinRecord*>(wins), cap, n_wins, err);
  return 1;
}

int launch_bsplit_sub(const DevCsr& B, int64_t nsub, const int32_t* bbase, uint32_t* split, int num_sms,
                      cudaStream_t s) {
  if (B.rows <= 0) return 0;
  int64_t g = (B.rows + kSplitWarps - 1) / kSplitWarps;
  if (g > int64_t(num_sms) * 64) g = int64_t(num_sms) * 64;
  k_bsplit_sub<<<static_cast<unsigned>(g), kSplitWarps * 32, 0, s>>>(B, nsub, bbase, split);
  return 1;
}

int launch_num_winteam(const DevCsr& A, const DevCsr& B, const void* wins, const int32_t* n_wins, int64_t wins_cap,
                       int32_t* counter, const uint16_t* subcnt, int64_t nsub, const uint32_t* split, int32_t* ccol,
                       void* cval, const uint32_t* wbits, const int32_t* negflag, int32_t* row_flag, int num_sms,
                       uint32_t* err, cudaStream_t s) {
  const unsigned grid = static_cast<unsigned>(num_sms * kTeamBlocks);
  cudaMemsetAsync(counter, 0, sizeof(int32_t), s);
  auto go = [&](auto kernel, auto* out) {
    constexpr int smem = static_cast<int>(sizeof(TeamSmem<std::remove_pointer_t<decltype(out)>>));
    static_assert(kTeamBlocks * (smem + 1024) <= 228 * 1024, "blocks per SM");
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    kernel<<<grid, kTeam * 32, smem, s>>>(A, B, static_cast<const WinRecord*>(wins), n_wins, wins_cap, counter, subcnt,
                                          nsub, split, ccol, out, wbits, negflag, row_flag, err);
  };
  if (negflag) go(k_num_winteam<float>, static_cast<float*>(cval));
  else go(k_num_winteam<double>, static_cast<double*>(cval));
  return 1;
}

}  // namespace spg
