// binning.cu -- per-tile Gaussian lists (Sec. 3: each pixel's list of the
// Gaussians that cover it, sorted by depth).
//
// The lists are the (tile, depth, id)-ordered pairs of every visible
// (view, Gaussian) row with every tile of its rect.  Instead of sorting all
// P pairs, the sort works on rows and on row x super-tile items (a
// super-tile is 8x8 tiles), and the pairs are only ever written once, into
// their final slots:
//   1. drop the rows without tiles (an ordered compaction in the one-launch sort;
//      above 2M rows the depth sort's first pass reads the rows and leaves them out);
//   2. stable LSD radix sort of the visible rows by FP32 depth bits, on the
//      bits that vary over the visible rows (digits of up to 8 bits: 3 passes
//      for a range of up to 24 bits; ties keep row order = Gaussian id order);
//   3. gather every row's rect in depth order (16-bit packed); block scans
//      give the pair count P and each block's first super-tile item (count
//      Q <= P);
//   4. duplicate: each block of rows scans its rows' item offsets and writes
//      (super-tile, row) for the super-tiles each rect meets, in depth order
//      (4 consecutive items per thread, owners by binary search);
//   5. stable radix sort of the items by super-tile id (one pass for up to
//      256 super-tiles), so every super-tile holds its rows in depth order;
//   6. per segment of 1024 rows of a super-tile: each row's rect within the
//      super-tile and per-tile counts; scans over segments and over all
//      tiles give every tile's list start (the ranges);
//   7. expansion: each segment writes its rows into the lists of the tiles
//      they cover, a warp per tile row, ranked by warp scans, which keeps the
//      depth order.
// The result is exactly the order of a 64-bit (tile << 32 | depth) key sort
// with ties by Gaussian id.
//
// All kernels read their element counts from device memory and use grids
// sized from host-known upper bounds (blocks beyond the actual counts leave
// at once), so the whole sequence can be captured in a CUDA graph (no host
// synchronisation needed).  Up to 2M rows steps 1 to 3 are one cooperative
// launch whose blocks meet at grid barriers with bounded waits
// (depth_sort_kernel); no other kernel waits on another block: where a
// single-block scan follows one, its last block to finish runs the scan (each
// block counts its arrival after a __threadfence).
#include <cuda.h>

#include <algorithm>
#include <mutex>

#include <atomic>

#include "gs_internal.cuh"

namespace gs {
namespace {

constexpr int kScanThreads = 256;
// Scan blocks: ITEMS rows per thread (4 or 16, chosen from the row count at
// launch); the workspace is sized for the smaller blocks (the most blocks).
constexpr int kScanItems = 4;
constexpr int kScanTile = kScanThreads * kScanItems;  // 1024 rows per block

// ----------------------------------------------------------------------------
// Block-wide exclusive scan helpers (256 threads).
// ----------------------------------------------------------------------------
__device__ __forceinline__ unsigned long long warp_incl_scan(unsigned long long x) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  return x;
}

// Returns the exclusive prefix of x over the block; *total receives the block
// total in every thread.
__device__ __forceinline__ unsigned long long block_excl_scan(unsigned long long x,
                                                              unsigned long long* total) {
  __shared__ unsigned long long s_w[kScanThreads / 32 + 1];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  unsigned long long inc = warp_incl_scan(x);
  if (lane == 31) s_w[w] = inc;
  __syncthreads();
  if (w == 0) {
    unsigned long long t = lane < kScanThreads / 32 ? s_w[lane] : 0ull;
    unsigned long long ti = warp_incl_scan(t);
    if (lane < kScanThreads / 32) s_w[lane] = ti - t;
    if (lane == 31) s_w[kScanThreads / 32] = ti;
  }
  __syncthreads();
  unsigned long long r = s_w[w] + inc - x;
  *total = s_w[kScanThreads / 32];
  __syncthreads();
  return r;
}

// The block's total of x (256 threads), in every thread.
__device__ __forceinline__ unsigned long long block_sum(unsigned long long x) {
  __shared__ unsigned long long s_ws[kScanThreads / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  if (lane == 0) s_ws[w] = x;
  __syncthreads();
  unsigned long long t = 0ull;
#pragma unroll
  for (int k = 0; k < kScanThreads / 32; ++k) t += s_ws[k];
  __syncthreads();  // s_ws is read by every thread before a later call reuses it
  return t;
}

// A CTA's arrival at the end of a kernel whose last CTA goes on to a step
// over every CTA's results (a scan of the block sums, say), in place of a
// separate single-CTA launch.  Each CTA makes its results visible (a fence by one
// thread behind a block barrier) before it counts itself, so the CTA that counts
// last sees all of them; it reads them through L2 (__ldcg).  No CTA waits for
// another.
// The counter is zeroed with the pipeline's counters before the launch.
// Returns true in every thread of the last CTA.
__device__ __forceinline__ bool last_block_arrives(unsigned long long* counter,
                                                   unsigned long long expected) {
  __shared__ int s_last;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();  // (after the block barrier: covers the whole CTA's results)
    s_last = atomicAdd(counter, 1ull) == expected - 1ull ? 1 : 0;
  }
  __syncthreads();
  const bool last = s_last != 0;
  if (last) __threadfence();
  return last;
}

__device__ __forceinline__ long long scan_blocks_dev(unsigned long long* block_sums, int nblocks);

// Exclusive scan of the block sums in one block (in place); returns
// the grand total.  Each warp takes a contiguous chunk of the sums: its total
// (a lane's loads in flight together), one scan of the warp totals, then the
// chunk again with the warp's running offset -- no block-wide barrier per
// round of 256 sums (cfg3-sized inputs have ~6,000 blocks).
__device__ __forceinline__ long long scan_blocks_dev(unsigned long long* block_sums, int nblocks) {
  constexpr int NW = kScanThreads / 32;
  __shared__ unsigned long long s_wt[NW + 1];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int per = (nblocks + NW - 1) / NW;
  const int b0 = min(nblocks, w * per), b1 = min(nblocks, b0 + per);
  unsigned long long tot = 0ull;
#pragma unroll 4
  for (int i = b0 + lane; i < b1; i += 32) tot += __ldcg(block_sums + i);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
  if (lane == 0) s_wt[w] = tot;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long run = 0ull;
    for (int k = 0; k < NW; ++k) {
      const unsigned long long x = s_wt[k];
      s_wt[k] = run;
      run += x;
    }
    s_wt[NW] = run;
  }
  __syncthreads();
  unsigned long long carry = s_wt[w];
  const long long total = (long long)s_wt[NW];
#pragma unroll 4
  for (int b = b0; b < b1; b += 32) {  // (warp-uniform)
    const int i = b + lane;
    const unsigned long long x = i < b1 ? __ldcg(block_sums + i) : 0ull;
    const unsigned long long incl = warp_incl_scan(x);
    if (i < b1) block_sums[i] = carry + incl - x;
    carry += __shfl_sync(0xffffffffu, incl, 31);
  }
  __syncthreads();  // s_wt is read by every thread before a later call reuses it
  return total;
}


// Exclusive scans of the super-tile counts (sums_q) and the pair counts
// (sums_p) over the blocks, then the capacity check: P, Q, the reported
// count, the status and the counts later stages use (0 on overflow).
struct CountsOut {
  unsigned long long* sums_q;
  unsigned long long* sums_p;
  long long capacity;
  long long *Q, *P, *q_eff, *p_eff, *num_pairs_dev;
  int* status;
};

// The totals q (super-tile items) and pp (pairs) into the counts (one thread).
__device__ __forceinline__ void counts_check(const CountsOut& o, long long q, long long pp) {
  const bool over = pp > o.capacity;
  *o.Q = q;
  *o.P = pp;
  *o.num_pairs_dev = pp;
  *o.status = over ? GS_ERR_CAPACITY : GS_OK;
  *o.p_eff = over ? 0 : pp;  // on overflow every later stage sees zero pairs
  *o.q_eff = over ? 0 : q;   // (Q <= P: a super-pair holds at least one pair)
}

__device__ __forceinline__ void scan_counts_check_dev(const CountsOut& o, int nblocks);

__global__ void __launch_bounds__(kScanThreads) scan_counts_check_kernel(const CountsOut o,
                                                                         int nblocks) {
  behind_previous();
  scan_counts_check_dev(o, nblocks);
}

__device__ __forceinline__ void scan_counts_check_dev(const CountsOut& o, int nblocks) {
  const long long q = scan_blocks_dev(o.sums_q, nblocks);
  const long long pp = scan_blocks_dev(o.sums_p, nblocks);
  if (threadIdx.x == 0) counts_check(o, q, pp);
}


// ----------------------------------------------------------------------------
// Per visible row (depth order): its tile rect clamped to the view, the
// number of pairs it makes (rect area) and the number of super-tiles its
// rect meets.  Every later stage derives counts from this same clamped rect,
// so the pair and super-tile counts agree everywhere.
// ----------------------------------------------------------------------------
static_assert(kSuperTile == 8, "super-tile masks hold 8x8 tiles");

__device__ __forceinline__ int4 view_rect(const int* rect, unsigned row, int N,
                                          const CamTable& ct) {
  int4 r = reinterpret_cast<const int4*>(rect)[row];
  const CamInfo& c = ct.c[row / (unsigned)N];
  r.x = max(r.x, 0);
  r.y = max(r.y, 0);
  r.z = min(r.z, c.TX);
  r.w = min(r.w, c.TY);
  if (r.z <= r.x || r.w <= r.y) r = make_int4(0, 0, 0, 0);
  return r;
}

// The descriptor of a rect inside a super-tile, in tiles relative to the
// super-tile's origin: bit r set when it covers tile row r, bit 8 + c when it
// covers tile column c (x0 < 8, x1 > 0, y0 < 8, y1 > 0: the rect meets it).
__device__ __forceinline__ unsigned rect_masks(int x0, int x1, int y0, int y1) {
  const unsigned cols = (0xffu << max(x0, 0)) & (0xffu >> (8 - min(x1, 8)));
  const unsigned rows = (0xffu << max(y0, 0)) & (0xffu >> (8 - min(y1, 8)));
  return rows | (cols << 8);
}

// Super-tile span [x0, x1) x [y0, y1) of a non-empty tile rect.
__device__ __forceinline__ int4 st_span(const int4 r) {
  return make_int4(r.x >> 3, r.y >> 3, ((r.z - 1) >> 3) + 1, ((r.w - 1) >> 3) + 1);
}

__device__ __forceinline__ unsigned st_count(const int4 r) {
  if (r.z <= r.x) return 0u;
  const int4 q = st_span(r);
  return (unsigned)((q.z - q.x) * (q.w - q.y));
}

// A clamped tile rect packed in 16-bit fields (x0 | y0 << 16, x1 | y1 << 16);
// views are at most 65535 tiles wide and high.
__device__ __forceinline__ uint2 pack_rect(const int4 r) {
  return make_uint2((unsigned)r.x | ((unsigned)r.y << 16), (unsigned)r.z | ((unsigned)r.w << 16));
}
__device__ __forceinline__ int4 unpack_rect(const uint2 p) {
  return make_int4((int)(p.x & 0xffffu), (int)(p.x >> 16), (int)(p.y & 0xffffu), (int)(p.y >> 16));
}

// The projection's 8-bit packed rect (gs_proj.rect8: x0 | y0 << 8 | x1 << 16 |
// y1 << 24, views of at most 255 tiles per side): the depth-ordered gather
// reads 4 bytes from an array a quarter the size of the int4 rects, most of
// which stays in L2 (a random 16-byte gather from the int4 rects fetches
// several times its size from DRAM).
__device__ __forceinline__ int4 unpack_rect8(unsigned p) {
  return make_int4((int)(p & 0xffu), (int)((p >> 8) & 0xffu), (int)((p >> 16) & 0xffu),
                   (int)(p >> 24));
}

__device__ __forceinline__ int radix_result(const unsigned* range, int bits);

// The depth-sorted rows: the buffer the sort left them in follows from the
// device-side key range (the number of passes it ran); buf0 without a range.
struct SortedRows {
  const unsigned* buf0;
  const unsigned* buf1;
  const unsigned* range;
  __device__ __forceinline__ const unsigned* get() const {
    return range && radix_result(range, 32) ? buf1 : buf0;
  }
};

// Gathers the clamped rect of every depth-ordered row (so later stages read
// them in order) and forms per-block sums of the super-tile counts and of
// the pair counts.
// The last CTA to finish scans both sums over the blocks and runs the
// capacity check (scan_counts_check_dev).
template <int ITEMS>
__global__ void __launch_bounds__(kScanThreads) rows_gather_kernel(
    const SortedRows sorted, const long long* n_dev,
    const int* rect, const unsigned* rect8, int N, const CamTable ct,
    uint2* rect_sorted, unsigned long long* arrive,
    const CountsOut co) {
  behind_previous();
  unsigned long long* sums_q = co.sums_q;
  unsigned long long* sums_p = co.sums_p;
  const unsigned* rows = sorted.get();
  const long long n = *n_dev;
  const long long base = (long long)blockIdx.x * (kScanThreads * ITEMS);
  if (base >= n) {  // (the whole CTA) no rows: zero sums
    if (threadIdx.x == 0) {
      sums_q[blockIdx.x] = 0ull;
      sums_p[blockIdx.x] = 0ull;
    }
    if (last_block_arrives(arrive, gridDim.x)) scan_counts_check_dev(co, (int)gridDim.x);
    return;
  }
  unsigned long long q = 0, pp = 0;
  // groups of kGather rows: their ids, then their rect gathers in flight
  // before any use (more per group would cost occupancy on large inputs)
  constexpr int kGather = 4;
  static_assert(ITEMS % kGather == 0, "whole groups");
#pragma unroll 1
  for (int k0 = 0; k0 < ITEMS; k0 += kGather) {
    unsigned row[kGather];
#pragma unroll
    for (int k = 0; k < kGather; ++k) {
      const long long i = base + (long long)(k0 + k) * kScanThreads + threadIdx.x;
      row[k] = i < n ? __ldcs(rows + i) : 0xffffffffu;  // streamed: evict first
    }
    int4 rr[kGather];
    if (rect8) {  // (uniform)
      unsigned p8[kGather];
#pragma unroll
      for (int k = 0; k < kGather; ++k)
        p8[k] = row[k] != 0xffffffffu && GS_IN_BOUNDS(row[k], (long long)N * ct.V, 205)
                    ? rect8[row[k]] : 0u;
#pragma unroll
      for (int k = 0; k < kGather; ++k) rr[k] = unpack_rect8(p8[k]);
    } else {
#pragma unroll
      for (int k = 0; k < kGather; ++k)
        rr[k] = row[k] != 0xffffffffu && GS_IN_BOUNDS(row[k], (long long)N * ct.V, 204)
                    ? view_rect(rect, row[k], N, ct) : make_int4(0, 0, 0, 0);
    }
#pragma unroll
    for (int k = 0; k < kGather; ++k) {
      const long long i = base + (long long)(k0 + k) * kScanThreads + threadIdx.x;
      if (i < n) {
        const int4 r = rr[k];
        __stcs(rect_sorted + i, pack_rect(r));  // streamed: keeps rect8 in L2
        q += st_count(r);
        pp += (unsigned long long)((r.z - r.x) * (r.w - r.y));
      }
    }
  }
  const unsigned long long tq = block_sum(q), tp = block_sum(pp);
  if (threadIdx.x == 0) {
    sums_q[blockIdx.x] = tq;
    sums_p[blockIdx.x] = tp;
  }
  if (last_block_arrives(arrive, gridDim.x)) scan_counts_check_dev(co, (int)gridDim.x);
}

// ----------------------------------------------------------------------------
// Stable LSD radix sort of (u32 key, u32 value) pairs, up to 8-bit digits,
// reduce-then-scan with a fixed grid.  Each block owns a contiguous chunk of
// whole 2048-item tiles; n is read from device memory.
//
// The depth sort reads the rows themselves in its first pass (RadixRows):
// the visible rows' depth bits with their row ids, the culled rows dropped,
// so no separate compaction runs.  That pass's upsweep folds in the visible
// rows' key range (smallest and largest depth bits); the later passes sort
// digits of (key - min) on the range's significant bits, their number and
// width following from the range on the device (radix_plan).  The kernels of
// passes beyond the plan return at once, so the launch sequence, and a graph
// of it, is fixed.  The result is in buffer (passes mod 2).
// ----------------------------------------------------------------------------
constexpr int kRadixThreads = 256;
constexpr int kRadixWarps = kRadixThreads / 32;
constexpr int kRadixIpt = 8;                                // items per thread per tile
constexpr int kRadixTile = kRadixThreads * kRadixIpt;       // 2048
constexpr int kRadixMaxBits = 8;
constexpr int kRadixBins = 1 << kRadixMaxBits;              // 256
constexpr int kRadixMaxPasses = (32 + kRadixMaxBits - 1) / kRadixMaxBits;  // 4
static_assert(kRadixThreads == kRadixBins, "the scatter's threads own one digit each");

struct RadixPlan {
  unsigned kmin;  // subtracted from every key
  int passes;
  int d0;         // digit width of the first pass
  int dbits;      // digit width of the later passes
};

// bits: significant bits of (key - kmin), in digits of equal width.
__host__ __device__ __forceinline__ RadixPlan radix_plan_bits(unsigned kmin, int bits) {
  RadixPlan p;
  p.kmin = kmin;
  p.passes = (bits + kRadixMaxBits - 1) / kRadixMaxBits;
  p.dbits = p.passes ? (bits + p.passes - 1) / p.passes : 0;
  p.d0 = p.dbits;
  return p;
}

// range (device, nullable): [0] = ~(smallest key), [1] = largest key, both
// folded in with atomicMax from zero (no key: range[0] = range[1] = 0, an
// empty range).  Without a range every one of `bits` bits is sorted.
//
// With a range the first pass reads the rows themselves and runs before the
// range is known (its upsweep folds the range in): its digit is the low byte
// of the key.  The smallest key is therefore rounded down to a multiple of
// 256, which leaves the low byte of (key - kmin) equal to that of the key;
// the later passes take the remaining significant bits of (key - kmin) in
// digits of equal width.  There is always at least the first pass.
__device__ __forceinline__ RadixPlan radix_plan(const unsigned* range, int bits) {
  if (!range) return radix_plan_bits(0u, bits);
  RadixPlan p;
  p.kmin = 0u;
  p.passes = 1;
  p.d0 = kRadixMaxBits;
  p.dbits = kRadixMaxBits;
  const unsigned kmin = ~__ldcg(range), kmax = __ldcg(range + 1);
  if (kmax > kmin) {
    p.kmin = kmin & ~(unsigned)(kRadixBins - 1);
    const int b = 32 - __clz(kmax - p.kmin);
    if (b > p.d0) {
      const int rest = (b - p.d0 + kRadixMaxBits - 1) / kRadixMaxBits;
      p.passes = 1 + rest;
      p.dbits = (b - p.d0 + rest - 1) / rest;
    }
  }
  return p;
}

// Bit offset of a pass's digit in (key - kmin), and its mask.
__device__ __forceinline__ int radix_shift(const RadixPlan& p, int pass) {
  return pass == 0 ? 0 : p.d0 + (pass - 1) * p.dbits;
}
__device__ __forceinline__ unsigned radix_mask(const RadixPlan& p, int pass) {
  return (1u << (pass == 0 ? p.d0 : p.dbits)) - 1u;
}
__device__ __forceinline__ unsigned radix_digit(unsigned key, const RadixPlan& p, int shift,
                                                unsigned mask) {
  return ((key - p.kmin) >> shift) & mask;
}

// Rows as the first pass's input (the depth sort): the key of row j is the
// bits of depth[j], its value j, and only the rows with tiles_touched[j] > 0
// take part (the visible rows: depth > near_z > 0, so the bits order like
// the values).  The pass writes the visible rows' count to *n_vis.
struct RadixRows {
  const float* depth;
  const unsigned* tiles_touched;
  long long n;     // rows
  long long* n_vis;
};

// Arguments of one pass.
struct RadixPass {
  const unsigned* keys_in;
  const unsigned* vals_in;
  unsigned* keys_out;
  unsigned* vals_out;
  const long long* n_dev;  // item count (the later passes with rows)
  const unsigned* range;   // device key range or nullptr
  int bits;                // significant bits without a range
  int pass;                // pass index
  unsigned* hist;          // [256][grid] per-CTA digit counts, then their scan
  unsigned* digit_tot;     // [256] items per digit
  int keys_last;           // write the keys in the last pass too
  RadixRows rows;          // rows.depth set: the first pass reads the rows
  __device__ __forceinline__ bool from_rows() const { return pass == 0 && rows.depth; }
  __device__ __forceinline__ long long count() const { return from_rows() ? rows.n : *n_dev; }
};

__device__ __forceinline__ long long radix_chunk(long long n, int nblocks) {
  long long per = (n + nblocks - 1) / nblocks;
  return (per + kRadixTile - 1) / kRadixTile * kRadixTile;
}

// CTAs of a pass that own items: the grid is sized for the bound on the
// item count, so with few items (a small visible set) most CTAs own none;
// they leave at once and the histogram scan covers only the active ones.
__device__ __forceinline__ int radix_active(long long n, int nblocks) {
  const long long chunk = radix_chunk(n, nblocks);
  return chunk > 0 ? (int)min((long long)nblocks, (n + chunk - 1) / chunk) : 0;
}

// Item j of a pass: key, value and whether it takes part.
__device__ __forceinline__ void radix_load(const RadixPass& a, long long j, long long end,
                                           unsigned& k, unsigned& v, bool& in) {
  if (a.from_rows()) {
    const unsigned t = j < end ? a.rows.tiles_touched[j] : 0u;
    k = j < end ? __float_as_uint(a.rows.depth[j]) : 0u;
    in = t > 0u;
    v = (unsigned)j;
  } else {
    in = j < end;
    k = in ? a.keys_in[j] : 0u;
    v = in ? a.vals_in[j] : 0u;
  }
}

__global__ void __launch_bounds__(kRadixThreads) radix_upsweep_kernel(const RadixPass a) {
  behind_previous();
  // the first pass over rows folds the key range in, so it cannot read the
  // plan: its digit is the low byte of the key
  const bool rows = a.from_rows();
  RadixPlan pl;
  if (rows) {
    pl.kmin = 0u;
    pl.passes = 1;
    pl.d0 = pl.dbits = kRadixMaxBits;
  } else {
    pl = radix_plan(a.range, a.bits);
    if (a.pass >= pl.passes) return;  // (the whole grid)
  }
  const int shift = radix_shift(pl, a.pass);
  const unsigned mask = radix_mask(pl, a.pass);
  unsigned* hist = a.hist;  // [256][nblocks]
  __shared__ unsigned s_h[kRadixWarps][kRadixBins];
  __shared__ unsigned s_kmin[kRadixWarps], s_kmax[kRadixWarps];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const long long n = a.count();
  if ((int)blockIdx.x >= radix_active(n, gridDim.x)) return;  // (the whole CTA)
  const long long chunk = radix_chunk(n, gridDim.x);
  const long long b0 = (long long)blockIdx.x * chunk;
  const long long b1 = min(n, b0 + chunk);
  // kRadixIpt loads in flight per thread; the first tile's are requested
  // before the histogram is cleared
  unsigned kk[kRadixIpt], unused;
  bool in[kRadixIpt];
#pragma unroll
  for (int i = 0; i < kRadixIpt; ++i)
    radix_load(a, b0 + i * kRadixThreads + threadIdx.x, b1, kk[i], unused, in[i]);
  for (int i = threadIdx.x; i < kRadixWarps * kRadixBins; i += kRadixThreads)
    (&s_h[0][0])[i] = 0u;
  __syncthreads();
  unsigned kmin = 0xffffffffu, kmax = 0u;  // (rows) range of the keys taking part
  for (long long t0 = b0; t0 < b1; t0 += kRadixTile) {
    if (t0 != b0) {
#pragma unroll
      for (int i = 0; i < kRadixIpt; ++i)
        radix_load(a, t0 + i * kRadixThreads + threadIdx.x, b1, kk[i], unused, in[i]);
    }
#pragma unroll
    for (int i = 0; i < kRadixIpt; ++i) {
      if (in[i]) {
        atomicAdd(&s_h[w][radix_digit(kk[i], pl, shift, mask)], 1u);
        if (rows) {
          kmin = min(kmin, kk[i]);
          kmax = max(kmax, kk[i]);
        }
      }
    }
  }
  if (rows) {
    kmin = __reduce_min_sync(0xffffffffu, kmin);
    kmax = __reduce_max_sync(0xffffffffu, kmax);
    if (lane == 0) {
      s_kmin[w] = kmin;
      s_kmax[w] = kmax;
    }
  }
  __syncthreads();
  for (int d = threadIdx.x; d < kRadixBins; d += kRadixThreads) {
    unsigned s = 0;
    for (int k = 0; k < kRadixWarps; ++k) s += s_h[k][d];
    hist[(long long)d * gridDim.x + blockIdx.x] = s;
  }
  if (rows && threadIdx.x == 0) {
    for (int q = 1; q < kRadixWarps; ++q) {
      kmin = min(kmin, s_kmin[q]);
      kmax = max(kmax, s_kmax[q]);
    }
    if (kmin <= kmax) {  // (folded in from zero: range[0] holds the complement)
      atomicMax(const_cast<unsigned*>(a.range), ~kmin);
      atomicMax(const_cast<unsigned*>(a.range) + 1, kmax);
    }
  }
}

// Per-digit exclusive scan over the blocks: block d scans hist[d][0..Ga) in
// place (Ga = the pass's active CTAs) and writes the digit total to
// totals[d].  G <= 1024.
__global__ void __launch_bounds__(kScanThreads) radix_scan_kernel(const RadixPass a, int G) {
  behind_previous();
  const RadixPlan pl = radix_plan(a.range, a.bits);
  if (a.pass >= pl.passes) return;
  unsigned* totals = a.digit_tot;
  unsigned* h = a.hist + (long long)blockIdx.x * G;
  const int Ga = radix_active(a.count(), G);
  constexpr int kPer = 4;  // 256 threads x 4 >= 1024 blocks
  unsigned loc[kPer];
  unsigned long long s = 0;
  const int first = threadIdx.x * kPer;
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    loc[k] = first + k < Ga ? h[first + k] : 0u;
    s += loc[k];
  }
  unsigned long long tot;
  unsigned long long off = block_excl_scan(s, &tot);
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    if (first + k < Ga) h[first + k] = (unsigned)off;
    off += loc[k];
  }
  if (threadIdx.x == 0) totals[blockIdx.x] = (unsigned)tot;
}

// Scatter of one radix pass (digit = (key >> shift) & dmask, at most 8
// bits).  Per 2048-item tile: digits ranked within each warp from bit
// ballots (stable within the tile), the tile is reordered by digit in shared
// memory, then written out so that consecutive threads store consecutive
// addresses of one digit's run (coalesced), and each digit's running global
// offset advances by the tile's count.  The next tile's keys and values are
// loaded into registers while the current one is ranked and written.
#ifndef GS_RADIX_CTAS
#define GS_RADIX_CTAS 3  // resident scatter CTAs per SM the register budget targets
#endif
__global__ void __launch_bounds__(kRadixThreads, GS_RADIX_CTAS) radix_downsweep_kernel(
    const RadixPass a) {
  behind_previous();
  const RadixPlan pl = radix_plan(a.range, a.bits);
  if (a.pass >= pl.passes) return;
  unsigned* keys_out = a.keys_out;
  unsigned* vals_out = a.vals_out;
  const unsigned* offsets = a.hist;
  const unsigned* totals = a.digit_tot;
  const int shift = radix_shift(pl, a.pass);
  const unsigned mask = radix_mask(pl, a.pass);
  const bool wkeys = a.keys_last || a.pass + 1 < pl.passes;
  __shared__ unsigned s_wc[kRadixWarps][kRadixBins + 1];  // per-warp digit counters (+ dummy)
  __shared__ unsigned s_pre[kRadixWarps][kRadixBins];     // per-warp start within the digit's run
  __shared__ unsigned s_off[kRadixBins];                  // tile-local start per digit
  __shared__ unsigned s_gl[kRadixBins];                   // global minus tile-local start per digit
  __shared__ unsigned s_ws[kRadixWarps];                  // warp totals of the digit scan
  __shared__ unsigned s_nt;                               // items of the tile taking part
  __shared__ unsigned s_key[kRadixTile];
  __shared__ unsigned s_val[kRadixTile];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const unsigned lt_mask = (1u << lane) - 1u;
  const long long n = a.count();
  if ((int)blockIdx.x >= radix_active(n, gridDim.x)) return;  // (the whole CTA)
  const long long chunk = radix_chunk(n, gridDim.x);
  const long long b0 = (long long)blockIdx.x * chunk;
  const long long b1 = min(n, b0 + chunk);
  // the first tile's keys and values are requested before the digit bases
  // (independent loads, their latency overlaps the scan)
  unsigned nk[kRadixIpt], nv[kRadixIpt];
  unsigned nin = 0u;  // bit i: item i takes part
  const int lbase = w * (32 * kRadixIpt) + lane;
#pragma unroll
  for (int i = 0; i < kRadixIpt; ++i) {
    bool in;
    radix_load(a, b0 + lbase + i * 32, b1, nk[i], nv[i], in);
    nin |= (in ? 1u : 0u) << i;
  }
  // thread d owns digit d (kRadixThreads == kRadixBins): its running global
  // offset = exclusive scan of the digit totals + this CTA's offset
  const int dd = threadIdx.x;
  unsigned gbase;
  {
    const unsigned off = offsets[(long long)dd * gridDim.x + blockIdx.x];
    unsigned long long tot;
    gbase = (unsigned)block_excl_scan(totals[dd], &tot) + off;
    // the first pass over rows reports the count of the rows taking part
    if (a.from_rows() && blockIdx.x == 0 && threadIdx.x == 0) *a.rows.n_vis = (long long)tot;
  }
  for (int i = threadIdx.x; i < kRadixWarps * (kRadixBins + 1); i += kRadixThreads)
    (&s_wc[0][0])[i] = 0u;
  __syncthreads();
  // Four barriers per tile.  The counters s_wc are read and cleared between
  // the first two, so the next tile's ranking may start while this tile is
  // still being written out; the next tile's first barrier orders that
  // write-out before the shared tile and the offsets are overwritten.
  for (long long t0 = b0; t0 < b1; t0 += kRadixTile) {
    unsigned k[kRadixIpt], v[kRadixIpt], dg[kRadixIpt], loc[kRadixIpt];
#pragma unroll
    for (int i = 0; i < kRadixIpt; ++i) {
      k[i] = nk[i];
      v[i] = nv[i];
      dg[i] = (nin >> i) & 1u ? radix_digit(k[i], pl, shift, mask) : (unsigned)kRadixBins;
    }
    const long long t1 = t0 + kRadixTile;
    if (t1 < b1) {
      nin = 0u;
#pragma unroll
      for (int i = 0; i < kRadixIpt; ++i) {
        bool in;
        radix_load(a, t1 + lbase + i * 32, b1, nk[i], nv[i], in);
        nin |= (in ? 1u : 0u) << i;
      }
    }
#pragma unroll
    for (int i = 0; i < kRadixIpt; ++i) {
      // lanes holding the same digit: one ballot per digit bit plus validity
      const bool valid = dg[i] < (unsigned)kRadixBins;
      const unsigned vm = __ballot_sync(0xffffffffu, valid);
      unsigned peers = valid ? vm : ~vm;
      // (digit bits at or above the pass's width are zero in every lane:
      // their ballots leave peers unchanged)
#pragma unroll
      for (int b = 0; b < kRadixMaxBits; ++b) {
        const bool bit = (dg[i] >> b) & 1u;
        const unsigned m = __ballot_sync(0xffffffffu, bit);
        peers &= bit ? m : ~m;
      }
      const unsigned rank = __popc(peers & lt_mask);
      const unsigned base = s_wc[w][dg[i]];
      __syncwarp();
      if (rank == 0) s_wc[w][dg[i]] = base + __popc(peers);
      __syncwarp();
      loc[i] = base + rank;
    }
    __syncthreads();
    unsigned run = 0, inc;
    {
      // digit dd: prefix over the warps (counters cleared for the next
      // tile), then a 32-bit scan of the tile counts over the digits
#pragma unroll
      for (int ww = 0; ww < kRadixWarps; ++ww) {
        const unsigned c = s_wc[ww][dd];
        s_pre[ww][dd] = run;
        s_wc[ww][dd] = 0u;
        run += c;
      }
      inc = run;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
      }
      if (lane == 31) s_ws[w] = inc;
    }
    __syncthreads();
    {
      unsigned wo = 0;
#pragma unroll
      for (int ww = 0; ww < kRadixWarps - 1; ++ww) wo += ww < w ? s_ws[ww] : 0u;
      const unsigned off = wo + inc - run;
      s_off[dd] = off;
      s_gl[dd] = gbase - off;
      gbase += run;
      if (dd == kRadixBins - 1) s_nt = off + run;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kRadixIpt; ++i) {
      if (dg[i] < (unsigned)kRadixBins) {
        const unsigned lp = s_off[dg[i]] + s_pre[w][dg[i]] + loc[i];
        s_key[lp] = k[i];
        s_val[lp] = v[i];
      }
    }
    __syncthreads();
    const int nt = (int)s_nt;
    for (int i = threadIdx.x; i < nt; i += kRadixThreads) {
      const unsigned kk = s_key[i];
      const unsigned pos = s_gl[radix_digit(kk, pl, shift, mask)] + (unsigned)i;
      if (!GS_IN_BOUNDS(pos, n, 202)) continue;
      if (wkeys) keys_out[pos] = kk;
      vals_out[pos] = s_val[i];
    }
  }
}

// Buffer index (0 or 1) holding the sorted result.
__device__ __forceinline__ int radix_result(const unsigned* range, int bits) {
  return radix_plan(range, bits).passes & 1;
}

// ----------------------------------------------------------------------------
// Steps 1 to 3 in one cooperative launch, for up to kCoopRows rows: compaction
// of the visible rows, the depth sort and the depth-ordered gather with its
// counts, with a grid barrier between dependent phases.  As separate kernels
// they are 13 launches of 4 to 10 us each whatever the rows, most of it
// launching, filling and draining the chip and re-reading arguments: 10k rows
// took about 75 us, 1M rows of which 70k are visible about 110 us.  Here the
// counts a phase needs from all CTAs are summed by each CTA for itself, and up to
// kCountAhead visible rows a pass's scatter also counts the next pass's digits (one
// reduction per item into the chunk that will own it), so a pass is one phase.
// Beyond, those reductions collide in L2 and a CTA counts its own chunk in shared
// memory instead, a phase more.  Above kCoopRows the passes are long enough for the
// separate kernels, whose three CTAs per SM hide more latency.
//
// Measured, whole list construction replayed from a graph, us:
//   counted ahead / counted in the pass, all rows visible: 20k 66 / 66, 60k 76 / 76,
//   80k 76 / 75, 200k 90 / 87, 1M 168 / 152, 2.1M 281 / 247; 7 % visible (8k: 560 rows)
//   51 / 56, 50k 62 / 64, 1M (70k visible) 86 / 84.
//   one launch / separate kernels, all rows visible: 100k 80 / 80, 1M 152 / 148, 1.5M
//   197 / 182, 2.1M 247 / 239, 2.6M 295 / 270, 6M 560 / 479; 30 % visible: 1M 98 / 113,
//   2.1M 139 / 150, 6M 270 / 253; 7 %: 1M 84 / 105, 2.1M 94 / 127, 6M 162 / 177.
//   (The host knows the rows, not how many are visible: the line lies where the one
//   launch costs at most 8 % with all of them visible and gains a quarter with few.)
//   one cluster / the grid, all rows visible: 2k 55 / 60, 16k 66 / 68, 32,768 70 / 72,
//   40k (two tiles per CTA of the cluster) 88 / 74; 7 % visible: 32,768 58 / 62.
//
// Every CTA is resident (cooperative launch).  The barrier's wait is bounded:
// when it runs out, the CTA reports GS_ERR_TIMEOUT and leaves, the others run
// out in turn, and the later kernels find zero counts.
// ----------------------------------------------------------------------------
constexpr int kCoopThreads = 512;
constexpr int kCoopWarps = kCoopThreads / 32;
constexpr int kCoopTile = kCoopThreads * kRadixIpt;  // 4096 items
constexpr int kCoopShift = 12;                       // log2(kCoopTile)
constexpr int kCoopBlock = kScanThreads;             // rows per block of the expansion
constexpr int kCoopGrid = 152;                       // most CTAs (one per SM)
constexpr long long kCoopRows = 2ll << 20;
// Row groups of 32 of a warp: at most kCoopRows over the warps of the whole
// grid (smaller grids take fewer rows: a CTA per 1,024 rows).
constexpr int kCoopGroups = (int)((kCoopRows / (kCoopGrid * kCoopWarps) + 31) / 32 + 1);
// Up to this many rows the grid is one cluster of up to 8 CTAs.
constexpr int kCoopCluster = 8;
constexpr long long kClusterRows = (long long)kCoopCluster * kCoopTile;
static_assert(kClusterRows / (kCoopCluster * kCoopWarps) <= 32 * kCoopGroups,
              "a warp's rows of the cluster form fit");
constexpr unsigned kCountAhead = 65536;
static_assert(kCoopTile == 1 << kCoopShift, "chunks are whole tiles");

struct CoopArgs {
  RadixRows rows;
  unsigned* k[2];
  unsigned* v[2];
  unsigned* hist;   // [passes][grid][256] digit counts of every chunk (zeroed here)
  unsigned* cnt;    // [grid] visible rows per CTA
  unsigned* range;  // [~smallest, largest] visible key (zero)
  unsigned* bar;    // barrier arrivals (zero)
  int polls;        // reads of bar after which a barrier's wait gives up
  const int* rect;
  const unsigned* rect8;
  int N;
  uint2* rect_sorted;
  unsigned long long* arrive;  // (zero)
  CountsOut co;
};

struct CoopShared {
  unsigned key[kCoopTile], val[kCoopTile];
  unsigned wc[kCoopWarps][kRadixBins + 1];  // per-warp digit counters (+ dummy)
  unsigned pre[kCoopWarps][kRadixBins];     // per-warp start within the digit's run
  unsigned off[kRadixBins];                 // tile-local start per digit
  unsigned gl[kRadixBins];                  // global minus tile-local start per digit
  unsigned part[2][kRadixBins];
  unsigned ws[kCoopWarps], ws2[kCoopWarps];
  unsigned vis[kCoopWarps][kCoopGroups];    // visible lanes of the warp's rows
  unsigned long long wt[2][9];
  int ok;
};

// Barrier number `phase` (1, 2, ...) over the grid.  CLUSTER: the grid is one
// cluster, whose hardware barrier takes a fraction of the time.  Otherwise
// through an arrival counter: false when the wait ran out.
template <bool CLUSTER>
__device__ __forceinline__ bool coop_barrier(const CoopArgs& a, CoopShared& s, unsigned phase) {
  if constexpr (CLUSTER) {
    asm volatile(
        "barrier.cluster.arrive.release.aligned;\n\t"
        "barrier.cluster.wait.acquire.aligned;" ::: "memory");
    return true;
  } else {
    __syncthreads();
    if (threadIdx.x == 0) {
      const unsigned want = phase * gridDim.x;
      __threadfence();  // (after the block barrier: covers the whole CTA's writes)
      atomicAdd(a.bar, 1u);
      int ok = 0;
      for (int i = 0; i < a.polls && !ok; ++i) {
        unsigned x;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(x) : "l"(a.bar) : "memory");
        ok = x >= want;
      }
      if (!ok) {
        *a.co.status = GS_ERR_TIMEOUT;
        *a.co.num_pairs_dev = 0;
        *a.co.P = -1;  // (for the host's read of the count)
      }
      __threadfence();
      s.ok = ok;
    }
    __syncthreads();
    return s.ok != 0;
  }
}

// Inclusive warp scan (32-bit).
__device__ __forceinline__ unsigned warp_scan32(unsigned x) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  return x;
}

template <bool CLUSTER>
__global__ void __launch_bounds__(kCoopThreads, 1) depth_sort_kernel(const CoopArgs a,
                                                                     const CamTable ct) {
  extern __shared__ __align__(16) unsigned char coop_smem[];
  CoopShared& s = *reinterpret_cast<CoopShared*>(coop_smem);
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const unsigned lt = (1u << lane) - 1u;
  const int G = gridDim.x, cta = blockIdx.x;
  const long long n_rows = a.rows.n;
  // A. visible rows of the CTA's chunk (a contiguous part per warp) and the
  //    visible rows' key range; the digit counts are cleared
  const long long sub = ((n_rows + (long long)G * kCoopWarps - 1) / ((long long)G * kCoopWarps) + 31) / 32 * 32;
  const long long r0 = ((long long)cta * kCoopWarps + w) * sub, r1 = min(n_rows, r0 + sub);
  const int groups = (int)((max(r1 - r0, 0ll) + 31) / 32);
  unsigned mine = 0u, kmin = 0xffffffffu, kmax = 0u;
#pragma unroll 8
  for (int i = 0; i < groups; ++i) {
    const long long j = r0 + 32 * i + lane;
    const unsigned t = j < r1 ? a.rows.tiles_touched[j] : 0u;
    const unsigned k = j < r1 ? __float_as_uint(a.rows.depth[j]) : 0u;
    const unsigned m = __ballot_sync(0xffffffffu, t > 0u);
    if (lane == 0) s.vis[w][i] = m;
    mine += __popc(m);
    if (t > 0u) {
      kmin = min(kmin, k);
      kmax = max(kmax, k);
    }
  }
  for (int i = tid; i < kRadixMaxPasses * kRadixBins; i += kCoopThreads)
    a.hist[(long long)cta * (kRadixMaxPasses * kRadixBins) + i] = 0u;
  kmin = __reduce_min_sync(0xffffffffu, kmin);
  kmax = __reduce_max_sync(0xffffffffu, kmax);
  if (lane == 0) {
    s.ws[w] = mine;
    if (kmin <= kmax) {
      atomicMax(a.range, ~kmin);
      atomicMax(a.range + 1, kmax);
    }
  }
  __syncthreads();
  unsigned woff = 0u, total = 0u;  // the warp's start in the CTA, the CTA's rows
#pragma unroll
  for (int i = 0; i < kCoopWarps; ++i) {
    woff += i < w ? s.ws[i] : 0u;
    total += s.ws[i];
  }
  if (tid == 0) a.cnt[cta] = total;
  unsigned phase = 1u;
  if (!coop_barrier<CLUSTER>(a, s, phase++)) return;
  // B. ordered compaction, with the first pass's digit counts
  unsigned before = 0u, all = 0u;
  if (tid < G) {
    const unsigned c = __ldcg(a.cnt + tid);
    all = c;
    before = tid < cta ? c : 0u;
  }
  before = __reduce_add_sync(0xffffffffu, before);
  all = __reduce_add_sync(0xffffffffu, all);
  if (lane == 0) {
    s.ws[w] = before;
    s.ws2[w] = all;
  }
  __syncthreads();
  before = all = 0u;
#pragma unroll
  for (int i = 0; i < kCoopWarps; ++i) {
    before += s.ws[i];
    all += s.ws2[i];
  }
  const unsigned n = all;
  if (cta == 0 && tid == 0) *a.rows.n_vis = (long long)n;
  const unsigned lo = ~__ldcg(a.range), hi = __ldcg(a.range + 1);
  const unsigned base = n ? lo : 0u;
  const int bits = n && hi > lo ? 32 - __clz(hi - lo) : 0;
  const RadixPlan pl = radix_plan_bits(base, bits);
  const unsigned dmask = (1u << pl.dbits) - 1u;  // (dbits 0: no pass)
  // chunks of `tiles` whole tiles: the chunk of tile t is t / tiles, by a reciprocal
  // that is exact below 2^16 / tiles tiles (here at most kCoopRows / kCoopTile)
  const unsigned tiles = max(1u, (n + (unsigned)G * kCoopTile - 1u) / ((unsigned)G * kCoopTile));
  const unsigned per_chunk = 65536u / tiles + 1u, chunk = tiles * kCoopTile;
  auto count = [&](int pass, unsigned pos, unsigned k) {
    const unsigned c = ((pos >> kCoopShift) * per_chunk) >> 16;
    atomicAdd(a.hist + ((long long)pass * G + c) * kRadixBins +
                  (((k - base) >> (pass * pl.dbits)) & dmask), 1u);
  };
  const bool ahead = n <= kCountAhead;  // (see the top)
  int buf = pl.passes & 1;  // (the result lands in buffer 0)
  {
    unsigned at = before + woff;
    unsigned* __restrict__ ko = a.k[buf];
    unsigned* __restrict__ vo = a.v[buf];
#pragma unroll 8
    for (int i = 0; i < groups; ++i) {
      const long long j = r0 + 32 * i + lane;
      const unsigned m = s.vis[w][i];
      if ((m >> lane) & 1u) {
        const unsigned k = __float_as_uint(a.rows.depth[j]), pos = at + __popc(m & lt);
        if (pl.passes) {
          ko[pos] = k;
          if (ahead) count(0, pos, k);
        }
        vo[pos] = (unsigned)j;
      }
      at += __popc(m);
    }
  }
  if (!coop_barrier<CLUSTER>(a, s, phase++)) return;
  // C. stable passes over the digits, as radix_downsweep_kernel
  const int chunks = (int)((n + chunk - 1u) / chunk);
  for (int pass = 0; pass < pl.passes; ++pass, buf ^= 1) {
    if (!ahead) {  // this chunk's digit counts
      if (cta < chunks) {
        const unsigned c0 = (unsigned)cta * chunk, c1 = min(n, c0 + chunk);
        for (int i = tid; i < kCoopWarps * (kRadixBins + 1); i += kCoopThreads) (&s.wc[0][0])[i] = 0u;
        __syncthreads();
        for (unsigned t0 = c0; t0 < c1; t0 += kCoopTile) {
          unsigned kk[kRadixIpt];
#pragma unroll
          for (int i = 0; i < kRadixIpt; ++i) {
            const unsigned p = t0 + tid + kCoopThreads * i;
            kk[i] = p < c1 ? __ldcg(a.k[buf] + p) : 0u;
          }
#pragma unroll
          for (int i = 0; i < kRadixIpt; ++i)
            if (t0 + tid + kCoopThreads * i < c1)
              atomicAdd(&s.wc[w][((kk[i] - base) >> (pass * pl.dbits)) & dmask], 1u);
        }
        __syncthreads();
        if (tid < kRadixBins) {
          unsigned sum = 0u;
#pragma unroll
          for (int ww = 0; ww < kCoopWarps; ++ww) sum += s.wc[ww][tid];
          a.hist[((long long)pass * G + cta) * kRadixBins + tid] = sum;
        }
      }
      if (!coop_barrier<CLUSTER>(a, s, phase++)) return;
    }
    if (cta < chunks) {
      const unsigned* __restrict__ ki = a.k[buf];
      const unsigned* __restrict__ vi = a.v[buf];
      const unsigned c0 = (unsigned)cta * chunk, c1 = min(n, c0 + chunk);
      // (a tile's items are requested while the one before is ranked)
      unsigned nk[kRadixIpt], nv[kRadixIpt];
      auto request = [&](unsigned t0) {
#pragma unroll
        for (int i = 0; i < kRadixIpt; ++i) {
          const unsigned p = t0 + w * (32 * kRadixIpt) + lane + 32 * i;
          nk[i] = p < c1 ? __ldcg(ki + p) : 0u;
          nv[i] = p < c1 ? __ldcg(vi + p) : 0u;
        }
      };
      request(c0);
      // digit starts: the digits below over all chunks, then the chunks before
      const int dd = tid & (kRadixBins - 1), half = tid >> kRadixMaxBits;
      const unsigned* __restrict__ h = a.hist + (long long)pass * G * kRadixBins + dd;
      unsigned hb = 0u, ha = 0u;
#pragma unroll 8
      for (int c = half; c < chunks; c += 2) {
        const unsigned x = __ldcg(h + c * kRadixBins);
        ha += x;
        hb += c < cta ? x : 0u;
      }
      if (half) {
        s.part[0][dd] = hb;
        s.part[1][dd] = ha;
      }
      for (int i = tid; i < kCoopWarps * (kRadixBins + 1); i += kCoopThreads) (&s.wc[0][0])[i] = 0u;
      __syncthreads();
      unsigned gbase = 0u;
      if (!half) {
        hb += s.part[0][dd];
        ha += s.part[1][dd];
        gbase = warp_scan32(ha);
        if (lane == 31) s.ws[w] = gbase;
      }
      __syncthreads();
      if (!half) {
        unsigned wo = 0u;
        for (int i = 0; i < kRadixBins / 32; ++i) wo += i < w ? s.ws[i] : 0u;
        gbase += wo - ha + hb;
      }
      unsigned* __restrict__ ko = a.k[buf ^ 1];
      unsigned* __restrict__ vo = a.v[buf ^ 1];
      const int dshift = pass * pl.dbits;
      const bool more = pass + 1 < pl.passes;
      for (unsigned t0 = c0; t0 < c1; t0 += kCoopTile) {
        unsigned k[kRadixIpt], v[kRadixIpt], dg[kRadixIpt], loc[kRadixIpt];
        const unsigned p0 = t0 + w * (32 * kRadixIpt) + lane;
#pragma unroll
        for (int i = 0; i < kRadixIpt; ++i) {
          k[i] = nk[i];
          v[i] = nv[i];
          dg[i] = p0 + 32 * i < c1 ? ((k[i] - base) >> dshift) & dmask : (unsigned)kRadixBins;
        }
        if (t0 + kCoopTile < c1) request(t0 + kCoopTile);
#pragma unroll
        for (int i = 0; i < kRadixIpt; ++i) {
          const bool valid = dg[i] < (unsigned)kRadixBins;
          const unsigned vm = __ballot_sync(0xffffffffu, valid);
          unsigned peers = valid ? vm : ~vm;
#pragma unroll
          for (int b = 0; b < kRadixMaxBits; ++b) {
            const bool bit = (dg[i] >> b) & 1u;
            const unsigned m = __ballot_sync(0xffffffffu, bit);
            peers &= bit ? m : ~m;
          }
          const unsigned rank = __popc(peers & lt);
          const unsigned old = s.wc[w][dg[i]];
          __syncwarp();
          if (rank == 0) s.wc[w][dg[i]] = old + __popc(peers);
          __syncwarp();
          loc[i] = old + rank;
        }
        __syncthreads();
        unsigned run = 0u, inc = 0u;
        if (tid < kRadixBins) {
#pragma unroll
          for (int ww = 0; ww < kCoopWarps; ++ww) {
            const unsigned c = s.wc[ww][tid];
            s.pre[ww][tid] = run;
            s.wc[ww][tid] = 0u;
            run += c;
          }
          inc = warp_scan32(run);
          if (lane == 31) s.ws2[w] = inc;
        }
        __syncthreads();
        if (tid < kRadixBins) {
          unsigned wo = 0u;
#pragma unroll
          for (int ww = 0; ww < kRadixBins / 32 - 1; ++ww) wo += ww < w ? s.ws2[ww] : 0u;
          const unsigned off = wo + inc - run;
          s.off[tid] = off;
          s.gl[tid] = gbase - off;
          gbase += run;
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < kRadixIpt; ++i) {
          if (dg[i] < (unsigned)kRadixBins) {
            const unsigned lp = s.off[dg[i]] + s.pre[w][dg[i]] + loc[i];
            s.key[lp] = k[i];
            s.val[lp] = v[i];
          }
        }
        __syncthreads();
        const unsigned nt = min(c1 - t0, (unsigned)kCoopTile);
        for (unsigned i = tid; i < nt; i += kCoopThreads) {
          const unsigned kk = s.key[i];
          const unsigned pos = s.gl[((kk - base) >> dshift) & dmask] + i;
          if (!GS_IN_BOUNDS(pos, n, 202)) continue;
          if (more) {
            ko[pos] = kk;
            if (ahead) count(pass + 1, pos, kk);
          }
          vo[pos] = s.val[i];
        }
      }
    }
    if (!coop_barrier<CLUSTER>(a, s, phase++)) return;
  }
  // D. the rects in depth order and the counts per block of 256 rows (the
  //    blocks rows_expand_kernel<1> takes), a warp per block and 8 rows per
  //    lane; the last CTA scans them
  const unsigned* __restrict__ rows = a.v[0];
  const int nb = (int)((n + kCoopBlock - 1) / kCoopBlock);
  for (int b = cta + G * w; b < nb; b += G * kCoopWarps) {
    unsigned long long q = 0ull, pp = 0ull;
    constexpr int kPer = kCoopBlock / 32;
    unsigned row[kPer];
    int4 rr[kPer];
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const unsigned at = (unsigned)b * kCoopBlock + 32 * i + lane;
      row[i] = at < n ? __ldcg(rows + at) : 0xffffffffu;
    }
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      rr[i] = make_int4(0, 0, 0, 0);
      if (row[i] != 0xffffffffu && GS_IN_BOUNDS(row[i], n_rows, 205))
        rr[i] = a.rect8 ? unpack_rect8(a.rect8[row[i]]) : view_rect(a.rect, row[i], a.N, ct);
    }
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const unsigned at = (unsigned)b * kCoopBlock + 32 * i + lane;
      if (at < n) {
        a.rect_sorted[at] = pack_rect(rr[i]);
        q += st_count(rr[i]);
        pp += (unsigned long long)((rr[i].z - rr[i].x) * (rr[i].w - rr[i].y));
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      q += __shfl_xor_sync(0xffffffffu, q, o);
      pp += __shfl_xor_sync(0xffffffffu, pp, o);
    }
    if (lane == 0) {
      a.co.sums_q[b] = q;
      a.co.sums_p[b] = pp;
    }
  }
  if (!last_block_arrives(a.arrive, (unsigned long long)G)) return;
  // warps 0-7 scan the super-tile counts, 8-15 the pair counts: each warp a
  // contiguous part of the blocks
  const int which = w >> 3, wi = w & 7;
  unsigned long long* sums = which ? a.co.sums_p : a.co.sums_q;
  const int per = (nb + 7) / 8, b0 = min(nb, wi * per), b1 = min(nb, b0 + per);
  unsigned long long tot = 0ull;
#pragma unroll 4
  for (int i = b0 + lane; i < b1; i += 32) tot += __ldcg(sums + i);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
  if (lane == 0) s.wt[which][wi] = tot;
  __syncthreads();
  unsigned long long carry = 0ull, grand = 0ull;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    carry += i < wi ? s.wt[which][i] : 0ull;
    grand += s.wt[which][i];
  }
  for (int b = b0; b < b1; b += 32) {  // (warp-uniform)
    const int i = b + lane;
    const unsigned long long x = i < b1 ? __ldcg(sums + i) : 0ull;
    const unsigned long long incl = warp_incl_scan(x);
    if (i < b1) sums[i] = carry + incl - x;
    carry += __shfl_sync(0xffffffffu, incl, 31);
  }
  if (tid == 0) {
    unsigned long long pp = 0ull;
    for (int i = 0; i < 8; ++i) pp += s.wt[1][i];
    counts_check(a.co, (long long)grand, (long long)pp);
  }
}

// A barrier's wait, about a second.  The bounds-checked debug build lets a test
// shorten it for the calling thread's next calls (gs_debug_sort_polls).
constexpr int kBarrierPolls = 1 << 21;
#ifdef GS_DEBUG_BOUNDS
thread_local int g_barrier_polls = kBarrierPolls;
int barrier_polls() { return g_barrier_polls; }
#else
int barrier_polls() { return kBarrierPolls; }
#endif

template <bool CLUSTER>
cudaError_t allow_coop_smem() {
  return cudaFuncSetAttribute(depth_sort_kernel<CLUSTER>,
                              cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(CoopShared));
}

// Whether the current device can hold depth_sort_kernel's largest grid at once
// (not a part of a GPU with fewer SMs); cached per device.
bool coop_available() {
  static std::atomic<int> cache[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
  const int c = cache[dev].load(std::memory_order_relaxed);
  if (c) return c > 0;
  int per_sm = 0, sms = 0, coop = 0;
  int v = -1;
  if (allow_coop_smem<false>() == cudaSuccess &&
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, depth_sort_kernel<false>,
                                                    kCoopThreads, sizeof(CoopShared)) ==
          cudaSuccess &&
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
      cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) == cudaSuccess && coop &&
      per_sm > 0 && sms >= kCoopGrid)
    v = 1;
  cudaGetLastError();
  cache[dev].store(v, std::memory_order_relaxed);
  return v > 0;
}

// ----------------------------------------------------------------------------
// Super-pair generation, per-tile expansion.
// ----------------------------------------------------------------------------
// Super-pair duplication.  Each CTA takes one scan block of the depth-sorted
// visible rows (the blocks of rows_gather_kernel, whose item counts are
// already scanned into the blocks' item bases), scans its rows' super-tile
// counts in shared memory, and expands its items: every thread takes 4
// consecutive items, finds the row owning the first by a binary search over
// the rows' item offsets, walks through the owner's super-tile span (and on
// to the next rows) and stores the 4 (super-tile, row) items with one
// 16-byte store per array where aligned.  Items keep the rows' depth order.
// floor(a / d) for a < 2^32 from m = floor(2^32 / d) (d >= 2) or m = 2^32 - 1
// (d = 1): the product's high word is the quotient or one less.
__device__ __forceinline__ unsigned div_magic(unsigned a, unsigned d, unsigned m) {
  unsigned q = __umulhi(a, m);
  if (a - q * d >= d) ++q;
  return q;
}
unsigned div_magic_host(unsigned d) {
  return d <= 1u ? 0xffffffffu : (unsigned)((1ull << 32) / d);
}

// floor(a / d) for 0 <= a < 2^27, d >= 1 from a float reciprocal, corrected
// to the exact quotient.
__device__ __forceinline__ int div_small(int a, int d) {
  int q = __float2int_rz(__int2float_rn(a) * __frcp_rn(__int2float_rn(d)));
  while (q * d > a) --q;
  while ((q + 1) * d <= a) ++q;
  return q;
}

template <int ITEMS>
__global__ void __launch_bounds__(kScanThreads) rows_expand_kernel(
    const SortedRows sorted, const uint2* rect_sorted,
    const long long* n_dev, const unsigned long long* block_items,
    const long long* q_eff, int N, unsigned n_magic, const CamTable ct,
    unsigned* skeys, unsigned* svals, int vec16, int packed,
    unsigned* hist, int hgrid, unsigned hmask) {
  behind_previous();
  constexpr int RB = kScanThreads * ITEMS;
  __shared__ unsigned s_off[RB + 1];  // item offset of each row in the block (+ the total)
  // the super-tile sort's first-pass histogram (hist: [256][hgrid], zeroed):
  // the block's items are one contiguous range of positions, which meets
  // one or two of the sort's chunks; their digit counts are summed here
  __shared__ unsigned s_h[2][kRadixBins];
  const long long n = *n_dev, Q = *q_eff;
  const long long base = (long long)blockIdx.x * RB;
  if (base >= n || Q == 0) return;  // (the whole CTA)
  if (hist)
    for (int i = threadIdx.x; i < 2 * kRadixBins; i += kScanThreads) (&s_h[0][0])[i] = 0u;
  const int nr = (int)min((long long)RB, n - base);
  const int first = threadIdx.x * ITEMS;
  unsigned loc[ITEMS];
  unsigned long long sum = 0;
#pragma unroll
  for (int k = 0; k < ITEMS; ++k) {
    const int i = first + k;
    loc[k] = i < nr ? st_count(unpack_rect(rect_sorted[base + i])) : 0u;
    sum += loc[k];
  }
  unsigned long long tot;
  unsigned off = (unsigned)block_excl_scan(sum, &tot);
#pragma unroll
  for (int k = 0; k < ITEMS; ++k) {
    s_off[first + k] = off;
    off += loc[k];
  }
  if (threadIdx.x == 0) s_off[RB] = (unsigned)tot;
  __syncthreads();
  const unsigned total = (unsigned)tot;
  const long long gbase = (long long)block_items[blockIdx.x];
  const unsigned* rows = sorted.get();
  // the sort's chunk of a position: div_magic by the chunk (Q < 2^32)
  const unsigned hchunk = hist ? (unsigned)radix_chunk(Q, hgrid) : 1u;
  const unsigned hmagic = hist ? (unsigned)(0x100000000ull / hchunk) : 0u;
  const unsigned hc0 = hist ? div_magic((unsigned)gbase, hchunk, hmagic) : 0u;
  for (unsigned c0 = 0; c0 < total; c0 += 4 * kScanThreads) {
    const unsigned e0 = c0 + 4u * threadIdx.x;
    if (e0 >= total) continue;
    // the owner of e0: the last row whose items start at or before it (rows
    // without items share their start with the next row)
    int lo = 0, hi = nr - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (s_off[mid] <= e0) lo = mid;
      else hi = mid - 1;
    }
    int j = lo;
    unsigned kk[4], vv[4];
    unsigned row = 0u;
    int4 r = make_int4(0, 0, 0, 0), q = r;
    int id0 = 0, wdt = 1, stx = 1, x = 0, y = 0;
    int cur = -1;
    int cnt = 0;
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const unsigned e = e0 + (unsigned)t;
      if (e >= total) break;
      while (s_off[j + 1] <= e) ++j;  // (s_off[nr .. RB] = total > e)
      if (j != cur) {
        row = rows[base + j];
        if (!GS_IN_BOUNDS(row, (long long)N * ct.V, 205)) row = 0u;
        r = unpack_rect(rect_sorted[base + j]);
        q = st_span(r);
        const CamInfo& c = ct.c[div_magic(row, (unsigned)N, n_magic)];
        id0 = c.st_off + q.y * c.STX + q.x;
        wdt = max(q.z - q.x, 1);
        stx = c.STX;
        const int k = (int)(e - s_off[j]);
        y = div_small(k, wdt);
        x = k - y * wdt;
        cur = j;
      } else if (++x == wdt) {  // next span row
        x = 0;
        ++y;
      }
      unsigned key = (unsigned)(id0 + y * stx + x);
      if (packed) {
        // the rows and columns of this super-tile that the rect covers
        const int ox = 8 * (q.x + x), oy = 8 * (q.y + y);
        key |= rect_masks(r.x - ox, r.z - ox, r.y - oy, r.w - oy) << 16;
      }
      kk[t] = key;
      vv[t] = row;
      cnt = t + 1;
    }
    const long long g0 = gbase + e0;
    if (hist) {
      // the 4 positions cross at most one chunk boundary (chunks hold whole
      // 2048-item tiles)
      const unsigned c = div_magic((unsigned)g0, hchunk, hmagic);
      const unsigned long long next = (unsigned long long)(c + 1u) * hchunk;
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        if (t < cnt && g0 + t < Q) {
          const unsigned ct_ = (unsigned long long)(g0 + t) >= next ? c + 1u : c;
          const unsigned d = kk[t] & hmask;
          if (ct_ - hc0 < 2u) atomicAdd(&s_h[ct_ - hc0][d], 1u);
          else atomicAdd(hist + (long long)d * hgrid + ct_, 1u);
        }
      }
    }
    if (vec16 && cnt == 4 && (g0 & 3) == 0 && g0 + 3 < Q) {  // skeys, svals 16-byte aligned
      reinterpret_cast<uint4*>(skeys + g0)[0] = make_uint4(kk[0], kk[1], kk[2], kk[3]);
      reinterpret_cast<uint4*>(svals + g0)[0] = make_uint4(vv[0], vv[1], vv[2], vv[3]);
    } else {
#pragma unroll
      for (int t = 0; t < 4; ++t)
        if (t < cnt && g0 + t < Q) {
          skeys[g0 + t] = kk[t];
          svals[g0 + t] = vv[t];
        }
    }
  }
  if (hist) {
    __syncthreads();
    for (int i = threadIdx.x; i < 2 * kRadixBins; i += kScanThreads) {
      const unsigned v = (&s_h[0][0])[i];
      if (v) atomicAdd(hist + (long long)(i % kRadixBins) * hgrid + hc0 + i / kRadixBins, v);
    }
  }
}

// Per-key [start, end) from sorted u32 keys: each thread reads 4
// consecutive keys with one 16-byte load (the array is 256-byte aligned) plus
// its neighbours, and marks where the key changes.
__global__ void __launch_bounds__(256) ranges_kernel(const unsigned* tkeys,
                                                     const long long* p_eff,
                                                     unsigned kmask,
                                                     unsigned* ranges) {
  behind_previous();
  const long long P = *p_eff;
  const long long groups = (P + 3) / 4;
  for (long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x; g < groups;
       g += (long long)gridDim.x * blockDim.x) {
    const long long i0 = 4 * g;
    unsigned k[6];
    if (i0 + 3 < P) {
      const uint4 v = reinterpret_cast<const uint4*>(tkeys)[g];
      k[1] = v.x & kmask; k[2] = v.y & kmask; k[3] = v.z & kmask; k[4] = v.w & kmask;
    } else {
      for (int q = 0; q < 4; ++q) k[1 + q] = i0 + q < P ? tkeys[i0 + q] & kmask : 0u;
    }
    k[0] = i0 > 0 ? tkeys[i0 - 1] & kmask : 0xffffffffu;
    k[5] = i0 + 4 < P ? tkeys[i0 + 4] & kmask : 0xffffffffu;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const long long i = i0 + q;
      if (i >= P) break;
      const unsigned t = k[1 + q];
      if (i == 0 || k[q] != t) ranges[2ll * t] = (unsigned)i;
      const unsigned nxt = (i == P - 1) ? 0xffffffffu : (q < 3 ? k[2 + q] : k[5]);
      if (i == P - 1 || nxt != t) ranges[2ll * t + 1] = (unsigned)(i + 1);
    }
  }
}

// ----------------------------------------------------------------------------
// Expansion of the super-tile-sorted rows into per-tile lists.  A super-tile's
// rows (depth order) are cut into segments of kSeg; per segment and per tile
// of the super-tile (64), the count of rows covering the tile; per tile, the
// exclusive scan of those counts over the super-tile's segments; per tile,
// the list start (scan over all tiles); then every segment writes each of
// its rows into the lists of the tiles it covers, in the rows' order, so
// each list keeps their depth order.
// ----------------------------------------------------------------------------
constexpr int kSeg = 1024;
static_assert(kSeg % 256 == 0, "a segment is loaded in groups of 256");

__device__ __forceinline__ int view_of_st(const CamTable& ct, int s) {
  int v = 0;
  while (v + 1 < ct.V && ct.c[v + 1].st_off <= s) ++v;
  return v;
}

// A segment as st_segments_kernel lists it: its items [b, e), the global id of
// its super-tile's first tile, and (packed) the view's tiles per row and the
// tile columns and rows of the super-tile that lie in the view.
struct __align__(16) Segment {
  unsigned b, e;
  int tile;
  unsigned shape;  // TX | columns << 16 | rows << 20
  __device__ __forceinline__ int tx() const { return (int)(shape & 0xffffu); }
  __device__ __forceinline__ int cols() const { return (int)((shape >> 16) & 15u); }
  __device__ __forceinline__ int rows() const { return (int)(shape >> 20); }
};

__device__ __forceinline__ Segment load_segment(const Segment* segs, long long g) {
  const uint4 v = *reinterpret_cast<const uint4*>(segs + g);
  return Segment{v.x, v.y, (int)v.z, v.w};
}

// Segments of every super-tile: seg_first[s] (exclusive scan of
// ceil(len_s / kSeg)), seg_first[S] = total, segs[g] and (when not NULL)
// seg_st[g] = super-tile of g.
// One CTA of 1024 threads; for more than 256 super-tiles (up to that many
// st_count_kernel forms the segments itself).
__global__ void __launch_bounds__(1024) st_segments_kernel(
    const uint2* st_ranges, int S, unsigned* seg_first,
    Segment* segs, unsigned* seg_st, const CamTable ct,
    long long* n_seg) {
  behind_previous();
  __shared__ unsigned s_w[32];
  __shared__ unsigned s_carry;
  __shared__ Segment s_seg[1024];    // the super-tile's whole range, tile and shape
  __shared__ unsigned s_first[1024];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  if (tid == 0) s_carry = 0u;
  __syncthreads();
  for (int base = 0; base < S; base += 1024) {
    const int s = base + tid;
    uint2 r = make_uint2(0u, 0u);
    if (s < S) r = st_ranges[s];
    const unsigned cnt = (r.y - r.x + kSeg - 1) / kSeg;
    unsigned incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31) s_w[w] = incl;
    __syncthreads();
    if (w == 0) {
      const unsigned t = s_w[lane];
      unsigned ti = t;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, ti, o);
        if (lane >= o) ti += y;
      }
      s_w[lane] = ti - t;
    }
    __syncthreads();
    const unsigned first = s_carry + s_w[w] + incl - cnt;
    if (s < S) {
      seg_first[s] = first;
      const CamInfo& c = ct.c[view_of_st(ct, s)];
      const int sl = s - c.st_off;
      const int ox = (sl % c.STX) * kSuperTile, oy = (sl / c.STX) * kSuperTile;
      s_seg[tid] = Segment{r.x, r.y, c.tile_off + oy * c.TX + ox,
                           (unsigned)c.TX | (unsigned)min(kSuperTile, c.TX - ox) << 16 |
                               (unsigned)min(kSuperTile, c.TY - oy) << 20};
    }
    s_first[tid] = first;
    __syncthreads();
    if (tid == 1023) s_carry = first + cnt;
    // the segments of these super-tiles: a warp per super-tile
    for (int k = w; k < 1024 && base + k < S; k += 32) {
      const Segment sg = s_seg[k];
      const unsigned n = (sg.e - sg.b + kSeg - 1) / kSeg, g0 = s_first[k];
      for (unsigned j = lane; j < n; j += 32) {
        const unsigned b = sg.b + j * (unsigned)kSeg;
        segs[g0 + j] = Segment{b, min(sg.e, b + (unsigned)kSeg), sg.tile, sg.shape};
        if (seg_st) seg_st[g0 + j] = (unsigned)(base + k);
      }
    }
    __syncthreads();
  }
  if (tid == 0) {
    seg_first[S] = s_carry;
    *n_seg = (long long)s_carry;
  }
}

// Rect of row `row` inside the super-tile with tile origin (ox, oy), as a
// descriptor (0 when it covers no tile of it).
__device__ __forceinline__ unsigned st_desc(const int* rect, unsigned row, int N,
                                            const CamTable& ct, int ox, int oy) {
  const int4 r = view_rect(rect, row, N, ct);
  const int x0 = r.x - ox, x1 = r.z - ox, y0 = r.y - oy, y1 = r.w - oy;
  if (x0 >= kSuperTile || y0 >= kSuperTile || x1 <= 0 || y1 <= 0 || x1 <= x0 || y1 <= y0)
    return 0u;  // (not produced by consistent inputs)
  return rect_masks(x0, x1, y0, y1);
}

// Per segment: the count of rows covering each of the 64 tiles.  The count of
// tile (r, c) is the sum over the rows of [covers tile row r] [covers tile
// column c]: an 8 x 8 product of two 0/1 matrices over up to 1024 rows, which
// the tensor cores take 16 rows at a time (mma.sync m16n8k16 on bf16 with
// FP32 sums: whole numbers of at most 4 * 1024, exact).  A lane needs, of four
// items, the bits of one tile row and one tile column; a set bit moved to bit
// 14 of its 16-bit half is bf16 2.0, so every covering row adds 4.  The 8
// unused rows of A are zero.  About 11 instructions per 16 items; counting by
// row and column ballots took about 60 and was bound by issue (45 M items:
// 258 -> 97 us; what is left is the latency of the key loads).
// The descriptors travel in the items' keys (bits 16-31) when `packed`;
// otherwise they are formed here from the rects and stored in desc for the
// expansion.
__device__ __forceinline__ void mma_count(float d[4], unsigned a0, unsigned a2, unsigned b0,
                                          unsigned b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %5}, "
      "{%7, %8}, {%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(0u), "r"(a2), "r"(b0), "r"(b1));
}

// With `totals` (the items were sorted by super-tile in at most one pass: S <=
// 256) every CTA forms the segments itself from the super-tiles' item counts,
// two scans of 256 values, and writes the table entries of the segments it
// takes, instead of a launch of st_segments_kernel before.
__device__ __forceinline__ unsigned block_scan256(unsigned x, unsigned* s_w) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  unsigned inc = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) s_w[w] = inc;
  __syncthreads();
  unsigned wo = 0u;
#pragma unroll
  for (int i = 0; i < 8; ++i) wo += i < w ? s_w[i] : 0u;
  __syncthreads();
  return wo + inc - x;
}

__global__ void __launch_bounds__(256) st_count_kernel(
    const unsigned* sp_keys, const unsigned* sp_rows,
    Segment* segs, const unsigned* seg_st,
    long long* n_seg, int packed, const int* rect, int N,
    const CamTable ct, unsigned* desc, unsigned* hist,
    const unsigned* totals, const long long* q_eff, int S,
    unsigned* seg_first) {
  behind_previous();
  __shared__ unsigned s_cnt[8][64];
  constexpr int kPer = kSeg / 8;  // items of a warp
  __shared__ __align__(16) unsigned short s_desc[8][kPer];
  __shared__ unsigned s_start[256], s_first[257];  // (totals) items, segments before a super-tile
  __shared__ unsigned s_w[8];
  __shared__ __align__(16) Segment s_seg[256];  // (totals) the CTA's segments
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int t = lane & 3, q = lane >> 2;  // the lane's four items of 16; its tile row and column
  const int sr = 14 - q, sc = 6 - q;      // moves its bits to bit 14 (a rotation by -1 for column 7)
  long long G;
  static_assert(kRadixBins == 256, "one digit per thread: S <= 256 where the segments are formed here");
  const bool own = totals || S == 1;  // the segments are formed here
  if (own) {
    const unsigned items = tid < S ? (S == 1 ? (unsigned)*q_eff : totals[tid]) : 0u;
    const unsigned start = block_scan256(items, s_w);
    const unsigned first = block_scan256((items + kSeg - 1) / kSeg, s_w);
    s_start[tid] = start;
    s_first[tid] = first;
    if (tid == 255) s_first[256] = first + (items + kSeg - 1) / kSeg;
    __syncthreads();
    G = s_first[256];
    if (blockIdx.x == 0) {
      if (tid < S) seg_first[tid] = first;
      if (tid == 0) {
        seg_first[S] = (unsigned)G;
        *n_seg = G;
      }
    }
  } else {
    G = *n_seg;
  }
  for (long long g = blockIdx.x, it = 0; g < G; g += gridDim.x, ++it) {
    if (own && (it & 255) == 0) {
      // the CTA's next 256 segments, one per thread
      const long long gt = g + (long long)tid * gridDim.x;
      __syncthreads();
      if (gt < G) {
        // the last super-tile whose segments start at or before gt (those
        // without segments share their start with the next)
        int s = 0;
        for (int hi = S - 1; s < hi;) {
          const int mid = (s + hi + 1) >> 1;
          if (s_first[mid] <= (unsigned)gt) s = mid;
          else hi = mid - 1;
        }
        Segment si;
        si.b = s_start[s] + ((unsigned)gt - s_first[s]) * (unsigned)kSeg;
        si.e = min(s + 1 < S ? s_start[s + 1] : (unsigned)*q_eff, si.b + (unsigned)kSeg);
        const CamInfo& c = ct.c[view_of_st(ct, s)];
        const int sl = s - c.st_off;
        const int ox = (sl % c.STX) * kSuperTile, oy = (sl / c.STX) * kSuperTile;
        si.tile = c.tile_off + oy * c.TX + ox;
        si.shape = (unsigned)c.TX | (unsigned)min(kSuperTile, c.TX - ox) << 16 |
                   (unsigned)min(kSuperTile, c.TY - oy) << 20;
        s_seg[tid] = si;
        segs[gt] = si;
      }
      __syncthreads();
    }
    const Segment si = own ? s_seg[it & 255] : load_segment(segs, g);
    int ox = 0, oy = 0;
    if (!packed) {  // (over 65,536 super-tiles or 8,000 tiles a side: not own)
      const int s = (int)seg_st[g];
      const CamInfo& c = ct.c[view_of_st(ct, s)];
      ox = ((s - c.st_off) % c.STX) * kSuperTile;
      oy = ((s - c.st_off) / c.STX) * kSuperTile;
    }
    unsigned dd[kPer / 32];
#pragma unroll
    for (int k = 0; k < kPer / 32; ++k) {
      const unsigned i = si.b + kPer * w + 32u * k + lane;
      dd[k] = 0u;
      if (i < si.e) {
        if (packed) {
          dd[k] = sp_keys[i] >> 16;
        } else {
          dd[k] = st_desc(rect, sp_rows[i], N, ct, ox, oy);
          desc[i] = dd[k] << 16;
        }
      }
    }
#pragma unroll
    for (int k = 0; k < kPer / 32; ++k) s_desc[w][32 * k + lane] = (unsigned short)dd[k];
    __syncwarp();
    float d[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int j = 0; j < kPer / 16; ++j) {
      const uint2 v = *reinterpret_cast<const uint2*>(&s_desc[w][16 * j + 4 * t]);
      mma_count(d, (v.x << sr) & 0x40004000u, (v.y << sr) & 0x40004000u,
                __funnelshift_l(v.x, v.x, sc) & 0x40004000u,
                __funnelshift_l(v.y, v.y, sc) & 0x40004000u);
    }
    // d[0], d[1]: tile row q, columns 2t and 2t + 1
    *reinterpret_cast<uint2*>(&s_cnt[w][8 * q + 2 * t]) =
        make_uint2((unsigned)(0.25f * d[0]), (unsigned)(0.25f * d[1]));
    __syncthreads();
    if (tid < 64) {
      unsigned sum = 0u;
#pragma unroll
      for (int ww = 0; ww < 8; ++ww) sum += s_cnt[ww][tid];
      hist[g * 64 + tid] = sum;
    }
    __syncthreads();
  }
}

// One CTA per super-tile, 64 groups of segments x 16 quads of tiles: exclusive
// scan of every tile's counts over the super-tile's segments (in place), and
// the tile's total list length.
__device__ __forceinline__ void tile_scan_dev(const unsigned* tile_cnt, int T,
                                              unsigned* tile_start,
                                              unsigned* ranges);

__device__ __forceinline__ uint4 add4(uint4 a, uint4 b) {
  return make_uint4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
}

__global__ void __launch_bounds__(1024) st_scan_kernel(const unsigned* seg_first,
                                                       const CamTable ct,
                                                       uint4* hist,
                                                       unsigned* tile_cnt,
                                                       unsigned long long* arrive,
                                                       unsigned* tile_start,
                                                       unsigned* ranges) {
  behind_previous();
  __shared__ uint4 s_part[64][16];
  const int s = blockIdx.x;
  const int k = threadIdx.x >> 4, q = threadIdx.x & 15;
  const unsigned g0 = seg_first[s], L = seg_first[s + 1] - g0;
  const unsigned per = (L + 63u) / 64u;
  const unsigned a = min(L, (unsigned)k * per), e = min(L, a + per);
  constexpr unsigned kBatch = 4;  // counts loaded together
  const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
  uint4 sum = zero;
  for (unsigned g = a; g < e; g += kBatch) {
    const uint4* h = hist + (long long)(g0 + g) * 16 + q;
    uint4 x[kBatch];
#pragma unroll
    for (unsigned j = 0; j < kBatch; ++j) x[j] = g + j < e ? h[16 * j] : zero;
#pragma unroll
    for (unsigned j = 0; j < kBatch; ++j) sum = add4(sum, x[j]);
  }
  s_part[k][q] = sum;
  __syncthreads();
  if (threadIdx.x < 64) {
    // tile bt: exclusive scan over the 64 groups
    const int bt = threadIdx.x;
    unsigned* p = &s_part[0][0].x + bt;
    unsigned run = 0u;
#pragma unroll 16
    for (int kk = 0; kk < 64; ++kk) {
      const unsigned x = p[64 * kk];
      p[64 * kk] = run;
      run += x;
    }
    const CamInfo& c = ct.c[view_of_st(ct, s)];
    const int sl = s - c.st_off;
    const int tx = (sl % c.STX) * kSuperTile + (bt & 7);
    const int ty = (sl / c.STX) * kSuperTile + (bt >> 3);
    if (tx < c.TX && ty < c.TY) tile_cnt[c.tile_off + ty * c.TX + tx] = run;
  }
  __syncthreads();
  uint4 run = s_part[k][q];
  for (unsigned g = a; g < e; g += kBatch) {
    uint4* h = hist + (long long)(g0 + g) * 16 + q;
    uint4 x[kBatch];
#pragma unroll
    for (unsigned j = 0; j < kBatch; ++j) x[j] = g + j < e ? h[16 * j] : zero;
#pragma unroll
    for (unsigned j = 0; j < kBatch; ++j) {
      if (g + j < e) h[16 * j] = run;
      run = add4(run, x[j]);
    }
  }
  if (last_block_arrives(arrive, gridDim.x)) tile_scan_dev(tile_cnt, ct.total_tiles, tile_start, ranges);
}

// Exclusive scan of the list lengths over all T tiles (one CTA of 1024
// threads, 4 consecutive tiles per thread and round): list starts, and ranges
// [start, end) ((0, 0) for an empty list).  Run by the last CTA of
// st_scan_kernel (tile_cnt read through L2; it is padded to whole 16 bytes).
__device__ __forceinline__ void tile_scan_dev(const unsigned* tile_cnt, int T,
                                              unsigned* tile_start,
                                              unsigned* ranges) {
  __shared__ unsigned s_w[2][32];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  unsigned carry = 0u;
  int buf = 0;
  for (int base = 0; base < T; base += 4096, buf ^= 1) {
    const int t = base + 4 * tid;
    unsigned c[4] = {0u, 0u, 0u, 0u};
    if (t < T) {
      const uint4 v = __ldcg(reinterpret_cast<const uint4*>(tile_cnt + t));
      c[0] = v.x;
      c[1] = t + 1 < T ? v.y : 0u;
      c[2] = t + 2 < T ? v.z : 0u;
      c[3] = t + 3 < T ? v.w : 0u;
    }
    const unsigned sum = c[0] + c[1] + c[2] + c[3];
    unsigned incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31) s_w[buf][w] = incl;
    __syncthreads();  // (two buffers: one barrier per round)
    unsigned wt = s_w[buf][lane];
    const unsigned own = wt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned y = __shfl_up_sync(0xffffffffu, wt, o);
      if (lane >= o) wt += y;
    }
    unsigned start = carry + __shfl_sync(0xffffffffu, wt - own, w) + incl - sum;
    carry += __shfl_sync(0xffffffffu, wt, 31);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (t + j < T) {
        tile_start[t + j] = start;
        ranges[2ll * (t + j)] = c[j] ? start : 0u;
        ranges[2ll * (t + j) + 1] = c[j] ? start + c[j] : 0u;
        start += c[j];
      }
    }
  }
}

// Inclusive warp scan of four byte fields each (sums stay below 256).
__device__ __forceinline__ unsigned warp_scan_bytes(unsigned x) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1)
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b32 t;\n\t"
        "shfl.sync.up.b32 t|p, %0, %1, 0x0, 0xffffffff;\n\t"
        "@p add.u32 %0, %0, t;\n\t}"
        : "+r"(x)
        : "r"(o));
  return x;
}

// Bits 0..3 of x as the low bits of four bytes.
__device__ __forceinline__ unsigned spread4(unsigned x) {
  return ((x & 15u) * 0x00204081u) & 0x01010101u;
}

// Address of the list slot n after the one at address a (one instruction).
__device__ __forceinline__ unsigned long long slot_after(unsigned long long a, unsigned n) {
  unsigned long long r;
  asm("mad.wide.u32 %0, %1, 4, %2;" : "=l"(r) : "r"(n), "l"(a));
  return r;
}

// Expansion.  Per segment, the items (row, descriptor) are staged in shared
// memory and warp r takes tile row r of the super-tile: it walks the items in
// (depth) order, keeps those that cover its tile row in a ring of its own,
// and whenever 64 of them are there writes them out to the row's 8 lists, two
// consecutive items per lane: the ranks of all 8 columns come from one warp
// scan of byte counters.  (Ranks from ballots take a population count per
// column and 32 rows, which runs at an eighth of the issue rate and bound this
// kernel.)  The next slots of the 8 lists stay in registers, so no barrier and
// no prefix over the warps is needed between the segment's staging and its
// end, and only the rows that cover the tile row reach the 8 column steps.
//
// What bounds it: instruction issue while the lists fit in L2 (21 M pairs: 58
// -> 43 us against the ballot form), the stores' way to DRAM beyond (351 M
// pairs: 590 -> 420 us, 3.4 TB/s).  CTAs per SM the register budget targets: 4;
// left to itself the compiler takes 32 registers, which recomputes addresses
// (351 M pairs: 567 us).  Grid: up to 64 CTAs per SM, so that most CTAs write
// one segment and they run in list order (500 us with 8 per SM, whose rounds
// drift apart and leave a partly empty last one).
constexpr int kEmitCtas = 4;
constexpr long long kEmitGrid = 152ll * 64;
template <bool KEYS>
__global__ void __launch_bounds__(256, kEmitCtas) st_emit_kernel(
    const unsigned* sp_keys, const unsigned* sp_rows,
    const unsigned* desc, int packed, const Segment* segs,
    const long long* n_seg, const unsigned* hist,
    const unsigned* tile_start, const float* depth,
    unsigned* out_vals, unsigned long long* out_keys, long long cap) {
  behind_previous();
  constexpr unsigned kRing = 128;  // at most 63 waiting + 32 new items
  __shared__ uint2 s_item[kSeg];                     // row, descriptor
  __shared__ __align__(16) uint2 s_ring[8][kRing];   // row, columns covered
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const unsigned lt = (1u << lane) - 1u;
  const long long G = *n_seg;
  const unsigned* keys = packed ? sp_keys : desc;
  for (long long g = blockIdx.x; g < G; g += gridDim.x) {
    const Segment si = load_segment(segs, g);
    const int n = (int)(si.e - si.b);
    constexpr int kPer = kSeg / 256;
    uint2 it[kPer];
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const int i = tid + 256 * k;
      it[k] = make_uint2(0u, 0u);
      if (i < n) it[k] = make_uint2(sp_rows[si.b + i], keys[si.b + i] >> 16);
    }
    // the first slots of this warp's tiles (lane c: column c)
    int tile = -1;
    unsigned first = 0u;
    if (lane < si.cols() && w < si.rows()) {
      tile = si.tile + w * si.tx() + lane;
      first = tile_start[tile] + hist[g * 64 + 8 * w + lane];
    }
    __syncthreads();  // the previous segment's items have been read
#pragma unroll
    for (int k = 0; k < kPer; ++k) s_item[tid + 256 * k] = it[k];
    __syncthreads();
    unsigned long long run[8];  // address of the next slot of each list
#pragma unroll
    for (int k = 0; k < 8; ++k)
      run[k] = slot_after(reinterpret_cast<unsigned long long>(out_vals),
                          __shfl_sync(0xffffffffu, first, k));
    auto store = [&](unsigned long long at, unsigned row, int tk) {
      unsigned* p = reinterpret_cast<unsigned*>(at);
      if (!GS_IN_BOUNDS(p - out_vals, cap, 201)) return;
      *p = row;
      if (KEYS)
        out_keys[p - out_vals] =
            ((unsigned long long)(unsigned)tk << 32) | __float_as_uint(depth[row]);
    };
    // writes out the first `m` (at most 64) of the 64 items from ring position `at`
    auto flush = [&](unsigned at, unsigned m) {
      uint4 e = *reinterpret_cast<const uint4*>(&s_ring[w][(at + 2 * lane) & (kRing - 1)]);
      if (2u * lane >= m) e.y = 0u;
      if (2u * lane + 1u >= m) e.w = 0u;
      const unsigned a0 = spread4(e.y), a1 = spread4(e.y >> 4);
      const unsigned t0 = a0 + spread4(e.w), t1 = a1 + spread4(e.w >> 4);
      const unsigned i0 = warp_scan_bytes(t0), i1 = warp_scan_bytes(t1);
      const unsigned x0 = i0 - t0, x1 = i1 - t1;    // ranks of the lane's first item
      const unsigned y0 = x0 + a0, y1 = x1 + a1;    // and of its second
      const unsigned n0 = __shfl_sync(0xffffffffu, i0, 31), n1 = __shfl_sync(0xffffffffu, i1, 31);
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const unsigned sel = 0x4440u | (k & 3);
        int tk = 0;
        if (KEYS) tk = __shfl_sync(0xffffffffu, tile, k);
        if (e.y & (1u << k))
          store(slot_after(run[k], __byte_perm(k < 4 ? x0 : x1, 0u, sel)), e.x, tk);
        if (e.w & (1u << k))
          store(slot_after(run[k], __byte_perm(k < 4 ? y0 : y1, 0u, sel)), e.z, tk);
        run[k] = slot_after(run[k], __byte_perm(k < 4 ? n0 : n1, 0u, sel));
      }
    };
    unsigned head = 0u, cnt = 0u;  // ring: `cnt` items from position `head`
    for (int b = 0; b < n; b += 32) {
      const uint2 e = s_item[b + lane];  // (items past n: descriptor 0)
      const bool in = (e.y >> w) & 1u;
      const unsigned m = __ballot_sync(0xffffffffu, in);
      if (in) s_ring[w][(head + cnt + __popc(m & lt)) & (kRing - 1)] = make_uint2(e.x, e.y >> 8);
      cnt += __popc(m);
      if (cnt >= 64u) {
        __syncwarp();
        flush(head, 64u);
        head += 64u;
        cnt -= 64u;
        __syncwarp();
      }
    }
    __syncwarp();
    if (cnt) flush(head, cnt);
    __syncwarp();
  }
}


__global__ void set_value_kernel(long long* dst, long long v) {
  behind_previous();
  if (threadIdx.x == 0 && blockIdx.x == 0) *dst = v;
}

// ----------------------------------------------------------------------------
// Workspace layout.
// ----------------------------------------------------------------------------
inline size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

struct Workspace {
  unsigned long long* block_sums;  // scan block sums
  unsigned long long* block_sums2; // second scan's block sums
  long long* counters;             // [0] n_vis, [1] P, [2] P eff., [3] Q, [4] Q eff., [5] segments
  unsigned* rk[2];                 // row keys (depth bits), double buffer
  unsigned* rv[2];                 // row values, double buffer
  uint2* rect_sorted;              // clamped rect per visible row, depth order (16-bit packed)
  unsigned* pk[2];                 // super-pair keys (super-tile), double buffer; later descriptors
  unsigned* pv;                    // super-pair values (rows)
  unsigned* hist;                  // radix histograms
  unsigned* st_ranges;             // [2 * super-tiles] rows of each super-tile
  unsigned* seg_first;             // [super-tiles + 1] first segment of each super-tile
  Segment* segs;                   // the segments
  unsigned* seg_st;                // super-tile of every segment
  unsigned* seg_hist;              // [segments][64] per-tile counts, then bases
  unsigned* tile_cnt;              // [tiles] list lengths
  unsigned* tile_start;            // [tiles] list starts
  size_t bytes;
};

constexpr int kRadixGrid = 4 * 152;  // largest radix grid (4 CTAs per SM of a GB300)

// Radix histograms: [256][grid] per-CTA digit counts and their scan, then the
// 256 digit totals.
constexpr size_t radix_hist_bytes() { return 4ull * kRadixBins * (kRadixGrid + 1); }
// (depth_sort_kernel: a table of [kCoopGrid][256] per pass, then a count per CTA)
static_assert((size_t)kRadixMaxPasses * kCoopGrid * kRadixBins + kCoopGrid <= radix_hist_bytes() / 4,
              "the sort's counts fit the histogram buffer");

// CTAs of radix_downsweep_kernel resident on the current device at once
// (cached per device).
int radix_resident_ctas() {
  static std::atomic<int> cache[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return kRadixGrid;
  int v = cache[dev].load(std::memory_order_relaxed);
  if (v > 0) return v;
  int per_sm = 0, sms = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, radix_downsweep_kernel,
                                                    kRadixThreads, 0) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      per_sm < 1 || sms < 1) {
    cudaGetLastError();
    return kRadixGrid;
  }
  v = per_sm * sms;
  cache[dev].store(v, std::memory_order_relaxed);
  return v;
}

inline long long scan_blocks(long long n) { return (n + kScanTile - 1) / kScanTile; }

// Upper bound of the expansion segments: sum over super-tiles of
// ceil(len / kSeg) <= Q / kSeg + super-tiles, and Q <= P <= cap.
inline long long max_segments(long long cap, long long tiles) { return cap / kSeg + tiles + 2; }

constexpr int kCounters = 14;  // 8 counts, 3 arrival counters, the grid barrier, the depth-key range

Workspace carve(void* base, long long n_rows, long long cap, long long tiles) {
  Workspace w;
  char* p = reinterpret_cast<char*>(base);
  size_t off = 0;
  auto take = [&](size_t bytes) {
    char* r = p ? p + off : nullptr;
    off += align256(bytes);
    return r;
  };
  // (blocks of 256 rows up to kCoopRows, of 1,024 or 4,096 above)
  const long long nb = std::max(scan_blocks(n_rows > cap ? n_rows : cap),
                                (std::min(n_rows, kCoopRows) + kCoopBlock - 1) / kCoopBlock) + 1;
  const long long ms = max_segments(cap, tiles);
  w.block_sums = reinterpret_cast<unsigned long long*>(take(sizeof(unsigned long long) * nb));
  w.block_sums2 = reinterpret_cast<unsigned long long*>(take(sizeof(unsigned long long) * nb));
  w.counters = reinterpret_cast<long long*>(take(sizeof(long long) * kCounters));
  for (int i = 0; i < 2; ++i) w.rk[i] = reinterpret_cast<unsigned*>(take(4 * (n_rows + 1)));
  for (int i = 0; i < 2; ++i) w.rv[i] = reinterpret_cast<unsigned*>(take(4 * (n_rows + 1)));
  w.rect_sorted = reinterpret_cast<uint2*>(take(8 * (n_rows + 1)));
  for (int i = 0; i < 2; ++i) w.pk[i] = reinterpret_cast<unsigned*>(take(4 * (cap + 1)));
  w.pv = reinterpret_cast<unsigned*>(take(4 * (cap + 1)));
  w.hist = reinterpret_cast<unsigned*>(take(radix_hist_bytes()));
  w.st_ranges = reinterpret_cast<unsigned*>(take(8ull * (tiles + 1)));
  w.seg_first = reinterpret_cast<unsigned*>(take(4ull * (tiles + 2)));
  w.segs = reinterpret_cast<Segment*>(take(sizeof(Segment) * ms));
  w.seg_st = reinterpret_cast<unsigned*>(take(4ull * ms));
  w.seg_hist = reinterpret_cast<unsigned*>(take(4ull * 64 * ms));
  w.tile_cnt = reinterpret_cast<unsigned*>(take(4ull * (tiles + 4)));
  w.tile_start = reinterpret_cast<unsigned*>(take(4ull * (tiles + 1)));
  w.bytes = off;
  return w;
}

// Radix sort of the pairs in (k[0], v[0]) (n_dev items, at most n_bound):
// with `range` on the significant bits of (key - smallest key), else on
// `bits` bits.  The result is in buffer (passes mod 2): radix_result on the
// device, or the host's plan when there is no range.  keys_last: the last
// pass writes the keys as well (only the values are needed otherwise).
// The radix grid for at most n_bound items.
int radix_grid(long long n_bound) {
  return (int)std::max<long long>(
      1, std::min<long long>(std::min(kRadixGrid, radix_resident_ctas()),
                             (n_bound + kRadixTile - 1) / kRadixTile));
}

void radix_sort(unsigned* k[2], unsigned* v[2], const long long* n_dev, long long n_bound,
                const unsigned* range, int bits, unsigned* hist, bool keys_last,
                cudaStream_t st, const RadixRows* rows = nullptr, bool hist0_ready = false) {
  if (n_bound == 0) return;
  const int passes = range ? kRadixMaxPasses : radix_plan_bits(0u, bits).passes;
  // one wave: at most the CTAs of the scatter kernel resident on the device
  const int grid = radix_grid(n_bound);
  RadixPass a;
  a.n_dev = n_dev;
  a.range = range;
  a.bits = bits;
  a.hist = hist;
  a.digit_tot = hist + kRadixBins * grid;
  a.keys_last = keys_last ? 1 : 0;
  a.rows = rows ? *rows : RadixRows{nullptr, nullptr, 0, nullptr};
  for (int p = 0; p < passes; ++p) {
    a.keys_in = k[p & 1];
    a.vals_in = v[p & 1];
    a.keys_out = k[(p + 1) & 1];
    a.vals_out = v[(p + 1) & 1];
    a.pass = p;
    // (hist0_ready: the first pass's per-CTA digit counts are already in
    // hist, summed by the kernel that wrote the items)
    if (p > 0 || !hist0_ready)
      launch_behind(radix_upsweep_kernel, dim3(grid), kRadixThreads, st, a);
    launch_behind(radix_scan_kernel, dim3(kRadixBins), kScanThreads, st, a, grid);
    launch_behind(radix_downsweep_kernel, dim3(grid), kRadixThreads, st, a);
    count_launches(p > 0 || !hist0_ready ? 3 : 2);
  }
}

// Steps 1 to 3 in one launch (depth_sort_kernel).  An error of the launch itself
// that says the grid cannot be resident at once (a part of the GPU, say) is
// reported as cudaErrorCooperativeLaunchTooLarge: the caller then takes the
// separate kernels.
cudaError_t launch_depth_sort(const CoopArgs& args_in, const CamTable& ct, cudaStream_t st) {
  CoopArgs a = args_in;
  CamTable cams = ct;
  void* args[] = {&a, &cams};
  // a CTA per 1,024 rows, at most one per SM: fewer CTAs meet at a barrier sooner
  int ctas = (int)std::min<long long>(kCoopGrid, (a.rows.n + 1023) / 1024);
  cudaError_t e;
  if (a.rows.n <= kClusterRows) {
    int c = 1;  // (cluster sizes are powers of two)
    while (c < kCoopCluster && c < ctas) c *= 2;
    if ((e = allow_coop_smem<true>()) != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(c);
    cfg.blockDim = dim3(kCoopThreads);
    cfg.dynamicSmemBytes = sizeof(CoopShared);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = c;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelExC(&cfg, reinterpret_cast<const void*>(depth_sort_kernel<true>), args);
  } else {
    if ((e = allow_coop_smem<false>()) != cudaSuccess) return e;
    e = cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(depth_sort_kernel<false>),
                                    dim3(ctas), dim3(kCoopThreads), args, sizeof(CoopShared), st);
  }
  if (e == cudaErrorLaunchOutOfResources) e = cudaErrorCooperativeLaunchTooLarge;
  return e;
}

int bits_for(long long count) {
  int b = 0;
  while (b < 32 && (1ll << b) < count) ++b;
  return b;
}

}  // namespace

GS_BOUNDS_READER(bounds_status_binning)

#ifdef GS_DEBUG_BOUNDS
extern "C" void gs_debug_sort_polls(int polls) {
  g_barrier_polls = polls >= 0 ? polls : kBarrierPolls;
}
#endif

size_t bin_sort_workspace_size(long long n_rows, long long cap, long long total_tiles) {
  return carve(nullptr, n_rows, cap, total_tiles).bytes;
}

int launch_bin_sort(const gs_proj* proj, int N, const CamTable& ct, void* workspace,
                    size_t ws_bytes, long long cap, unsigned* sorted_vals,
                    unsigned long long* sorted_keys, unsigned* ranges, long long* num_pairs_dev,
                    long long* num_pairs_host, int* status_dev, cudaStream_t st) {
  const long long n_rows = (long long)N * ct.V;
  const long long T = ct.total_tiles;
  const int S = ct.total_st;
  Workspace w = carve(workspace, n_rows, cap, T);
  if (ws_bytes < w.bytes) return GS_ERR_INVALID_ARG;
  long long* n_vis = w.counters;
  long long* P = w.counters + 1;
  long long* p_eff = w.counters + 2;
  long long* Q = w.counters + 3;
  long long* q_eff = w.counters + 4;
  long long* n_seg = w.counters + 5;
  // arrival counters of the kernels whose last CTA runs the following scan
  unsigned long long* arrive = reinterpret_cast<unsigned long long*>(w.counters + 8);
  GS_TRY_CUDA(cudaMemsetAsync(w.counters, 0, kCounters * sizeof(long long), st));
  const CountsOut co{w.block_sums, w.block_sums2, cap, Q, P, q_eff, p_eff, num_pairs_dev,
                     status_dev};
  // the visible rows' depth-bit range (complement of the smallest, largest)
  unsigned* range = reinterpret_cast<unsigned*>(w.counters + 12);
  // the projection's 8-bit packed rects (views of at most 255 tiles per side)
  const unsigned* rect8 = rect8_fits(ct) ? proj->rect8 : nullptr;
  bool coop = n_rows > 0 && n_rows <= kCoopRows && coop_available();
  if (coop) {
    CoopArgs a;
    a.rows = RadixRows{proj->depth, proj->tiles_touched, n_rows, n_vis};
    for (int i = 0; i < 2; ++i) {
      a.k[i] = w.rk[i];
      a.v[i] = w.rv[i];
    }
    a.hist = w.hist;
    a.cnt = w.hist + (size_t)kRadixMaxPasses * kCoopGrid * kRadixBins;
    a.range = range;
    a.bar = reinterpret_cast<unsigned*>(w.counters + 11);
    a.polls = barrier_polls();
    a.rect = proj->rect;
    a.rect8 = rect8;
    a.N = N;
    a.rect_sorted = w.rect_sorted;
    a.arrive = arrive + 1;
    a.co = co;
    const cudaError_t e = launch_depth_sort(a, ct, st);
    if (e == cudaErrorCooperativeLaunchTooLarge) {
      cudaGetLastError();
      coop = false;
    } else {
      GS_TRY_CUDA(e);
    }
  }
  const SortedRows rows_sorted{w.rv[0], w.rv[1], coop ? nullptr : range};
  // scan blocks: 256 rows (one per thread) behind the one-launch sort, whose warps
  // count them; in the separate kernels 1,024 rows (4 per thread), which keep many
  // CTAs in flight when few rows are visible, and above 4M rows 4,096 (16 per thread),
  // which are faster there
  const bool small = n_rows <= (4ll << 20);
  const int items = coop ? 1 : small ? 4 : 16;
  const long long nb = (n_rows + kScanThreads * items - 1) / (kScanThreads * items);
  if (n_rows > 0 && coop) {
    count_launches(1);  // 1-3. in one launch (above)
  } else if (n_rows > 0) {
    // 1-2. stable depth sort of the visible rows (ties keep row order = id
    //    order) on the significant bits of their depth range; the first pass
    //    reads the rows (depth bits, visible when tiles_touched > 0), drops
    //    the culled ones, folds the range in and counts the visible rows
    const RadixRows rr{proj->depth, proj->tiles_touched, n_rows, n_vis};
    radix_sort(w.rk, w.rv, n_vis, n_rows, range, 32, w.hist, false, st, &rr);
    // 3. per row in depth order: super-tile offsets, the super-pair count Q
    //    and the pair count P
    //    (its last CTA: the scans of Q and P over the blocks, the capacity
    //    check and the reported count)
    if (small)
      launch_behind(rows_gather_kernel<4>, dim3((unsigned)nb), kScanThreads, st, rows_sorted,
                    n_vis, proj->rect, rect8, N, ct, w.rect_sorted, arrive + 1, co);
    else
      launch_behind(rows_gather_kernel<16>, dim3((unsigned)nb), kScanThreads, st, rows_sorted,
                    n_vis, proj->rect, rect8, N, ct, w.rect_sorted, arrive + 1, co);
    count_launches(1);
  } else {
    launch_behind(scan_counts_check_kernel, dim3(1), kScanThreads, st, co, 0);
    count_launches(1);
  }
  GS_TRY_CUDA(cudaGetLastError());
  long long p_bound = cap;
  if (num_pairs_host) {
    long long p_host = 0;
    GS_TRY_CUDA(cudaMemcpyAsync(&p_host, P, sizeof(long long), cudaMemcpyDeviceToHost, st));
    GS_TRY_CUDA(cudaStreamSynchronize(st));
    if (p_host < 0) {
      *num_pairs_host = 0;
      GS_TRY_CUDA(cudaMemsetAsync(ranges, 0, 2 * sizeof(unsigned) * (size_t)T, st));
      return GS_ERR_TIMEOUT;
    }
    *num_pairs_host = p_host;
    if (p_host > cap) {
      GS_TRY_CUDA(cudaMemsetAsync(ranges, 0, 2 * sizeof(unsigned) * (size_t)T, st));
      return GS_ERR_CAPACITY;
    }
    p_bound = p_host;
  }
  if (n_rows == 0 || p_bound == 0 || S == 0) {
    GS_TRY_CUDA(cudaMemsetAsync(ranges, 0, 2 * sizeof(unsigned) * (size_t)T, st));
    return check_launch();
  }
  // 4. super-pairs (super-tile, row) in depth order of the rows, into the
  //    buffers that the super-tile sort leaves in (pk[res], pv)
  const int sbits = bits_for(S);
  const int spasses = radix_plan_bits(0u, sbits).passes;
  unsigned* sk[2] = {w.pk[0], w.pk[1]};
  unsigned* sv[2];
  if (spasses % 2 == 0) {
    sv[0] = w.pv;
    sv[1] = sorted_vals;
  } else {
    sv[0] = sorted_vals;
    sv[1] = w.pv;
  }
  const long long q_bound = p_bound;  // Q <= P
  // the rect descriptors ride in the keys' upper 16 bits when the super-tile
  // ids fit the lower 16 and every rect end fits the packed field
  int packed = S <= 65536 ? 1 : 0;
  for (int v = 0; v < ct.V; ++v)
    if (ct.c[v].TX > 8000 || ct.c[v].TY > 8000) packed = 0;
  // the expansion sums the super-tile sort's first-pass histogram as it
  // writes the items (positions below 2^31)
  const bool hist0 = q_bound < (1ll << 31);
  const int sgrid = radix_grid(q_bound);
  if (hist0)
    GS_TRY_CUDA(cudaMemsetAsync(w.hist, 0, sizeof(unsigned) * kRadixBins * (size_t)sgrid, st));
  {
    // (the scan blocks of rows_gather_kernel: their item bases are scanned)
    const int vec16 = (reinterpret_cast<uintptr_t>(sv[0]) % 16 == 0 &&
                       reinterpret_cast<uintptr_t>(sk[0]) % 16 == 0) ? 1 : 0;
    unsigned* h = hist0 ? w.hist : nullptr;
    const unsigned hmask = (1u << radix_plan_bits(0u, sbits).d0) - 1u;
    if (coop)
      launch_behind(rows_expand_kernel<1>, dim3((unsigned)nb), kScanThreads, st, rows_sorted,
                    w.rect_sorted, n_vis, w.block_sums, q_eff, N, div_magic_host((unsigned)N), ct,
                    sk[0], sv[0], vec16, packed, h, sgrid, hmask);
    else if (small)
      launch_behind(rows_expand_kernel<4>, dim3((unsigned)nb), kScanThreads, st, rows_sorted,
                    w.rect_sorted, n_vis, w.block_sums, q_eff, N, div_magic_host((unsigned)N), ct,
                    sk[0], sv[0], vec16, packed, h, sgrid, hmask);
    else
      launch_behind(rows_expand_kernel<16>, dim3((unsigned)nb), kScanThreads, st, rows_sorted,
                    w.rect_sorted, n_vis, w.block_sums, q_eff, N, div_magic_host((unsigned)N), ct,
                    sk[0], sv[0], vec16, packed, h, sgrid, hmask);
    count_launches(1);
  }
  // 5. stable sort of the super-pairs by super-tile id
  radix_sort(sk, sv, q_eff, q_bound, nullptr, sbits, w.hist, true, st, nullptr, hist0);
  const int sres = spasses & 1;
  const unsigned* sp_keys = sk[sres];
  const unsigned* sp_rows = sv[sres];  // == w.pv
  unsigned* desc = sk[1 - sres];
  // 6. rows of every super-tile (from the one-pass sort's digit totals, or
  //    marked on the sorted keys), segments, per-tile counts and list starts
  const unsigned* st_totals = nullptr;
  if (spasses == 1) {  // the digit totals are the per-super-tile item counts
    st_totals = w.hist + kRadixBins * radix_grid(q_bound);
  } else if (spasses > 1) {
    GS_TRY_CUDA(cudaMemsetAsync(w.st_ranges, 0, 2 * sizeof(unsigned) * (size_t)S, st));
    const unsigned gq = (unsigned)std::min<long long>((q_bound + 1023) / 1024, 152ll * 16);
    launch_behind(ranges_kernel, dim3(gq), 256, st, sp_keys, q_eff, packed ? 0xffffu : 0xffffffffu,
                  w.st_ranges);
    count_launches(1);
  }
  if (spasses > 1) {  // (else st_count_kernel forms the segments)
    launch_behind(st_segments_kernel, dim3(1), 1024, st,
                  reinterpret_cast<const uint2*>(w.st_ranges), S, w.seg_first, w.segs,
                  packed ? nullptr : w.seg_st, ct, n_seg);
    count_launches(1);
  }
  const unsigned gs = (unsigned)std::min<long long>(max_segments(q_bound, S), 152ll * 8);
  launch_behind(st_count_kernel, dim3(gs), 256, st, sp_keys, sp_rows, w.segs, w.seg_st, n_seg,
                packed, proj->rect, N, ct, desc, w.seg_hist, st_totals, q_eff, S, w.seg_first);
  launch_behind(st_scan_kernel, dim3((unsigned)S), 1024, st, w.seg_first, ct,
                reinterpret_cast<uint4*>(w.seg_hist), w.tile_cnt, arrive + 2, w.tile_start,
                ranges);
  // 7. every row into the lists of the tiles it covers, in depth order
  {
    const int e = stage_event(GS_STAGE_EXPANSION, false, st);
    if (e != GS_OK) return e;
  }
  const unsigned ge = (unsigned)std::min<long long>(max_segments(q_bound, S), kEmitGrid);
  if (sorted_keys)
    launch_behind(st_emit_kernel<true>, dim3(ge), 256, st, sp_keys, sp_rows, desc, packed, w.segs,
                  n_seg, w.seg_hist, w.tile_start, proj->depth, sorted_vals, sorted_keys, cap);
  else
    launch_behind(st_emit_kernel<false>, dim3(ge), 256, st, sp_keys, sp_rows, desc, packed, w.segs,
                  n_seg, w.seg_hist, w.tile_start, proj->depth, sorted_vals, nullptr, cap);
  {
    const int e = stage_event(GS_STAGE_EXPANSION, true, st);
    if (e != GS_OK) return e;
  }
  count_launches(3);
  return check_launch();
}

// ----------------------------------------------------------------------------
// Tile queue: global tile ids ordered by list length, longest first.
// ----------------------------------------------------------------------------
namespace {
__global__ void queue_keys_kernel(const unsigned* ranges, long long T,
                                  unsigned* keys, unsigned* vals) {
  behind_previous();
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < T;
       t += (long long)gridDim.x * blockDim.x) {
    unsigned len = ranges[2 * t + 1] - ranges[2 * t];
    keys[t] = 0xffffffffu - len;
    vals[t] = (unsigned)t;
  }
}
}  // namespace

size_t tile_queue_workspace_size(long long T) {
  return align256(4 * (T + 1)) * 3 + align256(sizeof(long long) * 2) +
         align256(radix_hist_bytes());
}

int launch_tile_queue(const unsigned* ranges, long long T, unsigned* order, void* ws,
                      size_t ws_bytes, cudaStream_t st) {
  if (ws_bytes < tile_queue_workspace_size(T)) return GS_ERR_INVALID_ARG;
  if (T == 0) return GS_OK;
  char* p = reinterpret_cast<char*>(ws);
  unsigned* k0 = reinterpret_cast<unsigned*>(p);
  p += align256(4 * (T + 1));
  unsigned* k1 = reinterpret_cast<unsigned*>(p);
  p += align256(4 * (T + 1));
  unsigned* v1 = reinterpret_cast<unsigned*>(p);
  p += align256(4 * (T + 1));
  long long* n_dev = reinterpret_cast<long long*>(p);
  p += align256(sizeof(long long) * 2);
  unsigned* hist = reinterpret_cast<unsigned*>(p);
  launch_behind(set_value_kernel, dim3(1), 32, st, n_dev, T);
  count_launches(1);
  unsigned grid = (unsigned)std::min<long long>((T + 255) / 256, 1024);
  // 4 passes (even): the result ends in the first buffer, i.e. `order`
  launch_behind(queue_keys_kernel, dim3(grid), 256, st, ranges, T, k0, order);
  count_launches(1);
  unsigned* k[2] = {k0, k1};
  unsigned* v[2] = {order, v1};
  radix_sort(k, v, n_dev, T, nullptr, 32, hist, false, st);
  return check_launch();
}

}  // namespace gs

// ----------------------------------------------------------------------------
// Tile queue without allocation: the same sort, run in a fixed scratch array
// in device global memory that the library owns (see gs_tile_queue_static in
// include/gs.h).
// ----------------------------------------------------------------------------

// Scratch of the no-allocation tile queue, sized for
// GS_TILE_QUEUE_STATIC_MAX_TILES tiles with the layout of launch_tile_queue:
// three key/value arrays, the count, and the radix histograms.  Every GPU that
// loads the library holds these bytes until the process exits.
static __device__ __align__(256) unsigned char g_queue_scratch[
    ((4ull * (GS_TILE_QUEUE_STATIC_MAX_TILES + 1) + 255) / 256 * 256) * 3 + 256 +
    (gs::radix_hist_bytes() + 255) / 256 * 256];

namespace {

constexpr int kMaxDevices = 64;
std::mutex g_queue_scratch_mutex;
struct ScratchAddr {
  unsigned long long ctx_id;  // context the address belongs to (0: none yet)
  void* ptr;
};
ScratchAddr g_queue_scratch_addr[kMaxDevices] = {};

// Unique id of the calling thread's current CUDA context (ids are never
// reused within a process), through the driver entry points the runtime
// exposes; 0 when there is no current context or the query is unavailable.
unsigned long long current_context_id() {
  typedef CUresult (*GetCurrent)(CUcontext*);
  typedef CUresult (*GetId)(CUcontext, unsigned long long*);
  static GetCurrent get_current = nullptr;
  static GetId get_id = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f, 12000, cudaEnableDefault, &q) ==
            cudaSuccess && q == cudaDriverEntryPointSuccess)
      get_current = reinterpret_cast<GetCurrent>(f);
    f = nullptr;
    if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &f, 12000, cudaEnableDefault, &q) ==
            cudaSuccess && q == cudaDriverEntryPointSuccess)
      get_id = reinterpret_cast<GetId>(f);
    cudaGetLastError();
  });
  CUcontext ctx = nullptr;
  unsigned long long id = 0;
  if (!get_current || !get_id || get_current(&ctx) != CUDA_SUCCESS || !ctx ||
      get_id(ctx, &id) != CUDA_SUCCESS)
    return 0;
  return id;
}

// Device address of g_queue_scratch in the current device's context (in host
// code the array's name is only a stand-in, not a device address).  Looked
// up once per device and context: a device reset or a new primary context
// (the module is then loaded again, at another address) brings a new lookup.
int queue_scratch_address(void** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return gs::set_cuda_error(e);
  if (dev < 0 || dev >= kMaxDevices)
    return gs::set_error_text_and_status("unsupported device index", GS_ERR_UNSUPPORTED);
  std::lock_guard<std::mutex> lock(g_queue_scratch_mutex);
  ScratchAddr& a = g_queue_scratch_addr[dev];
  unsigned long long ctx = current_context_id();
  if (!a.ptr || ctx == 0 || ctx != a.ctx_id) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_queue_scratch);  // makes the primary context current if needed
    if (e != cudaSuccess) return gs::set_cuda_error(e);
    if (ctx == 0) ctx = current_context_id();
    a.ptr = p;
    a.ctx_id = ctx;
  }
  *out = a.ptr;
  return GS_OK;
}

}  // namespace

extern "C" int gs_tile_queue_static(const unsigned* tile_ranges, long long total_tiles,
                                    unsigned* tile_order, gs_stream stream) {
  if (total_tiles < 0 || total_tiles > GS_TILE_QUEUE_STATIC_MAX_TILES) {
    char buf[160];
    snprintf(buf, sizeof buf,
             "invalid argument: gs_tile_queue_static supports at most %d tiles (got %lld)",
             GS_TILE_QUEUE_STATIC_MAX_TILES, total_tiles);
    return gs::set_error_text_and_status(buf, GS_ERR_INVALID_ARG);
  }
  if (total_tiles > 0 && (!tile_ranges || !tile_order))
    return gs::set_error_text_and_status("invalid argument: pointers", GS_ERR_INVALID_ARG);
  void* scratch = nullptr;
  const int rc = queue_scratch_address(&scratch);
  if (rc != GS_OK) return rc;
  // Nothing in the scratch needs to start at zero: each call writes every word
  // it reads (keys, values, histograms, the count) before reading it.
  return gs::launch_tile_queue(tile_ranges, total_tiles, tile_order, scratch,
                               sizeof(g_queue_scratch), (cudaStream_t)stream);
}
