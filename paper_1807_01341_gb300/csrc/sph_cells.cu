// Top-level cells and leaves (Sec. III-A of arXiv 1807.01341).
//
// Particles are binned into an n_c^3 grid whose width is at least the largest
// kernel support, so a particle only interacts with the 27 cells around its
// own.  Inside a cell the particles are ordered by the Morton code of their
// cell-relative position; the Morton order is the cell's octree, and the
// leaves are octree nodes holding at most leaf_max particles -- the GPU form
// of the paper's refinement of top-level cells into small sub-cells.  The
// (cell, Morton) keys are sorted by a stable LSD radix sort, so ties keep the
// previous particle order and the result is deterministic.
//
// A build is a fixed chain of launches whose sizes live on the device (no
// host read between the keys and the finished structure): keys, one launch
// per 8-bit digit (up to 65,536 particles one for all of them), every particle
// packed into a record and the records unpacked in the new order, one pass that
// splits every octree node and one compaction, for the particles (leaves) and
// again for the leaves (chunks and work groups).
#include <cooperative_groups.h>

#include <algorithm>
#include <cstddef>
#include <utility>

#include "sph_internal.cuh"

namespace sph {

namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int TILE = 4096;                 // items of a sort or compaction tile
constexpr int RS_DIGITS = 256;
constexpr int RS_PASSES_MAX = 7;           // 30 Morton + at most 24 cell bits
// Polls of a look-back before it gives up: wait_limit, where it is given, but
// enough for the tiles before to run (a poll is one load; a staging wait's
// suspends the warp).
constexpr int POLL_LIMIT = 1 << 22, POLL_MIN = 4096;

// ---------------------------------------------------------------------------
// maximum smoothing length
// ---------------------------------------------------------------------------
__global__ void k_reduce_hmax(const float *__restrict__ h, long long n, unsigned int *out) {
  float m = 0.0f;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    m = fmaxf(m, h[i]);
  for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(FULL, m, o));
  if ((threadIdx.x & 31) == 0) atomic_max_float_pos(out, m);
}

// ---------------------------------------------------------------------------
// cell keys: exact FP64 arithmetic (no contraction) so the cell of every
// particle is a function of its FP64 position alone
// ---------------------------------------------------------------------------
__device__ __forceinline__ double wrap_box(double x, double box) {
  if (x < 0.0) x = __dadd_rn(x, box);
  if (x >= box) x = __dsub_rn(x, box);
  return x;
}

__device__ __forceinline__ int axis_cell(double x, double w, int nc) {
  int c = (int)floor(__ddiv_rn(x, w));
  return c < 0 ? 0 : (c > nc - 1 ? nc - 1 : c);
}

__device__ __forceinline__ unsigned int axis_morton(double x, int c, double w) {
  double t = __ddiv_rn(__dsub_rn(x, __dmul_rn((double)c, w)), w);
  t = __dmul_rn(t, (double)(1 << MORTON_BITS));
  double ft = floor(t);
  long long q = (long long)ft;
  if (ft < 0.0) q = 0;
  if (q > (1 << MORTON_BITS) - 1) q = (1 << MORTON_BITS) - 1;
  return (unsigned int)q;
}

// Cell and Morton coordinate of one axis, cell * 1024 + Morton: the two
// functions above, whose four FP64 divisions and roundings per axis made the
// keys FP64-bound (1/64 of the FP32 rate: 336 us at 2.1M particles).  One
// fused multiply-add puts x (1024 / w) into the mantissa with 22 fractional
// bits; its error and the rounding of the divisions are below 2^-30 of a
// Morton step, so unless the fraction lies within 2^-21 of a whole number
// (or x outside the box) the whole part is what the divisions give.  There the
// divisions decide.
__device__ __forceinline__ unsigned int axis_code(double x, double w, double inv, int nc) {
  constexpr long long MAGIC = 0x41D0000000000000ll;  // 2^30: one ulp is 2^-22
  const double t = __fma_rn(x, inv, __longlong_as_double(MAGIC));
  const unsigned long long m = (unsigned long long)(__double_as_longlong(t) - MAGIC);
  const unsigned int frac = (unsigned int)m & ((1u << 22) - 1u);
  if (m < ((unsigned long long)nc << (MORTON_BITS + 22)) && frac - 2u < (1u << 22) - 4u)
    return (unsigned int)(m >> 22);
  const int c = axis_cell(x, w, nc);
  return ((unsigned int)c << MORTON_BITS) | axis_morton(x, c, w);
}

__device__ __forceinline__ unsigned int spread3(unsigned int v) {  // 10 bits, every third place
  v = (v | (v << 16)) & 0x030000FFu;
  v = (v | (v << 8)) & 0x0300F00Fu;
  v = (v | (v << 4)) & 0x030C30C3u;
  v = (v | (v << 2)) & 0x09249249u;
  return v;
}

// A position as the build takes it: wrapped into the box by one box length
// (the test on the bit patterns: no FP64 instruction in the common case).
__device__ __forceinline__ bool out_of_box(double x, double box) {
  const long long b = __double_as_longlong(x);
  return b < 0 || b >= __double_as_longlong(box);
}

// Totals of every digit of the sort, counted while the keys are made.
__device__ __forceinline__ void digits_begin(int passes, unsigned int *s_hist) {
  for (int k = threadIdx.x; k < passes * RS_DIGITS; k += blockDim.x) s_hist[k] = 0;
  __syncthreads();
}

__device__ __forceinline__ void digits_add(int passes, unsigned int *s_hist, unsigned long long key) {
  for (int p = 0; p < passes; p++)
    atomicAdd(&s_hist[p * RS_DIGITS + ((key >> (8 * p)) & 255u)], 1u);
}

__device__ __forceinline__ void digits_end(int passes, unsigned int *s_hist, unsigned int *totals) {
  __syncthreads();
  for (int k = threadIdx.x; k < passes * RS_DIGITS; k += blockDim.x)
    if (s_hist[k]) atomicAdd(&totals[k], s_hist[k]);
}

// (also counts in ds->build_bad the particles whose position is not finite or
// whose h is not a positive finite number: the rest of the build then leaves
// everything as it is and the caller rejects the input)
__global__ void __launch_bounds__(256)
    k_cell_keys(View v, int nc, double w, double inv, unsigned long long *__restrict__ keys,
                unsigned int *totals, int passes) {
  __shared__ unsigned int s_hist[RS_PASSES_MAX * RS_DIGITS];
  digits_begin(passes, s_hist);
  const unsigned int mort_mask = (1u << MORTON_BITS) - 1u;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < v.n;
       i += (long long)gridDim.x * blockDim.x) {
    const float hi = v.h[i];
    double x = v.x[i], y = v.y[i], z = v.z[i];
    if (!(isfinite(x) && isfinite(y) && isfinite(z) && hi > 0.0f && isfinite(hi)))
      atomicAdd(&v.ds->build_bad, 1u);
    if (out_of_box(x, v.box)) v.x[i] = x = wrap_box(x, v.box);
    if (out_of_box(y, v.box)) v.y[i] = y = wrap_box(y, v.box);
    if (out_of_box(z, v.box)) v.z[i] = z = wrap_box(z, v.box);
    const unsigned int ax = axis_code(x, w, inv, nc), ay = axis_code(y, w, inv, nc),
                       az = axis_code(z, w, inv, nc);
    const unsigned long long cid =
        ((unsigned long long)(ax >> MORTON_BITS) * nc + (ay >> MORTON_BITS)) * nc + (az >> MORTON_BITS);
    const unsigned int mort = (spread3(ax & mort_mask) << 2) | (spread3(ay & mort_mask) << 1) |
                              spread3(az & mort_mask);
    const unsigned long long key = (cid << KEY_MORTON_BITS) | mort;
    keys[i] = key;
    digits_add(passes, s_hist, key);
  }
  digits_end(passes, s_hist, totals);
}

// ---------------------------------------------------------------------------
// scans and look-back
// ---------------------------------------------------------------------------
// exclusive scan over the block of one value per thread; every thread calls it
// (s_sums: 33 words)
template <class T>
__device__ __forceinline__ T block_exclusive(T x, T *s_sums, T *total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  T inc = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const T y = __shfl_up_sync(FULL, inc, o);
    if (lane >= o) inc += y;
  }
  __syncthreads();  // (s_sums may still be read from an earlier call)
  if (lane == 31) s_sums[wid] = inc;
  __syncthreads();
  if (wid == 0) {
    const T s = lane < nw ? s_sums[lane] : (T)0;
    T si = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const T y = __shfl_up_sync(FULL, si, o);
      if (lane >= o) si += y;
    }
    s_sums[lane] = si - s;
    if (lane == 31) s_sums[32] = si;
  }
  __syncthreads();
  if (total) *total = s_sums[32];
  return s_sums[wid] + inc - x;
}

template <class T>
__device__ __forceinline__ T ld_relaxed(const T *p) {
  return *reinterpret_cast<const volatile T *>(p);
}
template <class T>
__device__ __forceinline__ void st_relaxed(T *p, T x) {
  *reinterpret_cast<volatile T *>(p) = x;
}

// Status of a tile in a chain: 0 not there yet, AGG its own counts, INC its
// counts and those of every tile before it.  Tiles are handed out by a ticket,
// so every tile before a running one is running or done and a wait ends; a
// wait that exceeds its limit all the same (or meets another block's failure)
// sets *fail and the build's later kernels return without writing.
__device__ __forceinline__ bool poll_failed(int polls, int limit, unsigned int *fail) {
  if (polls >= limit) {
    atomicCAS(fail, 0u, (unsigned int)SPH_ERR_TIMEOUT);
    return true;
  }
  return (polls & 1023) == 1023 && ld_relaxed(fail) != 0u;
}

// Testing (a library built with SPH_CHECKS; sph_params.test_build_stall):
// whether this tile keeps its status to itself (one thread of the tile asks).
enum { STALL_SORT = 1, STALL_LEAVES = 2, STALL_CHUNKS = 3 };
#ifdef SPH_CHECKS
constexpr bool PLANTS = true;
#else
constexpr bool PLANTS = false;
#endif
__device__ __forceinline__ bool planted_stall(DevState *ds, int stage, int tile) {
  return PLANTS && ds && tile == 0 && gridDim.x > 1 &&
         atomicCAS(&ds->test_build_stall, stage, 0) == stage;
}

// Chain of one 64-bit word per tile (two counts of 31 bits; bits 62-63: the
// state), looked back 32 tiles at a time by one warp.
constexpr unsigned long long CH_AGG = 1ull << 62, CH_INC = 2ull << 62, CH_VAL = (1ull << 62) - 1ull;
__device__ bool chain_prefix(unsigned long long *status, int tile, unsigned long long mine,
                             unsigned long long *prefix, DevState *ds, int stage, int limit) {
  const int lane = threadIdx.x & 31;
  unsigned int *const fail = &ds->build_fail;
  unsigned long long pre = 0ull;
  if (lane == 0 && !planted_stall(ds, stage, tile))
    st_relaxed(&status[tile], (tile == 0 ? CH_INC : CH_AGG) | mine);
  for (int p = tile - 1; p >= 0; p -= 32) {
    const int t = p - lane;
    unsigned long long s = CH_INC;
    for (int polls = 0;; polls++) {
      s = t >= 0 ? ld_relaxed(&status[t]) : CH_INC;
      if (!__any_sync(FULL, (s & ~CH_VAL) == 0ull)) break;
      if (__any_sync(FULL, poll_failed(polls, limit, fail))) return false;
    }
    const unsigned inc = __ballot_sync(FULL, (s & CH_INC) != 0ull);
    const int last = inc ? __ffs(inc) - 1 : 31;
    unsigned long long x = lane <= last ? (s & CH_VAL) : 0ull;
#pragma unroll
    for (int o = 16; o; o >>= 1) x += __shfl_xor_sync(FULL, x, o);
    pre += x;
    if (inc) break;
  }
  if (lane == 0 && tile > 0) st_relaxed(&status[tile], CH_INC | (pre + mine));
  *prefix = pre;
  return true;
}

// The lanes whose low `bits` bits of x equal this lane's, by one vote per bit
// (match.any takes a round per distinct value: 32 for the random low digits).
template <int BITS>
__device__ __forceinline__ unsigned equal_lanes(unsigned int x) {
  unsigned peers = FULL;
#pragma unroll
  for (int b = 0; b < BITS; b++) {
    const bool one = (x >> b) & 1u;
    const unsigned m = __ballot_sync(FULL, one);
    peers &= one ? m : ~m;
  }
  return peers;
}

// ---------------------------------------------------------------------------
// stable LSD radix sort, 8-bit digits: one launch per digit
// ---------------------------------------------------------------------------
// A block takes a tile of 4,096 pairs, warp w the 32 ITEMS pairs from w 32 ITEMS
// on, in rounds of 32: a pair's rank among the equal digits of its tile is the
// count in the warps before, in the warp's earlier rounds and in the lanes
// below.  The tile is laid out by digit in shared memory and written out in
// runs.  The pairs of a digit in the tiles before this one come by look-back
// over those tiles (one status word per tile and digit: 2 bits of state, 30 of
// count), the digits' starts from totals counted with the keys, so a pass is
// one launch that reads and writes each pair once (before: three to five
// launches a pass, each key read twice, 256 pairs at a time).  Bound by the
// votes of the ranking and the latency of a tile's phases, not by its 24 bytes
// a pair: 2.1M pairs, 6 passes 275 -> 173 us; 16.8M 2340 -> 1030 us; 33k, 5
// passes 140 -> 40 us.  (Three blocks per SM spill and lengthen the look-back:
// 197 us at 2.1M.  Counting the next digit by destination tile during the
// scatter needs no look-back but was slower at every size it could serve:
// 47 against 37 us at one tile, 68 against 58 us at 64.)
//
// The look-back is that of Merrill and Garland's single-pass scan (2016) over
// one status word per tile and digit.  Without CHAIN the tiles' digit counts
// are there already (k_rs_tile_counts, `cur`; none for a single tile) and
// nothing waits: for callers that have no way to hear of a wait that gave up.
constexpr int RS_THREADS = 512;
template <bool CHAIN>
__global__ void __launch_bounds__(RS_THREADS, 2)
    k_rs_pass(const unsigned long long *__restrict__ keys, const unsigned int *__restrict__ vals,
              unsigned long long *__restrict__ okeys, unsigned int *__restrict__ ovals, int n,
              int shift, unsigned int *cur, unsigned int *clear,
              const unsigned int *__restrict__ totals, unsigned int *ticket, unsigned int *fail,
              const unsigned int *bad, DevState *ds, int limit) {
  constexpr int THREADS = RS_THREADS, ITEMS = TILE / THREADS, WARPS = THREADS / 32;
  constexpr unsigned AGG = 1u << 30, INC = 2u << 30, VAL = AGG - 1u;
  __shared__ unsigned long long s_keys[TILE];
  __shared__ unsigned int s_lofs[RS_DIGITS], s_gofs[RS_DIGITS], s_sums[33];
  __shared__ int s_tile, s_fail, s_hold;
  unsigned int *const wcnt = reinterpret_cast<unsigned int *>(s_keys);  // [WARPS][256], until the scatter
  static_assert(WARPS * RS_DIGITS * 4 <= TILE * 8, "the warps' counters fit the staging area");
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (CHAIN && tid == 0) {
    s_tile = (int)atomicAdd(ticket, 1u);
    s_fail = ld_relaxed(fail) != 0u || (bad && *bad != 0u);
    if (PLANTS) s_hold = planted_stall(ds, STALL_SORT, s_tile) ? 1 : 0;
  }
  for (int k = lane; k < RS_DIGITS; k += 32) wcnt[warp * RS_DIGITS + k] = 0u;
  __syncthreads();
  if (CHAIN && s_fail) return;
  const int tile = CHAIN ? s_tile : (int)blockIdx.x;
  const int base = tile * TILE, count = min(TILE, n - base);
  if (CHAIN && tid < RS_DIGITS) clear[tile * RS_DIGITS + tid] = 0u;
  unsigned long long key[ITEMS];
  unsigned int rank[ITEMS];
#pragma unroll
  for (int r = 0; r < ITEMS; r++) {
    const int o = warp * (32 * ITEMS) + r * 32 + lane;
    // (past the end: the largest digit, after every pair of the tile)
    key[r] = o < count ? keys[base + o] : ~0ull;
  }
#pragma unroll
  for (int r = 0; r < ITEMS; r++) {
    const unsigned int d = (unsigned int)(key[r] >> shift) & 255u;
    const unsigned peers = equal_lanes<8>(d);
    const int leader = __ffs(peers) - 1;
    unsigned int old = 0u;
    if (lane == leader) {
      old = wcnt[warp * RS_DIGITS + d];
      wcnt[warp * RS_DIGITS + d] = old + __popc(peers);
    }
    rank[r] = __shfl_sync(FULL, old, leader) + __popc(peers & ((1u << lane) - 1u));
    __syncwarp();
  }
  __syncthreads();
  unsigned int mine = 0u, tot = 0u, prev = 0u;
  if (tid < RS_DIGITS) {
#pragma unroll 8
    for (int q = 0; q < WARPS; q++) {
      const unsigned int c = wcnt[q * RS_DIGITS + tid];
      wcnt[q * RS_DIGITS + tid] = mine;
      mine += c;
    }
    // (the padding of the last tile counts there, where nothing follows)
    if (CHAIN) {
      if (!PLANTS || !s_hold)
        st_relaxed(&cur[tile * RS_DIGITS + tid], (tile == 0 ? INC : AGG) | mine);
      tot = totals[tid];
    } else {
      const int tiles = (int)gridDim.x;
      tot = mine;
      if (tiles > 1) {
        tot = 0u;
        for (int t = 0; t < tiles; t++) {
          const unsigned int c = cur[t * RS_DIGITS + tid];
          prev += t < tile ? c : 0u;
          tot += c;
        }
      }
    }
  }
  const unsigned int lofs = block_exclusive<unsigned int>(mine, s_sums, nullptr);
  const unsigned int gofs = block_exclusive<unsigned int>(tot, s_sums, nullptr);
  if (CHAIN && tid < RS_DIGITS && tile > 0) {
    // LB tiles a round, their words loaded together: blocks that start
    // together walk back over one another, one word at a time half as many
    // rounds as there are tiles in flight
    constexpr int LB = 8;
    bool ok = true, found = false;
    for (int t = tile - 1; ok && !found; t -= LB) {
      unsigned int w[LB];
      for (int polls = 0;; polls++) {
        bool ready = true;
#pragma unroll
        for (int q = 0; q < LB; q++)
          w[q] = t - q >= 0 ? ld_relaxed(&cur[(t - q) * RS_DIGITS + tid]) : INC;
        // (every word up to the first complete one must be there)
        bool open = true;
#pragma unroll
        for (int q = 0; q < LB; q++) {
          if (open && !(w[q] & (AGG | INC))) ready = false;
          if (w[q] & INC) open = false;
        }
        if (ready) break;
        if (poll_failed(polls, limit, fail)) {
          ok = false;
          break;
        }
      }
#pragma unroll
      for (int q = 0; q < LB; q++) {
        if (!found) prev += w[q] & VAL;
        found = found || (w[q] & INC) != 0u;
      }
    }
    if (ok) st_relaxed(&cur[tile * RS_DIGITS + tid], INC | (prev + mine));
    else s_fail = 1;
  }
  if (tid < RS_DIGITS) {
    s_lofs[tid] = lofs;
    s_gofs[tid] = gofs + prev - lofs;
  }
  __syncthreads();
  if (CHAIN && s_fail) return;
#pragma unroll
  for (int r = 0; r < ITEMS; r++) {
    const unsigned int d = (unsigned int)(key[r] >> shift) & 255u;
    rank[r] += s_lofs[d] + wcnt[warp * RS_DIGITS + d];  // the pair's place in the tile
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < ITEMS; r++) s_keys[rank[r]] = key[r];
  __syncthreads();
  unsigned int pos[ITEMS], val[ITEMS];
#pragma unroll
  for (int r = 0; r < ITEMS; r++) {
    const int o = warp * (32 * ITEMS) + r * 32 + lane;
    val[r] = o < count ? (vals ? vals[base + o] : (unsigned int)(base + o)) : 0u;
  }
#pragma unroll
  for (int r = 0; r < ITEMS; r++) {
    const int p = r * THREADS + tid;
    const unsigned long long k = s_keys[p];
    pos[r] = s_gofs[(unsigned int)(k >> shift) & 255u] + (unsigned int)p;
    if (p < count && SPH_IN(ds, pos[r], n, SPH_CHECK_SCATTER)) okeys[pos[r]] = k;
  }
  __syncthreads();
  unsigned int *const s_vals = reinterpret_cast<unsigned int *>(s_keys);
#pragma unroll
  for (int r = 0; r < ITEMS; r++) s_vals[rank[r]] = val[r];
  __syncthreads();
#pragma unroll
  for (int r = 0; r < ITEMS; r++) {
    const int p = r * THREADS + tid;
    if (p < count && SPH_IN(ds, pos[r], n, SPH_CHECK_SCATTER)) ovals[pos[r]] = s_vals[p];
  }
}

// digit counts of every tile
__global__ void __launch_bounds__(RS_THREADS)
    k_rs_tile_counts(const unsigned long long *__restrict__ keys, int n, int shift,
                     unsigned int *__restrict__ counts) {
  __shared__ unsigned int s_hist[RS_DIGITS];
  if (threadIdx.x < RS_DIGITS) s_hist[threadIdx.x] = 0u;
  __syncthreads();
  const int end = min(n, ((int)blockIdx.x + 1) * TILE);
#pragma unroll 8
  for (int i = (int)blockIdx.x * TILE + (int)threadIdx.x; i < end; i += RS_THREADS)
    atomicAdd(&s_hist[(keys[i] >> shift) & 255u], 1u);
  __syncthreads();
  if (threadIdx.x < RS_DIGITS) counts[blockIdx.x * RS_DIGITS + threadIdx.x] = s_hist[threadIdx.x];
}

// The same sort of up to 65,536 pairs in one launch: the 8 or 16 blocks of a
// cluster hold them all in shared memory, a pair in one word (key << 16 |
// index, so keys of up to 48 bits), every pass within the cluster.  Block c
// holds the places [c T, (c + 1) T), T = 1024 ITEMS, past the end filled with
// the largest word, which every digit leaves at the end.  A pass ranks the words as k_rs_pass
// does, gives its digit counts to every block, orders its words by digit and
// writes them in runs to their places, the other blocks' shared memory among
// them; a cluster barrier before the counts are read and one before the words
// are.  (Keys and indices are read before the first barrier and written after
// the last: in place.)
//
// A small sort is latency: a launch per digit took 7 to 8 us and a gap of 2 us
// with one to 16 blocks at work, a pass in here takes what its barriers and the
// votes of its ranking do.  Keys counted to records packed, 5 passes: 4,096
// pairs 48 -> 24 us, 16,384 52 -> 26, 32,768 53 -> 32, 40,000 52 -> 36, 65,536 (6
// passes) 65 -> 49.  With 8 blocks for all sizes 40,000 took 56 us and 32,768 37;
// 16 blocks for 4,096 take 27.  The line is the 16-bit index: keys of more than
// 48 bits (64 cells an axis) and more pairs take a launch per digit, and so does
// what the device cannot place (cluster_sort_max: a partition of a GPU may have
// no 16, or no 8, SMs that form a cluster).
constexpr int RC_THREADS = 1024, RC_INDEX_BITS = 16;
constexpr int RC_MAX = 16 * RC_THREADS * 4;  // of the largest instance below
static_assert(RC_MAX <= 1 << RC_INDEX_BITS, "an index has 16 bits");
template <int BLOCKS, int ITEMS>
__global__ void __cluster_dims__(BLOCKS, 1, 1) __launch_bounds__(RC_THREADS, 1)
    k_rs_cluster(unsigned long long *keys, unsigned int *vals, int n, int passes,
                 const unsigned int *bad, DevState *ds) {
  namespace cg = cooperative_groups;
  constexpr int T = RC_THREADS * ITEMS, WARPS = RC_THREADS / 32;
  extern __shared__ unsigned long long s_words[];  // in order, then by digit of the block
  unsigned long long *const s_order = s_words, *const s_stage = s_words + T;
  __shared__ unsigned short s_wcnt[WARPS][RS_DIGITS];
  __shared__ unsigned int s_all[BLOCKS][RS_DIGITS];  // every block's digit counts
  __shared__ unsigned int s_lofs[RS_DIGITS], s_gofs[RS_DIGITS], s_sums[33];
  if (bad && *bad != 0u) return;  // (the whole cluster: an earlier launch wrote it)
  cg::cluster_group cluster = cg::this_cluster();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int self = (int)cluster.block_rank();
  unsigned long long word[ITEMS];
#pragma unroll
  for (int r = 0; r < ITEMS; r++) {
    const int o = self * T + warp * (32 * ITEMS) + r * 32 + lane;
    word[r] = o < n ? keys[o] << RC_INDEX_BITS | (unsigned int)o : ~0ull;
  }
  cluster.sync();  // every block runs before its shared memory is written
  for (int p = 0; p < passes; p++) {
    const int shift = RC_INDEX_BITS + 8 * p;
    auto digit = [&](unsigned long long w) { return (unsigned int)(w >> shift) & 255u; };
    for (int k = lane; k < RS_DIGITS; k += 32) s_wcnt[warp][k] = 0;
    __syncwarp();
    unsigned int rank[ITEMS];
#pragma unroll
    for (int r = 0; r < ITEMS; r++) {
      const unsigned int d = digit(word[r]);
      const unsigned peers = equal_lanes<8>(d);
      const int leader = __ffs(peers) - 1;
      unsigned int old = 0u;
      if (lane == leader) {
        old = s_wcnt[warp][d];
        s_wcnt[warp][d] = (unsigned short)(old + __popc(peers));
      }
      rank[r] = __shfl_sync(FULL, old, leader) + __popc(peers & ((1u << lane) - 1u));
      __syncwarp();
    }
    __syncthreads();
    unsigned int mine = 0u;
    if (tid < RS_DIGITS) {
#pragma unroll
      for (int q = 0; q < WARPS; q++) {
        const unsigned int c = s_wcnt[q][tid];
        s_wcnt[q][tid] = (unsigned short)mine;
        mine += c;
      }
#pragma unroll
      for (int b = 0; b < BLOCKS; b++) *cluster.map_shared_rank(&s_all[self][tid], b) = mine;
    }
    const unsigned int lofs = block_exclusive<unsigned int>(mine, s_sums, nullptr);
    cluster.sync();
    unsigned int tot = 0u, prev = 0u;
    if (tid < RS_DIGITS) {
#pragma unroll
      for (int b = 0; b < BLOCKS; b++) {
        const unsigned int c = s_all[b][tid];
        prev += b < self ? c : 0u;
        tot += c;
      }
    }
    const unsigned int gofs = block_exclusive<unsigned int>(tot, s_sums, nullptr);
    if (tid < RS_DIGITS) {
      s_lofs[tid] = lofs;
      s_gofs[tid] = gofs + prev - lofs;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < ITEMS; r++) {
      const unsigned int d = digit(word[r]);
      s_stage[s_lofs[d] + s_wcnt[warp][d] + rank[r]] = word[r];
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < ITEMS; r++) {
      const int k = r * RC_THREADS + tid;
      const unsigned long long w = s_stage[k];
      const unsigned int to = s_gofs[digit(w)] + (unsigned int)k;
      if (SPH_IN(ds, to, BLOCKS * T, SPH_CHECK_SCATTER))
        *cluster.map_shared_rank(&s_order[to % T], to / T) = w;
    }
    cluster.sync();
#pragma unroll
    for (int r = 0; r < ITEMS; r++) word[r] = s_order[warp * (32 * ITEMS) + r * 32 + lane];
  }
#pragma unroll
  for (int r = 0; r < ITEMS; r++) {
    const int o = self * T + warp * (32 * ITEMS) + r * 32 + lane;
    if (o < n) {
      keys[o] = word[r] >> RC_INDEX_BITS;
      vals[o] = (unsigned int)word[r] & ((1u << RC_INDEX_BITS) - 1u);
    }
  }
}

// ---------------------------------------------------------------------------
// permutation of the particle arrays
// ---------------------------------------------------------------------------
// Every array of a particle packed into one 128-byte record, in the caller's
// order (coalesced reads, whole-sector writes), then the records fetched in
// the sorted order, one line each, and written back to the arrays.  A gather
// per array reads a 32-byte sector for every 4 or 8 bytes where the caller's
// order is random: 2.1M clustered particles 350 us in 26 gathers and copies
// back (297 + 84 us as one gather into scratch and one copy back), 81 + 91 us
// here, 5.4 TB/s of the 460 + 536 MB both move.
constexpr int PF8 = 6, PF4 = 19;  // 8-byte and 4-byte arrays of a particle
struct Fields {
  unsigned long long *p8[PF8];
  unsigned int *p4[PF4];
  uint8_t *bin;
  char *records;
};

__device__ __forceinline__ void st_32b(void *p, const unsigned int *w) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(w[0]),
               "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
               : "memory");
}
__device__ __forceinline__ void ld_32b(const void *p, unsigned int *w) {
  asm volatile("ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]), "=r"(w[4]), "=r"(w[5]), "=r"(w[6]),
                 "=r"(w[7])
               : "l"(p)
               : "memory");
}

__device__ __forceinline__ bool build_stopped(const DevState *ds) {
  return ds->build_bad != 0u || ds->build_fail != 0u;
}

// No work queue survives a build: their entries are indices into the structure
// before it, and the density loop's lie in the build's scratch.
__device__ __forceinline__ void clear_queues(DevState *ds) {
  ds->n_active_leaves = ds->n_active_groups = ds->n_heavy_groups = 0;
  ds->n_active_cells = ds->n_drift_chunks = 0;
  ds->n_bin_groups = ds->n_bin_coop = 0;
  ds->n_wake = 0;
  ds->n_big = ds->head_big = ds->dens_split = 0;
}

// Words 0-11 the 8-byte arrays, 12-30 the 4-byte ones (the mass first), 31 the
// particle's index in the first build's order (below 2^24) with its bin above.
// (old: the composed permutation of the first n_old particles; the others are
// new to it and start at their own place.)  Also the masses' range, as float bits: masses are positive, and any other value
// only makes the two ends differ, which selects the general density loop.
static_assert(2 * PF8 + PF4 + 1 == 32 && BUILD_SCRATCH == 128 && BUILD_MAX <= 1ll << 24,
              "a particle's arrays fill one record");
__global__ void __launch_bounds__(256)
    k_pack(View v, Fields f, const int32_t *__restrict__ old, long long n_old) {
  DevState *ds = v.ds;
  unsigned int nlo = 0u, hi = 0u;
  for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < v.n;
       k += (long long)gridDim.x * blockDim.x) {
    unsigned int w[32];
#pragma unroll
    for (int q = 0; q < PF8; q++) {
      const unsigned long long a = f.p8[q][k];
      w[2 * q] = (unsigned int)a;
      w[2 * q + 1] = (unsigned int)(a >> 32);
    }
#pragma unroll
    for (int q = 0; q < PF4; q++) w[2 * PF8 + q] = f.p4[q] ? f.p4[q][k] : 0u;
    w[31] = (unsigned int)(k < n_old ? old[k] : (int32_t)k) | ((unsigned int)f.bin[k] << 24);
    char *r = f.records + k * BUILD_SCRATCH;
#pragma unroll
    for (int q = 0; q < 4; q++) st_32b(r + 32 * q, w + 8 * q);
    nlo = max(nlo, ~w[2 * PF8]);
    hi = max(hi, w[2 * PF8]);
  }
  nlo = __reduce_max_sync(FULL, nlo);
  hi = __reduce_max_sync(FULL, hi);
  if ((threadIdx.x & 31) == 0) {
    atomicMax(&ds->m_nlo_bits, nlo);
    atomicMax(&ds->m_hi_bits, hi);
  }
  if (blockIdx.x == 0 && threadIdx.x < MAX_BINS && !build_stopped(ds))
    ds->bin_count[threadIdx.x] = 0;
}

// The records in the sorted order; cleared leaf marks, the occupancy of the
// time bins and the state of the new structure.
__global__ void __launch_bounds__(256)
    k_unpack(View v, Fields f, const unsigned int *__restrict__ order, int32_t *__restrict__ perm,
             uint8_t *__restrict__ lead, int nc, double w) {
  DevState *ds = v.ds;
  if (build_stopped(ds)) return;
  __shared__ int h[MAX_BINS];
  if (threadIdx.x < MAX_BINS) h[threadIdx.x] = 0;
  __syncthreads();
  const long long n = v.n;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    ds->nc = nc;
    ds->n_cells = nc * nc * nc;
    ds->w = w;
    ds->build_moved = 1u;
    clear_queues(ds);
    ds->excursion_bits = ds->Hmax_bits = ds->want_h_bits = 0u;
    ds->group_cost_sum = 0ull;
    // equal masses: the density loop sums the kernel alone (rho = m sum w)
    const unsigned int lo = ~ds->m_nlo_bits, hi = ds->m_hi_bits;
    const float m = __uint_as_float(lo);
    ds->m_uniform = n > 0 && lo == hi && m > 0.0f && isfinite(m) ? m : 0.0f;
  }
  for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n;
       k += (long long)gridDim.x * blockDim.x) {
    const unsigned int s = order[k];
    if (!SPH_IN(ds, s, n, SPH_CHECK_SCATTER)) continue;
    const char *r = f.records + (long long)s * BUILD_SCRATCH;
    unsigned int a[32];
#pragma unroll
    for (int q = 0; q < 4; q++) ld_32b(r + 32 * q, a + 8 * q);
#pragma unroll
    for (int q = 0; q < PF8; q++)
      f.p8[q][k] = (unsigned long long)a[2 * q] | ((unsigned long long)a[2 * q + 1] << 32);
#pragma unroll
    for (int q = 0; q < PF4; q++)
      if (f.p4[q]) f.p4[q][k] = a[2 * PF8 + q];
    const unsigned int bin = a[31] >> 24;
    f.bin[k] = (uint8_t)bin;
    perm[k] = (int32_t)(a[31] & 0xffffffu);
    v.active[k] = 0;
    lead[k] = 0;
    atomicAdd(&h[bin & (MAX_BINS - 1)], 1);
  }
  __syncthreads();
  if (threadIdx.x < MAX_BINS && h[threadIdx.x]) atomicAdd(&ds->bin_count[threadIdx.x], h[threadIdx.x]);
}

// ---------------------------------------------------------------------------
// cell boundaries and leaves
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t compact3(unsigned long long m) {
  uint32_t r = 0;
#pragma unroll
  for (int b = 0; b < MORTON_BITS; b++) r |= (uint32_t)((m >> (3 * b)) & 1ull) << b;
  return r;
}

// Morton-grid corner (packed kx | ky << 10 | kz << 20) of a particle's code,
// truncated to the octree level of its node
__device__ __forceinline__ uint32_t corner_of(unsigned long long key, int level) {
  const unsigned long long m = key & ((1ull << KEY_MORTON_BITS) - 1ull);
  const int drop = 3 * (MORTON_BITS - level);
  const unsigned long long t = drop >= KEY_MORTON_BITS ? 0ull : (m >> drop) << drop;
  return compact3(t >> 2) | (compact3(t >> 1) << 10) | (compact3(t) << 20);
}

// Deepest octree level (0: the cell, 10: the finest) whose node holds both
// keys; -1 when their cells differ.
__device__ __forceinline__ int common_level(unsigned long long a, unsigned long long b) {
  const unsigned long long x = a ^ b;
  if (x >> KEY_MORTON_BITS) return -1;
  if (x == 0ull) return MORTON_BITS;
  return (KEY_MORTON_BITS - 1 - (31 - __clz((unsigned int)x))) / 3;
}

// First index in (i, n) whose key is at least target; i when key_i already is.
__device__ __forceinline__ int first_at_least(const unsigned long long *__restrict__ keys, int i,
                                              unsigned long long key_i, int n,
                                              unsigned long long target) {
  if (key_i >= target) return i;
  int lo = i, step = 8, hi = i + 8;  // key[lo] < target
  while (hi < n && keys[hi] < target) {
    lo = hi;
    step <<= 1;
    hi = lo + step;
  }
  hi = min(hi, n);
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (keys[mid] < target) lo = mid;
    else hi = mid;
  }
  return hi;
}

// Leaves: the octree of each cell's Morton-ordered items.  A node holding more
// than `most` items is split into its 8 children; consecutive children that
// hold at most `most` items between them are merged into one leaf (siblings,
// so the leaf stays inside the parent node), and larger children are split in
// turn.  At the deepest level a node is cut into runs of `most`.  Every leaf
// is marked at its first item by lead[s] = 1 + the level of the node it lies
// in; the marks, compacted in item order, give the leaves cell by cell in the
// order of a depth-first walk.  All items of a leaf share the Morton prefix of
// that level, so its corner follows from the first item's code.
// Whether a node is split depends on its own count alone (a parent holds at
// least as many), so every node of every level is found at its first item i
// -- the levels at which key i - 1 lies in another node, as far as key
// i + most still lies in the same one -- and split in one pass: 8 lanes per
// node, each finding the first item of one child by a galloping search (one
// launch per level before, ten per tree: leaves and chunks of 2.1M clustered
// particles 150 us, now 39 us and, with the work groups beside them, 71 us).
__device__ __forceinline__ void split_nodes(const unsigned long long *__restrict__ keys, int n,
                                            int i, int most, uint8_t *__restrict__ lead,
                                            unsigned long long key, int first_level) {
  const int lane = threadIdx.x & 31, j = lane & 7;
  unsigned int pend = 0u;  // levels at which this lane's item starts a node to split
  if (i < n) {
    const int deep = i + most < n ? common_level(key, keys[i + most]) : -1;
    if (first_level == 0 && deep < 0) lead[i] = 1;  // a cell of at most `most` items
    const int last = min(deep, MORTON_BITS - 1);
    if (last >= first_level) pend = (2u << last) - (1u << first_level);
  }
  for (;;) {
    const unsigned m = __ballot_sync(FULL, pend != 0u);
    if (m == 0u) break;
    // the first four lanes with a node left, one node each
    unsigned t = m;
    for (int q = 0; q < (lane >> 3); q++) t &= t - 1u;
    const int src = t ? __ffs(t) - 1 : 0;
    const int level = __ffs(__shfl_sync(FULL, pend, src)) - 1;
    const unsigned long long k0 = __shfl_sync(FULL, key, src);
    const int i0 = __shfl_sync(FULL, i, src);
    if (pend && __popc(m & ((1u << lane) - 1u)) < 4) pend &= pend - 1u;
    if (t == 0u) continue;  // (8 lanes together)
    const unsigned gmask = 0xFFu << (lane & 24);
    const int sh = 3 * (MORTON_BITS - 1 - level);
    const unsigned long long node = (k0 >> (sh + 3)) << (sh + 3);
    // lane j: the first item of child j + 1 (j = 7: the node's end)
    const int mine = first_at_least(keys, i0, k0, n, node + ((unsigned long long)(j + 1) << sh));
    int bnd[9];
    bnd[0] = i0;
#pragma unroll
    for (int q = 0; q < 8; q++) bnd[q + 1] = __shfl_sync(gmask, mine, q, 8);
    if (j != 0) continue;
    int sum = 0;  // items of the leaf being merged (0: none open)
#pragma unroll
    for (int q = 0; q < 8; q++) {
      const int c = bnd[q + 1] - bnd[q];
      if (c == 0) continue;
      if (c > most) {
        // (split at its own first item, or, at the deepest level, cut into runs)
        if (level + 1 == MORTON_BITS)
          for (int s = bnd[q]; s < bnd[q + 1]; s += most) lead[s] = (uint8_t)(MORTON_BITS + 1);
        sum = 0;
        continue;
      }
      if (sum == 0 || sum + c > most) {
        lead[bnd[q]] = (uint8_t)(level + 1);
        sum = 0;
      }
      sum += c;
    }
  }
}

__global__ void __launch_bounds__(256)
    k_leaf_nodes(const unsigned long long *__restrict__ keys, int n, int n_cells, int leaf_max,
                 uint8_t *__restrict__ lead, int32_t *__restrict__ cell_start, const DevState *ds) {
  if (build_stopped(ds)) return;
  const int stride = gridDim.x * blockDim.x;
  for (int b = blockIdx.x * blockDim.x + (threadIdx.x & ~31); b < n; b += stride) {
    const int i = b + (threadIdx.x & 31);
    unsigned long long key = 0ull;
    int first_level = MORTON_BITS + 1;
    if (i < n) {
      key = keys[i];
      const int c = (int)(key >> KEY_MORTON_BITS);
      int cp = -1;
      first_level = 0;
      if (i > 0) {
        const unsigned long long prev = keys[i - 1];
        cp = (int)(prev >> KEY_MORTON_BITS);
        first_level = common_level(key, prev) + 1;
      }
      for (int cc = cp + 1; cc <= c; cc++) cell_start[cc] = i;
      if (i == n - 1)
        for (int cc = c + 1; cc <= n_cells; cc++) cell_start[cc] = n;
    }
    split_nodes(keys, n, i, leaf_max, lead, key, first_level);
  }
}

// Compaction of the leaves' marks, one tile of 4,096 particles per block: leaf
// records, the leaf of every particle, first leaf of every cell, the leaves'
// first keys and cleared marks for the chunks, closing entries.
constexpr int CT = 512;  // threads of a compaction block: 8 items each
__global__ void __launch_bounds__(CT)
    k_leaf_emit(const unsigned long long *__restrict__ keys, const uint8_t *__restrict__ lead, int n,
                int n_cells, unsigned long long *status, unsigned int *ticket,
                int32_t *__restrict__ leaf_start, int32_t *__restrict__ leaf_cell,
                uint32_t *__restrict__ leaf_k, int32_t *__restrict__ cell_leaf_start,
                int32_t *__restrict__ pleaf, unsigned long long *__restrict__ leaf_keys,
                uint8_t *__restrict__ chunk_lead, uint8_t *__restrict__ group_lead, DevState *ds,
                int limit) {
  __shared__ unsigned int s_sums[33];
  __shared__ unsigned long long s_pre;
  __shared__ int s_tile, s_stop;
  if (threadIdx.x == 0) {
    s_stop = build_stopped(ds) ? 1 : 0;
    s_tile = (int)atomicAdd(ticket, 1u);
  }
  __syncthreads();
  if (s_stop) return;
  const int tile = s_tile;
  const int base = tile * TILE + (int)threadIdx.x * 8;
  uint8_t l[8];
  unsigned int s = 0;
  if (base + 8 <= n) {
    const uint2 q = *reinterpret_cast<const uint2 *>(lead + base);
#pragma unroll
    for (int k = 0; k < 4; k++) {
      l[k] = (uint8_t)(q.x >> (8 * k));
      l[k + 4] = (uint8_t)(q.y >> (8 * k));
    }
  } else {
#pragma unroll
    for (int k = 0; k < 8; k++) l[k] = base + k < n ? lead[base + k] : (uint8_t)0;
  }
#pragma unroll
  for (int k = 0; k < 8; k++) s += l[k] != 0;
  unsigned int tot;
  unsigned int off = block_exclusive<unsigned int>(s, s_sums, &tot);
  if (threadIdx.x < 32) {
    unsigned long long pre = 0ull;
    const bool ok = chain_prefix(status, tile, tot, &pre, ds, STALL_LEAVES, limit);
    if (threadIdx.x == 0) {
      s_pre = pre;
      s_stop = ok ? 0 : 1;
    }
  }
  __syncthreads();
  if (s_stop) return;
  off += (unsigned int)s_pre;
#pragma unroll
  for (int k = 0; k < 8; k++) {
    const int i = base + k;
    if (i >= n) break;
    if (l[k]) {
      const unsigned long long key = keys[i];
      const int c = (int)(key >> KEY_MORTON_BITS);
      leaf_start[off] = i;
      leaf_cell[off] = c;
      leaf_k[off] = corner_of(key, l[k] - 1);
      leaf_keys[off] = key;
      chunk_lead[off] = 0;
      group_lead[off] = 0;
      // the first particle of a cell always starts a leaf
      const int cp = i > 0 ? (int)(keys[i - 1] >> KEY_MORTON_BITS) : -1;
      for (int cc = cp + 1; cc <= c; cc++) cell_leaf_start[cc] = (int32_t)off;
      off++;
    }
    pleaf[i] = (int32_t)off - 1;
    if (i == n - 1) {
      for (int cc = (int)(keys[i] >> KEY_MORTON_BITS) + 1; cc <= n_cells; cc++)
        cell_leaf_start[cc] = (int32_t)off;
      leaf_start[off] = n;
      ds->n_leaves = (int)off;
    }
  }
}

// Chunks: the leaves of a cell placed in the cell's octree by the Morton code
// of their first particles and split as the particles are split into leaves,
// with CHUNK leaves in place of leaf_max particles.  A chunk is then an octree
// node (or a run of consecutive sibling nodes) holding at most CHUNK leaves,
// so its box stays compact; runs of CHUNK consecutive leaves in Morton order
// can straddle the boundary of a large node and span a box far wider than
// their leaves.
__device__ void chunk_nodes(const unsigned long long *__restrict__ leaf_keys, int n_leaves,
                            uint8_t *__restrict__ lead, int b0, int nb) {
  const int stride = nb * blockDim.x;
  for (int b = (blockIdx.x - b0) * blockDim.x + (threadIdx.x & ~31); b < n_leaves; b += stride) {
    const int l = b + (threadIdx.x & 31);
    unsigned long long key = 0ull;
    int first_level = MORTON_BITS + 1;
    if (l < n_leaves) {
      key = leaf_keys[l];
      first_level = l > 0 ? common_level(key, leaf_keys[l - 1]) + 1 : 0;
    }
    split_nodes(leaf_keys, n_leaves, l, CHUNK, lead, key, first_level);
  }
}

// Work groups: the leaves of a cell taken in order, a new group whenever the
// next leaf would bring the group above WG_MAX particles.  A warp walks every
// nwarps-th cell (32 cells' ranges loaded at a time): the lanes hold the ends
// of 96 consecutive leaves (windows of 32, the third in flight; a group has at
// most 32 leaves), and one vote per group finds the first leaf that no longer
// fits (one thread walked a cell leaf by leaf before, twice: 120 us at 2.1M
// clustered particles, where a cell holds up to 1,500 leaves).
__device__ void group_marks(const int32_t *__restrict__ cell_leaf_start,
                            const int32_t *__restrict__ leaf_start, int n_cells,
                            uint8_t *__restrict__ lead, int b0, int nb) {
  const int lane = threadIdx.x & 31;
  const int nw = nb * (int)(blockDim.x >> 5);
  const int w0 = ((int)blockIdx.x - b0) * (int)(blockDim.x >> 5) + (int)(threadIdx.x >> 5);
  for (long long cb = w0; cb < n_cells; cb += 32ll * nw) {
    const long long c = cb + (long long)lane * nw;
    const int a = c < n_cells ? cell_leaf_start[c] : 0, b = c < n_cells ? cell_leaf_start[c + 1] : 0;
    const int first = b > a ? leaf_start[a] : 0;
    unsigned todo = __ballot_sync(FULL, b > a);
    while (todo) {
      const int q = __ffs(todo) - 1;
      todo &= todo - 1u;
      const int l0 = __shfl_sync(FULL, a, q), l1 = __shfl_sync(FULL, b, q);
      // ends of leaves wb + lane and wb + 32 + lane (past the cell: never fit)
      int wb = l0, s = l0, sv = __shfl_sync(FULL, first, q);
      auto window = [&](int l) { return l + lane < l1 ? leaf_start[l + lane + 1] : 0x7fffffff; };
      int e0 = window(wb), e1 = window(wb + 32), e2 = window(wb + 64);
      while (s < l1) {
        if (lane == 0) lead[s] = 1;
        // the first leaf from s on that ends more than WG_MAX particles after sv
        // (leaf s itself fits)
        const unsigned m0 = __ballot_sync(FULL, e0 - sv > WG_MAX);
        if (m0) {
          const int p = __ffs(m0) - 1;
          sv = __shfl_sync(FULL, e0, p - 1);
          s = wb + p;
        } else {
          // (in the next window: 32 leaves never fit one group and more)
          const int p = __ffs(__ballot_sync(FULL, e1 - sv > WG_MAX)) - 1;
          const int last0 = __shfl_sync(FULL, e0, 31);
          const int prev = __shfl_sync(FULL, e1, p > 0 ? p - 1 : 0);
          sv = p > 0 ? prev : last0;
          s = wb + 32 + p;
          wb += 32;
          e0 = e1;
          e1 = e2;
          e2 = window(wb + 64);
        }
      }
    }
  }
}

__global__ void __launch_bounds__(256)
    k_chunk_nodes(const unsigned long long *__restrict__ leaf_keys, uint8_t *__restrict__ chunk_lead,
                  const int32_t *__restrict__ cell_leaf_start,
                  const int32_t *__restrict__ leaf_start, int n_cells,
                  uint8_t *__restrict__ group_lead, int group_blocks, const DevState *ds) {
  if (build_stopped(ds)) return;
  if ((int)blockIdx.x < group_blocks)
    group_marks(cell_leaf_start, leaf_start, n_cells, group_lead, 0, group_blocks);
  else
    chunk_nodes(leaf_keys, ds->n_leaves, chunk_lead, group_blocks, (int)gridDim.x - group_blocks);
}

// Compaction of the chunks' and the work groups' marks in one pass over the
// leaves (both counts travel in one status word).
__global__ void __launch_bounds__(CT)
    k_chunk_emit(const int32_t *__restrict__ leaf_cell, const uint8_t *__restrict__ chunk_lead,
                 const uint8_t *__restrict__ group_lead, int n_cells, unsigned long long *status,
                 unsigned int *ticket, int32_t *__restrict__ chunk_leaf_start,
                 int32_t *__restrict__ chunk_cell, int32_t *__restrict__ cell_chunk_start,
                 int32_t *__restrict__ leaf_chunk, int32_t *__restrict__ group_leaf0,
                 int32_t *__restrict__ group_cell, DevState *ds, int limit) {
  __shared__ unsigned long long s_sums[33];
  __shared__ unsigned long long s_pre;
  __shared__ int s_tile, s_stop;
  const int n = ds->n_leaves;
  if (threadIdx.x == 0) {
    s_tile = (int)atomicAdd(ticket, 1u);
    s_stop = build_stopped(ds) || s_tile * TILE >= n ? 1 : 0;
  }
  __syncthreads();
  if (s_stop) return;
  const int tile = s_tile;
  const int base = tile * TILE + (int)threadIdx.x * 8;
  unsigned int lc = 0u, lg = 0u;  // one bit per item
#pragma unroll
  for (int k = 0; k < 8; k++) {
    if (base + k >= n) break;
    lc |= chunk_lead[base + k] ? 1u << k : 0u;
    lg |= group_lead[base + k] ? 1u << k : 0u;
  }
  unsigned long long tot;
  const unsigned long long mine =
      (unsigned long long)__popc(lc) | ((unsigned long long)__popc(lg) << 31);
  unsigned long long off = block_exclusive<unsigned long long>(mine, s_sums, &tot);
  if (threadIdx.x < 32) {
    unsigned long long pre = 0ull;
    const bool ok = chain_prefix(status, tile, tot, &pre, ds, STALL_CHUNKS, limit);
    if (threadIdx.x == 0) {
      s_pre = pre;
      s_stop = ok ? 0 : 1;
    }
  }
  __syncthreads();
  if (s_stop) return;
  off += s_pre;
  int oc = (int)(off & 0x7fffffffull), og = (int)(off >> 31);
#pragma unroll
  for (int k = 0; k < 8; k++) {
    const int l = base + k;
    if (l >= n) break;
    const int c = leaf_cell[l];
    if ((lc >> k) & 1u) {
      chunk_leaf_start[oc] = l;
      chunk_cell[oc] = c;
      // the first leaf of a cell always starts a chunk
      const int cp = l > 0 ? leaf_cell[l - 1] : -1;
      for (int cc = cp + 1; cc <= c; cc++) cell_chunk_start[cc] = oc;
      oc++;
    }
    leaf_chunk[l] = oc - 1;
    if ((lg >> k) & 1u) {
      group_leaf0[og] = l;
      group_cell[og] = c;
      og++;
    }
    if (l == n - 1) {
      for (int cc = c + 1; cc <= n_cells; cc++) cell_chunk_start[cc] = oc;
      chunk_leaf_start[oc] = n;
      group_leaf0[og] = n;
      ds->n_chunks = oc;
      ds->n_groups = og;
    }
  }
}

// the structure of an empty set
__global__ void k_build_empty(DevState *ds, int32_t *leaf_start, int32_t *chunk_leaf_start,
                              int32_t *group_leaf0, int nc, double w) {
  leaf_start[0] = chunk_leaf_start[0] = group_leaf0[0] = 0;
  ds->nc = nc;
  ds->n_cells = nc * nc * nc;
  ds->w = w;
  ds->n_leaves = ds->n_chunks = ds->n_groups = 0;
  clear_queues(ds);
  ds->excursion_bits = ds->Hmax_bits = ds->want_h_bits = 0u;
  ds->group_cost_sum = 0ull;
  ds->m_uniform = 0.0f;
  for (int b = 0; b < MAX_BINS; b++) ds->bin_count[b] = 0;
}

inline int blocks_for(long long n, int t) { return (int)((n + t - 1) / t); }
inline int tiles_of(long long n) { return (int)((n + TILE - 1) / TILE); }
inline int passes_of(int nbits) { return (nbits + 7) / 8; }

// The sort's scratch: [tickets 7, one unused][totals 7 x 256][status rows 2 x tiles x 256]
// (a row's sectors whole: shifted by a word the passes of 913k pairs take 93 us, not 88)
struct SortWork {
  unsigned int *ticket, *totals, *row[2];
  size_t zero_words;  // from `ticket` on, zero before the keys are counted
};
SortWork sort_work(unsigned int *w, int n_tiles) {
  SortWork s;
  const size_t row = (size_t)n_tiles * RS_DIGITS;
  s.ticket = w;
  s.totals = w + RS_PASSES_MAX + 1;
  s.row[0] = s.totals + RS_PASSES_MAX * RS_DIGITS;
  s.row[1] = s.row[0] + row;
  s.zero_words = (size_t)(s.row[1] - w);
  return s;
}

// Whether one cluster sorts them (k_rs_cluster); most: what this device's
// clusters hold (cluster_sort_max).
inline bool cluster_sorts(int n, int nbits, int most) {
  return n <= most && nbits + RC_INDEX_BITS <= 64;
}

template <int BLOCKS, int ITEMS>
struct ClusterSort {
  static constexpr int HOLDS = BLOCKS * RC_THREADS * ITEMS;
  static constexpr int SMEM = 2 * RC_THREADS * ITEMS * (int)sizeof(unsigned long long);
  static_assert(HOLDS <= RC_MAX, "an index has 16 bits");
  // sets the kernel's attributes; whether the device can place such a cluster
  static bool prepare() {
    const auto kernel = k_rs_cluster<BLOCKS, ITEMS>;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = BLOCKS;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3(BLOCKS);
    c.blockDim = dim3(RC_THREADS);
    c.dynamicSmemBytes = SMEM;
    c.attrs = &at;
    c.numAttrs = 1;
    int clusters = 0;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM) == cudaSuccess &&
        (BLOCKS <= 8 ||
         cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) &&
        cudaOccupancyMaxActiveClusters(&clusters, kernel, &c) == cudaSuccess)
      return clusters > 0;
    cudaGetLastError();
    return false;
  }
  static cudaError_t launch(unsigned long long *keys, unsigned int *vals, int n, int nbits,
                            const unsigned int *bad, DevState *ds, cudaStream_t st) {
    note_launches(1);
    k_rs_cluster<BLOCKS, ITEMS>
        <<<BLOCKS, RC_THREADS, SMEM, st>>>(keys, vals, n, passes_of(nbits), bad, ds);
    return cudaGetLastError();
  }
};

// the smallest instance that holds n (rising order)
template <class F>
auto with_cluster_sort(int n, F f) {
  return n <= ClusterSort<8, 1>::HOLDS    ? f(ClusterSort<8, 1>())
         : n <= ClusterSort<16, 1>::HOLDS ? f(ClusterSort<16, 1>())
         : n <= ClusterSort<16, 2>::HOLDS ? f(ClusterSort<16, 2>())
         : n <= ClusterSort<16, 3>::HOLDS ? f(ClusterSort<16, 3>())
                                          : f(ClusterSort<16, 4>());
}

cudaError_t cluster_sort(unsigned long long *keys, unsigned int *vals, int n, int nbits,
                         const unsigned int *bad, DevState *ds, bool *result_in_alt,
                         cudaStream_t st) {
  *result_in_alt = false;
  return with_cluster_sort(n, [&](auto s) { return s.launch(keys, vals, n, nbits, bad, ds, st); });
}

// Every pass.  Of more pairs than one cluster sorts, the keys' digits have been
// counted; a pass clears the status row that the next one chains on.
cudaError_t sort_passes(unsigned long long *const keys[2], unsigned int *const vals[2], int n,
                        int nbits, const SortWork &s, bool *result_in_alt, unsigned int *fail,
                        const unsigned int *bad, DevState *ds, int limit, int cluster_most,
                        cudaStream_t st) {
  if (cluster_sorts(n, nbits, cluster_most))
    return cluster_sort(keys[0], vals[0], n, nbits, bad, ds, result_in_alt, st);
  const int passes = passes_of(nbits);
  note_launches(passes);
  for (int p = 0; p < passes; p++) {
    const int a = p & 1, b = a ^ 1;
    k_rs_pass<true><<<tiles_of(n), RS_THREADS, 0, st>>>(
        keys[a], p == 0 ? nullptr : vals[a], keys[b], vals[b], n, 8 * p, s.row[a], s.row[b],
        s.totals + p * RS_DIGITS, s.ticket + p, fail, bad, ds, limit);
  }
  *result_in_alt = (passes & 1) != 0;
  return cudaGetLastError();
}

}  // namespace

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
cudaError_t launch_reduce_hmax(const View &v, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(SPH_DS_FIELD(v.ds, build_hmax_bits), 0, sizeof(unsigned int), st);
  if (e != cudaSuccess || v.n == 0) return e;
  note_launches(1);
  int blocks = (int)std::min<long long>(1024, std::max<long long>(1, (v.n + 255) / 256));
  k_reduce_hmax<<<blocks, 256, 0, st>>>(v.h, v.n, SPH_DS_FIELD(v.ds, build_hmax_bits));
  return cudaGetLastError();
}

int cluster_sort_max() {
  int most = 0;
  while (most < RC_MAX) {
    // (the next instance up)
    const int holds = with_cluster_sort(most + 1, [](auto s) { return s.prepare() ? s.HOLDS : 0; });
    if (holds == 0) break;
    most = holds;
  }
  return most;
}

size_t order_work_words(long long n) {
  return (size_t)tiles_of(std::max<long long>(n, 1)) * RS_DIGITS;
}

cudaError_t radix_sort_indices(unsigned long long *keys, unsigned int *vals,
                               unsigned long long *keys_alt, unsigned int *vals_alt, int n,
                               int nbits, int cluster_most, unsigned int *work, bool *result_in_alt,
                               cudaStream_t st) {
  unsigned long long *const ks[2] = {keys, keys_alt};
  unsigned int *const vs[2] = {vals, vals_alt};
  if (cluster_sorts(n, nbits, cluster_most))
    return cluster_sort(ks[0], vs[0], n, nbits, nullptr, nullptr, result_in_alt, st);
  // (7 passes: 4,096 keys 78 us, with the look-back 86; 20,000 107 and 98; 65,536 119 and 108)
  const int passes = passes_of(nbits), tiles = tiles_of(n);
  note_launches(tiles > 1 ? 2 * passes : passes);
  for (int p = 0; p < passes; p++) {
    const int a = p & 1, b = a ^ 1;
    if (tiles > 1) k_rs_tile_counts<<<tiles, RS_THREADS, 0, st>>>(ks[a], n, 8 * p, work);
    k_rs_pass<false><<<tiles, RS_THREADS, 0, st>>>(ks[a], p == 0 ? nullptr : vs[a], ks[b], vs[b], n,
                                                   8 * p, work, nullptr, nullptr, nullptr, nullptr,
                                                   nullptr, nullptr, 0);
  }
  *result_in_alt = (passes & 1) != 0;
  return cudaGetLastError();
}

size_t build_work_words(long long n) {
  const long long t = tiles_of(std::max<long long>(n, 1));
  return 4 + 4 * (size_t)t + (RS_PASSES_MAX + 1 + RS_PASSES_MAX * RS_DIGITS) +
         2 * (size_t)t * RS_DIGITS;
}

cudaError_t launch_build(const View &v, const BuildArrays &b, int nc, double w, int n_cells,
                         long long n_perm, cudaStream_t st) {
  const int n = (int)v.n;
  cudaError_t e = cudaMemsetAsync(SPH_DS_FIELD(v.ds, build_bad), 0, BUILD_WORDS * sizeof(unsigned int), st);
  if (e != cudaSuccess) return e;
  if (n == 0) {
    for (int32_t *p : {v.cell_start, v.cell_leaf_start, v.cell_chunk_start})
      if (e == cudaSuccess) e = cudaMemsetAsync(p, 0, sizeof(int32_t) * ((size_t)n_cells + 1), st);
    if (e != cudaSuccess) return e;
    note_launches(1);
    k_build_empty<<<1, 1, 0, st>>>(v.ds, v.leaf_start, v.chunk_leaf_start, v.group_leaf0, nc, w);
    return cudaGetLastError();
  }
  const int n_tiles = tiles_of(n);
  // [tickets 4][leaf chain][chunk and group chain][sort]
  unsigned int *ticket = b.work;
  auto *leaf_chain = reinterpret_cast<unsigned long long *>(b.work + 4);
  unsigned long long *group_chain = leaf_chain + n_tiles;
  const SortWork s = sort_work(b.work + 4 + 4 * (size_t)n_tiles, n_tiles);
  e = cudaMemsetAsync(b.work, 0, (4 + 4 * (size_t)n_tiles + s.zero_words) * sizeof(unsigned int), st);
  if (e != cudaSuccess) return e;
  int cell_bits = 1;
  while ((1LL << cell_bits) < n_cells) cell_bits++;
  const int nbits = KEY_MORTON_BITS + cell_bits;
  const int limit = v.wait_limit > 0 ? (int)std::max<long long>(v.wait_limit, POLL_MIN) : POLL_LIMIT;
  const int wide = 2 * v.grid_util;  // 8 blocks of 256 threads per SM
  note_launches(7);
  // (1024 / w = 1024 nc / box, rounded once more than a division by w would be:
  // inside the margin of axis_code)
  k_cell_keys<<<std::min(blocks_for(n, 256), v.grid_util), 256, 0, st>>>(
      v, nc, w, (double)(1 << MORTON_BITS) / w, b.keys[0], s.totals,
      cluster_sorts(n, nbits, b.cluster_most) ? 0 : passes_of(nbits));
  bool alt = false;
  unsigned int *const vals[2] = {b.vals[0], b.vals[1]};
  unsigned long long *const ks[2] = {b.keys[0], b.keys[1]};
  e = sort_passes(ks, vals, n, nbits, s, &alt, SPH_DS_FIELD(v.ds, build_fail),
                  SPH_DS_FIELD(v.ds, build_bad), v.ds, limit, b.cluster_most, st);
  if (e != cudaSuccess) return e;
  const unsigned long long *skeys = b.keys[alt ? 1 : 0];
  unsigned long long *leaf_keys = b.keys[alt ? 0 : 1];
  Fields f;
  unsigned long long *p8[PF8] = {
      (unsigned long long *)v.x, (unsigned long long *)v.y, (unsigned long long *)v.z,
      (unsigned long long *)v.ti_begin, (unsigned long long *)v.ti_end,
      (unsigned long long *)v.ti_drift};
  void *p4[PF4] = {v.m, v.vx, v.vy, v.vz, v.ax, v.ay, v.az, v.A, v.Adot, v.h, v.rho, v.f, v.P, v.c,
                   v.vsig, v.ngb_density, v.ngb_force, v.div_v, v.curl_v};
  for (int k = 0; k < PF8; k++) f.p8[k] = p8[k];
  for (int k = 0; k < PF4; k++) f.p4[k] = (unsigned int *)p4[k];
  f.bin = (uint8_t *)v.bin;
  f.records = b.scratch;
  // marks: of the particles, then of the leaves for the chunks and the groups
  uint8_t *lead = b.marks, *chunk_lead = b.marks + b.n_max, *group_lead = chunk_lead + b.n_max;
  k_pack<<<std::min(blocks_for(n, 256), wide), 256, 0, st>>>(v, f, b.perm, n_perm);
  k_unpack<<<std::min(blocks_for(n, 256), wide), 256, 0, st>>>(v, f, b.vals[alt ? 1 : 0], b.perm,
                                                               lead, nc, w);
  k_leaf_nodes<<<std::min(blocks_for(n, 256), wide), 256, 0, st>>>(skeys, n, n_cells, v.leaf_max,
                                                                   lead, v.cell_start, v.ds);
  k_leaf_emit<<<n_tiles, CT, 0, st>>>(skeys, lead, n, n_cells, leaf_chain, ticket, v.leaf_start,
                                      v.leaf_cell, v.leaf_k, v.cell_leaf_start, v.pleaf, leaf_keys,
                                      chunk_lead, group_lead, v.ds, limit);
  // (one half of the blocks splits the leaves' octrees, the other marks groups)
  const int gb = std::min(blocks_for(n_cells, 8), v.grid_util);
  k_chunk_nodes<<<gb + std::min(blocks_for(n, 256), v.grid_util), 256, 0, st>>>(
      leaf_keys, chunk_lead, v.cell_leaf_start, v.leaf_start, n_cells, group_lead, gb, v.ds);
  k_chunk_emit<<<n_tiles, CT, 0, st>>>(v.leaf_cell, chunk_lead, group_lead, n_cells, group_chain,
                                       ticket + 1, v.chunk_leaf_start, v.chunk_cell,
                                       v.cell_chunk_start, v.leaf_chunk, v.group_leaf0,
                                       v.group_cell, v.ds, limit);
  return cudaGetLastError();
}

}  // namespace sph
