// The three per-frame trees (vehicles, receivers, both merged) of up to
// kFrameTreesMax primitives, built together in four launches (one up to
// kSmallFrame: k_tree_small).  Same trees as
// the one-block, cooperative and device-wide builders of bvh.cu: the order by
// (Morton code, index), the radix tree over it, and boxes that are exact
// minima and maxima.
//
// At these sizes a build is a chain of latencies, not of work, so the steps
// are chosen to have none that wait on one another:
//  - The sorted position of a primitive is its bin's first position (bins of
//    the code's leading bits, counted while the codes are made) plus the
//    smaller keys of the bin, counted directly (k_tree_bins, k_tree_rank),
//    instead of sort passes with a barrier each.  One bin list serves all
//    three trees: the order of the merged tree, restricted to a class, is
//    that class's own.
//  - A node's box is the minimum and maximum over its range of leaves, read
//    from the aligned power-of-two blocks of k_tree_blocks, instead of a walk
//    from the leaves up with one atomic arrival per level.
// Measured, update replayed from a graph, against one-block (to 4096
// primitives) and cooperative builds on three streams: 1200 primitives 61 ->
// 29 us, 4000 124 -> 31, 15000 (the city) 109 -> 37, 32760 126 -> 54.
#include "bvh.cuh"
#include "lbvh.cuh"

namespace emrt {

namespace {

struct FrameTreesView {
  const float4 *veh_lo, *veh_hi, *rx;
  uint32_t V, R;                // vehicles, receivers: primitives 0..V-1, V..V+R-1
  const uint32_t *code, *slot;  // [V + R] Morton codes and places within their bins
  const uint32_t *count, *count_v;  // [kTreeBins] primitives, vehicles
  uint32_t *first, *first_v;    // [kTreeBins + 1] the same before a bin
  uint2 *member;                // [V + R] (code, primitive), bin by bin
  float4 *prims[3];             // leaves in order: vehicles (may be null), receivers, merged
  uint32_t *sorted[3];          // their codes in order
};

// Every block scans the bins' counts (8 bins a thread) and puts its own
// primitives into the bins' lists; block 0 keeps the scan for k_tree_rank.
constexpr int kBinsBlock = 512, kBinsPer = kTreeBins / kBinsBlock;
static_assert(kBinsPer == 8, "two 16-byte loads of each count a thread");
__global__ void __launch_bounds__(kBinsBlock) k_tree_bins(FrameTreesView T) {
  __shared__ uint32_t s_first[kTreeBins];
  __shared__ uint2 s_warp[kBinsBlock / 32];
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t c[kBinsPer], v[kBinsPer], sc = 0, sv = 0;
#pragma unroll
  for (int q = 0; q < kBinsPer / 4; q++) {
    const uint4 x = reinterpret_cast<const uint4 *>(T.count)[threadIdx.x * (kBinsPer / 4) + q];
    const uint4 y = reinterpret_cast<const uint4 *>(T.count_v)[threadIdx.x * (kBinsPer / 4) + q];
    c[4 * q] = x.x; c[4 * q + 1] = x.y; c[4 * q + 2] = x.z; c[4 * q + 3] = x.w;
    v[4 * q] = y.x; v[4 * q + 1] = y.y; v[4 * q + 2] = y.z; v[4 * q + 3] = y.w;
  }
#pragma unroll
  for (int q = 0; q < kBinsPer; q++) {
    sc += c[q];
    sv += v[q];
  }
  uint32_t ic = sc, iv = sv;
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t a = __shfl_up_sync(0xffffffffu, ic, o), b = __shfl_up_sync(0xffffffffu, iv, o);
    if (lane >= (uint32_t)o) {
      ic += a;
      iv += b;
    }
  }
  if (lane == 31) s_warp[warp] = make_uint2(ic, iv);
  __syncthreads();
  uint32_t bc = ic - sc, bv = iv - sv;
  for (uint32_t w = 0; w < warp; w++) {
    bc += s_warp[w].x;
    bv += s_warp[w].y;
  }
#pragma unroll
  for (int q = 0; q < kBinsPer; q++) {
    const uint32_t bin = threadIdx.x * kBinsPer + q;
    s_first[bin] = bc;
    if (blockIdx.x == 0) {
      T.first[bin] = bc;
      T.first_v[bin] = bv;
    }
    bc += c[q];
    bv += v[q];
  }
  if (blockIdx.x == 0 && threadIdx.x == kBinsBlock - 1) {
    T.first[kTreeBins] = bc;
    T.first_v[kTreeBins] = bv;
  }
  __syncthreads();
  const uint32_t p = blockIdx.x * kBinsBlock + threadIdx.x;
  if (p >= T.V + T.R) return;
  const uint32_t code = T.code[p];
  T.member[s_first[code >> kTreeBinShift] + T.slot[p]] = make_uint2(code, p);
}

// (code, primitive): equal codes are ordered by index
__device__ inline uint64_t order_key(uint2 m) { return (uint64_t)m.x << 32 | m.y; }

// One thread a list place (a warp's threads mostly share their bin, whose
// list they read together): smaller keys of the bin, of both classes and of
// its own, and the leaf written in its places.  A bin of more than kRankLong
// primitives (a crowd on one square) is not compared all with all: the block
// orders its own places of the bin, every member finds where it stands among
// them (8 steps) and is counted there, and a place's rank is the sum of the
// counts up to it.  Update with every receiver within 100 m: 4000 225 -> 42 us,
// 15000 770 -> 66, 32700 1650 -> 112 (spread over 2 km: 31, 37, 56); blocks of
// 128 places 155 at 32700, of 512 118.
constexpr int kRankBlock = 256;
constexpr uint32_t kRankLong = 256;
static_assert(kRankLong >= kRankBlock, "only the bins at a block's two ends can be long");
__global__ void __launch_bounds__(kRankBlock) k_tree_rank(FrameTreesView T) {
  __shared__ uint64_t s_own[kRankBlock], s_key[kRankBlock];
  __shared__ uint32_t s_hist[kRankBlock];
  const uint32_t n = T.V + T.R, i0 = blockIdx.x * kRankBlock, i = i0 + threadIdx.x;
  const bool live = i < n;
  const uint2 me = T.member[min(i, n - 1u)];
  const uint32_t p = me.y, bin = me.x >> kTreeBinShift;
  const bool veh = p < T.V;
  const uint32_t b0 = T.first[bin], b1 = T.first[bin + 1], v0 = T.first_v[bin];
  const float4 a = veh ? T.veh_lo[p] : T.rx[p - T.V], b = veh ? T.veh_hi[p] : a;
  // places before this one in its bin: all in the low half, vehicles in the high
  uint32_t rank = 0;
  static_assert(kFrameTreesMax < 65536u, "two counts a word");
  const bool is_long = live && b1 - b0 > kRankLong;
  if (live && !is_long) {
#pragma unroll 4
    for (uint32_t q = b0; q < b1; q++) {
      const uint2 m = T.member[q];
      if (order_key(m) < order_key(me)) rank += m.y < T.V ? 0x10001u : 1u;
    }
  }
  if (__syncthreads_or(is_long)) {
    s_own[threadIdx.x] = order_key(me);
    uint32_t done = 0xffffffffu;  // bin of the first round
    for (int end = 0; end < 2; end++) {
      const uint32_t e = T.member[end ? min(i0 + kRankBlock, n) - 1u : i0].x >> kTreeBinShift;
      const uint32_t e0 = T.first[e], e1 = T.first[e + 1];
      if (e == done || e1 - e0 <= kRankLong) continue;  // the same for the whole block
      done = e;
      const uint32_t q0 = max(e0, i0) - i0, q1 = min(e1, i0 + kRankBlock) - i0;
      const bool mine = live && bin == e;
      s_key[threadIdx.x] = ~0ull;
      s_hist[threadIdx.x] = 0u;
      __syncthreads();
      uint32_t at = 0;  // order among the block's own
      for (uint32_t q = q0; q < q1; q++) at += s_own[q] < s_own[threadIdx.x] ? 1u : 0u;
      if (mine) s_key[at] = s_own[threadIdx.x];
      __syncthreads();
      uint32_t first = 0;
#pragma unroll 4
      for (uint32_t q = e0 + threadIdx.x; q < e1; q += kRankBlock) {
        const uint2 m = T.member[q];
        const uint64_t k = order_key(m);
        const uint32_t one = m.y < T.V ? 0x10001u : 1u;
        uint32_t above = 0;  // own keys up to k, the last not counted
#pragma unroll
        for (uint32_t s = kRankBlock / 2; s; s >>= 1)
          if (s_key[above + s - 1] <= k) above += s;
        if (!above) {
          first += one;
        } else {
          if (s_key[above] <= k) above++;
          if (above < q1 - q0) atomicAdd(&s_hist[above], one);
        }
      }
      for (int o = 16; o; o >>= 1) first += __shfl_xor_sync(0xffffffffu, first, o);
      if ((threadIdx.x & 31) == 0 && first) atomicAdd(&s_hist[0], first);
      __syncthreads();
      if (mine)
        for (uint32_t q = 0; q <= at; q++) rank += s_hist[q];
      __syncthreads();
    }
  }
  if (!live) return;
  const uint32_t vehs = rank >> 16, all = rank & 0xffffu;
  const uint32_t own = veh ? v0 + vehs : b0 - v0 + all - vehs;
  const uint32_t mix = b0 + all;
  T.prims[2][2ull * mix] = make_float4(a.x, a.y, a.z, __uint_as_float(p));
  T.prims[2][2ull * mix + 1] = make_float4(b.x, b.y, b.z, 0.f);
  T.sorted[2][mix] = me.x;
  if (!veh) {
    T.prims[1][own] = make_float4(a.x, a.y, a.z, __uint_as_float(p - T.V));
    T.sorted[1][own] = me.x;
  } else if (T.prims[0]) {
    T.prims[0][2ull * own] = make_float4(a.x, a.y, a.z, __uint_as_float(p));
    T.prims[0][2ull * own + 1] = make_float4(b.x, b.y, b.z, 0.f);
    T.sorted[0][own] = me.x;
  }
}

// Boxes of aligned blocks of leaves: level l (1..kLevels) has ceil(n / 2^l)
// of them, two float4 (lo, hi) each, one level after the other.
constexpr int kLevels = 10;
constexpr int kBlocksBlock = 256;
constexpr uint32_t kBlocksLeaves = 1u << kLevels;  // leaves of a thread block

struct TreeView {       // one tree of the last two launches
  const float4 *prims;
  const uint32_t *sorted;
  float4 *blocks;
  float4 *nodes;
  uint32_t *leaf_parent;
  uint32_t n;
  uint32_t first;       // first thread block of the launch that serves it
  int points;           // 1: leaves are points (one float4), 0: boxes (two)
};
struct TreeSet {
  TreeView t[3];
};

struct LoHi {
  float3 lo, hi;
};
// Merging ignores NaN (fminf, fmaxf), so NaN is the box of nothing.
__device__ inline LoHi no_box() {
  const float q = __int_as_float(0x7fffffff);
  return LoHi{make_float3(q, q, q), make_float3(q, q, q)};
}
__device__ inline void merge(LoHi &a, const LoHi &b) {
  a.lo = make_float3(fminf(a.lo.x, b.lo.x), fminf(a.lo.y, b.lo.y), fminf(a.lo.z, b.lo.z));
  a.hi = make_float3(fmaxf(a.hi.x, b.hi.x), fmaxf(a.hi.y, b.hi.y), fmaxf(a.hi.z, b.hi.z));
}
__device__ inline LoHi leaf_of(const TreeView &t, uint32_t g) {
  LoHi b;
  if (t.points) {
    b.lo = b.hi = f3(t.prims[g]);
  } else {
    b.lo = f3(t.prims[2ull * g]);
    b.hi = f3(t.prims[2ull * g + 1]);
  }
  return b;
}
__device__ inline void put_block(const TreeView &t, uint32_t offset, int level, uint32_t i,
                                 const LoHi &b) {
  if (((uint64_t)i << level) >= t.n) return;
  t.blocks[2ull * (offset + i)] = make_float4(b.lo.x, b.lo.y, b.lo.z, 0.f);
  t.blocks[2ull * (offset + i) + 1] = make_float4(b.hi.x, b.hi.y, b.hi.z, 0.f);
}
__device__ inline LoHi shfl_box(const LoHi &b, int d) {
  LoHi r;
  r.lo = make_float3(__shfl_down_sync(0xffffffffu, b.lo.x, d), __shfl_down_sync(0xffffffffu, b.lo.y, d),
                     __shfl_down_sync(0xffffffffu, b.lo.z, d));
  r.hi = make_float3(__shfl_down_sync(0xffffffffu, b.hi.x, d), __shfl_down_sync(0xffffffffu, b.hi.y, d),
                     __shfl_down_sync(0xffffffffu, b.hi.z, d));
  return r;
}
// the tree a thread block of the launch serves (no dynamic indexing of the
// kernel's parameters)
__device__ inline TreeView tree_of(const TreeSet &S) {
  TreeView t = S.t[0];
  if (blockIdx.x >= S.t[1].first) t = S.t[1];
  if (blockIdx.x >= S.t[2].first) t = S.t[2];
  return t;
}

// Four leaves a thread (levels 1 and 2), a warp's 32 by shuffles (3-7), the
// block's eight warps by shuffles of the first (8-10): no step waits for
// another block.
__global__ void __launch_bounds__(kBlocksBlock) k_tree_blocks(TreeSet S) {
  __shared__ LoHi s_warp[kBlocksBlock / 32];
  const TreeView t = tree_of(S);
  const uint32_t base = (blockIdx.x - t.first) * kBlocksLeaves;
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t g = base + 4u * threadIdx.x;
  LoHi b[4];
#pragma unroll
  for (int q = 0; q < 4; q++) b[q] = g + q < t.n ? leaf_of(t, g + q) : no_box();
  merge(b[0], b[1]);
  merge(b[2], b[3]);
  uint32_t offset = 0;
  put_block(t, offset, 1, g / 2, b[0]);
  put_block(t, offset, 1, g / 2 + 1, b[2]);
  merge(b[0], b[2]);
  offset += (t.n + 1) >> 1;
  put_block(t, offset, 2, g / 4, b[0]);
  for (int l = 3; l <= 7; l++) {
    offset += (t.n + (1u << (l - 1)) - 1) >> (l - 1);
    const int d = 1 << (l - 3);
    merge(b[0], shfl_box(b[0], d));
    if ((lane & (2 * d - 1)) == 0) put_block(t, offset, l, g >> l, b[0]);
  }
  if (lane == 0) s_warp[warp] = b[0];
  __syncthreads();
  if (warp) return;
  b[0] = lane < kBlocksBlock / 32 ? s_warp[lane] : no_box();
  for (int l = 8; l <= kLevels; l++) {
    offset += (t.n + (1u << (l - 1)) - 1) >> (l - 1);
    const int d = 1 << (l - 8);
    merge(b[0], shfl_box(b[0], d));
    if (lane < kBlocksBlock / 32 && (lane & (2 * d - 1)) == 0)
      put_block(t, offset, l, (base >> l) + (lane >> (l - 7)), b[0]);
  }
}

// Boxes of leaves first..split and split + 1..last: the aligned blocks they
// are made of, at most two a level each and the run of the top level.  Both
// ranges go up the levels together and a level's loads are issued before its
// merges: the loads' latency is the time of this step.  at(level, i): box of
// block i of a level.
template <typename At>
__device__ inline void range_boxes(At at, int top, const NodeRange &r, LoHi &a, LoHi &b) {
  a = b = no_box();
  uint32_t l0 = r.first, r0 = r.split + 1, l1 = r.split + 1, r1 = r.last + 1;
  for (int level = 0; l0 < r0 || l1 < r1; level++) {
    if (level == top) {
      for (; l0 < r0; l0++) merge(a, at(level, l0));
      for (; l1 < r1; l1++) merge(b, at(level, l1));
      break;
    }
    const bool la = l0 < r0 && (l0 & 1u), ra = l0 + la < r0 && (r0 & 1u);
    const bool lb = l1 < r1 && (l1 & 1u), rb = l1 + lb < r1 && (r1 & 1u);
    const LoHi x = la ? at(level, l0) : no_box(), y = ra ? at(level, r0 - 1) : no_box();
    const LoHi z = lb ? at(level, l1) : no_box(), w = rb ? at(level, r1 - 1) : no_box();
    merge(a, x);
    merge(a, y);
    merge(b, z);
    merge(b, w);
    l0 = (l0 + 1) >> 1;
    r0 >>= 1;
    l1 = (l1 + 1) >> 1;
    r1 >>= 1;
  }
}

__device__ inline void put_boxes(float4 *n, const LoHi &a, const LoHi &b, float pad) {
  n[0] = make_float4(a.lo.x - pad, a.hi.x + pad, a.lo.y - pad, a.hi.y + pad);
  n[1] = make_float4(b.lo.x - pad, b.hi.x + pad, b.lo.y - pad, b.hi.y + pad);
  n[2] = make_float4(a.lo.z - pad, a.hi.z + pad, b.lo.z - pad, b.hi.z + pad);
}

// One thread an inner node: its range and split from the codes in shared
// memory, then the boxes of its two children.
constexpr int kNodesBlock = 256;
__global__ void __launch_bounds__(kNodesBlock) k_tree_nodes(TreeSet S, float pad) {
  extern __shared__ __align__(16) uint32_t s_codes[];
  const TreeView t = tree_of(S);
  {  // the tree's codes, 16 bytes at a time (arrays start and end on 16 bytes)
    const uint4 *in = reinterpret_cast<const uint4 *>(t.sorted);
    uint4 *out = reinterpret_cast<uint4 *>(s_codes);
#pragma unroll 4
    for (uint32_t k = threadIdx.x; k < (t.n + 3) / 4; k += kNodesBlock) out[k] = in[k];
  }
  __syncthreads();
  const uint32_t i = (blockIdx.x - t.first) * kNodesBlock + threadIdx.x;
  if (i + 1 >= t.n) return;
  const NodeRange r = hierarchy_node([](int q) { return s_codes[q]; }, (int)t.n, (int)i,
                                     t.nodes, t.leaf_parent);
  // the levels' offsets, in step with the level asked for (each level once)
  uint32_t offset = 0;
  int known = 1;
  auto at = [&](int level, uint32_t k) {
    if (level == 0) return leaf_of(t, k);
    for (; known < level; known++) offset += (t.n + (1u << known) - 1) >> known;
    return LoHi{f3(t.blocks[2ull * (offset + k)]), f3(t.blocks[2ull * (offset + k) + 1])};
  };
  LoHi a, b;
  range_boxes(at, kLevels, r, a, b);
  put_boxes(t.nodes + 4ull * i, a, b, pad);
}

// The same steps for a frame of up to kSmallFrame primitives, a block a tree
// with bins, lists, codes and boxes in shared memory: one launch instead of
// four (and no counts in the update), whose latencies are the time of a small
// frame's trees.  Update (graph / call by call): 16 primitives 22.7 -> 12.4 us /
// 34 -> 20, 1200 28.8 -> 26.7 / 40 -> 27, 2040 30.3 -> 32.9 / 43 -> 34; one
// block's own work is what bounds it there.
constexpr uint32_t kSmallBlock = 1024, kSmallPer = kSmallFrame / kSmallBlock;
constexpr uint32_t kSmallBoxes = 2 * kSmallFrame + 16;
struct SmallShared {
  uint32_t first[kTreeBins];
  uint2 member[kSmallFrame];
  uint32_t code[kSmallFrame];  // in order
  LoHi box[kSmallBoxes];       // level 0 (leaves), 1, ...
  uint32_t warp[32];
};
static_assert(kTreeBins == 4 * kSmallBlock, "four bins a thread");

// A bin of more than kSmallLong members: the block sorts all members (bitonic,
// 66 steps of 2048 keys, a warp's own 64 places without block barriers) instead
// of comparing the bin's with one another.  The sort adds 14 us to a 2048
// frame's 29, whatever the bins; bins of 200 add 8 by comparing (the line lies
// where the two meet), one bin of all 2000 added 154.
constexpr uint32_t kSmallLong = 256;
__device__ inline void sort_members(uint2 *member, uint32_t n) {
  uint32_t size = 2;
  while (size < n) size <<= 1;
  for (uint32_t i = threadIdx.x; i < size; i += kSmallBlock)
    if (i >= n) member[i] = make_uint2(0xffffffffu, 0xffffffffu);
  __syncthreads();
  for (uint32_t run = 2; run <= size; run <<= 1)
    for (uint32_t step = run >> 1; step; step >>= 1) {
      for (uint32_t t = threadIdx.x; t < size / 2; t += kSmallBlock) {
        const uint32_t i = 2 * t - (t & (step - 1)), k = i + step;
        const uint2 x = member[i], y = member[k];
        if ((order_key(x) > order_key(y)) == ((i & run) == 0)) {
          member[i] = y;
          member[k] = x;
        }
      }
      // steps up to 32 stay within the 64 places of a warp
      if (step > 32 || (step == 1 && run >= 64)) __syncthreads();
      else __syncwarp();
    }
  __syncthreads();
}

__global__ void __launch_bounds__(kSmallBlock) k_tree_small(FrameTreesView T, TreeSet S,
                                                            const float4 *bb, float pad) {
  extern __shared__ __align__(16) unsigned char s_raw[];
  SmallShared &s = *reinterpret_cast<SmallShared *>(s_raw);
  TreeView t = S.t[0];
  if (blockIdx.x == 1) t = S.t[1];
  if (blockIdx.x == 2) t = S.t[2];
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float4 *prims = blockIdx.x == 0 ? T.prims[0] : blockIdx.x == 1 ? T.prims[1] : T.prims[2];
  if (!t.n || !prims) return;
  // primitive e of this tree: its corners
  auto corners = [&](uint32_t e, float4 &a, float4 &b) {
    if (blockIdx.x == 0 || (blockIdx.x == 2 && e < T.V)) {
      a = T.veh_lo[e];
      b = T.veh_hi[e];
    } else {
      a = b = T.rx[blockIdx.x == 2 ? e - T.V : e];
    }
  };
#pragma unroll
  for (uint32_t q = 0; q < 4; q++) s.first[tid + q * kSmallBlock] = 0u;
  __syncthreads();
  uint32_t code[kSmallPer], slot[kSmallPer];
#pragma unroll
  for (uint32_t q = 0; q < kSmallPer; q++) {
    const uint32_t e = tid + q * kSmallBlock;
    if (e < t.n) {
      float4 a, b;
      corners(e, a, b);
      code[q] = frame_code_of(a, b, bb);
      slot[q] = atomicAdd(&s.first[code[q] >> kTreeBinShift], 1u);
    }
  }
  __syncthreads();
  bool sorts;  // some bin is long
  {  // bins' counts to first positions, four bins a thread
    const uint4 c = reinterpret_cast<const uint4 *>(s.first)[tid];
    const uint32_t sum = c.x + c.y + c.z + c.w;
    uint32_t incl = sum;
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= (uint32_t)o) incl += y;
    }
    if (lane == 31) s.warp[warp] = incl;
    sorts = __syncthreads_or(max(max(c.x, c.y), max(c.z, c.w)) > kSmallLong);
    uint32_t run = incl - sum;
    for (uint32_t w = 0; w < warp; w++) run += s.warp[w];
    reinterpret_cast<uint4 *>(s.first)[tid] =
        make_uint4(run, run + c.x, run + c.x + c.y, run + c.x + c.y + c.z);
  }
  __syncthreads();
#pragma unroll
  for (uint32_t q = 0; q < kSmallPer; q++) {
    const uint32_t e = tid + q * kSmallBlock;
    if (e < t.n) s.member[s.first[code[q] >> kTreeBinShift] + slot[q]] = make_uint2(code[q], e);
  }
  __syncthreads();
  if (sorts) sort_members(s.member, t.n);
  for (uint32_t i = tid; i < t.n; i += kSmallBlock) {
    const uint2 me = s.member[i];
    uint32_t at = i;
    if (!sorts) {
      const uint32_t bin = me.x >> kTreeBinShift;
      const uint32_t b0 = s.first[bin], b1 = bin + 1u < kTreeBins ? s.first[bin + 1u] : t.n;
      at = b0;
      for (uint32_t q = b0; q < b1; q++) at += order_key(s.member[q]) < order_key(me) ? 1u : 0u;
    }
    float4 a, b;
    corners(me.y, a, b);
    s.code[at] = me.x;
    s.box[at] = LoHi{f3(a), f3(b)};
    if (t.points) {
      prims[at] = make_float4(a.x, a.y, a.z, __uint_as_float(me.y));
    } else {
      prims[2ull * at] = make_float4(a.x, a.y, a.z, __uint_as_float(me.y));
      prims[2ull * at + 1] = make_float4(b.x, b.y, b.z, 0.f);
    }
  }
  __syncthreads();
  uint32_t below = 0, size = t.n;  // level under the one being made
  while (size > 1u) {
    const uint32_t up = (size + 1u) / 2u, made = below + size;
    for (uint32_t i = tid; i < up; i += kSmallBlock) {
      LoHi b = s.box[below + 2u * i];
      if (2u * i + 1u < size) merge(b, s.box[below + 2u * i + 1u]);
      s.box[made + i] = b;
    }
    __syncthreads();
    below = made;
    size = up;
  }
  for (uint32_t i = tid; i + 1u < t.n; i += kSmallBlock) {
    const NodeRange r = hierarchy_node([&](int q) { return s.code[q]; }, (int)t.n, (int)i, t.nodes,
                                       t.leaf_parent);
    uint32_t offset = 0;
    int known = 0;
    auto at = [&](int level, uint32_t k) {
      for (; known < level; known++) offset += (t.n + (1u << known) - 1u) >> known;
      return s.box[offset + k];
    };
    LoHi a, b;
    range_boxes(at, 31, r, a, b);
    put_boxes(t.nodes + 4ull * i, a, b, pad);
  }
}

}  // namespace

static uint32_t round4(uint32_t n) { return (n + 3u) & ~3u; }

cudaError_t frame_trees_alloc(FrameTreesBuf &b, uint32_t n) {
  frame_trees_free(b);
  if (n > kFrameTreesMax) n = kFrameTreesMax;  // larger frames take the other builders
  b.cap = n;
  // counts; codes, slots; first positions; member lists
  cudaError_t e = cudaMalloc((void **)&b.count, sizeof(uint32_t) * 2 * kTreeBins);
  if (!e) e = cudaMalloc((void **)&b.code, sizeof(uint32_t) * 2ull * n);
  if (!e) e = cudaMalloc((void **)&b.first, sizeof(uint32_t) * 2 * (kTreeBins + 1));
  if (!e) e = cudaMalloc((void **)&b.member, sizeof(uint2) * n);
  // sorted codes and block boxes (below n + kLevels a tree) of the three trees
  if (!e) e = cudaMalloc((void **)&b.sorted, sizeof(uint32_t) * (2ull * n + 12));
  if (!e) e = cudaMalloc((void **)&b.blocks, 2 * sizeof(float4) * (2ull * n + 3ull * (kLevels + 1)));
  return e;
}

void frame_trees_free(FrameTreesBuf &b) {
  cudaFree(b.count);
  cudaFree(b.code);
  cudaFree(b.first);
  cudaFree(b.member);
  cudaFree(b.sorted);
  cudaFree(b.blocks);
  b = FrameTreesBuf{};
}

cudaError_t frame_trees_build(const FrameTreesBuf &f, BVHBuf &veh, BVHBuf &rx, BVHBuf &mix,
                              const float4 *veh_lo, const float4 *veh_hi, uint32_t V,
                              bool vehicles, const float4 *rx_pos, uint32_t R,
                              const float4 *bbox, cudaStream_t s) {
  const uint32_t n = V + R;
  FrameTreesView T{};
  T.veh_lo = veh_lo;
  T.veh_hi = veh_hi;
  T.rx = rx_pos;
  T.V = V;
  T.R = R;
  T.code = f.code;
  T.slot = f.code + f.cap;
  T.count = f.count;
  T.count_v = f.count + kTreeBins;
  T.first = f.first;
  T.first_v = f.first + kTreeBins + 1;
  T.member = f.member;
  T.prims[0] = vehicles ? veh.prims : nullptr;
  T.prims[1] = rx.prims;
  T.prims[2] = mix.prims;
  T.sorted[2] = f.sorted;
  T.sorted[0] = f.sorted + round4(n);
  T.sorted[1] = T.sorted[0] + round4(V);
  if (vehicles) veh.n = V;
  rx.n = R;
  mix.n = n;
  if (n <= kSmallFrame) {
    TreeSet S{};
    BVHBuf *buf[3] = {&veh, &rx, &mix};
    for (int k = 0; k < 3; k++) {
      S.t[k].n = k == 0 ? (vehicles ? V : 0u) : k == 1 ? R : n;
      S.t[k].nodes = buf[k]->nodes;
      S.t[k].leaf_parent = buf[k]->leaf_parent;
      S.t[k].points = k == 1;
    }
    const cudaError_t e = cudaFuncSetAttribute(
        k_tree_small, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SmallShared));
    if (e) return e;
    emrt::note_launch(), k_tree_small<<<3, kSmallBlock, sizeof(SmallShared), s>>>(T, S, bbox, mix.pad);
    return cudaGetLastError();
  }
  emrt::note_launch(), k_tree_bins<<<ceil_div(n, kBinsBlock), kBinsBlock, 0, s>>>(T);
  emrt::note_launch(), k_tree_rank<<<ceil_div(n, kRankBlock), kRankBlock, 0, s>>>(T);
  TreeSet S{};
  BVHBuf *buf[3] = {&veh, &rx, &mix};
  float4 *blocks = f.blocks;
  uint32_t nodes_first[3], blocks_total = 0, nodes_total = 0, widest = 0;
  for (int k = 0; k < 3; k++) {
    TreeView &t = S.t[k];
    t.n = k == 0 ? (vehicles ? V : 0u) : k == 1 ? R : n;
    t.prims = buf[k]->prims;
    t.sorted = T.sorted[k];
    t.nodes = buf[k]->nodes;
    t.leaf_parent = buf[k]->leaf_parent;
    t.points = k == 1;
    t.blocks = blocks;
    t.first = blocks_total;
    nodes_first[k] = nodes_total;
    if (t.n < 2) t.n = 0;  // no inner node
    blocks += 2ull * (t.n + kLevels + 1);
    blocks_total += ceil_div(t.n, kBlocksLeaves);
    nodes_total += ceil_div(t.n, kNodesBlock);
    if (t.n > widest) widest = t.n;
  }
  if (!nodes_total) return cudaGetLastError();
  emrt::note_launch(), k_tree_blocks<<<blocks_total, kBlocksBlock, 0, s>>>(S);
  for (int k = 0; k < 3; k++) S.t[k].first = nodes_first[k];
  const size_t smem = sizeof(uint32_t) * round4(widest);
  // the attribute is the function's for all threads of the process: always the
  // largest size, so that no build lowers what another's launch needs
  const cudaError_t e = cudaFuncSetAttribute(k_tree_nodes, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)(sizeof(uint32_t) * kFrameTreesMax));
  if (e) return e;
  emrt::note_launch(), k_tree_nodes<<<nodes_total, kNodesBlock, smem, s>>>(S, mix.pad);
  return cudaGetLastError();
}

}  // namespace emrt
