// Device code shared by the LBVH builders: Morton codes and the nodes of the
// binary radix tree over sorted codes (Karras 2012, restated from the
// published algorithm).
#pragma once
#include "bvh.cuh"

namespace emrt {

__device__ inline uint64_t spread3(uint32_t v) {
  uint64_t x = v & 0x1fffffu;
  x = (x | x << 32) & 0x1f00000000ffffull;
  x = (x | x << 16) & 0x1f0000ff0000ffull;
  x = (x | x << 8) & 0x100f00f00f00f00full;
  x = (x | x << 4) & 0x10c30c30c30c30c3ull;
  x = (x | x << 2) & 0x1249249249249249ull;
  return x;
}

// Morton code (3 AB bits, AB <= 21 per axis) of p quantised in the cube
// spanned by the largest extent of the box (all axes share one scale), so
// that a flat scene is split along its long axes first instead of slicing it
// into thin horizontal slabs.  Equal codes are told apart by index in the
// hierarchy (delta), so coarse codes only cost tree quality.
template <int AB>
__device__ inline uint64_t morton_code(float3 p, const float4 *bb) {
  float4 lo = bb[0], hi = bb[1];
  float ext = fmaxf(fmaxf(hi.x - lo.x, hi.y - lo.y), fmaxf(hi.z - lo.z, 1e-6f));
  float q[3] = {(p.x - lo.x) / ext, (p.y - lo.y) / ext, (p.z - lo.z) / ext};
  uint32_t c[3];
  for (int k = 0; k < 3; k++)
    c[k] = (uint32_t)(fminf(fmaxf(q[k], 0.f), 1.f) * (float)((1u << AB) - 1u));
  return spread3(c[0]) << 2 | spread3(c[1]) << 1 | spread3(c[2]);
}
// Code bits per primitive kind: the static triangles (LBVH fallback) use 63;
// vehicle boxes and receiver points, rebuilt every frame, use 30 (2 m cells
// over a 2 km cube) so that their sort takes four passes instead of eight
constexpr int kMortonBitsTri = 21, kMortonBitsDyn = 10;
// Code of a per-frame primitive with corners a and b (a point: a = b).
__device__ inline uint32_t frame_code_of(float4 a, float4 b, const float4 *bb) {
  return (uint32_t)morton_code<kMortonBitsDyn>(
      make_float3(0.5f * (a.x + b.x), 0.5f * (a.y + b.y), 0.5f * (a.z + b.z)), bb);
}
// at[bin]++ for every calling lane, its place among them returned.  The lanes of
// the first lane's bin add together: in a crowd they are most of the warp, and
// atomics on one address complete one after the other (32k of them took 33 us).
// Finding every lane's peers (match) cost a spread frame 4 us.
__device__ inline uint32_t add_one(uint32_t *at, uint32_t bin) {
  const uint32_t lane = threadIdx.x & 31u, all = __activemask();
  const uint32_t lead = __ffs(all) - 1u;
  const uint32_t peers = __ballot_sync(all, bin == __shfl_sync(all, bin, lead));
  const bool together = peers >> lane & 1u;
  uint32_t place = 0;
  if (!together || lane == lead) place = atomicAdd(at + bin, together ? (uint32_t)__popc(peers) : 1u);
  const uint32_t base = __shfl_sync(all, place, lead);
  return together ? base + __popc(peers & ((1u << lane) - 1u)) : place;
}
// The code of primitive i kept and counted in its bin (f.count zero before).
__device__ inline void frame_code(const FrameTreesBuf &f, uint32_t i, bool vehicle, float4 a,
                                  float4 b, const float4 *bb) {
  const uint32_t code = frame_code_of(a, b, bb);
  f.code[i] = code;
  f.code[f.cap + i] = add_one(f.count, code >> kTreeBinShift);
  if (vehicle) add_one(f.count + kTreeBins, code >> kTreeBinShift);
}

// Inner node i in [0, n-2] of the radix tree over the sorted keys k: its
// children and their parent links; returns its range of leaves and the last
// leaf of its left child.
struct NodeRange {
  int first, last, split;
};
__device__ inline int leading_zeros(uint64_t v) { return __clzll(v); }
__device__ inline int leading_zeros(uint32_t v) { return __clz(v); }
template <typename KeyAt>
__device__ inline NodeRange hierarchy_node(KeyAt key, int n, int i, float4 *nodes,
                                           uint32_t *leaf_parent) {
  auto delta = [&](int a, int c) -> int {
    if (c < 0 || c >= n) return -1;
    const auto x = key(a), y = key(c);
    if (x == y) return 8 * (int)sizeof(x) + __clz(a ^ c);
    return leading_zeros(x ^ y);
  };
  int d = (delta(i, i + 1) - delta(i, i - 1)) >= 0 ? 1 : -1;
  int dmin = delta(i, i - d);
  int lmax = 2;
  while (delta(i, i + lmax * d) > dmin) lmax <<= 1;
  int l = 0;
  for (int t = lmax >> 1; t >= 1; t >>= 1)
    if (delta(i, i + (l + t) * d) > dmin) l += t;
  int j = i + l * d;
  int dnode = delta(i, j);
  int s = 0, t = l;
  do {
    t = (t + 1) >> 1;
    if (delta(i, i + (s + t) * d) > dnode) s += t;
  } while (t > 1);
  int gamma = i + s * d + min(d, 0);
  int left = min(i, j) == gamma ? ~gamma : gamma;
  int right = max(i, j) == gamma + 1 ? ~(gamma + 1) : gamma + 1;
  int *n3 = reinterpret_cast<int *>(nodes + 4ll * i + 3);
  n3[0] = left;
  n3[1] = right;
  n3[3] = 0;
  int code0 = 2 * i, code1 = 2 * i + 1;
  if (left < 0) leaf_parent[~left] = code0;
  else reinterpret_cast<int *>(nodes + 4ll * left + 3)[2] = code0;
  if (right < 0) leaf_parent[~right] = code1;
  else reinterpret_cast<int *>(nodes + 4ll * right + 3)[2] = code1;
  if (i == 0) n3[2] = -1;
  return NodeRange{min(i, j), max(i, j), gamma};
}

}  // namespace emrt
