// Path records after discovery: candidates to canonical order without
// duplicates, compaction of the kept ones, lookup in and merge into a path
// cache.
//
// A frame has some 1e4 candidates, so these steps are launches and latencies,
// not bytes; every launch taken out is 3-4 us.  The canonical order starts
// with the pair (tx, rx), and a pair holds few candidates, so instead of radix
// passes over a 128-bit key the candidates are counted per pair, put side by
// side in their pair's place and ordered there by counting, each thread
// reading its pair's list.  Duplicates stay in the list as records of no depth
// (kNoDepth), which acceptance passes over and the one compaction at the end
// leaves out: 9 launches from candidates to output where sorted keys, unique
// heads and two compactions took 28.  Measured with the launches that take the
// place of the merge's sort: district frame 691 -> 617 us, district cached
// frame about 575 -> 459, city cached frame 1065 -> 890.
#include "trace.cuh"

namespace emrt {

namespace {

constexpr int kPathsBlock = 256;
constexpr uint32_t kNoDepth = 15u;  // word 2 of a duplicate: no path has it

// Order of a record: (scene, tx), rx, depth, faces; faces past the depth do
// not count.
struct PathOrder {
  unsigned long long k0, k1, k2;
  uint32_t k3;
};
__device__ inline PathOrder order_of(uint4 a, uint4 b) {
  const uint32_t d = a.z & 15u;
  PathOrder o;
  o.k0 = (unsigned long long)a.x << 32 | a.y;
  o.k1 = (unsigned long long)d << 32 | (d > 0 ? a.w : 0u);
  o.k2 = (unsigned long long)(d > 1 ? b.x : 0u) << 32 | (d > 2 ? b.y : 0u);
  o.k3 = d > 3 ? b.z : 0u;
  return o;
}
__device__ inline PathOrder order_at(const uint32_t *rec, uint32_t i) {
  const uint4 *r = reinterpret_cast<const uint4 *>(rec + 8ull * i);
  return order_of(r[0], r[1]);
}
__device__ inline bool same(const PathOrder &a, const PathOrder &b) {
  return a.k0 == b.k0 && a.k1 == b.k1 && a.k2 == b.k2 && a.k3 == b.k3;
}
__device__ inline bool before(const PathOrder &a, const PathOrder &b) {
  if (a.k0 != b.k0) return a.k0 < b.k0;
  if (a.k1 != b.k1) return a.k1 < b.k1;
  if (a.k2 != b.k2) return a.k2 < b.k2;
  return a.k3 < b.k3;
}
// records of rec[0, n) before o
__device__ inline uint32_t lower_bound(const uint32_t *rec, uint32_t n, const PathOrder &o) {
  uint32_t lo = 0, hi = n;
  while (lo < hi) {
    const uint32_t mid = (lo + hi) >> 1;
    if (before(order_at(rec, mid), o)) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

// A receiver id past the frame's (a source list of backward discovery kept from
// a frame with more receivers) goes to the transmitter's last pair, behind that
// pair's own records in the order; acceptance rejects it.
__device__ inline uint32_t pair_of(const PairSpace &ps, uint32_t w0, uint32_t rx) {
  if (!ps.tab) return w0 * ps.per_tx + (min(rx, ps.n_rx - 1u) >> ps.shift);
  const BatchScene &t = ps.tab[w0 >> 8];
  return t.pair_begin + (w0 & 255u) * t.pair_rx + (rx >> ps.shift);
}

constexpr uint32_t kLeftOut = 0xffffffffu;  // place of a candidate left out

__device__ inline uint64_t slot_of(const PathOrder &o, uint64_t slots) {
  unsigned long long h = o.k0 * 0x9e3779b97f4a7c15ull;
  h = (h ^ (h >> 32) ^ o.k1) * 0xd6e8feb86659fd93ull;
  h = (h ^ (h >> 32) ^ o.k2) * 0x9e3779b97f4a7c15ull;
  h = (h ^ (h >> 32) ^ o.k3) * 0xd6e8feb86659fd93ull;
  return __umul64hi(h ^ (h >> 32), slots);
}

// Whether candidate i is the first of its path in the table; another lowers the
// first one's ray index.  The table has more slots than there are candidates.
__device__ inline bool first_met(uint32_t *cand, uint32_t i, uint32_t *table, uint64_t slots) {
  const PathOrder o = order_at(cand, i);
  uint64_t at = slot_of(o, slots);
  for (uint64_t k = 0; k < slots; k++) {
    uint32_t other = *reinterpret_cast<volatile uint32_t *>(table + at);
    if (!other) other = atomicCAS(table + at, 0u, i + 1u);
    if (!other) return true;
    const uint32_t c = other - 1u;
    if (same(order_at(cand, c), o)) {
      const uint32_t ray = cand[8ull * i + 7];
      if (ray < *reinterpret_cast<volatile uint32_t *>(cand + 8ull * c + 7))
        atomicMin(cand + 8ull * c + 7, ray);
      return false;
    }
    at = at + 1 == slots ? 0 : at + 1;
  }
  return true;
}

// Takes candidate i, a first one, out of the table.  Others are taken out at the
// same time, so an empty slot does not end the search.
__device__ inline void take_out(const uint32_t *cand, uint32_t i, uint32_t *table, uint64_t slots) {
  uint64_t at = slot_of(order_at(cand, i), slots);
  for (uint64_t k = 0; k < slots; k++) {
    uint32_t *t = table + at;
    if (*reinterpret_cast<volatile uint32_t *>(t) == i + 1u) {
      *t = 0u;
      return;
    }
    at = at + 1 == slots ? 0 : at + 1;
  }
}

// place of every candidate within its pair, in order of arrival; group[g]:
// candidates of pairs kPairGroup g .. kPairGroup (g + 1) - 1
__global__ void __launch_bounds__(kPathsBlock) k_pair_count(uint32_t *cand,
                                                            const uint32_t *n_cand, uint32_t cap,
                                                            PairSpace ps, PairBufs pb,
                                                            uint32_t *place, uint32_t *table,
                                                            uint64_t slots, Counters *ctr) {
  const uint32_t n = min(*n_cand, cap);
  uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0 && *n_cand > cap) atomicOr(&ctr->err, ERR_CAND_OVERFLOW);
  for (; i < n; i += gridDim.x * blockDim.x) {
    const uint32_t p = pair_of(ps, cand[8ull * i], cand[8ull * i + 1]);
    uint32_t at = atomicAdd(pb.count + p, 1u);
    if (at >= kPairLong)
      at = first_met(cand, i, table, slots) ? kPairLong + atomicAdd(pb.more + p, 1u) : kLeftOut;
    place[i] = at;
    if (at != kLeftOut) atomicAdd(pb.group + p / kPairGroup, 1u);
  }
}

// records of a pair's list
__device__ inline uint32_t list_length(const PairBufs &pb, uint32_t p, uint32_t count) {
  return count <= kPairLong ? count : kPairLong + pb.more[p];
}

// off[p] = records before pair p, off[n] and ctr->n_eff = all: a block scans one group of
// pairs, four a thread (16-byte loads; count is zero up to the next multiple
// of 4), after the sum of the groups before it.  One launch without a barrier:
// 40000 pairs in 3.0 us, 13.9 with one block scanning them all.
constexpr int kScanBlock = kPairGroup / 4;
__global__ void __launch_bounds__(kScanBlock) k_pair_scan(PairBufs pb, uint32_t n, Counters *ctr) {
  __shared__ uint32_t s_warp[kScanBlock / 32], s_base;
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t i = blockIdx.x * kScanBlock + threadIdx.x;  // of four pairs
  if (threadIdx.x == 0) s_base = 0;
  uint4 c = make_uint4(0u, 0u, 0u, 0u);
  if (4 * i < n) {
    c = reinterpret_cast<const uint4 *>(pb.count)[i];
    c.x = list_length(pb, 4 * i, c.x);
    c.y = list_length(pb, 4 * i + 1, c.y);
    c.z = list_length(pb, 4 * i + 2, c.z);
    c.w = list_length(pb, 4 * i + 3, c.w);
  }
  uint32_t before = 0;
  for (uint32_t g = threadIdx.x; g < blockIdx.x; g += kScanBlock) before += pb.group[g];
  const uint32_t sum = c.x + c.y + c.z + c.w;
  uint32_t incl = sum;
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= (uint32_t)o) incl += y;
  }
  for (int o = 16; o; o >>= 1) before += __shfl_xor_sync(0xffffffffu, before, o);
  if (lane == 31) s_warp[warp] = incl;
  __syncthreads();
  if (lane == 0) atomicAdd(&s_base, before);
  __syncthreads();
  uint32_t run = s_base + incl - sum;
  for (uint32_t w = 0; w < warp; w++) run += s_warp[w];
  if (4 * i >= n) return;
  reinterpret_cast<uint4 *>(pb.off)[i] = make_uint4(run, run + c.x, run + c.x + c.y, run + c.x + c.y + c.z);
  if (4 * i + 4 >= n) pb.off[n] = ctr->n_eff = run + sum;
}

__global__ void __launch_bounds__(kPathsBlock) k_pair_place(const uint32_t *cand,
                                                            const uint32_t *n_cand, uint32_t cap,
                                                            PairSpace ps, const uint32_t *off,
                                                            const uint32_t *place, uint32_t *lists,
                                                            uint32_t *table, uint64_t slots) {
  const uint32_t cnt = min(*n_cand, cap);
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < cnt; i += gridDim.x * blockDim.x) {
    const uint32_t at = place[i];
    if (at == kLeftOut) continue;
    const uint4 *r = reinterpret_cast<const uint4 *>(cand + 8ull * i);
    const uint4 a = r[0], b = r[1];
    uint4 *o = reinterpret_cast<uint4 *>(lists + 8ull * (off[pair_of(ps, a.x, a.y)] + at));
    o[0] = a;
    o[1] = b;
    if (at >= kPairLong) take_out(cand, i, table, slots);
  }
}

// The pair lists in canonical order: a record's position is the number of its
// list's records before it (equal ones by list position); of equal records the
// first gets the smallest ray index, the others become duplicates.
__global__ void __launch_bounds__(kPathsBlock) k_pair_order(const uint32_t *lists, const uint32_t *n,
                                                            PairSpace ps, const uint32_t *off,
                                                            uint32_t *out, Counters *ctr) {
  const uint32_t cnt = *n;
  uint32_t unique = 0;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < cnt; i += gridDim.x * blockDim.x) {
    const uint4 *r = reinterpret_cast<const uint4 *>(lists + 8ull * i);
    uint4 a = r[0], b = r[1];
    const PathOrder me = order_of(a, b);
    const uint32_t p = pair_of(ps, a.x, a.y), r0 = off[p], r1 = off[p + 1];
    uint32_t rank = 0, ray = b.w;
    bool dup = false;
#pragma unroll 2
    for (uint32_t q = r0; q < r1; q++) {
      const uint4 *s = reinterpret_cast<const uint4 *>(lists + 8ull * q);
      const uint4 c = s[0], d = s[1];
      const PathOrder it = order_of(c, d);
      if (same(it, me)) {
        ray = min(ray, d.w);
        if (q < i) {
          rank++;
          dup = true;
        }
      } else if (before(it, me)) {
        rank++;
      }
    }
    a.z = dup ? kNoDepth : a.z;
    b.w = ray;
    uint4 *o = reinterpret_cast<uint4 *>(out + 8ull * (r0 + rank));
    o[0] = a;
    o[1] = b;
    unique += dup ? 0u : 1u;
  }
  __syncwarp();
  for (int o = 16; o; o >>= 1) unique += __shfl_xor_sync(0xffffffffu, unique, o);
  if ((threadIdx.x & 31) == 0 && unique) atomicAdd(&ctr->n_unique, unique);
}

__device__ inline bool kept(const uint32_t *rec, uint32_t i, KeepWhich which) {
  const uint32_t w2 = rec[8ull * i + 2];
  if (which == KEEP_ALL) return true;
  if ((w2 & 15u) == kNoDepth) return false;
  return which == KEEP_PATHS || (w2 & EMRT_PATH_VALID);
}

// a block's share of the n records, a multiple of the block size
__device__ inline void share(uint32_t n, uint32_t &lo, uint32_t &hi) {
  uint32_t per = (n + gridDim.x - 1) / gridDim.x;
  per = (per + kPathsBlock - 1) / kPathsBlock * kPathsBlock;
  lo = min(n, blockIdx.x * per);
  hi = min(n, lo + per);
}

__global__ void __launch_bounds__(kPathsBlock) k_keep_count(const uint32_t *rec, const uint32_t *n,
                                                            KeepWhich which, uint32_t *partial) {
  __shared__ uint32_t s_sum;
  if (threadIdx.x == 0) s_sum = 0;
  __syncthreads();
  uint32_t lo, hi, sum = 0;
  share(*n, lo, hi);
  for (uint32_t i = lo + threadIdx.x; i < hi; i += kPathsBlock) sum += kept(rec, i, which) ? 1u : 0u;
  for (int o = 16; o; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if ((threadIdx.x & 31) == 0) atomicAdd(&s_sum, sum);
  __syncthreads();
  if (threadIdx.x == 0) partial[blockIdx.x] = s_sum;
}

// The kept records of a block's share, after those of the blocks before it
// (their counts summed here: at most kPrimGrid words).  pos (batches, may be
// null): kept records before each record, instead of writing them.
__global__ void __launch_bounds__(kPathsBlock) k_keep_write(const uint32_t *rec, const uint32_t *n,
                                                            KeepWhich which, const uint32_t *partial,
                                                            uint32_t *out, uint32_t cap,
                                                            uint32_t *pos, uint32_t *total,
                                                            uint32_t *count, Counters *ctr) {
  __shared__ uint32_t s_warp[kPathsBlock / 32], s_all[2];
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x < 2) s_all[threadIdx.x] = 0;
  __syncthreads();
  uint32_t mine = 0, all = 0;
  for (uint32_t b = threadIdx.x; b < gridDim.x; b += kPathsBlock) {
    const uint32_t c = partial[b];
    all += c;
    mine += b < blockIdx.x ? c : 0u;
  }
  for (int o = 16; o; o >>= 1) {
    mine += __shfl_xor_sync(0xffffffffu, mine, o);
    all += __shfl_xor_sync(0xffffffffu, all, o);
  }
  if (lane == 0) {
    atomicAdd(&s_all[0], mine);
    atomicAdd(&s_all[1], all);
  }
  __syncthreads();
  uint32_t base = s_all[0];
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    *total = s_all[1];
    if (count) *count = s_all[1];
    if (!pos && s_all[1] > cap) atomicOr(&ctr->err, ERR_PATH_OVERFLOW);
  }
  uint32_t lo, hi;
  share(*n, lo, hi);
  for (uint32_t r0 = lo; r0 < hi; r0 += kPathsBlock) {
    const uint32_t i = r0 + threadIdx.x;
    const bool keep = i < hi && kept(rec, i, which);
    const uint32_t m = __ballot_sync(0xffffffffu, keep);
    if (lane == 0) s_warp[warp] = __popc(m);
    __syncthreads();
    uint32_t at = base;
    for (uint32_t w = 0; w < kPathsBlock / 32; w++) {
      const uint32_t c = s_warp[w];
      at += w < warp ? c : 0u;
      base += c;
    }
    at += __popc(m & lanemask_lt());
    if (pos) {
      if (i < hi) pos[i] = at;
    } else if (keep && at < cap) {
      const uint4 *s = reinterpret_cast<const uint4 *>(rec + 8ull * i);
      uint4 *d = reinterpret_cast<uint4 *>(out + 8ull * at);
      d[0] = s[0];
      d[1] = s[1];
    }
    __syncthreads();
  }
}

// Kept, ordered records of a batch to each scene's output.  A scene's records
// start at the place of its first pair, so its kept ones are those between
// two scenes' starts.
__global__ void __launch_bounds__(kPathsBlock) k_batch_write(const BatchScene *tab, uint32_t n_scenes,
                                                             const uint32_t *rec, const uint32_t *n,
                                                             const uint32_t *off, uint32_t n_pairs,
                                                             const uint32_t *pos,
                                                             const uint32_t *total, Counters *ctr) {
  __shared__ uint32_t s_first[kBatchMaxScenes + 1];
  const uint32_t cnt = *n;
  for (uint32_t t = threadIdx.x; t <= n_scenes; t += kPathsBlock) {
    const uint32_t e = off[t < n_scenes ? tab[t].pair_begin : n_pairs];
    s_first[t] = e < cnt ? pos[e] : *total;
  }
  __syncthreads();
  const uint32_t t = blockIdx.x * kPathsBlock + threadIdx.x;
  if (t < n_scenes) {
    const uint32_t c = s_first[t + 1] - s_first[t];
    *tab[t].out_count = c;
    if (c > tab[t].out_cap) atomicOr(&ctr->err, ERR_PATH_OVERFLOW);
  }
  for (uint32_t i = t; i < cnt; i += gridDim.x * kPathsBlock) {
    if (!kept(rec, i, KEEP_VALID)) continue;
    const uint4 *src = reinterpret_cast<const uint4 *>(rec + 8ull * i);
    uint4 a = src[0];
    const uint4 b = src[1];
    const uint32_t sc = a.x >> 8, p = pos[i] - s_first[sc];
    if (p >= tab[sc].out_cap) continue;
    a.x &= 255u;
    uint4 *dst = reinterpret_cast<uint4 *>(tab[sc].out_rec + 8ull * p);
    dst[0] = a;
    dst[1] = b;
  }
}

// out = in, *n_out = records, min(*count, cap)
__global__ void __launch_bounds__(kPathsBlock) k_copy_paths(const uint32_t *in, const uint32_t *count,
                                                            uint32_t cap, uint32_t *out,
                                                            uint32_t *n_out) {
  const uint32_t cnt = min(*count, cap);
  uint32_t i = blockIdx.x * kPathsBlock + threadIdx.x;
  if (i == 0) *n_out = cnt;
  for (; i < cnt; i += gridDim.x * kPathsBlock) {
    const uint4 *s = reinterpret_cast<const uint4 *>(in + 8ull * i);
    uint4 *d = reinterpret_cast<uint4 *>(out + 8ull * i);
    d[0] = s[0];
    d[1] = s[1];
  }
}

// Candidates the cache already holds become duplicates; one that it holds as a
// valid path lowers that record's smallest ray index to its own (what merging
// the accepted candidate would have done; one candidate per record, so no two
// threads write the same word).  side (may be null): counters of the cache's
// revalidation on another stream, added to ctr.
__global__ void __launch_bounds__(kPathsBlock) k_known(uint32_t *cand, const uint32_t *n,
                                                       uint32_t *cache, const uint32_t *cache_n,
                                                       uint32_t cache_cap, const Counters *side,
                                                       Counters *ctr) {
  const uint32_t cnt = *n, nc = min(*cache_n, cache_cap);
  uint32_t i = blockIdx.x * kPathsBlock + threadIdx.x;
  if (i == 0 && side) {
    atomicOr(&ctr->err, side->err);
    ctr->occl_rays += side->occl_rays;
  }
  for (; i < cnt; i += gridDim.x * kPathsBlock) {
    uint32_t *c = cand + 8ull * i;
    if ((c[2] & 15u) == kNoDepth) continue;
    const PathOrder o = order_at(cand, i);
    const uint32_t at = lower_bound(cache, nc, o);
    if (at >= nc || !same(order_at(cache, at), o)) continue;
    uint32_t *h = cache + 8ull * at;
    if (h[2] & EMRT_PATH_VALID) h[7] = min(h[7], c[7]);
    c[2] = kNoDepth;
  }
}

// Merge of the cache's canonical records with the *n_new others (canonical,
// none of them in the cache) into out: a record goes to its own place plus the
// number of the other side's records before it.  Neighbours of the cache out
// of order raise ERR_UNSORTED.
__global__ void __launch_bounds__(kPathsBlock) k_merge_paths(const uint32_t *cache,
                                                             const uint32_t *cache_n,
                                                             uint32_t cache_cap, const uint32_t *fresh,
                                                             const uint32_t *n_new, uint32_t *out,
                                                             uint32_t out_cap, Counters *ctr) {
  const uint32_t nc = min(*cache_n, cache_cap), nn = *n_new;
  uint32_t i = blockIdx.x * kPathsBlock + threadIdx.x;
  if (i == 0) {
    ctr->n_accepted = min(nc + nn, out_cap);
    if (nc + nn > out_cap) atomicOr(&ctr->err, ERR_CAND_OVERFLOW);
  }
  for (; i < nc + nn; i += gridDim.x * kPathsBlock) {
    const bool old = i < nc;
    const uint32_t k = old ? i : i - nc;
    const uint4 *s = reinterpret_cast<const uint4 *>((old ? cache : fresh) + 8ull * k);
    const uint4 a = s[0], b = s[1];
    const PathOrder o = order_of(a, b);
    if (old && k > 0 && before(o, order_at(cache, k - 1))) atomicOr(&ctr->err, ERR_UNSORTED);
    const uint32_t p = k + lower_bound(old ? fresh : cache, old ? nn : nc, o);
    if (p >= out_cap) continue;
    uint4 *d = reinterpret_cast<uint4 *>(out + 8ull * p);
    d[0] = a;
    d[1] = b;
  }
}

// the merged records back into the cache (the first cap of them)
__global__ void __launch_bounds__(kPathsBlock) k_store_paths(const uint32_t *in, uint32_t *out,
                                                             uint32_t cap, uint32_t *count,
                                                             Counters *ctr) {
  const uint32_t n = ctr->n_accepted;
  uint32_t i = blockIdx.x * kPathsBlock + threadIdx.x;
  if (i == 0) {
    *count = n;
    if (n > cap) atomicOr(&ctr->err, ERR_PATH_OVERFLOW);
  }
  for (; i < min(n, cap); i += gridDim.x * kPathsBlock) {
    const uint4 *s = reinterpret_cast<const uint4 *>(in + 8ull * i);
    uint4 *d = reinterpret_cast<uint4 *>(out + 8ull * i);
    d[0] = s[0];
    d[1] = s[1];
  }
}

constexpr int kPathsGrid = 4 * 152;

}  // namespace

uint64_t pair_words(uint64_t n_pairs) {
  return 2 * ((n_pairs + 3) / 4 * 4) + (n_pairs + kPairGroup - 1) / kPairGroup;
}
PairBufs pair_bufs(uint32_t *count, uint32_t *off, uint64_t n_pairs) {
  const uint64_t n4 = (n_pairs + 3) / 4 * 4;
  return PairBufs{count, count + n4, count + 2 * n4, off};
}

void launch_dedup(uint32_t *cand, const uint32_t *n_cand, uint32_t cap, const PairSpace &ps,
                  const PairBufs &pb, uint32_t *lists, uint32_t *place, uint32_t *table,
                  Counters *ctr, cudaStream_t s) {
  const uint64_t slots = pair_slots(cap);
  emrt::note_launch(), k_pair_count<<<kPathsGrid, kPathsBlock, 0, s>>>(cand, n_cand, cap, ps, pb, place, table, slots,
                                                                     ctr);
  emrt::note_launch(), k_pair_scan<<<ceil_div(ps.n_pairs, kPairGroup), kScanBlock, 0, s>>>(pb, ps.n_pairs, ctr);
  emrt::note_launch(), k_pair_place<<<kPathsGrid, kPathsBlock, 0, s>>>(cand, n_cand, cap, ps, pb.off, place, lists,
                                                                     table, slots);
  emrt::note_launch(), k_pair_order<<<kPathsGrid, kPathsBlock, 0, s>>>(lists, &ctr->n_eff, ps, pb.off, cand, ctr);
}

void launch_keep(const uint32_t *rec, const uint32_t *n, KeepWhich which, uint32_t *out,
                 uint32_t cap, uint32_t *pos, uint32_t *total, uint32_t *count, Counters *ctr,
                 uint32_t *partial, cudaStream_t s) {
  emrt::note_launch(), k_keep_count<<<kPrimGrid, kPathsBlock, 0, s>>>(rec, n, which, partial);
  emrt::note_launch(), k_keep_write<<<kPrimGrid, kPathsBlock, 0, s>>>(rec, n, which, partial, out, cap, pos, total,
                                                                     count, ctr);
}

void launch_batch_write(const BatchScene *tab, uint32_t n_scenes, const uint32_t *rec,
                        const uint32_t *n, const uint32_t *off, uint32_t n_pairs,
                        const uint32_t *pos, const uint32_t *total, Counters *ctr,
                        cudaStream_t s) {
  emrt::note_launch(), k_batch_write<<<kPathsGrid, kPathsBlock, 0, s>>>(tab, n_scenes, rec, n, off, n_pairs, pos,
                                                                      total, ctr);
}

void launch_copy_paths(const uint32_t *in, const uint32_t *count, uint32_t cap, uint32_t *out,
                       uint32_t *n_out, cudaStream_t s) {
  emrt::note_launch(), k_copy_paths<<<kPathsGrid, kPathsBlock, 0, s>>>(in, count, cap, out, n_out);
}

void launch_known(uint32_t *cand, const uint32_t *n, uint32_t *cache, const uint32_t *cache_n,
                  uint32_t cache_cap, const Counters *side, Counters *ctr, cudaStream_t s) {
  emrt::note_launch(), k_known<<<kPathsGrid, kPathsBlock, 0, s>>>(cand, n, cache, cache_n, cache_cap, side, ctr);
}

void launch_merge_paths(uint32_t *cache, uint32_t *cache_n, uint32_t cache_cap,
                        const uint32_t *fresh, const uint32_t *n_new, uint32_t *tmp,
                        uint32_t tmp_cap, Counters *ctr, cudaStream_t s) {
  emrt::note_launch(), k_merge_paths<<<kPathsGrid, kPathsBlock, 0, s>>>(cache, cache_n, cache_cap, fresh, n_new, tmp,
                                                                      tmp_cap, ctr);
  emrt::note_launch(), k_store_paths<<<kPathsGrid, kPathsBlock, 0, s>>>(tmp, cache, cache_cap, cache_n, ctr);
}

}  // namespace emrt
