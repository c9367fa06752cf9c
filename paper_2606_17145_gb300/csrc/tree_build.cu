// tree_build.cu -- K3 permute, K4 octree build.
//
// Nodes are stored level by level (level-major), each level in the order of
// the sorted keys, so the children of a node are a contiguous range of the
// next level.  A node is a maximal run of sorted keys sharing the top 3*level
// bits; it is split (level < 21, more than leaf_size members) into the runs
// of its 8 possible next digits.
//
// Topology without a pass per level.  With L_i the number of digits key i
// shares with key i - 1, and D_i the deepest level at which more than
// leaf_size keys around i share a prefix (the largest common prefix of two
// keys leaf_size apart with i between them), the nodes that start at key i are
// those of the levels L_i + 1 .. D_i + 1, and all but the deepest are split.  So
// one pass counts the nodes of each level per block, a scan over the blocks
// gives every node its index, and a second pass writes them.
//
// Moments: all leaves in one launch, then the split nodes from the deepest
// level up in one launch whose blocks wait for the level below (one block alone
// where the levels are small).  One thread serves one node and sums its
// children (or a leaf's particles) in FP64 in index order, so the result does
// not depend on scheduling.
//
// A launch and its gap cost 2 - 3 us: a launch per level and direction (46 in
// all) cost 180 us on 4096 particles, most of it for empty levels.  Whole force
// passes, build alone changed: 4096 particles 500 -> 294 us, 64^3 leapfrog step
// 1050 -> 887 us, 100,003-particle SPH 1.15 -> 0.96 ms.  At 2.1 M particles the
// kernels take 0.065 (permute), 0.024 (count), 0.005 (scan), 0.032 (fill), 0.049
// (leaves) and 0.073 ms (upward).
#include <cfloat>

#include "og_internal.cuh"

namespace og {


// The order of the walk groups.  A walk takes the groups with the most work
// first, so that no long group starts when the others are done.  Started in
// tree order, the SMs of a 90^3 clustered walk are busy 75 % of its time, and
// with 78 % of their warps.  Work follows the sources within reach, and grows
// with the group's own box (its targets then share fewer of them):
//   w = (particles in the 8 cells nearest a target) (box volume / mean volume)^(1/4),
// the count averaged over four targets of the group, cells of 4 to 8 mean
// spacings.  Groups are sorted by half octaves of w, in tree order within one
// (which keeps neighbours together).  Forward walk, ms, tree order / this
// order / sorted by measured time: 187,501 zoom particles 16.7 / 12.3 / 11.8,
// clustered 64^3 1.74 / 1.38 / 1.38, 90^3 4.62 / 3.52 / 3.21, 128^3 18.2 / 16.8 /
// 15.8; 128^3 lattice 2.52 / 2.51.  The box volume alone says little (18.2 ->
// 20.0 at 128^3): the heavy groups are those that lie between dense clumps.  In
// the FP64 walk, where the pairs are nearly all of the work, the count alone
// tells more (clustered 64^3 7.6 / 6.5 / 6.8 ms, 7.7 with the volume).  Whole
// octaves: zoom 13.7 ms; other powers of the volume from 0.2 to 0.3: zoom
// 14.0 - 12.3, 90^3 3.50 - 3.69.  (Every tile adding up all tiles' counts again
// made k_scan 0.32 ms of a 60 M-particle build; with their prefix sums 0.08.)

// Counts the particles per cell (consecutive particles of a cell together) and
// leaves each group's box volume in T.gorder.  Every lane of the warp calls it.
__device__ __forceinline__ void group_cells(const TreeDev& T, int64_t g, bool live, const float hi[3]) {
  const int lane = threadIdx.x & 31;
  const int N = 1 << T.cell_level;
  int cell = 0;
  float v = 1.0f;
#pragma unroll
  for (int c = 0; c < 3; ++c) {  // split parts are not negative: they order like their bits
    const uint32_t a = __reduce_min_sync(0xffffffffu, live ? __float_as_uint(hi[c]) : 0x7f800000u);
    const uint32_t b = __reduce_max_sync(0xffffffffu, live ? __float_as_uint(hi[c]) : 0u);
    v *= __uint_as_float(b) - __uint_as_float(a) + 1.1920929e-07f;
    cell = cell * N + min(max((int)(hi[c] * (float)N), 0), N - 1);
  }
  const int before = __shfl_up_sync(0xffffffffu, cell, 1);
  const uint32_t lives = __ballot_sync(0xffffffffu, live);
  const bool head = live && (lane == 0 || before != cell);
  const uint32_t heads = __ballot_sync(0xffffffffu, head);
  if (head) {
    const uint32_t after = heads & ~((2u << lane) - 1u);
    const int end = after ? __ffs(after) - 1 : __popc(lives);
    atomicAdd(&T.gcell[cell], end - lane);
  }
  if (lane == 0) T.gorder[0][g] = __float_as_int(v);
}

// The buckets of this block's kTopoThreads / 4 groups, four threads a group.
__device__ __forceinline__ void group_buckets(const TreeDev& T, int64_t block) {
  const int64_t g = (block * kTopoBlock + threadIdx.x) >> 2;
  const int N = 1 << T.cell_level;
  float cnt = 0.f;
  if (g < T.ngroups) {
    const int64_t k = min(g * kGroup + 4 + 8 * (threadIdx.x & 3), T.n - 1);
    const float4 p = T.pA[k];
    const float x[3] = {p.x, p.y, p.z};
    int c0[3], c1[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const int f = (int)(x[c] * (float)N + 0.5f);  // the nearest face: the cells on both sides of it
      c0[c] = (f + N - 1) & (N - 1);
      c1[c] = f & (N - 1);
    }
    int s = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i)
      s += T.gcell[((i & 4 ? c1[0] : c0[0]) * N + (i & 2 ? c1[1] : c0[1])) * N + (i & 1 ? c1[2] : c0[2])];
    cnt = (float)s;
  }
  cnt += __shfl_xor_sync(0xffffffffu, cnt, 1);
  cnt += __shfl_xor_sync(0xffffffffu, cnt, 2);
  if (g < T.ngroups && (threadIdx.x & 3) == 0) {
    const float v = __int_as_float(T.gorder[0][g]) * (float)T.ngroups;
    const float n2 = 2.0f * __log2f(cnt);  // half octaves
#pragma unroll
    for (int o = 0; o < 2; ++o) {
      const float w2 = o ? n2 : n2 + 0.5f * __log2f(v);
      const int bucket = (int)fminf(fmaxf(96.0f - w2, 0.0f), (float)(kBuckets - 1));
      T.gbucket[o][g] = (unsigned char)bucket;
      atomicAdd(&T.gtile[o][(g / kOrderTile) * kBuckets + bucket], 1);
    }
  }
}

// The buckets [32 q, 32 q + 32) of order o: their counts in the tiles before each
// tile, and in all (1024 threads: a warp's lanes are the buckets, its rows a
// 32nd of the tiles).
__device__ __forceinline__ void bucket_columns(const TreeDev& T, int o, int q) {
  __shared__ int s_sum[32][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int* col = T.gtile[o] + 32 * q + lane;
  const int64_t rows = (T.ntiles + 31) / 32;
  const int64_t t0 = min(w * rows, T.ntiles), t1 = min(t0 + rows, T.ntiles);
  int sum = 0;
#pragma unroll 8
  for (int64_t t = t0; t < t1; ++t) sum += col[t * kBuckets];
  s_sum[w][lane] = sum;
  __syncthreads();
  int at = 0;
  for (int ww = 0; ww < w; ++ww) at += s_sum[ww][lane];
  for (int64_t t = t0; t < t1; t += 8) {
    int c[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) c[u] = t + u < t1 ? col[(t + u) * kBuckets] : 0;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      if (t + u < t1) col[(t + u) * kBuckets] = at;
      at += c[u];
    }
  }
  if (w == 31) col[T.ntiles * kBuckets] = at;
}

// Order o of one tile's groups, kOrderTile threads.
__device__ __forceinline__ void group_places(const TreeDev& T, int64_t tile, int o) {
  __shared__ int s_at[kOrderTile / 32][kBuckets];
  __shared__ int s_base[kBuckets];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int i = lane; i < kBuckets; i += 32) s_at[w][i] = 0;
  const int64_t g = tile * kOrderTile + threadIdx.x;
  const int bucket = g < T.ngroups ? T.gbucket[o][g] : -1;
  if (w == 0) {  // exclusive scan of the buckets' totals, 4 a lane
    const int4 c = reinterpret_cast<const int4*>(T.gtile[o] + T.ntiles * kBuckets)[lane];
    const int sum = c.x + c.y + c.z + c.w;
    int x = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, d);
      if (lane >= d) x += y;
    }
    x -= sum;
    reinterpret_cast<int4*>(s_base)[lane] = make_int4(x, x + c.x, x + c.x + c.y, x + c.x + c.y + c.z);
  }
  __syncthreads();
  const uint32_t peers = __match_any_sync(0xffffffffu, bucket);
  if (bucket >= 0 && lane == __ffs(peers) - 1) s_at[w][bucket] = __popc(peers);
  __syncthreads();
  if (threadIdx.x < kBuckets) {
    int at = s_base[threadIdx.x] + T.gtile[o][tile * kBuckets + threadIdx.x];
    for (int i = 0; i < kOrderTile / 32; ++i) {
      const int c = s_at[i][threadIdx.x];
      s_at[i][threadIdx.x] = at;
      at += c;
    }
  }
  __syncthreads();
  if (bucket >= 0) T.gorder[o][s_at[w][bucket] + __popc(peers & ((1u << lane) - 1u))] = (int32_t)g;
}

__global__ void k_permute(BuildArgs A, BoxScale B) {
  const TreeDev& T = A.T;
  const double invL2 = B.invL * B.invL;
  // a warp's 32 particles are one walk group
  for (int64_t k0 = blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31); k0 < T.n;
       k0 += (int64_t)gridDim.x * blockDim.x) {
    const int64_t k = k0 + (threadIdx.x & 31);
    const bool live = k < T.n;
    const int32_t i = live ? A.order[k] : 0;
    double w[3];
    float hi[3] = {0.f, 0.f, 0.f}, lo[3];
    bool ok = true;
    if (live) {
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const double x = A.pos[3 * (int64_t)i + c];
        ok = ok && finite_bits(x);
        w[c] = wrap_coord(x, B);
        split_box(w[c], B, hi[c], lo[c]);
        T.x64[3 * k + c] = w[c];
      }
    }
    group_cells(T, k0 / kGroup, live, hi);
    if (!live) continue;
    const double m = A.mass[i];
    const double eps = A.eps ? A.eps[i] : A.eps_scalar;
    if (!(ok && positive_finite_bits(m) && positive_finite_bits(eps))) set_status(T.sb, ST_BADINPUT);
    const double h = 2.8 * eps;
    T.m64[k] = m;
    T.h64[k] = h;
    T.order[k] = i;
    // m / L^2 and (h / L)^2 in FP32.  For a power-of-two side with 2^-2e an
    // exact double (invL2 then equals it), m invL2 = m 2^-2e and
    // (h invL)^2 = (h h) 2^-2e wherever the FP32 result is normal, and the
    // rounding to FP32 is done on the integer pipe.
    const bool sq = B.pow2 && B.e >= -511 && B.e <= 537;
    float mw, h2;
    if (!(sq && d2f_scaled((uint64_t)__double_as_longlong(m), 2 * B.e, mw))) mw = (float)(m * invL2);
    const double hh = h * h;
    if (!(sq && d2f_scaled((uint64_t)__double_as_longlong(hh), 2 * B.e, h2))) {
      const double hb = h * B.invL;
      h2 = (float)(hb * hb);
    }
    if (!(mw <= FLT_MAX)) atomicOr(&T.sb->pad[kTreeWildMass], 1);
    T.pA[k] = make_float4(hi[0], hi[1], hi[2], mw);
    T.pB[k] = make_float4(lo[0], lo[1], lo[2], h2);
  }
}

constexpr int kTopoThreads = kTopoBlock;
constexpr int kMaxLeaf = 32;        // largest leaf_size

// Octal digits two 63-bit keys share from the top (0 .. 21).
__device__ __forceinline__ int common_digits(uint64_t a, uint64_t b) {
  const uint64_t x = a ^ b;
  return x == 0 ? kMaxLevel : (__clzll((long long)x) - 1) / 3;
}

// Levels [lo, hi] of the nodes that start at sorted key i of this block (none
// if lo > hi): all but the one at hi are split.  Every thread of the block calls
// it.  LEAF: leaf_size, or 0 for any.
template <int LEAF>
__device__ __forceinline__ void node_levels(const uint64_t* __restrict__ keys, int64_t n, int leaf_size, int64_t i0,
                                            short* s_far, int& lo, int& hi) {
  const int leaf = LEAF ? LEAF : leaf_size;
  // s_far[j]: digits shared by keys i0 - leaf + j and i0 + j
  for (int j = threadIdx.x; j < kTopoThreads + leaf; j += kTopoThreads) {
    const int64_t a = i0 - leaf + j, b = i0 + j;
    s_far[j] = (short)(a >= 0 && b < n ? common_digits(keys[a], keys[b]) : -1);
  }
  __syncthreads();
  const int64_t i = i0 + threadIdx.x;
  lo = 1;
  hi = 0;
  if (i < n) {
    // two at a time from the even place on; those outside the window, one on
    // either side at most, are left out of the first and the last pair
    const uint32_t* f = reinterpret_cast<const uint32_t*>(s_far) + (threadIdx.x >> 1);
    const int odd = threadIdx.x & 1, last = (odd + leaf) >> 1;
    uint32_t m = odd ? f[0] | 0x0000ffffu : f[0];
    if (last > 0) {
#pragma unroll
      for (int j = 1; j < last; ++j) m = __vmaxs2(m, f[j]);
      m = __vmaxs2(m, (odd + leaf) & 1 ? f[last] : f[last] | 0xffff0000u);
    } else if (((odd + leaf) & 1) == 0) {
      m |= 0xffff0000u;
    }
    const int deep = max((int)(short)(m & 0xffffu), (int)(short)(m >> 16));
    lo = i == 0 ? 0 : common_digits(keys[i - 1], keys[i]) + 1;
    hi = min(deep + 1, kMaxLevel);
  }
}

// Nodes of each level that start in this block's keys.  The levels of each key's
// go to T.leaf_of (until k_leaves fills it), which saves k_fill from finding
// them again (16.8 M keys, us: k_fill 447 -> 352).  The blocks after those of
// the keys find the groups' buckets.
template <int LEAF>
__global__ void __launch_bounds__(kTopoThreads) k_count(TreeDev T, const uint64_t* __restrict__ keys, int leaf_size) {
  __shared__ __align__(4) short s_far[kTopoThreads + kMaxLeaf + 2];
  __shared__ int s_cnt[kLevels];
  if (blockIdx.x >= T.nblk) {
    group_buckets(T, blockIdx.x - T.nblk);
    return;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) T.sb->magic = kMagicTree;
  if (threadIdx.x < kLevels) s_cnt[threadIdx.x] = 0;
  int lo, hi;
  const int64_t i0 = blockIdx.x * (int64_t)kTopoThreads, i = i0 + threadIdx.x;
  node_levels<LEAF>(keys, T.n, leaf_size, i0, s_far, lo, hi);
  if (i < T.n) T.leaf_of[i] = lo | hi << 8;
  // All that follows holds for sorted keys.  Of others the nodes' ranges still
  // lie inside the particles, but a node may be nobody's child.
  if (i > 0 && i < T.n && keys[i - 1] > keys[i]) set_status(T.sb, ST_TREELINK);
  for (int l = lo; l <= hi; ++l) atomicAdd(&s_cnt[l], 1);
  __syncthreads();
  if (threadIdx.x < kLevels) T.blk[threadIdx.x * T.nblk + blockIdx.x] = s_cnt[threadIdx.x];
}

// One block per level: exclusive scan of its counts over the blocks, in
// place, and the level's total.  The blocks after those do the same for the
// buckets of the groups.
constexpr int kScanThreads = 1024;
constexpr int kScanItems = 8;
constexpr int kScanBlocks = kLevels + 2 * (kBuckets / 32);
__global__ void __launch_bounds__(kScanThreads) k_scan(TreeDev T) {
  __shared__ int s_w[32];
  if (blockIdx.x >= kLevels) {
    bucket_columns(T, (blockIdx.x - kLevels) & 1, (blockIdx.x - kLevels) >> 1);
    return;
  }
  int* row = T.blk + blockIdx.x * T.nblk;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int carry = 0;
  for (int64_t b0 = 0; b0 < T.nblk; b0 += kScanThreads * kScanItems) {
    const int64_t i = b0 + threadIdx.x * kScanItems;
    int v[kScanItems], sum = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) v[k] = i + k < T.nblk ? row[i + k] : 0;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) sum += v[k];
    int x = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) s_w[w] = x;
    __syncthreads();
    int y = s_w[lane];  // the warps' sums, then those up to each warp
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int z = __shfl_up_sync(0xffffffffu, y, o);
      if (lane >= o) y += z;
    }
    const int before = __shfl_sync(0xffffffffu, y, (w + 31) & 31), all = __shfl_sync(0xffffffffu, y, 31);
    int at = carry + (w > 0 ? before : 0) + x - sum;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
      if (i + k < T.nblk) row[i + k] = at;
      at += v[k];
    }
    carry += all;
    __syncthreads();
  }
  if (threadIdx.x == 0) T.sb->level_cnt[blockIdx.x] = carry;
}

__device__ __forceinline__ int level_base(const StatusBlock* sb, int level) {
  int b = 0;
  for (int l = 0; l < level; ++l) b += sb->level_cnt[l];
  return b;
}

// First key from `end` on whose prefix is not pre (n if there is none), by a
// whole warp: probes at distances that double, then 32 at a time between the
// last one inside the run and the first outside it.
__device__ __forceinline__ int64_t run_end(const uint64_t* __restrict__ keys, int64_t n, int64_t end, uint64_t pre,
                                           int shift) {
  const int lane = threadIdx.x & 31;
  auto inside = [&](int64_t j) {  // how many of the lanes' probes, from the first on
    return __ffs(~__ballot_sync(0xffffffffu, j < n && (keys[j] >> shift) == pre)) - 1;
  };
  int in = inside(end + ((int64_t)1 << lane) - 1);
  if (in < 0) in = 32;
  if (in == 0) return end;
  // the run ends in [a, b]
  int64_t a = end + ((int64_t)1 << (in - 1)), b = min(n, end + ((int64_t)1 << in) - 1);
  while (a < b) {
    const int64_t step = (b - a + 31) >> 5;
    const int64_t j = a + lane * step;
    in = inside(j < b ? j : n);
    if (in < 0) in = 32;
    b = min(b, a + in * step);
    if (in > 0) a += (in - 1) * step + 1;
  }
  return a;
}

// Writes the nodes' ranges.  nchild and the parent links follow with the
// moments, where a node meets its children.  A warp lists the nodes that start
// at its 32 keys and takes 32 of them at a time: going through the levels with a
// lane per key left 3 lanes of 32 at work (16.8 M keys, us: 352 -> 314).  Runs that
// go on past the block are searched for by whole warps, a level each (314 -> 279,
// 259 with the levels' counts read once).
// The blocks after those of the keys write the walks' orders of the groups, one
// tile in one order each.
__global__ void __launch_bounds__(kTopoThreads) k_fill(TreeDev T, const uint64_t* __restrict__ keys) {
  constexpr int kWarps = kTopoThreads / 32;
  __shared__ uint32_t s_ends[kWarps][kLevels];  // keys at which a run of the level (and a node) starts
  __shared__ uint32_t s_here[kWarps][kLevels];  // keys at which a node of the level starts (the warp's levels)
  __shared__ int s_warp[kWarps][kLevels];       // their number, then the index of the warp's first
  __shared__ uint16_t s_list[kWarps][32];       // nodes: lane of the key | level << 8
  __shared__ int s_past[kLevels];               // where the level's last run in the block ends
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (blockIdx.x >= T.nblk) {
    group_places(T, (blockIdx.x - T.nblk) >> 1, (blockIdx.x - T.nblk) & 1);
    return;
  }
  const int64_t i0 = blockIdx.x * (int64_t)kTopoThreads, i = i0 + threadIdx.x;
  const int levels = i < T.n ? T.leaf_of[i] : 1;  // lowest level 1, highest 0: none
  const int c_l = lane < kLevels ? T.sb->level_cnt[lane] : 0;
  // index of this block's first node of level threadIdx.x
  int first = threadIdx.x < kLevels ? T.blk[threadIdx.x * T.nblk + blockIdx.x] - c_l : 0;
  const int top = 31 - __clz((int)__ballot_sync(0xffffffffu, c_l > 0));  // the last level there is
  if (w == 0) {
    int x = c_l;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    first += x;
  }
  const int lo = levels & 255, hi = levels >> 8;
  const bool any = lo <= hi;
  const int wlo = (int)__reduce_min_sync(0xffffffffu, (unsigned)(any ? lo : kLevels));
  const int whi = (int)__reduce_max_sync(0xffffffffu, (unsigned)(any ? hi + 1 : 0)) - 1;
  if (lane < kLevels) s_warp[w][lane] = 0;
  __syncwarp();
  for (int l = 0; l <= top; ++l) {
    const uint32_t e = __ballot_sync(0xffffffffu, any && lo <= l);
    if (lane == 0) s_ends[w][l] = e;
    if (l < wlo || l > whi) continue;
    const uint32_t h = __ballot_sync(0xffffffffu, l >= lo && l <= hi);
    if (lane == 0) {
      s_here[w][l] = h;
      s_warp[w][l] = __popc(h);
    }
  }
  __syncthreads();
  if (threadIdx.x < kLevels) {
#pragma unroll
    for (int ww = 0; ww < kWarps; ++ww) {
      const int c = s_warp[ww][threadIdx.x];
      s_warp[ww][threadIdx.x] = first;
      first += c;
    }
  }
  // the runs that go on past the block, a warp a level
  const int64_t past = min(i0 + kTopoThreads, T.n);
  for (int l = w + 1; l <= top; l += kWarps) {
    const bool starts = __any_sync(0xffffffffu, lane < kWarps && s_ends[lane & (kWarps - 1)][l] != 0u);
    if (!starts) continue;  // none of its nodes starts here
    const int64_t e = run_end(keys, T.n, past, keys[past - 1] >> (63 - 3 * l), 63 - 3 * l);
    if (lane == 0) s_past[l] = (int)e;
  }
  const int cnt = any ? hi - lo + 1 : 0;
  int off = cnt;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, off, o);
    if (lane >= o) off += y;
  }
  const int nodes = __shfl_sync(0xffffffffu, off, 31);
  off -= cnt;
  __syncthreads();
  for (int b = 0; b < nodes; b += 32) {
    for (int k = max(b - off, 0); k < min(cnt, b + 32 - off); ++k)
      s_list[w][off + k - b] = (uint16_t)(lane | (lo + k) << 8);
    __syncwarp();
    const int e = b + lane < nodes ? s_list[w][lane] : 0;
    const int at = e & 31, l = e >> 8;  // key and level of this lane's node
    const bool leaf = l == __shfl_sync(0xffffffffu, hi, at);
    __syncwarp();
    if (b + lane >= nodes) break;
    const int64_t ki = i0 + 32 * w + at;
    const uint32_t before = (1u << at) - 1u;
    const int64_t p = (int64_t)s_warp[w][l] + __popc(s_here[w][l] & before);
    int64_t end = T.n;
    if (l > 0) {
      // The run ends at the next key that starts a run of level l.  A node
      // starts there too: the two keys' deepest common node is split, so the
      // first level at which they differ has one.  In this block the starts
      // are in s_ends.
      int ww = w;
      uint32_t next = at < 31 ? s_ends[w][l] & (0xfffffffeu << at) : 0u;
      while (next == 0u && ++ww < kWarps) next = s_ends[ww][l];
      end = next ? i0 + 32 * ww + __ffs(next) - 1 : s_past[l];
    }
    if (p < T.cap) {
      // the first child starts at the same key, one level down
      const int child = leaf ? -1 : s_warp[w][l + 1] + __popc(s_here[w][l + 1] & before);
      T.nD[p] = make_int4((int)ki, (int)(end - ki), child, make_meta(0, l, leaf));
      if (l == 0) T.nParent[p] = -1;
    } else {
      set_status(T.sb, ST_NOSPACE);
    }
  }
}

// A node's sums and everything derived from them: centre of mass, split FP32
// copies and cube centre.  On this GPU an FP64 warp instruction costs the same
// however many lanes are active, so each lane serves its own node (rather than
// one node spread over several lanes).
__device__ __forceinline__ void write_moments(const TreeDev& T, const BoxScale& B, int p, const int4& D, double M,
                                              double S0, double S1, double S2, double H) {
  const int lev = meta_level(D.w);
  const double side = ldexp(B.L, -lev);
  const float side_b = ldexpf(1.0f, -lev);
  const double invL = B.invL, invL2 = B.invL * B.invL;
  const double invM = 1.0 / M;
  const double com[3] = {S0 * invM, S1 * invM, S2 * invM};
  float hi[3], lo[3];
  double cen[3];
  float cenb[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    if (!(B.pow2 && split_bits((uint64_t)__double_as_longlong(com[c]), B.e, hi[c], lo[c])))
      split_coord(com[c] * invL, hi[c], lo[c]);
    const uint32_t q = quantise(T.x64[3 * (int64_t)D.x + c], B) >> (kMaxLevel - lev);
    // (q + 1/2) side, exact for a power-of-two box: (2q + 1) 2^(e - lev - 1)
    if (!(B.pow2 && double_odd_scaled(2u * q + 1u, B.e - lev - 1, cen[c]))) cen[c] = __dmul_rn((double)q + 0.5, side);
    cenb[c] = ((float)q + 0.5f) * side_b;
  }
  // M / L^2 and (hmax / L)^2 in FP32, as in k_permute
  const bool sq = B.pow2 && B.e >= -511 && B.e <= 537;
  float mw, h2;
  if (!(sq && d2f_scaled((uint64_t)__double_as_longlong(M), 2 * B.e, mw))) mw = (float)(M * invL2);
  const double HH = H * H;
  if (!(sq && d2f_scaled((uint64_t)__double_as_longlong(HH), 2 * B.e, h2))) {
    const double hb = H * invL;
    h2 = (float)(hb * hb);
  }
  T.mass64[p] = M;
  T.hmax64[p] = H;
  T.S64[3 * (int64_t)p] = S0;
  T.S64[3 * (int64_t)p + 1] = S1;
  T.S64[3 * (int64_t)p + 2] = S2;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    T.com64[3 * (int64_t)p + c] = com[c];
    T.cen64[3 * (int64_t)p + c] = cen[c];
  }
  if (!(mw <= FLT_MAX)) atomicOr(&T.sb->pad[kTreeWildMass], 1);
  T.nA[p] = make_float4(hi[0], hi[1], hi[2], mw);
  T.nB[p] = make_float4(lo[0], lo[1], lo[2], h2);
  T.nC[p] = make_float4(cenb[0], cenb[1], cenb[2], side_b);
}

// The leaves of all levels.  hmax as an integer max of the bit patterns:
// softenings are positive (checked by k_permute), and positive doubles order
// like their bits.
__global__ void __launch_bounds__(256) k_leaves(TreeDev T, BoxScale B) {
  const int total = level_base(T.sb, kLevels);
  if (total > T.cap) return;  // flagged by k_fill
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < total; p += gridDim.x * blockDim.x) {
    const int4 D = T.nD[p];
    if (!meta_leaf(D.w)) continue;
    double M = 0.0, S0 = 0.0, S1 = 0.0, S2 = 0.0;
    long long Hb = 0;
    for (int j = D.x; j < D.x + D.y; ++j) {
      const double m = T.m64[j];
      M += m;
      S0 += m * T.x64[3 * (int64_t)j];
      S1 += m * T.x64[3 * (int64_t)j + 1];
      S2 += m * T.x64[3 * (int64_t)j + 2];
      Hb = max(Hb, __double_as_longlong(T.h64[j]));
      T.leaf_of[j] = p;
    }
    write_moments(T, B, p, D, M, S0, S1, S2, __longlong_as_double(Hb));
  }
}

// A split node's moments from its children's.
constexpr int kUpThreads = 512;
__device__ __forceinline__ void node_moments(const TreeDev& T, const BoxScale& B, int p, int l, int total) {
  int4 D = T.nD[p];
  if (meta_leaf(D.w)) return;
  // the children's counts first (independent loads), which give their
  // number, then their sums: two memory latencies a level instead of one
  // a child (4096 particles: 28 -> 23 us)
  int nch = 0, left = D.y;
  int cy[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) cy[c] = D.z + c < total ? T.nD[D.z + c].y : 0;
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    if (left > 0) ++nch;
    left -= cy[c];
  }
  // children past the last node or more than eight: the keys are not sorted,
  // or not of 63 bits
  if (left > 0 || D.z + nch > total) {
    set_status(T.sb, ST_TREELINK);
    return;
  }
  double m8[8], s8[3][8], h8[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const int64_t q = D.z + (c < nch ? c : 0);
    m8[c] = T.mass64[q];
    s8[0][c] = T.S64[3 * q];
    s8[1][c] = T.S64[3 * q + 1];
    s8[2][c] = T.S64[3 * q + 2];
    h8[c] = T.hmax64[q];
  }
  double M = 0.0, S0 = 0.0, S1 = 0.0, S2 = 0.0;
  long long Hb = 0;
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    if (c < nch) {
      M += m8[c];
      S0 += s8[0][c];
      S1 += s8[1][c];
      S2 += s8[2][c];
      Hb = max(Hb, __double_as_longlong(h8[c]));
      T.nParent[D.z + c] = p;
    }
  }
  D.w = make_meta(nch, l, 0);
  T.nD[p] = D;
  write_moments(T, B, p, D, M, S0, S1, S2, __longlong_as_double(Hb));
}

// The split nodes, from the deepest level up, in parts (take_part) of
// nodes of one level.  The last part is the levels from the root on that have at
// most kUpThreads nodes each.
__global__ void __launch_bounds__(kUpThreads) k_upward(TreeDev T, BoxScale B) {
  __shared__ int s_split[kUpThreads / 32][64];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int part = take_part(T.sb);  // on its way while the levels are read
  int cnt[kLevels];
#pragma unroll
  for (int l = 0; l < kLevels; ++l) cnt[l] = T.sb->level_cnt[l];
  int total = 0, lone = -1;
#pragma unroll
  for (int l = 0; l < kLevels; ++l) {
    total += cnt[l];
    if (lone == l - 1 && cnt[l] <= kUpThreads) lone = l;
  }
  if (total > T.cap) return;  // flagged by k_fill
  int l = kLevels - 1, c_l = T.sb->level_cnt[l], base = total - c_l, parts = level_parts(c_l, kUpThreads);
  int first = 0;  // the level's first part: as many belong to the levels below
  int ready = 0;
  for (;; finish_part(T.sb), part = take_part(T.sb)) {
    part = share_part(part);
    while (l > lone && part - first >= parts) {
      first += parts;
      c_l = T.sb->level_cnt[--l];
      base -= c_l;
      parts = level_parts(c_l, kUpThreads);
    }
    if (l <= lone && part > first) return;
    if (first > ready) {
      if (!wait_parts(T.sb, first)) {
        if (threadIdx.x == 0) set_status(T.sb, ST_WALKCAP);
        return;
      }
      ready = first;
    }
    if (l > lone) {
      // a warp collects split nodes until there is one for every lane: taken as
      // they come, one lane in eight is at work, and FP64 instructions cost the
      // same for it (16.8 M clustered particles, us: 430 -> 358)
      int have = 0;
      for (int s0 = (part - first) * kUpThreads + (threadIdx.x & ~31); s0 < c_l; s0 += parts * kUpThreads) {
        const int s = s0 + lane;
        const bool split = s < c_l && !meta_leaf(T.nD[base + s].w);
        const uint32_t m = __ballot_sync(0xffffffffu, split);
        if (split) s_split[w][have + __popc(m & ((1u << lane) - 1u))] = base + s;
        have += __popc(m);
        __syncwarp();
        if (have >= 32) {
          have -= 32;
          node_moments(T, B, s_split[w][have + lane], l, total);
          __syncwarp();
        }
      }
      if (lane < have) node_moments(T, B, s_split[w][lane], l, total);
      continue;
    }
    for (;;) {
      if ((int)threadIdx.x < c_l) node_moments(T, B, base + threadIdx.x, l, total);
      if (l == 0) return;
      __threadfence_block();
      __syncthreads();
      c_l = T.sb->level_cnt[--l];
      base -= c_l;
    }
  }
}

cudaError_t launch_tree_build(const BuildArgs& A, cudaStream_t s) {
  const TreeDev& T = A.T;
  int64_t grid = (T.n + 255) / 256;
  if (grid > grid_cap(32)) grid = grid_cap(32);
  const BoxScale B = box_scale(A.L);
  k_permute<<<(unsigned)grid, 256, 0, s>>>(A, B);
  const int64_t gblocks = (4 * T.ngroups + kTopoThreads - 1) / kTopoThreads;
  const unsigned cblocks = (unsigned)(T.nblk + gblocks);
  if (A.leaf_size == 16) k_count<16><<<cblocks, kTopoThreads, 0, s>>>(T, A.keys, 16);  // the default
  else k_count<0><<<cblocks, kTopoThreads, 0, s>>>(T, A.keys, A.leaf_size);
  k_scan<<<kScanBlocks, kScanThreads, 0, s>>>(T);
  k_fill<<<(unsigned)(T.nblk + 2 * T.ntiles), kTopoThreads, 0, s>>>(T, A.keys);
  // the node counts live on the device: grids are sized for the particles
  int64_t lgrid = (T.n / 2 + 255) / 256;
  if (lgrid > grid_cap(8)) lgrid = grid_cap(8);
  if (lgrid < 1) lgrid = 1;
  k_leaves<<<(unsigned)lgrid, 256, 0, s>>>(T, B);
  int64_t ugrid = (T.n / 8 + kUpThreads - 1) / kUpThreads;
  if (ugrid > grid_cap(1)) ugrid = grid_cap(1);
  if (ugrid < 1) ugrid = 1;
  k_upward<<<(unsigned)ugrid, kUpThreads, 0, s>>>(T, B);
  return cudaGetLastError();
}

__global__ void k_copy_nodes(TreeDev T, int64_t m, int32_t* level, int32_t* first, int32_t* count, int32_t* parent,
                             double* mass, double* com, double* hmax, int32_t* child_first, int32_t* nchild) {
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < m; p += (int64_t)gridDim.x * blockDim.x) {
    const int4 D = T.nD[p];
    if (level) level[p] = meta_level(D.w);
    if (first) first[p] = D.x;
    if (count) count[p] = D.y;
    if (parent) parent[p] = T.nParent[p];
    if (mass) mass[p] = T.mass64[p];
    if (com)
      for (int c = 0; c < 3; ++c) com[3 * p + c] = T.com64[3 * p + c];
    if (hmax) hmax[p] = T.hmax64[p];
    if (child_first) child_first[p] = meta_leaf(D.w) ? -1 : D.z;
    if (nchild) nchild[p] = meta_leaf(D.w) ? 0 : meta_nchild(D.w);
  }
}

cudaError_t launch_copy_nodes(const TreeDev& T, int64_t m, int32_t* level, int32_t* first, int32_t* count,
                              int32_t* parent, double* mass, double* com, double* hmax, int32_t* child_first,
                              int32_t* nchild, cudaStream_t s) {
  if (m <= 0) return cudaSuccess;
  int64_t grid = (m + 255) / 256;
  if (grid > grid_cap(16)) grid = grid_cap(16);
  k_copy_nodes<<<(unsigned)grid, 256, 0, s>>>(T, m, level, first, count, parent, mass, com, hmax, child_first,
                                              nchild);
  return cudaGetLastError();
}

}  // namespace og
