// keys_sort.cu -- K1 Peano-Hilbert keys and K2 stable LSD radix sort.
//
// K1: one thread per particle.  Position wrap and quantisation use explicitly
// rounded FP64 operations (no contraction) so the integer cell is a pure
// function of the input bits.  The 3-D Hilbert index follows Skilling's
// transpose construction (J. Skilling, "Programming the Hilbert curve", 2004):
// from the most significant bit down, the low bits of axis 0 are inverted or
// exchanged with those of axis i; the axes are then Gray-coded against one
// another and a running parity of the last axis is folded in.  Here the
// parity fold is a bit-parallel suffix XOR and the final interleave uses
// magic-mask bit spreading.  That is about 350 integer instructions a key, and
// bound the kernel (123 us at 5.0 M keys, 24 us of memory time), so where keys
// are counted for the passes the index is looked up instead, three levels of
// the curve at a time, in a 24 KB table of its 24 states: 57 us.
//
// K2: 8 passes of 8-bit digits (63-bit keys), one launch each.  K1 counts all
// eight digits' histograms while it writes the keys.  A pass ranks its tile's
// keys by digit with warp match masks, publishes the tile's digit counts, and
// finds the keys of equal digit in the tiles before it by looking back over
// their published counts (a tile publishes its own counts first and the sum
// up to itself once it knows it, so a look-back ends at the nearest sum);
// then it stages the tile in shared memory in digit order and writes
// contiguous runs.  (The scheme is the one-pass radix sort of Adinets and Merrill,
// 2022, on the look-back of Merrill and Garland, 2016.)  Tiles are numbered by a
// counter as blocks start, so every tile that is looked back at is running or
// done.  Stability of every pass gives the (key, original index) order.
//
// Bound by HBM: 220 B a key (32 for the keys, 20 for the first pass, whose
// values are the indices themselves, 24 for each other pass), against 310 B and 25
// launches for a histogram, a scan and a scatter per pass.
// Measured (keys and sort): 2.1 M 0.38 -> 0.24 ms, 5.0 M clustered 0.69 -> 0.41,
// 16.8 M 2.07 -> 1.14.  A pass takes 2.4 times its memory
// time at 16.8 M keys: a tile's chain of ranking, look-back and scattered writes
// is 12 us long and three tiles fit an SM.  Tile shapes, 5.0 M / 16.8 M, with the
// index computed bit by bit: 256 x 16 keys
// 0.481 / 1.38 ms, 256 x 12 0.488 / 1.43, 384 x 16 0.488 / 1.43, 512 x 8 0.52 / 1.57, 256 x 8
// 0.55 / 1.63; predecessors read at a time 4 / 8 / 16: 0.481 / 0.488 / 0.524 ms at 5.0 M.  Up to
// 262,144 keys a tile is 256 x 4 (sort_items).
#include "og_internal.cuh"

namespace og {

__device__ __forceinline__ uint64_t spread3(uint32_t v) {
  uint64_t x = v & 0x1fffffu;
  x = (x | (x << 32)) & 0x001f00000000ffffull;
  x = (x | (x << 16)) & 0x001f0000ff0000ffull;
  x = (x | (x << 8)) & 0x100f00f00f00f00full;
  x = (x | (x << 4)) & 0x10c30c30c30c30c3ull;
  x = (x | (x << 2)) & 0x1249249249249249ull;
  return x;
}

__device__ __forceinline__ uint64_t hilbert63(uint32_t a, uint32_t b, uint32_t c) {
#pragma unroll
  for (int bit = 20; bit >= 1; --bit) {
    const uint32_t top = 1u << bit;
    const uint32_t low = top - 1u;
    if (a & top) a ^= low;
    if (b & top) {
      a ^= low;
    } else {
      const uint32_t t = (a ^ b) & low;
      a ^= t;
      b ^= t;
    }
    if (c & top) {
      a ^= low;
    } else {
      const uint32_t t = (a ^ c) & low;
      a ^= t;
      c ^= t;
    }
  }
  b ^= a;
  c ^= b;
  // bit p of par = XOR of the bits of c at positions p+1 .. 20
  uint32_t par = (c & 0x1ffffeu) >> 1;
  par ^= par >> 1;
  par ^= par >> 2;
  par ^= par >> 4;
  par ^= par >> 8;
  par ^= par >> 16;
  a ^= par;
  b ^= par;
  c ^= par;
  return (spread3(a) << 2) | (spread3(b) << 1) | spread3(c);
}

constexpr int kKeyThreads = 256;

// The same index three levels at a time.  What the levels above leave behind
// is one of 24 states: which axis each of the three is exchanged with, which
// are inverted, and the parity.  e[512 s + (a, b, c)], three bits of each axis, is
// the next state << 9 | nine bits of the index.  Built from the steps of
// hilbert63 at compile time; states that give the same digits are one.
constexpr int kHilbertStates = 24;
struct alignas(16) HilbertTable {
  uint16_t e[kHilbertStates * 512];
  constexpr HilbertTable() : e() {
    int key[kHilbertStates] = {};    // the state's digits of the eight octants, 3 bits each
    int rep[kHilbertStates][7] = {};  // source axis of each axis, its inversion, parity
    int next[kHilbertStates][8] = {};
    int ns = 0;
    const int first[7] = {0, 1, 2, 0, 0, 0, 0};
    find(first, key, rep, ns);
    for (int s = 0; s < ns; ++s)
      for (int o = 0; o < 8; ++o) {
        int to[7] = {};
        step(rep[s], o, to);
        next[s][o] = find(to, key, rep, ns);
      }
    for (int s = 0; s < ns; ++s)
      for (int i = 0; i < 512; ++i) {
        int st = s, digits = 0;
        for (int b = 2; b >= 0; --b) {
          const int o = ((i >> (6 + b)) & 1) << 2 | ((i >> (3 + b)) & 1) << 1 | ((i >> b) & 1);
          digits = digits << 3 | ((key[st] >> (3 * o)) & 7);
          st = next[st][o];
        }
        e[512 * s + i] = (uint16_t)(st << 9 | digits);
      }
  }
  // One level of hilbert63 for the octant o: its digit and the state below.
  static constexpr int step(const int st[7], int o, int to[7]) {
    int v[3] = {};
    for (int x = 0; x < 3; ++x) v[x] = ((o >> (2 - st[x])) & 1) ^ st[3 + x];
    for (int x = 0; x < 7; ++x) to[x] = st[x];
    const int B = v[1] ^ v[0], C = v[2] ^ B;
    if (v[0]) to[3] ^= 1;
    for (int x = 1; x < 3; ++x) {
      if (v[x]) {
        to[3] ^= 1;
      } else {
        const int src = to[0], inv = to[3];
        to[0] = to[x];
        to[3] = to[3 + x];
        to[x] = src;
        to[3 + x] = inv;
      }
    }
    to[6] ^= C;
    return (v[0] << 2 | B << 1 | C) ^ (st[6] ? 7 : 0);
  }
  static constexpr int find(const int st[7], int* key, int (*rep)[7], int& ns) {
    int k = 0, unused[7] = {};
    for (int o = 0; o < 8; ++o) k |= step(st, o, unused) << (3 * o);
    for (int s = 0; s < ns; ++s)
      if (key[s] == k) return s;
    key[ns] = k;
    for (int x = 0; x < 7; ++x) rep[ns][x] = st[x];
    return ns++;
  }
};
__device__ const HilbertTable kHilbertTable;

__device__ __forceinline__ uint64_t hilbert63(const uint16_t* __restrict__ table, uint32_t a, uint32_t b,
                                              uint32_t c) {
  uint64_t key = 0;
  uint32_t st = 0;
#pragma unroll
  for (int bit = 18; bit >= 0; bit -= 3) {
    const uint32_t i = (((a >> bit) & 7u) << 6) | (((b >> bit) & 7u) << 3) | ((c >> bit) & 7u);
    const uint32_t e = table[(st & ~511u) | i];
    key = key << 9 | (e & 511u);
    st = e;
  }
  return key;
}

// Key of one position; 0 and the status flag for a non-finite one.
template <bool TABLE>
__device__ __forceinline__ uint64_t position_key(const double* __restrict__ pos, int64_t i, const BoxScale& B,
                                                 const uint16_t* table, StatusBlock* sb) {
  const double x0 = pos[3 * i], x1 = pos[3 * i + 1], x2 = pos[3 * i + 2];
  if (!(finite_bits(x0) && finite_bits(x1) && finite_bits(x2))) {
    set_status(sb, ST_BADINPUT);
    return 0;
  }
  const uint32_t a = quantise(wrap_coord(x0, B), B), b = quantise(wrap_coord(x1, B), B),
                 c = quantise(wrap_coord(x2, B), B);
  return TABLE ? hilbert63(table, a, b, c) : hilbert63(a, b, c);
}

// PASSES: also what the radix passes need, the digits' counts and clear tile counts.
template <bool PASSES>
__global__ void __launch_bounds__(kKeyThreads) k_keys(const double* __restrict__ pos, int64_t n, BoxScale B,
                                                      uint64_t* __restrict__ keys, SortWs W) {
  __shared__ uint32_t h[PASSES ? 8 * 256 : 1];
  __shared__ uint4 s_table[PASSES ? sizeof(HilbertTable) / sizeof(uint4) : 1];
  if (PASSES) {
    for (int i = threadIdx.x; i < 8 * 256; i += kKeyThreads) h[i] = 0u;
    for (int i = threadIdx.x; i < (int)(sizeof(HilbertTable) / sizeof(uint4)); i += kKeyThreads)
      s_table[i] = reinterpret_cast<const uint4*>(kHilbertTable.e)[i];
    __syncthreads();
  }
  const int64_t stride = (int64_t)gridDim.x * kKeyThreads;
  const int64_t first = blockIdx.x * (int64_t)kKeyThreads + threadIdx.x;
  // the first pass's tile counts start at zero
  if (PASSES)
    for (int64_t i = first; i < W.ntiles * 256; i += stride) W.tile_state[0][i] = 0u;
  for (int64_t i = first; i < n; i += stride) {
    const uint64_t key = position_key<PASSES>(pos, i, B, reinterpret_cast<const uint16_t*>(s_table), W.sb);
    keys[i] = key;
    if (PASSES) {
#pragma unroll
      for (int d = 0; d < 8; ++d) atomicAdd(&h[256 * d + ((key >> (8 * d)) & 255u)], 1u);
    }
  }
  if (PASSES) {
    __syncthreads();
    for (int i = threadIdx.x; i < 8 * 256; i += kKeyThreads)
      if (h[i]) atomicAdd(&W.hist[i], h[i]);
  }
}

// A tile's published state for one digit: 0 nothing yet, 1 + count its own
// count, kStateSum | sum the keys of the digit in all tiles up to it.  One
// word that other blocks poll while it is written, hence relaxed accesses of
// device scope (volatile, so that a tile publishes before it polls); nothing else is
// read on the strength of it.
constexpr uint32_t kStateSum = 1u << 31;
__device__ __forceinline__ uint32_t ld_relaxed(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ void st_relaxed(uint32_t* p, uint32_t v) {
  asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v));
}
// Polls of one state before a look-back gives up (seconds, far above any
// tile's run time; the tiles looked at are always running).
constexpr int kStatePolls = 1 << 22;
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kStateAhead = 4;

// Shared memory of a pass (dynamic: above the static limit).
template <int ITEMS>
struct SortSmem {
  uint64_t keys[kSortThreads * ITEMS];
  int32_t vals[kSortThreads * ITEMS];
  uint32_t wcnt[kSortWarps][256];
  uint32_t base[256];  // where the tile's first key of each digit goes, less its place in the tile
  unsigned long long scan[8];
  uint32_t tile;
};

template <bool FIRST, int ITEMS>
__global__ void __launch_bounds__(kSortThreads, ITEMS == 16 ? 3 : 6)
    k_sort_pass(const uint64_t* __restrict__ kin, const int32_t* __restrict__ vin, int64_t n, int pass, SortWs W,
                uint64_t* __restrict__ kout, int32_t* __restrict__ vout) {
  extern __shared__ __align__(16) unsigned char s_raw[];
  constexpr int kTile = kSortThreads * ITEMS;
  SortSmem<ITEMS>& S = *reinterpret_cast<SortSmem<ITEMS>*>(s_raw);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int shift = 8 * pass;
  if (threadIdx.x == 0) S.tile = (uint32_t)atomicAdd(&W.sb->pad[pass], 1);
  for (int i = threadIdx.x; i < kSortWarps * 256; i += kSortThreads) (&S.wcnt[0][0])[i] = 0u;
  __syncthreads();
  const int64_t tile = S.tile;
  const int64_t base = tile * kTile;
  const int tile_n = (int)((n - base) < kTile ? (n - base) : kTile);
  const int l0 = w * 32 * ITEMS + lane;  // this lane's first key of the tile

  uint64_t key[ITEMS];
  uint32_t place[ITEMS];
  const uint32_t lt = (1u << lane) - 1u;
  // padding slots lie behind every key of the tile: the largest digit keeps them last
#pragma unroll
  for (int k = 0; k < ITEMS; ++k) key[k] = l0 + 32 * k < tile_n ? kin[base + l0 + 32 * k] : ~0ull;
  // rank among the warp's keys of the same digit: the first of the 32 lanes
  // with the digit takes their number from the warp's counter; the rounds'
  // atomics go out in order and are not waited for between rounds
#pragma unroll
  for (int k = 0; k < ITEMS; ++k) {
    const uint32_t d = (uint32_t)((key[k] >> shift) & 255u);
    uint32_t peers = 0xffffffffu;
#pragma unroll
    for (int b = 0; b < 8; ++b) {
      const uint32_t v = __ballot_sync(0xffffffffu, (d >> b) & 1u);
      peers &= (d >> b) & 1u ? v : ~v;
    }
    const int first = __ffs(peers) - 1;
    uint32_t before = 0;
    if (lane == first) before = atomicAdd(&S.wcnt[w][d], (uint32_t)__popc(peers));
    __syncwarp();
    place[k] = __shfl_sync(0xffffffffu, before, first) + __popc(peers & lt);
  }
  __syncthreads();
  // thread d serves digit d: the warps' offsets inside the tile's run of the
  // digit, then one scan over the digits of (tile count, global count)
  const int d = threadIdx.x;
  uint32_t* state = W.tile_state[pass & 1];
  uint32_t cnt = 0;
  unsigned long long x = 0, own = 0;
  if (d < 256) {
    const uint32_t all = W.hist[256 * pass + d];
#pragma unroll
    for (int ww = 0; ww < kSortWarps; ++ww) {
      const uint32_t c = S.wcnt[ww][d];
      S.wcnt[ww][d] = cnt;
      cnt += c;
    }
    own = ((unsigned long long)cnt << 32) | all;
    if (d == 255) cnt -= (uint32_t)(kTile - tile_n);  // less the padding
    st_relaxed(&state[tile * 256 + d], tile == 0 ? (kStateSum | cnt) : cnt + 1u);
    if (pass < 7) W.tile_state[(pass + 1) & 1][tile * 256 + d] = 0u;  // the next pass's
    x = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) S.scan[w] = x;
  }
  __syncthreads();
  uint32_t tstart = 0, gbase = 0;
  if (d < 256) {
    for (int ww = 0; ww < w; ++ww) x += S.scan[ww];
    x -= own;
    tstart = (uint32_t)(x >> 32);
    gbase = (uint32_t)x;
#pragma unroll
    for (int ww = 0; ww < kSortWarps; ++ww) S.wcnt[ww][d] += tstart;
  }
  __syncthreads();
  // the tile in digit order
  int32_t val[ITEMS];
#pragma unroll
  for (int k = 0; k < ITEMS; ++k) {
    place[k] += S.wcnt[w][(key[k] >> shift) & 255u];
    S.keys[place[k]] = key[k];
  }
#pragma unroll
  for (int k = 0; k < ITEMS; ++k)
    val[k] = FIRST ? (int32_t)(base + l0 + 32 * k) : l0 + 32 * k < tile_n ? vin[base + l0 + 32 * k] : 0;
  // keys of this digit in the tiles before
  if (d < 256) {
    uint32_t sum = 0;
    if (tile > 0) {
      int64_t t = tile - 1;
      int polls = 0;
      for (;;) {
        // several predecessors at a time: their loads are independent
        uint32_t st[kStateAhead];
#pragma unroll
        for (int u = 0; u < kStateAhead; ++u) st[u] = t - u >= 0 ? ld_relaxed(state + (t - u) * 256 + d) : kStateSum;
        bool done = false;
        int used = 0;
#pragma unroll
        for (int u = 0; u < kStateAhead; ++u) {
          if (done || used < u || st[u] == 0u) continue;
          ++used;
          done = (st[u] & kStateSum) != 0u;
          sum += done ? st[u] & ~kStateSum : st[u] - 1u;
        }
        if (done) break;
        t -= used;
        if (used == 0 && ++polls > kStatePolls) {
          set_status(W.sb, ST_WALKCAP);
          break;
        }
      }
      st_relaxed(&state[tile * 256 + d], kStateSum | (sum + cnt));
    }
    S.base[d] = gbase + sum - tstart;
  }
#pragma unroll
  for (int k = 0; k < ITEMS; ++k) S.vals[place[k]] = val[k];
  __syncthreads();
#pragma unroll
  for (int k = 0; k < ITEMS; ++k) key[k] = S.keys[k * kSortThreads + threadIdx.x];
#pragma unroll
  for (int k = 0; k < ITEMS; ++k) val[k] = S.vals[k * kSortThreads + threadIdx.x];
#pragma unroll
  for (int k = 0; k < ITEMS; ++k) place[k] = S.base[(key[k] >> shift) & 255u] + (uint32_t)(k * kSortThreads + threadIdx.x);
#pragma unroll
  for (int k = 0; k < ITEMS; ++k) {
    if (k * kSortThreads + (int)threadIdx.x < tile_n && (int64_t)place[k] < n) {
      kout[place[k]] = key[k];
      vout[place[k]] = val[k];
    }
  }
}

// A small sort by counting: a key's place is the number of keys before it.  32
// keys a block (lane = key), which compare themselves with all keys, a chunk
// at a time from shared memory, each warp its share of the chunk.  n^2
// comparisons, but two launches and no pass after pass: 4096 keys 78 -> 18 us
// (host-bound), 8192 83 -> 28, 16,384 83 -> 63; at 20,000 the passes (82 us) catch up.
constexpr int kRankWarps = 16;
constexpr int kRankChunk = 4096;
constexpr int64_t kRankMax = 16384;
__global__ void __launch_bounds__(kRankWarps * 32) k_sort_rank(const uint64_t* __restrict__ keys, int n,
                                                               uint64_t* __restrict__ keys_out,
                                                               int32_t* __restrict__ order_out) {
  __shared__ __align__(16) uint64_t s_keys[kRankChunk];
  __shared__ int s_before[kRankWarps][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int i = blockIdx.x * 32 + lane;
  const uint64_t key = i < n ? keys[i] : 0;
  int before = 0;
  constexpr int kShare = kRankChunk / kRankWarps;
  for (int c0 = 0; c0 < n; c0 += kRankChunk) {
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kRankChunk; k += kRankWarps * 32) {
      const int j = c0 + k + threadIdx.x;
      s_keys[k + threadIdx.x] = j < n ? keys[j] : ~0ull;  // past the end: behind every key
    }
    __syncthreads();
    const ulonglong2* s = reinterpret_cast<const ulonglong2*>(s_keys + w * kShare);
    const int j0 = c0 + w * kShare, own = blockIdx.x * 32;
    // equal keys keep their order: those ahead of this block's keys count,
    // those behind do not, and in its own part the index decides
    if (j0 + kShare <= own) {
#pragma unroll 8
      for (int k = 0; k < kShare / 2; ++k) before += (s[k].x <= key ? 1 : 0) + (s[k].y <= key ? 1 : 0);
    } else if (j0 >= own + 32) {
#pragma unroll 8
      for (int k = 0; k < kShare / 2; ++k) before += (s[k].x < key ? 1 : 0) + (s[k].y < key ? 1 : 0);
    } else {
      for (int k = 0; k < kShare; ++k) {
        const uint64_t other = s_keys[w * kShare + k];
        before += other < key || (other == key && j0 + k < i) ? 1 : 0;
      }
    }
  }
  s_before[w][lane] = before;
  __syncthreads();
  if (w == 0 && i < n) {
    int at = 0;
#pragma unroll
    for (int ww = 0; ww < kRankWarps; ++ww) at += s_before[ww][lane];
    keys_out[at] = key;
    order_out[at] = i;
  }
}

template <int ITEMS>
static cudaError_t launch_sort_pass(const uint64_t* kin, const int32_t* vin, int64_t n, int pass, const SortWs& W,
                                    uint64_t* ko, int32_t* vo, cudaStream_t s) {
  auto kernel = pass == 0 ? k_sort_pass<true, ITEMS> : k_sort_pass<false, ITEMS>;
  const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)sizeof(SortSmem<ITEMS>));
  if (e != cudaSuccess) return e;
  kernel<<<(unsigned)W.ntiles, kSortThreads, sizeof(SortSmem<ITEMS>), s>>>(kin, vin, n, pass, W, ko, vo);
  return cudaGetLastError();
}

cudaError_t launch_keys_sort(const double* pos, int64_t n, double L, uint64_t* keys_out, int32_t* order_out,
                             const SortWs& W, cudaStream_t s) {
  // status, tile counters and histograms start at zero
  cudaError_t e = cudaMemsetAsync(W.sb, 0, kSortZeroBytes, s);
  if (e != cudaSuccess) return e;
  int64_t kgrid = (n + kKeyThreads - 1) / kKeyThreads;
  if (kgrid > grid_cap(4)) kgrid = grid_cap(4);  // each block copies the table: 8 an SM +2 us at 262,144 keys
  if (n <= kRankMax) {
    k_keys<false><<<(unsigned)kgrid, kKeyThreads, 0, s>>>(pos, n, box_scale(L), W.keys_alt, W);
    k_sort_rank<<<(unsigned)((n + 31) / 32), kRankWarps * 32, 0, s>>>(W.keys_alt, (int)n, keys_out, order_out);
    return cudaGetLastError();
  }
  k_keys<true><<<(unsigned)kgrid, kKeyThreads, 0, s>>>(pos, n, box_scale(L), keys_out, W);
  uint64_t* kin = keys_out;
  int32_t* vin = order_out;
  uint64_t* ko = W.keys_alt;
  int32_t* vo = W.vals_alt;
  const int items = sort_items(n);
  for (int pass = 0; pass < 8; ++pass) {
    e = items == 4 ? launch_sort_pass<4>(kin, vin, n, pass, W, ko, vo, s)
                   : launch_sort_pass<16>(kin, vin, n, pass, W, ko, vo, s);
    if (e != cudaSuccess) return e;
    uint64_t* tk = kin; kin = ko; ko = tk;
    int32_t* tv = vin; vin = vo; vo = tv;
  }
  return cudaGetLastError();
}

}  // namespace og

// ----------------------------------------------------------------------------
// og_keys_sort_noalloc: the same keys and sort with the workspace in a static
// device array instead of a caller buffer (declared in include/og.h).
#include <cmath>
#include <mutex>

namespace {

constexpr int64_t kNoAllocMaxN = int64_t(1) << 20;
constexpr size_t noalloc_round(size_t x) { return (x + og::kAlign - 1) / og::kAlign * og::kAlign; }
// Same carving as og::carve_sort: status block, histograms, alternate keys,
// alternate indices, two passes' tile counts.
constexpr size_t kNoAllocBytes =
    og::kSortZeroBytes + noalloc_round(sizeof(uint64_t) * kNoAllocMaxN) + noalloc_round(sizeof(int32_t) * kNoAllocMaxN) +
    2 * noalloc_round(sizeof(uint32_t) * 256 * og::sort_tiles_room(kNoAllocMaxN));

// Held by every GPU that loads the library, until the process exits.
static __device__ __align__(256) unsigned char g_noalloc_sort_ws[kNoAllocBytes];

constexpr int kNoAllocMaxDevices = 256;
std::mutex g_noalloc_mu;
void* g_noalloc_base[kNoAllocMaxDevices] = {};

}  // namespace

extern "C" og_status og_keys_sort_noalloc(const double* pos, int64_t n, double box, uint64_t* keys_sorted,
                                          int32_t* order, og_stream stream) {
  if (!pos || !keys_sorted || !order) return OG_EINVAL;
  if (n < 1 || !std::isfinite(box) || !(box > 0.0)) return OG_EINVAL;
  if (n > kNoAllocMaxN) return OG_ENOSPACE;
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kNoAllocMaxDevices) return OG_ECUDA;
  void* base = nullptr;
  {
    // First call on this device: look up the device address of the static
    // array (the host-side name is only a stand-in for it).
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    if (!g_noalloc_base[dev]) {
      void* p = nullptr;
      if (cudaGetSymbolAddress(&p, g_noalloc_sort_ws) != cudaSuccess || !p) return OG_ECUDA;
      g_noalloc_base[dev] = p;
    }
    base = g_noalloc_base[dev];
  }
  og::SortWs W;
  if (og::carve_sort(base, n, &W) > kNoAllocBytes) return OG_ENOSPACE;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  return og::launch_keys_sort(pos, n, box, keys_sorted, order, W, s) == cudaSuccess ? OG_OK : OG_ECUDA;
}
