// sph.cu -- SPH density and smoothing length on the device (declared in
// include/og.h: og_sph_ws_bytes / og_sph_density).
//
// The paper's SPH density module iterates each particle's smoothing length
// until its sphere holds a fixed number of neighbours, gathering the
// neighbours inside a sphere before evaluating them; its walks group nearby
// targets (Sec. 2, 2.1).  The reading is GADGET-2's: W is the cubic spline
// with support h, rho_i = sum_j m_j W(r_ij, h_i) (the particle itself
// included), and h_i is the root of the kernel-weighted count
// N_eff(h) = (4 pi / 3) h^3 sum_j W(r_ij, h) = (32 / 3) sum_j w(r_ij / h) = N_ngb.
//
// Grouped walk.  One warp serves a group of 32 Hilbert-consecutive targets, as
// in the gravity walk (two or four warps, each its part of the targets, where
// the groups do not fill the chip).  Each pass gathers, from one traversal of
// the tree (a range stack popped 32 nodes at a time), every leaf whose cube
// comes within R of the box of the targets still iterating (R their largest
// radius).  The leaves' particles are fetched 32 at a time, a particle beyond
// the reach of all four sub-groups of 8 targets is dropped, and the staged ones
// are evaluated by tiles of 8 targets x 8 particles.
//   1. Start: the density of the smallest ancestor of the target's leaf that
//      holds at least N_ngb particles gives h = (3 N_ngb / 4 pi n)^(1/3).
//   2. FP32 passes (k_sph_radius): third-order steps on ln h towards
//      ln N_eff(h) = ln N_ngb from sum w, sum q w' and sum q^2 w'', a bracket of
//      the root kept from every evaluation (a step leaving it is replaced by
//      the bracket's geometric mean) and steps clamped to a factor 2, until a
//      step below 2e-2 (taken, leaving ~6e-5).
//   3. Finishing pass (k_sph_density): the candidates within h (1 + 4e-4)
//      (FP32 test with a margin) are listed per target in shared memory, and
//      the lists are evaluated lane-parallel in float-float arithmetic on the
//      split-float positions (about 1e-11 relative in q; the FP64 pipe, 1/64
//      of FP32 on this GPU, keeps only the sums): sum w and sum m w in FP64;
//      sum q w' and sum m q w' (compensated FP32) and sum q^2 w'' and sum m q^2
//      w'' (FP32).  A second-order step in ln h from those sums gives h (error
//      ~20 d^3 for a step d; steps up to 3e-4 are accepted) and the density at
//      it; the neighbour count at the new h is the count at the evaluated one
//      corrected by the neighbours within 4e-4 h of it (their distances are
//      kept, up to two; with more, or a larger step, the pass is repeated at
//      the new h).
// Two kernels: the passes need 63 registers and 6.0 KB of shared memory a warp,
// the finishing pass 95 and 12.1 KB (17 warps an SM); in one kernel, of 126
// registers, the passes ran at 16 warps an SM.
//
// Measured, ms (one target per lane against every staged particle, Newton
// steps until 1e-2, one kernel of two warps a block -> now): 128^3 clustered
// N_ngb 32 24.9 -> 10.9; 128^3 lattice 5.05 -> 3.7; 4096 uniform 0.33 -> 0.20; 100,003
// uniform, N_ngb 64 0.73 -> 0.69.  By part on the clustered set: tiles 24.8 -> 19.8,
// two kernels 16.8, one warp a block 15.3, third-order steps 14.2, conversions on
// the integer pipe 13.6, groups by estimated work 10.9.  On a 90^3 clustered set
// k_sph_radius issues on 74 % of its cycles; k_sph_density (58 %) waits for
// latencies at 15 of 17 warps an SM and keeps the FP64 pipe 32 % busy.
// Every loop is bounded (node-visit cap, pass caps, the stack bound); a
// particle whose h does not converge below half the box gets NaN / -1 and
// sets a status bit.
#include <cmath>

#include "og_internal.cuh"

namespace og {

constexpr int kSphWarps = 1;          // warps per block
constexpr int kSphStack = 276;        // range stack entries (same bound as the gravity walk)
constexpr int kSphStackNeed = 32;     // pushes of one step
constexpr int kSphDeep = 64;          // above this depth a step pops a single range
static_assert(kSphDeep + 31 + 7 * 20 + 8 <= kSphStack - kSphStackNeed, "stack bound");
constexpr int kSphQueue = 128;        // queued leaves per warp
constexpr int kSphQueueNeed = 32;     // a step queues at most one leaf per popped node
constexpr int kSphList = 48;          // finishing pass: listed candidates per lane before a flush
constexpr int kSphPass32 = 32;        // FP32 Newton passes at most
constexpr int kSphPass64 = 8;         // finishing passes at most
// FP32 passes stop once a step on ln h is below this; the step is still taken,
// and its cubic convergence leaves an error of about 7 dl^3 ~ 6e-5, inside the
// 3e-4 step that the finishing pass accepts in one evaluation (at 3e-2 a 32^3
// clustered set needs a second one: 0.97 ms against 0.84).
constexpr float kSphConv32 = 2e-2f;
// The finishing pass lists neighbours within (1 + kSphBand) h and accepts a
// second-order step of up to kSphStep in ln h.
constexpr double kSphBand = 4e-4;
constexpr double kSphStep = 3e-4;

struct SphArgs {
  TreeDev T;
  StatusBlock* wsb;
  BoxScale B;
  double n_ngb;
  long long max_visits;  // node visits per gather
  int split;             // 2^split warps per group, each its part of the targets
  double* h_out;
  double* rho_out;
  int32_t* ngb_out;
};

// Minimum image of a box-unit difference t (|t| < 1.5): t - rint(t).
__device__ __forceinline__ float sph_round1(float t) { return __fadd_rn(__fadd_rn(t, 12582912.0f), -12582912.0f); }
__device__ __forceinline__ float sph_mi1(float t) { return __fadd_rn(t, -sph_round1(t)); }

// Packed pairs of floats.
__device__ __forceinline__ unsigned long long sph_pack(float lo, float hi) {
  return ((unsigned long long)__float_as_uint(hi) << 32) | __float_as_uint(lo);
}
__device__ __forceinline__ float sph_lo(unsigned long long a) { return __uint_as_float((uint32_t)a); }
__device__ __forceinline__ float sph_hi(unsigned long long a) { return __uint_as_float((uint32_t)(a >> 32)); }
__device__ __forceinline__ unsigned long long sph_add2(unsigned long long a, unsigned long long b) {
  unsigned long long d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ unsigned long long sph_mul2(unsigned long long a, unsigned long long b) {
  unsigned long long d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ unsigned long long sph_fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
  unsigned long long d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ float sph_rsqrt(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Compensated (Kahan) addition: the sum is T - C.  The _rn intrinsics keep
// the compiler from reassociating it away.
__device__ __forceinline__ void sph_kahan_add(float& T, float& C, float x) {
  const float y = __fsub_rn(x, C);
  const float t = __fadd_rn(T, y);
  C = __fsub_rn(__fsub_rn(t, T), y);
  T = t;
}

// Float-float arithmetic (a value is hi + lo, |lo| <= ulp(hi) / 2): the
// error-free sum and product of two floats (Knuth's two-sum; the product's
// error from one fused multiply-add) and the products and sums built on
// them, about 2^-46 relative.  The _rn intrinsics keep the compiler from
// contracting or reordering the steps.
struct FF {
  float hi, lo;
};
__device__ __forceinline__ FF ff_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}
__device__ __forceinline__ FF ff_quick(float a, float b) {  // |a| >= |b| (or a == 0)
  const float s = __fadd_rn(a, b);
  return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ FF ff_two_prod(float a, float b) {
  const float p = __fmul_rn(a, b);
  return {p, __fmaf_rn(a, b, -p)};
}
__device__ __forceinline__ FF ff_mul(const FF& a, const FF& b) {
  const FF p = ff_two_prod(a.hi, b.hi);
  return ff_quick(p.hi, __fmaf_rn(a.hi, b.lo, __fmaf_rn(a.lo, b.hi, p.lo)));
}
__device__ __forceinline__ FF ff_add(const FF& a, const FF& b) {
  const FF s = ff_two_sum(a.hi, b.hi);
  return ff_quick(s.hi, __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo)));
}
// max(c - q, 0) for c = 1 or 1/2
__device__ __forceinline__ FF ff_pos_diff(float c, const FF& q) {
  const FF d = ff_two_sum(c, -q.hi);
  const FF r = ff_quick(d.hi, __fsub_rn(d.lo, q.lo));
  return (r.hi > 0.f) ? r : FF{0.f, 0.f};
}

// Float -> double on the integer pipe (subnormals flush to zero): a conversion
// costs the FP64 pipe as much as an addition.
__device__ __forceinline__ double sph_f2d(float x) {
  const uint32_t u = __float_as_uint(x);
  const uint64_t b = (((uint64_t)(u & 0x7fffffffu) << 29) + (896ull << 52)) | ((uint64_t)(u >> 31) << 63);
  return (u & 0x7f800000u) == 0u ? 0.0 : __longlong_as_double((long long)b);
}

// Staged candidates: up to 64, two adjacent slots component by component so
// that one 16-byte load gives two packed (f32x2) operands, and behind them a
// pair far outside every sphere that pads the lists.
constexpr int kSphStage = 64;
constexpr int kSphFar = kSphStage / 2;  // index of the padding pair
struct SphStage {
  float4 s0[kSphFar + 1];  // -hi.x of both, -hi.y of both (nearest image to the group centre)
  float4 s1[kSphFar + 1];  // -hi.z, -lo.x
  float4 s2[kSphFar + 1];  // -lo.y, -lo.z
  int id[kSphStage];       // sorted index
  unsigned char sub[kSphStage];        // sub-groups within reach
  unsigned char list[4][kSphFar + 4];  // slot pairs of each sub-group
};

struct SphBufs {
  int* stack;
  int2* queue;
  int* qoff;        // [kSphQueue + 1] slot offsets of the queued leaves
  SphStage* St;
  float4* box;      // [8] per sub-group: centre and squared reach, half extents
  float4* tA;       // [32] targets: hi part
  float4* tB;       // [32] lo part
  int (*list)[32];  // finishing pass: [kSphList][lane] candidates of each target
  int* cnt;         // [32] their number, then the sub-groups' list lengths
  // some target's list could overflow in the next iteration (8 at most)
  __device__ __forceinline__ bool any_full(int lane) const {
    return __any_sync(0xffffffffu, cnt[lane] > kSphList - 8);
  }
};

struct SphGroup {
  float cx, cy, cz, ex, ey, ez;  // box centre and half extents (box units, padded)
};

// Bounding box of the active lanes' targets (hi parts, box units), padded by
// 1e-6 for the lo parts and rounding, and the boxes and reaches of the four
// sub-groups of 8 (W.box).  A pass gathers around the lanes it still has to
// serve, so a group whose other lanes have converged reaches fewer leaves.
__device__ __forceinline__ SphGroup active_boxes(const SphBufs& W, const float3& th, bool act, float reach, int lane) {
  float lo[3] = {act ? th.x : 8.f, act ? th.y : 8.f, act ? th.z : 8.f};
  float hi[3] = {act ? th.x : -8.f, act ? th.y : -8.f, act ? th.z : -8.f};
  float rr = act ? reach : 0.f;
  SphGroup G;
#pragma unroll 1
  for (int o = 1; o < 32; o <<= 1) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      lo[c] = fminf(lo[c], __shfl_xor_sync(0xffffffffu, lo[c], o));
      hi[c] = fmaxf(hi[c], __shfl_xor_sync(0xffffffffu, hi[c], o));
    }
    rr = fmaxf(rr, __shfl_xor_sync(0xffffffffu, rr, o));
    G.cx = 0.5f * (lo[0] + hi[0]);
    G.cy = 0.5f * (lo[1] + hi[1]);
    G.cz = 0.5f * (lo[2] + hi[2]);
    G.ex = 0.5f * (hi[0] - lo[0]) * 1.0001f + 1e-6f;
    G.ey = 0.5f * (hi[1] - lo[1]) * 1.0001f + 1e-6f;
    G.ez = 0.5f * (hi[2] - lo[2]) * 1.0001f + 1e-6f;
    if (o == 4 && (lane & 7) == 0) {
      const float R = rr * 1.00001f + 1e-7f;
      W.box[2 * (lane >> 3)] = make_float4(G.cx, G.cy, G.cz, lo[0] <= hi[0] ? R * R : -1.f);
      W.box[2 * (lane >> 3) + 1] = make_float4(G.ex, G.ey, G.ez, 0.f);
    }
  }
  __syncwarp();
  return G;
}

// The slot pairs within reach of each sub-group, padded to a multiple of four
// with the far pair.
__device__ __forceinline__ void sph_lists(const SphBufs& W, int cnt, int lane) {
  SphStage& St = *W.St;
  const uint32_t lt = (1u << lane) - 1u;
  const uint32_t m0 = 2 * lane < cnt ? St.sub[2 * lane] : 0u, m1 = 2 * lane + 1 < cnt ? St.sub[2 * lane + 1] : 0u;
  if ((cnt & 1) && lane < 6) {  // the empty second slot of the last pair lies far outside as well
    float4* p = lane < 2 ? &St.s0[cnt >> 1] : lane < 4 ? &St.s1[cnt >> 1] : &St.s2[cnt >> 1];
    (&p->x)[2 * (lane & 1) + 1] = -4.f;
  }
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    const uint32_t um = __ballot_sync(0xffffffffu, ((m0 | m1) >> g) & 1u);
    const int n = __popc(um);
    if ((um >> lane) & 1u) St.list[g][__popc(um & lt)] = (unsigned char)lane;
    if (lane < 3) St.list[g][n + lane] = (unsigned char)kSphFar;
    if (lane == 0) W.cnt[32 + g] = n;
  }
  __syncwarp();
}

// One gather: the particles within reach of a sub-group (R, box units, the
// largest reach) are staged, and every full stage is passed to eval(mi, end);
// mi: some staged particle has no image common to the whole group; end: the
// last call of the gather.
// Warp-uniform control flow.  Returns status bits (0 if clean).
template <class Eval>
__device__ __forceinline__ uint32_t sph_gather(const SphArgs& A, const SphBufs& W, const SphGroup& G, float R,
                                               int nodes_total, int lane, Eval& eval) {
  const TreeDev& T = A.T;
  SphStage& St = *W.St;
  const float R2 = (R * 1.00001f + 1e-7f) * (R * 1.00001f + 1e-7f);
  const float uni_lim = 0.9999f - R;
  const uint32_t lt = (1u << lane) - 1u;
  if (lane == 0) W.stack[0] = (int)(1u << 28);  // the root: node 0, one node
  int sp = 1, nq = 0, pend = 0;
  int run = 0, s0 = 0, ecur = 0;  // windows of the queued leaves: slots, next slot, its leaf
  bool mi = false;
  long long visits = 0;
  __syncwarp();
  for (;;) {
    const bool end = sp == 0 && nq == 0;
    if (end || pend > kSphStage - 32) {
      sph_lists(W, pend, lane);
      eval(W, mi, end);
      if (end) break;
      __syncwarp();
      pend = 0;
      mi = false;
    } else if (sp > 0 && run == 0 && nq <= kSphQueue - kSphQueueNeed) {
      if (sp > kSphStack - kSphStackNeed) return ST_STACK;
      const int m = sp > kSphDeep ? 1 : min(sp, 32);
      const uint32_t E = (uint32_t)W.stack[max(sp - 1 - lane, 0)];
      __syncwarp();
      const int rcnt = lane < m ? (int)(E >> 28) : 0;
      const int rfirst_l = (int)(E & 0x0fffffffu);
      if (__any_sync(0xffffffffu, lane < m && (rcnt < 1 || rcnt > 8))) return ST_TREELINK;
      int incl = rcnt;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      const int take = __popc(__ballot_sync(0xffffffffu, lane < m && incl <= 32));
      const int total = __shfl_sync(0xffffffffu, incl, take - 1);
      sp -= take;
      visits += total;
      if (visits > A.max_visits) return ST_WALKCAP;
      // lane s takes node s of the gathered ranges: r = ranges ending at or before s
      int r = 0;
#pragma unroll
      for (int b = 16; b > 0; b >>= 1) {
        const int cand = r + b;
        const int v = __shfl_sync(0xffffffffu, incl, (cand - 1) & 31);
        if (cand <= take && v <= lane) r = cand;
      }
      const int prev = __shfl_sync(0xffffffffu, incl, (r - 1) & 31);
      const int excl = r > 0 ? prev : 0;
      const int rfirst = __shfl_sync(0xffffffffu, rfirst_l, r & 31);
      const bool has = lane < total;
      const int node = has ? rfirst + (lane - excl) : 0;
      if (__any_sync(0xffffffffu, has && (node < 0 || node >= nodes_total))) return ST_TREELINK;
      const float4 NC = T.nC[node];
      const int4 ND = T.nD[node];
      bool keep = false;
      if (has) {
        const float hs = 0.5f * NC.w;
        const float gx = fmaxf(fabsf(sph_mi1(NC.x - G.cx)) - (hs + G.ex), 0.f);
        const float gy = fmaxf(fabsf(sph_mi1(NC.y - G.cy)) - (hs + G.ey), 0.f);
        const float gz = fmaxf(fabsf(sph_mi1(NC.z - G.cz)) - (hs + G.ez), 0.f);
        keep = fmaf(gx, gx, fmaf(gy, gy, gz * gz)) <= R2;
      }
      const bool leaf = meta_leaf(ND.w);
      const int nch = meta_nchild(ND.w);
      bool bad = false;
      if (keep) {
        if (leaf) bad = ND.x < 0 || ND.y < 1 || (int64_t)ND.x + ND.y > T.n;
        else bad = nch <= 0 || nch > 8 || ND.z <= node || ND.z + nch > nodes_total;
      }
      if (__any_sync(0xffffffffu, bad)) return ST_TREELINK;
      const bool push = keep && !leaf;
      const uint32_t pm = __ballot_sync(0xffffffffu, push);
      if (push) W.stack[sp + __popc(pm & lt)] = (int)((uint32_t)ND.z | ((uint32_t)nch << 28));
      sp += __popc(pm);
      const bool q = keep && leaf;
      const uint32_t qm = __ballot_sync(0xffffffffu, q);
      if (q) W.queue[nq + __popc(qm & lt)] = make_int2(ND.x, ND.y);
      nq += __popc(qm);
      __syncwarp();
    } else if (run == 0) {
      // slot offsets of the queued leaves (warp scan, 32 entries at a time)
      s0 = 0;
      ecur = 0;
#pragma unroll 1
      for (int b0 = 0; b0 < nq; b0 += 32) {
        const int e = b0 + lane;
        const int c = e < nq ? W.queue[e].y : 0;
        int incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int y = __shfl_up_sync(0xffffffffu, incl, o);
          if (lane >= o) incl += y;
        }
        if (e < nq) W.qoff[e] = run + incl - c;
        run += __shfl_sync(0xffffffffu, incl, 31);
      }
      __syncwarp();
    } else {
      // The leaves' particles 32 at a time (one coalesced load per lane); a
      // particle out of reach of every sub-group is not staged.  Each window
      // of 32 slots finds its slots' leaves without a search: ecur holds the
      // window's first slot, the leaves starting inside the window set bit
      // (start - s0) of one OR-reduced mask (leaves hold at least one
      // particle, so at most 31 start inside it), and slot s0 + l lies in leaf
      // ecur + (number of starts at or before bit l).
        const int ek = ecur + 1 + lane;
        const int sk = ek < nq ? W.qoff[ek] - s0 : 32;
        const uint32_t starts = __reduce_or_sync(0xffffffffu, (sk > 0 && sk < 32) ? (1u << sk) : 0u);
        const int slot = s0 + lane;
        uint32_t sub = 0;
        bool uni = true;
        float4 pa = make_float4(0.f, 0.f, 0.f, 0.f), pb = pa;
        int j = 0;
        if (slot < run) {
          const int e = ecur + __popc(starts & ((2u << lane) - 1u));
          j = W.queue[e].x + (slot - W.qoff[e]);
          pa = T.pA[j];
          pb = T.pB[j];
          // the image nearest to the group centre; uni: the minimum image of
          // every target that it can be within reach of
          pa.x -= sph_round1(pa.x - G.cx);
          pa.y -= sph_round1(pa.y - G.cy);
          pa.z -= sph_round1(pa.z - G.cz);
          uni = fmaxf(fabsf(pa.x - G.cx) + G.ex, fmaxf(fabsf(pa.y - G.cy) + G.ey, fabsf(pa.z - G.cz) + G.ez)) < uni_lim;
#pragma unroll
          for (int g = 0; g < 4; ++g) {
            const float4 c4 = W.box[2 * g], e4 = W.box[2 * g + 1];
            const float gx = fmaxf(fabsf(pa.x - c4.x) - e4.x, 0.f);
            const float gy = fmaxf(fabsf(pa.y - c4.y) - e4.y, 0.f);
            const float gz = fmaxf(fabsf(pa.z - c4.z) - e4.z, 0.f);
            if (c4.w >= 0.f && (!uni || fmaf(gx, gx, fmaf(gy, gy, gz * gz)) <= c4.w)) sub |= 1u << g;
          }
        }
        const uint32_t sm = __ballot_sync(0xffffffffu, sub != 0u);
        if (sub) {
          const int at = pend + __popc(sm & lt);
          const int e = 4 * (at >> 1) + (at & 1);
          float* p0 = &St.s0[0].x + e;
          float* p1 = &St.s1[0].x + e;
          float* p2 = &St.s2[0].x + e;
          p0[0] = -pa.x;
          p0[2] = -pa.y;
          p1[0] = -pa.z;
          p1[2] = -pb.x;
          p2[0] = -pb.y;
          p2[2] = -pb.z;
          St.id[at] = j;
          St.sub[at] = (unsigned char)sub;
        }
        mi = mi || __any_sync(0xffffffffu, sub != 0u && !uni);
        pend += __popc(sm);
        __syncwarp();
        // the leaf holding the next window's first slot
        int en = ecur + __popc(starts);
        if (en + 1 < nq && W.qoff[en + 1] == s0 + 32) ++en;
        ecur = en;
        s0 += 32;
        if (s0 >= run) {
          run = 0;
          nq = 0;
        }
    }
  }
  return 0u;
}

// Displacement of one target (each component twice) from a slot pair and the
// squared distances, packed, by the split-float positions (the FP64 difference
// rounded to FP32).
struct SphTarget {
  unsigned long long x, y, z, u, v, w;
};
__device__ __forceinline__ SphTarget sph_target(const SphBufs& W, int t) {
  const float4 a = W.tA[t], b = W.tB[t];
  return {sph_pack(a.x, a.x), sph_pack(a.y, a.y), sph_pack(a.z, a.z), sph_pack(b.x, b.x), sph_pack(b.y, b.y),
          sph_pack(b.z, b.z)};
}
__device__ __forceinline__ unsigned long long sph_mi2(unsigned long long d) {
  return sph_pack(sph_mi1(sph_lo(d)), sph_mi1(sph_hi(d)));
}
__device__ __forceinline__ unsigned long long sph_r2(const SphStage& St, const SphTarget& T, int k, bool mi) {
  const float4 v0 = St.s0[k], v1 = St.s1[k], v2 = St.s2[k];
  unsigned long long dx = sph_add2(T.x, sph_pack(v0.x, v0.y));
  unsigned long long dy = sph_add2(T.y, sph_pack(v0.z, v0.w));
  unsigned long long dz = sph_add2(T.z, sph_pack(v1.x, v1.y));
  if (mi) {
    dx = sph_mi2(dx);
    dy = sph_mi2(dy);
    dz = sph_mi2(dz);
  }
  dx = sph_add2(dx, sph_add2(T.u, sph_pack(v1.z, v1.w)));
  dy = sph_add2(dy, sph_add2(T.v, sph_pack(v2.x, v2.y)));
  dz = sph_add2(dz, sph_add2(T.w, sph_pack(v2.z, v2.w)));
  return sph_fma2(dx, dx, sph_fma2(dy, dy, sph_mul2(dz, dz)));
}

// FP32 passes: sums of w(q), q w'(q) and q^2 w''(q) over the particles within h.
//
// Both kinds of pass work by tiles, as in the gravity walk: a warp iteration
// takes the 8 targets of one sub-group against 4 slot pairs, lane = (pair of
// the four, target of the eight), two particles per lane in packed arithmetic.
// The sub-group's own box and reach leave a third of the group's candidates
// for each of its targets.
struct SphEval32 {
  int lane;
  float ih2_32, F0, F1, F2;  // this lane's target: 1 / h^2 (box units) and its sums
  // One sub-group.  Branch-free: w(q) = 2 u^3 - 8 v^3, w'(q) = 24 v^2 - 6 u^2 and
  // w''(q) = 12 u - 48 v with u = max(1 - q, 0), v = max(1/2 - q, 0) (both zero
  // beyond the support).
  __device__ __forceinline__ void sums32(const SphStage& St, const SphTarget& T, int g, int n, int t, bool mi) {
    const unsigned long long one = sph_pack(1.f, 1.f), half = sph_pack(0.5f, 0.5f), neg = sph_pack(-1.f, -1.f);
    const float i2 = __shfl_sync(0xffffffffu, ih2_32, t);
    const unsigned long long i22 = sph_pack(i2, i2);
    unsigned long long a0 = 0, a1 = 0, a2 = 0;
    unsigned long long rn = sph_r2(St, T, St.list[g][lane >> 3], mi);
#pragma unroll 1
    for (int e0 = 0; e0 < n; e0 += 4) {
      const unsigned long long x0 = sph_mul2(rn, i22);
      if (e0 + 4 < n) rn = sph_r2(St, T, St.list[g][e0 + 4 + (lane >> 3)], mi);
      const unsigned long long x = sph_pack(fmaxf(sph_lo(x0), 1e-30f), fmaxf(sph_hi(x0), 1e-30f));
      const unsigned long long q = sph_mul2(x, sph_pack(sph_rsqrt(sph_lo(x)), sph_rsqrt(sph_hi(x))));
      const unsigned long long u0 = sph_fma2(q, neg, one), v0 = sph_fma2(q, neg, half);
      const unsigned long long u = sph_pack(fmaxf(sph_lo(u0), 0.f), fmaxf(sph_hi(u0), 0.f));
      const unsigned long long v = sph_pack(fmaxf(sph_lo(v0), 0.f), fmaxf(sph_hi(v0), 0.f));
      const unsigned long long u2 = sph_mul2(u, u), v2 = sph_mul2(v, v);
      a0 = sph_fma2(sph_mul2(u2, sph_pack(2.f, 2.f)), u, a0);
      a0 = sph_fma2(sph_mul2(v2, sph_pack(-8.f, -8.f)), v, a0);
      a1 = sph_fma2(q, sph_fma2(v2, sph_pack(24.f, 24.f), sph_mul2(u2, sph_pack(-6.f, -6.f))), a1);
      a2 = sph_fma2(sph_mul2(q, q), sph_fma2(v, sph_pack(-48.f, -48.f), sph_mul2(u, sph_pack(12.f, 12.f))), a2);
    }
    float s0 = sph_lo(a0) + sph_hi(a0), s1 = sph_lo(a1) + sph_hi(a1), s2 = sph_lo(a2) + sph_hi(a2);
    s0 += __shfl_xor_sync(0xffffffffu, s0, 8);
    s1 += __shfl_xor_sync(0xffffffffu, s1, 8);
    s2 += __shfl_xor_sync(0xffffffffu, s2, 8);
    s0 += __shfl_xor_sync(0xffffffffu, s0, 16);
    s1 += __shfl_xor_sync(0xffffffffu, s1, 16);
    s2 += __shfl_xor_sync(0xffffffffu, s2, 16);
    if ((lane >> 3) == g) {
      F0 += s0;
      F1 += s1;
      F2 += s2;
    }
  }
  __device__ __forceinline__ void operator()(const SphBufs& W, bool mi, bool) {
#pragma unroll 1
    for (int g = 0; g < 4; ++g) {
      const int n = W.cnt[32 + g];
      if (n == 0) continue;
      const int t = 8 * g + (lane & 7);
      sums32(*W.St, sph_target(W, t), g, n, t, mi);
    }
  }
};

// Finishing pass: candidates within hb (FP32 test with a margin, by the same
// tiles) go to their targets' lists; before a list can overflow all are
// flushed, i.e. every lane evaluates its target's candidates in float-float and
// adds w to FP64 sums (sum w, sum m w, which set h and rho to ~1e-12); the
// derivatives, which scale the step from here (about 6e-5 of h after the FP32
// passes, 3e-4 at most), are FP32 sums of the same neighbours: a relative error of
// 1e-7 in them is 3e-11 of h at the largest step.
struct SphEval64 {
  const SphArgs* A;
  const SphBufs* W;
  int lane;
  int64_t k;           // this lane's sorted index
  float3 th, tl;
  float hb2_32;        // FP32 prefilter radius^2 (box units), with margin; negative once done
  FF ih2;              // 1 / h^2 (box units)
  double S0, R0;
  // the step's derivatives at this h: sum q w'(q) and sum (m / L^2) q w'(q)
  // (FP32, compensated: C1, Q1), sum q^2 w''(q) and sum (m / L^2) q^2 w''(q)
  float S1, R1, C1, Q1;
  float S2, R2;
  double bq0, bq1;     // q = r / h of the first two neighbours in the band
  int clt, band;
  __device__ __forceinline__ void flush() {
    const TreeDev& T = A->T;
    const float qhi2 = (float)((1.0 + kSphBand) * (1.0 + kSphBand)), qlo = (float)(1.0 - kSphBand);
    const int cnt = W->cnt[lane];
    const int top = __reduce_max_sync(0xffffffffu, (unsigned)cnt);
#pragma unroll 1
    for (int t = 0; t < top; ++t) {
      if (t < cnt) {
        const int j = W->list[t][lane];
        const float4 a = T.pA[j], b = T.pB[j];
        // d = x_i - x_j - s (box units), s the nearest periodic image: the hi
        // parts are multiples of 2^-23 in [0, 1), so their difference minus s
        // is exact; the lo difference is rounded once (2^-48).  d = dh + dl and
        // r^2 = |d|^2 as a float-float.
        const float dh0 = sph_mi1(__fsub_rn(th.x, a.x));
        const float dh1 = sph_mi1(__fsub_rn(th.y, a.y));
        const float dh2 = sph_mi1(__fsub_rn(th.z, a.z));
        const float dl0 = __fsub_rn(tl.x, b.x), dl1 = __fsub_rn(tl.y, b.y), dl2 = __fsub_rn(tl.z, b.z);
        const FF p0 = ff_two_prod(dh0, dh0), p1 = ff_two_prod(dh1, dh1), p2 = ff_two_prod(dh2, dh2);
        const FF s01 = ff_two_sum(p0.hi, p1.hi), s012 = ff_two_sum(s01.hi, p2.hi);
        // the small terms: the products' errors, 2 dh dl and dl^2
        float c = __fmaf_rn(2.0f * dh0 + dl0, dl0, __fmaf_rn(2.0f * dh1 + dl1, dl1, __fmul_rn(2.0f * dh2 + dl2, dl2)));
        c = __fadd_rn(c, __fadd_rn(__fadd_rn(p0.lo, p1.lo), __fadd_rn(p2.lo, __fadd_rn(s01.lo, s012.lo))));
        const FF q2 = ff_mul(ff_quick(s012.hi, c), ih2);
        if (q2.hi < qhi2) {
          // q = sqrt(q2): the rounded root and one correction,
          // q0 + (q2 - q0^2) / (2 q0), with q0^2 exact
          FF q = {0.f, 0.f};
          const float q0 = __fsqrt_rn(q2.hi);
          if (q0 > 0.f) {
            const FF sq = ff_two_prod(q0, q0);
            const float res = __fadd_rn(__fsub_rn(__fsub_rn(q2.hi, sq.hi), sq.lo), q2.lo);
            q = ff_quick(q0, __fmul_rn(res, __fdiv_rn(0.5f, q0)));
          }
          // w = 2 u^3 - 8 v^3, u = max(1 - q, 0), v = max(1/2 - q, 0)
          const FF u = ff_pos_diff(1.0f, q), v = ff_pos_diff(0.5f, q);
          const FF u3 = ff_mul(ff_mul(u, u), u), v3 = ff_mul(ff_mul(v, v), v);
          const FF w = ff_add(FF{2.0f * u3.hi, 2.0f * u3.lo}, FF{-8.0f * v3.hi, -8.0f * v3.lo});
          const double wd = sph_f2d(w.hi) + sph_f2d(w.lo);
          S0 += wd;
          R0 = fma(T.m64[j], wd, R0);
          const bool in = q.hi < 1.0f || (q.hi == 1.0f && q.lo < 0.0f);
          if (in) {
            // q w'(q) and q^2 w''(q): w' = 18 q^2 - 12 q, w'' = 36 q - 12 for
            // q <= 1/2; w' = -6 u^2, w'' = 12 u (u = 1 - q) beyond
            const float qf = q.hi, uf = 1.0f - qf;
            const bool inner = qf <= 0.5f;
            const float wq = inner ? qf * qf * fmaf(18.0f, qf, -12.0f) : -6.0f * qf * uf * uf;
            const float wqq = inner ? qf * qf * fmaf(36.0f, qf, -12.0f) : 12.0f * qf * qf * uf;
            sph_kahan_add(S1, C1, wq);
            sph_kahan_add(R1, Q1, a.w * wq);
            S2 += wqq;
            R2 = fmaf(a.w, wqq, R2);
          }
          if (j != (int)k) {
            if (in) ++clt;
            if (q.hi >= qlo) {
              const double qd = (double)q.hi + (double)q.lo;
              if (band == 0) bq0 = qd;
              else if (band == 1) bq1 = qd;
              ++band;
            }
          }
        }
      }
    }
    W->cnt[lane] = 0;
    __syncwarp();
  }
  // Lists the candidates of one sub-group's targets from list position e0 on;
  // returns where it stopped, below n if some list could overflow next.
  __device__ __forceinline__ int list64(const SphBufs& Wb, const SphTarget& T, int g, int n, int t, int e0, bool mi) {
    const SphStage& St = *Wb.St;
    const float hb2 = __shfl_sync(0xffffffffu, hb2_32, t);
    const uint32_t earlier = (1u << (lane & 24)) - 1u;
    int have = Wb.cnt[t];
    bool full = false;
#pragma unroll 1
    for (; e0 < n && !full; e0 += 4) {
      const int k = St.list[g][e0 + (lane >> 3)];
      const unsigned long long r2 = sph_r2(St, T, k, mi);
      const bool h0 = sph_lo(r2) < hb2, h1 = sph_hi(r2) < hb2;
      // this target's hits over its four lanes
      const uint32_t b0 = (__ballot_sync(0xffffffffu, h0) >> (lane & 7)) & 0x01010101u;
      const uint32_t b1 = (__ballot_sync(0xffffffffu, h1) >> (lane & 7)) & 0x01010101u;
      int at = have + __popc(b0 & earlier) + __popc(b1 & earlier);
      if (h0) Wb.list[at++][t] = St.id[2 * k];
      if (h1) Wb.list[at][t] = St.id[2 * k + 1];
      have += __popc(b0) + __popc(b1);
      full = __any_sync(0xffffffffu, have > kSphList - 8);
    }
    if (lane < 8) Wb.cnt[t] = have;
    __syncwarp();
    return full ? e0 : n;
  }
  __device__ __forceinline__ void operator()(const SphBufs& Wb, bool mi, bool end) {
    int g = 0, e0 = 0;
#pragma unroll 1
    while (g < 4 || end) {
      bool full = false;
      if (g < 4) {
        const int n = Wb.cnt[32 + g];
        const int t = 8 * g + (lane & 7);
        if (e0 < n) {
          e0 = list64(Wb, sph_target(Wb, t), g, n, t, e0, mi);
          full = Wb.any_full(lane);
        }
        if (e0 >= n) {
          ++g;
          e0 = 0;
        }
        if (!full) continue;
      }
      flush();
      if (g >= 4) break;
    }
  }
};

// Warps per group (log2): two or four shorten a call whose groups do not fill
// the chip.
static int sph_split(int64_t n_groups) { return n_groups <= 1024 ? 2 : 0; }

// Shared memory of a warp; the finishing pass's lists come with that kernel.
struct SphWarp {
  int stack[kSphStack];
  int2 queue[kSphQueue];
  int qoff[kSphQueue + 1];
  SphStage stage;
  float4 box[8];
  float4 t[2][32];
  int cnt[36];  // candidates of each target, then list lengths of the sub-groups
};

// What both kernels begin with: the tree is usable (otherwise every output is
// NaN / -1 and the status is flagged), this warp has a group, and its shared
// buffers are set up.
__device__ __forceinline__ bool sph_begin(const SphArgs& A, SphWarp& S, SphBufs& W, int64_t g, bool mine, int lane,
                                          int& nodes_total) {
  const TreeDev& T = A.T;
  if (T.sb->status != 0 || T.sb->magic != kMagicTree) {
    if (threadIdx.x == 0) set_status(A.wsb, ST_NOTREE);
    for (int64_t kk = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; kk < T.n;
         kk += (int64_t)gridDim.x * blockDim.x) {
      A.h_out[kk] = NAN;
      A.rho_out[kk] = NAN;
      A.ngb_out[kk] = -1;
    }
    return false;
  }
  if (g >= T.ngroups || !__any_sync(0xffffffffu, mine && g * kGroup + lane < T.n)) return false;
  W.stack = S.stack;
  W.queue = S.queue;
  W.qoff = S.qoff;
  W.St = &S.stage;
  W.box = S.box;
  W.tA = S.t[0];
  W.tB = S.t[1];
  W.cnt = S.cnt;
  W.list = nullptr;
  nodes_total = 0;
#pragma unroll 1
  for (int l = 0; l < kLevels; ++l) nodes_total += T.sb->level_cnt[l];
  if (nodes_total > T.cap) nodes_total = (int)T.cap;
  const int64_t k = g * kGroup + lane;
  const int64_t kc = k < T.n ? k : 0;
  W.tA[lane] = T.pA[kc];
  W.tB[lane] = T.pB[kc];
  W.cnt[lane] = 0;
  if (lane < 3) {
    float4* far = lane == 0 ? S.stage.s0 : lane == 1 ? S.stage.s1 : S.stage.s2;
    far[kSphFar] = make_float4(-4.f, -4.f, -4.f, -4.f);
  }
  __syncwarp();
  return true;
}

__device__ __forceinline__ float sph_max(float x) {  // over the warp, x >= 0
  return __int_as_float((int)__reduce_max_sync(0xffffffffu, (unsigned)__float_as_int(x)));
}

// Group at place i: those of most estimated work first, in the FP32 walk's order
// (tree_build.cu).  Against tree order, ms: clustered 64^3 3.20 -> 2.86, 90^3 6.86 ->
// 5.44, 128^3 13.6 -> 10.9; 10^6 uniform particles 2.65 -> 2.65; 128^3 lattice
// 3.67 -> 3.70.  (Ordered by count alone: 11.6 ms at 128^3.)
__device__ __forceinline__ int64_t sph_group(const SphArgs& A, int64_t i) {
  const TreeDev& T = A.T;
  const bool usable = i < T.ngroups && T.sb->status == 0 && T.sb->magic == kMagicTree;
  return usable ? group_at(T, 0, i, A.wsb) : i;
}

// FP32 Newton passes on ln h.  Leaves h (box units) in h_out for the finishing
// kernel, negative where there is no root below half the box.
__global__ void __launch_bounds__(kSphWarps * 32) k_sph_radius(SphArgs A) {
  __shared__ SphWarp s_warp[kSphWarps];
  const TreeDev& T = A.T;
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int64_t vw = (int64_t)blockIdx.x * kSphWarps + wib, g = sph_group(A, vw >> A.split);
  const bool mine = (lane >> (5 - A.split)) == (int)(vw & ((1 << A.split) - 1));
  SphBufs W;
  int nodes_total;
  if (!sph_begin(A, s_warp[wib], W, g, mine, lane, nodes_total)) return;
  const int64_t k = g * kGroup + lane;
  const bool valid = mine && k < T.n;
  const float3 th = make_float3(W.tA[lane].x, W.tA[lane].y, W.tA[lane].z);
  const float nngb = (float)A.n_ngb;

  // start: the density of the smallest ancestor holding >= N_ngb particles
  float h = 0.5f;
  {
    int p = T.leaf_of[valid ? k : 0];
#pragma unroll 1
    for (int up = 0; up < kLevels + 1 && p >= 0 && p < nodes_total; ++up) {
      const int c = T.nD[p].y;
      if ((double)c >= A.n_ngb || T.nParent[p] < 0) {
        const float s = T.nC[p].w;
        h = s * cbrtf(3.0f * nngb / (4.0f * 3.14159265f * (float)c));
        break;
      }
      p = T.nParent[p];
    }
    h = fminf(fmaxf(h, 1e-7f), 0.5f);
  }

  bool conv = !valid, fail = false;
  float blo = 0.f, bhi = 1e30f;
  uint32_t st = 0;
  SphEval32 ev;
  ev.lane = lane;
#pragma unroll 1
  for (int pass = 0; pass < kSphPass32 && __any_sync(0xffffffffu, !conv); ++pass) {
    ev.ih2_32 = 1.0f / (h * h);
    ev.F0 = 0.f;
    ev.F1 = 0.f;
    ev.F2 = 0.f;
    const float R = sph_max(conv ? 0.f : h);
    st |= sph_gather(A, W, active_boxes(W, th, !conv, h, lane), R, nodes_total, lane, ev);
    if (st) break;
    if (!conv) {
      const float N = (32.0f / 3.0f) * ev.F0;
      if (N < nngb) blo = h;
      else bhi = h;
      float dl;
      if (ev.F1 < 0.f) {
        // y(l) = ln N_eff at l = ln h: y' = -S1 / S0, y'' = (S1 + S2) / S0 - y'^2;
        // a Newton step, and near the root the one that solves
        // y + y' d + y'' d^2 / 2 = ln N_ngb to third order
        const float dy = __logf(nngb) - __logf(N), y1 = -ev.F1 / ev.F0;
        const float y2 = (ev.F1 + ev.F2) / ev.F0 - y1 * y1;
        dl = dy / y1;
        if (fabsf(dl) < 0.3f) dl = dy / fmaxf(y1 + 0.5f * y2 * dl, 0.5f * y1);
      } else dl = N >= nngb ? -0.7f : 0.7f;
      dl = fminf(fmaxf(dl, -0.7f), 0.7f);
      if (h >= 0.5f && N < nngb) {
        fail = true;  // no root below half the box
        conv = true;
      } else if (fabsf(dl) < kSphConv32) {
        // converged: take the step itself (it may round to h, which
        // is a bracket end by now, so it is not tested against the bracket)
        h = fminf(h * __expf(dl), 0.5f);
        conv = true;
      } else {
        float hn = h * __expf(dl);
        if (blo > 0.f && bhi < 1e30f && !(hn > blo && hn < bhi)) hn = sqrtf(blo * bhi);
        if (hn > 0.5f) hn = 0.5f;
        conv = bhi < 1e30f && bhi - blo < 2e-6f * bhi;
        h = hn;
      }
    }
  }
  if (st && lane == 0) set_status(A.wsb, st);
  if (valid) A.h_out[T.order[k]] = fail || st ? -1.0 : (double)h;
}

// Finishing pass(es): second-order step, density and neighbour count.
__global__ void __launch_bounds__(kSphWarps * 32, 17) k_sph_density(SphArgs A) {
  __shared__ SphWarp s_warp[kSphWarps];
  __shared__ int s_list[kSphWarps][kSphList][32];
  const TreeDev& T = A.T;
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int64_t vw = (int64_t)blockIdx.x * kSphWarps + wib, g = sph_group(A, vw >> A.split);
  const bool mine = (lane >> (5 - A.split)) == (int)(vw & ((1 << A.split) - 1));
  SphBufs W;
  int nodes_total;
  if (!sph_begin(A, s_warp[wib], W, g, mine, lane, nodes_total)) return;
  W.list = s_list[wib];
  const int64_t k = g * kGroup + lane;
  const bool valid = mine && k < T.n;
  const int32_t i = valid ? T.order[k] : 0;
  const float4 pa = W.tA[lane], pb = W.tB[lane];
  const float3 th = make_float3(pa.x, pa.y, pa.z);
  const double L = A.B.L;
  double hd = valid ? A.h_out[i] * L : -1.0;
  const bool fail = !(hd > 0.0);
  bool done = fail;
  double lo64 = 0.0, hi64 = 0.0;  // FP64 bracket (hi64 = 0: none yet)
  double h_out = NAN, rho_out = NAN;
  int ngb_out = -1;
  uint32_t st = 0;
  SphEval64 ev;
  ev.A = &A;
  ev.W = &W;
  ev.lane = lane;
  ev.k = k;
  ev.th = th;
  ev.tl = make_float3(pb.x, pb.y, pb.z);
#pragma unroll 1
  for (int pass = 0; pass < kSphPass64 && __any_sync(0xffffffffu, !done); ++pass) {
    {
      const double v = (L * L) / (hd * hd);  // 1 / h^2 in box units, as a float-float
      ev.ih2.hi = (float)v;
      ev.ih2.lo = (float)(v - (double)ev.ih2.hi);
    }
    const float hb = (float)(hd * (1.0 + kSphBand) / L);
    ev.hb2_32 = done ? -1.f : hb * hb * 1.0001f + 1e-14f;
    ev.S0 = ev.R0 = 0.0;
    ev.S1 = ev.R1 = ev.C1 = ev.Q1 = 0.f;
    ev.S2 = ev.R2 = 0.f;
    ev.bq0 = ev.bq1 = 0.0;
    ev.clt = ev.band = 0;
    const float R = sph_max(done ? 0.f : hb);
    st |= sph_gather(A, W, active_boxes(W, th, !done, hb, lane), R, nodes_total, lane, ev);
    if (st) break;
    if (!done) {
      // Second-order step in d = ln(h / hd): with q' = q e^-d,
      //   sum w(q') = S0 - d S1 + d^2 / 2 (S1 + S2) + O(d^3)
      // (S1 = sum q w', S2 = sum q^2 w''; the spline is C^2, and neighbours
      // entering or leaving the sphere add O(d^3)).  Solve (32/3) of it =
      // N_ngb by Newton steps on the quadratic; its error, ~20 d^3 of N_ngb,
      // is below 1e-9 for the accepted |d| <= kSphStep.
      const double N = (32.0 / 3.0) * ev.S0;
      if (N < A.n_ngb) lo64 = hd;
      else hi64 = hd;
      const double c0 = ev.S0 - (3.0 / 32.0) * A.n_ngb;
      const double s1 = (double)ev.S1 - (double)ev.C1, r1 = (double)ev.R1 - (double)ev.Q1;
      const double c1 = -s1, c2 = 0.5 * (s1 + (double)ev.S2);
      double d;
      if (c1 > 0.0) {
        d = -c0 / c1;
        for (int it = 0; it < 2; ++it) {
          const double den = c1 + 2.0 * c2 * d;
          if (den > 0.0) d -= (c0 + (c1 + c2 * d) * d) / den;
        }
      } else {
        d = N >= A.n_ngb ? -0.69 : 0.69;
      }
      double hn = hd * exp(d);
      const bool small = fabs(d) <= kSphStep;
      if (!small && hi64 > 0.0 && lo64 > 0.0 && !(hn > lo64 && hn < hi64)) hn = 0.5 * (lo64 + hi64);
      // with more than two band neighbours (their distances are not kept)
      // the step must be at the FP64 resolution: no neighbour then lies
      // between hd and hn short of an exact tie
      if (small && (ev.band <= 2 || fabs(d) <= 1e-12)) {
        // the step stays inside the band (kSphBand > kSphStep), so only band
        // neighbours can change side between hd and hn
        const double qn = hn / hd;
        int c = ev.clt;
        if (ev.band >= 1) c += (int)(ev.bq0 < qn) - (int)(ev.bq0 < 1.0);
        if (ev.band >= 2) c += (int)(ev.bq1 < qn) - (int)(ev.bq1 < 1.0);
        // rho at hn from sum m w to second order in d, as sum w above
        const double L2 = L * L;
        const double R0f = ev.R0 + (-d * r1 + 0.5 * d * d * (r1 + (double)ev.R2)) * L2;
        h_out = hn;
        rho_out = 8.0 * R0f / (M_PI * hn * hn * hn);
        ngb_out = c;
        done = true;
      } else {
        hd = hn > 0.5 * L ? 0.5 * L : hn;
      }
    }
  }
  if (st && lane == 0) set_status(A.wsb, st);
  if (valid) {
    if (!done || fail || st) {
      if (!st) set_status(A.wsb, ST_WALKCAP);
      h_out = NAN;
      rho_out = NAN;
      ngb_out = -1;
    }
    A.h_out[i] = h_out;
    A.rho_out[i] = rho_out;
    A.ngb_out[i] = ngb_out;
  }
}

}  // namespace og

extern "C" {

size_t og_sph_ws_bytes(void) { return og::align_up(sizeof(og::StatusBlock)); }

og_status og_sph_density(const og_tree* t, double n_ngb, void* ws, size_t ws_bytes, double* h, double* rho,
                         int32_t* ngb, og_stream stream) {
  if (!t || !t->built || !t->mem) return OG_ETREE;
  if (!ws || !h || !rho || !ngb) return OG_EINVAL;
  if (!std::isfinite(n_ngb) || n_ngb <= 0.0) return OG_EINVAL;
  if ((reinterpret_cast<uintptr_t>(ws) % og::kAlign) != 0) return OG_EINVAL;
  if (ws_bytes < og_sph_ws_bytes()) return OG_ENOSPACE;
  if (t->node_capacity >= (int64_t(1) << 28)) return OG_EINVAL;  // node indices are packed in 28 bits
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  og::SphArgs A;
  A.T = og::tree_view(t);
  A.wsb = static_cast<og::StatusBlock*>(ws);
  A.B = og::box_scale(t->box);
  A.n_ngb = n_ngb;
  A.max_visits = t->max_walk_iters;
  A.h_out = h;
  A.rho_out = rho;
  A.ngb_out = ngb;
  if (cudaMemsetAsync(A.wsb, 0, sizeof(og::StatusBlock), s) != cudaSuccess) return OG_ECUDA;
  A.split = og::sph_split(t->n_groups);
  const int64_t grid = ((t->n_groups << A.split) + og::kSphWarps - 1) / og::kSphWarps;
  if (grid <= 0) return OG_OK;
  og::k_sph_radius<<<(unsigned)grid, og::kSphWarps * 32, 0, s>>>(A);
  og::k_sph_density<<<(unsigned)grid, og::kSphWarps * 32, 0, s>>>(A);
  return cudaGetLastError() == cudaSuccess ? OG_OK : OG_ECUDA;
}

}  // extern "C"
