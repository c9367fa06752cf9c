// walk.cu -- K6 FP32+Kahan walk, K6d FP64 walk, K7 adjoint walk.
//
// One warp walks the tree for one group of 32 Hilbert-consecutive targets
// (lane = target).  The warp keeps a stack of (first node, node count, lane
// mask) ranges in shared memory and pops up to 32 nodes per step, one per
// lane.  Each node is first classified against the bounding box of the whole
// group (drop / open / accept / mixed); a mixed node is classified again
// against the boxes of the four 8-target sub-groups, and only the sub-groups
// left undecided take per-lane decisions.  Opened internal nodes push their
// children as one range with the mask of the lanes that opened them; opened
// leaves and accepted nodes are queued.  Each target therefore receives
// exactly the terms of its own per-particle walk (the rules are listed in
// og.h), while node data is read once per warp.
//
// Evaluation.  Queued entries are expanded into source slots, 32 at a time
// (fetched by cp.async while the previous ones are evaluated); a source
// beyond r_cut of the group box is dropped and the others are staged, up to
// 64 for a batch.  In the FP32 walks a batch is evaluated by tiles of 8
// targets x 8 sources: each of the group's four sub-groups of 8 lists the
// pairs of adjacent slots within r_cut of its box, and a warp iteration takes
// four listed pairs against its 8 targets, two sources per lane in packed
// (f32x2) arithmetic, with the exact cut taken per pair.  A target's sum stays
// in registers over its sub-group's list, in a fixed order, so the result
// does not depend on scheduling; in the adjoint the sources' sums over the 8
// targets are exchanged by shuffles.  The FP64 variant lists the pairs inside
// a conservative cut filter (|x_i|^2 + |x_j|^2 - 2 x_i.x_j against r_cut^2)
// target by target, evaluates 32 listed pairs per iteration and sums each
// target's run by a segmented scan.
//
// The kernel is bound by instruction issue and by the instruction cache: its
// warps are at different places of a loop nest of about 2000 instructions, and
// an adjoint build with 20 % more code runs 40 % slower on the clustered set
// and no slower with one warp per SM.  Hence the loops that are not unrolled,
// and the softened and cut-band pairs evaluated after their list.
//
// FP32 path.  Positions are split floats in box units (hi a multiple of 2^-23,
// lo the rest), so hi_i - hi_j is exact and every displacement
// (hi_i - hi_j) + (lo_i - lo_j) is the FP64 difference rounded to FP32.  A
// decision whose FP32 test falls within a small relative band of its
// threshold is re-taken in FP64 with the same operation order as the CPU
// reference, so decisions agree with an FP64 walk.  Interactions use the
// special-function unit (rsqrt, ex2) and a polynomial for
// erfcx(u) + 2u/sqrt(pi); per-target sums are Kahan-compensated after every
// batch (at most 64 terms per target, 8 per lane and slot parity).
#include <type_traits>

#include "og_internal.cuh"
#include "short_range_poly.inc"
#include "short_range_table.inc"

namespace og {

enum : int { DEC_DISCARD = 0, DEC_OPEN = 1, DEC_ACCEPT = 2, DEC_ACCEPT_OUT = 3 };


// ------------------------------------------------------------------ helpers

__device__ __forceinline__ float rsqrt_approx(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(smem)), "l"(gmem)
               : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }
// Minimum image of a box-unit difference t (|t| < 1.5): t - rint(t), with
// rint by the 1.5 * 2^23 rounding constant (round to nearest even, so
// +-0.5 stay), equal bit for bit to t - 1 / t + 1 / t on t > 0.5 / t < -0.5 /
// otherwise.
__device__ __forceinline__ float round1(float t) { return __fadd_rn(__fadd_rn(t, 12582912.0f), -12582912.0f); }
__device__ __forceinline__ float mi1(float t) { return __fadd_rn(t, -round1(t)); }

__device__ __forceinline__ float sr_poly(float t) {
  float p = og_sr_poly[OG_SR_POLY_DEG];
#pragma unroll
  for (int k = OG_SR_POLY_DEG - 1; k >= 0; --k) p = fmaf(p, t, og_sr_poly[k]);
  return p;
}

// FP64 forms with the reference's operation order (no contraction).
__device__ __forceinline__ double mi64(double t, double L) {
  const double h = __dmul_rn(0.5, L);
  if (t > h) return __dsub_rn(t, L);
  if (t < -h) return __dadd_rn(t, L);
  return t;
}
__device__ __forceinline__ double norm2_64(double a, double b, double c) {
  return __dadd_rn(__dadd_rn(__dmul_rn(a, a), __dmul_rn(b, b)), __dmul_rn(c, c));
}

// Exact (FP64) node decision for sorted target k.
__device__ __noinline__ int decide_exact(const WalkArgs& A, int64_t k, int node, int level) {
  const TreeDev& T = A.T;
  const double L = A.box;
  const double side = ldexp(L, -level);
  const double half = __dmul_rn(0.5, side);
  double dc[3], cmax = 0.0, e[3], f[3], d[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    dc[c] = fabs(mi64(__dsub_rn(T.x64[3 * k + c], T.cen64[3 * (int64_t)node + c]), L));
    if (dc[c] > cmax) cmax = dc[c];
    e[c] = __dsub_rn(dc[c], half);
    if (e[c] < 0.0) e[c] = 0.0;
  }
  const double e2 = norm2_64(e[0], e[1], e[2]);
  if (e2 > A.rc2_64) return DEC_DISCARD;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    f[c] = __dadd_rn(dc[c], half);
    d[c] = mi64(__dsub_rn(T.x64[3 * k + c], T.com64[3 * (int64_t)node + c]), L);
  }
  const double far2 = norm2_64(f[0], f[1], f[2]);
  const double d2 = norm2_64(d[0], d[1], d[2]);
  const bool inside = cmax <= __dmul_rn(0.6, side);
  if (__dmul_rn(side, side) < __dmul_rn(A.th2_64, d2) && !inside && far2 < A.rc2_64)
    return d2 < A.rc2_64 ? DEC_ACCEPT : DEC_ACCEPT_OUT;
  return DEC_OPEN;
}

__device__ __noinline__ bool pair_inside_exact(const WalkArgs& A, int64_t k, int64_t j) {
  const double* x = A.T.x64;
  const double L = A.box;
  const double a = mi64(__dsub_rn(x[3 * k], x[3 * j]), L);
  const double b = mi64(__dsub_rn(x[3 * k + 1], x[3 * j + 1]), L);
  const double c = mi64(__dsub_rn(x[3 * k + 2], x[3 * j + 2]), L);
  return norm2_64(a, b, c) < A.rc2_64;
}

// Softened kernel K_h(r) inside r < h (v = r / h), FP32.
__device__ __forceinline__ void spline_f32(float r, float h2, float& K, float& Kp_r) {
  const float h = sqrtf(h2);
  const float hinv = 1.0f / h;
  const float v = r * hinv;
  const float h3 = hinv * hinv * hinv;
  if (v < 0.5f) {
    K = h3 * (10.6666666667f + v * v * (32.0f * v - 38.4f));
    Kp_r = h3 * hinv * hinv * (96.0f * v - 76.8f);
  } else {
    const float v3 = v * v * v;
    K = h3 * (21.3333333333f - 48.0f * v + 38.4f * v * v - 10.6666666667f * v3 - 0.0666666667f / v3);
    Kp_r = h3 * hinv * hinv * (-48.0f / v + 76.8f - 32.0f * v + 0.2f / (v3 * v * v));
  }
}

// Force factor F = K_h(r) f(r) (and its radial derivative over r if wanted).
template <bool DERIV>
__device__ __forceinline__ void force_f32(const WalkArgs& A, float r2, float h2, float& F, float& Fr) {
  float K, Kp_r, r;
  if (r2 >= h2) {
    const float ri = rsqrt_approx(r2);
    r = r2 * ri;
    K = ri * ri * ri;
    Kp_r = -3.0f * K * ri * ri;
  } else {
    r = sqrtf(r2);
    spline_f32(r, h2, K, Kp_r);
  }
  const float e = ex2_approx(r2 * A.ex2c);
  const float g = sr_poly(fmaf(r, A.t_scale, -1.0f));
  const float f = g * e;
  F = K * f;
  if (DERIV) Fr = fmaf(Kp_r, f, K * (A.fp_c * e * r));  // f'(r)/r = fp_c r exp(-u^2)
  else Fr = 0.0f;
}

__device__ __forceinline__ void kahan_add(float& T, float& C, float x) {
  const float y = x - C;
  const float t = T + y;
  C = (t - T) - y;
  T = t;
}

// Exact float -> double by bit manipulation on the integer pipe (the FP64
// pipe is a small fraction of the FP32 rate on this GPU).  Subnormal inputs
// flush to zero, like the FP32 arithmetic that produced them.
__device__ __forceinline__ double f2d_exact(float x) {
  const uint32_t u = __float_as_uint(x);
  const uint32_t e = (u >> 23) & 0xffu;
  const uint64_t sign = (uint64_t)(u >> 31) << 63;
  const uint64_t exp = e == 0xffu ? 0x7ffull : (uint64_t)(e + (1023u - 127u));
  const uint64_t man = (uint64_t)(u & 0x7fffffu) << 29;
  const uint64_t bits = e == 0u ? sign : (sign | (exp << 52) | man);
  return __longlong_as_double((long long)bits);
}

struct GroupInfo {
  float cx, cy, cz;  // group box centre
  float ex, ey, ez;  // group box half extents (padded outward)
};

// ------------------------------------------------------------------ per-warp shared buffers

// Traversal stack of child ranges.  A step pops ranges holding up to 32
// nodes and pushes at most one range per popped node (net growth <= 31).
// Above kDeep entries a step pops a single range (<= 8 nodes, growth <= 7
// per level), so the depth stays below kDeep + 31 + 7 x 20 + 8 for any tree.
constexpr int kStack = 276;
constexpr int kStackNeed = 32;   // pushes of one step
constexpr int kDeep = 64;
static_assert(kDeep + 31 + 7 * 20 + 8 <= kStack - kStackNeed, "stack bound");
constexpr int kSub = 4;          // sub-groups of 8 Hilbert-consecutive targets
constexpr int kQueue = 128;      // queued leaves / accepted nodes per warp
constexpr int kQueueNeed = 64;   // a step queues at most 2 entries per node
constexpr int kSlots = 32;       // sources fetched at a time
constexpr int kStage = 2 * kSlots; // staged sources: one batch
constexpr int kList = 512;       // FP64 variant: listed pairs; the FP32 walk lists at most kSub * kGroup entries

// Stack entry: (first node | node count << 28, lane mask); node indices stay
// below 2^28 (checked on the host).  Queue entry: (first particle or node,
// particle count or -1 for an accepted node, lane mask, unused).
struct WarpBufs {
  int2* stack;
  int4* queue;
  int* qoff;
  unsigned short* list;  // per-lane decision list (traversal) or pair list (evaluation)
};

// Nodes of one traversal step that need per-lane decisions.
struct MixedScratch {
  int4 D[kGroup];
  float4 C[kGroup], A[kGroup], B[kGroup];  // C, A image-shifted when the node has a common image
  int node[kGroup], fl[kGroup];
  uint32_t mask[kGroup], acc[kGroup], open[kGroup];
};

enum : int { CL_NONE = -1, CL_DROP = 0, CL_OPEN = 1, CL_ACCEPT = 2, CL_MIXED = 3 };

// Group-level classification of a node against the whole group box (box
// units, FP32, conservative margins): DROP if the cube is beyond rcut of
// every point of the box; OPEN if no point of the box can accept it; ACCEPT
// if every point of the box accepts it (cube inside rcut, outside the 1.2x
// cube, side < theta d); MIXED otherwise (exact per-lane decisions follow).
__device__ __forceinline__ int classify(const WalkArgs& A, const GroupInfo& G, const float4& NC, const float4& NA,
                                        const float4& NB) {
  const float s = NC.w, hs = 0.5f * s;
  const float tcx = fabsf(mi1(NC.x - G.cx)), tcy = fabsf(mi1(NC.y - G.cy)), tcz = fabsf(mi1(NC.z - G.cz));
  const float gx = fmaxf(tcx - G.ex - hs, 0.f), gy = fmaxf(tcy - G.ey - hs, 0.f), gz = fmaxf(tcz - G.ez - hs, 0.f);
  if (fmaf(gx, gx, fmaf(gy, gy, gz * gz)) > A.grp_rc2) return CL_DROP;
  if (s > 0.25f || G.ex > 0.125f || G.ey > 0.125f || G.ez > 0.125f) return CL_MIXED;
  if (A.th2_hi == 0.0f) return CL_OPEN;  // theta = 0: nothing is ever accepted
  const float txx = fabsf(mi1((NA.x - G.cx) + NB.x));
  const float txy = fabsf(mi1((NA.y - G.cy) + NB.y));
  const float txz = fabsf(mi1((NA.z - G.cz) + NB.z));
  const float m_lo = 0.999f, m_hi = 1.001f;
  const float ax = txx + G.ex, ay = txy + G.ey, az = txz + G.ez;
  const float dmax2 = fmaf(ax, ax, fmaf(ay, ay, az * az));
  const float bx = fmaxf(txx - G.ex, 0.f), by = fmaxf(txy - G.ey, 0.f), bz = fmaxf(txz - G.ez, 0.f);
  const float dmin2 = fmaf(bx, bx, fmaf(by, by, bz * bz));
  const float fx0 = fmaxf(tcx - G.ex, 0.f) + hs, fy0 = fmaxf(tcy - G.ey, 0.f) + hs, fz0 = fmaxf(tcz - G.ez, 0.f) + hs;
  const float minfar2 = fmaf(fx0, fx0, fmaf(fy0, fy0, fz0 * fz0));
  const float fx1 = tcx + G.ex + hs, fy1 = tcy + G.ey + hs, fz1 = tcz + G.ez + hs;
  const float maxfar2 = fmaf(fx1, fx1, fmaf(fy1, fy1, fz1 * fz1));
  const float lim = 0.6f * s;
  const bool all_inside = tcx + G.ex < lim * m_lo && tcy + G.ey < lim * m_lo && tcz + G.ez < lim * m_lo;
  const bool all_outside = tcx - G.ex > lim * m_hi || tcy - G.ey > lim * m_hi || tcz - G.ez > lim * m_hi;
  const float s2 = s * s;
  if (s2 > A.th2_hi * dmax2 * m_hi || all_inside || minfar2 > A.rc2 * m_hi) return CL_OPEN;
  if (s2 < A.th2_lo * dmin2 * m_lo && all_outside && maxfar2 < A.rc2 * m_lo) return CL_ACCEPT;
  return CL_MIXED;
}

// Image shift that puts every (target, source) pair of a node that can lie
// inside rcut at its minimum image, if one exists for the whole cube.
__device__ __forceinline__ bool node_image(const WalkArgs& A, const GroupInfo& G, const float4& NC, float& nx, float& ny,
                                           float& nz) {
  const float hs = 0.5f * NC.w;
  const float dx = NC.x - G.cx, dy = NC.y - G.cy, dz = NC.z - G.cz;
  nx = round1(dx);
  ny = round1(dy);
  nz = round1(dz);
  return fabsf(dx - nx) + G.ex + hs < A.uni_lim && fabsf(dy - ny) + G.ey + hs < A.uni_lim &&
         fabsf(dz - nz) + G.ez + hs < A.uni_lim;
}

// Validates the queue and writes the slot offsets; returns the slot count or
// -1 if an entry is malformed (then nothing may be evaluated).
__device__ __forceinline__ int queue_offsets(const WalkArgs& A, const WarpBufs& W, int nq, int lane) {
  int run = 0;
  bool badq = false;
#pragma unroll 1
  for (int b0 = 0; b0 < nq; b0 += 32) {
    const int e = b0 + lane;
    int c = 0;
    if (e < nq) {
      const int4 Q = W.queue[e];
      if (Q.y == -1) {
        c = 1;
        badq = badq || Q.x < 0 || Q.x >= A.T.cap;
      } else {
        c = Q.y;
        badq = badq || Q.y < 1 || Q.x < 0 || (int64_t)Q.x + Q.y > A.T.n;
      }
    }
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
  if (__any_sync(0xffffffffu, badq)) return -1;
  return run;
}


// 32 x 32 bit-matrix transpose across the warp: lane r holds row r (bit c =
// column c) and receives column r.  Five stages swap the off-diagonal blocks
// of side 16, 8, 4, 2, 1 between partner lanes.  (Unrolled, the forward walk
// needs 110 registers instead of 96 and loses a resident block; the adjoint
// is 2-5 % faster with it.)
template <int kUnroll>
__device__ __forceinline__ uint32_t transpose32(uint32_t x, int lane) {
  const uint32_t keep[5] = {0x0000ffffu, 0x00ff00ffu, 0x0f0f0f0fu, 0x33333333u, 0x55555555u};
  int j = 16;
#pragma unroll kUnroll
  for (int st = 0; st < 5; ++st, j >>= 1) {
    const uint32_t y = __shfl_xor_sync(0xffffffffu, x, j);
    x = (lane & j) == 0 ? ((x & keep[st]) | ((y & keep[st]) << j)) : ((x & ~keep[st]) | ((y & ~keep[st]) >> j));
  }
  return x;
}

// ------------------------------------------------------------------ lanes

__device__ __forceinline__ unsigned long long pack2(float lo, float hi) {
  return ((unsigned long long)__float_as_uint(hi) << 32) | __float_as_uint(lo);
}
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b) {
  unsigned long long d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
  unsigned long long d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}

__device__ __forceinline__ unsigned long long mul2(unsigned long long a, unsigned long long b) {
  unsigned long long d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ float lo2(unsigned long long a) { return __uint_as_float((uint32_t)a); }
__device__ __forceinline__ float hi2(unsigned long long a) { return __uint_as_float((uint32_t)(a >> 32)); }
// sr_poly of both halves; the doubled coefficients sit in constant memory
// (a 64-bit operand cannot be an immediate).
__device__ __forceinline__ unsigned long long sr_poly2(unsigned long long t) {
  const unsigned long long* c = reinterpret_cast<const unsigned long long*>(og_sr_poly2);
  unsigned long long p = c[OG_SR_POLY_DEG];
#pragma unroll
  for (int k = OG_SR_POLY_DEG - 1; k >= 0; --k) p = fma2(p, t, c[k]);
  return p;
}
__device__ __forceinline__ uint32_t low_bits(int n) { return n >= 32 ? 0xffffffffu : ((1u << n) - 1u); }

// Exact per-target decision for a node (FP32 with an FP64 re-check in the
// band), target given by its split position.  With uni, NC and NA are
// already shifted to the image that is the minimum image for every target
// of the group, so no per-target minimum image is taken.  A node beyond
// rcut is opened rather than discarded: none of its descendants gives this
// target a term, and the test is saved.  A node whose farthest corner is
// inside the cut has its centre of mass inside it.
__device__ __forceinline__ float mi1_if(bool per_target, float t) { return per_target ? mi1(t) : t; }

__device__ __forceinline__ int decide_f32(const WalkArgs& A, int64_t k, const float4& th, const float4& tl, int node,
                                          int level, const float4& NC, const float4& NA, const float4& NB,
                                          bool uni) {
  const float s = NC.w, hs = 0.5f * s;
  // hi differences are exact: the minimum image is taken before the lo parts are added
  const float ax = fabsf(mi1_if(!uni, NC.x - th.x) - tl.x);
  const float ay = fabsf(mi1_if(!uni, NC.y - th.y) - tl.y);
  const float az = fabsf(mi1_if(!uni, NC.z - th.z) - tl.z);
  const float d0 = mi1_if(!uni, th.x - NA.x) + (tl.x - NB.x);
  const float d1 = mi1_if(!uni, th.y - NA.y) + (tl.y - NB.y);
  const float dz = mi1_if(!uni, th.z - NA.z) + (tl.z - NB.z);
  const float d2 = fmaf(d0, d0, fmaf(d1, d1, dz * dz));
  const float fx = ax + hs, fy = ay + hs, fz = az + hs;
  const float far2 = fmaf(fx, fx, fmaf(fy, fy, fz * fz));
  const float lhs = s * s;
  const float cmax = fmaxf(ax, fmaxf(ay, az));
  if (lhs > A.th2_hi * d2 || cmax < A.lim_lo * s || far2 > A.rc2_hi) return DEC_OPEN;
  if (lhs < A.th2_lo * d2 && cmax > A.lim_hi * s && far2 < A.rc2_lo) return DEC_ACCEPT;
  return decide_exact(A, k, node, level);
}

// The short-range factor f(u) = erfc(u) + (2 u / sqrt(pi)) exp(-u^2) in FP64:
// a degree-6 polynomial about the centre of each interval of width 1 / 64
// (its error, below 1e-17, is far under the rounding), four 16-byte loads and
// seven FP64 operations.  uf: u to FP32 accuracy (beside a boundary either
// interval's polynomial serves).  u stays below 2.25 at the default cut of
// 4.5 r_s; beyond the table CUDA's functions take over.
__device__ __forceinline__ double short_range_f64(double u, float uf) {
  const float fi = uf * (float)OG_SR_TABLE_PER_UNIT;
  if (fi < (float)OG_SR_TABLE_N) {
    const int i = (int)fi;
    const double2* e = reinterpret_cast<const double2*>(og_sr_table) + 4 * i;
    const double2 a = __ldg(e), b = __ldg(e + 1), c = __ldg(e + 2), d = __ldg(e + 3);
    const double x = u - a.x;
    return fma(fma(fma(fma(fma(fma(d.y, x, d.x), x, c.y), x, c.x), x, b.y), x, b.x), x, a.y);
  }
  return erfc(u) + 1.1283791670955126 * u * exp(-u * u);
}

// Lane of the walk: FP32 + Kahan forward (ADJ = false) or adjoint
// (ADJ = true), or the all-FP64 forward variant (F64 = true: FP64 pair
// arithmetic, plain double sums).  All share the traversal, its decisions
// (which agree with FP64) and the box test.
// FUSED (with ADJ): the adjoint walk that also writes the forward
// accelerations, each pair's force factor serving both (one traversal for a
// loss whose weights are known before the walk).
template <bool ADJ, bool F64, bool FUSED = false>
struct LaneFP {
  static_assert(!FUSED || (ADJ && !F64), "the fused walk is the FP32 adjoint plus the forward sums");
  static constexpr int kListSize = F64 ? kList : kSub * kGroup;
  static constexpr int kOrder = F64 ? 1 : 0;  // of T.gorder
  // per-warp data that lives through the whole walk
  struct Smem {
    float4 tA[kGroup];    // targets: hi part, h^2
    float4 tB[kGroup];    // targets: lo part
    float4 tW[ADJ ? kGroup : 1];   // adjoint: dL/da of each target
    float4 SG[ADJ ? kStage : 1];   // adjoint: source-side sums (G, S) of each staged slot over the batch
    int self[kGroup];     // staged slot holding the target itself, or -1
    // FP64 variant: targets; each target's sum over the batch; the sum of each
    // lane's first run where that run began in an earlier lane
    double tx[F64 ? 3 : 1][F64 ? kGroup : 1], th2[F64 ? kGroup : 1];
    double Ps[F64 ? 3 : 1][F64 ? kGroup : 1], Hd[F64 ? 3 : 1][F64 ? kGroup : 1];
    int fneg[F64 ? kGroup : 1];  // listed pairs of the batch outside the exact cut
  };
  // per-batch staging (dead between evaluations; shares memory with the
  // traversal's scratch)
  // Survivors of the box test are appended; a batch is evaluated once the
  // next 32 might not fit.  The FP32 walk keeps the two sources of adjacent
  // slots 2k, 2k + 1 component by component, so that one 16-byte load gives
  // two register pairs of a packed (f32x2) operand.
  struct Stage {
    float4 s0[F64 ? 1 : kStage / 2];  // -hi.x of both, -hi.y of both (image-shifted)
    float4 s1[F64 ? 1 : kStage / 2];  // -hi.z, -mass
    float4 s2[F64 ? 1 : kStage / 2];  // -lo.x, -lo.y
    float4 s3[F64 ? 1 : kStage / 2];  // -lo.z, h^2
    float4 ra[F64 ? 1 : kSlots], rb[F64 ? 1 : kSlots];  // the next 32 sources as they arrive from the tree
    int id[kStage];       // particle, or -2 - node
    uint32_t sq[kStage];  // lane mask of the source's queue entry
    double sx[F64 ? 3 : 1][F64 ? kStage : 1], sm[F64 ? kStage : 1], sh2[F64 ? kStage : 1];  // FP64: position, -mass, h^2
    float fX[F64 ? kStage : 1], fY[F64 ? kStage : 1], fZ[F64 ? kStage : 1], fW[F64 ? kStage : 1];  // filter form (see put)
  };
  // a slot's source as read from the tree
  struct Fetch {
    float4 a, b;
    int id;  // particle, or -2 - node
    uint32_t q;
    bool shifted;  // FP64 variant: not at its stored image
  };

  int64_t k;          // sorted index of this lane's target
  bool valid;
  float xr[3], sr;    // position relative to the group centre and its square (filter)
  float P[3];         // partial sum since the last fold
  float S[3], C[3];   // Kahan total and compensation
  float Pf[3], Sf[3], Cf[3];  // fused: the forward sums likewise
  double a64[3];      // FP64 variant: plain double sums
  int nint;

  // True if the warp's batches need batch_wild.
  __device__ bool init(const WalkArgs& A, Smem& M, int64_t kk, bool v, int lane, const GroupInfo& G) {
    k = kk;
    valid = v;
    const int64_t kc = v ? kk : 0;  // never form an out-of-range address
    const float4 a = A.T.pA[kc];
    const float4 b = A.T.pB[kc];
    M.tA[lane] = make_float4(a.x, a.y, a.z, b.w);
    M.tB[lane] = make_float4(b.x, b.y, b.z, 0.f);
    if constexpr (F64) {
#pragma unroll
      for (int c = 0; c < 3; ++c) M.tx[c][lane] = A.T.x64[3 * kc + c];
      const double h = A.T.h64[kc];
      M.th2[lane] = h * h;
    }
    a64[0] = a64[1] = a64[2] = 0.0;
    if constexpr (F64) M.fneg[lane] = 0;
    if constexpr (ADJ) M.SG[lane] = M.SG[lane + 32] = make_float4(0.f, 0.f, 0.f, 0.f);
    xr[0] = (a.x - G.cx) + b.x;
    xr[1] = (a.y - G.cy) + b.y;
    xr[2] = (a.z - G.cz) + b.z;
    sr = fmaf(xr[0], xr[0], fmaf(xr[1], xr[1], xr[2] * xr[2]));
#pragma unroll
    for (int c = 0; c < 3; ++c) { P[c] = 0.f; S[c] = 0.f; C[c] = 0.f; Pf[c] = 0.f; Sf[c] = 0.f; Cf[c] = 0.f; }
    bool wild = A.T.sb->pad[kTreeWildMass] != 0;
    if (ADJ) {
      float4 w = make_float4(0.f, 0.f, 0.f, 0.f);
      if (v) {
        const int32_t i = A.T.order[kk];
        w = make_float4(A.w[3 * (int64_t)i], A.w[3 * (int64_t)i + 1], A.w[3 * (int64_t)i + 2], 0.f);
      }
      M.tW[lane] = w;
      wild = wild || !(fabsf(w.x) <= kWildWeight && fabsf(w.y) <= kWildWeight && fabsf(w.z) <= kWildWeight);
    }
    nint = 0;
    return !F64 && __any_sync(0xffffffffu, wild);
  }

  // FP64 variant: force of staged slot s on target i, added to acc; false
  // (and nothing added) outside the cut.  1 / r by a third-order step from the
  // FP32 reciprocal root.  The cut is taken on r^2 in the reference's order of
  // operations where the contracted r^2 is within rounding of it (accepted
  // nodes are inside by decision).  Bound by the FP64 pipe, 1/64 of the FP32
  // rate: 28 operations a pair (displacement 3, r^2 3, 1 / r and r 6, factor 8,
  // force 8) where CUDA's erfc, exp, sqrt and divisions and a segmented scan of
  // the sums took about 220.  64^3 clustered 30.6 -> 6.5 ms, 128^3 lattice 52.9 ->
  // 12.3, zoom set 347 -> 68; error against 64 bits unchanged (1.4e-14).
  __device__ __forceinline__ bool pair_eval64(const WalkArgs& A, const Stage& St, const Smem& M, int i, int s,
                                              bool wrap, double (&acc)[3]) const {
    double d0 = M.tx[0][i] - St.sx[0][s], d1 = M.tx[1][i] - St.sx[1][s], d2 = M.tx[2][i] - St.sx[2][s];
    if (wrap) {
      d0 = mi64(d0, A.box);
      d1 = mi64(d1, A.box);
      d2 = mi64(d2, A.box);
    }
    const double r2 = fma(d0, d0, fma(d1, d1, d2 * d2));
    // positive doubles order like their bits
    const long long rb = __double_as_longlong(r2);
    if (rb >= A.rc2_lo_bits && St.id[s] >= 0 && !(rb <= A.rc2_hi_bits && norm2_64(d0, d1, d2) < A.rc2_64)) return false;
    const long long hb = max(__double_as_longlong(M.th2[i]), __double_as_longlong(St.sh2[s]));
    double r, K;
    float uf;
    if (rb < hb || (uint32_t)(rb >> 52) - 923u > 200u) {  // softened, or r^2 outside 2^-100 .. 2^101
      const double hh = sqrt(__longlong_as_double(hb));
      r = sqrt(r2);
      uf = (float)(r * A.inv2rs64);
      if (r >= hh) {
        K = 1.0 / (r * r * r);
      } else {
        const double v = r / hh;
        const double h3 = 1.0 / (hh * hh * hh);
        if (v < 0.5) K = h3 * (32.0 / 3.0 + v * v * (32.0 * v - 38.4));
        else K = h3 * (64.0 / 3.0 - 48.0 * v + 38.4 * v * v - (32.0 / 3.0) * v * v * v - (1.0 / 15.0) / (v * v * v));
      }
    } else {
      // conversions on the integer pipe
      const float r2f = __uint_as_float((uint32_t)((rb >> 29) - (896ll << 23)));
      const float yf = rsqrt_approx(r2f);
      const double y = __longlong_as_double(((long long)__float_as_uint(yf) << 29) + (896ll << 52));
      const double e = fma(-(r2 * y), y, 1.0);
      const double y1 = fma(y * e, fma(e, 0.375, 0.5), y);
      r = r2 * y1;
      K = y1 * y1 * y1;
      uf = r2f * yf * A.inv2rs;
    }
    const double sc = St.sm[s] * (K * short_range_f64(r * A.inv2rs64, uf));
    acc[0] = fma(sc, d0, acc[0]);
    acc[1] = fma(sc, d1, acc[1]);
    acc[2] = fma(sc, d2, acc[2]);
    return true;
  }

  // Start fetching slot s of queue entry e: its two 16-byte records go to
  // this lane's place in the staging buffer, asynchronously in the FP32 walk.
  __device__ __forceinline__ void fetch(const WalkArgs& A, const WarpBufs& W, Stage& St, int e, int s, int lane,
                                        Fetch& f) const {
    const int4 Q = W.queue[e];
    const bool node = Q.y < 0;
    const int j = node ? Q.x : Q.x + (s - W.qoff[e]);
    const float4* pa = (node ? A.T.nA : A.T.pA) + j;
    const float4* pb = (node ? A.T.nB : A.T.pB) + j;
    f.id = node ? -2 - j : j;
    f.q = (uint32_t)Q.z;
    if constexpr (F64) {
      f.a = *pa;
      f.b = *pb;
    } else {
      cp_async16(&St.ra[lane], pa);
      cp_async16(&St.rb[lane], pb);
    }
  }

  // The fetched source, once arrived: shifted to its image nearest to the
  // group centre (x: its position relative to that centre), and whether it
  // can have a pair inside the cut with some target of the group (its
  // distance to the padded group box within the conservative threshold).
  // uni: that image is the minimum image of every target of the group that
  // it can have such a pair with.
  __device__ __forceinline__ bool arrive(const WalkArgs& A, const Stage& St, int lane, const GroupInfo& G, Fetch& f,
                                         float (&x)[3], bool& uni) const {
    if constexpr (!F64) {
      cp_async_wait();
      f.a = St.ra[lane];
      f.b = St.rb[lane];
    }
    x[0] = f.a.x - G.cx;
    x[1] = f.a.y - G.cy;
    x[2] = f.a.z - G.cz;
    const float n0 = round1(x[0]), n1 = round1(x[1]), n2 = round1(x[2]);
    f.a.x -= n0;
    f.a.y -= n1;
    f.a.z -= n2;
    x[0] = (x[0] - n0) + f.b.x;
    x[1] = (x[1] - n1) + f.b.y;
    x[2] = (x[2] - n2) + f.b.z;
    const float a0 = fabsf(x[0]), a1 = fabsf(x[1]), a2 = fabsf(x[2]);
    uni = fmaxf(a0 + G.ex, fmaxf(a1 + G.ey, a2 + G.ez)) < A.uni_lim;
    if (F64) f.shifted = n0 != 0.f || n1 != 0.f || n2 != 0.f;
    const float g0 = fmaxf(a0 - G.ex, 0.f), g1 = fmaxf(a1 - G.ey, 0.f), g2 = fmaxf(a2 - G.ez, 0.f);
    return fmaf(g0, g0, fmaf(g1, g1, g2 * g2)) <= A.grp_rc2;
  }

  // Stage a fetched source in slot pos.
  // FP64 variant, filter form: (-2 x, -2 y, -2 z, |x|^2 - r_cut^2 - margin)
  // relative to the group centre, so |x_i - x_j|^2 - r_cut^2 - margin
  // evaluates as fW + |x_i|^2 + fX x_i + fY y_i + fZ z_i.  The FP32 evaluation
  // of that chain is within 18 u (|x_i| + |x_j|)^2 + 18 u r_cut^2 of the exact
  // value (u = 2^-24); the margin is 64 u times that bound's bracket, so every
  // pair inside the cut gives a negative value.
  __device__ __forceinline__ void put(const WalkArgs& A, Stage& S, Smem& M, const Fetch& f, int pos,
                                      const float (&x)[3], bool uni, int64_t gbase, float Rg) const {
    if constexpr (!F64) {
      const int e = 4 * (pos >> 1) + (pos & 1);  // this slot's first word of its pair's 16 bytes
      float* p0 = &S.s0[0].x + e;
      float* p1 = &S.s1[0].x + e;
      float* p2 = &S.s2[0].x + e;
      float* p3 = &S.s3[0].x + e;
      p0[0] = -f.a.x;
      p0[2] = -f.a.y;
      p1[0] = -f.a.z;
      p1[2] = -f.a.w;
      p2[0] = -f.b.x;
      p2[2] = -f.b.y;
      p3[0] = -f.b.z;
      p3[2] = f.b.w;
    } else {
      float fx = 0.f, fy = 0.f, fz = 0.f, fw = -1e30f;  // accepted node or per-pair image: always a candidate
      if (uni && f.id >= 0) {
        const float sj = fmaf(x[0], x[0], fmaf(x[1], x[1], x[2] * x[2]));
        const float rr = sqrtf(sj) + Rg;
        fx = -2.f * x[0];
        fy = -2.f * x[1];
        fz = -2.f * x[2];
        fw = (sj - A.rc2_hi) - 3.814697265625e-06f * fmaf(rr, rr, A.rc2_hi);
      }
      const int64_t j = f.id >= 0 ? f.id : -2 - f.id;
      const double* sp = f.id >= 0 ? A.T.x64 : A.T.com64;
#pragma unroll
      for (int c = 0; c < 3; ++c) S.sx[c][pos] = sp[3 * j + c];
      S.sm[pos] = -(f.id >= 0 ? A.T.m64 : A.T.mass64)[j];
      const double h = (f.id >= 0 ? A.T.h64 : A.T.hmax64)[j];
      S.sh2[pos] = h * h;
      S.fX[pos] = fx;
      S.fY[pos] = fy;
      S.fZ[pos] = fz;
      S.fW[pos] = fw;
    }
    S.id[pos] = f.id;
    S.sq[pos] = f.q;
    if (f.id >= gbase && f.id < gbase + kGroup) M.self[f.id - gbase] = pos;
  }

  __device__ __forceinline__ void fold() {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      kahan_add(S[c], C[c], P[c]);
      P[c] = 0.f;
      if constexpr (FUSED) {
        kahan_add(Sf[c], Cf[c], Pf[c]);
        Pf[c] = 0.f;
      }
    }
  }

  // Evaluate the queued entries (see the header comment).
  template <bool WILD>
  __device__ void evaluate(const WalkArgs& A, const WarpBufs& W, Stage& St, Smem& M, int nq, int lane,
                           const GroupInfo& G, const float4* SGB, int64_t gbase, uint32_t vmask, float Rg) {
    const int total = queue_offsets(A, W, nq, lane);
    if (total < 0) {
      if (lane == 0) set_status(A.wsb, ST_TREELINK);
      return;
    }
    const uint32_t lt = (1u << lane) - 1u;
    M.self[lane] = -1;
    __syncwarp();
    // slots are fetched 32 at a time and the survivors of the box test are
    // appended to the staged ones
    // Each window of 32 slots finds its slots' entries without a search:
    // ecur holds the window's first slot, the entries starting inside the
    // window set bit (start - rb) of one OR-reduced mask (an entry holds at
    // least one slot, so at most 31 start inside it), and slot rb + l lies
    // in entry ecur + (number of starts at or before bit l).
    // The next window is fetched while the current one is staged and evaluated.
    int pend = 0;
    // some staged source has no image common to the whole group (FP64 variant:
    // or one that is not its stored position)
    bool mi = false;
    int ecur = 0;
    Fetch cur = {};
    auto window = [&](int rb, Fetch& f) {
      const int ek = ecur + 1 + lane;
      const int sk = ek < nq ? W.qoff[ek] - rb : 32;
      const uint32_t starts = __reduce_or_sync(0xffffffffu, (sk > 0 && sk < 32) ? (1u << sk) : 0u);
      if (rb + lane < total) fetch(A, W, St, ecur + __popc(starts & ((2u << lane) - 1u)), rb + lane, lane, f);
      // the entry holding the following window's first slot
      const int en = ecur + __popc(starts);
      ecur = en + (en + 1 < nq && W.qoff[en + 1] == rb + 32 ? 1 : 0);
    };
    window(0, cur);
#pragma unroll 1
    for (int rb = 0; rb < total; rb += 32) {
      bool uni = true;
      float x[3] = {0.f, 0.f, 0.f};
      const bool kp = rb + lane < total && arrive(A, St, lane, G, cur, x, uni);
      const uint32_t km = __ballot_sync(0xffffffffu, kp);
      if (kp) put(A, St, M, cur, pend + __popc(km & lt), x, uni, gbase, Rg);
      mi = mi || __any_sync(0xffffffffu, kp && (!uni || (F64 && cur.shifted)));
      pend += __popc(km);
      if (rb + 32 < total) window(rb + 32, cur);
      __syncwarp();
      if (pend > 0 && (pend > kStage - 32 || rb + 32 >= total)) {
        if constexpr (F64) {
#pragma unroll 1
          for (int hb = 0; hb < pend; hb += 32) batch_list(A, W, St, M, hb, min(pend - hb, 32), lane, vmask, mi);
        } else if constexpr (WILD) {
          batch_wild(A, St, M, pend, lane, gbase + lane, mi);
        } else {
          batch_tiles(A, W, St, M, SGB, pend, lane, gbase, vmask, mi);
        }
        pend = 0;
        mi = false;
      }
    }
  }

  // Conservative cut test of this lane's target against the slots s and
  // s + 1 .. s + 3 of the filter arrays, two per instruction; a result's sign
  // bit is set where the pair can lie inside the cut.
  struct Filter {
    unsigned long long X2, Y2, Z2, S2;
    __device__ __forceinline__ void four(const Stage& St, int s, unsigned long long& r01,
                                         unsigned long long& r23) const {
      const float4 fx = *reinterpret_cast<const float4*>(St.fX + s);
      const float4 fy = *reinterpret_cast<const float4*>(St.fY + s);
      const float4 fz = *reinterpret_cast<const float4*>(St.fZ + s);
      const float4 fw = *reinterpret_cast<const float4*>(St.fW + s);
      r01 = add2(pack2(fw.x, fw.y), S2);
      r23 = add2(pack2(fw.z, fw.w), S2);
      r01 = fma2(pack2(fz.x, fz.y), Z2, r01);
      r23 = fma2(pack2(fz.z, fz.w), Z2, r23);
      r01 = fma2(pack2(fy.x, fy.y), Y2, r01);
      r23 = fma2(pack2(fy.z, fy.w), Y2, r23);
      r01 = fma2(pack2(fx.x, fx.y), X2, r01);
      r23 = fma2(pack2(fx.z, fx.w), X2, r23);
    }
  };
  __device__ __forceinline__ Filter filter() const {
    return {pack2(xr[0], xr[0]), pack2(xr[1], xr[1]), pack2(xr[2], xr[2]), pack2(sr, sr)};
  }

  // One target against one slot pair: displacements, squared distances and
  // -mass, packed over the pair's two slots.
  struct Pair {
    unsigned long long dx, dy, dz, r2, nm;
    float h20, h21;  // softening: max of the target's and the source's h^2
  };
  // A sub-group's target as this lane holds it, each component twice.
  struct Target {
    unsigned long long x, y, z, u, v, w;  // hi and lo parts
    unsigned long long wx, wy, wz;        // adjoint: dL/da
    float h2;
  };
  // Packed sums of this lane's pairs with its target, even and odd slots.
  struct Sums {
    unsigned long long ax, ay, az;  // target side: the force, or m J w in the adjoint
    unsigned long long bx, by, bz;  // fused: the force
  };

  __device__ __forceinline__ Pair load_pair(const Stage& St, const Target& T, int k, bool mi) const {
    const float4 v0 = St.s0[k], v1 = St.s1[k], v2 = St.s2[k], v3 = St.s3[k];
    Pair p;
    p.dx = add2(T.x, pack2(v0.x, v0.y));
    p.dy = add2(T.y, pack2(v0.z, v0.w));
    p.dz = add2(T.z, pack2(v1.x, v1.y));
    if (mi) {
      p.dx = pack2(mi1(lo2(p.dx)), mi1(hi2(p.dx)));
      p.dy = pack2(mi1(lo2(p.dy)), mi1(hi2(p.dy)));
      p.dz = pack2(mi1(lo2(p.dz)), mi1(hi2(p.dz)));
    }
    p.dx = add2(p.dx, add2(T.u, pack2(v2.x, v2.y)));
    p.dy = add2(p.dy, add2(T.v, pack2(v2.z, v2.w)));
    p.dz = add2(p.dz, add2(T.w, pack2(v3.x, v3.y)));
    p.r2 = fma2(p.dx, p.dx, fma2(p.dy, p.dy, mul2(p.dz, p.dz)));
    p.nm = pack2(v1.z, v1.w);
    p.h20 = fmaxf(T.h2, v3.z);
    p.h21 = fmaxf(T.h2, v3.w);
    return p;
  }

  // Adds a pair with force factors F (zero for a slot that is no hit) to the
  // lane's sums and, in the adjoint, to the slots' sums.  own: this lane's
  // slot pair is its own (lanes past the end of the list repeat the last one).
  __device__ __forceinline__ void add_pair(Smem& M, const Target& T, const Pair& p, unsigned long long F,
                                           unsigned long long Fr, int k, bool own, int lane, Sums& S) const {
    if constexpr (!ADJ) {
      const unsigned long long sc = mul2(p.nm, F);
      S.ax = fma2(sc, p.dx, S.ax);
      S.ay = fma2(sc, p.dy, S.ay);
      S.az = fma2(sc, p.dz, S.az);
    } else {
      const unsigned long long dw = fma2(p.dx, T.wx, fma2(p.dy, T.wy, mul2(p.dz, T.wz)));
      const unsigned long long qq = mul2(Fr, dw);
      // J w and F d.w; the source side takes their negatives
      const unsigned long long j0 = fma2(F, T.wx, mul2(qq, p.dx));
      const unsigned long long j1 = fma2(F, T.wy, mul2(qq, p.dy));
      const unsigned long long j2 = fma2(F, T.wz, mul2(qq, p.dz));
      const unsigned long long js = mul2(F, dw);
      S.ax = fma2(p.nm, j0, S.ax);
      S.ay = fma2(p.nm, j1, S.ay);
      S.az = fma2(p.nm, j2, S.az);
      if constexpr (FUSED) {
        const unsigned long long sc = mul2(p.nm, F);
        S.bx = fma2(sc, p.dx, S.bx);
        S.by = fma2(sc, p.dy, S.by);
        S.bz = fma2(sc, p.dz, S.bz);
      }
      // sum over the 8 targets: each step exchanges half of the values with
      // the partner lane, so that lane (k, t) ends with one of the eight sums
      // (slot 2k + bit 2 of t, component t & 3)
      const bool s2 = lane & 4, s1 = lane & 2, s0 = lane & 1;
      float c0 = s2 ? hi2(j0) : lo2(j0), c1 = s2 ? hi2(j1) : lo2(j1);
      float c2 = s2 ? hi2(j2) : lo2(j2), c3 = s2 ? hi2(js) : lo2(js);
      c0 += __shfl_xor_sync(0xffffffffu, s2 ? lo2(j0) : hi2(j0), 4);
      c1 += __shfl_xor_sync(0xffffffffu, s2 ? lo2(j1) : hi2(j1), 4);
      c2 += __shfl_xor_sync(0xffffffffu, s2 ? lo2(j2) : hi2(j2), 4);
      c3 += __shfl_xor_sync(0xffffffffu, s2 ? lo2(js) : hi2(js), 4);
      float d0 = s1 ? c2 : c0, d1 = s1 ? c3 : c1;
      d0 += __shfl_xor_sync(0xffffffffu, s1 ? c0 : c2, 2);
      d1 += __shfl_xor_sync(0xffffffffu, s1 ? c1 : c3, 2);
      float v = s0 ? d1 : d0;
      v += __shfl_xor_sync(0xffffffffu, s0 ? d0 : d1, 1);
      if (own) (&M.SG[0].x)[8 * k + (lane & 7)] -= v;
    }
  }

  // Outside the softening length and below the cut band: the packed form holds.
  __device__ __forceinline__ bool plain(const WalkArgs& A, float r2, float h2) const {
    return r2 < A.pp_lo && r2 >= h2;
  }

  // The packed force factors of both slots, zero where h0 / h1 is false.
  __device__ __forceinline__ void force_pair(const WalkArgs& A, const Pair& p, bool h0, bool h1,
                                             unsigned long long& F, unsigned long long& Fr) const {
    const unsigned long long ri = pack2(rsqrt_approx(lo2(p.r2)), rsqrt_approx(hi2(p.r2)));
    const unsigned long long r = mul2(p.r2, ri);
    const unsigned long long ri2 = mul2(ri, ri);
    const unsigned long long K = mul2(ri2, ri);
    const unsigned long long ea = mul2(p.r2, pack2(A.ex2c, A.ex2c));
    const unsigned long long ex = pack2(ex2_approx(lo2(ea)), ex2_approx(hi2(ea)));
    const unsigned long long f = mul2(sr_poly2(fma2(r, pack2(A.t_scale, A.t_scale), pack2(-1.0f, -1.0f))), ex);
    F = mul2(K, f);
    F = pack2(h0 ? lo2(F) : 0.f, h1 ? hi2(F) : 0.f);
    if constexpr (ADJ) {
      // F'/r = (K'/r) f + K f'/r, K'/r = -3 K / r^2, f'(r)/r = fp_c r exp(-u^2)
      Fr = fma2(mul2(mul2(pack2(-3.0f, -3.0f), K), ri2), f, mul2(K, mul2(mul2(pack2(A.fp_c, A.fp_c), ex), r)));
      Fr = pack2(h0 ? lo2(Fr) : 0.f, h1 ? hi2(Fr) : 0.f);
    }
  }

  // A pair the packed form does not cover: the exact cut (an accepted node is
  // inside by decision, a particle in the band is decided in FP64), then the
  // force with the softened kernel.  False if outside the cut.
  __device__ __forceinline__ bool force_rare(const WalkArgs& A, const Stage& St, int64_t i, int s, float r2, float h2,
                                             float& F, float& Fr) const {
    if (!(r2 < A.pp_lo)) {
      const int id = St.id[s];
      if (id >= 0 && !pair_inside_exact(A, i, id)) return false;
    }
    force_f32<ADJ>(A, r2, h2, F, Fr);
    return true;
  }

  // Adjoint: a source's sums into its accumulators (id: particle, or -2 - node).
  static __device__ __forceinline__ void add_source(const WalkArgs& A, int id, const float4& g) {
    double* Gd = id >= 0 ? A.Gp + 3 * (int64_t)id : A.Gn + 3 * (int64_t)(-2 - id);
    double* Sd = id >= 0 ? A.Sp + id : A.Sn + (-2 - id);
    atomicAdd(Gd, f2d_exact(g.x));
    atomicAdd(Gd + 1, f2d_exact(g.y));
    atomicAdd(Gd + 2, f2d_exact(g.z));
    atomicAdd(Sd, f2d_exact(g.w));
  }

  // The tiles add every listed pair, those that are no hits with a factor of
  // zero, which clears the term only while its operands are finite: dL/da up to
  // kWildWeight (three products with displacements below 1 stay below FLT_MAX) and
  // masses that do not overflow FP32.  A warp with others evaluates its batches
  // here, hit by hit: lane = target, slot after slot.
  static constexpr float kWildWeight = 1e38f;
  __device__ void batch_wild(const WalkArgs& A, const Stage& St, Smem& M, int cnt, int lane, int64_t i, bool mi) {
    const float4 ta = M.tA[lane], tb = M.tB[lane];
    const int so = M.self[lane];
#pragma unroll 1
    for (int s = 0; s < cnt; ++s) {
      const int e = 4 * (s >> 1) + (s & 1);
      const float* p0 = &St.s0[0].x + e;
      const float* p1 = &St.s1[0].x + e;
      const float* p2 = &St.s2[0].x + e;
      const float* p3 = &St.s3[0].x + e;
      float d0 = ta.x + p0[0], d1 = ta.y + p0[2], d2 = ta.z + p1[0];
      if (mi) {
        d0 = mi1(d0);
        d1 = mi1(d1);
        d2 = mi1(d2);
      }
      d0 += tb.x + p2[0];
      d1 += tb.y + p2[2];
      d2 += tb.z + p3[0];
      const float r2 = fmaf(d0, d0, fmaf(d1, d1, d2 * d2));
      const int id = St.id[s];
      float v[4] = {0.f, 0.f, 0.f, 0.f};
      if (((St.sq[s] >> lane) & 1u) && s != so && r2 <= A.pp_hi &&
          (r2 < A.pp_lo || id < 0 || pair_inside_exact(A, i, id))) {
        float F, Fr;
        force_f32<ADJ>(A, r2, fmaxf(ta.w, p3[2]), F, Fr);
        ++nint;
        const float nm = p1[2], sc = nm * F;
        float(&f)[3] = ADJ ? Pf : P;
        f[0] = fmaf(sc, d0, f[0]);
        f[1] = fmaf(sc, d1, f[1]);
        f[2] = fmaf(sc, d2, f[2]);
        if constexpr (ADJ) {
          const float4 w = M.tW[lane];
          const float dw = fmaf(d0, w.x, fmaf(d1, w.y, d2 * w.z));
          const float qq = Fr * dw;
          v[0] = fmaf(F, w.x, qq * d0);
          v[1] = fmaf(F, w.y, qq * d1);
          v[2] = fmaf(F, w.z, qq * d2);
          v[3] = F * dw;
#pragma unroll
          for (int c = 0; c < 3; ++c) P[c] = fmaf(nm, v[c], P[c]);
        }
      }
      if constexpr (ADJ) {
#pragma unroll
        for (int o = 1; o < 32; o <<= 1)
#pragma unroll
          for (int c = 0; c < 4; ++c) v[c] += __shfl_xor_sync(0xffffffffu, v[c], o);
        if (lane == 0) add_source(A, id, make_float4(-v[0], -v[1], -v[2], -v[3]));
      }
    }
    M.self[lane] = -1;
    fold();
    __syncwarp();
  }

  // One FP32 batch: the cnt staged sources, as pairs of adjacent slots.
  //
  // Tile: a warp iteration takes the 8 targets of one sub-group against 4
  // slot pairs (8 sources), lane = (pair of the four, target of the eight),
  // each lane both sources of its pair in packed arithmetic.  A sub-group
  // lists the slot pairs with a source inside the cut of its box.  The 8
  // targets lie close together and adjacent slots come from one leaf, so
  // about half of the 64 (target, source) pairs of an iteration are hits
  // (a third of a whole group's would be).  A target's sum stays in
  // registers over the sub-group's iterations and is reduced over its four
  // lanes once per batch.  Measured against listing the pairs one by one,
  // 32 per iteration, with a segmented scan for the sums (full lanes, but the
  // list, the gathered operands and the scan cost two thirds of the pair
  // work): forward 3.17 -> 2.56 ms on the 128^3 lattice, 23.2 -> 18.5 ms on the
  // 128^3 clustered set, 0.66 -> 0.36 ms on 4096 particles (one group per SM);
  // adjoint 4.61 -> 3.73 and 33.3 -> 25.0 ms.  The next list entry is read
  // ahead; loading its pair ahead as well costs 4 % (19.2 and 2.68 ms forward,
  // 27.3 against 25.3 ms with both directions in one walk).
  __device__ void batch_tiles(const WalkArgs& A, const WarpBufs& W, Stage& St, Smem& M, const float4* SGB,
                              int cnt, int lane, int64_t gbase, uint32_t vmask, bool mi) {
    const uint2 qq = *reinterpret_cast<const uint2*>(St.sq + 2 * lane);
    const bool has0 = 2 * lane < cnt, has1 = 2 * lane + 1 < cnt;
    const uint32_t q0 = has0 ? qq.x : 0u, q1 = has1 ? qq.y : 0u;
    // lane = slot pair: the sub-groups within reach of either slot's source
    // (the source's distance to the padded box; the exact cut is taken per
    // pair), listed per sub-group
    unsigned char* list = reinterpret_cast<unsigned char*>(W.list);
    const uint32_t lt = (1u << lane) - 1u;
    const float reach2 = mi ? 8.0f : A.grp_rc2;  // without a common image every pair is listed
    uint32_t U = 0;  // slot pairs listed for this lane's sub-group
    {
      const float4 v0 = St.s0[lane], v1 = St.s1[lane];
#pragma unroll
      for (int g = 0; g < kSub; ++g) {
        const float4 c4 = SGB[2 * g], e4 = SGB[2 * g + 1];
        const unsigned long long x = add2(pack2(c4.x, c4.x), pack2(v0.x, v0.y));
        const unsigned long long y = add2(pack2(c4.y, c4.y), pack2(v0.z, v0.w));
        const unsigned long long z = add2(pack2(c4.z, c4.z), pack2(v1.x, v1.y));
        const unsigned long long gx = pack2(fmaxf(fabsf(lo2(x)) - e4.x, 0.f), fmaxf(fabsf(hi2(x)) - e4.x, 0.f));
        const unsigned long long gy = pack2(fmaxf(fabsf(lo2(y)) - e4.y, 0.f), fmaxf(fabsf(hi2(y)) - e4.y, 0.f));
        const unsigned long long gz = pack2(fmaxf(fabsf(lo2(z)) - e4.z, 0.f), fmaxf(fabsf(hi2(z)) - e4.z, 0.f));
        const unsigned long long g2 = fma2(gx, gx, fma2(gy, gy, mul2(gz, gz)));
        const uint32_t gm = 0xffu << (8 * g);
        const bool in0 = (q0 & gm) != 0u && lo2(g2) <= reach2;
        const bool in1 = (q1 & gm) != 0u && hi2(g2) <= reach2;
        const uint32_t um = __ballot_sync(0xffffffffu, in0 || in1);
        if ((um >> lane) & 1u) list[32 * g + __popc(um & lt)] = (unsigned char)lane;
        if ((lane >> 3) == g) U = um;
      }
    }
    // bit k of m0 / m1: slot 2k / 2k + 1 holds a source of this lane's target
    uint32_t m0, m1;
    if (__any_sync(0xffffffffu, (has0 && q0 != vmask) || (has1 && q1 != vmask))) {
      m0 = transpose32<ADJ ? 5 : 1>(q0, lane);
      m1 = transpose32<ADJ ? 5 : 1>(q1, lane);
    } else {
      m0 = valid ? low_bits((cnt + 1) >> 1) : 0u;
      m1 = valid ? low_bits(cnt >> 1) : 0u;
    }
    const int so = M.self[lane];
    if (so >= 0) {
      const uint32_t others = ~(1u << (so >> 1));
      if (so & 1) m1 &= others;
      else m0 &= others;
    }
    __syncwarp();  // every lane has read its slot pair
    // an odd count leaves the last pair's second slot empty: its data must be finite
    if ((cnt & 1) && lane < 8) {
      float4* p = lane < 2 ? &St.s0[cnt >> 1] : lane < 4 ? &St.s1[cnt >> 1] : lane < 6 ? &St.s2[cnt >> 1] : &St.s3[cnt >> 1];
      (&p->x)[2 * (lane & 1) + 1] = 0.f;
    }
    __syncwarp();
#pragma unroll 1
    for (int g = 0; g < kSub; ++g) {
      const int n = __popc(__shfl_sync(0xffffffffu, U, 8 * g));
      if (n == 0) continue;
      const int t = 8 * g + (lane & 7);
      const uint32_t q0m = __shfl_sync(0xffffffffu, m0, t), q1m = __shfl_sync(0xffffffffu, m1, t);
      int hits = 0;
      Target T;
      {
        const float4 ta = M.tA[t], tb = M.tB[t];
        T.x = pack2(ta.x, ta.x); T.y = pack2(ta.y, ta.y); T.z = pack2(ta.z, ta.z);
        T.u = pack2(tb.x, tb.x); T.v = pack2(tb.y, tb.y); T.w = pack2(tb.z, tb.z);
        T.h2 = ta.w;
        if constexpr (ADJ) {
          const float4 w = M.tW[t];
          T.wx = pack2(w.x, w.x); T.wy = pack2(w.y, w.y); T.wz = pack2(w.z, w.z);
        }
      }
      Sums S = {0, 0, 0, 0, 0, 0};
      uint32_t rare = 0u;  // bit i: iteration i of the list holds a pair the packed form does not cover
      // the next iteration's list entry is read ahead
      int kn = list[32 * g + min(lane >> 3, n - 1)];
#pragma unroll 1
      for (int e0 = 0; e0 < n; e0 += 4) {
        const int e = e0 + (lane >> 3);
        const int k = kn;
        kn = list[32 * g + min(e + 4, n - 1)];
        const Pair p = load_pair(St, T, k, mi);
        const bool h0 = e < n && ((q0m >> k) & 1u) && lo2(p.r2) <= A.pp_hi;
        const bool h1 = e < n && ((q1m >> k) & 1u) && hi2(p.r2) <= A.pp_hi;
        const bool p0 = h0 && plain(A, lo2(p.r2), p.h20), p1 = h1 && plain(A, hi2(p.r2), p.h21);
        if (h0 != p0 || h1 != p1) rare |= 1u << (e0 >> 2);
        hits += (p0 ? 1 : 0) + (p1 ? 1 : 0);
        unsigned long long F, Fr = 0;
        force_pair(A, p, p0, p1, F, Fr);
        add_pair(M, T, p, F, Fr, k, e < n, lane, S);
      }
      rare = __reduce_or_sync(0xffffffffu, rare);
#pragma unroll 1
      while (rare) {
        const int e0 = 4 * (__ffs(rare) - 1);
        rare &= rare - 1u;
        const int e = e0 + (lane >> 3);
        const int k = list[32 * g + min(e, n - 1)];
        const Pair p = load_pair(St, T, k, mi);
        float F[2] = {0.f, 0.f}, Fr[2] = {0.f, 0.f};
#pragma unroll 1
        for (int c = 0; c < 2; ++c) {
          const float r2 = c ? hi2(p.r2) : lo2(p.r2), h2 = c ? p.h21 : p.h20;
          const bool h = e < n && (((c ? q1m : q0m) >> k) & 1u) && r2 <= A.pp_hi;
          float f = 0.f, fr = 0.f;
          if (h && !plain(A, r2, h2) && force_rare(A, St, gbase + t, 2 * k + c, r2, h2, f, fr)) ++hits;
          if (c) { F[1] = f; Fr[1] = fr; }
          else { F[0] = f; Fr[0] = fr; }
        }
        add_pair(M, T, p, pack2(F[0], F[1]), pack2(Fr[0], Fr[1]), k, e < n, lane, S);
      }
      // the target's sum over its four lanes (even and odd slots first)
      float p0 = lo2(S.ax) + hi2(S.ax), p1 = lo2(S.ay) + hi2(S.ay), p2 = lo2(S.az) + hi2(S.az);
      p0 += __shfl_xor_sync(0xffffffffu, p0, 8);
      p1 += __shfl_xor_sync(0xffffffffu, p1, 8);
      p2 += __shfl_xor_sync(0xffffffffu, p2, 8);
      p0 += __shfl_xor_sync(0xffffffffu, p0, 16);
      p1 += __shfl_xor_sync(0xffffffffu, p1, 16);
      p2 += __shfl_xor_sync(0xffffffffu, p2, 16);
      hits += __shfl_xor_sync(0xffffffffu, hits, 8);
      hits += __shfl_xor_sync(0xffffffffu, hits, 16);
      if ((lane >> 3) == g) {
        nint += hits;
        P[0] = p0;
        P[1] = p1;
        P[2] = p2;
      }
      if constexpr (FUSED) {
        float f0 = lo2(S.bx) + hi2(S.bx), f1 = lo2(S.by) + hi2(S.by), f2 = lo2(S.bz) + hi2(S.bz);
        f0 += __shfl_xor_sync(0xffffffffu, f0, 8);
        f1 += __shfl_xor_sync(0xffffffffu, f1, 8);
        f2 += __shfl_xor_sync(0xffffffffu, f2, 8);
        f0 += __shfl_xor_sync(0xffffffffu, f0, 16);
        f1 += __shfl_xor_sync(0xffffffffu, f1, 16);
        f2 += __shfl_xor_sync(0xffffffffu, f2, 16);
        if ((lane >> 3) == g) {
          Pf[0] = f0;
          Pf[1] = f1;
          Pf[2] = f2;
        }
      }
      __syncwarp();  // the slots' sums of this sub-group before the next one's
    }
    M.self[lane] = -1;
    fold();
    if constexpr (ADJ) {
#pragma unroll 1
      for (int u = 0; u < 2; ++u) {
        const int s = lane + 32 * u;
        const float4 g = M.SG[s];
        if (s < cnt && (g.x != 0.f || g.y != 0.f || g.z != 0.f || g.w != 0.f)) {
          add_source(A, St.id[s], g);
        }
        M.SG[s] = make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
    __syncwarp();
  }

  // One FP64 batch: the cnt staged sources at slots [hb, hb + cnt).  The FP64
  // pipe runs a warp instruction at the same cost however few lanes are
  // active (16 cycles of the SM), so the hit pairs are listed target by target
  // and each lane evaluates an equal share of consecutive pairs.  A run of
  // one target's pairs sums in the lane's registers; the lane in which the run
  // begins stores its part, the lanes that continue it keep theirs aside, and
  // the target's owner adds them in lane order: three FP64 additions a
  // target where a segmented scan took fifteen an iteration.
  __device__ void batch_list(const WalkArgs& A, const WarpBufs& W, Stage& St, Smem& M, int hb, int cnt, int lane,
                             uint32_t vmask, bool wrap) {
    // bit s of msk: slot s is in this lane's part of its entry's lane mask
    const bool has = lane < cnt;
    const uint32_t q = has ? St.sq[hb + lane] : 0u;
    uint32_t msk;
    if (__any_sync(0xffffffffu, has && q != vmask)) msk = transpose32<1>(q, lane);
    else msk = valid ? low_bits(cnt) : 0u;
    // conservative cut test for all 32 slots; the sign bit of each result is
    // shifted into acc (slot 0 ends up at bit 31)
    uint32_t acc = 0;
    const Filter f = filter();
#pragma unroll
    for (int s = 0; s < kSlots; s += 4) {
      unsigned long long r01, r23;
      f.four(St, hb + s, r01, r23);
      acc = __funnelshift_l((uint32_t)r01, acc, 1);
      acc = __funnelshift_l((uint32_t)(r01 >> 32), acc, 1);
      acc = __funnelshift_l((uint32_t)r23, acc, 1);
      acc = __funnelshift_l((uint32_t)(r23 >> 32), acc, 1);
    }
    uint32_t hit = __brev(acc) & msk;
    const int so = M.self[lane];
    const bool self_here = so >= hb && so < hb + cnt;
    if (self_here) hit &= ~(1u << (so - hb));
    const int nhit = (int)__reduce_add_sync(0xffffffffu, (unsigned)__popc(hit));
    // a batch with more pairs than the list holds is processed in two
    // halves of its slots (at most 32 x 16 pairs each)
    const bool split = nhit > kList;
#pragma unroll 1
    for (int part = 0; part < (split ? 2 : 1); ++part) {
      const uint32_t hp = split ? (hit & (part == 0 ? 0x0000ffffu : 0xffff0000u)) : hit;
      // compaction: target-major pair list
      const int c = __popc(hp);
      int incl = c;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      const int T = __shfl_sync(0xffffffffu, incl, 31);
      const int off = incl - c;
      {
        uint32_t m = hp;
        int t = off;
        while (m) {
          const int s = __ffs(m) - 1;
          m &= m - 1;
          W.list[t++] = (unsigned short)((lane << 5) | s);
        }
      }
      nint += c;  // listed pairs; those outside the exact cut are subtracted below
      __syncwarp();
      if (T == 0) continue;
      const int share = (T + 31) >> 5;  // consecutive pairs of each lane
      const int p0 = lane * share, p1 = min(p0 + share, T);
      int cur = p0 < T ? W.list[p0] >> 5 : -1;               // target of the run being summed
      bool head = p0 > 0 && p0 < T && (W.list[p0 - 1] >> 5) == cur;  // it began in an earlier lane
      double sum[3] = {0.0, 0.0, 0.0};
#pragma unroll 1
      for (int u = 0; u < share; ++u) {
        const int p = p0 + u;
        if (p < p1) {
          const int e = W.list[p];
          const int i = e >> 5;
          if (i != cur) {
#pragma unroll
            for (int a = 0; a < 3; ++a) {
              if (head) M.Hd[a][lane] = sum[a];
              else M.Ps[a][cur] = sum[a];
              sum[a] = 0.0;
            }
            head = false;
            cur = i;
          }
          if (!pair_eval64(A, St, M, i, hb + (e & 31), wrap, sum)) atomicAdd(&M.fneg[i], 1);
        }
      }
      if (p0 < T) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          if (head) M.Hd[a][lane] = sum[a];
          else M.Ps[a][cur] = sum[a];
        }
      }
      __syncwarp();
      if (c > 0) {
        // the run began in lane off / share and goes on in those after it
        const int l1 = (off + c - 1) / share;
        double s0 = M.Ps[0][lane], s1 = M.Ps[1][lane], s2 = M.Ps[2][lane];
        for (int l = off / share + 1; l <= l1; ++l) {
          s0 += M.Hd[0][l];
          s1 += M.Hd[1][l];
          s2 += M.Hd[2][l];
        }
        a64[0] += s0;
        a64[1] += s1;
        a64[2] += s2;
      }
      __syncwarp();
    }
    nint -= M.fneg[lane];
    M.fneg[lane] = 0;
    // this batch held the target's own slot
    if (self_here) M.self[lane] = -1;
    __syncwarp();
  }

  __device__ void finish(const WalkArgs& A) {
    if (!valid) return;
    const int32_t i = A.T.order[k];
    if (F64) {
#pragma unroll
      for (int c = 0; c < 3; ++c) A.accd[3 * (int64_t)i + c] = a64[c];
      if (A.counts) A.counts[i] = nint;
    } else if (!ADJ) {
#pragma unroll
      for (int c = 0; c < 3; ++c) A.accf[3 * (int64_t)i + c] = S[c] - C[c];
      if (A.counts) A.counts[i] = nint;
    } else {
#pragma unroll
      for (int c = 0; c < 3; ++c) A.tgt[3 * k + c] = (double)S[c] - (double)C[c];
      if constexpr (FUSED) {
#pragma unroll
        for (int c = 0; c < 3; ++c) A.accf[3 * (int64_t)i + c] = Sf[c] - Cf[c];
        if (A.counts) A.counts[i] = nint;
      }
    }
  }
};

template <bool ADJ>
using LaneF32 = LaneFP<ADJ, false>;
using LaneF64 = LaneFP<false, true>;
using LaneFused = LaneFP<true, false, true>;

// ------------------------------------------------------------------ traversal

template <class Lane>
union WarpScratch {
  MixedScratch mix;
  typename Lane::Stage stage;
};

// Shared memory of a warp.
template <class Lane>
struct WalkShared {
  int2 stack[kStack];
  int4 queue[kQueue];
  int qoff[kQueue + 1];
  unsigned short list[Lane::kListSize];
  WarpScratch<Lane> scr;
  typename Lane::Smem lane;
  float4 sgb[2 * kSub];
};

// The walk of this warp's group.  Without WILD it returns true, having done
// nothing, if the group needs the variant with it (batch_wild).
template <class Lane, int kWarpsPerBlock, bool WILD>
__device__ __forceinline__ bool walk_groups(const WalkArgs& A, WalkShared<Lane>& S) {
  const TreeDev& T = A.T;
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  // 2^split warps serve a group, each its part of the targets
  const int64_t v = (int64_t)blockIdx.x * kWarpsPerBlock + wib;
  const int64_t gi = A.g_begin + (v >> A.split);
  if (gi >= A.g_end) return false;
  const bool usable = T.sb->status == 0 && T.sb->magic == kMagicTree;
  const int64_t g = A.ordered && usable ? group_at(T, Lane::kOrder, gi, A.wsb) : gi;
  const bool mine = (lane >> (5 - A.split)) == (int)(v & ((1 << A.split) - 1));
  if (!usable) {
    // a failed or missing tree: flag it and give every output of this
    // group's targets NaN, so that nothing downstream can take stale values
    // for forces.  A tree whose build started wrote its permutation first;
    // for one that was never built the sorted index stands in for it.
    if (lane == 0) set_status(A.wsb, ST_NOTREE);
    const int64_t kk = g * kGroup + lane;
    if (mine && kk < T.n) {
      const float nf = __int_as_float(0x7fc00000);
      const double nd = __longlong_as_double(0x7ff8000000000000ll);
      int64_t io = kk;
      if (T.sb->magic == kMagicTree) {
        const int64_t o = T.order[kk];
        if (o >= 0 && o < T.n) io = o;
      }
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        if (A.accf) A.accf[3 * io + c] = nf;
        if (A.accd) A.accd[3 * io + c] = nd;
        if (A.tgt) A.tgt[3 * kk + c] = nd;
      }
      if (A.counts) A.counts[io] = -1;
    }
    return false;
  }
  WarpBufs W;
  W.stack = S.stack;
  W.queue = S.queue;
  W.qoff = S.qoff;
  W.list = S.list;
  MixedScratch& X = S.scr.mix;
  typename Lane::Stage& St = S.scr.stage;
  typename Lane::Smem& M = S.lane;
  int nodes_total = 0;
#pragma unroll 1
  for (int l = 0; l < kLevels; ++l) nodes_total += T.sb->level_cnt[l];
  if (nodes_total > T.cap) nodes_total = (int)T.cap;

  const int64_t gbase = g * kGroup;
  const int64_t k = gbase + lane;
  const bool valid = mine && k < T.n;
  const uint32_t vmask = __ballot_sync(0xffffffffu, valid);
  if (vmask == 0u) return false;  // a part beyond the last particle
  const uint32_t lt = (1u << lane) - 1u;

  // boxes of this warp's targets and of the 4 sub-groups of 8 targets (box
  // units, padded outward by more than the FP32 rounding of a position in
  // [0, 1))
  GroupInfo G;
  float4* SGB = S.sgb;
  {
    const float4 pa = T.pA[valid ? k : 0], pb = T.pB[valid ? k : 0];
    float lo[3] = {pa.x + pb.x, pa.y + pb.y, pa.z + pb.z};
    float hi[3] = {lo[0], lo[1], lo[2]};
    if (!valid) {
#pragma unroll
      for (int c = 0; c < 3; ++c) { lo[c] = 1e30f; hi[c] = -1e30f; }
    }
#pragma unroll 1
    for (int o = 1; o < 32; o <<= 1) {
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        lo[c] = fminf(lo[c], __shfl_xor_sync(0xffffffffu, lo[c], o));
        hi[c] = fmaxf(hi[c], __shfl_xor_sync(0xffffffffu, hi[c], o));
      }
      G.cx = 0.5f * (lo[0] + hi[0]); G.cy = 0.5f * (lo[1] + hi[1]); G.cz = 0.5f * (lo[2] + hi[2]);
      G.ex = 0.5f * (hi[0] - lo[0]) * 1.0001f + 2e-7f;
      G.ey = 0.5f * (hi[1] - lo[1]) * 1.0001f + 2e-7f;
      G.ez = 0.5f * (hi[2] - lo[2]) * 1.0001f + 2e-7f;
      if (o == 4 && (lane & 7) == 0) {
        SGB[2 * (lane >> 3)] = make_float4(G.cx, G.cy, G.cz, 0.f);
        SGB[2 * (lane >> 3) + 1] = make_float4(G.ex, G.ey, G.ez, 0.f);
      }
    }
  }
  // bound on |x_i - group centre| for the FP64 variant's cut filter
  const float Rg = sqrtf(fmaf(G.ex, G.ex, fmaf(G.ey, G.ey, G.ez * G.ez))) * 1.0001f + 1e-6f;

  Lane L;
  if (L.init(A, M, k, valid, lane, G) && !WILD) return true;

  if (lane == 0) W.stack[0] = make_int2((int)(1u << 28), (int)vmask);  // the root: node 0, one node
  int sp = 1, nq = 0;
  long long visits = 0;
  __syncwarp();
  for (;;) {
    if (sp > 0 && nq <= kQueue - kQueueNeed) {
      if (sp > kStack - kStackNeed) {
        if (lane == 0) set_status(A.wsb, ST_STACK);
        break;
      }
      // Pop whole child ranges from the top until up to 32 nodes are gathered
      // (one range when the stack is deep).  The index is clamped so no lane
      // forms an address outside the stack, and every pop completes before
      // any push.
      const int m = sp > min(A.deep, kDeep) ? 1 : min(sp, 32);
      const int2 E = W.stack[max(sp - 1 - lane, 0)];
      __syncwarp();
      const uint32_t ex = (uint32_t)E.x;
      const int rcnt = lane < m ? (int)(ex >> 28) : 0;
      const int rfirst_l = (int)(ex & 0x0fffffffu);
      if (__any_sync(0xffffffffu, lane < m && (rcnt < 1 || rcnt > 8))) {
        if (lane == 0) set_status(A.wsb, ST_TREELINK);
        break;
      }
      int incl = rcnt;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      const int take = __popc(__ballot_sync(0xffffffffu, lane < m && incl <= 32));  // >= 4 ranges or all
      const int total = __shfl_sync(0xffffffffu, incl, take - 1);
      sp -= take;
      visits += total;
      if (visits > A.max_iters) {
        if (lane == 0) set_status(A.wsb, ST_WALKCAP);
        break;
      }
      // lane s takes node s of the gathered ranges: r = ranges ending at or before s
      int r = 0;
#pragma unroll
      for (int b = 16; b > 0; b >>= 1) {
        const int cand = r + b;
        const int v = __shfl_sync(0xffffffffu, incl, (cand - 1) & 31);
        if (cand <= take && v <= lane) r = cand;
      }
      // every lane executes the shuffle (a full-mask shuffle reached by only
      // some lanes is undefined); the value is selected afterwards
      const int prev = __shfl_sync(0xffffffffu, incl, (r - 1) & 31);
      const int excl = r > 0 ? prev : 0;
      const int rfirst = __shfl_sync(0xffffffffu, rfirst_l, r & 31);
      const uint32_t mask = (uint32_t)__shfl_sync(0xffffffffu, E.y, r & 31);
      const bool has = lane < total;
      const int node = has ? rfirst + (lane - excl) : 0;
      if (__any_sync(0xffffffffu, has && (node < 0 || node >= nodes_total))) {
        if (lane == 0) set_status(A.wsb, ST_TREELINK);
        break;
      }
      const int nc = has ? node : 0;
      const float4 NC = T.nC[nc];
      const int4 ND = T.nD[nc];
      const float4 NA = T.nA[nc];
      const float4 NB = T.nB[nc];
      const int cls = has ? classify(A, G, NC, NA, NB) : CL_NONE;
      const bool leaf = meta_leaf(ND.w);
      const int nch = meta_nchild(ND.w);
      bool bad = false;
      if (has && cls != CL_DROP) {
        if (leaf) bad = ND.x < 0 || ND.y < 1 || (int64_t)ND.x + ND.y > T.n;
        else bad = nch <= 0 || nch > 8 || ND.z <= node || ND.z + nch > nodes_total;
      }
      if (__any_sync(0xffffffffu, bad)) {
        if (lane == 0) set_status(A.wsb, ST_TREELINK);
        break;
      }
      // OPEN internal nodes: push their child range with the same lanes
      const bool push = cls == CL_OPEN && !leaf;
      const uint32_t pm = __ballot_sync(0xffffffffu, push);
      if (push) W.stack[sp + __popc(pm & lt)] = make_int2((int)((uint32_t)ND.z | ((uint32_t)nch << 28)), (int)mask);
      sp += __popc(pm);
      // OPEN leaves and ACCEPTed nodes: queue them for evaluation
      const bool q = (cls == CL_OPEN && leaf) || cls == CL_ACCEPT;
      const uint32_t qm = __ballot_sync(0xffffffffu, q);
      if (q)
        W.queue[nq + __popc(qm & lt)] =
            cls == CL_ACCEPT ? make_int4(node, -1, (int)mask, 0) : make_int4(ND.x, ND.y, (int)mask, 0);
      nq += __popc(qm);
      // MIXED nodes: decisions for the targets in their masks, OR-ed into
      // per-node accept / open masks
      const uint32_t mm = __ballot_sync(0xffffffffu, cls == CL_MIXED);
      if (mm) {
        const int nm = __popc(mm);
        if (cls == CL_MIXED) {
          const int ix = __popc(mm & lt);
          float sx, sy, sz;
          const bool uni = node_image(A, G, NC, sx, sy, sz);
          float4 SC = NC, SA = NA;
          if (uni) {
            SC.x -= sx; SC.y -= sy; SC.z -= sz;
            SA.x -= sx; SA.y -= sy; SA.z -= sz;
          }
          X.node[ix] = node;
          X.fl[ix] = uni ? 1 : 0;
          X.D[ix] = ND;
          X.C[ix] = SC;
          X.A[ix] = SA;
          X.B[ix] = NB;
          X.mask[ix] = mask & vmask;
          X.acc[ix] = 0u;
          X.open[ix] = 0u;
        }
        __syncwarp();
        // each (node, sub-group) pair is first classified against the
        // sub-group's box; the undecided ones are listed
        int nd = 0;
#pragma unroll 1
        for (int j0 = 0; j0 < kSub * nm; j0 += 32) {
          const int j = j0 + lane;
          const int ix = j >> 2, g = j & 3;
          int cg = CL_NONE;
          const uint32_t gm = j < kSub * nm ? X.mask[ix] & (0xffu << (8 * g)) : 0u;
          if (gm) {
            const float4 c4 = SGB[2 * g], e4 = SGB[2 * g + 1];
            GroupInfo Gs;
            Gs.cx = c4.x; Gs.cy = c4.y; Gs.cz = c4.z;
            Gs.ex = e4.x; Gs.ey = e4.y; Gs.ez = e4.z;
            cg = classify(A, Gs, X.C[ix], X.A[ix], X.B[ix]);
            if (cg == CL_OPEN) atomicOr(&X.open[ix], gm);
            else if (cg == CL_ACCEPT) atomicOr(&X.acc[ix], gm);
          }
          const uint32_t um = __ballot_sync(0xffffffffu, cg == CL_MIXED);
          if (cg == CL_MIXED) W.list[nd + __popc(um & lt)] = (unsigned short)j;
          nd += __popc(um);
        }
        __syncwarp();
        // per-target decisions, four listed (node, sub-group) pairs at a
        // time: lane = (pair of the four, target of the eight)
#pragma unroll 1
        for (int d0 = 0; d0 < nd; d0 += 4) {
          const int d = d0 + (lane >> 3);
          const int j = W.list[min(d, nd - 1)];
          const int ix = j >> 2, t = 8 * (j & 3) + (lane & 7);
          int dec = DEC_DISCARD;
          if (d < nd && ((X.mask[ix] >> t) & 1u))
            dec = decide_f32(A, gbase + t, M.tA[t], M.tB[t], X.node[ix], meta_level(X.D[ix].w), X.C[ix], X.A[ix],
                             X.B[ix], X.fl[ix] != 0);
          const uint32_t da = (__ballot_sync(0xffffffffu, dec == DEC_ACCEPT) >> (lane & 24)) & 0xffu;
          const uint32_t dn = (__ballot_sync(0xffffffffu, dec == DEC_OPEN) >> (lane & 24)) & 0xffu;
          if ((lane & 7) == 0) {
            if (da) atomicOr(&X.acc[ix], da << (8 * (j & 3)));
            if (dn) atomicOr(&X.open[ix], dn << (8 * (j & 3)));
          }
        }
        __syncwarp();
        const bool hm = lane < nm;
        const int hx = hm ? lane : 0;
        const uint32_t am = hm ? X.acc[hx] : 0u;
        const uint32_t om = hm ? X.open[hx] : 0u;
        const int4 XD = X.D[hx];
        const int xnode = X.node[hx];
        const bool xleaf = meta_leaf(XD.w);
        const bool qa = am != 0u, qo = om != 0u && xleaf, po = om != 0u && !xleaf;
        const uint32_t ba = __ballot_sync(0xffffffffu, qa);
        const uint32_t bo = __ballot_sync(0xffffffffu, qo);
        const uint32_t bp = __ballot_sync(0xffffffffu, po);
        if (qa) W.queue[nq + __popc(ba & lt)] = make_int4(xnode, -1, (int)am, 0);
        nq += __popc(ba);
        if (qo) W.queue[nq + __popc(bo & lt)] = make_int4(XD.x, XD.y, (int)om, 0);
        nq += __popc(bo);
        if (po)
          W.stack[sp + __popc(bp & lt)] =
              make_int2((int)((uint32_t)XD.z | ((uint32_t)meta_nchild(XD.w) << 28)), (int)om);
        sp += __popc(bp);
      }
      __syncwarp();
    } else if (nq > 0) {
      L.template evaluate<WILD>(A, W, St, M, nq, lane, G, SGB, gbase, vmask, Rg);
      nq = 0;
      __syncwarp();
    } else {
      break;
    }
  }
  L.finish(A);
  if (A.total) {
    const unsigned cnt = __reduce_add_sync(0xffffffffu, (unsigned)(valid ? L.nint : 0));
    if (lane == 0 && cnt) atomicAdd(A.total, (unsigned long long)cnt);
  }
  return false;
}

// Not inlined, so that the walk of all other groups keeps its registers.
template <class Lane, int kWarpsPerBlock>
__device__ __noinline__ void walk_wild(const WalkArgs& A, WalkShared<Lane>& S) {
  walk_groups<Lane, kWarpsPerBlock, true>(A, S);
}
template <class Lane, int kWarpsPerBlock>
__device__ __forceinline__ void walk_block(const WalkArgs& A) {
  __shared__ WalkShared<Lane> s_walk[kWarpsPerBlock];
  WalkShared<Lane>& S = s_walk[threadIdx.x >> 5];
  const bool wild = walk_groups<Lane, kWarpsPerBlock, false>(A, S);
  if constexpr (!std::is_same<Lane, LaneF64>::value)
    if (wild) walk_wild<Lane, kWarpsPerBlock>(A, S);
}

// Forward walks of many groups run 18 warps an SM, in blocks of one (96
// registers); the others 16, in blocks of two (118 to 128 registers), whose groups
// are neighbours and share their sources in L1.  Forward, ms, blocks of two / one:
// lattice 128^3 2.55 / 2.36, clustered 128^3 17.1 / 15.7, 256^3 405 / 368, 90^3 (22,782
// groups) 3.61 / 3.43; 5860 groups (zoom) 12.7 / 12.4, 128 groups 0.217 / 0.233.  Adjoint
// 128^3 clustered 22.8 / 24.2: its code fits the instruction cache less well.  The
// FP64 walk, which shares little in L1 for its arithmetic, runs 15 in blocks of
// one (shared memory, 14 KB a warp and 1 KB a block): of two groups in a block one
// waits for the other.  16 in blocks of two / 15 in blocks of one: 64^3 lattice
// 1.90 / 1.81 ms, clustered 58^3 5.3 / 5.0, 64^3 6.5 / 6.35; zoom 68.6 / 69.2.
constexpr int64_t kManyGroups = 24576;

template <class Lane>
__global__ void __launch_bounds__(64) k_walk(WalkArgs A) {
  walk_block<Lane, 2>(A);
}
template <class Lane, int kBlocks>
__global__ void __launch_bounds__(32, kBlocks) k_walk_one(WalkArgs A) {
  walk_block<Lane, 1>(A);
}

// Warps per group (log2).  A walk of fewer groups than the chip holds warps
// leaves it idle, and one of a few times as many waits for its longest groups;
// two or four warps a group, each with its part of the targets and its own
// traversal, shorten them for some repeated traversal.  It depends on the
// tree alone, so a walk over a range of groups gives the full walk's sums.
// Measured, ms with 1 / 2 / 4 warps a group, forward: 128 groups (4096
// uniform) 0.37 / 0.27 / 0.22, 1024 groups (32^3) clustered 0.30 / 0.26 / 0.23,
// zoom 3.38 / 2.37 / 2.48, lattice 0.15 / 0.13 / 0.15; 5860 groups (zoom) 12.4 /
// 13.8 / 17.2; 8192 groups (64^3) lattice 0.41 / 0.48 / 0.62, clustered 1.35 /
// 1.16 / 1.37.  FP64: 128 groups 1.58 / 0.94 / 0.67, 1024 clustered 1.50 / 1.04 /
// 0.80, zoom 7.5 / 7.1 / 8.7, lattice 0.38 / 0.36 / 0.42; 5860 (zoom) 67.5 / 69.5 /
// 80.6, 8192 clustered 6.4 / 5.8 / 6.4, lattice 1.81 / 1.90 / 2.27.  Between 1024 and
// 5860 groups nothing was measured.
static int walk_split(int64_t n_groups) { return n_groups <= 1024 ? 2 : n_groups <= 4096 ? 1 : 0; }

cudaError_t launch_walk(WalkArgs A, int prec, bool adjoint, cudaStream_t s, bool fused) {
  A.split = walk_split(A.T.ngroups);
  A.ordered = A.g_begin == 0 && A.g_end == A.T.ngroups;
  const int64_t warps = (A.g_end - A.g_begin) << A.split;
  if (warps <= 0) return cudaSuccess;
  const unsigned pairs = (unsigned)((warps + 1) / 2);
  if (fused) k_walk<LaneFused><<<pairs, 64, 0, s>>>(A);
  else if (adjoint) k_walk<LaneF32<true>><<<pairs, 64, 0, s>>>(A);
  else if (prec == OG_FP64) k_walk_one<LaneF64, 15><<<(unsigned)warps, 32, 0, s>>>(A);
  else if (A.T.ngroups >= kManyGroups) k_walk_one<LaneF32<false>, 18><<<(unsigned)warps, 32, 0, s>>>(A);
  else k_walk<LaneF32<false>><<<pairs, 64, 0, s>>>(A);
  return cudaGetLastError();
}

}  // namespace og
