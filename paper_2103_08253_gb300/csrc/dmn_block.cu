// The CTA organisation of the FP64 Newton iteration: k_newton_block and its launch.
//
// Newton's method of Sec. 3.2 with the FP64 step obtained by iterative refinement.  GB300 runs FP64 at
// 1/64 of its FP32 rate, and 152 k of the 183 kflop of an FP64 pass (depth 8) are the condensation that
// only serves to solve J da = -R.  Here each iteration
//   A  evaluates strains, leaf laws and the residual R in FP64 (and tests the criterion on it),
//   S  condenses the leaf tangents in FP32 and solves for da1 (relative error some 1e-6),
//   B  forms R + J da1 with pairs of FP32 numbers (about 46 bits) and solves again in FP32 for da2,
// and applies da = da1 + da2, whose relative error is the product of the two solves' (1e-11, at most
// some 1e-10 on the workloads' plastic paths).  Where a large step ends in a fixed set of plastic leaves, or in none,
// no quadratic term hides what the solves left of its linear residual: a residual no larger than that is taken off
// by a second part of the same step, which is not counted, also below the criterion (an elastic point's stress is
// then 5e-16 from the exact one as with the all-FP64 solve, 5e-14 without).  Below the criterion and with all leaves
// elastic it keeps the condensed tangents, solves once, R alone, and ends with the jumps, without S and another A
// (155000 elastic points of depth 8: 62.4 -> 54.7 ms, 52.2 without the second part).  So the iterates
// are those of the all-FP64 condensation, with its iteration counts.  A costs about 21 k FP64 instructions, a
// pass of the all-FP64 kernel 122 k; S and B cost none.  The tangent comes from one FP64
// sweep at the converged jumps, as in the mixed form.
//
// A point for which the FP32 solve does not contract (|R + J da1| > REFINE_MAX |R|: tangents near
// singular, moduli outside the FP32 range), which is not finite or which has not converged within BLOCK_ITERS
// corrections is put on a list (status RETRY) and updated from its start by the
// all-FP64 kernels, so that every call keeps their results and statuses.
//
// Components.  Strains are engineering, stresses, tangents and flow directions tensor components (Voigt): N(n) has
// the bare components of n, which saves the 6 multiplications per laminate of the Mandel form's 1 / sqrt 2.  The
// leaf tangents are formed in pairs.  Depth 8 compressed, 20001 points: 10.7 -> 9.7 ms; 8 points: 0.45 -> 0.42.
//
// Organisation.  A CTA of 256 threads holds 256 / S points, S = 2^(K-3) threads per point: thread (s, p)
// owns the s-th subtree of depth 3 (7 laminates, 8 leaves) of the point in slot p and, for s >= 1, the
// laminate s of the top K - 3 levels (heap number).  Subtrees run depth first in registers; the top
// levels run level by level, the strains (down) and results (up) handed over in shared memory.  All
// per-laminate data is laid out [field][laminate][thread], so that every access is coalesced whatever
// the tree's depth, with p fastest: a warp's lanes run the same instructions.  The top levels' laminates
// lie on different warps (laminate h on warp h P / 32), which balances the SM's four FP64 units.
// Every slot runs its own Newton iteration: a converged point is written out and its slot takes the next
// one, so uneven iteration counts do not idle the CTA.
#include <cuda_runtime.h>

#include "../../include/dmn.h"
#include "dmn_block.cuh"

namespace dmn {

namespace {

constexpr float REFINE_MAX = 1e-3f;
// A residual this many times what the solves left of the last step's linear system, or less, belongs to that step
constexpr double LEFT_MAX = 4.0;
// and is taken off also where it meets the criterion, unless it is at the rounding of FP64 stresses (times the root's)
constexpr double ROUNDING = 1e-15;
// What the second solve leaves at least, as a part of the residual it starts from: the pairs' 46 bits, less some for
// the sums that cancel.  (Without it elastic points at criteria of 1e-15 took a counted correction more than with
// the all-FP64 solve.)
constexpr double PAIR_LEFT = 9.1e-13;   // 2^-40
constexpr int BLOCK_ITERS = 16;

// scratch fields of a thread, in units of 8 laminates (7 of the subtree, then the top laminate)
enum { D_A = 0, D_N = 3, D_A2 = 6 };                                               // FP64 (D_A2: line search)
enum { F_H = 0, F_K = 18, F_G = 24, F_D = 27, F_T = 30, F_TL = 33, F_END = 36 };   // FP32

// Pairs of FP32 numbers, value h + l (Dekker 1971: error-free sum and product): a sum costs 8 FP32
// instructions, a product 4, against 64 cycles of the FP64 unit for a warp's FP64 instruction.
struct pair {
  float h, l;
};
__device__ __forceinline__ pair add(pair a, pair b) {
  const float s = __fadd_rn(a.h, b.h), t = __fsub_rn(s, a.h);
  const float e = __fadd_rn(__fsub_rn(a.h, __fsub_rn(s, t)), __fsub_rn(b.h, t));
  return {s, __fadd_rn(e, __fadd_rn(a.l, b.l))};
}
__device__ __forceinline__ pair neg(pair a) { return {-a.h, -a.l}; }
__device__ __forceinline__ pair mul(pair a, float b) {
  const float p = __fmul_rn(a.h, b);
  return {p, __fmaf_rn(a.l, b, __fmaf_rn(a.h, b, -p))};
}
__device__ __forceinline__ pair mul(pair a, pair b) {
  const float p = __fmul_rn(a.h, b.h);
  return {p, __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.l, __fmaf_rn(a.h, b.h, -p)))};
}
// x as a pair, with integer instructions (as narrow_rn): h the 24 leading bits truncated, l the 29 bits
// below them.  Magnitudes below FP32's normal range give 0 (l: below 2^-74), above it infinity.
__device__ __forceinline__ pair split(double x) {
  const unsigned long long b = bits_of(x);
  const unsigned hi = (unsigned)(b >> 32), lo = (unsigned)b, sign = hi & 0x80000000u, e = (hi >> 20) & 0x7ffu;
  unsigned h = ((e - 896u) << 23) + (((hi & 0xfffffu) << 3) | (lo >> 29));
  if (e <= 896u) h = 0u;
  if (e >= 1151u) h = 0x7f800000u;
  const float l = e > 948u && e < 1151u ? __uint2float_rn(lo & 0x1fffffffu) * float_of((e - 948u) << 23) : 0.f;
  return {float_of(sign | h), float_of(sign | bits_of(l))};
}

}  // namespace

// flags of a slot
enum { B_ACT = 1, B_FIRST = 4, B_CONT = 8, B_CONV = 16, B_CUR = 32, B_LAST = 64 };

// The Newton kernel for CTAs of BT threads.  A point's results do not depend on BT, bit for bit.
template <int BT>
struct Block {

struct Ctx {
  double* D;      // this thread's FP64 scratch: field f of laminate j at D[(8 f + j) BT]
  float* F;       // this thread's FP32 scratch
  double* z;      // leaf states: z[(6 leaf + c) BT]
  float* tan;     // leaf tangents mu, c, m as pairs: h at tan[(16 leaf + k) BT], l at tan[(16 leaf + 8 + k) BT]
  __device__ double& d(int f, int j) const { return D[(8 * f + j) * BT]; }
  __device__ float& f(int f, int j) const { return F[(8 * f + j) * BT]; }
};

static __device__ __forceinline__ void load3(const Ctx& c, int f, int j, double v[3]) {
#pragma unroll
  for (int k = 0; k < 3; ++k) v[k] = c.d(f + k, j);
}
static __device__ __forceinline__ void normal32(const Ctx& c, int j, float n[3]) {
#pragma unroll
  for (int k = 0; k < 3; ++k) n[k] = narrow_rn(c.d(D_N + k, j));
}

// The FP32 step of laminate j, g + H de.
static __device__ __forceinline__ void step32(const Ctx& c, int j, const float de[6], float da[3]) {
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    float v = c.f(F_G + k, j);
#pragma unroll
    for (int I = 0; I < 6; ++I) v += c.f(F_H + 6 * k + I, j) * de[I];
    da[k] = v;
  }
}

// A, downwards: the jumps of laminate j corrected (apply) and the children's strains.  de: the FP32
// correction of the second solve handed down (dL, dR: to the children; NULL for leaves).
template <bool CMP, bool LS>
static __device__ __forceinline__ void down_a(const TreeDev& t, const Ctx& c, int h, int j, int a_in, int a_out, bool apply,
                                       double step, const double e[6], const float de[6], double eL[6], double eR[6],
                                       float* dL, float* dR) {
  const Lam<CMP> q(t, h);
  if (CMP && q.mode) {
#pragma unroll
    for (int I = 0; I < 6; ++I) { eL[I] = eR[I] = e[I]; if (dL) dL[I] = dR[I] = de[I]; }
    return;
  }
  double nd[3], a[3];
  load3(c, D_N, j, nd);
  load3(c, a_in, j, a);
  if (apply) {
    float da[3];
    step32(c, j, de, da);
    if (dL) {
      const float c1 = __ldg(t.c1f + q.id), c2 = __ldg(t.c2f + q.id);
      const float n[3] = {narrow_rn(nd[0]), narrow_rn(nd[1]), narrow_rn(nd[2])};
      float Nd[6];
      N_apply<float>(n, n, da, Nd);
#pragma unroll
      for (int I = 0; I < 6; ++I) { dL[I] = de[I] - c2 * Nd[I]; dR[I] = de[I] + c1 * Nd[I]; }
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const double s = widen(c.f(F_D + k, j)) + widen(da[k]);
      a[k] = LS ? a[k] + step * s : a[k] + s;
      c.d(a_out + k, j) = a[k];
    }
  } else {
    if (dL) {
#pragma unroll
      for (int I = 0; I < 6; ++I) dL[I] = dR[I] = 0.f;
    }
    if (LS) {
#pragma unroll
      for (int k = 0; k < 3; ++k) c.d(a_out + k, j) = a[k];
    }
  }
  double Na[6];
  N_apply<double>(nd, nd, a, Na);
#pragma unroll
  for (int I = 0; I < 6; ++I) { eL[I] = e[I] - q.c2 * Na[I]; eR[I] = e[I] + q.c1 * Na[I]; }
}

// The last solve's correction of laminate j's jumps (at f), and its strains in the children (as in down_a).
template <bool CMP>
static __device__ __forceinline__ void down_last(const TreeDev& t, const Ctx& c, int h, int j, int f, const float de[6],
                                          float* dL, float* dR) {
  const Lam<CMP> q(t, h);
  if (CMP && q.mode) {
    if (dL) {
#pragma unroll
      for (int I = 0; I < 6; ++I) dL[I] = dR[I] = de[I];
    }
    return;
  }
  float da[3];
  step32(c, j, de, da);
#pragma unroll
  for (int k = 0; k < 3; ++k) c.d(f + k, j) += widen(da[k]);
  if (!dL) return;
  const float c1 = __ldg(t.c1f + q.id), c2 = __ldg(t.c2f + q.id);
  float n[3], Nd[6];
  normal32(c, j, n);
  N_apply<float>(n, n, da, Nd);
#pragma unroll
  for (int I = 0; I < 6; ++I) { dL[I] = de[I] - c2 * Nd[I]; dR[I] = de[I] + c1 * Nd[I]; }
}

static __device__ __forceinline__ void pair_normal(const Ctx& c, int j, pair n[3]) {
#pragma unroll
  for (int k = 0; k < 3; ++k) n[k] = split(c.d(D_N + k, j));
}

// B, downwards: the step da1 of laminate j stored, and its strains in the children.  Without `first` there is no
// first solve: da1 = 0.
template <bool CMP>
static __device__ __forceinline__ void down_b(const TreeDev& t, const Ctx& c, int h, int j, bool first, const pair e[6],
                                       pair eL[6], pair eR[6]) {
  const Lam<CMP> q(t, h);
  if (CMP && q.mode) {
#pragma unroll
    for (int I = 0; I < 6; ++I) eL[I] = eR[I] = e[I];
    return;
  }
  float de[6], x[3] = {0.f, 0.f, 0.f};
#pragma unroll
  for (int I = 0; I < 6; ++I) de[I] = e[I].h;
  if (first) step32(c, j, de, x);
#pragma unroll
  for (int k = 0; k < 3; ++k) c.f(F_D + k, j) = x[k];
  pair n[3];
  pair_normal(c, j, n);
  const pair Nx[6] = {mul(n[0], x[0]), mul(n[1], x[1]), mul(n[2], x[2]), add(mul(n[2], x[1]), mul(n[1], x[2])),
                      add(mul(n[2], x[0]), mul(n[0], x[2])), add(mul(n[1], x[0]), mul(n[0], x[1]))};
  const pair c2 = split(-q.c2);
#pragma unroll
  for (int I = 0; I < 6; ++I) { eL[I] = add(e[I], mul(c2, Nx[I])); eR[I] = add(eL[I], Nx[I]); }   // c1 = 1 - c2
}

// A, upwards: residual of laminate j (t = N^T (s_R - s_L), stored) and the average stress.
template <bool CMP>
static __device__ __forceinline__ void up_a(const TreeDev& t, const Ctx& c, int h, int j, const double sL[6],
                                     const double sR[6], double sb[6], double& r2) {
  const Lam<CMP> q(t, h);
  if (CMP && q.mode) {
#pragma unroll
    for (int I = 0; I < 6; ++I) sb[I] = q.mode == 2 ? sR[I] : sL[I];
    return;
  }
  double nd[3], u[3];
  load3(c, D_N, j, nd);
  double d[6];
#pragma unroll
  for (int I = 0; I < 6; ++I) { d[I] = sR[I] - sL[I]; sb[I] = sL[I] + q.c2 * d[I]; }
  Nt_apply<double>(nd, nd, d, u);
  const double sc = __ldg(t.sc + q.id);
  r2 += sc * sc * (u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const pair v = split(u[k]);
    c.f(F_T + k, j) = v.h;
    c.f(F_TL + k, j) = v.l;
  }
}

// B, upwards: the linearised residual of laminate j after da1, u = N^T (s_R - s_L) + N^T (tau_R - tau_L)
// in pairs, then the FP32 solve's upward half with the stored H and Kn^-1:
//   u += N^T (ds_R - ds_L),  g = -Kn^-1 u,  ds = c1 ds_L + c2 ds_R + c1 c2 H^T u.
// BOT: the children are leaves (ds = 0 there).
template <bool CMP, bool BOT>
static __device__ __forceinline__ void up_b(const TreeDev& t, const Ctx& c, int h, int j, const pair tL[6], const pair tR[6],
                                     const float dsL[6], const float dsR[6], pair tb[6], float ds[6], float& r2) {
  const Lam<CMP> q(t, h);
  if (CMP && q.mode) {
#pragma unroll
    for (int I = 0; I < 6; ++I) {
      tb[I] = q.mode == 2 ? tR[I] : tL[I];
      ds[I] = BOT ? 0.f : q.mode == 2 ? dsR[I] : dsL[I];
    }
    return;
  }
  pair n[3], d[6];
  pair_normal(c, j, n);
  const pair p2 = split(q.c2);
#pragma unroll
  for (int I = 0; I < 6; ++I) { d[I] = add(tR[I], neg(tL[I])); tb[I] = add(tL[I], mul(p2, d[I])); }
  const pair v[3] = {add(mul(n[0], d[0]), add(mul(n[2], d[4]), mul(n[1], d[5]))),
                     add(mul(n[1], d[1]), add(mul(n[2], d[3]), mul(n[0], d[5]))),
                     add(mul(n[2], d[2]), add(mul(n[1], d[3]), mul(n[0], d[4])))};
  float u[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const pair x = add(pair{c.f(F_T + k, j), c.f(F_TL + k, j)}, v[k]);
    u[k] = x.h + x.l;
  }
  const float sc = __ldg(t.scf + q.id), c2 = __ldg(t.c2f + q.id), c12 = __ldg(t.c12f + q.id);
#pragma unroll
  for (int k = 0; k < 3; ++k) r2 += (sc * u[k]) * (sc * u[k]);
  float dd[6];
  if (!BOT) {
    const float m[3] = {n[0].h, n[1].h, n[2].h};
    float w[3];
#pragma unroll
    for (int I = 0; I < 6; ++I) dd[I] = dsR[I] - dsL[I];
    Nt_apply<float>(m, m, dd, w);
#pragma unroll
    for (int k = 0; k < 3; ++k) u[k] += w[k];
  }
  float K[6];
#pragma unroll
  for (int k = 0; k < 6; ++k) K[k] = c.f(F_K + k, j);
  c.f(F_G, j) = -(K[0] * u[0] + K[1] * u[1] + K[2] * u[2]);
  c.f(F_G + 1, j) = -(K[1] * u[0] + K[3] * u[1] + K[4] * u[2]);
  c.f(F_G + 2, j) = -(K[2] * u[0] + K[4] * u[1] + K[5] * u[2]);
#pragma unroll
  for (int k = 0; k < 3; ++k) u[k] *= c12;
#pragma unroll
  for (int I = 0; I < 6; ++I) {
    float x = BOT ? 0.f : dsL[I] + c2 * dd[I];
#pragma unroll
    for (int k = 0; k < 3; ++k) x += c.f(F_H + 6 * k + I, j) * u[k];
    ds[I] = x;
  }
}

// S, upwards: FP32 condensation of laminate j (Sub without the FP64 stress).
struct Sub32 {
  float ds[6], C[21];
};

static __device__ __forceinline__ void solve32(const Ctx& c, int j, float c12, const float Ki[3][3], const float B[6][3],
                                        const float u[3], float ds[6], float C[21]) {
  float H[3][6], g[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
#pragma unroll
    for (int I = 0; I < 6; ++I) H[k][I] = -(Ki[k][0] * B[I][0] + Ki[k][1] * B[I][1] + Ki[k][2] * B[I][2]);
    g[k] = -(Ki[k][0] * u[0] + Ki[k][1] * u[1] + Ki[k][2] * u[2]);
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
#pragma unroll
    for (int I = 0; I < 6; ++I) c.f(F_H + 6 * k + I, j) = H[k][I];
    c.f(F_G + k, j) = g[k];
  }
  c.f(F_K, j) = Ki[0][0]; c.f(F_K + 1, j) = Ki[0][1]; c.f(F_K + 2, j) = Ki[0][2];
  c.f(F_K + 3, j) = Ki[1][1]; c.f(F_K + 4, j) = Ki[1][2]; c.f(F_K + 5, j) = Ki[2][2];
#pragma unroll
  for (int I = 0; I < 6; ++I) {
    const float b[3] = {c12 * B[I][0], c12 * B[I][1], c12 * B[I][2]};
    ds[I] += b[0] * g[0] + b[1] * g[1] + b[2] * g[2];
#pragma unroll
    for (int J = I; J < 6; ++J) C[sidx(I, J)] += b[0] * H[0][J] + b[1] * H[1][J] + b[2] * H[2][J];
  }
}

template <bool CMP>
static __device__ __forceinline__ void condense32(const TreeDev& t, const Ctx& c, int h, int j, const Sub32& L, const Sub32& R,
                                           Sub32& o) {
  const Lam<CMP> q(t, h);
  if (CMP && q.mode) {
    if (q.mode == 2) o = R; else o = L;
    return;
  }
  const float c2 = __ldg(t.c2f + q.id), c12 = __ldg(t.c12f + q.id);
  float n[3];
  normal32(c, j, n);
  float dC[21], Ch[21], X[6][3], B[6][3], u[3], w[3], dd[6];
#pragma unroll
  for (int k = 0; k < 21; ++k) { dC[k] = R.C[k] - L.C[k]; Ch[k] = R.C[k] - c2 * dC[k]; }
  SN_apply<float>(Ch, n, n, X);
  float Ki[3][3];
  {
    const float k00 = n[0] * X[0][0] + n[2] * X[4][0] + n[1] * X[5][0];
    const float k10 = n[1] * X[1][0] + n[2] * X[3][0] + n[0] * X[5][0];
    const float k20 = n[2] * X[2][0] + n[1] * X[3][0] + n[0] * X[4][0];
    const float k11 = n[1] * X[1][1] + n[2] * X[3][1] + n[0] * X[5][1];
    const float k21 = n[2] * X[2][1] + n[1] * X[3][1] + n[0] * X[4][1];
    const float k22 = n[2] * X[2][2] + n[1] * X[3][2] + n[0] * X[4][2];
    inv3_sym<float>(k00, k10, k20, k11, k21, k22, Ki);
  }
  SN_apply<float>(dC, n, n, B);
#pragma unroll
  for (int I = 0; I < 6; ++I) dd[I] = R.ds[I] - L.ds[I];
  Nt_apply<float>(n, n, dd, w);
#pragma unroll
  for (int k = 0; k < 3; ++k) u[k] = c.f(F_T + k, j) + w[k];
#pragma unroll
  for (int I = 0; I < 6; ++I) o.ds[I] = L.ds[I] + c2 * dd[I];
#pragma unroll
  for (int k = 0; k < 21; ++k) o.C[k] = L.C[k] + c2 * dC[k];
  solve32(c, j, c12, Ki, B, u, o.ds, o.C);
}

// leaf tangent in FP32: the phase's constants or the stored mu, c, m
static __device__ __forceinline__ void leaf_tan32(const PhaseDev& ph, const float* s, LeafTan<float>& D) {
  if (ph.kind == 0) {
    D.lam = ph.lamf; D.mu = ph.Gf; D.c = 0.f;
#pragma unroll
    for (int I = 0; I < 6; ++I) D.m[I] = 0.f;
  } else {
    D.mu = s[0]; D.c = s[BT];
    D.lam = ph.f.K - (float)(2.0 / 3.0) * D.mu;
#pragma unroll
    for (int I = 0; I < 6; ++I) D.m[I] = s[(2 + I) * BT];
  }
}

// the structured condensation of a bottom laminate (condense_bottom); a side passed on keeps its leaf's tangent
template <bool CMP>
static __device__ __forceinline__ void condense32_bottom(const TreeDev& t, const Ctx& c, int h, int j,
                                                  const LeafTan<float>& L, const LeafTan<float>& R, bool elL, bool elR,
                                                  Sub32& o) {
  const Lam<CMP> q(t, h);
#pragma unroll
  for (int I = 0; I < 6; ++I) o.ds[I] = 0.f;
  float c1, c2;
  if (CMP && q.mode) { c2 = q.mode == 2 ? 1.f : 0.f; c1 = 1.f - c2; }
  else { c1 = __ldg(t.c1f + q.id); c2 = __ldg(t.c2f + q.id); }
  // the average of the two tangents
  const float lam = c1 * L.lam + c2 * R.lam, mu2 = 2.f * (c1 * L.mu + c2 * R.mu);
  const float wL = c1 * L.c, wR = c2 * R.c;
#pragma unroll
  for (int I = 0; I < 6; ++I) {
    const float hL = wL * L.m[I], hR = wR * R.m[I];
#pragma unroll
    for (int J = I; J < 6; ++J) {
      float v = I < 3 && J < 3 ? lam : 0.f;
      if (I == J) v += I < 3 ? mu2 : 0.5f * mu2;
      if (!elL) v -= hL * L.m[J];
      if (!elR) v -= hR * R.m[J];
      o.C[sidx(I, J)] = v;
    }
  }
  if (CMP && q.mode) return;
  const float c12 = __ldg(t.c12f + q.id);
  float n[3];
  normal32(c, j, n);
  const float a = c2 * L.mu + c1 * R.mu, b = c2 * (L.lam + L.mu) + c1 * (R.lam + R.mu);
  const float dlam = R.lam - L.lam, dmu2 = 2.f * (R.mu - L.mu), dld = dlam + dmu2;
  float k[3][3], B[6][3];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int l = i; l < 3; ++l) k[i][l] = b * n[i] * n[l] + (i == l ? a : 0.f);
#pragma unroll
  for (int I = 0; I < 6; ++I)
#pragma unroll
    for (int l = 0; l < 3; ++l)
      B[I][l] = I < 3 ? (I == l ? dld : dlam) * n[l] : (N_nonzero(I, l) ? 0.5f * dmu2 * N_entry<float>(n, n, I, l) : 0.f);
  if (!elL) {
    float v[3];
    Nt_apply<float>(n, n, L.m, v);
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int l = i; l < 3; ++l) k[i][l] -= (c2 * L.c) * v[i] * v[l];
#pragma unroll
    for (int I = 0; I < 6; ++I)
#pragma unroll
      for (int l = 0; l < 3; ++l) B[I][l] += (L.c * L.m[I]) * v[l];
  }
  if (!elR) {
    float v[3];
    Nt_apply<float>(n, n, R.m, v);
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int l = i; l < 3; ++l) k[i][l] -= (c1 * R.c) * v[i] * v[l];
#pragma unroll
    for (int I = 0; I < 6; ++I)
#pragma unroll
      for (int l = 0; l < 3; ++l) B[I][l] -= (R.c * R.m[I]) * v[l];
  }
  float Ki[3][3];
  inv3_sym<float>(k[0][0], k[0][1], k[0][2], k[1][1], k[1][2], k[2][2], Ki);
  const float u[3] = {c.f(F_T, j), c.f(F_T + 1, j), c.f(F_T + 2, j)};
  solve32(c, j, c12, Ki, B, u, o.ds, o.C);
}

// A, the leaf: stress from the strain e and the state z (shear entries times 1 / sqrt 2), the law of leaf_iso in
// Voigt components; the tangent mu, c, m for S and B goes to T as pairs, formed in pairs from FP64 xi, 1 / |xi| and
// k2.  An elastic leaf's tangent is its phase's.  Returns whether the leaf is plastic.
static __device__ __forceinline__ bool leaf_a(const PhaseDev& ph, const double e[6], const double* zp, double sig[6], float* T) {
  const double tr = e[0] + e[1] + e[2];
  if (ph.kind == 0) {
    const double lt = ph.lam * tr, g2 = 2.0 * ph.G;
#pragma unroll
    for (int I = 0; I < 6; ++I) sig[I] = I < 3 ? g2 * e[I] + lt : ph.G * e[I];
    return false;
  }
  double z[6];
#pragma unroll
  for (int k = 0; k < 6; ++k) z[k] = zp[k * BT];
  const double twoG = 2.0 * ph.G, m3 = tr * (1.0 / 3.0);
  const double xi[6] = {e[0] - m3 - z[1],      e[1] - m3 - z[2],      e[2] - m3 + (z[1] + z[2]),
                        0.5 * e[3] - z[3], 0.5 * e[4] - z[4], 0.5 * e[5] - z[5]};
  const double n2 = xi[0] * xi[0] + xi[1] * xi[1] + xi[2] * xi[2] +
                    2.0 * (xi[3] * xi[3] + xi[4] * xi[4] + xi[5] * xi[5]);
  const double inx = rsqrt(fmax(n2, tiny_s<double>())), ns = twoG * (n2 * inx);   // 1 / |xi|, |s_tr|
  const bool explin = ph.kind == 2;
  const double e_n = explin ? exp(-ph.rate * z[0]) : 1.0;
  const double sy = ph.s0 + ph.H * z[0] + (explin ? ph.ds * (1.0 - e_n) : 0.0);
  const double f = ns - SQ23 * sy;
  const bool plastic = f > 0.0;
  double dg = plastic ? f * ph.inv_den : 0.0, thb0 = ph.thb0;
  if (explin && plastic) {   // the scalar Newton iteration of leaf_iso
    double slope = ph.H + ph.dk * e_n, ex = e_n, step = 0.0;
    dg = f / (twoG + (2.0 / 3.0) * slope);
    for (int it = 0; it < 40; ++it) {
      const double a = z[0] + SQ23 * dg;
      ex = exp(-ph.rate * a);
      slope = ph.H + ph.dk * ex;
      const double r = ns - twoG * dg - SQ23 * (ph.s0 + ph.H * a + ph.ds * (1.0 - ex));
      step = r / (twoG + (2.0 / 3.0) * slope);
      dg += step;
      if (fabs(step) <= 1e-10 * dg) break;
    }
    slope -= ph.rate * ph.dk * ex * SQ23 * step;
    thb0 = 1.0 / (1.0 + slope / (3.0 * ph.G));
  }
  const double k2 = dg * inx, Kt = ph.K * tr, g2 = twoG - twoG * k2;
#pragma unroll
  for (int I = 0; I < 6; ++I) sig[I] = I < 3 ? g2 * xi[I] + Kt : g2 * xi[I];
  const pair nk2 = neg(split(k2)), G = split(ph.G);
  pair ix = split(inx);
  if (!(ix.h < 1e37f)) ix = pair{0.f, 0.f};   // no strain: no direction (and c = 0)
  pair v = mul(G, add(pair{1.f, 0.f}, nk2));               // mu = G (1 - k2)
  T[0] = v.h; T[8 * BT] = v.l;
  v = mul(pair{2.f * G.h, 2.f * G.l}, add(split(thb0), nk2));   // c = 2 G (thb0 - k2)
  T[BT] = plastic ? v.h : 0.f; T[9 * BT] = plastic ? v.l : 0.f;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    v = mul(split(xi[k]), ix);
    T[(2 + k) * BT] = v.h; T[(10 + k) * BT] = v.l;
  }
  return plastic;
}

// D e of a leaf in pairs (B): the phase's constants or the stored mu, c, m
static __device__ __forceinline__ void leaf_apply(const PhaseDev& ph, const float* s, const pair e[6], pair tau[6]) {
  const pair tr = add(add(e[0], e[1]), e[2]);
  if (ph.kind == 0) {
    const pair lt = mul(split(ph.lam), tr), g = split(ph.G), g2 = {2.f * g.h, 2.f * g.l};
#pragma unroll
    for (int I = 0; I < 6; ++I) tau[I] = I < 3 ? add(mul(g2, e[I]), lt) : mul(g, e[I]);
    return;
  }
  pair m[6], me;
#pragma unroll
  for (int I = 0; I < 6; ++I) {
    m[I] = pair{s[(2 + I) * BT], s[(10 + I) * BT]};
    me = I ? add(me, mul(m[I], e[I])) : mul(m[I], e[I]);
  }
  const pair mu = {s[0], s[8 * BT]}, cm = neg(mul(pair{s[BT], s[9 * BT]}, me)), g2 = {2.f * mu.h, 2.f * mu.l};
  const pair lt = mul(add(split(ph.K), mul(split(-2.0 / 3.0), mu)), tr);
#pragma unroll
  for (int I = 0; I < 6; ++I) {
    tau[I] = add(mul(I < 3 ? g2 : mu, e[I]), mul(cm, m[I]));
    if (I < 3) tau[I] = add(tau[I], lt);
  }
}

// Own-column accesses: a thread's vector of 6 in rows 0 .. 5 of a shared array, at column x.
template <typename T>
static __device__ __forceinline__ void put6(T (*m)[BT], int x, const T v[6]) {
#pragma unroll
  for (int I = 0; I < 6; ++I) m[I][x] = v[I];
}
template <typename T>
static __device__ __forceinline__ void get6(T (*m)[BT], int x, T v[6]) {
#pragma unroll
  for (int I = 0; I < 6; ++I) v[I] = m[I][x];
}
static __device__ __forceinline__ void put6(float (*m)[BT], int x, const pair v[6]) {
#pragma unroll
  for (int I = 0; I < 6; ++I) { m[I][x] = v[I].h; m[6 + I][x] = v[I].l; }
}
static __device__ __forceinline__ void get6(float (*m)[BT], int x, pair v[6]) {
#pragma unroll
  for (int I = 0; I < 6; ++I) v[I] = pair{m[I][x], m[6 + I][x]};
}
static __device__ __forceinline__ void put27(float (*m)[BT], int x, const Sub32& v) {
#pragma unroll
  for (int I = 0; I < 6; ++I) m[I][x] = v.ds[I];
#pragma unroll
  for (int k = 0; k < 21; ++k) m[6 + k][x] = v.C[k];
}
static __device__ __forceinline__ void get27(float (*m)[BT], int x, Sub32& v) {
#pragma unroll
  for (int I = 0; I < 6; ++I) v.ds[I] = m[I][x];
#pragma unroll
  for (int k = 0; k < 21; ++k) v.C[k] = m[6 + k][x];
}

// Shared memory: what a level hands to the next, at the column of its leftmost subtree (in place: a
// laminate's own column is its left child's); between levels a thread's own column keeps what its depth-first
// walk sets aside, with sh_s for the level below.
struct BlockShared {
  double e[6][BT];       // strains down, stresses up (FP64, or pairs in 12 FP32 rows)
  float c[27][BT];       // FP32 condensation up; rows 0 .. 5 also the FP32 corrections
  float s[27][BT];       // the bottom walk's set-aside vectors (FP64: the first 12 rows)
  double r[BT];          // partial residual norms
  long long pt[BT];
  int fl[BT];
  float st[BT];
  int pl[BT];            // the point has a plastic leaf in this round
  int n_in, n_out;       // slots that take a point in / hand one out in this round
  short in[BT], out[BT];
};

// Laminate h (0-based) of the full tree of depth Kt + 3 lies with subtree thread s as its laminate j.
static __device__ __forceinline__ void owner(int h, int Kt, int& s, int& j) {
  const int h1 = h + 1, d = 31 - __clz(h1) - Kt, S = 1 << Kt;
  if (d < 0) { s = h1; j = 7; }
  else { s = (h1 >> d) - S; j = (1 << d) - 1 + (h1 & ((1 << d) - 1)); }
}

// The two CTAs of an SM should alternate between the FP64 phase A and the FP32 phases S and B: in step, both in A
// or both out of it, the FP64 units idle half of the time.  A token per SM is held during A.  The wait for it is
// bounded, and its holder waits for nothing; a CTA that gives up goes on without it (two SMs whose ids share a
// token only wait more).  Depth 8, 200003 points: 72.8 ms always; without it 70 ms to 87 ms, also where the two
// CTAs start half a round apart.  With several trees the rounds of an SM's CTAs differ in length and the wait
// costs more than it orders (depths 3 to 8 with the line search: 5.9 against 5.4 ms).
static __device__ __forceinline__ unsigned long long* token(const BlockParams& P) {
  unsigned smid;
  asm volatile("mov.u32 %0, %%smid;" : "=r"(smid));
  return P.counter + 32 + (smid & (BLOCK_TOKENS - 1));
}
static __device__ __forceinline__ bool acquire(unsigned long long* tok) {
  for (int k = 0; k < 500; ++k) {
    if (atomicCAS(tok, 0ull, 1ull) == 0ull) return true;
    __nanosleep(400);
  }
  return false;
}

template <bool LS, bool CMP>
static __device__ void newton(const BlockParams& P) {
  extern __shared__ __align__(16) char dyn[];
  BlockShared& M = *reinterpret_cast<BlockShared*>(dyn);
  double (*const sh_e)[BT] = M.e;
  float (*const sh_c)[BT] = M.c;
  double (*const sh_s)[BT] = reinterpret_cast<double (*)[BT]>(M.s);
  float (*const sh_p)[BT] = reinterpret_cast<float (*)[BT]>(M.e);   // pairs
  float (*const sh_x)[BT] = M.s + 12;
  double* const sh_r = M.r;
  long long* const sh_pt = M.pt;
  int* const sh_fl = M.fl;
  float* const sh_st = M.st;
  int* const sh_pl = M.pl;
  const int tid = threadIdx.x;
  const size_t n = (size_t)P.n;
  unsigned long long* const tok = token(P);
  bool own = false;
  Ctx c;
  double *D0, *z0;
  {
    char* base = P.scratch + (size_t)blockIdx.x * block_scratch_bytes(BT, P.leaf_slots, LS);
    double* D = (double*)base;
    D0 = D;
    z0 = D + (size_t)8 * (LS ? 9 : 6) * BT;
    c.D = D + tid;
    c.z = D + (size_t)8 * (LS ? 9 : 6) * BT + tid;
    float* F = (float*)(D + (size_t)(8 * (LS ? 9 : 6) + 6 * P.leaf_slots) * BT);
    c.F = F + tid;
    c.tan = F + (size_t)8 * F_END * BT + tid;
  }
  for (int tr = 0; tr < P.F.n; ++tr) {
    const TreeDev& t = P.F.t[tr];
    const int K = t.K, Kt = K - 3, S = 1 << Kt, nP = BT >> Kt, p = tid & (nP - 1), s = tid / nP;
    // with several trees the points are sorted by tree: this tree's are [begin, end)
    const unsigned long long end = P.perm ? P.counter[10 + tr] : (tr ? 0ull : (unsigned long long)P.n);
    const unsigned long long begin = P.perm ? end - P.counter[1 + tr] : 0ull;
    const int nzf = 6 * t.nz;
    const bool both = t.z_both;
    // the thread's top laminate: heap number s on level `lev`, its results at place pos, its right child's at pos + half
    const int lev = s ? 31 - __clz(s) : -1;
    const int pos = s ? (((s << (Kt - lev)) - S) * nP + p) : p, half = s ? (S >> (lev + 1)) * nP : 0;
    const int R1 = S + s;                      // heap number of the thread's subtree
    auto heap = [&](int j) { return (j == 0 ? R1 : j < 3 ? 2 * R1 + j - 1 : j < 7 ? 4 * R1 + j - 3 : s) - 1; };
    // a subtree with nothing alive in it is skipped (its results are never used, only kept finite)
    const bool dead = CMP && __ldg(t.hdir + heap(0)) == 3;
    // state of slot p, kept by thread p < nP
    long long pt = -1;
    int it = 0, halv = 0, np = 0;
    double rn_acc = 0.0, left = 0.0;
    bool again = false;   // a step in two parts (LEFT_MAX)
    bool met = false;     // whose first part met the criterion
    bool linear = false;  // all leaves elastic in the step's condensation
    // a point that is done: its counts, and its jumps in the state's order (by the CTA)
    auto done = [&](int st) {
      P.iters[pt] = it;
      P.status[pt] = st;
      if (P.passes) atomicAdd(P.passes, (unsigned long long)np);
      M.out[atomicAdd(&M.n_out, 1)] = (short)tid;
    };
    auto write_out = [&]() {
      for (int i = tid; i < M.n_out << K; i += BT) {
        const int x = M.out[i >> K], h = i & (t.L - 1);
        const int row = h == t.L - 1 ? -1 : CMP ? __ldg(t.hcid + h) : (1 << K) - 3 * (1 << (31 - __clz(h + 1))) + h + 1;
        if (row < 0) continue;
        int os, oj;
        owner(h, Kt, os, oj);
        const double* w = D0 + 8 * (LS && (sh_fl[x] & B_CUR) ? D_A2 : D_A) * BT + oj * BT + os * nP + x;
        double* st = P.state_out + (nzf + 3 * row) * n + (size_t)sh_pt[x];
#pragma unroll
        for (int k = 0; k < 3; ++k) st[k * n] = w[8 * k * BT];
      }
    };
    bool more = tid < nP;
    if (tid < nP) sh_fl[tid] = 0;
    if (tid == 0) M.n_in = 0;
    __syncthreads();
    for (;;) {
      if (tid < nP && more && !(sh_fl[tid] & B_ACT)) {
        for (;;) {
          const unsigned long long i = begin + atomicAdd(P.counter + 21 + tr, 1ull);
          if (i >= end) { more = false; break; }
          int tt;
          int64_t x;
          point_of(P.perm, P.tid, P.F.n, (int64_t)i, x, tt);
          if (tt == tr) {
            pt = x; it = 0; halv = 0; np = 0; rn_acc = 0.0; left = 0.0; again = met = false;
            sh_pt[tid] = pt; sh_st[tid] = 1.f;
            sh_fl[tid] = B_ACT | B_FIRST;
            M.in[atomicAdd(&M.n_in, 1)] = (short)tid;
            break;
          }
          block_bad_tree(P, x);
        }
      }
      if (tid < nP) sh_pl[tid] = 0;
      const bool any = tid < nP && (sh_fl[tid] & B_ACT);
      if (!__syncthreads_or(any)) break;
      int fl = sh_fl[p];
      const size_t mypt = (size_t)sh_pt[p];
      // the CTA's threads load the new points together, a laminate and a leaf each: independent loads, where
      // the slot's own S threads would wait for one after another (a quarter of a round; now a twentieth)
      for (int i = tid; i < M.n_in << K; i += BT) {
        const int x = M.in[i >> K], h = i & (t.L - 1);
        const size_t q = (size_t)sh_pt[x];
        const int id = h == t.L - 1 ? -1 : CMP ? __ldg(t.hcid + h) : h;
        if (id >= 0) {
          const int row = CMP ? id : (1 << K) - 3 * (1 << (31 - __clz(h + 1))) + h + 1;
          int os, oj;
          owner(h, Kt, os, oj);
          double* w = D0 + oj * BT + os * nP + x;
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            w[8 * (D_A + k) * BT] = __ldg(P.state_in + (nzf + 3 * row + k) * n + q);
            w[8 * (D_N + k) * BT] = __ldg(P.nbuf + (3 * id + k) * n + q);
          }
        }
        const int leaf = h;   // as many leaves as laminates and one
        if (t.ph[leaf & 1].kind != 0) {
          const int slot = CMP ? __ldg(t.lslot + leaf) : both ? leaf : leaf >> 1;
          const int l = leaf & 7;
          double* w = z0 + (6 * (both ? l : l >> 1)) * BT + (leaf >> 3) * nP + x;
#pragma unroll
          for (int k = 0; k < 6; ++k)
            w[k * BT] = slot >= 0 ? (k < 3 ? 1.0 : RS2) * __ldg(P.state_in + (6 * slot + k) * n + q) : 0.0;
        }
      }
      if (tid == 0) {
        M.n_out = 0;
        own = P.F.n == 1 && acquire(tok);
      }
      const bool act = fl & B_ACT, apply = act && !(fl & B_FIRST);
      const int a_in = LS && (fl & B_CUR) ? D_A2 : D_A, a_out = LS ? (a_in == D_A ? D_A2 : D_A) : D_A;
      const double step = LS ? (double)sh_st[p] : 1.0;
      // ---- A: strains down, leaf laws, residual up (FP64)
      float(*sd)[BT] = sh_c;
      if (act && s == 0) {
#pragma unroll
        for (int I = 0; I < 6; ++I) {
          sh_e[I][p] = (I < 3 ? 1.0 : 1.41421356237309504880) * P.nbuf[(3 * P.N_max + I) * n + mypt];
          sd[I][p] = 0.f;
        }
      }
      __syncthreads();
      for (int l = 0; l < Kt; ++l) {
        if (act && lev == l) {
          double e[6], eL[6], eR[6];
          float de[6], dL[6], dR[6];
          get6(sh_e, pos, e);
          get6(sd, pos, de);
          down_a<CMP, LS>(t, c, s - 1, 7, a_in, a_out, apply, step, e, de, eL, eR, dL, dR);
          put6(sh_e, pos, eL); put6(sh_e, pos + half, eR);
          put6(sd, pos, dL); put6(sd, pos + half, dR);
        }
        __syncthreads();
      }
      double r2 = 0.0;
      if (act && !dead) {
        double e[6], eL[6], eR[6], sb[6];
        float de[6], dL[6], dR[6];
        get6(sh_e, tid, e);
        get6(sd, tid, de);
        down_a<CMP, LS>(t, c, heap(0), 0, a_in, a_out, apply, step, e, de, eL, eR, dL, dR);
        put6(sh_e, tid, eR);
        put6(sd, tid, dR);
#pragma unroll
        for (int I = 0; I < 6; ++I) { e[I] = eL[I]; de[I] = dL[I]; }
#pragma unroll 1
        for (int q = 0; q < 4; ++q) {
          const int mid = 1 + (q >> 1);
          if (!(q & 1)) {
            down_a<CMP, LS>(t, c, heap(mid), mid, a_in, a_out, apply, step, e, de, eL, eR, dL, dR);
            put6(sh_s, tid, eR);
            put6(sh_x, tid, dR);
#pragma unroll
            for (int I = 0; I < 6; ++I) { e[I] = eL[I]; de[I] = dL[I]; }
          }
          down_a<CMP, LS>(t, c, heap(3 + q), 3 + q, a_in, a_out, apply, step, e, de, eL, eR, nullptr, nullptr);
          double s0[6], s1[6];
#pragma unroll
          for (int side = 0; side < 2; ++side) {
            const int ls = both ? 2 * q + side : q;
            if (leaf_a(t.ph[side], side ? eR : eL, c.z + 6 * ls * BT, side ? s1 : s0, c.tan + 16 * ls * BT)) sh_pl[p] = 1;
          }
          up_a<CMP>(t, c, heap(3 + q), 3 + q, s0, s1, sb, r2);
          if (!(q & 1)) {
            get6(sh_s, tid, e);
            get6(sh_x, tid, de);
            put6(sh_s, tid, sb);
          } else {
            get6(sh_s, tid, s0);
            up_a<CMP>(t, c, heap(mid), mid, s0, sb, s1, r2);
            if (q == 1) {
              get6(sh_e, tid, e);
              get6(sd, tid, de);
              put6(sh_e, tid, s1);
            }
          }
          if (q == 3) {
            get6(sh_e, tid, s0);
            up_a<CMP>(t, c, heap(0), 0, s0, s1, sb, r2);
            put6(sh_e, tid, sb);
          }
        }
      } else if (act) {
#pragma unroll
        for (int I = 0; I < 6; ++I) sh_e[I][tid] = 0.0;
      }
      __syncthreads();
      for (int l = Kt - 1; l >= 0; --l) {
        if (act && lev == l) {
          double sL[6], sR[6], sb[6];
          get6(sh_e, pos, sL);
          get6(sh_e, pos + half, sR);
          up_a<CMP>(t, c, s - 1, 7, sL, sR, sb, r2);
          put6(sh_e, pos, sb);
        }
        __syncthreads();
      }
      // sum of the point's shares in an order that does not depend on BT: 2^nb neighbouring subtrees by shuffles
      // (as many as a warp of the large CTA holds), then the groups in turn
      const int nb = Kt > 3 ? Kt - 3 : 0, groups = S >> nb;
      for (int b = nb - 1; b >= 0; --b) r2 += __shfl_xor_sync(0xffffffffu, r2, nP << b);
      if (!(s & ((1 << nb) - 1))) sh_r[(s >> nb) * nP + p] = r2;
      __syncthreads();
      if (own) { own = false; atomicExch(tok, 0ull); }
      double rn = 0.0;
      if (tid < nP && (sh_fl[tid] & B_ACT)) {
        double r = 0.0, sn2 = 0.0;
        for (int k = 0; k < groups; ++k) r += sh_r[k * nP + tid];
        rn = sqrt(r);
#pragma unroll
        for (int I = 0; I < 6; ++I) sn2 += (I < 3 ? 1.0 : 2.0) * sh_e[I][tid] * sh_e[I][tid];
        const double sn = sqrt(sn2);
        int f = sh_fl[tid] & (B_ACT | B_FIRST | B_CUR);
        if (!again) ++np;
        bool retry = false;
        int st = -1;   // the point's status once it is done
        const bool ok = !LS || (f & B_FIRST) || rn < rn_acc;
        if (ok) {
          if (LS) { f ^= B_CUR; sh_st[tid] = 1.f; halv = 0; }
          rn_acc = rn;
          f &= ~B_FIRST;
          const bool crit = rn <= P.tol * (double)t.N * sn, rest = !again && rn <= LEFT_MAX * left;
          if (!isfinite(rn) || !isfinite(sn)) retry = true;
          else if (crit && !(rest && rn > ROUNDING * sn)) st = DMN_STATUS_OK;
          else if (rest) { again = true; met = crit; f |= crit && linear && !sh_pl[tid] ? B_CONT | B_LAST : B_CONT; }
          else if (it >= P.max_iter) st = DMN_STATUS_MAXITER;
          else if (it >= BLOCK_ITERS) retry = true;
          else { ++it; again = met = false; f |= B_CONT; }
          linear = !sh_pl[tid];
        } else if (met) {
          st = DMN_STATUS_OK;   // at its rounding: the accepted iterate stands
        } else if (++halv > 8) {
          st = DMN_STATUS_LINESEARCH;   // no halving lowered the residual: the accepted iterate stands
          ++it;
        } else {
          sh_st[tid] *= 0.5f;
        }
        if (retry) { block_retry(P, pt); f = 0; }
        if (st >= 0) {
          f |= B_CONV;
          done(st);
          f &= ~B_ACT;
        }
        sh_fl[tid] = f;
      }
      __syncthreads();
      fl = sh_fl[p];
      if (tid == 0) M.n_in = 0;
      write_out();
      const bool cont = fl & B_CONT, last = fl & B_LAST, solve = cont && !last;
      if (!__syncthreads_or(cont)) {
        if (tid < nP) sh_fl[tid] &= ~B_CONV;
        continue;
      }
      // ---- S: FP32 condensation up
      if (solve && !dead) {
        Sub32 res, sib, o;
#pragma unroll 1
        for (int q = 0; q < 4; ++q) {
          const int mid = 1 + (q >> 1);
          LeafTan<float> DL, DR;
          leaf_tan32(t.ph[0], c.tan + 16 * (both ? 2 * q : q) * BT, DL);
          leaf_tan32(t.ph[1], c.tan + 16 * (both ? 2 * q + 1 : q) * BT, DR);
          condense32_bottom<CMP>(t, c, heap(3 + q), 3 + q, DL, DR, t.ph[0].kind == 0, t.ph[1].kind == 0, res);
          if (!(q & 1)) {
            put27(M.s, tid, res);
          } else {
            get27(M.s, tid, sib);
            condense32<CMP>(t, c, heap(mid), mid, sib, res, o);
            if (q == 1) put27(sh_c, tid, o);
          }
        }
        get27(sh_c, tid, sib);
        condense32<CMP>(t, c, heap(0), 0, sib, o, res);
        put27(sh_c, tid, res);
      } else if (solve) {
#pragma unroll
        for (int k = 0; k < 27; ++k) sh_c[k][tid] = 0.f;
      }
      __syncthreads();
      for (int l = Kt - 1; l >= 0; --l) {
        if (solve && lev == l) {
          Sub32 L, R, o;
          get27(sh_c, pos, L);
          get27(sh_c, pos + half, R);
          condense32<CMP>(t, c, s - 1, 7, L, R, o);
          put27(sh_c, pos, o);
        }
        __syncthreads();
      }
      // ---- B: the step down, J times it up (pairs), the second FP32 solve up
      if (cont && s == 0) {
#pragma unroll
        for (int I = 0; I < 12; ++I) sh_p[I][p] = 0.f;
      }
      __syncthreads();
      for (int l = 0; l < Kt; ++l) {
        if (cont && lev == l) {
          pair e[6], eL[6], eR[6];
          get6(sh_p, pos, e);
          down_b<CMP>(t, c, s - 1, 7, solve, e, eL, eR);
          put6(sh_p, pos, eL); put6(sh_p, pos + half, eR);
        }
        __syncthreads();
      }
      float q2 = 0.f;
      if (cont && !dead) {
        pair e[6], eL[6], eR[6], t0[6], t1[6];
        float x0[6], x1[6];
        get6(sh_p, tid, e);
        down_b<CMP>(t, c, heap(0), 0, solve, e, eL, eR);
        put6(sh_p, tid, eR);
#pragma unroll
        for (int I = 0; I < 6; ++I) e[I] = eL[I];
#pragma unroll 1
        for (int q = 0; q < 4; ++q) {
          const int mid = 1 + (q >> 1);
          if (!(q & 1)) {
            down_b<CMP>(t, c, heap(mid), mid, solve, e, eL, eR);
            put6(M.s, tid, eR);
#pragma unroll
            for (int I = 0; I < 6; ++I) e[I] = eL[I];
          }
          down_b<CMP>(t, c, heap(3 + q), 3 + q, solve, e, eL, eR);
          leaf_apply(t.ph[0], c.tan + 16 * (both ? 2 * q : q) * BT, eL, t0);
          leaf_apply(t.ph[1], c.tan + 16 * (both ? 2 * q + 1 : q) * BT, eR, t1);
          up_b<CMP, true>(t, c, heap(3 + q), 3 + q, t0, t1, nullptr, nullptr, eL, x1, q2);
          if (!(q & 1)) {
            get6(M.s, tid, e);
            put6(M.s, tid, eL);
            put6(sh_x, tid, x1);
          } else {
            get6(M.s, tid, t0);
            get6(sh_x, tid, x0);
            float y[6];
            up_b<CMP, false>(t, c, heap(mid), mid, t0, eL, x0, x1, t1, y, q2);
#pragma unroll
            for (int I = 0; I < 6; ++I) x1[I] = y[I];
            if (q == 1) {
              get6(sh_p, tid, e);
              put6(sh_p, tid, t1);
              put6(sd, tid, x1);
            }
          }
          if (q == 3) {
            get6(sh_p, tid, t0);
            get6(sd, tid, x0);
            float y[6];
            up_b<CMP, false>(t, c, heap(0), 0, t0, t1, x0, x1, eL, y, q2);
            put6(sh_p, tid, eL);
            put6(sd, tid, y);
          }
        }
      } else if (cont) {
#pragma unroll
        for (int I = 0; I < 12; ++I) sh_p[I][tid] = 0.f;
#pragma unroll
        for (int I = 0; I < 6; ++I) sd[I][tid] = 0.f;
      }
      __syncthreads();
      for (int l = Kt - 1; l >= 0; --l) {
        if (cont && lev == l) {
          pair tL[6], tR[6], tb[6];
          float xL[6], xR[6], xb[6];
          get6(sh_p, pos, tL);
          get6(sh_p, pos + half, tR);
          get6(sd, pos, xL);
          get6(sd, pos + half, xR);
          up_b<CMP, false>(t, c, s - 1, 7, tL, tR, xL, xR, tb, xb, q2);
          put6(sh_p, pos, tb);
          put6(sd, pos, xb);
        }
        __syncthreads();
      }
      for (int b = nb - 1; b >= 0; --b) q2 += __shfl_xor_sync(0xffffffffu, q2, nP << b);
      if (!(s & ((1 << nb) - 1))) sh_r[(s >> nb) * nP + p] = (double)q2;
      const bool ends = __syncthreads_or(last);
      if (tid < nP) {
        int f = sh_fl[tid] & ~B_CONV;
        if ((f & B_CONT) && !last) {
          double r = 0.0;
          for (int k = 0; k < groups; ++k) r += sh_r[k * nP + tid];
          r = sqrt(r);                 // of the linear residual; the second solve leaves about r / rn_acc of it
          left = fmax(r * (r / rn_acc), PAIR_LEFT * rn_acc);
          if (!(r <= (double)REFINE_MAX * rn_acc)) {
            block_retry(P, pt);
            f = 0;
          }
        }
        sh_fl[tid] = f;
      }
      // ---- an elastic point's second part ends with the jumps: no more A
      if (!ends) continue;
      const int buf = LS && (fl & B_CUR) ? D_A2 : D_A;
      if (tid == 0) M.n_out = 0;
      if (last && s == 0) {
#pragma unroll
        for (int I = 0; I < 6; ++I) sd[I][p] = 0.f;
      }
      __syncthreads();
      for (int l = 0; l < Kt; ++l) {
        if (last && lev == l) {
          float de[6], dL[6], dR[6];
          get6(sd, pos, de);
          down_last<CMP>(t, c, s - 1, 7, buf, de, dL, dR);
          put6(sd, pos, dL); put6(sd, pos + half, dR);
        }
        __syncthreads();
      }
      if (last && !dead) {
        float de[6], dL[6], dR[6];
        get6(sd, tid, de);
        down_last<CMP>(t, c, heap(0), 0, buf, de, dL, dR);
        put6(sd, tid, dR);
#pragma unroll
        for (int I = 0; I < 6; ++I) de[I] = dL[I];
#pragma unroll 1
        for (int q = 0; q < 4; ++q) {
          const int mid = 1 + (q >> 1);
          if (!(q & 1)) {
            down_last<CMP>(t, c, heap(mid), mid, buf, de, dL, dR);
            put6(sh_x, tid, dR);
#pragma unroll
            for (int I = 0; I < 6; ++I) de[I] = dL[I];
          }
          down_last<CMP>(t, c, heap(3 + q), 3 + q, buf, de, nullptr, nullptr);
          if (!(q & 1)) get6(sh_x, tid, de);
          else if (q == 1) get6(sd, tid, de);
        }
      }
      if (tid < nP && last) {
        done(DMN_STATUS_OK);
        sh_fl[tid] &= B_CUR;
      }
      __syncthreads();
      write_out();
      __syncthreads();
    }
    __syncthreads();
  }
  // points of unknown trees (the last bucket of the sort)
  if (P.perm) {
    const unsigned long long end = P.counter[10 + P.F.n], begin = end - P.counter[1 + P.F.n];
    for (unsigned long long i = begin + blockIdx.x * (unsigned long long)BT + tid; i < end;
         i += (unsigned long long)gridDim.x * BT)
      block_bad_tree(P, P.perm[i]);
  }
}

};

template <int BT, bool LS, bool CMP>
__global__ void __launch_bounds__(BT, BLOCK_THREADS * BLOCK_CTAS_PER_SM / BT) k_newton_block(BlockParams P) {
  Block<BT>::template newton<LS, CMP>(P);
}

// ---------------------------------------------------------------------------
// The FP64 sweep at the converged jumps in the same organisation: stress, algorithmic tangent and leaf states
// of every point (the FP64 form after k_newton_block, the mixed form after its Newton kernel).  One pass:
// strains down, leaf laws (which give the FP64 form's new leaf states too), condensation up, rotation.  It
// replaces one sweep per thread, whose last wave and per-thread stacks cost 20 % at 10^5 points, or 8 lanes per
// point.  The FP64 pipe bounds it, so its algebra is the shortest form
// found: tangents in Voigt components (C_IJ / (w_I w_J), w = sqrt 2 in the shear rows), in which N(n) has the
// bare components of n; Kn as quadratic forms in n instead of N^T (C N); and, without a Newton step to store,
// Kn = L D L^T and C -= c1 c2 (B L^-T) D^-1 (B L^-T)^T in place of the inverse and H.  88 k FP64 instructions
// per point at depth 8 instead of 107 k.
// Points left to the all-FP64 kernels (RETRY) are skipped; a point that the mixed forms' Newton kernel found not finite
// gets NaN here, its leaf states in k_final (k_newton_block leaves no such point).
// STATES: also the leaf states.  The mixed form leaves them to k_final, as its FP32-tangent variant does: the two
// return the same state bit for bit.
template <bool CMP, bool STATES>
__global__ void __launch_bounds__(ST, SWEEP_CTAS_PER_SM) k_sweep_block(SweepParams P) {
  extern __shared__ __align__(16) char dyn[];
  SweepShared& M = *reinterpret_cast<SweepShared*>(dyn);
  const int tid = threadIdx.x;
  const size_t n = (size_t)P.n;
  const double qnan = __longlong_as_double(0x7ff8000000000000LL);
  for (unsigned long long g = blockIdx.x;; g += gridDim.x) {
    // group g: nP consecutive points of one tree
    int tr = 0;
    unsigned long long b = g, begin = 0, end = 0;
    for (; tr < P.F.n; ++tr) {
      const int w = ST >> (P.F.t[tr].K - 3);
      end = P.perm ? P.counter[10 + tr] : (tr ? 0ull : (unsigned long long)P.n);
      begin = P.perm ? end - P.counter[1 + tr] : 0ull;
      const unsigned long long groups = (end - begin + w - 1) / w;
      if (b < groups) break;
      b -= groups;
    }
    if (tr == P.F.n) return;
    const TreeDev& t = P.F.t[tr];
    const int K = t.K, Kt = K - 3, S = 1 << Kt, nP = ST >> Kt, p = tid & (nP - 1), s = tid / nP;
    const int nzf = 6 * t.nz, R1 = S + s, lev = s ? 31 - __clz(s) : -1;
    const int pos = s ? (((s << (Kt - lev)) - S) * nP + p) : p, half = s ? (S >> (lev + 1)) * nP : 0;
    const bool both = t.z_both;
    auto heap = [&](int j) { return (j == 0 ? R1 : j < 3 ? 2 * R1 + j - 1 : 4 * R1 + j - 3) - 1; };
    const bool dead = CMP && __ldg(t.hdir + heap(0)) == 3;
    const unsigned long long i = begin + b * nP + p;
    int64_t pt = 0;
    int st = STATUS_RETRY;
    if (i < end) {
      int tt;
      point_of(P.perm, P.tid, P.F.n, (int64_t)i, pt, tt);
      if (tt == tr) st = P.status[pt];
    }
    const bool act = st != STATUS_RETRY && st != DMN_STATUS_NONFINITE;
    const double* zin = P.state_in + pt;
    double* zout = P.state_out + pt;
    auto normal = [&](const Lam<CMP>& q, double v[3]) {
#pragma unroll
      for (int k = 0; k < 3; ++k) v[k] = P.nbuf[(3 * q.id + k) * n + pt];
    };
    auto down = [&](int h, const double e[6], double eL[6], double eR[6]) {
      const Lam<CMP> q(t, h);
      if (CMP && q.mode) {
#pragma unroll
        for (int I = 0; I < 6; ++I) eL[I] = eR[I] = e[I];
        return;
      }
      const int row = CMP ? q.id : (1 << K) - 3 * (1 << (31 - __clz(h + 1))) + h + 1;
      double v[3], a[3], Na[6];
      normal(q, v);
#pragma unroll
      for (int k = 0; k < 3; ++k) a[k] = zout[(nzf + 3 * row + k) * n];
      const double vr[3] = {v[0] * RS2, v[1] * RS2, v[2] * RS2};
      N_apply<double>(v, vr, a, Na);
#pragma unroll
      for (int I = 0; I < 6; ++I) { eL[I] = e[I] - q.c2 * Na[I]; eR[I] = e[I] + q.c1 * Na[I]; }
    };
    auto up = [&](int h, const Sub64& L, const Sub64& R, Sub64& o) {
      const Lam<CMP> q(t, h);
      if (CMP && q.mode) {
        if (q.mode == 2) o = R; else o = L;
        return;
      }
      double v[3];
      normal(q, v);
      condense64(v, q.c2, q.c1 * q.c2, L, R, o, Downdate{});
    };
    if (act && s == 0) {
#pragma unroll
      for (int I = 0; I < 6; ++I) M.e[I][p] = P.nbuf[(3 * P.N_max + I) * n + pt];
    }
    __syncthreads();
    for (int l = 0; l < Kt; ++l) {
      if (act && lev == l) {
        double e[6], eL[6], eR[6];
        sget6(M.e, pos, e);
        down(s - 1, e, eL, eR);
        sput6(M.e, pos, eL);
        sput6(M.e, pos + half, eR);
      }
      __syncthreads();
    }
    if (act && !dead) {
      double e[6], eL[6], eR[6];
      Sub64 res, sib, o;
      sget6(M.e, tid, e);
      down(heap(0), e, eL, eR);
      sput6(M.e, tid, eR);
#pragma unroll
      for (int I = 0; I < 6; ++I) e[I] = eL[I];
#pragma unroll 1
      for (int q = 0; q < 4; ++q) {
        const int mid = 1 + (q >> 1);
        if (!(q & 1)) {
          down(heap(mid), e, eL, eR);
          sput6(M.f, tid, eR);
#pragma unroll
          for (int I = 0; I < 6; ++I) e[I] = eL[I];
        }
        const int h = heap(3 + q);
        down(h, e, eL, eR);
        LeafTan<double> D[2];
        double s0[6], s1[6];
#pragma unroll
        for (int side = 0; side < 2; ++side) {
          const int leaf = 8 * s + 2 * q + side;
          const int slot = t.ph[side].kind == 0 ? -1 : CMP ? __ldg(t.lslot + leaf) : both ? leaf : leaf >> 1;
          double z[6], zn[6];
#pragma unroll
          for (int k = 0; k < 6; ++k) z[k] = slot >= 0 ? zin[(6 * slot + k) * n] : 0.0;
          leaf_iso<double, double>(t.ph[side], side ? eR : eL, z, side ? s1 : s0, &D[side], STATES ? zn : nullptr, nullptr);
          if (STATES && slot >= 0) {
#pragma unroll
            for (int k = 0; k < 6; ++k) zout[(6 * slot + k) * n] = zn[k];
          }
        }
        {
          const Lam<CMP> lam(t, h);
          double v[3] = {0.0, 0.0, 0.0}, c1 = lam.c1, c2 = lam.c2, c12 = lam.c1 * lam.c2;
          if (CMP && lam.mode) { c2 = lam.mode == 2 ? 1.0 : 0.0; c1 = 1.0 - c2; c12 = 0.0; }
          else normal(lam, v);
          condense64_bottom(v, c1, c2, c12, s0, D[0], t.ph[0].kind == 0, s1, D[1], t.ph[1].kind == 0, res, Downdate{});
          if (CMP && lam.mode) {
#pragma unroll
            for (int I = 0; I < 6; ++I) res.sb[I] = lam.mode == 2 ? s1[I] : s0[I];
          }
        }
        if (!(q & 1)) {
          put27(M.s, tid, res);
          sget6(M.f, tid, e);
        } else {
          get27(M.s, tid, sib);
          up(heap(mid), sib, res, o);
          if (q == 1) {
            put27(M.c, tid, o);
            sget6(M.e, tid, e);
          }
        }
      }
      get27(M.c, tid, sib);
      up(heap(0), sib, o, res);
      put27(M.c, tid, res);
    } else if (act) {
#pragma unroll
      for (int k = 0; k < 27; ++k) M.c[k][tid] = 0.0;
    }
    __syncthreads();
    for (int l = Kt - 1; l >= 0; --l) {
      if (act && lev == l) {
        Sub64 L, R, o;
        get27(M.c, pos, L);
        get27(M.c, pos + half, R);
        up(s - 1, L, R, o);
        put27(M.c, pos, o);
      }
      __syncthreads();
    }
    // rotation to the global frame by a thread per entry: R (6 x 6), R C, (R C) R^T
    const int pi[6] = {0, 1, 2, 1, 0, 0}, pj[6] = {0, 1, 2, 2, 2, 1};
    constexpr double W2 = 1.41421356237309504880;
    double* rot = &M.s[0][0];           // [36][nP] R, then [36][nP] R C (in chunks of at most 32 points)
    const int w = min(nP, 32);
    for (int p0 = 0; p0 < nP; p0 += w) {
      for (int x = tid; x < 36 * w; x += ST) {
        const int pp = x % w, I = x / w / 6, J = x / w % 6;
        const unsigned long long ii = begin + b * nP + p0 + pp;
        if (ii >= end) continue;
        const double* Q = P.Q + 9 * (P.perm ? P.perm[ii] : (int64_t)ii);
        const double wIJ = (I < 3 ? 1.0 : W2) * (J < 3 ? 1.0 : W2) * 0.5;
        rot[x] = wIJ * (Q[3 * pi[I] + pi[J]] * Q[3 * pj[I] + pj[J]] + Q[3 * pi[I] + pj[J]] * Q[3 * pj[I] + pi[J]]);
      }
      __syncthreads();
      for (int x = tid; x < 36 * w; x += ST) {
        const int pp = x % w, I = x / w / 6, J = x / w % 6;
        double v = 0.0;
        for (int k = 0; k < 6; ++k) v += rot[(6 * I + k) * w + pp] * (k < 3 ? 1.0 : W2) * M.c[6 + sidx(k, J)][p0 + pp];
        rot[36 * w + x] = (J < 3 ? 1.0 : W2) * v;
      }
      __syncthreads();
      for (int x = tid; x < 42 * w; x += ST) {
        const int pp = x % w, y = x / w;
        const unsigned long long ii = begin + b * nP + p0 + pp;
        if (ii >= end) continue;
        int64_t q;
        int tt;
        point_of(P.perm, P.tid, P.F.n, (int64_t)ii, q, tt);
        if (tt != tr) continue;
        const int qs = P.status[q];
        if (qs == STATUS_RETRY) continue;
        double v = 0.0;
        if (y < 36) {
          for (int k = 0; k < 6; ++k) v += rot[(36 + 6 * (y / 6) + k) * w + pp] * rot[(6 * (y % 6) + k) * w + pp];
          P.tangent[36 * q + y] = qs == DMN_STATUS_NONFINITE ? qnan : v;
        } else {
          for (int k = 0; k < 6; ++k) v += rot[(6 * (y - 36) + k) * w + pp] * M.c[k][p0 + pp];
          P.stress[6 * q + y - 36] = qs == DMN_STATUS_NONFINITE ? qnan : v;
        }
      }
      __syncthreads();
    }
  }
}

template <bool CMP, bool STATES>
static cudaError_t sweep(const SweepParams& P, unsigned grid, cudaStream_t s) {
  const int bytes = (int)sizeof(SweepShared);
  const cudaError_t e = cudaFuncSetAttribute(k_sweep_block<CMP, STATES>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e != cudaSuccess) return e;
  k_sweep_block<CMP, STATES><<<grid, ST, bytes, s>>>(P);
  return cudaSuccess;
}

cudaError_t launch_sweep_block(const SweepParams& P, bool cmp, bool states, unsigned grid, cudaStream_t s) {
  if (cmp) return states ? sweep<true, true>(P, grid, s) : sweep<true, false>(P, grid, s);
  return states ? sweep<false, true>(P, grid, s) : sweep<false, false>(P, grid, s);
}

template <int BT, bool LS, bool CMP>
static cudaError_t launch(const BlockParams& P, unsigned grid, cudaStream_t s) {
  const int bytes = (int)sizeof(typename Block<BT>::BlockShared);
  const cudaError_t e = cudaFuncSetAttribute(k_newton_block<BT, LS, CMP>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e != cudaSuccess) return e;
  k_newton_block<BT, LS, CMP><<<grid, BT, bytes, s>>>(P);
  return cudaSuccess;
}
template <int BT>
static cudaError_t launch(const BlockParams& P, bool ls, bool cmp, unsigned grid, cudaStream_t s) {
  if (ls && cmp) return launch<BT, true, true>(P, grid, s);
  if (ls) return launch<BT, true, false>(P, grid, s);
  if (cmp) return launch<BT, false, true>(P, grid, s);
  return launch<BT, false, false>(P, grid, s);
}

// K: the depth of the handle's deepest tree.  A call that gives every SM at most one CTA of 256 threads runs in
// CTAs of 128, a warp per FP64 unit instead of two (8 points of depth 8: 0.58 -> 0.42 ms).  With more points the
// larger CTA is ahead (100003 points: 36 against 43 ms), whose top levels lie on more warps.
cudaError_t launch_block(const BlockParams& P, int K, bool ls, bool cmp, cudaStream_t s) {
  const int64_t big = (P.n + (BLOCK_THREADS >> (K - 3)) - 1) / (BLOCK_THREADS >> (K - 3));
  if (big <= P.n_sm) {
    constexpr int SMALL = BLOCK_THREADS / 2;
    return launch<SMALL>(P, ls, cmp, (unsigned)((P.n + (SMALL >> (K - 3)) - 1) / (SMALL >> (K - 3))), s);
  }
  const int64_t most = (int64_t)P.n_sm * BLOCK_CTAS_PER_SM;
  return launch<BLOCK_THREADS>(P, ls, cmp, (unsigned)(big < most ? big : most), s);
}

}  // namespace dmn
