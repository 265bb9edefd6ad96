// The adjoints of dmn_grad in the CTA organisation (trees of depth 3 or more): stress seeds (the implicit-function
// gradient of the converged update, see AdjWork in dmn_device.cuh) and tangent seeds (reverse mode through the
// laminate recursion of a tree of elastic phases, see lam_tangent_adjoint there).
//
// Both are bound by the FP64 pipe, once it is fed: one thread per point (stress) kept 128 warps busy at the offline
// training's 4096 samples and took 9.3 ms; one warp per point (tangent) with its per-laminate data point-strided
// moved a sector per value and took 7.2 ms.  Here a thread owns a subtree of depth 3 of one of a CTA's 128 / S
// points (the organisation of k_sweep_block) and keeps per-laminate data in the CTA's scratch, [field][laminate]
// [thread]; the sines and cosines come from a kernel of their own, a thread per point and share of the laminates.
// At depth 8 and 4096 points: stress 9.3 -> 1.6 ms, tangent 7.2 -> 2.3 ms.
#include <cuda_runtime.h>

#include <type_traits>

#include "../../include/dmn.h"
#include "dmn_block.cuh"

namespace dmn {

namespace {

constexpr double W2 = 1.41421356237309504880;

// shape-function values of one point (Sec. 2.3), as in point_normals
__device__ __forceinline__ void shape_values(int M, double l1, double l2, double ph[6]) {
  const double v[3] = {l1 - l2, 3.0 * (1.0 - l1 - l2), 2.0 * l1 + 4.0 * l2 - 2.0};
#pragma unroll
  for (int k = 0; k < 6; ++k) ph[k] = 0.0;
  if (M == 3) {
    ph[0] = v[0]; ph[1] = v[1]; ph[2] = v[2];
  } else if (M == 4) {
    const double b = v[0] * v[1] * v[2];
    ph[0] = v[0] - 9.0 * b; ph[1] = v[1] - 9.0 * b; ph[2] = v[2] - 9.0 * b; ph[3] = 27.0 * b;
  } else {
    ph[0] = v[0] * (2.0 * v[0] - 1.0); ph[1] = v[1] * (2.0 * v[1] - 1.0); ph[2] = v[2] * (2.0 * v[2] - 1.0);
    ph[3] = 4.0 * v[0] * v[1]; ph[4] = 4.0 * v[0] * v[2]; ph[5] = 4.0 * v[1] * v[2];
  }
}

// Normals, sin(alpha), cos(beta), sin(beta) of every laminate and the shape-function values; blockIdx.y: the
// share of the laminates.
__global__ void k_grad_normals(GradWork G) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= G.nc) return;
  const TreeDev& t = G.t;
  const size_t ws = (size_t)G.nc;
  double* w = G.work + i;
  double ph[6];
  shape_values(t.M, G.lam[2 * (G.n0 + i)], G.lam[2 * (G.n0 + i) + 1], ph);
  if (blockIdx.y == 0) {
#pragma unroll
    for (int k = 0; k < 6; ++k) w[(G.ph() + k) * ws] = ph[k];
  }
  for (int j = blockIdx.y; j < t.N; j += gridDim.y) {
    double al = 0.0, be = 0.0, sa, ca, sb, cb;
#pragma unroll
    for (int k = 0; k < 6; ++k)
      if (k < t.M) {
        al += __ldg(t.p + j * t.M + k) * ph[k];
        be += __ldg(t.q + j * t.M + k) * ph[k];
      }
    sincos(al, &sa, &ca);
    sincos(be, &sb, &cb);
    w[(3 * j) * ws] = sa * cb; w[(3 * j + 1) * ws] = sa * sb; w[(3 * j + 2) * ws] = ca;
    w[(3 * (t.N + j)) * ws] = sa; w[(3 * (t.N + j) + 1) * ws] = cb; w[(3 * (t.N + j) + 2) * ws] = sb;
  }
}

struct GradShared {
  double e[6][ST], f[6][ST];     // vectors handed down; set aside by the bottom walk
  double c[27][ST], s[27][ST];   // results handed up; set aside
  double g[6][ST];               // the points' seeds (local frame)
  double r[ST];                  // partial sums
};

__device__ __forceinline__ void gput6(double (*m)[ST], int x, const double v[6]) {
#pragma unroll
  for (int k = 0; k < 6; ++k) m[k][x] = v[k];
}
__device__ __forceinline__ void gget6(double (*m)[ST], int x, double v[6]) {
#pragma unroll
  for (int k = 0; k < 6; ++k) v[k] = m[k][x];
}
__device__ __forceinline__ void gput21(double (*m)[ST], int x, const double v[21]) {
#pragma unroll
  for (int k = 0; k < 21; ++k) m[k][x] = v[k];
}
__device__ __forceinline__ void gget21(double (*m)[ST], int x, double v[21]) {
#pragma unroll
  for (int k = 0; k < 21; ++k) v[k] = m[k][x];
}

// A thread's place in the CTA (K: the tree's depth) for one group of points.
struct Place {
  int K, Kt, S, nP, p, s, lev, pos, half;
  __device__ Place(int K_) : K(K_) {
    Kt = K - 3; S = 1 << Kt; nP = ST >> Kt;
    p = threadIdx.x & (nP - 1); s = threadIdx.x / nP;
    lev = s ? 31 - __clz(s) : -1;
    pos = s ? (((s << (Kt - lev)) - S) * nP + p) : p;
    half = s ? (S >> (lev + 1)) * nP : 0;
  }
  __device__ int heap(int j) const {   // laminate j of the thread (7: its top laminate), heap order
    const int R = S + s;
    return (j == 0 ? R : j < 3 ? 2 * R + j - 1 : j < 7 ? 4 * R + j - 3 : s) - 1;
  }
};

// dL/d alpha and dL/d beta of a laminate from dL/dn
__device__ __forceinline__ void put_angles(const GradWork& G, size_t i, int id, const double n[3], const double gn[3]) {
  const size_t ws = (size_t)G.nc;
  const double* tr = G.work + (size_t)(3 * (G.t.N + id)) * ws + i;
  G.work[(G.gab() + id) * ws + i] = n[2] * (gn[0] * tr[ws] + gn[1] * tr[2 * ws]) - gn[2] * tr[0];
  G.work[(G.gab() + G.t.N + id) * ws + i] = gn[1] * n[0] - gn[0] * n[1];
}

// The leaf-weight gradients of a group's points: with y = W Xi of every laminate (fields y at Y[j ST]) each leaf
// takes +c2 y from a laminate whose left subtree holds it and -c1 y from the right one, and its direct term
// (fields at X[l ST], or none); then the normalisation is undone: dL/dw_k = (G_k - sum_l G_l w_l) / S.
template <bool CMP, bool DIRECT>
__device__ void weights(const GradWork& G, GradShared& M, const Place& L, bool act, bool dead, size_t i, const double* Y,
                        const double* X) {
  const TreeDev& t = G.t;
  const int tid = threadIdx.x;
  double* acc = M.f[0];
  auto down = [&](int h, int j, double a, double& l, double& r) {
    const Lam<CMP> q(t, h);
    l = r = a;
    if (CMP && q.mode) return;
    const double y = Y[j * ST];
    l += q.c2 * y;
    r -= q.c1 * y;
  };
  if (L.s == 0) acc[L.p] = 0.0;
  __syncthreads();
  for (int l = 0; l < L.Kt; ++l) {
    if (act && L.lev == l) {
      double a, b;
      down(L.s - 1, 7, acc[L.pos], a, b);
      acc[L.pos] = a;
      acc[L.pos + L.half] = b;
    }
    __syncthreads();
  }
  double g[8], sum = 0.0;
#pragma unroll
  for (int l = 0; l < 8; ++l) g[l] = 0.0;
  if (act && !dead) {
    double a[2], b[4];
    down(L.heap(0), 0, acc[tid], a[0], a[1]);
#pragma unroll
    for (int k = 0; k < 2; ++k) down(L.heap(1 + k), 1 + k, a[k], b[2 * k], b[2 * k + 1]);
#pragma unroll
    for (int k = 0; k < 4; ++k) down(L.heap(3 + k), 3 + k, b[k], g[2 * k], g[2 * k + 1]);
#pragma unroll
    for (int l = 0; l < 8; ++l) {
      const double w = __ldg(t.wl + 8 * L.s + l);
      if (DIRECT) g[l] += X[l * ST];
      if (CMP && !(w > 0.0)) g[l] = 0.0;
      sum += g[l] * w;
    }
  }
  for (int o = 16; o >= L.nP; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  const int lane = tid & 31, groups = L.nP < 32 ? ST / 32 : L.S;
  if (L.nP >= 32) M.r[tid] = sum;
  else if (lane < L.nP) M.r[(tid >> 5) * L.nP + lane] = sum;
  __syncthreads();
  sum = 0.0;
  for (int k = 0; k < groups; ++k) sum += M.r[k * L.nP + L.p];
  if (act) {
#pragma unroll
    for (int l = 0; l < 8; ++l) {
      const bool alive = !CMP || __ldg(t.wl + 8 * L.s + l) > 0.0;
      G.work[(G.gw() + 8 * L.s + l) * (size_t)G.nc + i] = alive ? (g[l] - sum) / t.wsum : 0.0;
    }
  }
  __syncthreads();
}

// scratch of a thread: H [8][18], mu [8][3], jumps [8][3], y [8], leaf stresses [8][6], tangents [8][8], direct [8]
enum { X_H = 0, X_MU = 144, X_A = 168, X_Y = 192, X_S = 200, X_T = 248, X_D = 312, X_END = 320 };
// tangent seeds: C [8][21], y [8]
enum { Z_C = 0, Z_Y = 168 };
static_assert(X_END == GRAD_SCRATCH_DOUBLES && Z_Y + 8 <= GRAD_SCRATCH_DOUBLES, "scratch layout");

}  // namespace

template <bool CMP>
__global__ void __launch_bounds__(ST, SWEEP_CTAS_PER_SM) k_grad_block(GradWork G) {
  extern __shared__ __align__(16) char dyn[];
  GradShared& M = *reinterpret_cast<GradShared*>(dyn);
  const int tid = threadIdx.x;
  const TreeDev& t = G.t;
  const Place L(t.K);
  const int K = L.K, Kt = L.Kt, nP = L.nP, s = L.s, p = L.p;
  double* X = G.scratch + (size_t)blockIdx.x * GRAD_SCRATCH_DOUBLES * ST + tid;
  const size_t n = (size_t)G.n, ws = (size_t)G.nc;
  const int nzf = 6 * t.nz;
  const bool both = t.z_both, dead = CMP && __ldg(t.hdir + L.heap(0)) == 3;
  for (int64_t g0 = (int64_t)blockIdx.x * nP; g0 < G.nc; g0 += (int64_t)gridDim.x * nP) {
    const size_t i = (size_t)(g0 + p);
    const bool act = (int64_t)i < G.nc;
    const size_t pt = (size_t)G.n0 + i;
    auto normal = [&](int id, double v[3]) {
#pragma unroll
      for (int k = 0; k < 3; ++k) v[k] = G.work[(3 * id + k) * ws + i];
    };
    if (act && s == 0) {   // local strain and seed
      double R[6][6];
      mandel_rotation(G.Q + 9 * pt, R);
#pragma unroll
      for (int J = 0; J < 6; ++J) {
        double e = 0.0, gl = 0.0;
#pragma unroll
        for (int I = 0; I < 6; ++I) {
          e += R[I][J] * (G.En[6 * pt + I] + G.dE[6 * pt + I]);
          gl += R[I][J] * G.g_stress[6 * pt + I];
        }
        M.e[J][p] = e;
        M.g[J][p] = gl;
      }
    }
    __syncthreads();
    // ---- strains down, leaf laws, condensation up: H of every laminate, the root's tangent
    auto down = [&](int j, const double e[6], double eL[6], double eR[6]) {
      const int h = L.heap(j);
      const Lam<CMP> q(t, h);
      if (CMP && q.mode) {
#pragma unroll
        for (int I = 0; I < 6; ++I) eL[I] = eR[I] = e[I];
        return;
      }
      const int row = CMP ? q.id : (1 << K) - 3 * (1 << (31 - __clz(h + 1))) + h + 1;
      double v[3], a[3], Na[6];
      normal(q.id, v);
#pragma unroll
      for (int k = 0; k < 3; ++k) X[(X_A + 3 * j + k) * ST] = a[k] = G.state_out[(nzf + 3 * row + k) * n + pt];
      const double vr[3] = {v[0] * RS2, v[1] * RS2, v[2] * RS2};
      N_apply<double>(v, vr, a, Na);
#pragma unroll
      for (int I = 0; I < 6; ++I) { eL[I] = e[I] - q.c2 * Na[I]; eR[I] = e[I] + q.c1 * Na[I]; }
    };
    auto up = [&](int j, const Sub64& A, const Sub64& B, Sub64& o) {
      const Lam<CMP> q(t, L.heap(j));
      if (CMP && q.mode) {
        if (q.mode == 2) o = B; else o = A;
        return;
      }
      double v[3];
      normal(q.id, v);
      condense64(v, q.c2, q.c1 * q.c2, A, B, o, StoreH{X + (X_H + 18 * j) * ST, (size_t)ST});
    };
    for (int l = 0; l < Kt; ++l) {
      if (act && L.lev == l) {
        double e[6], eL[6], eR[6];
        gget6(M.e, L.pos, e);
        down(7, e, eL, eR);
        gput6(M.e, L.pos, eL);
        gput6(M.e, L.pos + L.half, eR);
      }
      __syncthreads();
    }
    if (act && !dead) {
      double e[6], eL[6], eR[6];
      Sub64 res, sib, o;
      gget6(M.e, tid, e);
      down(0, e, eL, eR);
      gput6(M.e, tid, eR);
#pragma unroll
      for (int I = 0; I < 6; ++I) e[I] = eL[I];
#pragma unroll 1
      for (int q = 0; q < 4; ++q) {
        const int mid = 1 + (q >> 1);
        if (!(q & 1)) {
          down(mid, e, eL, eR);
          gput6(M.f, tid, eR);
#pragma unroll
          for (int I = 0; I < 6; ++I) e[I] = eL[I];
        }
        down(3 + q, e, eL, eR);
        LeafTan<double> D[2];
        double s0[6], s1[6];
#pragma unroll
        for (int side = 0; side < 2; ++side) {
          const int l = 2 * q + side, leaf = 8 * s + l;
          const int slot = t.ph[side].kind == 0 ? -1 : CMP ? __ldg(t.lslot + leaf) : both ? leaf : leaf >> 1;
          double z[6];
#pragma unroll
          for (int k = 0; k < 6; ++k) z[k] = slot >= 0 ? G.state_in[(6 * slot + k) * n + pt] : 0.0;
          double* sg = side ? s1 : s0;
          leaf_iso<double, double>(t.ph[side], side ? eR : eL, z, sg, &D[side], nullptr, nullptr);
#pragma unroll
          for (int k = 0; k < 6; ++k) X[(X_S + 6 * l + k) * ST] = sg[k];
          X[(X_T + 8 * l) * ST] = D[side].mu;
          X[(X_T + 8 * l + 1) * ST] = D[side].c;
#pragma unroll
          for (int k = 0; k < 6; ++k) X[(X_T + 8 * l + 2 + k) * ST] = D[side].m[k];
        }
        {
          const Lam<CMP> lam(t, L.heap(3 + q));
          double v[3] = {0.0, 0.0, 0.0}, c1 = lam.c1, c2 = lam.c2, c12 = lam.c1 * lam.c2;
          if (CMP && lam.mode) { c2 = lam.mode == 2 ? 1.0 : 0.0; c1 = 1.0 - c2; c12 = 0.0; }
          else normal(lam.id, v);
          condense64_bottom(v, c1, c2, c12, s0, D[0], t.ph[0].kind == 0, s1, D[1], t.ph[1].kind == 0, res,
                            StoreH{X + (X_H + 18 * (3 + q)) * ST, (size_t)ST});
        }
        if (!(q & 1)) {
          put27(M.s, tid, res);
          gget6(M.f, tid, e);
        } else {
          get27(M.s, tid, sib);
          up(mid, sib, res, o);
          if (q == 1) {
            put27(M.c, tid, o);
            gget6(M.e, tid, e);
          }
        }
      }
      get27(M.c, tid, sib);
      up(0, sib, o, res);
      put27(M.c, tid, res);
    } else if (act) {
#pragma unroll
      for (int k = 0; k < 27; ++k) M.c[k][tid] = 0.0;
    }
    __syncthreads();
    for (int l = Kt - 1; l >= 0; --l) {
      if (act && L.lev == l) {
        Sub64 A, B, o;
        get27(M.c, L.pos, A);
        get27(M.c, L.pos + L.half, B);
        up(7, A, B, o);
        put27(M.c, L.pos, o);
      }
      __syncthreads();
    }
    if (act && s == 0) {
      double gl[6];
      gget6(M.g, p, gl);
      gput6(M.e, p, gl);
      if (G.g_E) {   // dL/dE = C^T g (C symmetric), rotated back
        double R[6][6], ge[6];
        mandel_rotation(G.Q + 9 * pt, R);
#pragma unroll
        for (int I = 0; I < 6; ++I) {
          double v = 0.0;
#pragma unroll
          for (int J = 0; J < 6; ++J) v += M.c[6 + sidx(I, J)][p] * ((J < 3 ? 1.0 : W2) * gl[J]);
          ge[I] = (I < 3 ? 1.0 : W2) * v;
        }
#pragma unroll
        for (int I = 0; I < 6; ++I) {
          double v = 0.0;
#pragma unroll
          for (int J = 0; J < 6; ++J) v += R[I][J] * ge[J];
          G.g_E[6 * pt + I] = v;
        }
      }
    }
    __syncthreads();
    // ---- the jumps' response to the seed down (mu = H d_eps), D g_i of the leaves, the laminates' terms up
    auto down2 = [&](int j, const double e[6], double eL[6], double eR[6]) {
      const Lam<CMP> q(t, L.heap(j));
      if (CMP && q.mode) {
#pragma unroll
        for (int I = 0; I < 6; ++I) eL[I] = eR[I] = e[I];
        return;
      }
      double v[3], mu[3], Nm[6];
      normal(q.id, v);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        double m = 0.0;
#pragma unroll
        for (int I = 0; I < 6; ++I) m += X[(X_H + 18 * j + 6 * k + I) * ST] * e[I];
        X[(X_MU + 3 * j + k) * ST] = mu[k] = m;
      }
      const double vr[3] = {v[0] * RS2, v[1] * RS2, v[2] * RS2};
      N_apply<double>(v, vr, mu, Nm);
#pragma unroll
      for (int I = 0; I < 6; ++I) { eL[I] = e[I] - q.c2 * Nm[I]; eR[I] = e[I] + q.c1 * Nm[I]; }
    };
    auto up2 = [&](int j, const double sL[6], const double tL[6], const double sR[6], const double tR[6], double so[6],
                   double to[6]) {
      const Lam<CMP> q(t, L.heap(j));
      if (CMP && q.mode) {
#pragma unroll
        for (int I = 0; I < 6; ++I) { so[I] = q.mode == 2 ? sR[I] : sL[I]; to[I] = q.mode == 2 ? tR[I] : tL[I]; }
        return;
      }
      double v[3], a[3], mu[3], ds[6], dt[6], u1[3], u2[3], Nm[6], Na[6];
      normal(q.id, v);
#pragma unroll
      for (int k = 0; k < 3; ++k) { a[k] = X[(X_A + 3 * j + k) * ST]; mu[k] = X[(X_MU + 3 * j + k) * ST]; }
#pragma unroll
      for (int I = 0; I < 6; ++I) {
        ds[I] = sR[I] - sL[I]; dt[I] = tR[I] - tL[I];
        so[I] = sL[I] + q.c2 * ds[I]; to[I] = tL[I] + q.c2 * dt[I];
      }
      const double ar[3] = {a[0] * RS2, a[1] * RS2, a[2] * RS2}, mr[3] = {mu[0] * RS2, mu[1] * RS2, mu[2] * RS2};
      Nt_apply<double>(a, ar, dt, u1);    // N(a)^T (tau_R - tau_L)
      Nt_apply<double>(mu, mr, ds, u2);   // N(mu)^T (sb_R - sb_L)
      const double sc = __ldg(t.sc + q.id);
      const double gn[3] = {sc * (u1[0] + u2[0]), sc * (u1[1] + u2[1]), sc * (u1[2] + u2[2])};
      put_angles(G, i, q.id, v, gn);
      // W Xi = c1 Gam_L + c2 Gam_R = (N mu) . s + (N a) . tau of the averages
      const double vr[3] = {v[0] * RS2, v[1] * RS2, v[2] * RS2};
      N_apply<double>(v, vr, mu, Nm);
      N_apply<double>(v, vr, a, Na);
      double y = 0.0;
#pragma unroll
      for (int I = 0; I < 6; ++I) y += Nm[I] * so[I] + Na[I] * to[I];
      X[(X_Y + j) * ST] = y;
    };
    for (int l = 0; l < Kt; ++l) {
      if (act && L.lev == l) {
        double e[6], eL[6], eR[6];
        gget6(M.e, L.pos, e);
        down2(7, e, eL, eR);
        gput6(M.e, L.pos, eL);
        gput6(M.e, L.pos + L.half, eR);
      }
      __syncthreads();
    }
    if (act && !dead) {
      double e[6], eL[6], eR[6], s0[6], s1[6], t0[6], t1[6], so[6], to[6];
      gget6(M.e, tid, e);
      down2(0, e, eL, eR);
      gput6(M.e, tid, eR);
#pragma unroll
      for (int I = 0; I < 6; ++I) e[I] = eL[I];
#pragma unroll 1
      for (int q = 0; q < 4; ++q) {
        const int mid = 1 + (q >> 1);
        if (!(q & 1)) {
          down2(mid, e, eL, eR);
          gput6(M.f, tid, eR);
#pragma unroll
          for (int I = 0; I < 6; ++I) e[I] = eL[I];
        }
        down2(3 + q, e, eL, eR);
#pragma unroll
        for (int side = 0; side < 2; ++side) {
          const int l = 2 * q + side;
          const double* gi = side ? eR : eL;
          double* sg = side ? s1 : s0;
          double* tv = side ? t1 : t0;
          double gs = 0.0, mg = 0.0, m[6];
          const double mu = X[(X_T + 8 * l) * ST], lam = t.ph[side].K - (2.0 / 3.0) * mu;
#pragma unroll
          for (int I = 0; I < 6; ++I) {
            sg[I] = X[(X_S + 6 * l + I) * ST];
            m[I] = X[(X_T + 8 * l + 2 + I) * ST];
            gs += gi[I] * sg[I];
            mg += m[I] * gi[I];
          }
          const double cm = X[(X_T + 8 * l + 1) * ST] * mg, lt = lam * (gi[0] + gi[1] + gi[2]);
#pragma unroll
          for (int I = 0; I < 6; ++I) tv[I] = 2.0 * mu * gi[I] - cm * m[I] + (I < 3 ? lt : 0.0);
          X[(X_D + l) * ST] = gs;
        }
        up2(3 + q, s0, t0, s1, t1, so, to);
        if (!(q & 1)) {
          gget6(M.f, tid, e);
          gput6(M.s, tid, so);
          gput6(M.s + 6, tid, to);
        } else {
          gget6(M.s, tid, s0);
          gget6(M.s + 6, tid, t0);
          up2(mid, s0, t0, so, to, s1, t1);
          if (q == 1) {
            gget6(M.e, tid, e);
            gput6(M.c, tid, s1);
            gput6(M.c + 6, tid, t1);
          }
        }
      }
      gget6(M.c, tid, s0);
      gget6(M.c + 6, tid, t0);
      up2(0, s0, t0, s1, t1, so, to);
      gput6(M.c, tid, so);
      gput6(M.c + 6, tid, to);
    } else if (act) {
#pragma unroll
      for (int k = 0; k < 12; ++k) M.c[k][tid] = 0.0;
    }
    __syncthreads();
    for (int l = Kt - 1; l >= 0; --l) {
      if (act && L.lev == l) {
        double s0[6], s1[6], t0[6], t1[6], so[6], to[6];
        gget6(M.c, L.pos, s0);
        gget6(M.c + 6, L.pos, t0);
        gget6(M.c, L.pos + L.half, s1);
        gget6(M.c + 6, L.pos + L.half, t1);
        up2(7, s0, t0, s1, t1, so, to);
        gput6(M.c, L.pos, so);
        gput6(M.c + 6, L.pos, to);
      }
      __syncthreads();
    }
    weights<CMP, true>(G, M, L, act, dead, i, X + X_Y * ST, X + X_D * ST);
  }
}

// ---------------------------------------------------------------------------
// Tangent seeds.  Voigt components throughout (dL/dC of a Voigt tangent is w_I w_J times that of the Mandel one).

namespace {

// row . (row J of N(n)), N's rows (x, 0, 0), (0, y, 0), (0, 0, z), (0, z, y), (z, 0, x), (y, x, 0)
__device__ __forceinline__ double dot_n(const double r[3], const double n[3], int J) {
  return J < 3 ? r[J] * n[J] : J == 3 ? r[1] * n[2] + r[2] * n[1] : J == 4 ? r[0] * n[2] + r[2] * n[0]
                                                                           : r[0] * n[1] + r[1] * n[0];
}
// G += P N^T + N P^T (packed)
__device__ __forceinline__ void add_sym(const double P[6][3], const double n[3], double G[21]) {
#pragma unroll
  for (int I = 0; I < 6; ++I)
#pragma unroll
    for (int J = I; J < 6; ++J) G[sidx(I, J)] += dot_n(P[I], n, J) + dot_n(P[J], n, I);
}

// lam_tangent_adjoint: from G = dL/dC of a laminate its children's (in GL, GR; KIDS), dL/dn and dL/dc1
template <bool KIDS>
__device__ __forceinline__ void tangent_adjoint(const double n[3], double c1, double c2, const double CL[21],
                                                const double CR[21], const double G[21], double GL[21], double GR[21],
                                                double nb[3], double& c1b) {
  double dC[21], H[21], B[6][3], A[6][3], Ki[3][3], T[6][3], Kb[3][3];
#pragma unroll
  for (int k = 0; k < 21; ++k) { dC[k] = CR[k] - CL[k]; H[k] = CR[k] - c2 * dC[k]; }
  times_n(H, n, A);
  times_n(dC, n, B);
  double col[6];
  double Km[3][3], NB[3][3];
#pragma unroll
  for (int j = 0; j < 3; ++j) {   // N^T A and N^T B (symmetric)
#pragma unroll
    for (int I = 0; I < 6; ++I) col[I] = A[I][j];
    Km[0][j] = n[0] * col[0] + n[2] * col[4] + n[1] * col[5];
    Km[1][j] = n[1] * col[1] + n[2] * col[3] + n[0] * col[5];
    Km[2][j] = n[2] * col[2] + n[1] * col[3] + n[0] * col[4];
#pragma unroll
    for (int I = 0; I < 6; ++I) col[I] = B[I][j];
    NB[0][j] = n[0] * col[0] + n[2] * col[4] + n[1] * col[5];
    NB[1][j] = n[1] * col[1] + n[2] * col[3] + n[0] * col[5];
    NB[2][j] = n[2] * col[2] + n[1] * col[3] + n[0] * col[4];
  }
  inv3_sym<double>(Km[0][0], Km[0][1], Km[0][2], Km[1][1], Km[1][2], Km[2][2], Ki);
  const double c12 = c1 * c2;
  double gBY = 0.0, gLR = 0.0, kNB = 0.0;
  {
    double Y[3][6];
#pragma unroll
    for (int m = 0; m < 3; ++m)
#pragma unroll
      for (int J = 0; J < 6; ++J) Y[m][J] = Ki[m][0] * B[J][0] + Ki[m][1] * B[J][1] + Ki[m][2] * B[J][2];
#pragma unroll
    for (int I = 0; I < 6; ++I)
#pragma unroll
      for (int m = 0; m < 3; ++m) {
        double v = 0.0;
#pragma unroll
        for (int J = 0; J < 6; ++J) v += G[sidx(I, J)] * Y[m][J];
        T[I][m] = v;
        gBY += B[I][m] * v;
      }
#pragma unroll
    for (int m = 0; m < 3; ++m)
#pragma unroll
      for (int k = m; k < 3; ++k) {
        double v = 0.0;
#pragma unroll
        for (int I = 0; I < 6; ++I) v += Y[m][I] * T[I][k];
        Kb[m][k] = Kb[k][m] = c12 * v;
      }
  }
#pragma unroll
  for (int I = 0; I < 6; ++I)
#pragma unroll
    for (int J = I; J < 6; ++J) gLR -= (I == J ? 1.0 : 2.0) * G[sidx(I, J)] * dC[sidx(I, J)];
#pragma unroll
  for (int m = 0; m < 3; ++m)
#pragma unroll
    for (int k = 0; k < 3; ++k) kNB += Kb[m][k] * NB[m][k];
  c1b = gLR - (c2 - c1) * gBY + kNB;
  const double b2 = -2.0 * c12;
#pragma unroll
  for (int I = 0; I < 6; ++I)
#pragma unroll
    for (int m = 0; m < 3; ++m) T[I][m] *= b2;   // dL/dB
  // dL/dN = 2 A Kb + dC (dL/dB) at N's entries, summed into dL/dn
  auto Nb = [&](int I, int k) {
    double v = 2.0 * (A[I][0] * Kb[0][k] + A[I][1] * Kb[1][k] + A[I][2] * Kb[2][k]);
#pragma unroll
    for (int J = 0; J < 6; ++J) v += dC[sidx(I, J)] * T[J][k];
    return v;
  };
  nb[0] = Nb(0, 0) + Nb(4, 2) + Nb(5, 1);
  nb[1] = Nb(1, 1) + Nb(3, 2) + Nb(5, 0);
  nb[2] = Nb(2, 2) + Nb(3, 1) + Nb(4, 0);
  if (!KIDS) return;   // leaves
  double P[6][3], NK[6][3];
#pragma unroll
  for (int I = 0; I < 6; ++I)
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const double r[3] = {Kb[0][k], Kb[1][k], Kb[2][k]};
      NK[I][k] = 0.5 * dot_n(r, n, I);
      P[I][k] = c2 * NK[I][k] - 0.5 * T[I][k];
    }
#pragma unroll
  for (int k = 0; k < 21; ++k) GL[k] = c1 * G[k];
  add_sym(P, n, GL);
#pragma unroll
  for (int I = 0; I < 6; ++I)
#pragma unroll
    for (int k = 0; k < 3; ++k) P[I][k] = c1 * NK[I][k] + 0.5 * T[I][k];
#pragma unroll
  for (int k = 0; k < 21; ++k) GR[k] = c2 * G[k];
  add_sym(P, n, GR);
}

__device__ __forceinline__ void voigt_iso(const PhaseDev& ph, double C[21]) {
#pragma unroll
  for (int I = 0; I < 6; ++I)
#pragma unroll
    for (int J = I; J < 6; ++J)
      C[sidx(I, J)] = J < 3 ? (I == J ? ph.lam + 2.0 * ph.G : ph.lam) : (I == J ? ph.G : 0.0);
}

}  // namespace

template <bool CMP>
__global__ void __launch_bounds__(ST, SWEEP_CTAS_PER_SM) k_grad_tangent_block(GradWork G) {
  extern __shared__ __align__(16) char dyn[];
  GradShared& M = *reinterpret_cast<GradShared*>(dyn);
  const int tid = threadIdx.x;
  const TreeDev& t = G.t;
  const Place L(t.K);
  const int Kt = L.Kt, nP = L.nP, s = L.s, p = L.p;
  double* Z = G.scratch + (size_t)blockIdx.x * GRAD_SCRATCH_DOUBLES * ST + tid;
  const size_t ws = (size_t)G.nc;
  const bool dead = CMP && __ldg(t.hdir + L.heap(0)) == 3;
  for (int64_t g0 = (int64_t)blockIdx.x * nP; g0 < G.nc; g0 += (int64_t)gridDim.x * nP) {
    const size_t i = (size_t)(g0 + p);
    const bool act = (int64_t)i < G.nc;
    const size_t pt = (size_t)G.n0 + i;
    auto normal = [&](int id, double v[3]) {
#pragma unroll
      for (int k = 0; k < 3; ++k) v[k] = G.work[(3 * id + k) * ws + i];
    };
    auto load = [&](int j, double C[21]) {
#pragma unroll
      for (int k = 0; k < 21; ++k) C[k] = Z[(Z_C + 21 * j + k) * ST];
    };
    // ---- stiffnesses up (a laminate's own result kept)
    auto up = [&](int j, const double A[21], const double B[21], double o[21]) {
      const Lam<CMP> q(t, L.heap(j));
      if (CMP && q.mode) {
#pragma unroll
        for (int k = 0; k < 21; ++k) o[k] = q.mode == 2 ? B[k] : A[k];
      } else {
        double v[3], dC[21], H[21], Bn[6][3], k00, k01, k02, k11, k12, k22;
        normal(q.id, v);
#pragma unroll
        for (int k = 0; k < 21; ++k) { dC[k] = B[k] - A[k]; H[k] = B[k] - q.c2 * dC[k]; o[k] = A[k] + q.c2 * dC[k]; }
        acoustic(H, v, k00, k01, k02, k11, k12, k22);
        times_n(dC, v, Bn);
        Downdate{}(k00, k01, k02, k11, k12, k22, Bn, q.c1 * q.c2, o);
      }
#pragma unroll
      for (int k = 0; k < 21; ++k) Z[(Z_C + 21 * j + k) * ST] = o[k];
    };
    if (act && !dead) {
      double x[21], y[21], o[21];
#pragma unroll 1
      for (int q = 0; q < 4; ++q) {
        voigt_iso(t.ph[0], x);
        voigt_iso(t.ph[1], y);
        up(3 + q, x, y, o);
      }
#pragma unroll 1
      for (int j = 2; j >= 0; --j) {
        load(2 * j + 1, x);
        load(2 * j + 2, y);
        up(j, x, y, o);
      }
      gput21(M.c, tid, o);
    } else if (act) {
#pragma unroll
      for (int k = 0; k < 21; ++k) M.c[k][tid] = 0.0;
    }
    __syncthreads();
    for (int l = Kt - 1; l >= 0; --l) {
      if (act && L.lev == l) {
        double A[21], B[21], o[21];
        gget21(M.c, L.pos, A);
        gget21(M.c, L.pos + L.half, B);
        up(7, A, B, o);
        gput21(M.c, L.pos, o);
      }
      __syncthreads();
    }
    if (act && s == 0) {   // the seed in the local frame, symmetrised: C_glob = R C_loc R^T => R^T G R
      double R[6][6], RG[6][6];
      mandel_rotation(G.Q + 9 * pt, R);
      const double* g = G.g_tangent + 36 * pt;
      for (int a = 0; a < 6; ++a)
        for (int J = 0; J < 6; ++J) {
          double v = 0.0;
          for (int I = 0; I < 6; ++I) v += R[I][a] * g[6 * I + J];
          RG[a][J] = v;
        }
      for (int I = 0; I < 6; ++I)
        for (int J = I; J < 6; ++J) {
          double a = 0.0, b = 0.0;
          for (int k = 0; k < 6; ++k) { a += RG[I][k] * R[k][J]; b += RG[J][k] * R[k][I]; }
          M.c[sidx(I, J)][p] = 0.5 * (a + b) * (I < 3 ? 1.0 : W2) * (J < 3 ? 1.0 : W2);
        }
      if (G.g_E)   // the tangent of elastic phases does not depend on the macro strain
        for (int I = 0; I < 6; ++I) G.g_E[6 * pt + I] = 0.0;
    }
    __syncthreads();
    // ---- adjoints down
    auto rev = [&](int j, const double A[21], const double B[21], const double g[21], double GL[21], double GR[21],
                   auto kids) {
      const Lam<CMP> q(t, L.heap(j));
      if (CMP && q.mode) {
#pragma unroll
        for (int k = 0; k < 21; ++k) { GL[k] = g[k]; GR[k] = g[k]; }   // the weightless side's is never used
        return;
      }
      double v[3], nb[3], c1b;
      normal(q.id, v);
      tangent_adjoint<decltype(kids)::value>(v, q.c1, q.c2, A, B, g, GL, GR, nb, c1b);
      put_angles(G, i, q.id, v, nb);
      Z[(Z_Y + j) * ST] = c1b / (__ldg(t.sc + q.id) * __ldg(t.ic12 + q.id));   // W Xi = (dL/dc1) / W
    };
    // a top laminate's children: laminates of this CTA's threads s' = 2 s, 2 s + 1 (their top laminate, or the
    // root of their subtree)
    auto kid = [&](int side, double C[21]) {
      const int h1 = 2 * s + side;
      const int os = h1 < L.S ? h1 : h1 - L.S, oj = h1 < L.S ? 7 : 0;
      const double* o = Z - tid + (os * nP + p);
      const bool none = CMP && oj == 0 && __ldg(t.hdir + h1 - 1) == 3;
#pragma unroll
      for (int k = 0; k < 21; ++k) C[k] = none ? 0.0 : o[(Z_C + 21 * oj + k) * ST];
    };
    for (int l = 0; l < Kt; ++l) {
      if (act && L.lev == l) {
        double A[21], B[21], g[21], GL[21], GR[21];
        kid(0, A);
        kid(1, B);
        gget21(M.c, L.pos, g);
        rev(7, A, B, g, GL, GR, std::true_type{});
        gput21(M.c, L.pos, GL);
        gput21(M.c, L.pos + L.half, GR);
      }
      __syncthreads();
    }
    if (act && !dead) {
      double A[21], B[21], g[21], GL[21], GR[21];
      gget21(M.c, tid, g);
      load(1, A);
      load(2, B);
      rev(0, A, B, g, GL, GR, std::true_type{});
      gput21(M.c, tid, GR);
#pragma unroll
      for (int k = 0; k < 21; ++k) g[k] = GL[k];
#pragma unroll 1
      for (int q = 0; q < 4; ++q) {
        if (!(q & 1)) {
          const int mid = 1 + (q >> 1);
          load(2 * mid + 1, A);
          load(2 * mid + 2, B);
          rev(mid, A, B, g, GL, GR, std::true_type{});
          gput21(M.s, tid, GR);
#pragma unroll
          for (int k = 0; k < 21; ++k) g[k] = GL[k];
        }
        voigt_iso(t.ph[0], A);
        voigt_iso(t.ph[1], B);
        rev(3 + q, A, B, g, GL, GR, std::false_type{});
        if (!(q & 1)) gget21(M.s, tid, g);
        else if (q == 1) gget21(M.c, tid, g);
      }
    }
    __syncthreads();
    weights<CMP, false>(G, M, L, act, dead, i, Z + Z_Y * ST, nullptr);
  }
}

template <typename Kernel>
static cudaError_t run(Kernel k, const GradWork& G, unsigned grid, cudaStream_t s) {
  const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(GradShared));
  if (e != cudaSuccess) return e;
  k<<<grid, ST, sizeof(GradShared), s>>>(G);
  return cudaSuccess;
}

cudaError_t launch_grad_normals(const GradWork& G, unsigned split, cudaStream_t s) {
  k_grad_normals<<<dim3((unsigned)((G.nc + 127) / 128), split), 128, 0, s>>>(G);
  return cudaSuccess;
}
cudaError_t launch_grad_block(const GradWork& G, bool cmp, bool tangent, unsigned grid, cudaStream_t s) {
  if (tangent) return cmp ? run(k_grad_tangent_block<true>, G, grid, s) : run(k_grad_tangent_block<false>, G, grid, s);
  return cmp ? run(k_grad_block<true>, G, grid, s) : run(k_grad_block<false>, G, grid, s);
}

}  // namespace dmn
