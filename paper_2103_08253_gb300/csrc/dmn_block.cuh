// The CTA organisation's laminate lookup and FP64 condensation, shared by the sweep (csrc/dmn_block.cu) and the
// adjoints (csrc/dmn_grad.cu).  See dmn_block.cu for the organisation.
#pragma once
#include "dmn_launch.cuh"

namespace dmn {

// laminate h (heap order, 0-based) of the full tree: its number in the handle's arrays and its fractions.
// mode 0: a laminate; 1 / 2: passes its left / right side on (the other is weightless); 3: nothing alive
template <bool CMP>
struct Lam {
  int id, mode;
  double c1, c2;
  __device__ Lam(const TreeDev& t, int h) {
    mode = CMP ? __ldg(t.hdir + h) : 0;
    id = CMP ? __ldg(t.hcid + h) : h;
    if (!CMP || mode == 0) { c1 = __ldg(t.c1 + id); c2 = __ldg(t.c2 + id); }
    else { c1 = c2 = 0.0; }
  }
};

constexpr int ST = SWEEP_THREADS;

struct Sub64 {
  double sb[6], C[21];
};

// The two ends of a condensation, from Kn (symmetric positive definite), B = (C_R - C_L) N and the average C:
// Downdate, C -= c12 B Kn^-1 B^T alone;
struct Downdate {
  __device__ __forceinline__ void operator()(double k00, double k01, double k02, double k11, double k12, double k22,
                                             double B[6][3], double c12, double C[21]) const {
  const double i0 = 1.0 / k00, l10 = k01 * i0, l20 = k02 * i0;
  const double d1 = k11 - l10 * k01, s12 = k12 - l10 * k02, s22 = k22 - l20 * k02;
  const double t = s22 * d1 - s12 * s12, r = 1.0 / (d1 * t);   // t = d1 d2: one division for 1 / d1 and 1 / d2
  const double i1 = r * t, i2 = d1 * (r * d1), l21 = s12 * i1;
  const double w0 = -c12 * i0, w1 = -c12 * i1, w2 = -c12 * i2;
#pragma unroll
  for (int I = 0; I < 6; ++I) {
    B[I][1] -= l10 * B[I][0];
    B[I][2] -= l20 * B[I][0] + l21 * B[I][1];
  }
#pragma unroll
  for (int I = 0; I < 6; ++I) {
    const double z0 = w0 * B[I][0], z1 = w1 * B[I][1], z2 = w2 * B[I][2];
#pragma unroll
    for (int J = I; J < 6; ++J) {
      double v = C[sidx(I, J)];
      v += z0 * B[J][0];
      v += z1 * B[J][1];
      v += z2 * B[J][2];
      C[sidx(I, J)] = v;
    }
  }
}
};
// StoreH, the same and H = -Kn^-1 B^T for Mandel strain perturbations, the jump response (entry k at H[k * stride]).
struct StoreH {
  double* H;
  size_t stride;
  __device__ __forceinline__ void operator()(double k00, double k01, double k02, double k11, double k12, double k22,
                                             double B[6][3], double c12, double C[21]) const {
    double Ki[3][3], h[3][6];
    inv3_sym<double>(k00, k01, k02, k11, k12, k22, Ki);
#pragma unroll
    for (int m = 0; m < 3; ++m)
#pragma unroll
      for (int I = 0; I < 6; ++I) {
        h[m][I] = -(Ki[m][0] * B[I][0] + Ki[m][1] * B[I][1] + Ki[m][2] * B[I][2]);
        H[(6 * m + I) * stride] = I < 3 ? h[m][I] : 1.41421356237309504880 * h[m][I];
      }
#pragma unroll
    for (int I = 0; I < 6; ++I) {
      const double b[3] = {c12 * B[I][0], c12 * B[I][1], c12 * B[I][2]};
#pragma unroll
      for (int J = I; J < 6; ++J) {
        double v = C[sidx(I, J)];
        v += b[0] * h[0][J];
        v += b[1] * h[1][J];
        v += b[2] * h[2][J];
        C[sidx(I, J)] = v;
      }
    }
  }
};

// Kn = N^T Ch N of a packed Voigt tangent Ch, as quadratic forms in n
__device__ __forceinline__ void acoustic(const double H[21], const double n[3], double& k00, double& k01, double& k02,
                                         double& k11, double& k12, double& k22) {
  const double x = n[0], y = n[1], z = n[2], xx = x * x, yy = y * y, zz = z * z, xy = x * y, xz = x * z, yz = y * z;
  const double xy2 = 2.0 * xy, xz2 = 2.0 * xz, yz2 = 2.0 * yz;
#define C_(i, j) H[sidx(i, j)]
  k00 = C_(0, 0) * xx + C_(5, 5) * yy + C_(4, 4) * zz + C_(0, 5) * xy2 + C_(0, 4) * xz2 + C_(4, 5) * yz2;
  k11 = C_(5, 5) * xx + C_(1, 1) * yy + C_(3, 3) * zz + C_(1, 5) * xy2 + C_(3, 5) * xz2 + C_(1, 3) * yz2;
  k22 = C_(4, 4) * xx + C_(3, 3) * yy + C_(2, 2) * zz + C_(3, 4) * xy2 + C_(2, 4) * xz2 + C_(2, 3) * yz2;
  k01 = C_(0, 5) * xx + C_(1, 5) * yy + C_(3, 4) * zz + (C_(0, 1) + C_(5, 5)) * xy +
                     (C_(0, 3) + C_(4, 5)) * xz + (C_(1, 4) + C_(3, 5)) * yz;
  k02 = C_(0, 4) * xx + C_(3, 5) * yy + C_(2, 4) * zz + (C_(0, 3) + C_(4, 5)) * xy +
                     (C_(0, 2) + C_(4, 4)) * xz + (C_(2, 5) + C_(3, 4)) * yz;
  k12 = C_(4, 5) * xx + C_(1, 3) * yy + C_(2, 3) * zz + (C_(3, 5) + C_(1, 4)) * xy +
                     (C_(2, 5) + C_(3, 4)) * xz + (C_(1, 2) + C_(3, 3)) * yz;
#undef C_
}
// B = dC N: the columns of N are (x, 0, 0, 0, z, y), (0, y, 0, z, 0, x), (0, 0, z, y, x, 0)
__device__ __forceinline__ void times_n(const double dC[21], const double n[3], double B[6][3]) {
  const double x = n[0], y = n[1], z = n[2];
#pragma unroll
  for (int I = 0; I < 6; ++I) {
    B[I][0] = dC[sidx(I, 0)] * x + dC[sidx(I, 4)] * z + dC[sidx(I, 5)] * y;
    B[I][1] = dC[sidx(I, 1)] * y + dC[sidx(I, 3)] * z + dC[sidx(I, 5)] * x;
    B[I][2] = dC[sidx(I, 2)] * z + dC[sidx(I, 3)] * y + dC[sidx(I, 4)] * x;
  }
}

// laminate with normal n: L and R condensed into o (Voigt tangents)
template <typename End>
__device__ __forceinline__ void condense64(const double n[3], double c2, double c12, const Sub64& L, const Sub64& R,
                                           Sub64& o, const End& end) {
#pragma unroll
  for (int I = 0; I < 6; ++I) o.sb[I] = L.sb[I] + c2 * (R.sb[I] - L.sb[I]);
  double dC[21], H[21], B[6][3];
#pragma unroll
  for (int k = 0; k < 21; ++k) { dC[k] = R.C[k] - L.C[k]; H[k] = R.C[k] - c2 * dC[k]; o.C[k] = L.C[k] + c2 * dC[k]; }
  double k00, k01, k02, k11, k12, k22;
  acoustic(H, n, k00, k01, k02, k11, k12, k22);
  times_n(dC, n, B);
  end(k00, k01, k02, k11, k12, k22, B, c12, o.C);
}

// bottom laminate from its leaves' tangents lam 1(x)1 + 2 mu I - c m(x)m (condense_bottom in Voigt components);
// el: the phase is elastic, c = 0.  c1 + c2 = 1; a passed-on side has fraction 1 and no normal (n = 0, c12 = 0).
template <typename End>
__device__ __forceinline__ void condense64_bottom(const double n[3], double c1, double c2, double c12,
                                                  const double sL[6], const LeafTan<double>& L, bool elL,
                                                  const double sR[6], const LeafTan<double>& R, bool elR, Sub64& o,
                                                  const End& end) {
#pragma unroll
  for (int I = 0; I < 6; ++I) o.sb[I] = sL[I] + c2 * (sR[I] - sL[I]);
  const double lam = c1 * L.lam + c2 * R.lam, mu = c1 * L.mu + c2 * R.mu;
#pragma unroll
  for (int I = 0; I < 6; ++I)
#pragma unroll
    for (int J = I; J < 6; ++J) o.C[sidx(I, J)] = J < 3 ? (I == J ? lam + 2.0 * mu : lam) : (I == J ? mu : 0.0);
  const double a = c2 * L.mu + c1 * R.mu, b = c2 * (L.lam + L.mu) + c1 * (R.lam + R.mu);
  const double bx = b * n[0], by = b * n[1], bz = b * n[2];
  double k00 = bx * n[0] + a, k01 = bx * n[1], k02 = bx * n[2], k11 = by * n[1] + a, k12 = by * n[2], k22 = bz * n[2] + a;
  const double dlam = R.lam - L.lam, dmu = R.mu - L.mu, dld = dlam + 2.0 * dmu;
  double B[6][3];
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const double l = dlam * n[j], d = dmu * n[j];
#pragma unroll
    for (int I = 0; I < 3; ++I) B[I][j] = I == j ? dld * n[j] : l;
    // shear rows 23, 13, 12: entry (row, column) is dmu times the other index's component
    if (j == 0) { B[4][2] = d; B[5][1] = d; }
    if (j == 1) { B[3][2] = d; B[5][0] = d; }
    if (j == 2) { B[3][1] = d; B[4][0] = d; }
  }
  B[3][0] = 0.0; B[4][1] = 0.0; B[5][2] = 0.0;
  auto leaf = [&](const LeafTan<double>& D, double frac, double other, double sign) {
    const double m[6] = {D.m[0], D.m[1], D.m[2], RS2 * D.m[3], RS2 * D.m[4], RS2 * D.m[5]};
    const double u[3] = {m[0] * n[0] + m[4] * n[2] + m[5] * n[1], m[1] * n[1] + m[3] * n[2] + m[5] * n[0],
                         m[2] * n[2] + m[3] * n[1] + m[4] * n[0]};
    const double w = -other * D.c, wx = w * u[0], wy = w * u[1], wz = w * u[2];
    k00 += wx * u[0]; k01 += wx * u[1]; k02 += wx * u[2]; k11 += wy * u[1]; k12 += wy * u[2]; k22 += wz * u[2];
#pragma unroll
    for (int I = 0; I < 6; ++I) {
      const double cm = D.c * m[I], h = -frac * cm, s = sign * cm;
#pragma unroll
      for (int j = 0; j < 3; ++j) B[I][j] += s * u[j];
#pragma unroll
      for (int J = I; J < 6; ++J) o.C[sidx(I, J)] += h * m[J];
    }
  };
  if (!elL) leaf(L, c1, c2, 1.0);
  if (!elR) leaf(R, c2, c1, -1.0);
  end(k00, k01, k02, k11, k12, k22, B, c12, o.C);
}

struct SweepShared {
  double e[6][ST], f[6][ST];       // strains handed down; set aside by the bottom walk
  double c[27][ST], s[27][ST];     // results handed up; set aside
};
__device__ __forceinline__ void put27(double (*m)[ST], int x, const Sub64& v) {
#pragma unroll
  for (int I = 0; I < 6; ++I) m[I][x] = v.sb[I];
#pragma unroll
  for (int k = 0; k < 21; ++k) m[6 + k][x] = v.C[k];
}
__device__ __forceinline__ void get27(double (*m)[ST], int x, Sub64& v) {
#pragma unroll
  for (int I = 0; I < 6; ++I) v.sb[I] = m[I][x];
#pragma unroll
  for (int k = 0; k < 21; ++k) v.C[k] = m[6 + k][x];
}
__device__ __forceinline__ void sput6(double (*m)[ST], int x, const double v[6]) {
#pragma unroll
  for (int I = 0; I < 6; ++I) m[I][x] = v[I];
}
__device__ __forceinline__ void sget6(double (*m)[ST], int x, double v[6]) {
#pragma unroll
  for (int I = 0; I < 6; ++I) v[I] = m[I][x];
}

}  // namespace dmn
