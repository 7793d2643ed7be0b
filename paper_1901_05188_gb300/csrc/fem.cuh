// Device-side finite-element arithmetic (Sec. 2): orthotropic Hooke law,
// ply rotation and blocks of the trilinear hexahedral element stiffness.
#pragma once

#include "common.cuh"

namespace geneo {

// Voigt index of the symmetric pair (i, j): order 11, 22, 33, 23, 13, 12.
__device__ __forceinline__ int voigt(int i, int j) {
  // table {{0,5,4},{5,1,3},{4,3,2}} packed 3 bits per entry
  const unsigned t = 0u | (5u << 3) | (4u << 6) | (5u << 9) | (1u << 12) | (3u << 15) |
                     (4u << 18) | (3u << 21) | (2u << 24);
  return (t >> (3 * (3 * i + j))) & 7u;
}

// 6x6 stiffness (row-major) of an orthotropic material in its own axes:
// invert the compliance built from the nine engineering constants (Sec. 2).
__device__ inline void material_stiffness(const geneo_ortho &m, double C[36]) {
  double S[36];
  for (int i = 0; i < 36; ++i) S[i] = 0.0;
  S[0] = 1.0 / m.E1;
  S[7] = 1.0 / m.E2;
  S[14] = 1.0 / m.E3;
  S[1] = S[6] = -m.nu12 / m.E1;
  S[2] = S[12] = -m.nu13 / m.E1;
  S[8] = S[13] = -m.nu23 / m.E2;
  S[21] = 1.0 / m.G23;
  S[28] = 1.0 / m.G13;
  S[35] = 1.0 / m.G12;
  // Gauss-Jordan with partial pivoting on [S | I]
  double Aug[6][12];
  for (int i = 0; i < 6; ++i)
    for (int j = 0; j < 12; ++j) Aug[i][j] = j < 6 ? S[6 * i + j] : (j - 6 == i ? 1.0 : 0.0);
  for (int c = 0; c < 6; ++c) {
    int piv = c;
    for (int r = c + 1; r < 6; ++r)
      if (fabs(Aug[r][c]) > fabs(Aug[piv][c])) piv = r;
    if (piv != c)
      for (int j = 0; j < 12; ++j) {
        double t = Aug[c][j];
        Aug[c][j] = Aug[piv][j];
        Aug[piv][j] = t;
      }
    double inv = 1.0 / Aug[c][c];
    for (int j = 0; j < 12; ++j) Aug[c][j] *= inv;
    for (int r = 0; r < 6; ++r) {
      if (r == c) continue;
      double f = Aug[r][c];
      for (int j = 0; j < 12; ++j) Aug[r][j] -= f * Aug[c][j];
    }
  }
  for (int i = 0; i < 6; ++i)
    for (int j = 0; j < 6; ++j) C[6 * i + j] = Aug[i][6 + j];
}

// Rotate an orthotropic Voigt stiffness from ply axes to global axes with the
// stress transformation (Bond) matrix M of Q = R_z(theta) R_y(phi): C' = M C M^T.
// The fibre direction Q e1 is (cos t cos p, sin t cos p, -sin p).  In its own
// axes C couples only the three normal components and is diagonal in the
// shears, and C' is symmetric: 198 multiply-adds instead of 432.
__device__ inline void rotate_voigt(const double *__restrict__ C, double theta, double phi,
                                    double *__restrict__ Cr) {
  double ct, st, cp, sp;
  sincos(theta, &st, &ct);
  sincos(phi, &sp, &cp);
  // Q = Rz * Ry
  const double Q[3][3] = {{ct * cp, -st, ct * sp}, {st * cp, ct, st * sp}, {-sp, 0.0, cp}};
  constexpr int VI[6] = {0, 1, 2, 1, 0, 0};
  constexpr int VJ[6] = {0, 1, 2, 2, 2, 1};
  double M[6][6];
#pragma unroll
  for (int I = 0; I < 6; ++I)
#pragma unroll
    for (int J = 0; J < 6; ++J) {
      const int i = VI[I], j = VJ[I], k = VI[J], l = VJ[J];
      double v = Q[i][k] * Q[j][l];
      if (k != l) v += Q[i][l] * Q[j][k];
      M[I][J] = v;
    }
#pragma unroll
  for (int I = 0; I < 6; ++I) {
    double t[6];                                // row I of M C
#pragma unroll
    for (int J = 0; J < 3; ++J)
      t[J] = M[I][0] * C[J] + M[I][1] * C[6 + J] + M[I][2] * C[12 + J];
#pragma unroll
    for (int J = 3; J < 6; ++J) t[J] = M[I][J] * C[7 * J];
#pragma unroll
    for (int J = I; J < 6; ++J) {
      double s = 0.0;
#pragma unroll
      for (int K = 0; K < 6; ++K) s += t[K] * M[J][K];
      Cr[6 * I + J] = s;
      Cr[6 * J + I] = s;
    }
  }
}

// ---- rows of the Q1 stiffness, node by node ----------------------------------
// The 3x3 (or 1x1) block of local nodes a, b of an axis-aligned box element is
//   K_ab[i][k] = sum_{j,l} C_ijkl int d_j N_a d_l N_b,
// with trilinear N and integrals that are products of 1D integrals of linear
// factors (equal to the 2x2x2 Gauss rule, which is exact for them).  With the
// corner signs s_a, s_b in {-1, 1}^3 a 1D mass factor is h/4 + s_a s_b h/12, a
// mixed one s/2 and a stiffness one s_a s_b / h, so for one component pair
// (i, k) all 64 blocks follow from the nine numbers
//   T[j][l] = C_ijkl g_jl,  g_jj = h_e h_f / (16 h_j),  g_jl = h_e / 16
// (e, f the other axes): with w = s_0 s_1 s_2, r = T^T s_a, t = tr T,
//   K_ab = r . s_b + w_a w_b (q . s_b + t / 9),
//   3 q = T s_a + s_a o (t - 2 diag T).
// Every s is a compile-time sign, so a corner's row of eight blocks takes
// about 45 FP64 operations per component pair instead of the 81 multiply-adds
// per block of the direct sum over (j, l); FP64 issue (two per clock and SM)
// is what bounds the assembly on this GPU.

// Axis data of a node's two adjacent elements: [0] starts at the node, [1] ends there.
struct NodeAxis {
  double h[2], r[2];   // size and 1 / size
  bool in[2];          // the element exists (in [lo, hi))
};
__device__ __forceinline__ NodeAxis node_axis(const double *__restrict__ X, int i, int lo, int hi) {
  NodeAxis a;
#pragma unroll
  for (int b = 0; b < 2; ++b) {
    const int e = i - b;
    a.in[b] = e >= lo && e < hi;
    a.h[b] = a.in[b] ? X[e + 1] - X[e] : 1.0;
    a.r[b] = 1.0 / a.h[b];
  }
  return a;
}

// Adds r . s_b + w_a w_b (q . s_b + t9) to the slot of every local node b of
// the element in which the node is corner A (slot = dx + 3 dy + 9 dz, offset
// of b from A in -1..1 per axis, plus 13).
__device__ __forceinline__ void spread_corner(int A, const double (&r)[3], const double (&q)[3],
                                              double t9, double (&acc)[27]) {
  const int wa = ((A & 1) ^ ((A >> 1) & 1) ^ (A >> 2)) ? 1 : -1;   // s_0 s_1 s_2 of corner A
#pragma unroll
  for (int half = 0; half < 2; ++half) {      // corners b with w_a w_b = +1, then -1
    const int sg = half ? -1 : 1;
    const double p0 = r[0] + sg * q[0], p1 = r[1] + sg * q[1], p2 = r[2] + sg * q[2];
    const double t = sg * t9;
    const double up = t + p0, dn = t - p0, su = p1 + p2, di = p1 - p2;
#pragma unroll
    for (int b = 0; b < 8; ++b) {
      const int b0 = b & 1, b1 = (b >> 1) & 1, b2 = b >> 2;
      const int wb = (b0 ^ b1 ^ b2) ? 1 : -1;
      if (wa * wb != sg) continue;
      const double in = b1 == b2 ? su : di, ou = b0 ? up : dn;
      const int slot = 13 + (b0 - (A & 1)) + 3 * (b1 - ((A >> 1) & 1)) + 9 * (b2 - (A >> 2));
      acc[slot] += b1 ? ou + in : ou - in;
    }
  }
}

// The nine numbers T of one component pair from the element's coefficients
// c[off[3 j + l]] and the box scalings of corner A's element.
__device__ __forceinline__ void corner_T(const double *__restrict__ c, const int (&off)[9], double hx,
                                         double hy, double hz, double rx, double ry, double rz,
                                         double (&T)[9]) {
  const double fx = 0.0625 * hx, fy = 0.0625 * hy, fz = 0.0625 * hz;
  T[0] = __ldg(c + off[0]) * (fy * hz * rx);
  T[4] = __ldg(c + off[4]) * (fx * hz * ry);
  T[8] = __ldg(c + off[8]) * (fx * hy * rz);
  T[1] = __ldg(c + off[1]) * fz;
  T[3] = __ldg(c + off[3]) * fz;
  T[2] = __ldg(c + off[2]) * fy;
  T[6] = __ldg(c + off[6]) * fy;
  T[5] = __ldg(c + off[5]) * fx;
  T[7] = __ldg(c + off[7]) * fx;
}

// Blocks (i, k) in acc and, for a pair i != k, (k, i) in acct of a node's 27
// slots, summed over its (up to eight) elements for which take(e) holds.
// `off` indexes the element's 6x6 Voigt stiffness.
template <bool kPair, typename Take>
__device__ __forceinline__ void elastic_rows(const double *__restrict__ Cel, const int (&off)[9],
                                             const NodeAxis &ax, const NodeAxis &ay,
                                             const NodeAxis &az, int gi, int gj, int gk, int nx,
                                             int ny, Take take, double (&acc)[27],
                                             double (&acct)[27]) {
  const double third = 1.0 / 3.0;
#pragma unroll
  for (int A = 0; A < 8; ++A) {
    const int a0 = A & 1, a1 = (A >> 1) & 1, a2 = A >> 2;
    if (!(ax.in[a0] && ay.in[a1] && az.in[a2])) continue;
    const int ex = gi - a0, ey = gj - a1, ez = gk - a2;
    if (!take(ex, ey, ez)) continue;
    double T[9];
    corner_T(Cel + 36 * (size_t)(ex + nx * (ey + ny * ez)), off, ax.h[a0], ay.h[a1], az.h[a2],
             ax.r[a0], ay.r[a1], az.r[a2], T);
    const int s0 = a0 ? 1 : -1, s1 = a1 ? 1 : -1, s2 = a2 ? 1 : -1;
    const double tr = (T[0] + T[4]) + T[8], t9 = tr * (1.0 / 9.0);
    double r[3], q[3];
    r[0] = s0 * T[0] + s1 * T[3] + s2 * T[6];
    r[1] = s0 * T[1] + s1 * T[4] + s2 * T[7];
    r[2] = s0 * T[2] + s1 * T[5] + s2 * T[8];
    const double e0 = s0 * third * (tr - 2.0 * T[0]), e1 = s1 * third * (tr - 2.0 * T[4]),
                 e2 = s2 * third * (tr - 2.0 * T[8]);
    if (kPair) {
      double rt[3];                            // T s_a: the same for the transposed block
      rt[0] = s0 * T[0] + s1 * T[1] + s2 * T[2];
      rt[1] = s0 * T[3] + s1 * T[4] + s2 * T[5];
      rt[2] = s0 * T[6] + s1 * T[7] + s2 * T[8];
      q[0] = fma(third, rt[0], e0);
      q[1] = fma(third, rt[1], e1);
      q[2] = fma(third, rt[2], e2);
      spread_corner(A, r, q, t9, acc);
      q[0] = fma(third, r[0], e0);
      q[1] = fma(third, r[1], e1);
      q[2] = fma(third, r[2], e2);
      spread_corner(A, rt, q, t9, acct);
    } else {                                   // i = k: T is symmetric
      q[0] = fma(third, r[0], e0);
      q[1] = fma(third, r[1], e1);
      q[2] = fma(third, r[2], e2);
      spread_corner(A, r, q, t9, acc);
    }
  }
}

// The same for int K grad N_a . grad N_b with K = diag(kd) per element.
template <typename Take>
__device__ __forceinline__ void darcy_rows(const double *__restrict__ perm, const NodeAxis &ax,
                                           const NodeAxis &ay, const NodeAxis &az, int gi, int gj,
                                           int gk, int nx, int ny, Take take, double (&acc)[27]) {
  const double third = 1.0 / 3.0;
#pragma unroll
  for (int A = 0; A < 8; ++A) {
    const int a0 = A & 1, a1 = (A >> 1) & 1, a2 = A >> 2;
    if (!(ax.in[a0] && ay.in[a1] && az.in[a2])) continue;
    const int ex = gi - a0, ey = gj - a1, ez = gk - a2;
    if (!take(ex, ey, ez)) continue;
    const double *kd = perm + 3 * (size_t)(ex + nx * (ey + ny * ez));
    const double fx = 0.0625 * ax.h[a0], fy = 0.0625 * ay.h[a1];
    const double T0 = __ldg(kd) * (fy * az.h[a2] * ax.r[a0]),
                 T1 = __ldg(kd + 1) * (fx * az.h[a2] * ay.r[a1]),
                 T2 = __ldg(kd + 2) * (fx * ay.h[a1] * az.r[a2]);
    const double tr = (T0 + T1) + T2;
    const int s0 = a0 ? 1 : -1, s1 = a1 ? 1 : -1, s2 = a2 ? 1 : -1;
    const double r[3] = {s0 * T0, s1 * T1, s2 * T2};
    const double q[3] = {s0 * third * (tr - T0), s1 * third * (tr - T1), s2 * third * (tr - T2)};
    spread_corner(A, r, q, tr * (1.0 / 9.0), acc);
  }
}

// Component pair p of 0..5: (0,1), (0,2), (1,2), then the diagonal (0,0),
// (1,1), (2,2); the offsets of C_ijkl, j, l = 0..2, in the 6x6 Voigt matrix.
__device__ __forceinline__ void component_pair(int p, int &ci, int &ck, int (&off)[9]) {
  ci = p < 3 ? (p == 2 ? 1 : 0) : p - 3;
  ck = p < 3 ? (p == 0 ? 1 : 2) : p - 3;
#pragma unroll
  for (int j = 0; j < 3; ++j)
#pragma unroll
    for (int l = 0; l < 3; ++l) off[3 * j + l] = 6 * voigt(ci, j) + voigt(ck, l);
}

}  // namespace geneo
