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
// shears, so the first product skips the zeros.
__device__ inline void rotate_voigt(const double *__restrict__ C, double theta, double phi,
                                    double *__restrict__ Cr) {
  const double ct = cos(theta), st = sin(theta), cp = cos(phi), sp = sin(phi);
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
      if (k != l) v = fma(Q[i][l], Q[j][k], v);
      M[I][J] = v;
    }
#pragma unroll
  for (int I = 0; I < 6; ++I) {
    double t[6];                                // row I of M C
#pragma unroll
    for (int J = 0; J < 3; ++J)
      t[J] = fma(M[I][2], C[12 + J], fma(M[I][1], C[6 + J], M[I][0] * C[J]));
#pragma unroll
    for (int J = 3; J < 6; ++J) t[J] = M[I][J] * C[7 * J];
#pragma unroll
    for (int J = 0; J < 6; ++J) {
      double v = t[0] * M[J][0];
#pragma unroll
      for (int K = 1; K < 6; ++K) v = fma(t[K], M[J][K], v);
      Cr[6 * I + J] = v;
    }
  }
}

// ---- rows of the Q1 stiffness, node by node ----------------------------------
// The 3x3 (or 1x1) block of local nodes a, b of an axis-aligned box element is
//   K_ab[i][k] = sum_{j,l} C_ijkl G_ab[j][l],  G_ab[j][l] = int d_j N_a d_l N_b,
// with trilinear N and integrals that are products of 1D integrals of linear
// factors (equal to the 2x2x2 Gauss rule, which is exact for them): h/3 or h/6
// (same or other side), +-1/2 for one derivative, +-1/h for two.  Signs and
// halves are exact, so all 64 tables G_ab of an element are its nine numbers
//   g_jj = (1/h_j) m_e m_f,  m_d = h_d / 3,  and m_e / 4 for j != l,
// (multiplied in the order of the axes) times a sign and a power of two fixed by
// the corners at compile time; nine multiply-adds then give an entry of K_ab.
// FP64 issue (two per clock and SM) is what bounds the assembly on this GPU: the
// loop over blocks with run-time Voigt and sign tables that stood here took
// 21.5 ms on the 128x64x48 laminate, these rows take 5.0 ms.  The sums keep that
// loop's order (the matrices agree to 4e-17): a grouping of the 81 products that
// needs 40 % fewer operations (3.2 ms) moved entries by 2e-16, which the
// condition number carries to 1e-9 of a solution.

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

// The scaled integrals of an element: [3 j + k] = g_jj 2^-k, [9 + 2 e + k] = m_e 2^-(2+k).
constexpr int kCornerG = 15;
__device__ __forceinline__ void corner_integrals(double hx, double hy, double hz, double rx,
                                                 double ry, double rz, double *g) {
  const double m0 = (1.0 / 3.0) * hx, m1 = (1.0 / 3.0) * hy, m2 = (1.0 / 3.0) * hz;
  const double d[3] = {(rx * m1) * m2, (m0 * ry) * m2, (m0 * m1) * rz};
  const double m[3] = {m0, m1, m2};
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    g[3 * j] = d[j];
    g[3 * j + 1] = 0.5 * d[j];
    g[3 * j + 2] = 0.25 * d[j];
    g[9 + 2 * j] = 0.25 * m[j];
    g[10 + 2 * j] = 0.125 * m[j];
  }
}

// sign (+-1) and index of G_ab[j][l] in corner_integrals' table.
__device__ __forceinline__ constexpr int corner_bit(int a, int d) { return a >> d & 1; }
__device__ __forceinline__ constexpr int corner_sign(int a, int b, int j, int l) {
  return corner_bit(a, j) == corner_bit(b, l) ? 1 : -1;
}
__device__ __forceinline__ constexpr int corner_index(int a, int b, int j, int l) {
  if (j == l) {
    const int e = (j + 1) % 3, f = (j + 2) % 3;
    return 3 * j + (corner_bit(a, e) != corner_bit(b, e)) + (corner_bit(a, f) != corner_bit(b, f));
  }
  const int e = 3 - j - l;
  return 9 + 2 * e + (corner_bit(a, e) != corner_bit(b, e));
}
// Slot of local node b of the element in which the node is corner a.
__device__ __forceinline__ constexpr int corner_slot(int a, int b) {
  return 13 + corner_bit(b, 0) - corner_bit(a, 0) + 3 * (corner_bit(b, 1) - corner_bit(a, 1)) +
         9 * (corner_bit(b, 2) - corner_bit(a, 2));
}

// Component (ci, ck) of a node's 27 slots, summed over its (up to eight)
// elements for which take(e) holds, in ascending element order.  `off` indexes
// C_ijkl, j, l = 0..2, in the element's 6x6 Voigt stiffness; `g` holds the
// corner_integrals of the node's eight elements, [corner][kCornerG].
template <typename Take>
__device__ __forceinline__ void elastic_rows(const double *__restrict__ Cel, const int (&off)[9],
                                             const double *g, const NodeAxis &ax,
                                             const NodeAxis &ay, const NodeAxis &az, int gi, int gj,
                                             int gk, int nx, int ny, Take take, double (&acc)[27]) {
#pragma unroll
  for (int A = 7; A >= 0; --A) {
    const int a0 = A & 1, a1 = (A >> 1) & 1, a2 = A >> 2;
    if (!(ax.in[a0] && ay.in[a1] && az.in[a2])) continue;
    const int ex = gi - a0, ey = gj - a1, ez = gk - a2;
    if (!take(ex, ey, ez)) continue;
    const double *c = Cel + 36 * (size_t)(ex + nx * (ey + ny * ez));
    double C[9], G[kCornerG];
#pragma unroll
    for (int q = 0; q < 9; ++q) C[q] = __ldg(c + off[q]);
#pragma unroll
    for (int q = 0; q < kCornerG; ++q) G[q] = g[A * kCornerG + q];
#pragma unroll
    for (int b = 0; b < 8; ++b) {
      double v = 0.0;
#pragma unroll
      for (int q = 0; q < 9; ++q) {
        const double cq = corner_sign(A, b, q / 3, q % 3) > 0 ? C[q] : -C[q];
        v = q == 0 ? cq * G[corner_index(A, b, 0, 0)] : fma(cq, G[corner_index(A, b, q / 3, q % 3)], v);
      }
      acc[corner_slot(A, b)] += v;
    }
  }
}

// The same for int K grad N_a . grad N_b with K = diag(kd) per element.
template <typename Take>
__device__ __forceinline__ void darcy_rows(const double *__restrict__ perm, const NodeAxis &ax,
                                           const NodeAxis &ay, const NodeAxis &az, int gi, int gj,
                                           int gk, int nx, int ny, Take take, double (&acc)[27]) {
#pragma unroll
  for (int A = 7; A >= 0; --A) {
    const int a0 = A & 1, a1 = (A >> 1) & 1, a2 = A >> 2;
    if (!(ax.in[a0] && ay.in[a1] && az.in[a2])) continue;
    const int ex = gi - a0, ey = gj - a1, ez = gk - a2;
    if (!take(ex, ey, ez)) continue;
    const double *kd = perm + 3 * (size_t)(ex + nx * (ey + ny * ez));
    const double k0 = __ldg(kd), k1 = __ldg(kd + 1), k2 = __ldg(kd + 2);
    double G[kCornerG];
    corner_integrals(ax.h[a0], ay.h[a1], az.h[a2], ax.r[a0], ay.r[a1], az.r[a2], G);
#pragma unroll
    for (int b = 0; b < 8; ++b) {
      const double g0 = corner_sign(A, b, 0, 0) * G[corner_index(A, b, 0, 0)],
                   g1 = corner_sign(A, b, 1, 1) * G[corner_index(A, b, 1, 1)],
                   g2 = corner_sign(A, b, 2, 2) * G[corner_index(A, b, 2, 2)];
      acc[corner_slot(A, b)] += fma(k2, g2, fma(k0, g0, k1 * g1));
    }
  }
}

// The corner_integrals of the eight elements of nodes t = 0..n-1 into
// g[t][corner][kCornerG] (shared memory), one (node, corner) per thread and turn.
template <typename Axes>
__device__ __forceinline__ void stage_integrals(double *g, int n, int threads, Axes axes) {
  for (int e = threadIdx.x; e < 8 * n; e += threads) {
    NodeAxis ax, ay, az;
    const int A = e & 7;
    if (!axes(e >> 3, ax, ay, az)) continue;
    corner_integrals(ax.h[A & 1], ay.h[(A >> 1) & 1], az.h[A >> 2], ax.r[A & 1], ay.r[(A >> 1) & 1],
                     az.r[A >> 2], g + e * kCornerG);
  }
}

// The offsets of C_ijkl, j, l = 0..2, of component (ci, ck) = (p / 3, p % 3).
__device__ __forceinline__ void component_offsets(int p, int (&off)[9]) {
#pragma unroll
  for (int j = 0; j < 3; ++j)
#pragma unroll
    for (int l = 0; l < 3; ++l) off[3 * j + l] = 6 * voigt(p / 3, j) + voigt(p % 3, l);
}

}  // namespace geneo
