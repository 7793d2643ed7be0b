// Assembly of A u = b (Sec. 2, eqn:fe_matrix_system) into 3x3-block BSR.
//
// Rather than scattering element matrices with atomics, each (node, neighbour)
// block is gathered from the (1, 2, 4 or 8) elements that contain both nodes:
// every block is written once, in order, with no atomics, so assembly is
// deterministic.  The element integrals are in closed form (fem.cuh).
#include "fem.cuh"
#include "kernels.cuh"

namespace geneo {

__global__ void k_material_base(int n_mat, const geneo_ortho *__restrict__ mats,
                                double *__restrict__ C0) {
  int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= n_mat) return;
  material_stiffness(mats[m], C0 + 36 * m);
}

__global__ void k_element_C(int nel, int n_mat, const double *__restrict__ C0,
                            const int32_t *__restrict__ emat, const double *__restrict__ th,
                            const double *__restrict__ ph, double *__restrict__ Cel,
                            DevStatus *st) {
  int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= nel) return;
  int m = emat[e];
  if (m < 0 || m >= n_mat) {
    atomicCAS(&st->code, 0, GENEO_ERR_INVALID_ARG);
    m = 0;
  }
  rotate_voigt(C0 + 36 * m, th[e], ph ? ph[e] : 0.0, Cel + 36 * (size_t)e);
}

__device__ __forceinline__ void node_ijk(int n, int nnx, int nny, int &i, int &j, int &k) {
  i = n % nnx;
  int r = n / nnx;
  j = r % nny;
  k = r / nny;
}

// Blocks in the rows of the nodes before i on an axis of n nodes (n >= 2): a
// node couples to three positions, an end node to two.  The row pointer of the
// tensor-product pattern is a product of these, so it needs no scan (the
// single-block scan that stood here took 0.53 ms of a 23.3 ms assembly with
// 0.41 M nodes, 1.49 ms with 1.16 M).
__device__ __forceinline__ int axis_rows_before(int i, int n) { return 3 * i - (i > 0) - (i == n); }
__device__ __forceinline__ int axis_row(int i, int n) { return 3 - (i == 0) - (i == n - 1); }
__device__ __forceinline__ int row_start(int i, int j, int k, int nnx, int nny, int nnz) {
  const int tx = 3 * nnx - 2, ty = 3 * nny - 2, cy = axis_row(j, nny), cz = axis_row(k, nnz);
  return tx * (ty * axis_rows_before(k, nnz) + cz * axis_rows_before(j, nny)) +
         cz * cy * axis_rows_before(i, nnx);
}

// Rows of the matrix, assembled with the Dirichlet set eliminated: one block
// per kRowNodes consecutive nodes.  The sums over the elements are formed in
// registers -- elasticity: lane = node, one warp per component (i, k); Darcy:
// thread = node -- and staged in shared memory, from where the rows
// (contiguous in `val`) are written coalesced, with the Dirichlet rows and
// columns replaced by the identity and the lifting
//   lift_i = -sum_{c in D} A_ic g_c on free rows, g_i on Dirichlet rows
// formed on the way (kept so that a new load needs no eliminated columns).
// FP64 issue bounds it: about 6,000 FP64 operations per node for elasticity,
// 500 for Darcy.
template <int NC>
constexpr int kRowNodes = NC == 3 ? 32 : 128;
template <int NC>
constexpr int kRowThreads = NC == 3 ? 288 : 128;
template <int NC>
constexpr int kRowSmem = kRowNodes<NC> * (27 * (NC * NC * 8 + 4 + 1) + (NC == 3 ? 8 * 8 * kCornerG : 0));

template <int NC>
__global__ void __launch_bounds__(kRowThreads<NC>)
    k_assemble_rows(int nx, int ny, int nz, const double *__restrict__ X,
                    const double *__restrict__ Y, const double *__restrict__ Z,
                    const double *__restrict__ coef, const uint8_t *__restrict__ mask,
                    const double *__restrict__ g, double *__restrict__ lift,
                    int32_t *__restrict__ row_ptr, int32_t *__restrict__ col,
                    double *__restrict__ val) {
  constexpr int N = kRowNodes<NC>, NC2 = NC * NC;
  extern __shared__ __align__(16) double sv[];               // [N][27][NC2]
  double *gs = sv + N * 27 * NC2;                            // [N][8][kCornerG] (elasticity)
  int *pos = reinterpret_cast<int *>(gs + (NC == 3 ? N * 8 * kCornerG : 0));   // [N][27] block index in val, or -1
  uint8_t *mk = reinterpret_cast<uint8_t *>(pos + N * 27);   // [N][27] Dirichlet bits of the column node
  const int nnx = nx + 1, nny = ny + 1, nnz = nz + 1, nnode = nnx * nny * nnz;
  const int n0 = blockIdx.x * N, tid = threadIdx.x;
  for (int e = tid; e < N * 27; e += kRowThreads<NC>) {
    const int t = e / 27, s = e - 27 * t, n = n0 + t;
    int p = -1;
    uint8_t m = 0;
    if (n < nnode) {
      int i, j, k;
      node_ijk(n, nnx, nny, i, j, k);
      const int i2 = i + s % 3 - 1, j2 = j + (s / 3) % 3 - 1, k2 = k + s / 9 - 1;
      const int first = row_start(i, j, k, nnx, nny, nnz);
      if (s == 0) row_ptr[n] = first;
      if (s == 0 && n == nnode - 1)
        row_ptr[nnode] = first + axis_row(i, nnx) * axis_row(j, nny) * axis_row(k, nnz);
      if ((unsigned)i2 < (unsigned)nnx && (unsigned)j2 < (unsigned)nny && (unsigned)k2 < (unsigned)nnz) {
        const int dx = s % 3 - (i == 0), dy = (s / 3) % 3 - (j == 0), dz = s / 9 - (k == 0);
        p = first + dx + axis_row(i, nnx) * (dy + axis_row(j, nny) * dz);
        const int cn = i2 + nnx * (j2 + nny * k2);
        col[p] = cn;
        for (int c = 0; c < NC; ++c) m |= (uint8_t)((mask[NC * cn + c] != 0) << c);
      }
    }
    pos[e] = p;
    mk[e] = m;
  }
  if constexpr (NC == 3) {
    stage_integrals(gs, N, kRowThreads<NC>, [&](int t, NodeAxis &ax, NodeAxis &ay, NodeAxis &az) {
      if (n0 + t >= nnode) return false;
      int i, j, k;
      node_ijk(n0 + t, nnx, nny, i, j, k);
      ax = node_axis(X, i, 0, nx);
      ay = node_axis(Y, j, 0, ny);
      az = node_axis(Z, k, 0, nz);
      return true;
    });
    __syncthreads();
  }
  const int t = NC == 3 ? (tid & 31) : tid, n = n0 + t;
  if (n < nnode) {
    int i, j, k;
    node_ijk(n, nnx, nny, i, j, k);
    const NodeAxis ax = node_axis(X, i, 0, nx), ay = node_axis(Y, j, 0, ny), az = node_axis(Z, k, 0, nz);
    auto all = [](int, int, int) { return true; };
    double acc[27];
#pragma unroll
    for (int s = 0; s < 27; ++s) acc[s] = 0.0;
    double *out = sv + t * 27 * NC2;
    if constexpr (NC == 3) {
      const int p = tid >> 5;
      int off[9];
      component_offsets(p, off);
      elastic_rows(coef, off, gs + t * 8 * kCornerG, ax, ay, az, i, j, k, nx, ny, all, acc);
#pragma unroll
      for (int s = 0; s < 27; ++s) out[9 * s + p] = acc[s];
    } else {
      darcy_rows(coef, ax, ay, az, i, j, k, nx, ny, all, acc);
#pragma unroll
      for (int s = 0; s < 27; ++s) out[s] = acc[s];
    }
  }
  __syncthreads();
  if (lift)
    for (int e = tid; e < N * NC; e += kRowThreads<NC>) {
      const int t2 = e / NC, r = e - NC * t2, m = n0 + t2;
      if (m >= nnode) break;
      if (mk[27 * t2 + 13] >> r & 1) {
        lift[NC * m + r] = g[NC * m + r];
        continue;
      }
      double sum = 0.0;
      for (int s = 0; s < 27; ++s) {
        const int b = mk[27 * t2 + s];
        if (!b) continue;
        const int cn = m + s % 3 - 1 + nnx * ((s / 3) % 3 - 1 + nny * (s / 9 - 1));
        for (int c = 0; c < NC; ++c)
          if (b >> c & 1) sum += sv[(27 * t2 + s) * NC2 + NC * r + c] * g[NC * cn + c];
      }
      lift[NC * m + r] = -sum;
    }
  for (int e = tid; e < N * 27 * NC2; e += kRowThreads<NC>) {
    const int b = e / NC2, q = e - NC2 * b, p = pos[b];
    if (p < 0) continue;
    const int t2 = b / 27, r = q / NC, c = q - NC * r;
    const bool drop = (mk[27 * t2 + 13] >> r & 1) || (mk[b] >> c & 1);
    val[(size_t)NC2 * p + q] = drop ? ((b - 27 * t2 == 13 && r == c) ? 1.0 : 0.0) : sv[e];
  }
}

// Consistent nodal load of the traction (0, 0, -q) on the face z = z_max
// (int over a bilinear face of N_a = area / 4) plus an optional nodal load.
__global__ void k_load(int nx, int ny, int nz, const double *__restrict__ X,
                       const double *__restrict__ Y, double q,
                       const double *__restrict__ nodal, double *__restrict__ b) {
  int nnx = nx + 1, nny = ny + 1;
  int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= nnx * nny * (nz + 1)) return;
  int i, j, k;
  node_ijk(n, nnx, nny, i, j, k);
  double f[3] = {0.0, 0.0, 0.0};
  if (k == nz && q != 0.0) {
    for (int ey = max(j - 1, 0); ey <= min(j, ny - 1); ++ey)
      for (int ex = max(i - 1, 0); ex <= min(i, nx - 1); ++ex)
        f[2] -= q * (X[ex + 1] - X[ex]) * (Y[ey + 1] - Y[ey]) * 0.25;
  }
  for (int c = 0; c < 3; ++c) b[3 * n + c] = f[c] + (nodal ? nodal[3 * n + c] : 0.0);
}

__global__ void k_dirichlet_mark(int nd, const int32_t *__restrict__ dofs,
                                 const double *__restrict__ vals, int ndof,
                                 uint8_t *__restrict__ mask, double *__restrict__ g,
                                 DevStatus *st) {
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nd) return;
  int d = dofs[t];
  if (d < 0 || d >= ndof) {
    atomicCAS(&st->code, 0, GENEO_ERR_INVALID_ARG);
    return;
  }
  mask[d] = 1;
  g[d] = vals ? vals[t] : 0.0;
}

// b_i = f_i + lift_i on free rows, b_i = g_i on Dirichlet rows.
__global__ void k_apply_lift(int n3, const uint8_t *__restrict__ mask,
                             const double *__restrict__ lift, double *__restrict__ b) {
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n3) return;
  b[t] = mask[t] ? lift[t] : b[t] + lift[t];
}

// b_n = int f N_n dx = sum over the elements of node n of f V_e / 8, plus nodal.
__global__ void k_load_darcy(int nx, int ny, int nz, const double *__restrict__ X,
                             const double *__restrict__ Y, const double *__restrict__ Z,
                             double f, const double *__restrict__ nodal, double *__restrict__ b) {
  int nnx = nx + 1, nny = ny + 1;
  int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= nnx * nny * (nz + 1)) return;
  int i, j, k;
  node_ijk(n, nnx, nny, i, j, k);
  double v = 0.0;
  if (f != 0.0)
    for (int ex = max(i - 1, 0), e = min(i, nx - 1), q = 0; q < 1; ++q) {
      // f dx, f dx dy, f dx dy dz of the (up to) eight elements, summed in element order
      const double fx[2] = {f * (X[ex + 1] - X[ex]), f * (X[e + 1] - X[e])};
      for (int ez = max(k - 1, 0); ez <= min(k, nz - 1); ++ez) {
        const double dz = Z[ez + 1] - Z[ez];
        for (int ey = max(j - 1, 0); ey <= min(j, ny - 1); ++ey) {
          const double dy = Y[ey + 1] - Y[ey];
          v = fma(fx[0] * dy * dz, 0.125, v);
          if (e > ex) v = fma(fx[1] * dy * dz, 0.125, v);
        }
      }
    }
  b[n] = v + (nodal ? nodal[n] : 0.0);
}

// ---------------------------------------------------------------------------
// Dirichlet mask and values, then the matrix rows with the set eliminated, the
// pattern and the lifting; b = load (launched by the caller) plus the lifting.
template <int NC>
static int launch_rows(const AssemblyArgs &a, const double *coef, cudaStream_t s) {
  const int T = 256, nnode = (a.nx + 1) * (a.ny + 1) * (a.nz + 1);
  GENEO_CUDA_TRY(cudaMemsetAsync(a.mask, 0, NC * (size_t)nnode, s));
  GENEO_CUDA_TRY(cudaMemsetAsync(a.g, 0, NC * (size_t)nnode * sizeof(double), s));
  if (a.n_dir > 0) {
    k_dirichlet_mark<<<(a.n_dir + T - 1) / T, T, 0, s>>>(a.n_dir, a.dir_dofs, a.dir_vals,
                                                         NC * nnode, a.mask, a.g, a.status); GENEO_COUNT_LAUNCH();
  }
  if (int st = ensure_smem(k_assemble_rows<NC>, kRowSmem<NC>)) return st;
  k_assemble_rows<NC><<<(nnode + kRowNodes<NC> - 1) / kRowNodes<NC>, kRowThreads<NC>, kRowSmem<NC>, s>>>(
      a.nx, a.ny, a.nz, a.X, a.Y, a.Z, coef, a.mask, a.g, a.n_dir > 0 ? a.lift : nullptr,
      a.row_ptr, a.col, a.val); GENEO_COUNT_LAUNCH();
  return launch_load(a, s);
}

int launch_assembly(const AssemblyArgs &a, cudaStream_t s) {
  const int nel = a.nx * a.ny * a.nz, T = 128;
  k_material_base<<<(a.n_mat + 63) / 64, 64, 0, s>>>(a.n_mat, a.mats, a.C0); GENEO_COUNT_LAUNCH();
  k_element_C<<<(nel + T - 1) / T, T, 0, s>>>(nel, a.n_mat, a.C0, a.emat, a.theta, a.phi,
                                              a.Cel, a.status); GENEO_COUNT_LAUNCH();
  return launch_rows<3>(a, a.Cel, s);
}

int launch_assembly_darcy(const AssemblyArgs &a, cudaStream_t s) {
  return launch_rows<1>(a, a.perm, s);
}

// Stress recovery at the element centres: sigma_e = C_e B(0) u_e (Voigt order
// 11, 22, 33, 23, 13, 12; engineering shear strains).  At the centre of a box
// element dN_a/dx_d = s_d / (4 h_d) with the corner sign s_d = +-1.
__global__ void k_element_stress(int nx, int ny, int nz, const double *__restrict__ X,
                                 const double *__restrict__ Y, const double *__restrict__ Z,
                                 const double *__restrict__ Cel, const double *__restrict__ u,
                                 double *__restrict__ sig) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= nx * ny * nz) return;
  const int ex = e % nx, ey = (e / nx) % ny, ez = e / (nx * ny);
  const int nnx = nx + 1, nny = ny + 1;
  const double ih[3] = {0.25 / (X[ex + 1] - X[ex]), 0.25 / (Y[ey + 1] - Y[ey]),
                        0.25 / (Z[ez + 1] - Z[ez])};
  double du[3][3] = {{0.0, 0.0, 0.0}, {0.0, 0.0, 0.0}, {0.0, 0.0, 0.0}};   // du_i / dx_d
  for (int a = 0; a < 8; ++a) {
    const int ia = a & 1, ja = (a >> 1) & 1, ka = (a >> 2) & 1;
    const long long n = (ex + ia) + (long long)nnx * ((ey + ja) + (long long)nny * (ez + ka));
    const double g[3] = {(2 * ia - 1) * ih[0], (2 * ja - 1) * ih[1], (2 * ka - 1) * ih[2]};
    for (int i = 0; i < 3; ++i) {
      const double ui = u[3 * n + i];
      for (int d = 0; d < 3; ++d) du[i][d] += g[d] * ui;
    }
  }
  const double eps[6] = {du[0][0], du[1][1], du[2][2], du[1][2] + du[2][1], du[0][2] + du[2][0],
                         du[0][1] + du[1][0]};
  const double *C = Cel + 36 * (size_t)e;
  for (int r = 0; r < 6; ++r) {
    double s = 0.0;
    for (int c = 0; c < 6; ++c) s += C[6 * r + c] * eps[c];
    sig[6 * (size_t)e + r] = s;
  }
}

int launch_element_stress(int nx, int ny, int nz, const double *X, const double *Y,
                          const double *Z, const double *Cel, const double *u, double *sig,
                          cudaStream_t s) {
  const int nel = nx * ny * nz, T = 256;
  k_element_stress<<<(nel + T - 1) / T, T, 0, s>>>(nx, ny, nz, X, Y, Z, Cel, u, sig); GENEO_COUNT_LAUNCH();
  GENEO_CUDA_TRY(cudaGetLastError());
  return GENEO_OK;
}

int launch_load(const AssemblyArgs &a, cudaStream_t s) {
  const int T = 256;
  int nnode = (a.nx + 1) * (a.ny + 1) * (a.nz + 1);
  const int nc = a.nc == 1 ? 1 : 3;
  if (nc == 1) {
    k_load_darcy<<<(nnode + T - 1) / T, T, 0, s>>>(a.nx, a.ny, a.nz, a.X, a.Y, a.Z, a.top_pressure,
                                                   a.nodal, a.b); GENEO_COUNT_LAUNCH();
  } else {
    k_load<<<(nnode + T - 1) / T, T, 0, s>>>(a.nx, a.ny, a.nz, a.X, a.Y, a.top_pressure,
                                             a.nodal, a.b); GENEO_COUNT_LAUNCH();
  }
  if (a.n_dir > 0) {
    k_apply_lift<<<(nc * nnode + T - 1) / T, T, 0, s>>>(nc * nnode, a.mask, a.lift, a.b); GENEO_COUNT_LAUNCH();
  }
  GENEO_CUDA_TRY(cudaGetLastError());
  return GENEO_OK;
}

}  // namespace geneo
