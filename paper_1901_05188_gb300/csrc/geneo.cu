// GenEO coarse space on the device (Sec. 3.2, Sec. 3.3.1-3.3.3).
//
// Per subdomain j the generalised eigenproblem (eqm:matrixForm)
//   A_{Omega_j} p = lambda X_j A_{Omega_j^o} X_j p
// is solved with the shift-and-invert transformation the paper uses
// (Sec. 3.3.2): S = A - sigma B = L L^T for a small sigma < 0, and the
// symmetric operator C = L^-1 B L^-T has eigenvalues mu = 1 / (lambda - sigma),
// so the wanted smallest lambda are the largest mu.  Instead of ARPACK's
// implicitly restarted Lanczos, a block Lanczos process (block size 8, full
// re-orthogonalisation, Cholesky-QR) runs batched over all subdomains and the
// projected matrix is diagonalised by tridiagonalisation, bisection and inverse
// iteration; p = L^-T y.
#include "geneo.cuh"
#include "fem.cuh"

namespace geneo {

namespace {

__device__ __forceinline__ double *tile_at(double *pool, const BandLayout &L, int I, int d) {
  return pool + L.off + ((long long)I * (L.w + 1) + d) * L.slot;
}

__device__ __forceinline__ int cand_count(const int *c) {
  int n = 0;
  while (n < kMaxCand && c[n] >= 0) ++n;
  return n;
}

// Partition-of-unity weight X_j at node (gi, gj, gk) of subdomain j's
// interior: 1 / multiplicity (Sec. 3.3.1), or Sarkis's d_j / sum_k d_k with
// d the distance to each interior subdomain's artificial boundary in element
// layers (Sec. 3.2).  The caller zeroes it on global Dirichlet dofs.
__device__ double pou_weight(const SubDesc *subs, int j, int gi, int gj, int gk, const int *cand,
                             int co0, int co1, int co2, int px, int py, int nx, int ny, int nz,
                             int kind) {
  const int *ci = cand + (co0 + gi) * kMaxCand;
  const int *cj = cand + (co1 + gj) * kMaxCand;
  const int *ck = cand + (co2 + gk) * kMaxCand;
  const int nci = cand_count(ci), ncj = cand_count(cj), nck = cand_count(ck);
  if (kind == 0) return 1.0 / double(nci * ncj * nck);
  int sum = 0;
  for (int c = 0; c < nck; ++c)
    for (int b = 0; b < ncj; ++b)
      for (int a = 0; a < nci; ++a)
        sum += artificial_distance(subs[ci[a] + px * (cj[b] + py * ck[c])], gi, gj, gk, nx, ny, nz);
  return double(artificial_distance(subs[j], gi, gj, gk, nx, ny, nz)) / double(sum);
}

__global__ void k_pou_neumann(const SubDesc *subs, const int *cand, int co0, int co1, int co2,
                              const uint8_t *mask, int nnx, int nny, int nnz, int px, int py,
                              int kind, double *Xneu) {
  const int j = blockIdx.y;
  const SubDesc &S = subs[j];
  const int nc = S.nc;
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nc * S.nbox.count()) return;
  int l = t / nc, comp = t - nc * l;
  int gi, gj, gk;
  S.nbox.global(l, gi, gj, gk);
  double x = 0.0;
  if (S.ibox.local(gi, gj, gk) >= 0) {
    x = pou_weight(subs, j, gi, gj, gk, cand, co0, co1, co2, px, py, nnx - 1, nny - 1, nnz - 1,
                   kind);
    if (mask[nc * (gi + nnx * (gj + nny * gk)) + comp]) x = 0.0;
  }
  Xneu[S.x_neu + t] = x;
}

// The same weights on the interior dofs, laid out like the local solutions
// (offset v_int): the one-level weight D_j = X_j of the gather.
__global__ void k_pou_interior(const SubDesc *subs, const int *cand, int co0, int co1, int co2,
                               const uint8_t *mask, int nnx, int nny, int nnz, int px, int py,
                               int kind, double *wloc) {
  const int j = blockIdx.y;
  const SubDesc &S = subs[j];
  const int nc = S.nc;
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nc * S.ibox.count()) return;
  int l = t / nc, comp = t - nc * l;
  int gi, gj, gk;
  S.ibox.global(l, gi, gj, gk);
  double x = pou_weight(subs, j, gi, gj, gk, cand, co0, co1, co2, px, py, nnx - 1, nny - 1,
                        nnz - 1, kind);
  if (mask[nc * (gi + nnx * (gj + nny * gk)) + comp]) x = 0.0;
  wloc[S.v_int + t] = x;
}

// S_j = A_Omega_j - sigma B_j in band tiles (lower part) and B_j as 27-slot
// rows, from the rows of the node's elements inside Omega_j (fem.cuh): one
// block per kNeuNodes consecutive local nodes, summed in registers (elasticity:
// lane = node, one warp per component) and staged in shared memory, from
// where B's rows are written coalesced and S's entries column by column.  The
// overlap elements' rows are summed only in blocks that have some.  FP64 issue
// bounds it, as for the global matrix.
template <int NC>
constexpr int kNeuNodes = NC == 3 ? 32 : 128;
template <int NC>
constexpr int kNeuThreads = NC == 3 ? 288 : 128;
template <int NC>
constexpr int kNeuSmem = kNeuNodes<NC> * (27 * (NC * NC * 8 + 4 + 1) + (NC == 3 ? 8 * 8 * kCornerG : 0));

template <int NC>
__global__ void __launch_bounds__(kNeuThreads<NC>)
    k_neumann_assemble(const SubDesc *subs, const BandLayout *lay, int nx, int ny, int nz,
                       const double *__restrict__ X, const double *__restrict__ Y,
                       const double *__restrict__ Z, const double *__restrict__ coef,
                       const int *__restrict__ ecnt, int eo0, int eo1, int eo2,
                       const uint8_t *__restrict__ mask, const double *__restrict__ Xneu,
                       double sigma, double *poolS, double *Bloc) {
  constexpr int N = kNeuNodes<NC>, NC2 = NC * NC, kT = kNeuThreads<NC>;
  const SubDesc &S = subs[blockIdx.y];
  const int nn = S.nbox.count(), l0 = blockIdx.x * N, tid = threadIdx.x;
  if (l0 >= nn) return;
  extern __shared__ __align__(16) double sv[];               // [N][27][NC2]
  double *gs = sv + N * 27 * NC2;                            // [N][8][kCornerG] (elasticity)
  int *nb = reinterpret_cast<int *>(gs + (NC == 3 ? N * 8 * kCornerG : 0));   // [N][27] local neighbour node, or -1
  uint8_t *mk = reinterpret_cast<uint8_t *>(nb + N * 27);    // [N][27] its Dirichlet bits
  const int nnx = nx + 1, nny = ny + 1;
  for (int e = tid; e < N * 27; e += kT) {
    const int t = e / 27, s = e - 27 * t, l = l0 + t;
    int l2 = -1;
    uint8_t m = 0;
    if (l < nn) {
      int i, j, k;
      S.nbox.global(l, i, j, k);
      i += s % 3 - 1, j += (s / 3) % 3 - 1, k += s / 9 - 1;
      l2 = S.nbox.local(i, j, k);
      if (l2 >= 0)
        for (int c = 0; c < NC; ++c)
          m |= (uint8_t)((mask[(size_t)NC * (i + nnx * (j + nny * k)) + c] != 0) << c);
    }
    nb[e] = l2;
    mk[e] = m;
  }
  const int t = NC == 3 ? (tid & 31) : tid, l = l0 + t;
  const bool live = l < nn;
  int gi = 0, gj = 0, gk = 0;
  if (live) S.nbox.global(l, gi, gj, gk);
  NodeAxis ax, ay, az;
  bool touch = false;                      // the node has an overlap element
  auto ov = [&](int ex, int ey, int ez) { return ecnt[eo0 + ex] * ecnt[eo1 + ey] * ecnt[eo2 + ez] >= 2; };
  if (live) {
    ax = node_axis(X, gi, S.elo[0], S.ehi[0]);
    ay = node_axis(Y, gj, S.elo[1], S.ehi[1]);
    az = node_axis(Z, gk, S.elo[2], S.ehi[2]);
#pragma unroll
    for (int A = 0; A < 8; ++A)
      if (ax.in[A & 1] && ay.in[(A >> 1) & 1] && az.in[A >> 2])
        touch = touch || ov(gi - (A & 1), gj - ((A >> 1) & 1), gk - (A >> 2));
  }
  int off[9];
  if constexpr (NC == 3) {
    component_offsets(tid >> 5, off);
    stage_integrals(gs, N, kT, [&](int t, NodeAxis &bx, NodeAxis &by, NodeAxis &bz) {
      if (l0 + t >= nn) return false;
      int i, j, k;
      S.nbox.global(l0 + t, i, j, k);
      bx = node_axis(X, i, S.elo[0], S.ehi[0]);
      by = node_axis(Y, j, S.elo[1], S.ehi[1]);
      bz = node_axis(Z, k, S.elo[2], S.ehi[2]);
      return true;
    });
  }
  // this thread's rows over the elements `take` picks: to the stage, or
  // S = A - sigma B with the stage holding B
  auto rows = [&](auto take, bool shift) {
    double acc[27];
#pragma unroll
    for (int s = 0; s < 27; ++s) acc[s] = 0.0;
    double *out = sv + t * 27 * NC2 + (NC == 3 ? tid >> 5 : 0);
    if constexpr (NC == 3)
      elastic_rows(coef, off, gs + t * 8 * kCornerG, ax, ay, az, gi, gj, gk, nx, ny, take, acc);
    else
      darcy_rows(coef, ax, ay, az, gi, gj, gk, nx, ny, take, acc);
#pragma unroll
    for (int s = 0; s < 27; ++s) out[NC2 * s] = shift ? fma(-sigma, out[NC2 * s], acc[s]) : acc[s];
  };
  const bool any = __syncthreads_or(touch);
  if (any) {
    if (live) rows(ov, false);
    __syncthreads();
  }
  double *bl = Bloc + (S.b_neu + (long long)l0 * 27) * NC2;
  for (int e = tid; e < N * 27 * NC2; e += kT) {
    const int b = e / NC2, q = e - NC2 * b, t2 = b / 27, r = q / NC, c = q - NC * r, l2 = nb[b];
    if (l0 + t2 >= nn) break;
    double bv = 0.0;
    if (any && l2 >= 0 && !((mk[27 * t2 + 13] >> r & 1) || (mk[b] >> c & 1)))
      bv = Xneu[S.x_neu + NC * (l0 + t2) + r] * sv[e] * Xneu[S.x_neu + NC * l2 + c];
    bl[e] = bv;
    sv[e] = bv;
  }
  __syncthreads();
  if (live) rows([](int, int, int) { return true; }, true);
  __syncthreads();
  // column C = NC l + c of S: rows R = NC l2 + r >= C (S is symmetric)
  const BandLayout L = lay[blockIdx.y];
  for (int e = tid; e < N * 27 * NC2; e += kT) {
    const int r = e % NC, s = (e / NC) % 27, c = (e / (27 * NC)) % NC, t2 = e / (27 * NC2);
    const int b = 27 * t2 + s, l2 = nb[b];
    const int C = NC * (l0 + t2) + c, R = NC * l2 + r;
    if (l2 < 0 || R < C) continue;
    const bool drop = (mk[27 * t2 + 13] >> c & 1) || (mk[b] >> r & 1);
    const int I = R >> 5, J = C >> 5;
    tile_at(poolS, L, I, I - J)[(C & 31) * 32 + (R & 31)] =
        drop ? (R == C ? 1.0 : 0.0) : sv[b * NC2 + NC * c + r];
  }
}

__global__ void k_bloc_mv(const SubDesc *subs, const double *__restrict__ Bloc,
                          const double *__restrict__ T, double *__restrict__ W,
                          long long stride, int p) {
  const int j = blockIdx.y;
  const SubDesc &S = subs[j];
  const int nc = S.nc;
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nc * S.nbox.count()) return;
  int l = t / nc, r = t - nc * l;
  int gi, gj, gk;
  S.nbox.global(l, gi, gj, gk);
  double acc[kLanczosBlock];
#pragma unroll
  for (int q = 0; q < kLanczosBlock; ++q) acc[q] = 0.0;
  const double *Tj = T + j * stride;
  for (int s = 0; s < 27; ++s) {
    int l2 = S.nbox.local(gi + s % 3 - 1, gj + (s / 3) % 3 - 1, gk + s / 9 - 1);
    if (l2 < 0) continue;
    const double *bl = Bloc + (S.b_neu + (long long)l * 27 + s) * (nc * nc) + nc * r;
    for (int c = 0; c < nc; ++c) {
      double bv = bl[c];
      if (bv == 0.0) continue;
      const double *tr = Tj + (long long)(nc * l2 + c) * p;
#pragma unroll
      for (int q = 0; q < kLanczosBlock; ++q)
        if (q < p) acc[q] += bv * tr[q];
    }
  }
  double *wr = W + j * stride + (long long)t * p;
#pragma unroll
  for (int q = 0; q < kLanczosBlock; ++q)
    if (q < p) wr[q] = acc[q];
}

__device__ __forceinline__ unsigned long long splitmix64(unsigned long long x) {
  x += 0x9E3779B97F4A7C15ull;
  x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
  x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
  return x ^ (x >> 31);
}

__global__ void k_random_block(const SubDesc *subs, int npad, double *V, int ld, long long stride,
                               int p, unsigned long long seed) {
  const int j = blockIdx.y;
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= npad * p) return;
  int row = t / p, c = t - row * p;
  double v = 0.0;
  if (row < subs[j].n_neu) {
    unsigned long long h = splitmix64(seed ^ splitmix64(((unsigned long long)j << 40) ^
                                                        ((unsigned long long)row << 8) ^ c));
    v = double(h >> 11) * (1.0 / 9007199254740992.0) * 2.0 - 1.0;
  }
  V[j * stride + (long long)row * ld + c] = v;
}

// Second re-orthogonalisation pass needed?  After one projection W -= V H,
// column b of W has squared norm G_bb and lost sum_a H_ab^2; the pass is
// repeated where more than half of the column's squared norm was removed,
// G_bb < sum_a H_ab^2 (the criterion of Daniel, Gragg, Kaufman and Stewart with
// eta = 1/sqrt(2): "twice is enough").
__global__ void k_reorth_gate(const double *G, int p, const double *H, int na, long long hs,
                              int *gate) {
  const int j = blockIdx.x;
  __shared__ int need;
  if (threadIdx.x == 0) need = 0;
  __syncthreads();
  if (threadIdx.x < p) {
    const int b = threadIdx.x;
    double lost = 0.0;
    for (int a = 0; a < na; ++a) {
      const double h = H[j * hs + (long long)a * p + b];
      lost += h * h;
    }
    if (!(G[(long long)j * p * p + b * p + b] >= lost)) atomicOr(&need, 1);
  }
  __syncthreads();
  if (threadIdx.x == 0) gate[j] = need;
}

// Cholesky of the p x p Gram matrix, inverse, and Racc update: one warp per
// subdomain, lane = column.  A chain of square roots and divisions bounds it:
// 25 us a launch, with one thread for everything 57 us.
__global__ void k_cholqr_small(const double *G, int p, double *Rinv, double *Racc, int first,
                               double abs_tiny) {
  const int j = blockIdx.x, c = threadIdx.x;
  __shared__ double R[kLanczosBlock][kLanczosBlock];
  __shared__ double Ri[kLanczosBlock][kLanczosBlock];
  const double *g = G + (long long)j * p * p;
  if (c < p)
    for (int a = 0; a < p; ++a) R[a][c] = 0.0;
  __syncwarp();
  // upper factor R with G = R^T R; dead columns get R[k][k] = 0
  for (int k = 0; k < p; ++k) {
    double d = g[k * p + k];
    for (int i = 0; i < k; ++i) d -= R[i][k] * R[i][k];
    // numerically dependent (angle to the block's span below 1e-7) or
    // negligible against the operator scale: deflate the column
    const bool dead = !(d > 1e-14 * g[k * p + k]) || !(d > abs_tiny);
    const double rk = dead ? 0.0 : sqrt(d);
    if (c > k && c < p) {
      double v = g[k * p + c];
      for (int i = 0; i < k; ++i) v -= R[i][k] * R[i][c];
      R[k][c] = dead ? 0.0 : v / rk;
    } else if (c == k) {
      R[k][k] = rk;
    }
    __syncwarp();
  }
  // Rinv (upper); a dead column maps to zero
  if (c < p)
    for (int a = p - 1; a >= 0; --a) {
      if (a > c || R[a][a] == 0.0) {
        Ri[a][c] = 0.0;
        continue;
      }
      double s = (a == c) ? 1.0 : 0.0;
      for (int k = a + 1; k <= c; ++k) s -= R[a][k] * Ri[k][c];
      Ri[a][c] = s / R[a][a];
    }
  double *racc = Racc + (long long)j * p * p;
  if (c < p) {
    double in[kLanczosBlock];
    for (int k = 0; k < p; ++k) in[k] = first ? 0.0 : racc[k * p + c];
    for (int a = 0; a < p; ++a) {
      double s = 0.0;
      if (first) {
        s = R[a][c];
      } else {
        for (int k = 0; k < p; ++k) s += R[a][k] * in[k];
      }
      racc[a * p + c] = s;
      Rinv[(long long)j * p * p + a * p + c] = Ri[a][c];
    }
  }
}

__global__ void k_rowmul(const SubDesc *subs, int npad, double *W, int p, const double *Rinv) {
  const int j = blockIdx.y;
  int row = blockIdx.x * blockDim.x + threadIdx.x;
  if (row >= npad) return;
  double *w = W + ((long long)j * npad + row) * p;
  const double *ri = Rinv + (long long)j * p * p;
  double in[kLanczosBlock];
  for (int q = 0; q < p; ++q) in[q] = w[q];
  for (int b = 0; b < p; ++b) {
    double s = 0.0;
    for (int a = 0; a <= b; ++a) s += in[a] * ri[a * p + b];
    w[b] = row < subs[j].n_neu ? s : 0.0;
  }
}

__global__ void k_hm_accum(double *Hm, int kdim, const double *Hs, int rows, int k, int p) {
  const int j = blockIdx.x;
  for (int e = threadIdx.x; e < rows * p; e += blockDim.x) {
    int r = e / p, b = e - r * p;
    Hm[(long long)j * kdim * kdim + (long long)r * kdim + k * p + b] +=
        Hs[(long long)j * rows * p + e];
  }
}

__global__ void k_hm_subdiag(double *Hm, int kdim, const double *Racc, int k, int p,
                             double *Rblk) {
  const int j = blockIdx.x;
  for (int e = threadIdx.x; e < p * p; e += blockDim.x) {
    int a = e / p, b = e - a * p;
    double v = Racc[(long long)j * p * p + e];
    if ((k + 1) * p < kdim)
      Hm[(long long)j * kdim * kdim + (long long)((k + 1) * p + a) * kdim + k * p + b] = v;
    else
      Rblk[(long long)j * p * p + e] = v;
  }
}

__global__ void k_restart_hm(double *Hm, int kdim, const double *Eval, const double *Evec,
                             const double *Rblk, int kk, int p) {
  const int j = blockIdx.x;
  double *H = Hm + (long long)j * kdim * kdim;
  const double *S = Evec + (long long)j * kdim * kdim;
  const double *R = Rblk + (long long)j * p * p;
  for (int e = threadIdx.x; e < kdim * kdim; e += blockDim.x) {
    int r = e / kdim, c = e - r * kdim;
    double v = 0.0;
    if (r < kk && c < kk) {
      v = (r == c) ? Eval[(long long)j * kdim + r] : 0.0;
    } else if (r >= kk && r < kk + p && c < kk) {
      int a = r - kk;
      for (int b = 0; b < p; ++b) v += R[a * p + b] * S[(long long)(kdim - p + b) * kdim + c];
    }
    H[e] = v;
  }
}

__global__ void k_copy_block(const SubDesc *subs, int npad, const double *W, int ldw,
                             long long sw, double *V, int ldv, long long sv, int p) {
  const int j = blockIdx.y;
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= npad * p) return;
  int row = t / p, b = t - row * p;
  V[j * sv + (long long)row * ldv + b] = W[j * sw + (long long)row * ldw + b];
}

// Ritz pairs of the symmetrised projected matrix H (n x n, n <= kMaxKdim):
// Householder reduction to tridiagonal form (H = Q T Q^T), the nw largest
// eigenvalues of T by Sturm-sequence multisection, their eigenvectors by inverse
// iteration (re-orthogonalised inside clusters of close eigenvalues), and the
// back-transformation y = Q x.  One block per subdomain; eigenvalues are
// returned in descending order, columns nw..n-1 of Evec are zero.
constexpr int kMaxKdim = 128;

// Number of eigenvalues of T smaller than x: sign changes of the leading
// principal minors of T - x, p_i = (d_i - x) p_{i-1} - e_{i-1}^2 p_{i-2}: three
// instructions of the FP64 pipe a step (64 cycles each) where the quotients
// p_i / p_{i-1} take a division and comparisons, about fourteen; signs and
// sizes are read from the bits.  T is scaled to norm <= 1, so |p| grows at most
// threefold a step (n <= 128: below 2^203); pairs below 2^-303 are scaled up.
__device__ __forceinline__ int sturm_count(const double *d, const double *e2, int n, double x) {
  int cnt = 0;
  double p0 = 1.0, p1 = d[0] - x;
  int h0 = __double2hiint(p0), h1 = __double2hiint(p1);
  for (int i = 0;; ++i) {
    if (((h1 & 0x7fffffff) | __double2loint(p1)) == 0) {     // as a small negative quotient
      p1 = p0 * -1e-30;
      h1 = __double2hiint(p1);
    }
    cnt += (unsigned)(h0 ^ h1) >> 31;
    if (i + 1 == n) return cnt;
    if (max(h0 & 0x7fffffff, h1 & 0x7fffffff) < 0x2d000000) {
      const double up = __hiloint2double(0x52b00000, 0);     // 2^300
      p0 *= up;
      p1 *= up;
    }
    const double p2 = fma(d[i + 1] - x, p1, -(e2[i] * p0));
    p0 = p1;
    p1 = p2;
    h0 = __double2hiint(p0);
    h1 = __double2hiint(p1);
  }
}

__global__ void __launch_bounds__(256)
    k_ritz_eig(const double *Hm, int n, int nw, int p, const double *Rblk, double *Eval,
               double *Evec, double *Eres) {
  const int j = blockIdx.x;
  const int ld = n + 1;
  extern __shared__ __align__(16) unsigned char smraw[];
  double *A = reinterpret_cast<double *>(smraw);   // n x ld, Householder vectors below diagonal
  double *d = A + n * ld;                          // diagonal of T
  double *e = d + n;                               // off-diagonal of T
  double *e2 = e + n;                              // squares
  double *lam = e2 + n;                            // wanted eigenvalues (descending)
  double *vs = lam + n;                            // current Householder vector / work
  double *ps = vs + n;                             // A v / q
  __shared__ double red[8];
  __shared__ double bounds[2];
  const double *H = Hm + (long long)j * n * n;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int t = tid; t < n * n; t += blockDim.x) {
    int r = t / n, c = t - r * n;
    A[r * ld + c] = 0.5 * (H[t] + H[c * n + r]);
  }
  __syncthreads();
  // ---- Householder tridiagonalisation (lower)
  for (int k = 0; k + 2 < n; ++k) {
    const int m = n - k - 1;
    double s2 = 0.0;
    for (int i = tid; i < m; i += blockDim.x) {
      double x = A[(k + 1 + i) * ld + k];
      s2 += x * x;
    }
    s2 = warp_sum(s2);
    if (lane == 0) red[warp] = s2;
    __syncthreads();
    if (tid == 0) {
      double t = 0.0;
      for (int w = 0; w < 8; ++w) t += red[w];
      double x0 = A[(k + 1) * ld + k];
      double nrm = sqrt(t);
      double alpha = (x0 >= 0.0) ? -nrm : nrm;
      double vnorm2 = t - x0 * x0 + (x0 - alpha) * (x0 - alpha);
      d[k] = A[k * ld + k];
      if (nrm == 0.0 || vnorm2 <= 0.0) {
        e[k] = 0.0;
        red[0] = 0.0;           // no reflection
      } else {
        e[k] = alpha;
        red[0] = 1.0 / sqrt(vnorm2);
        red[1] = alpha;
      }
    }
    __syncthreads();
    const double inv = red[0];
    if (inv == 0.0) {
      for (int i = tid; i < m; i += blockDim.x) A[(k + 1 + i) * ld + k] = 0.0;
      __syncthreads();
      continue;
    }
    const double alpha = red[1];
    for (int i = tid; i < m; i += blockDim.x) {
      double v = A[(k + 1 + i) * ld + k] - (i == 0 ? alpha : 0.0);
      v *= inv;
      vs[i] = v;
      A[(k + 1 + i) * ld + k] = v;       // keep v for the back-transformation
    }
    __syncthreads();
    // p = A_sub v
    for (int i = tid; i < m; i += blockDim.x) {
      const double *row = A + (k + 1 + i) * ld + (k + 1);
      double s = 0.0;
      for (int c = 0; c < m; ++c) s += row[c] * vs[c];
      ps[i] = s;
    }
    __syncthreads();
    double b = 0.0;
    for (int i = tid; i < m; i += blockDim.x) b += vs[i] * ps[i];
    b = warp_sum(b);
    if (lane == 0) red[warp] = b;
    __syncthreads();
    double beta = 0.0;
    for (int w = 0; w < 8; ++w) beta += red[w];
    __syncthreads();
    for (int i = tid; i < m; i += blockDim.x) ps[i] = 2.0 * ps[i] - 2.0 * beta * vs[i];
    __syncthreads();
    // A_sub -= v q^T + q v^T
    for (int t = tid; t < m * m; t += blockDim.x) {
      int r = t / m, c = t - r * m;
      A[(k + 1 + r) * ld + (k + 1 + c)] -= vs[r] * ps[c] + ps[r] * vs[c];
    }
    __syncthreads();
  }
  if (tid == 0) {
    if (n >= 2) {
      d[n - 2] = A[(n - 2) * ld + (n - 2)];
      e[n - 2] = A[(n - 1) * ld + (n - 2)];
    }
    d[n - 1] = A[(n - 1) * ld + (n - 1)];
    e[n - 1] = 0.0;
    double lo = 1e300, hi = -1e300, mx = 0.0;
    for (int i = 0; i < n; ++i) {
      double r = (i > 0 ? fabs(e[i - 1]) : 0.0) + fabs(e[i]);
      lo = fmin(lo, d[i] - r);
      hi = fmax(hi, d[i] + r);
      mx = fmax(mx, fabs(d[i]) + r);
    }
    bounds[0] = lo - 1e-12 * mx - 1e-300;
    bounds[1] = hi + 1e-12 * mx + 1e-300;
    red[0] = mx;
  }
  __syncthreads();
  const double tnorm = red[0];
  // T times a power of two, norm at most one: vs = diagonal, e2 = squares
  const int tex = tnorm > 0.0 ? ilogb(tnorm) + 1 : 0;
  const double down = ldexp(1.0, -tex);
  for (int i = tid; i < n; i += blockDim.x) {
    vs[i] = d[i] * down;
    e2[i] = (e[i] * down) * (e[i] * down);
  }
  __syncthreads();
  // ---- multisection on four warps, one per SM sub-partition: G lanes cut the
  // interval of an eigenvalue into G + 1, as many lanes as nw leaves (80 columns,
  // 40 wanted: G = 3, 27 evaluations; the kernel takes 2.06 ms, bisection by one
  // thread with the quotients took 2.3 of its 3.65 ms)
  if (warp < 4) {
    const int G = nw <= 16 ? 8 : nw <= 20 ? 6 : nw <= 24 ? 5 : nw <= 32 ? 4 : nw <= 40 ? 3 : nw <= 64 ? 2 : 1;
    const int per = 32 / G, grp = lane / G, sub = lane - grp * G, q = warp * per + grp;
    const int target = n - 1 - q;          // index from the bottom
    double a = bounds[0] * down, bnd = bounds[1] * down;
    const double cut = 1.0 / (G + 1);
    bool open = grp < per && q < nw;
    for (int it = 0; it < 200; ++it) {
      open = open && bnd - a > 2.2e-16 * (fabs(a) + fabs(bnd)) + 1e-300;
      if (!__any_sync(0xffffffffu, open)) break;
      const double h = (bnd - a) * cut;
      const bool above = open && sturm_count(vs, e2, n, fma(h, (double)(sub + 1), a)) > target;
      const unsigned m = (__ballot_sync(0xffffffffu, above) >> (grp * G)) & ((1u << G) - 1u);
      if (!open) continue;
      const int f = m ? __ffs(m) : G + 1;  // the first point above
      const double lo = f > 1 ? fma(h, (double)(f - 1), a) : a;
      if (f <= G) bnd = fma(h, (double)f, a);
      a = lo;
    }
    if (grp < per && q < nw && sub == 0) lam[q] = ldexp(0.5 * (a + bnd), tex);
  }
  __syncthreads();
  // ---- inverse iteration on T - lam I (partial pivoting), vectors to Evec columns
  double *Ev = Evec + (long long)j * n * n;
  for (int q = tid; q < nw; q += blockDim.x) {
    double u0[kMaxKdim], u1[kMaxKdim], u2[kMaxKdim], lm[kMaxKdim], x[kMaxKdim];
    unsigned char piv[kMaxKdim];
    const double lq = lam[q];
    const double tiny = 1e-15 * fmax(tnorm, 1e-300);
    for (int i = 0; i < n; ++i) {
      u0[i] = d[i] - lq;
      u1[i] = (i + 1 < n) ? e[i] : 0.0;
      u2[i] = 0.0;
    }
    for (int i = 0; i + 1 < n; ++i) {
      double sub = e[i];
      if (fabs(u0[i]) >= fabs(sub)) {
        piv[i] = 0;
        if (fabs(u0[i]) < tiny) u0[i] = (u0[i] >= 0 ? tiny : -tiny);
        lm[i] = sub / u0[i];
        u0[i + 1] -= lm[i] * u1[i];
      } else {
        piv[i] = 1;
        lm[i] = u0[i] / sub;
        double t0 = u0[i + 1], t1 = (i + 2 < n) ? u1[i + 1] : 0.0;
        u0[i] = sub;
        double n11 = u1[i] - lm[i] * t0;
        double n12 = -lm[i] * t1;
        u1[i] = t0;
        u2[i] = t1;
        u0[i + 1] = n11;
        if (i + 2 < n) u1[i + 1] = n12;
      }
    }
    if (fabs(u0[n - 1]) < tiny) u0[n - 1] = (u0[n - 1] >= 0 ? tiny : -tiny);
    // deterministic start vector
    unsigned long long h = 0x9E3779B97F4A7C15ull * (unsigned long long)(q + 1) ^ (unsigned long long)j;
    for (int i = 0; i < n; ++i) {
      h = splitmix64(h + i);
      x[i] = double(h >> 11) * (1.0 / 9007199254740992.0) - 0.5;
    }
    for (int it = 0; it < 3; ++it) {
      for (int i = 0; i + 1 < n; ++i) {
        if (piv[i]) {
          double t = x[i];
          x[i] = x[i + 1];
          x[i + 1] = t;
        }
        x[i + 1] -= lm[i] * x[i];
      }
      x[n - 1] /= u0[n - 1];
      if (n >= 2) x[n - 2] = (x[n - 2] - u1[n - 2] * x[n - 1]) / u0[n - 2];
      for (int i = n - 3; i >= 0; --i) x[i] = (x[i] - u1[i] * x[i + 1] - u2[i] * x[i + 2]) / u0[i];
      double s = 0.0;
      for (int i = 0; i < n; ++i) s += x[i] * x[i];
      s = 1.0 / sqrt(s);
      for (int i = 0; i < n; ++i) x[i] *= s;
    }
    for (int i = 0; i < n; ++i) Ev[(long long)i * n + q] = x[i];
  }
  for (int t = tid; t < n * n; t += blockDim.x) {
    int c = t - (t / n) * n;
    if (c >= nw) Ev[t] = 0.0;
  }
  __syncthreads();
  // ---- re-orthogonalise inside clusters of close eigenvalues (warp 0, in order)
  if (warp == 0) {
    const double ctol = 1e-7 * fmax(fabs(lam[0]), 1e-300);
    int c0 = 0;
    for (int q = 1; q < nw; ++q) {
      if (fabs(lam[q] - lam[q - 1]) > ctol) {
        c0 = q;
        continue;
      }
      for (int pass = 0; pass < 2; ++pass) {
        for (int r = c0; r < q; ++r) {
          double s = 0.0;
          for (int i = lane; i < n; i += 32) s += Ev[(long long)i * n + r] * Ev[(long long)i * n + q];
          s = warp_sum(s);
          for (int i = lane; i < n; i += 32) Ev[(long long)i * n + q] -= s * Ev[(long long)i * n + r];
          __syncwarp();
        }
        double s = 0.0;
        for (int i = lane; i < n; i += 32) s += Ev[(long long)i * n + q] * Ev[(long long)i * n + q];
        s = warp_sum(s);
        s = s > 0.0 ? 1.0 / sqrt(s) : 0.0;
        for (int i = lane; i < n; i += 32) Ev[(long long)i * n + q] *= s;
        __syncwarp();
      }
    }
  }
  __syncthreads();
  // ---- back-transformation y = H_0 H_1 ... H_{n-3} x (thread q owns column q)
  for (int q = tid; q < nw; q += blockDim.x) {
    double x[kMaxKdim];
    for (int i = 0; i < n; ++i) x[i] = Ev[(long long)i * n + q];
    for (int k = n - 3; k >= 0; --k) {
      double s = 0.0;
      for (int i = k + 1; i < n; ++i) s += A[i * ld + k] * x[i];
      s *= 2.0;
      for (int i = k + 1; i < n; ++i) x[i] -= s * A[i * ld + k];
    }
    for (int i = 0; i < n; ++i) Ev[(long long)i * n + q] = x[i];
    Eval[(long long)j * n + q] = lam[q];
    // residual estimate || R_s y[n-p .. n-1] ||
    const double *Rb = Rblk + (long long)j * p * p;
    double r2 = 0.0;
    for (int a = 0; a < p; ++a) {
      double v = 0.0;
      for (int b = 0; b < p; ++b) v += Rb[a * p + b] * x[n - p + b];
      r2 += v * v;
    }
    Eres[(long long)j * n + q] = sqrt(r2);
  }
  for (int q = nw + tid; q < n; q += blockDim.x) {
    Eval[(long long)j * n + q] = 0.0;
    Eres[(long long)j * n + q] = 0.0;
  }
}

__global__ void k_build_Z(const SubDesc *subs, const double *P, int ldp, long long sp,
                          const double *Xneu, double *Zp) {
  const int j = blockIdx.y;
  const SubDesc &S = subs[j];
  if (S.m == 0) return;
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (long long)S.n_int * S.m) return;
  int row = (int)(t / S.m), k = (int)(t - (long long)row * S.m);
  const int nc = S.nc;
  int node = row / nc, comp = row - nc * node;
  int gi, gj, gk;
  S.ibox.global(node, gi, gj, gk);
  int ln = S.nbox.local(gi, gj, gk);
  int nd = nc * ln + comp;
  Zp[S.z_off + t] = Xneu[S.x_neu + nd] * P[j * sp + (long long)nd * ldp + k];
}

__global__ void k_AZ(const SubDesc *subs, int nnx, int nny, int nnz, const int32_t *__restrict__ rp,
                     const int32_t *__restrict__ col, const double *__restrict__ val,
                     const double *__restrict__ Zp, const long long *yoff, double *Yp) {
  const int j = blockIdx.y;
  const SubDesc &S = subs[j];
  const int m = S.m;
  if (m == 0) return;
  const int nc = S.nc;
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nc * S.nbox.count()) return;
  int l = t / nc, r = t - nc * l;
  int gi, gj, gk;
  S.nbox.global(l, gi, gj, gk);
  int g = gi + nnx * (gj + nny * gk);
  double acc[kMaxModes];
#pragma unroll
  for (int q = 0; q < kMaxModes; ++q) acc[q] = 0.0;
  for (int pidx = rp[g]; pidx < rp[g + 1]; ++pidx) {
    int g2 = col[pidx];
    int i2 = g2 % nnx, rr = g2 / nnx, j2 = rr % nny, k2 = rr / nny;
    int l2 = S.ibox.local(i2, j2, k2);
    if (l2 < 0) continue;
    for (int c = 0; c < nc; ++c) {
      double a = val[(size_t)nc * nc * pidx + nc * r + c];
      const double *zr = Zp + S.z_off + (long long)(nc * l2 + c) * m;
#pragma unroll
      for (int q = 0; q < kMaxModes; ++q)
        if (q < m) acc[q] += a * zr[q];
    }
  }
  double *yr = Yp + yoff[j] + (long long)t * m;
#pragma unroll
  for (int q = 0; q < kMaxModes; ++q)
    if (q < m) yr[q] = acc[q];
}

// A_H block of a pair of meeting subdomains, Z_j^T (A Z_k) over the nodes of
// V_{h,0}(Omega_j) inside Omega_k's box.  The rows are staged 32 at a time; a
// thread keeps one or two 2 x 2 blocks of the m_j x m_k products.  FP64 issue
// bounds it: the previous form (one entry per thread, its rows in a serial
// loop with index arithmetic per row) took 11.5 ms for 72 subdomains of 13,600
// unknowns and 28 ms for 108 Darcy ones.  Every entry is still one chain of
// multiply-adds over the rows: splitting the rows over the idle threads saved
// nothing more and made the coarse correction two to eight times less accurate
// (the entries cancel against each other along the rigid displacements).
constexpr int kCbRows = 32, kCbLd = kMaxModes + 2, kCbThreads = 128;
constexpr int kCbGroups = kMaxModes / 2 * kMaxModes / 2 / kCbThreads;
__global__ void __launch_bounds__(kCbThreads)
    k_coarse_blocks(const SubDesc *subs, const int2 *pairs, const double *__restrict__ Zp,
                    const double *__restrict__ Yp, const long long *yoff, double *AH, int nH) {
  const int2 pr = pairs[blockIdx.x];
  const SubDesc &Sj = subs[pr.x];
  const SubDesc &Sk = subs[pr.y];
  const int mj = Sj.m, mk = Sk.m, nc = Sj.nc, tid = threadIdx.x;
  __shared__ __align__(16) double zs[kCbRows][kCbLd], ys[kCbRows][kCbLd];
  __shared__ int zrow[kCbRows], yrow[kCbRows];
  int lo[3], ext[3];
  for (int d = 0; d < 3; ++d) {
    lo[d] = max(Sj.ibox.lo[d], Sk.nbox.lo[d]);
    ext[d] = max(0, min(Sj.ibox.lo[d] + Sj.ibox.n[d], Sk.nbox.lo[d] + Sk.nbox.n[d]) - lo[d]);
  }
  const int nrow = nc * ext[0] * ext[1] * ext[2];
  const int gk = (mk + 1) / 2, groups = (mj + 1) / 2 * gk;
  double acc[kCbGroups][2][2] = {};
  // odd counts: the last column of a 2 x 2 block multiplies zeros
  for (int e = tid; e < kCbRows * kCbLd; e += kCbThreads) zs[e / kCbLd][e % kCbLd] = ys[e / kCbLd][e % kCbLd] = 0.0;
  for (int r0 = 0; r0 < nrow; r0 += kCbRows) {
    const int rows = min(kCbRows, nrow - r0);
    __syncthreads();                       // the stage has been read
    if (tid < rows) {
      const int q = (r0 + tid) / nc, c = r0 + tid - nc * q;
      const int i = lo[0] + q % ext[0], t = q / ext[0], jj = lo[1] + t % ext[1], k = lo[2] + t / ext[1];
      zrow[tid] = nc * Sj.ibox.local(i, jj, k) + c;
      yrow[tid] = nc * Sk.nbox.local(i, jj, k) + c;
    }
    __syncthreads();
    for (int e = tid; e < rows * mj; e += kCbThreads) {
      const int r = e / mj, a = e - r * mj;
      zs[r][a] = __ldg(Zp + Sj.z_off + (long long)zrow[r] * mj + a);
    }
    for (int e = tid; e < rows * mk; e += kCbThreads) {
      const int r = e / mk, b = e - r * mk;
      ys[r][b] = __ldg(Yp + yoff[pr.y] + (long long)yrow[r] * mk + b);
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kCbGroups; ++q) {
      const int g = tid + q * kCbThreads;
      if (g >= groups) break;
      const int a0 = 2 * (g / gk), b0 = 2 * (g % gk);
      for (int r = 0; r < rows; ++r) {
        const double2 z = *reinterpret_cast<const double2 *>(&zs[r][a0]);
        const double2 y = *reinterpret_cast<const double2 *>(&ys[r][b0]);
        acc[q][0][0] = fma(z.x, y.x, acc[q][0][0]);
        acc[q][0][1] = fma(z.x, y.y, acc[q][0][1]);
        acc[q][1][0] = fma(z.y, y.x, acc[q][1][0]);
        acc[q][1][1] = fma(z.y, y.y, acc[q][1][1]);
      }
    }
  }
#pragma unroll
  for (int q = 0; q < kCbGroups; ++q) {
    const int g = tid + q * kCbThreads;
    if (g >= groups) break;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int a = 2 * (g / gk) + (e >> 1), b = 2 * (g % gk) + (e & 1);
      if (a >= mj || b >= mk) continue;
      const double s = acc[q][e >> 1][e & 1];
      AH[(long long)(Sj.coff + a) * nH + Sk.coff + b] = s;
      if (pr.x != pr.y) AH[(long long)(Sk.coff + b) * nH + Sj.coff + a] = s;
    }
  }
}

__global__ void k_dense_to_tiles(const double *AH, int n, const BandLayout *lay, double *pool) {
  const BandLayout L = lay[0];
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (long long)n * n) return;
  int R = (int)(t / n), C = (int)(t - (long long)R * n);
  if (R < C) return;
  tile_at(pool, L, R >> 5, (R >> 5) - (C >> 5))[(C & 31) * 32 + (R & 31)] = AH[t];
}

__global__ void k_symmetrize(double *M, int n) {
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (long long)n * n) return;
  int r = (int)(t / n), c = (int)(t - (long long)r * n);
  if (r >= c) return;
  double a = M[(long long)r * n + c], b = M[(long long)c * n + r];
  double v = 0.5 * (a + b);
  M[(long long)r * n + c] = v;
  M[(long long)c * n + r] = v;
}

__global__ void k_identity(double *M, int n) {
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (long long)n * n) return;
  int r = (int)(t / n), c = (int)(t - (long long)r * n);
  M[t] = r == c ? 1.0 : 0.0;
}

__global__ void k_normalize_cols(const SubDesc *subs, int npad, double *P, int ld, long long sp,
                                 int ncol, const double *G) {
  const int j = blockIdx.y;
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (long long)npad * ncol) return;
  int row = (int)(t / ncol), c = (int)(t - (long long)row * ncol);
  double g = G[(long long)j * ncol * ncol + c * ncol + c];
  double *pv = P + j * sp + (long long)row * ld + c;
  if (row >= subs[j].n_neu) {
    *pv = 0.0;
    return;
  }
  if (g > 0.0) *pv /= sqrt(g);
}

// Rigid displacements of the Neumann nodes of every subdomain (Sec. 5, zero
// energy modes): P[j][row][k] for k < 6 -- translations along x, y, z and
// rotations omega x (X - c) about the axes through the centre c of the
// subdomain's node box; columns 6.. and the padding rows are zero.
__global__ void k_rigid_modes(const SubDesc *subs, int npad, const double *__restrict__ X,
                              const double *__restrict__ Y, const double *__restrict__ Z,
                              double *P, int ld, long long sp) {
  const int j = blockIdx.y;
  const SubDesc &S = subs[j];
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (long long)npad * ld) return;
  const int row = (int)(t / ld), k = (int)(t - (long long)row * ld);
  double v = 0.0;
  if (S.nc == 1) {                // scalar problem: the constants
    v = (row < S.n_neu && k == 0) ? 1.0 : 0.0;
  } else if (row < S.n_neu && k < 6) {
    const int node = row / 3, comp = row - 3 * node;
    int gi, gj, gk;
    S.nbox.global(node, gi, gj, gk);
    const NodeBox &B = S.nbox;
    const double dx = X[gi] - 0.5 * (X[B.lo[0]] + X[B.lo[0] + B.n[0] - 1]);
    const double dy = Y[gj] - 0.5 * (Y[B.lo[1]] + Y[B.lo[1] + B.n[1] - 1]);
    const double dz = Z[gk] - 0.5 * (Z[B.lo[2]] + Z[B.lo[2] + B.n[2] - 1]);
    if (k < 3) {
      v = comp == k ? 1.0 : 0.0;
    } else if (k == 3) {          // about x: (0, -dz, dy)
      v = comp == 1 ? -dz : (comp == 2 ? dy : 0.0);
    } else if (k == 4) {          // about y: (dz, 0, -dx)
      v = comp == 0 ? dz : (comp == 2 ? -dx : 0.0);
    } else {                      // about z: (-dy, dx, 0)
      v = comp == 0 ? -dy : (comp == 1 ? dx : 0.0);
    }
  }
  P[j * sp + t] = v;
}

}  // namespace

void launch_rigid_modes(const SubDesc *d_subs, int nsub, int npad, const double *X,
                        const double *Y, const double *Z, double *P, int ld, long long sp,
                        cudaStream_t s) {
  long long tot = (long long)npad * ld;
  dim3 g((unsigned)((tot + 255) / 256), nsub);
  k_rigid_modes<<<g, 256, 0, s>>>(d_subs, npad, X, Y, Z, P, ld, sp); GENEO_COUNT_LAUNCH();
}

void launch_pou_neumann(const SubDesc *d_subs, int nsub, int max_nodes, const int *cand,
                        const int cand_off[3], const uint8_t *mask, int nnx, int nny, int nnz,
                        int px, int py, int kind, double *Xneu, cudaStream_t s) {
  dim3 g((3 * max_nodes + 255) / 256, nsub);
  k_pou_neumann<<<g, 256, 0, s>>>(d_subs, cand, cand_off[0], cand_off[1], cand_off[2], mask, nnx,
                                  nny, nnz, px, py, kind, Xneu); GENEO_COUNT_LAUNCH();
}

void launch_pou_interior(const SubDesc *d_subs, int nsub, int max_nodes, const int *cand,
                         const int cand_off[3], const uint8_t *mask, int nnx, int nny, int nnz,
                         int px, int py, int kind, double *wloc, cudaStream_t s) {
  dim3 g((3 * max_nodes + 255) / 256, nsub);
  k_pou_interior<<<g, 256, 0, s>>>(d_subs, cand, cand_off[0], cand_off[1], cand_off[2], mask,
                                   nnx, nny, nnz, px, py, kind, wloc); GENEO_COUNT_LAUNCH();
}

template <int NC>
static void launch_neumann(const SubDesc *d_subs, const BandLayout *d_lay, int nsub,
                           int max_nodes, int nx, int ny, int nz, const double *X, const double *Y,
                           const double *Z, const double *coef, const int *ecnt,
                           const int ecnt_off[3], const uint8_t *mask, const double *Xneu,
                           double sigma, double *poolS, double *Bloc, cudaStream_t s) {
  (void)ensure_smem(k_neumann_assemble<NC>, kNeuSmem<NC>);   // a failure surfaces as a launch error
  const dim3 g((unsigned)((max_nodes + kNeuNodes<NC> - 1) / kNeuNodes<NC>), nsub);
  k_neumann_assemble<NC><<<g, kNeuThreads<NC>, kNeuSmem<NC>, s>>>(
      d_subs, d_lay, nx, ny, nz, X, Y, Z, coef, ecnt, ecnt_off[0], ecnt_off[1], ecnt_off[2], mask,
      Xneu, sigma, poolS, Bloc); GENEO_COUNT_LAUNCH();
}

// Exactly one of Cel (elasticity) and perm (Darcy) is set.
void launch_neumann_assemble(const SubDesc *d_subs, const BandLayout *d_lay, int nsub,
                             int max_nodes, int nx, int ny, int nz, const double *X,
                             const double *Y, const double *Z, const double *Cel,
                             const double *perm,
                             const int *ecnt, const int ecnt_off[3], const uint8_t *mask,
                             const double *Xneu, double sigma, double *poolS, double *Bloc,
                             cudaStream_t s) {
  if (Cel)
    launch_neumann<3>(d_subs, d_lay, nsub, max_nodes, nx, ny, nz, X, Y, Z, Cel, ecnt, ecnt_off,
                      mask, Xneu, sigma, poolS, Bloc, s);
  else
    launch_neumann<1>(d_subs, d_lay, nsub, max_nodes, nx, ny, nz, X, Y, Z, perm, ecnt, ecnt_off,
                      mask, Xneu, sigma, poolS, Bloc, s);
}

void launch_bloc_mv(const SubDesc *d_subs, int nsub, int max_nodes, const double *Bloc,
                    const double *T, double *W, long long sys_stride, int p, cudaStream_t s) {
  dim3 g((3 * max_nodes + 127) / 128, nsub);
  k_bloc_mv<<<g, 128, 0, s>>>(d_subs, Bloc, T, W, sys_stride, p); GENEO_COUNT_LAUNCH();
}

void launch_random_block(const SubDesc *d_subs, int nsub, int npad, double *V, int ld,
                         long long sys_stride, int p, unsigned long long seed, cudaStream_t s) {
  dim3 g((npad * p + 255) / 256, nsub);
  k_random_block<<<g, 256, 0, s>>>(d_subs, npad, V, ld, sys_stride, p, seed); GENEO_COUNT_LAUNCH();
}

void launch_reorth_gate(int nsub, const double *G, int p, const double *H, int na, long long hs,
                        int *gate, cudaStream_t s) {
  k_reorth_gate<<<nsub, 32, 0, s>>>(G, p, H, na, hs, gate); GENEO_COUNT_LAUNCH();
}
void launch_cholqr(const SubDesc *d_subs, int nsub, int npad, const double *G, double *W,
                   int p, double *Racc, double *Rinv, int first, double abs_tiny, cudaStream_t s) {
  k_cholqr_small<<<nsub, 32, 0, s>>>(G, p, Rinv, Racc, first, abs_tiny); GENEO_COUNT_LAUNCH();
  dim3 g((npad + 255) / 256, nsub);
  k_rowmul<<<g, 256, 0, s>>>(d_subs, npad, W, p, Rinv); GENEO_COUNT_LAUNCH();
}

void launch_hm_accum(int nsub, double *Hm, int kdim, const double *Hs, int rows, int k, int p,
                     cudaStream_t s) {
  k_hm_accum<<<nsub, 256, 0, s>>>(Hm, kdim, Hs, rows, k, p); GENEO_COUNT_LAUNCH();
}

void launch_hm_subdiag(int nsub, double *Hm, int kdim, const double *Racc, int k, int p,
                       double *Rblk, cudaStream_t s) {
  k_hm_subdiag<<<nsub, 64, 0, s>>>(Hm, kdim, Racc, k, p, Rblk); GENEO_COUNT_LAUNCH();
}

void launch_restart_hm(int nsub, double *Hm, int kdim, const double *Eval, const double *Evec,
                       const double *Rblk, int kk, int p, cudaStream_t s) {
  k_restart_hm<<<nsub, 256, 0, s>>>(Hm, kdim, Eval, Evec, Rblk, kk, p); GENEO_COUNT_LAUNCH();
}

void launch_copy_block(const SubDesc *d_subs, int nsub, int npad, const double *W, int ldw,
                       long long sw, double *V, int ldv, long long sv, int p, cudaStream_t s) {
  dim3 g((npad * p + 255) / 256, nsub);
  k_copy_block<<<g, 256, 0, s>>>(d_subs, npad, W, ldw, sw, V, ldv, sv, p); GENEO_COUNT_LAUNCH();
}

int launch_ritz_eig(int nsub, const double *Hm, int kdim, int nw, int p, const double *Rblk,
                    double *Eval, double *Evec, double *Eres, cudaStream_t s) {
  if (kdim > kMaxKdim || nw > kdim) return GENEO_ERR_INVALID_ARG;
  int sm = (kdim * (kdim + 1) + 6 * kdim) * (int)sizeof(double);
  if (int st = ensure_smem(k_ritz_eig, sm)) return st;
  k_ritz_eig<<<nsub, 256, sm, s>>>(Hm, kdim, nw, p, Rblk, Eval, Evec, Eres); GENEO_COUNT_LAUNCH();
  GENEO_CUDA_TRY(cudaGetLastError());
  return GENEO_OK;
}

void launch_build_Z(const SubDesc *d_subs, int nsub, int max_nint, const double *P, int ldp,
                    long long sp, const double *Xneu, double *Zp, cudaStream_t s) {
  long long tot = (long long)max_nint * kMaxModes;
  dim3 g((unsigned)((tot + 255) / 256), nsub);
  k_build_Z<<<g, 256, 0, s>>>(d_subs, P, ldp, sp, Xneu, Zp); GENEO_COUNT_LAUNCH();
}

void launch_AZ(const SubDesc *d_subs, int nsub, int max_nodes, int nnx, int nny, int nnz,
               const int32_t *rp, const int32_t *col, const double *val, const double *Zp,
               const long long *yoff, double *Yp, cudaStream_t s) {
  dim3 g((3 * max_nodes + 127) / 128, nsub);
  k_AZ<<<g, 128, 0, s>>>(d_subs, nnx, nny, nnz, rp, col, val, Zp, yoff, Yp); GENEO_COUNT_LAUNCH();
}

void launch_coarse_blocks(const SubDesc *d_subs, const int2 *pairs, int npairs, const double *Zp,
                          const double *Yp, const long long *yoff, double *AH, int nH,
                          cudaStream_t s) {
  if (npairs > 0) {
    k_coarse_blocks<<<npairs, kCbThreads, 0, s>>>(d_subs, pairs, Zp, Yp, yoff, AH, nH);
    GENEO_COUNT_LAUNCH();
  }
}

void launch_dense_to_tiles(const double *AH, int nH, const BandLayout *d_lay, double *pool,
                           cudaStream_t s) {
  long long tot = (long long)nH * nH;
  k_dense_to_tiles<<<(unsigned)((tot + 255) / 256), 256, 0, s>>>(AH, nH, d_lay, pool); GENEO_COUNT_LAUNCH();
}

void launch_symmetrize(double *M, int n, cudaStream_t s) {
  long long tot = (long long)n * n;
  k_symmetrize<<<(unsigned)((tot + 255) / 256), 256, 0, s>>>(M, n); GENEO_COUNT_LAUNCH();
}

void launch_identity(double *M, int n, cudaStream_t s) {
  long long tot = (long long)n * n;
  k_identity<<<(unsigned)((tot + 255) / 256), 256, 0, s>>>(M, n); GENEO_COUNT_LAUNCH();
}

void launch_normalize_cols(const SubDesc *d_subs, int nsub, int npad, double *P, int ld,
                           long long sp, int ncol, const double *G, cudaStream_t s) {
  long long tot = (long long)npad * ncol;
  dim3 g((unsigned)((tot + 255) / 256), nsub);
  k_normalize_cols<<<g, 256, 0, s>>>(d_subs, npad, P, ld, sp, ncol, G); GENEO_COUNT_LAUNCH();
}

}  // namespace geneo
