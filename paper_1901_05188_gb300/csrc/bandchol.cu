// FP64 band Cholesky and the band solves with several right-hand sides, on the
// tensor cores by exact digit products (digits.cuh):
// the shift-invert operators of the GenEO eigenproblems (Sec. 3.3.2), the
// FP64 subdomain factors (Sec. 3.1) and the coarse matrix (Sec. 3.3.3).  The paper
// factors with a sparse direct solver (UMFPack); here every matrix is a band in
// a box numbering whose longest axis runs slowest, held as dense 32 x 32 tiles,
// with the diagonal blocks stored inverted so that triangular sweeps are
// streams of small products.
//
// Both were bound by the FP64 pipe (128 shifted Neumann matrices of
// about 16,000 unknowns and half-bandwidth 905: 1.31 s per factorisation, 32 ms
// per sweep with eight right-hand sides).
#include <cooperative_groups.h>

#include <algorithm>

#include "band.cuh"
#include "digits.cuh"

namespace geneo {

namespace cg = cooperative_groups;

namespace {

__device__ __forceinline__ double *tile_ptr(double *base, const BandLayout &L, int I, int d) {
  return base + L.off + ((long long)I * (L.w + 1) + d) * L.slot;
}

// Tile (I, d) of system j in the digit pool: in place of the FP64 tile, or only the
// w + 1 tile rows the factorisation can still touch (row I in slot I mod (w + 1)).
__device__ __forceinline__ __half *dig_tile(const DigitBand &D, const BandLayout &L, int j, int I,
                                            int d) {
  if (!D.window) return reinterpret_cast<__half *>(tile_ptr(static_cast<double *>(D.pool), L, I, d));
  return static_cast<__half *>(D.pool) +
         ((long long)j * D.window + (long long)(I % (L.w + 1)) * (L.w + 1) + d) * kDigTile;
}
static_assert(kDigSlot * 8 == kDigBytes && kDigHalves == kDigTile, "a slot holds a tile's digits");

// Scale of row i of the factor: |L_ik| <= sqrt(a_ii) < 2^E.
__global__ void k_row_exps(const BandLayout *lay, int sys0, double *poolL, DigitBand D) {
  const int j = sys0 + blockIdx.y;
  const BandLayout L = lay[j];
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= L.nt * 32) return;
  const double a = tile_ptr(poolL, L, i >> 5, 0)[(i & 31) * 33];
  const int e = a > 0.0 ? exp_above(a) : 0;
  D.rexp[(long long)j * D.npad + i] = e == kNoExp ? 0 : (e + 1) >> 1;
}

// Adds the products of one K tile to the integer sums of a 16 x 16 block: rows
// m0 of tile a times rows n0 of tile b (both in shared memory, [row][k] digit
// slices), eight columns at a time to stay within 128 registers.
__device__ __forceinline__ void block_product(long long (&hi)[8], long long (&lo)[8], uint32_t a,
                                              uint32_t b, int m0, int n0, int lane) {
  __syncwarp();
#pragma unroll
  for (int nb = 0; nb < 2; ++nb) {
    float S[kDig][4];
#pragma unroll
    for (int l = 0; l < kDig; ++l)
#pragma unroll
      for (int e = 0; e < 4; ++e) S[l][e] = 0.f;
#pragma unroll
    for (int kb = 0; kb < 2; ++kb) {
      uint32_t br[kDig][2];
      const uint32_t ab = a + ldsm_a(m0, 16 * kb, lane), bb = b + ldsm_b(n0 + 8 * nb, 16 * kb, lane);
#pragma unroll
      for (int t = 0; t < kDig; ++t) ldsm2(br[t], bb + t * 2048);
#pragma unroll
      for (int s = 0; s < kDig; ++s) {
        uint32_t ar[4];
        ldsm4(ar, ab + s * 2048);
#pragma unroll
        for (int t = 0; t < kDig - s; ++t) mma_f16(S[s + t], ar, br[t][0], br[t][1]);
      }
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      long long h, l;
      level_parts(S, e, h, l);
      hi[4 * nb + e] += h;
      lo[4 * nb + e] += l;
    }
  }
}
// Row and column of entry e (0..7) of a lane's 16 x 16 block.
__device__ __forceinline__ int blk_row(int e, int lane) { return (lane >> 2) + 8 * ((e >> 1) & 1); }
__device__ __forceinline__ int blk_col(int e, int lane) { return 2 * (lane & 3) + (e & 1) + 8 * (e >> 2); }

// Digits of a row-major 32 x 32 block in shared memory (row stride 33), rows
// [r0, r0 + n), with this lane's column taken times 2^cs: one warp, lane =
// column; scale 2^G per row, its own maximum (G written to rowexp) or the given
// one.  A row has one scale, so its entries have to be of one natural size:
// column k of R = L_IJ L_JJ^T is taken divided by the row scale of L at k, about
// sqrt(a_kk), and column k of inv(L_JJ) times it.  Without, a coefficient that
// jumps by 1e12 inside a tile cost the factor 2e-13 of sqrt(a_ii a_jj).  False
// if an entry is not finite or, at a given scale, not below it: the row scale of L
// is an upper bound of sqrt(a_ii), so the matrix is not positive definite (and
// fixed62 would cut the entry short, which can leave a positive pivot).
template <bool kOwn>
__device__ __forceinline__ bool slice_rows(const double *v, int r0, int n, int cs, int *rowexp,
                                           __half *dst, int lane) {
  bool fits = true;
  for (int r = r0; r < r0 + n; ++r) {
    const double x = v[r * 33 + lane];
    const int ex = exp_above(x);
    int G;
    if (kOwn) {
      G = __reduce_max_sync(0xffffffffu, ex == kNoExp ? ex : ex + cs);
      if (lane == 0) rowexp[r] = G;
    } else {
      G = rowexp[r];
    }
    fits = fits && ex < 1025 && (kOwn || ex <= G);
    const long long xb = fixed62(x, G - cs) + kDigBias;
    __half *o = dst + dig_index(r, lane);
#pragma unroll
    for (int s = 0; s < kDig; ++s) o[s * 1024] = digit_half(xb, s);
  }
  return fits;
}

__device__ __forceinline__ void not_spd(DevStatus *st, int j, int detail) {
  if (atomicCAS(&st->code, 0, GENEO_ERR_NOT_SPD) == 0) {
    st->where = j;
    st->detail = detail;
  }
}

// 1 / d for d > 0 (single-precision estimate, one third-order step: the error
// of the estimate, 2^-23, to the third power).
__device__ __forceinline__ double inv_pos(double d) {
  if (!(d >= 1e-30 && d <= 1e30)) return 1.0 / d;     // outside float range: exact path
  const double r = (double)__frcp_rn((float)d);
  const double e = fma(-d, r, 1.0);
  return fma(r, fma(e, e, e), r);
}
// 1 / sqrt(d), d > 0: Newton's iteration for 1 / y^2 - d from a single-precision estimate.
__device__ __forceinline__ double inv_sqrt(double d) {
  if (!(d >= 1e-30 && d <= 1e30)) return 1.0 / sqrt(d);
  double y = (double)rsqrtf((float)d);
  y = y * (1.5 - 0.5 * d * y * y);
  return y * (1.5 - 0.5 * d * y * y);
}

__device__ __forceinline__ void diag_bar() {
  __syncwarp();
  asm volatile("bar.sync 1, 128;" ::: "memory");
}

// Shared memory of a diagonal tile's factorisation.
struct DiagSmem {
  double A[32 * 33];
  double colv[32][32];
  double rinv[32];
  int ex[32], bad;
  __align__(16) __half dg[kDigTile];
};

// L D L^T of the diagonal tile J in Sm.A (updates applied) and the inverse of the
// unit factor together, one elimination step per column; the inverse of the
// Cholesky factor goes to the pools (in place, D.window = 0: only its digits).  Four warps, one per SM sub-partition;
// lane = row, warp w owns columns 4 q + w.  The FP64 pipe takes 64 cycles per
// warp instruction, so a step costs its eight updates (the entries of L right
// of the pivot and of the inverse left of it); the warp that owns the next
// column publishes it and its reciprocal pivot before its other updates.  One
// entry per thread with three barriers per column and the inverse afterwards
// took 44 us.
__device__ __forceinline__ void diag_factor(DiagSmem &Sm, const BandLayout &L, int j, int J,
                                            double *poolL, const DigitBand &D, DevStatus *st) {
  const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
  double *t = tile_ptr(poolL, L, J, 0), *A = Sm.A, *rinv = Sm.rinv;
  double (*colv)[32] = Sm.colv;
  int *ex = Sm.ex, *bad = &Sm.bad;
  __half *dg = Sm.dg;
  double a[8], x[8];
  const int cs = D.rexp[(long long)j * D.npad + J * 32 + lane];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    a[q] = A[lane * 33 + 4 * q + w];
    x[q] = lane == 4 * q + w ? 1.0 : 0.0;
  }
  auto publish = [&](int k, double v) {     // column k, final, and its reciprocal pivot
    colv[k][lane] = v;
    if (lane == k) {
      double d = v;
      if (!(d > 0.0)) {
        if (*bad < 0) *bad = J * 32 + k;
        d = 1.0;
        colv[k][lane] = d;
      }
      rinv[k] = inv_pos(d);
    }
  };
  if (w == 0) publish(0, a[0]);
  diag_bar();
#pragma unroll
  for (int k = 0; k < 32; ++k) {
    const int kq = k >> 2, kw = k & 3;
    const double li = lane > k ? colv[k][lane] * rinv[k] : 0.0;
    const bool own = k + 1 < 32 && w == ((k + 1) & 3);
    if (own) {
      const int q = (k + 1) >> 2;
      a[q] = fma(-li, colv[k][k + 1], a[q]);
      publish(k + 1, a[q]);
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      if (q > kq || (q == kq && w > kw)) {
        if (!(own && q == ((k + 1) >> 2))) a[q] = fma(-li, colv[k][4 * q + w], a[q]);
      } else {
        x[q] = fma(-li, __shfl_sync(0xffffffffu, x[q], k), x[q]);
      }
    }
    diag_bar();
  }
  const double rs = inv_sqrt(colv[lane][lane]);
  diag_bar();
#pragma unroll
  for (int q = 0; q < 8; ++q) A[lane * 33 + 4 * q + w] = x[q] * rs;      // inv(L_JJ)
  diag_bar();
  if (D.window)
    for (int e = tid; e < 1024; e += 128) t[e] = A[(e & 31) * 33 + (e >> 5)];
  const bool fits = slice_rows<true>(A, 8 * w, 8, cs, ex, dg, lane);
  if (!fits) *bad = J * 32;
  diag_bar();
  uint4 *dst = reinterpret_cast<uint4 *>(dig_tile(D, L, j, J, 0));
  for (int e = tid; e < kDigTile / 8; e += 128) dst[e] = reinterpret_cast<const uint4 *>(dg)[e];
  if (tid < 32) D.dexp[(long long)j * D.npad + J * 32 + tid] = ex[tid];
  if (tid == 0 && *bad >= 0) not_spd(st, j, *bad);
}

// The first diagonal tile of every system (all of them if no tiles couple); the
// others are factored by the panel launch before.
__global__ void __launch_bounds__(128)
    k_dchol_diag(const BandLayout *lay, int sys0, int J, double *poolL, DigitBand D, DevStatus *st) {
  const int j = sys0 + blockIdx.x;
  const BandLayout L = lay[j];
  if (J >= L.nt) return;
  __shared__ DiagSmem Sm;
  const double *t = tile_ptr(poolL, L, J, 0);
  for (int e = threadIdx.x; e < 1024; e += 128) Sm.A[(e & 31) * 33 + (e >> 5)] = t[e];
  if (threadIdx.x == 0) Sm.bad = -1;
  __syncthreads();
  diag_factor(Sm, L, j, J, poolL, D, st);
}

// Panel of tile column J, left-looking.  blockIdx.y = 2 + p takes the tiles (I, J),
// I = J + 2p + 2 and the next, subtracts sum_K L_IK L_JK^T over the band's
// columns K < J, multiplies by inv(L_JJ)^T (digits again) and writes the
// factor's FP64 tiles and digits.  The serial part of a column hides behind
// these: y = 0 finishes tile (J + 1, J), to which only column J - 1 is left to
// apply, then the diagonal tile J + 1 (columns J - 1 and J) and factors it, while
// y = 1 applies the columns K < J to the tiles (J + 2, J + 1) and (J + 2, J + 2),
// for y = 0 of the next launch.  With the diagonal tile in a launch of its own a
// column took 39 + 49 us on 16 systems of 7,600 unknowns, 53 + 119 us on 36 of
// 14,500 and 43 + 36 us on 54 Darcy ones (two such sets in flight); now 57, 115
// and 59 us, of which the serial part is 42.  Eight warps, 16 x 16 entries each; the K tiles
// come through two shared-memory stages, one copied while the other is used.
// Left-looking: the products of all K are summed as integers in registers, and
// each tile of A is read and written once (the right-looking FP64 update read
// and wrote the whole trailing triangle for every tile column).
constexpr int kPanStages = 2;
constexpr int kPanSmem = (3 * kPanStages + 1) * (int)kDigBytes;

__global__ void __launch_bounds__(256, 2)
    k_dchol_panel(const BandLayout *lay, int sys0, int J, double *poolL, DigitBand D, DevStatus *st) {
  const int j = sys0 + blockIdx.x;
  const BandLayout L = lay[j];
  if (J + 1 >= L.nt) return;
  const bool ahead = blockIdx.y == 1;
  const int I0 = ahead ? J + 2 : J + 2 * ((int)blockIdx.y - 1);
  if (blockIdx.y > 0 && (I0 >= L.nt || (ahead ? 1 : I0 - J) > L.w)) return;
  const bool two = !ahead && I0 + 1 < L.nt && I0 + 1 - J <= L.w;
  extern __shared__ __align__(128) unsigned char smraw[];
  __shared__ int rexp_s[64], rowe[64], cexp_s[32], dexp_s[32];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int tt = warp >> 2, m0 = 16 * ((warp >> 1) & 1), n0 = 16 * (warp & 1);
  const int K0 = max(0, I0 - L.w), nstep = max(0, J - K0);
  const uint32_t sm = dig_smem(smraw);
  __half *dinv = reinterpret_cast<__half *>(smraw + 3 * kPanStages * kDigBytes);
  auto tile_in = [&](uint32_t dst, const __half *src) {
    for (int e = tid; e < kDigTile / 8; e += 256) cp16(dst + 16 * e, src + 8 * e);
  };
  const long long eb = (long long)j * D.npad;
  if (blockIdx.y == 0) {
    // ---- tile (J + 1, J) and the diagonal tile J + 1
    const int I = J + 1;
    const bool tile = L.w >= 1, last = J >= 1 && L.w >= 2;
    double *R = reinterpret_cast<double *>(smraw + 2 * kDigBytes);      // [32][33]
    __half *dg = reinterpret_cast<__half *>(R + 32 * 33);
    DiagSmem &Sm = *reinterpret_cast<DiagSmem *>(dg + kDigTile);
    static_assert(2 * kDigBytes + 32 * 33 * 8 + kDigBytes + sizeof(DiagSmem) <= 3 * kPanStages * kDigBytes,
                  "the inverse of the diagonal tile follows the stages");
    if (tile) tile_in(dig_smem(dinv), dig_tile(D, L, j, J, 0));
    if (last) {
      tile_in(sm, dig_tile(D, L, j, I, 2));
      tile_in(sm + kDigBytes, dig_tile(D, L, j, J, 1));
    }
    cp_commit();
    if (tid < 32) {
      rexp_s[tid] = D.rexp[eb + I * 32 + tid];
      cexp_s[tid] = D.rexp[eb + J * 32 + tid];
      dexp_s[tid] = D.dexp[eb + J * 32 + tid];
    }
    const double *ta = tile_ptr(poolL, L, I, 0);
    double *tr = tile ? tile_ptr(poolL, L, I, 1) : nullptr;
    for (int e = tid; e < 1024; e += 256) {
      Sm.A[(e & 31) * 33 + (e >> 5)] = ta[e];
      if (tile) R[(e & 31) * 33 + (e >> 5)] = tr[e];
    }
    if (tid == 0) Sm.bad = -1;
    cp_wait<0>();
    __syncthreads();
    // warps 0..3 update the tile (J + 1, J), warps 4..7 the lower triangle of the diagonal tile
    auto update = [&](bool mine, uint32_t a, uint32_t b, double *T, const int *ec) {
      if (!mine) return;
      long long hi[8], lo[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) hi[e] = lo[e] = 0;
      block_product(hi, lo, a, b, m0, n0, lane);
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const int r = m0 + blk_row(e, lane), c = n0 + blk_col(e, lane);
        T[r * 33 + c] -= parts_value(hi[e], lo[e], rexp_s[r] + ec[c]);
      }
    };
    if (last)
      update(tt == 0 || m0 >= n0, sm, tt == 0 ? sm + kDigBytes : sm, tt == 0 ? R : Sm.A,
             tt == 0 ? cexp_s : rexp_s);
    __syncthreads();
    if (tile) {
      bool fits = slice_rows<true>(R, 4 * warp, 4, -cexp_s[lane], rowe, dg, lane);
      __syncthreads();
      if (tt == 0) {
        long long hi[8], lo[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) hi[e] = lo[e] = 0;
        block_product(hi, lo, dig_smem(dg), dig_smem(dinv), m0, n0, lane);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const int r = m0 + blk_row(e, lane), c = n0 + blk_col(e, lane);
          R[r * 33 + c] = parts_value(hi[e], lo[e], rowe[r] + dexp_s[c]);
        }
      }
      __syncthreads();
      fits = slice_rows<false>(R, 4 * warp, 4, 0, rexp_s, dg, lane) && fits;
      if (!fits) not_spd(st, j, J * 32);
      __syncthreads();
      update(tt == 1 && m0 >= n0, dig_smem(dg), dig_smem(dg), Sm.A, rexp_s);
      uint4 *dst = reinterpret_cast<uint4 *>(dig_tile(D, L, j, I, 1));
      const uint4 *src = reinterpret_cast<const uint4 *>(dg);
      for (int e = tid; e < kDigTile / 8; e += 256) dst[e] = src[e];
      if (D.window)
        for (int e = tid; e < 1024; e += 256) tr[e] = R[(e & 31) * 33 + (e >> 5)];
      __syncthreads();
    }
    if (warp < 4) diag_factor(Sm, L, j, I, poolL, D, st);
    return;
  }
  auto prefetch = [&](int it) {
    const uint32_t sp = sm + (it % kPanStages) * 3 * kDigBytes;
    const int K = K0 + it, C = ahead ? J + 1 : J;
    tile_in(sp, dig_tile(D, L, j, I0, I0 - K));
    if (two && I0 + 1 - K <= L.w) tile_in(sp + kDigBytes, dig_tile(D, L, j, I0 + 1, I0 + 1 - K));
    tile_in(sp + 2 * kDigBytes, dig_tile(D, L, j, C, C - K));
  };
  if (!ahead) tile_in(dig_smem(dinv), dig_tile(D, L, j, J, 0));
  if (nstep > 0) prefetch(0);
  cp_commit();
  if (tid < 64) rexp_s[tid] = (tid < 32 || two) ? D.rexp[eb + I0 * 32 + tid] : 0;
  if (tid < 32) {
    cexp_s[tid] = D.rexp[eb + (ahead ? J + 1 : J) * 32 + tid];
    dexp_s[tid] = D.dexp[eb + J * 32 + tid];
  }
  long long hi[8], lo[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) hi[e] = lo[e] = 0;
  for (int it = 0; it < nstep; ++it) {
    if (it + 1 < nstep) prefetch(it + 1);
    cp_commit();
    cp_wait<1>();
    __syncthreads();                        // the stage has landed
    const uint32_t sp = sm + (it % kPanStages) * 3 * kDigBytes;
    if (ahead) {                            // warps 0..3: (J + 2, J + 1), 4..7: (J + 2, J + 2)
      if (tt == 0 || m0 >= n0) block_product(hi, lo, sp, tt == 0 ? sp + 2 * kDigBytes : sp, m0, n0, lane);
    } else if (tt == 0 || (two && I0 + 1 - (K0 + it) <= L.w)) {
      block_product(hi, lo, sp + tt * kDigBytes, sp + 2 * kDigBytes, m0, n0, lane);
    }
    __syncthreads();                        // the stage is free
  }
  cp_wait<0>();
  __syncthreads();
  if (ahead) {
    if (nstep > 0 && (tt == 0 || m0 >= n0)) {
      double *t = tile_ptr(poolL, L, I0, tt == 0 ? 1 : 0);
      const int *ec = tt == 0 ? cexp_s : rexp_s;
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const int r = m0 + blk_row(e, lane), c = n0 + blk_col(e, lane);
        t[c * 32 + r] -= parts_value(hi[e], lo[e], rexp_s[r] + ec[c]);
      }
    }
  } else {
    double *R = reinterpret_cast<double *>(smraw);                              // [2][32][33]
    __half *dg = reinterpret_cast<__half *>(smraw + 2 * 32 * 33 * 8);           // [2] digit tiles
    double *Rt = R + tt * 32 * 33;
    const bool mine = tt == 0 || two;
    const int I = I0 + tt;
    if (mine) {
      const double *t = tile_ptr(poolL, L, I, I - J);
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const int r = m0 + blk_row(e, lane), c = n0 + blk_col(e, lane);
        Rt[r * 33 + c] = t[c * 32 + r] - parts_value(hi[e], lo[e], rexp_s[32 * tt + r] + cexp_s[c]);
      }
    }
    __syncthreads();
    bool fits = true;
    if (mine)
      fits = slice_rows<true>(Rt, 8 * (warp & 3), 8, -cexp_s[lane], rowe + 32 * tt, dg + tt * kDigTile, lane);
    __syncthreads();
    if (mine) {
#pragma unroll
      for (int e = 0; e < 8; ++e) hi[e] = lo[e] = 0;
      block_product(hi, lo, dig_smem(dg + tt * kDigTile), dig_smem(dinv), m0, n0, lane);
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const int r = m0 + blk_row(e, lane), c = n0 + blk_col(e, lane);
        Rt[r * 33 + c] = parts_value(hi[e], lo[e], rowe[32 * tt + r] + dexp_s[c]);
      }
    }
    __syncthreads();
    if (mine) {
      const int t4 = tid & 127;
      double *tl = tile_ptr(poolL, L, I, I - J);
      if (D.window)
        for (int e = t4; e < 1024; e += 128) tl[e] = Rt[(e & 31) * 33 + (e >> 5)];
      fits = slice_rows<false>(Rt, 8 * (warp & 3), 8, 0, rexp_s + 32 * tt, dg + tt * kDigTile, lane) && fits;
      if (!fits) not_spd(st, j, J * 32);
    }
    __syncthreads();
    if (mine) {
      uint4 *dst = reinterpret_cast<uint4 *>(dig_tile(D, L, j, I, I - J));
      const uint4 *src = reinterpret_cast<const uint4 *>(dg + tt * kDigTile);
      for (int e = tid & 127; e < kDigTile / 8; e += 128) dst[e] = src[e];
    }
  }
}

// The backward tile stream: U(J, d) = L(J + d, J)^T, one block per tile.  A pass of
// its own after the factorisation (which then never reads poolU), so that the
// digit windows can lie in poolU until here.
__global__ void __launch_bounds__(256)
    k_band_transpose(const BandLayout *lay, int w_max, const double *poolL, double *poolU) {
  const BandLayout L = lay[blockIdx.y];
  const int J = blockIdx.x / (w_max + 1), d = blockIdx.x - J * (w_max + 1);
  if (J >= L.nt || d > L.w || J + d >= L.nt) return;
  __shared__ double t[32][33];
  const double *l = poolL + L.off + ((long long)(J + d) * (L.w + 1) + d) * L.slot;
  double *u = tile_ptr(poolU, L, J, d);
  for (int e = threadIdx.x; e < 1024; e += 256) t[e >> 5][e & 31] = l[e];
  __syncthreads();
  for (int e = threadIdx.x; e < 1024; e += 256) u[e] = t[e & 31][e >> 5];
}

// ---- band solves with up to eight right-hand sides per cluster -----------------
// One cluster of one or two CTAs per (system, group of eight columns).  Row I needs
// s = b_I - sum_{d=1..w} L(I, I-d) y_{I-d} and y_I = inv(L_II) s; backward the
// transposes.  While the chain warps finish row I (the coupling d = 1, the
// inverse diagonal block), the eight far warps of every CTA multiply the tiles
// d >= 2 of the next row, which need only rows solved before; a pair of them
// takes one tile, 16 rows each, with the digits of L read by ldmatrix
// (transposed for the backward sweep, so one copy of the factor serves both) and
// those of y in fragment order.  Every row block of y has one scale per column,
// kept from row to row while it is at most four bits too large, so that the far
// warps can add the level sums of successive tiles as 32-bit integers; sums of
// different scales are aligned by shifting.  Each far warp copies its halves of
// the tiles into two private stages, the next one in flight while one is
// multiplied, across rows.  The window of y digits (w + 2 row blocks) lives in
// global scratch.
// The chain is a sequence of dependent integer instructions, at four to five
// cycles each, so it is spread wide and kept in integers: thread (c, r) of eight
// warps owns row r of column c.  Warps 0..3 multiply the chain's two tiles, a
// quarter each; meanwhile warps 4..7 form t = b - far sum and copy the next
// tiles.  s and y are cut into digits straight from the 128-bit sums; only the
// output becomes FP64, after the row's barrier.
// In a cluster the chain runs on the first CTA.  The second one only adds far
// warps: its other warps sum the CTA's partials of a row into the first CTA's
// buffer (integers: the result depends on the cluster only through the bits
// dropped when sums of different scales are aligned, below 2^-57 of the
// largest), and one cluster barrier ends the row.
// Bound: the larger of the chain (four barriers and two products, about 3 us a
// row) and a CTA's share of the tiles, where issuing the copies counts for as
// much as the matrix instructions.  Per launch of half the subdomains (forward
// or backward, eight right-hand sides): 36 of 14,500
// unknowns and 27 tiles half-bandwidth 1.4 ms, 54 Darcy ones of 16,000 and 7
// tiles 2.0 ms, 16 of 7,600 and 15 tiles 1.0 ms.  With four chain warps, FP64
// row values and one CTA per system they took 4.0, 2.3 and 1.7 ms.
constexpr int kSwChain = 8, kSwFar = 8;
constexpr int kSwThreads = (kSwChain + kSwFar) * 32;
constexpr int kSwHalf = kDigBytes / 2;      // a far warp's half of a tile
constexpr int kSwCol = 34;                  // row stride of a column of partial sums
constexpr int kSwPart = 8 * kSwCol;         // one 32 x 8 block of them
constexpr int kSwY = kDig * 128;            // words of one row block of y digits
constexpr int kSwSlack = 4;                 // bits a column's scale may be too large
constexpr int kSwFlush = 64;                // tiles added in 32 bits: 64 * 7 * 2^21 < 2^31
__host__ __device__ constexpr int sweep_smem(int w, int cl) {
  return 3 * (int)kDigBytes + kSwFar * 2 * kSwHalf + (2 * (3 + cl) + 2) * kSwPart * 16 +
         kSwY * 4 + 8 * 32 * 4 + 3 * 8 * 4 + (w + 2) * 16;
}

__device__ __forceinline__ void sw_bar_cta() {
  __syncwarp();                             // bar.sync is .aligned: converge first
  asm volatile("bar.sync 1, %0;" ::"n"(kSwThreads) : "memory");
}
// All CTAs of the cluster; their writes to shared and global memory are visible after it.
__device__ __forceinline__ void sw_bar_all(int cl) {
  if (cl == 1) return sw_bar_cta();
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void sw_bar_chain() {
  __syncwarp();
  asm volatile("bar.sync 2, %0;" ::"n"(kSwChain * 32) : "memory");
}

// hi 2^27 + lo, divided by 2^sh, added to the pair (hs, ls).
__device__ __forceinline__ void add_shifted(long long hi, long long lo, int sh, long long &hs,
                                            long long &ls) {
  const int s = min(sh, 62);
  const long long a = hi >> s, rem = hi - (a << s);          // 0 <= rem < 2^s
  hs += a;
  ls += s <= 30 ? ((rem << 27) + lo) >> s : (rem >> (s - 27)) + (lo >> s);
}

struct SweepArgs {
  const BandLayout *lay;
  DigitBand D;
  uint4 *ring;                              // y digits: [cluster][w_max + 2][kSwY / 4]
  int w_max;
  const double *in;
  long long in_sys;
  int in_row;
  double *out;
  long long out_sys;
  int out_row, ncols, mode, cl;
};

__global__ void __launch_bounds__(kSwThreads, 1) k_band_sweep(const SweepArgs P) {
  extern __shared__ __align__(128) unsigned char smraw[];
  const int cl = P.cl, rank = blockIdx.x % cl, j = blockIdx.x / cl, grp = blockIdx.y;
  const BandLayout L = P.lay[j];
  const int nt = L.nt, w = L.w, slots = w + 2, np = 3 + cl;
  unsigned char *chain_t = smraw;                                   // [diagonal x 2, coupling]
  unsigned char *far_t = chain_t + 3 * kDigBytes;                  // [warp][2] half tiles
  long long *part = reinterpret_cast<long long *>(far_t + kSwFar * 2 * kSwHalf);  // [2][np][hi, lo]
  long long *nearp = part + 2 * np * 2 * kSwPart;                   // [2][hi, lo]
  uint32_t *dig = reinterpret_cast<uint32_t *>(nearp + 2 * 2 * kSwPart);   // digits of s or y
  int *tf = reinterpret_cast<int *>(dig + kSwY);                    // [8][32] exponents of t
  int *fref = tf + 8 * 32;                                          // [2][8] scale of the far sums
  int *nanb = fref + 2 * 8;                                         // [8] b not finite in this row
  short *fexp = reinterpret_cast<short *>(nanb + 8);                // [w + 2][8]
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const cg::cluster_group cluster = cg::this_cluster();
  const char *tiles = static_cast<const char *>(P.D.pool) + L.off * 8;
  uint4 *yring = P.ring + ((long long)grp * (gridDim.x / cl) + j) * (P.w_max + 2) * (kSwY / 4);
  if (cl > 1) sw_bar_all(cl);               // every CTA is there before its memory is written
  for (int back = 0; back < 2; ++back) {
    if (!(P.mode & (1 << back))) continue;
    auto row = [&](int q) { return back ? nt - 1 - q : q; };
    auto dmax = [&](int I) { return back ? min(w, nt - 1 - I) : min(w, I); };
    auto tile_at = [&](int I, int d) {        // byte offset of the tile that couples row I to I -+ d
      return (long long)((back ? I + d : I) * (w + 1) + d) * (int)kDigBytes;
    };
    if (warp >= kSwChain) {
      // ---- far warps
      const int fw = warp - kSwChain, pl = fw >> 1, p = 4 * rank + pl, step = 4 * cl;
      const int m0 = 16 * (fw & 1), g = lane >> 2, t2 = 2 * (lane & 3);
      const uint32_t st0 = dig_smem(far_t) + fw * 2 * kSwHalf;
      // This warp's half of a tile, two 16 x 16 blocks of every slice: rows m0..
      // (forward) or columns m0.. (backward), the block of k = 16 kb.. at 512 kb.
      const char *lsrc = tiles + (back ? m0 * 32 : m0 * 64) + lane * 16;
      const int lnext = back ? 1024 : 512;
      auto load = [&](int stage, int I, int d) {
        const char *from = lsrc + tile_at(I, d);
        const uint32_t dst = st0 + stage * kSwHalf + lane * 16;
#pragma unroll
        for (int s = 0; s < kDig; ++s) {
          cp16(dst + s * 1024, from + s * 2048);
          cp16(dst + s * 1024 + 512, from + s * 2048 + lnext);
        }
      };
      const int ar0 = back ? (lane & 7) + 8 * (lane >> 4) : lane & 15;
      const uint32_t aoff = ar0 * 32 + (((back ? lane >> 3 : lane >> 4) ^ (ar0 >> 2)) & 1) * 16;
      // the warp's tiles in order: rows 1.. of the sweep, u = p, p + step, ... of each
      int pq = 0, pu = p, pn = 0;             // next tile to load: row q = pq, index pu of pn
      auto advance = [&]() {                  // to the next row that has one; false at the end
        while (pu >= pn) {
          if (++pq >= nt) return false;
          pn = max(dmax(row(pq)) - 1, 0);
          pu = p;
        }
        return true;
      };
      int stage = 0;
      if (advance()) {
        load(0, row(pq), 2 + pu);
        pu += step;
      }
      cp_commit();
      for (int q = 0; q < nt; ++q) {
        if (q + 1 < nt) {
          const int In = row(q + 1), n = max(dmax(In) - 1, 0);
          uint4 yb[kDig];
          auto y_in = [&](int slot) {
            const uint4 *yp = yring + slot * (kSwY / 4) + lane;
#pragma unroll
            for (int t = 0; t < kDig; ++t) yb[t] = rank ? __ldcg(yp + t * 32) : yp[t * 32];
          };
          int slot = (back ? In + 2 + p : In - 2 - p + slots) % slots;   // p <= w - 2 where it is used
          if (p < n) y_in(slot);
          const int fr0 = fref[((q + 1) & 1) * 8 + t2], fr1 = fref[((q + 1) & 1) * 8 + t2 + 1];
          long long *po = part + (((q + 1) & 1) * np + pl) * 2 * kSwPart;
          unsigned A[kDig][4];                // level sums of the tiles with scales (k0, k1)
          int k0 = 0, k1 = 0, cnt = 0;
          bool first = true;
#pragma unroll
          for (int l = 0; l < kDig; ++l)
#pragma unroll
            for (int e = 0; e < 4; ++e) A[l][e] = 0;
          auto flush = [&]() {                // A into this warp's partials
            const bool aligned = __all_sync(0xffffffffu, cnt == 0 || (k0 == fr0 && k1 == fr1));
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const int o = (t2 + (e & 1)) * kSwCol + m0 + g + 8 * (e >> 1);
              const unsigned z = cnt * 0x4b400000u;   // the start value of levels 0 and 1
              auto lev = [&](int l) { return (long long)(int)(l < 2 ? A[l][e] - z : A[l][e]); };
              const long long hi = lev(0) * 134217728 + lev(1) * 262144 + (lev(2) * 512 + lev(3)),
                              lo = lev(4) * 262144 + (lev(5) * 512 + lev(6));
              long long hs = first ? 0 : po[o], ls = first ? 0 : po[kSwPart + o];
              if (aligned) {
                hs += hi;
                ls += lo;
              } else {
                add_shifted(hi, lo, (e & 1) ? fr1 - k1 : fr0 - k0, hs, ls);
              }
              po[o] = hs;
              po[kSwPart + o] = ls;
#pragma unroll
              for (int l = 0; l < kDig; ++l) A[l][e] = 0u;
            }
            first = false;
            cnt = 0;
          };
          for (int u = p; u < n; u += step) {
            const short2 fk = *reinterpret_cast<const short2 *>(fexp + slot * 8 + t2);
            if (__any_sync(0xffffffffu, cnt == kSwFlush || (cnt > 0 && (fk.x != k0 || fk.y != k1)))) flush();
            k0 = fk.x;
            k1 = fk.y;
            if (advance()) {
              load(stage ^ 1, row(pq), 2 + pu);
              pu += step;
            }
            cp_commit();
            cp_wait<1>();
            __syncwarp();                     // this tile has landed, for every lane
            float S[kDig][4];
            level_start<2>(S);
#pragma unroll
            for (int kb = 0; kb < 2; ++kb) {
              const uint32_t ab = st0 + stage * kSwHalf + aoff + kb * 512;
              uint32_t ar[2][4];
              auto a_in = [&](int s) {
                if (back) ldsm4_trans(ar[s & 1], ab + s * 1024);
                else ldsm4(ar[s & 1], ab + s * 1024);
              };
              a_in(0);
#pragma unroll
              for (int s = 0; s < kDig; ++s) {
                if (s + 1 < kDig) a_in(s + 1);
#pragma unroll
                for (int t = 0; t < kDig - s; ++t)
                  mma_f16(S[s + t], ar[s & 1], kb ? yb[t].z : yb[t].x, kb ? yb[t].w : yb[t].y);
              }
            }
            __syncwarp();                     // every lane has read the stage
            stage ^= 1;
            if (u + step < n) {               // the next digits, in flight under the integer work
              slot += back ? step : -step;
              slot += slot < 0 ? slots : slot >= slots ? -slots : 0;
              y_in(slot);
            }
#pragma unroll
            for (int e = 0; e < 4; ++e)
#pragma unroll
              for (int l = 0; l < kDig; ++l)
                A[l][e] += l < 2 ? __float_as_int(S[l][e]) : __float2int_rn(S[l][e]);
            ++cnt;
          }
          if (cnt > 0 || first) flush();      // zeros if there was no tile
        }
        if (rank) sw_bar_cta();               // to this CTA's summing warps
        sw_bar_all(cl);
      }
    } else if (rank) {
      // ---- summing warps of the second CTA
      const int o = warp * kSwCol + lane;
      for (int q = 0; q < nt; ++q) {
        sw_bar_cta();
        if (q + 1 < nt) {
          const int buf = ((q + 1) & 1) * np;
          long long h = 0, l = 0;
#pragma unroll
          for (int p = 0; p < 4; ++p) {
            h += part[(buf + p) * 2 * kSwPart + o];
            l += part[(buf + p) * 2 * kSwPart + kSwPart + o];
          }
          long long *po = cluster.map_shared_rank(part, 0) + (buf + 3 + rank) * 2 * kSwPart + o;
          po[0] = h;
          po[kSwPart] = l;
        }
        sw_bar_all(cl);
      }
    } else {
      // ---- chain warps: thread (c, r) = (warp, lane) owns row r of column c
      const bool mult = warp < 4;             // the others: t = b - far sum, copies
      const int kb = warp & 1, m0 = 16 * ((warp >> 1) & 1), t2 = 2 * (lane & 3), g = lane >> 2;
      const int c = warp, o = c * kSwCol + lane, c2 = 2 * (warp & 3);
      const bool fresh = !(back && (P.mode & 1));
      const double *src = (fresh ? P.in + j * P.in_sys : P.out + j * P.out_sys) + grp * 8 + c2;
      const long long sst = fresh ? P.in_row : P.out_row;
      double *dst = P.out + j * P.out_sys + grp * 8 + c;
      const bool live0 = !mult && grp * 8 + c2 < P.ncols, live1 = !mult && grp * 8 + c2 + 1 < P.ncols;
      const int *re = P.D.rexp + (long long)j * P.D.npad + lane, *de = P.D.dexp + (long long)j * P.D.npad + lane;
      // half of row `lane`, column c in a row block of digits
      const int half = 2 * ((c * 4 + ((lane & 7) >> 1)) * 4 + 2 * (lane >> 4) + ((lane >> 3) & 1)) + (lane & 1);
      double b0 = 0.0, b1 = 0.0, n0 = 0.0, n1 = 0.0;
      int eR = 0, eD = 0, nR = 0, nD = 0;
      auto fetch = [&](int q) {
        const int i = row(q) * 32 + lane;
        n0 = live0 && i < L.n ? src[i * sst] : 0.0;
        n1 = live1 && i < L.n ? src[i * sst + 1] : 0.0;
        nR = re[row(q) * 32];
        nD = de[row(q) * 32];
      };
      const uint32_t diag_t = dig_smem(chain_t), near_t = diag_t + 2 * kDigBytes;
      const int ct = tid & 127;
      auto tile_in = [&](uint32_t to, int I, int d) {        // a chain tile, by four warps
        const char *from = tiles + tile_at(I, d) + ct * 16;
#pragma unroll
        for (int k = 0; k < 7; ++k) cp16(to + 16 * (k * 128 + ct), from + k * 2048);
      };
      auto near_in = [&](int q) {
        if (q < nt && dmax(row(q)) >= 1) tile_in(near_t, row(q), 1);
      };
      // product of this warp's quarter of a chain tile with the digit block, to nearp[kb]
      auto product = [&](uint32_t tile) {
        __syncwarp();
        float S[kDig][4];
        uint2 yb[kDig];
        uint32_t ar[kDig][4];
        const uint32_t ab = tile + (back ? ldsm_at(m0, 16 * kb, lane) : ldsm_a(m0, 16 * kb, lane));
#pragma unroll
        for (int s = 0; s < kDig; ++s) {
          yb[s] = *reinterpret_cast<const uint2 *>(dig + s * 128 + lane * 4 + 2 * kb);
          if (back) ldsm4_trans(ar[s], ab + s * 2048);
          else ldsm4(ar[s], ab + s * 2048);
        }
        level_start<4>(S);
#pragma unroll
        for (int s = 0; s < kDig; ++s)
#pragma unroll
          for (int t = 0; t < kDig - s; ++t) mma_f16(S[s + t], ar[s], yb[t].x, yb[t].y);
        long long *po = nearp + kb * 2 * kSwPart;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          long long hi, lo;
          level_parts<4>(S, e, hi, lo);
          const int oe = (t2 + (e & 1)) * kSwCol + m0 + g + 8 * (e >> 1);
          po[oe] = hi;
          po[kSwPart + oe] = lo;
        }
      };
      auto store_digits = [&](const Fixed &v, int G, __half *a, __half *z) {
        const long long xb = v.at(G) + kDigBias;
#pragma unroll
        for (int s = 0; s < kDig; ++s) {
          const __half d = digit_half(xb, s);
          a[s * 256] = d;
          if (z) z[s * 256] = d;
        }
      };
      __half *dh = reinterpret_cast<__half *>(dig) + half;
      fetch(0);
      for (int z = lane; z < slots; z += 32) fexp[z * 8 + c] = kNoExp;   // the first CTA's copy
      if (lane < 2) fref[lane * 8 + c] = kNoExp;
      if (!mult) tile_in(diag_t, row(0), 0);
      cp_commit();
      cp_wait<0>();
      sw_bar_chain();
      int F = kNoExp;                         // scale of the last solved row, this column
      Fixed y{0, kNoExp, false};
      int yi = L.n;                           // its unknown, not yet stored
      // A right-hand side that is not finite has no digits: its column is NaN from
      // that row on, as coupling by dense tiles makes it (w = 0: in that row).
      bool lost = false;
      auto store = [&]() {
        if (yi < L.n && grp * 8 + c < P.ncols)
          dst[(long long)yi * P.out_row] = lost ? __longlong_as_double(0x7ff8000000000000LL) : y.value();
      };
      int slot = row(0) % slots;              // of row I
      for (int q = 0; q < nt; ++q) {
        const int I = row(q);
        const bool has1 = dmax(I) >= 1;
        b0 = n0;
        b1 = n1;
        eR = nR;
        eD = nD;
        // powers of two: of the sums with L's rows and with inv(L_II), into the solved
        // row and into s (the digits of inv(L_II) carry the row scales of L in its columns)
        const int sR = back ? 0 : eR, sD = back ? -eR : eD, fR = back ? eR : 0, fD = back ? eD : -eR;
        if (mult) {
          if (has1) product(near_t);
        } else {
          // t = b - far sum, two entries, to the first block of partials
          long long *po = part + (q & 1) * np * 2 * kSwPart + c2 * kSwCol + lane;
#pragma unroll
          for (int x = 0; x < 2; ++x, po += kSwCol) {
            long long h = 0, l = 0;
            int ef = kNoExp;
            if (q > 0) {
              ef = fref[(q & 1) * 8 + c2 + x] + sR;
#pragma unroll 4
              for (int p = 0; p < np; ++p) {
                h += po[p * 2 * kSwPart];
                l += po[p * 2 * kSwPart + kSwPart];
              }
            }
            const double b = x ? b1 : b0;
            const int eb = exp_above(b) - 10, ft = max(ef, eb);
            const bool bad = __any_sync(0xffffffffu, eb >= 1015);     // infinite or NaN
            if (lane == 0) nanb[c2 + x] = bad;
            long long ht = 0, lt = 0;
            add_shifted(mantissa53(b), 0, ft - eb, ht, lt);
            add_shifted(-h, -l, ft - ef, ht, lt);
            po[0] = ht;
            po[kSwPart] = lt;
            tf[(c2 + x) * 32 + lane] = ft;
          }
          if (q + 1 < nt) tile_in(diag_t + ((q + 1) & 1) * kDigBytes, row(q + 1), 0);
        }
        cp_commit();
        store();
        if (q + 1 < nt) fetch(q + 1);
        sw_bar_chain();
        lost = nanb[c] || (lost && w > 0);
        int G;
        {
          const long long *tp = part + (q & 1) * np * 2 * kSwPart + o;
          const int ft = tf[c * 32 + lane], en = has1 ? F + sR : kNoExp, fs = max(ft, en);
          long long hs = 0, ls = 0;
          add_shifted(tp[0], tp[kSwPart], fs - ft, hs, ls);
          if (has1)
            add_shifted(-(nearp[o] + nearp[2 * kSwPart + o]), -(nearp[kSwPart + o] + nearp[3 * kSwPart + o]),
                        fs - en, hs, ls);
          // digits of s, its entries of one natural size
          Fixed s = fixed_of(hs, ls, fs);
          s.ex += fD;
          G = __reduce_max_sync(0xffffffffu, s.ex);
          store_digits(s, G, dh, nullptr);
        }
        sw_bar_chain();
        int fm = kNoExp;                      // the largest scale of the window so far
        for (int z = lane; z < slots; z += 32) fm = max(fm, (int)fexp[z * 8 + c]);
        if (mult) {
          product(diag_t + (q & 1) * kDigBytes);
        } else {
          near_in(q + 1);                     // the coupling tile has been read
          cp_commit();
        }
        fm = __reduce_max_sync(0xffffffffu, fm);
        sw_bar_chain();
        {
          y = fixed_of(nearp[o] + nearp[2 * kSwPart + o], nearp[kSwPart + o] + nearp[3 * kSwPart + o], G + sD);
          yi = I * 32 + lane;
          // digits of the solved row (backward: scaled by the factor's row scales)
          Fixed v = y;
          v.ex += fR;
          const int need = __reduce_max_sync(0xffffffffu, v.ex);
          if (need > F || (need > kNoExp / 2 && F - need > kSwSlack)) F = need + 1;
          store_digits(v, F, dh, reinterpret_cast<__half *>(yring + slot * (kSwY / 4)) + half);
          if (lane < cl) {                    // the far warps of every CTA read these
            cluster.map_shared_rank(fexp, lane)[slot * 8 + c] = (short)F;
            cluster.map_shared_rank(fref, lane)[(q & 1) * 8 + c] = max(fm, F);
          }
          slot += back ? -1 : 1;
          slot = slot < 0 ? slots - 1 : slot == slots ? 0 : slot;
        }
        cp_wait<0>();                         // the next row's tiles, before the barrier
        sw_bar_all(cl);
      }
      store();
      sw_bar_chain();                         // before the backward sweep fetches them
    }
  }
}

}  // namespace

int launch_band_cholesky64(const BandLayout *d_lay, int nsys, int nt_max, int w_max, double *poolL,
                           double *poolU, const DigitBand &D, DevStatus *st, cudaStream_t s,
                           cudaStream_t side) {
  if (int rc = ensure_smem(k_dchol_panel, kPanSmem)) return rc;
  // Two halves of the systems on two streams: one half's diagonal tiles (a
  // serial chain on a few warps) run under the other half's panels.
  const int half = side && nsys >= 2 ? (nsys + 1) / 2 : nsys;
  struct Events {
    cudaEvent_t fork = nullptr, join = nullptr;
    ~Events() {
      if (fork) cudaEventDestroy(fork);
      if (join) cudaEventDestroy(join);
    }
  } ev;
  if (half < nsys) {
    GENEO_CUDA_TRY(cudaEventCreateWithFlags(&ev.fork, cudaEventDisableTiming));
    GENEO_CUDA_TRY(cudaEventCreateWithFlags(&ev.join, cudaEventDisableTiming));
    GENEO_CUDA_TRY(cudaEventRecord(ev.fork, s));
    GENEO_CUDA_TRY(cudaStreamWaitEvent(side, ev.fork, 0));
  }
  for (int J = -1; J + 1 < nt_max; ++J)
    for (int h = 0; h < (half < nsys ? 2 : 1); ++h) {
      const int j0 = h ? half : 0, n = h ? nsys - half : half;
      cudaStream_t q = h ? side : s;
      if (J < 0) {
        k_row_exps<<<dim3((nt_max * 32 + 255) / 256, n), 256, 0, q>>>(d_lay, j0, poolL, D); GENEO_COUNT_LAUNCH();
        k_dchol_diag<<<n, 128, 0, q>>>(d_lay, j0, 0, poolL, D, st); GENEO_COUNT_LAUNCH();
      } else if (w_max == 0) {
        k_dchol_diag<<<n, 128, 0, q>>>(d_lay, j0, J + 1, poolL, D, st); GENEO_COUNT_LAUNCH();
      } else {
        const int d = std::min(w_max, nt_max - 1 - J);      // tiles (J + 2 .. J + d, J) in pairs
        k_dchol_panel<<<dim3(n, d / 2 + 2), 256, kPanSmem, q>>>(d_lay, j0, J, poolL, D, st); GENEO_COUNT_LAUNCH();
      }
    }
  if (half < nsys) {
    GENEO_CUDA_TRY(cudaEventRecord(ev.join, side));
    GENEO_CUDA_TRY(cudaStreamWaitEvent(s, ev.join, 0));
  }
  if (poolU) {
    const dim3 g((unsigned)(nt_max * (w_max + 1)), nsys);
    k_band_transpose<<<g, 256, 0, s>>>(d_lay, w_max, poolL, poolU); GENEO_COUNT_LAUNCH();
  }
  GENEO_CUDA_TRY(cudaGetLastError());
  return GENEO_OK;
}

// Widest half-bandwidth the set-up takes, in tiles: a vector's window of FP64 tile
// rows filled shared memory there.  This kernel fits up to 1,650.
constexpr int kSwMaxBand = 872;
static_assert(sweep_smem(kSwMaxBand, 1) <= 227 * 1024, "every accepted band has a launch");
bool band_solve_fits(int w_max) { return w_max <= kSwMaxBand; }

size_t band_solve_scratch(int nsys, int w_max, int ncols) {
  return (size_t)nsys * ((ncols + 7) / 8) * (w_max + 2) * kSwY * 4;
}

int launch_band_solve64(const BandLayout *d_lay, int nsys, int w_max, const DigitBand &D,
                        void *scratch, const double *in, long long in_sys, int in_row, double *out,
                        long long out_sys, int out_row, int ncols, int mode, cudaStream_t s,
                        int alongside, int ctas) {
  if (D.window || ctas < 0 || ctas > 2) return GENEO_ERR_INVALID_ARG;
  int dev = 0, sms = 0;
  GENEO_CUDA_TRY(cudaGetDevice(&dev));
  GENEO_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  // A second CTA for the far tiles while every CTA of the launches in flight
  // still has an SM of its own and a full row has a tile for each pair of warps.
  // All sweeps of one solve with and without: 93 and 135 ms (32 systems, 15 tiles),
  // 200 and 283 ms (72 systems, 27 tiles).
  const int groups = (ncols + 7) / 8;
  const int cl = ctas ? ctas
                 : 2 * groups * (nsys + alongside) <= sms && w_max - 1 > 4 &&
                         sweep_smem(w_max, 2) <= 227 * 1024 ? 2 : 1;
  const int sm = sweep_smem(w_max, cl);
  if (sm > 227 * 1024) return GENEO_ERR_INVALID_ARG;
  if (int rc = ensure_smem(k_band_sweep, sm)) return rc;
  const SweepArgs P{d_lay, D, static_cast<uint4 *>(scratch), w_max, in, in_sys, in_row, out, out_sys,
                    out_row, ncols, mode, cl};
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(nsys * cl, groups);
  cfg.blockDim = dim3(kSwThreads);
  cfg.dynamicSmemBytes = sm;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim = {(unsigned)cl, 1, 1};
  cfg.attrs = at;
  cfg.numAttrs = 1;
  GENEO_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_band_sweep, P)); GENEO_COUNT_LAUNCH();
  GENEO_CUDA_TRY(cudaGetLastError());
  return GENEO_OK;
}

}  // namespace geneo
