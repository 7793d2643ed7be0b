// Tall-skinny FP64 products of the block Lanczos process on the tensor cores, by
// exact digits (digits.cuh): H = V^T W (k_tsdots) and C = beta C + alpha V H
// (k_tsgemm), V of at most 128 and W of at most 32 columns, thousands of rows.
//
// Both were bound by the FP64 pipe: a row costs na * nb multiply-adds there, two
// a clock and SM.  Cutting an entry into digits costs about sixty integer
// instructions once and serves all its products, so the digits are made on the
// way, from the FP64 arrays, and nothing else changes hands.  Integer sums are
// exact.  Lost are what the entries have below 2^-60 of the largest of their
// column (k_tsdots) or row of A and column of H (k_tsgemm), the levels left out,
// as much again, and one FP64 rounding per entry, chunk of rows, 256 tiles and
// growth of a column's scale: over n terms 3 n 2^-60 of the product of the largest
// entries.  An FP64 sum errs by up to n 2^-53 of the sum of |v w|, which is less only
// where that sum is below 3/128 of the product of the largest.
//
// Half of 108 subdomains of 16,000 unknowns: V^T W of 64 columns 0.54 ms, W^T W
// 0.08 ms, V H of 64 columns 0.45 ms, on the FP64 pipe 0.76 ms (all sizes of V
// together), 0.3 ms and 0.99 ms; what is left is the cutting (integer issue) and,
// for the Gram matrices, reading W once.
#include <algorithm>

#include "digits.cuh"
#include "geneo.cuh"

namespace geneo {

namespace {

constexpr int kTsThreads = 256, kTsRows = 32;
constexpr int kTsFlush = 256;               // tiles summed in 32 bits: 256 * 7 * 2^20 < 2^31

// Digits of one entry, at element (r, c) of 32 x 32 tile `dst`.
__device__ __forceinline__ void ts_slice(__half *dst, int r, int c, double x, int G) {
  const long long xb = fixed62(x, G) + kDigBias;
  __half *o = dst + dig_index(r, c);
#pragma unroll
  for (int s = 0; s < kDig; ++s) o[s * 1024] = digit_half(xb, s);
}
// B operand of k = 0..31 (rows of the tile), columns n0..n0+7: words 2 kb, 2 kb + 1.
__device__ __forceinline__ void ts_b(uint32_t (&b)[4], uint32_t tile, int n0, int lane) {
  ldsm4_trans(b, tile + 2 * dig_index(lane, n0));
}

// ---- H = A^T B over a chunk of rows ----------------------------------------------
// One CTA per (chunk, subdomain, `width` columns of B: as many as leave at most
// sixteen blocks and halves).  Rows are taken 32 at a time: each thread reads
// its entries (lane = column), the running largest exponent of every column is
// kept, and the digits go to shared memory at a scale that may be up to two bits
// too large; only when a column outgrows its scale are the sums so far turned
// into FP64.  A warp owns one of the 16 x 8 blocks of H and half of the 32
// rows, as 32-bit level sums.
// NCG: 32-column groups of V, four at most (kMaxKdim).
template <int NCG>
__host__ __device__ constexpr int tsdots_smem() {
  return (NCG + 1) * (int)kDigBytes + 2 * 1024 * 8 + 2 * (32 * NCG + 32) * 4;
}

template <int NCG, int WARPS>
__global__ void __launch_bounds__(32 * WARPS, 16 / WARPS)
    k_tsdots(const SubDesc *subs, const double *__restrict__ A, int lda, long long sa, int na,
             const double *__restrict__ B, int ldb, long long sb, int nball, int width, double *Hpart,
             int chunks, const int *gate) {
  const int j = blockIdx.y, ch = blockIdx.x;
  if (gate && !gate[j]) return;                       // the reduction writes zeros
  const int n = subs[j].n_neu;
  const int per = ((n + chunks - 1) / chunks + kTsRows - 1) / kTsRows * kTsRows;
  const int r0 = min(n, ch * per), r1 = min(n, r0 + per);
  constexpr int T = 32 * WARPS, R = kTsRows / WARPS;  // threads; rows a warp reads of 32
  extern __shared__ __align__(128) unsigned char smraw[];
  __half *dA = reinterpret_cast<__half *>(smraw);     // [NCG] tiles [row][column]
  __half *dB = dA + NCG * kDigTile;
  double *sum = reinterpret_cast<double *>(dB + kDigTile);   // [2][16 x 8 blocks, 128 each]
  int *mx = reinterpret_cast<int *>(sum + 2 * 1024);  // largest exponents: A's, then B's columns
  int *G = mx + 32 * NCG + 32;                        // their scales
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int b0 = blockIdx.z * width, nb = min(width, nball - b0);     // this CTA's columns of B
  const int mt = (na + 15) / 16, jobs = 2 * mt * ((nb + 7) / 8);
  const double *Aj = A + j * sa, *Bj = B + j * sb + b0;
  for (int e = tid; e < 32 * NCG + 32; e += T) mx[e] = G[e] = kNoExp;
  for (int e = tid; e < 2 * 1024; e += T) sum[e] = 0.0;
  double x[NCG + 1][R];                               // rows R warp .. + R - 1
  auto fetch = [&](int rb) {
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const int r = rb + R * warp + i;
#pragma unroll
      for (int q = 0; q < NCG; ++q)
        x[q][i] = r < r1 && 32 * q + lane < na ? Aj[(long long)r * lda + 32 * q + lane] : 0.0;
      x[NCG][i] = r < r1 && lane < nb ? Bj[(long long)r * ldb + lane] : 0.0;
    }
  };
  // this warp's block of H, rows of A^T m0.. and columns n0.., and half kb of k
  const bool work = warp < jobs;
  const int blk = warp >> 1, kb = warp & 1, m0 = 16 * (blk % mt), n0 = 8 * (blk / mt);
  unsigned acc[kDig][4];
  int cnt = 0;
#pragma unroll
  for (int l = 0; l < kDig; ++l)
#pragma unroll
    for (int e = 0; e < 4; ++e) acc[l][e] = 0u;
  auto flush = [&]() {                                // the level sums, into this warp's block
    const unsigned z = cnt * 0x4b400000u;             // the start value of levels 0..3
    if (work)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int r = (lane >> 2) + 8 * (e >> 1), c = 2 * (lane & 3) + (e & 1);
        auto lev = [&](int l) { return (long long)(int)(l < 4 ? acc[l][e] - z : acc[l][e]); };
        const long long hi = lev(0) * 134217728 + lev(1) * 262144 + (lev(2) * 512 + lev(3)),
                        lo = lev(4) * 262144 + (lev(5) * 512 + lev(6));
        sum[kb * 1024 + blk * 128 + r * 8 + c] += parts_value(hi, lo, G[m0 + r] + G[32 * NCG + n0 + c]);
#pragma unroll
        for (int l = 0; l < kDig; ++l) acc[l][e] = 0u;
      }
    cnt = 0;
  };
  fetch(r0);
  __syncthreads();
  for (int rb = r0; rb < r1; rb += kTsRows) {
#pragma unroll
    for (int q = 0; q <= NCG; ++q) {
      int ex = exp_above(x[q][0]);
#pragma unroll
      for (int i = 1; i < R; ++i) ex = max(ex, exp_above(x[q][i]));
      if (ex > mx[32 * q + lane]) atomicMax(mx + 32 * q + lane, ex);
    }
    __syncthreads();                                  // also: the digits have been read
    bool grow = false;
    for (int e = tid; e < 32 * NCG + 32; e += T) grow = grow || mx[e] > G[e];
    if (__syncthreads_or(grow)) {
      if (cnt > 0) flush();
      __syncthreads();
      for (int e = tid; e < 32 * NCG + 32; e += T)
        if (mx[e] > G[e]) G[e] = mx[e] + 2;
      __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < R; ++i) {
#pragma unroll
      for (int q = 0; q < NCG; ++q)
        ts_slice(dA + q * kDigTile, R * warp + i, lane, x[q][i], G[32 * q + lane]);
      if (lane < 8 * ((nb + 7) / 8)) ts_slice(dB, R * warp + i, lane, x[NCG][i], G[32 * NCG + lane]);
    }
    __syncthreads();
    if (rb + kTsRows < r1) fetch(rb + kTsRows);       // in flight under the products
    if (work) {
      const uint32_t a = dig_smem(dA) + (m0 >> 5) * kDigBytes + ldsm_at(m0 & 31, 16 * kb, lane);
      float S[kDig][4];
      uint32_t bw[kDig][2];
#pragma unroll
      for (int t = 0; t < kDig; ++t) {
        uint32_t w4[4];
        ts_b(w4, dig_smem(dB) + t * 2048, n0, lane);
        bw[t][0] = kb ? w4[2] : w4[0];
        bw[t][1] = kb ? w4[3] : w4[1];
      }
      level_start<4>(S);
#pragma unroll
      for (int s = 0; s < kDig; ++s) {
        uint32_t ar[4];
        ldsm4_trans(ar, a + s * 2048);
#pragma unroll
        for (int t = 0; t < kDig - s; ++t) mma_f16(S[s + t], ar, bw[t][0], bw[t][1]);
      }
#pragma unroll
      for (int l = 0; l < kDig; ++l)
#pragma unroll
        for (int e = 0; e < 4; ++e)
          acc[l][e] += l < 4 ? __float_as_uint(S[l][e]) : (unsigned)__float2int_rn(S[l][e]);
    }
    if (++cnt == kTsFlush) flush();
  }
  if (cnt > 0) flush();
  __syncthreads();
  double *out = Hpart + ((long long)j * chunks + ch) * na * nball + b0;
  for (int o = tid; o < na * nb; o += T) {
    const int a = o / nb, b = o - a * nb, e = ((b >> 3) * mt + (a >> 4)) * 128 + (a & 15) * 8 + (b & 7);
    const bool finite = mx[a] < 1025 && mx[32 * NCG + b] < 1025;
    out[a * nball + b] = finite ? sum[e] + sum[1024 + e] : __longlong_as_double(0x7ff8000000000000LL);
  }
}

// H = W^T W for at most eight columns: 128 rows a turn, four entries per thread,
// one tile of digits for every 32 rows that serves as both operands.  A warp
// owns half of one of the four tiles; the eight sums are added at the end.
constexpr int kTgSmem = 4 * (int)kDigBytes + 8 * 64 * 8;
__global__ void __launch_bounds__(kTsThreads, 2)
    k_tsgram(const SubDesc *subs, const double *__restrict__ W, int ldw, long long sw, int p,
             double *Hpart, int chunks, const int *gate) {
  const int j = blockIdx.y, ch = blockIdx.x;
  if (gate && !gate[j]) return;
  const int n = subs[j].n_neu;
  const int per = ((n + chunks - 1) / chunks + 127) / 128 * 128;
  const int r0 = min(n, ch * per), r1 = min(n, r0 + per);
  extern __shared__ __align__(128) unsigned char smraw[];
  __half *dg = reinterpret_cast<__half *>(smraw);     // [4] tiles [row][column]
  double *sum = reinterpret_cast<double *>(dg + 4 * kDigTile);   // [warp][8][8]
  __shared__ int mx[8], G[8];                         // largest exponents and scales of the columns
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, col = tid & 7;
  const double *Wj = W + j * sw;
  for (int e = tid; e < 4 * kDigTile / 8; e += kTsThreads) reinterpret_cast<uint4 *>(dg)[e] = {0, 0, 0, 0};
  for (int e = tid; e < 8 * 64; e += kTsThreads) sum[e] = 0.0;
  if (tid < 8) mx[tid] = G[tid] = kNoExp;
  double x[4];                                        // row (tid >> 3) of each tile
  auto fetch = [&](int rb) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = rb + 32 * i + (tid >> 3);
      x[i] = r < r1 && col < p ? Wj[(long long)r * ldw + col] : 0.0;
    }
  };
  const int tile = warp >> 1, kb = warp & 1;
  unsigned acc[kDig][4];
  int cnt = 0;
#pragma unroll
  for (int l = 0; l < kDig; ++l)
#pragma unroll
    for (int e = 0; e < 4; ++e) acc[l][e] = 0u;
  auto flush = [&]() {
    const unsigned z = cnt * 0x4b400000u;
#pragma unroll
    for (int e = 0; e < 2; ++e) {                     // rows 8..15 of the block are padding
      const int r = lane >> 2, c = 2 * (lane & 3) + e;
      auto lev = [&](int l) { return (long long)(int)(l < 4 ? acc[l][e] - z : acc[l][e]); };
      const long long hi = lev(0) * 134217728 + lev(1) * 262144 + (lev(2) * 512 + lev(3)),
                      lo = lev(4) * 262144 + (lev(5) * 512 + lev(6));
      sum[warp * 64 + r * 8 + c] += parts_value(hi, lo, G[r] + G[c]);
#pragma unroll
      for (int l = 0; l < kDig; ++l) acc[l][e] = 0u;
    }
    cnt = 0;
  };
  fetch(r0);
  __syncthreads();
  for (int rb = r0; rb < r1; rb += 128) {
    int ex = max(max(exp_above(x[0]), exp_above(x[1])), max(exp_above(x[2]), exp_above(x[3])));
    ex = max(ex, __shfl_xor_sync(0xffffffffu, ex, 8));
    ex = max(ex, __shfl_xor_sync(0xffffffffu, ex, 16));
    if (lane < 8 && ex > mx[col]) atomicMax(mx + col, ex);
    __syncthreads();                                  // also: the digits have been read
    if (__syncthreads_or(mx[col] > G[col])) {
      if (cnt > 0) flush();
      __syncthreads();
      if (tid < 8 && mx[tid] > G[tid]) G[tid] = mx[tid] + 2;
      __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) ts_slice(dg + i * kDigTile, tid >> 3, col, x[i], G[col]);
    __syncthreads();
    if (rb + 128 < r1) fetch(rb + 128);               // in flight under the products
    const uint32_t t = dig_smem(dg) + tile * kDigBytes, a = t + ldsm_at(0, 16 * kb, lane);
    float S[kDig][4];
    uint32_t bw[kDig][2];
#pragma unroll
    for (int u = 0; u < kDig; ++u) {
      uint32_t w4[4];
      ts_b(w4, t + u * 2048, 0, lane);
      bw[u][0] = kb ? w4[2] : w4[0];
      bw[u][1] = kb ? w4[3] : w4[1];
    }
    level_start<4>(S);
#pragma unroll
    for (int s = 0; s < kDig; ++s) {
      uint32_t ar[4];
      ldsm4_trans(ar, a + s * 2048);
#pragma unroll
      for (int u = 0; u < kDig - s; ++u) mma_f16(S[s + u], ar, bw[u][0], bw[u][1]);
    }
#pragma unroll
    for (int l = 0; l < kDig; ++l)
#pragma unroll
      for (int e = 0; e < 4; ++e)
        acc[l][e] += l < 4 ? __float_as_uint(S[l][e]) : (unsigned)__float2int_rn(S[l][e]);
    if (++cnt == kTsFlush) flush();
  }
  if (cnt > 0) flush();
  __syncthreads();
  if (tid < p * p) {
    const int a = tid / p, b = tid - a * p;
    double v = 0.0;
#pragma unroll
    for (int w = 0; w < 8; ++w) v += sum[w * 64 + a * 8 + b];
    if (mx[a] >= 1025 || mx[b] >= 1025) v = __longlong_as_double(0x7ff8000000000000LL);
    Hpart[((long long)j * chunks + ch) * p * p + tid] = v;
  }
}

__global__ void k_tsdots_reduce(const double *Hpart, int chunks, int nout, double *H, long long hs,
                                const int *gate) {
  const int j = blockIdx.x;
  const bool skip = gate && !gate[j];
  for (int o = threadIdx.x; o < nout; o += blockDim.x) {
    double s = 0.0;
    if (!skip)
      for (int ch = 0; ch < chunks; ++ch) s += Hpart[((long long)j * chunks + ch) * nout + o];
    H[j * hs + o] = s;
  }
}

// ---- C = beta C + alpha A H ---------------------------------------------------------
// One CTA per (group of rows, subdomain, 32 columns of H).  The digits of H, one
// scale per column, stay in shared memory; rows of A are taken 32 at a time, one
// scale per row.  Eight columns of C are formed at a time: a warp multiplies 16
// rows with 32 of the columns of A and leaves two integers per entry, which the
// thread of the entry adds.
constexpr int kTsTiles = 8;                 // row tiles per CTA
template <int NCG>
__host__ __device__ constexpr int tsgemm_smem() {
  return 2 * NCG * (int)kDigBytes + NCG * 32 * 8 * 16 + (2 * 32 + 32) * 4;
}

template <int NCG>
__global__ void __launch_bounds__(kTsThreads, 2)
    k_tsgemm(const SubDesc *subs, int npad, const double *__restrict__ A, int lda, long long sa,
             int na, const double *__restrict__ H, int ldh, long long hs, double *C, int ldc,
             long long sc, int nb, double alpha, double beta, const int *gate) {
  const int j = blockIdx.y;
  if (gate && !gate[j]) return;
  extern __shared__ __align__(128) unsigned char smraw[];
  __half *dA = reinterpret_cast<__half *>(smraw);     // [NCG] tiles [row][column of A]
  __half *dH = dA + NCG * kDigTile;                   // [NCG] tiles [row of H][column]
  longlong2 *part = reinterpret_cast<longlong2 *>(dH + NCG * kDigTile);   // [NCG][32 rows][8]
  int *GR = reinterpret_cast<int *>(part + NCG * 256);    // [2][32] scales of the rows
  int *GH = GR + 2 * 32;                              // [32] scales of the columns of H
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n = subs[j].n_neu, nc0 = 32 * blockIdx.z, ncol = min(32, nb - nc0), kt = (na + 31) / 32;
  const double *Aj = A + j * sa, *Hj = H + j * hs + nc0;
  double *Cj = C + j * sc + nc0;
  if (tid < 32) GH[tid] = kNoExp;
  __syncthreads();
  for (int e = tid; e < na * 32; e += kTsThreads) {   // lane = column
    const double h = lane < ncol ? Hj[(long long)(e >> 5) * ldh + lane] : 0.0;
    atomicMax(GH + lane, exp_above(h));
  }
  __syncthreads();
  for (int e = tid; e < NCG * 1024; e += kTsThreads) {
    const int a = e >> 5;
    const double h = a < na && lane < ncol ? Hj[(long long)a * ldh + lane] : 0.0;
    ts_slice(dH + (a >> 5) * kDigTile, a & 31, lane, h, GH[lane]);
  }
  const int t0 = blockIdx.x * kTsTiles, t1 = min(npad / kTsRows, t0 + kTsTiles);
  double x[NCG][4];                                   // rows 4 warp .. + 3
  auto fetch = [&](int t) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = t * kTsRows + 4 * warp + i;
#pragma unroll
      for (int q = 0; q < NCG; ++q)
        x[q][i] = r < n && 32 * q + lane < na ? Aj[(long long)r * lda + 32 * q + lane] : 0.0;
    }
  };
  if (t0 < t1) fetch(t0);
  for (int t = t0; t < t1; ++t) {
    int *gr = GR + (t & 1) * 32;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      int ex = kNoExp;
#pragma unroll
      for (int q = 0; q < NCG; ++q) ex = max(ex, exp_above(x[q][i]));
      ex = __reduce_max_sync(0xffffffffu, ex);
      if (lane == 0) gr[4 * warp + i] = ex;
#pragma unroll
      for (int q = 0; q < NCG; ++q) ts_slice(dA + q * kDigTile, 4 * warp + i, lane, x[q][i], ex);
    }
    __syncthreads();
    if (t + 1 < t1) fetch(t + 1);                     // in flight under the products
    for (int n0 = 0; n0 < ncol; n0 += 8) {
      for (int job = warp; job < 2 * kt; job += 8) {  // 16 rows, 32 columns of A
        const int m0 = 16 * (job & 1), q = job >> 1;
        const uint32_t at = dig_smem(dA) + q * kDigBytes, bt = dig_smem(dH) + q * kDigBytes;
        float S[kDig][4];
        uint32_t bw[kDig][4];
#pragma unroll
        for (int s = 0; s < kDig; ++s) ts_b(bw[s], bt + s * 2048, n0, lane);
        level_start<2>(S);
#pragma unroll
        for (int kb = 0; kb < 2; ++kb)
#pragma unroll
          for (int s = 0; s < kDig; ++s) {
            uint32_t ar[4];
            ldsm4(ar, at + s * 2048 + ldsm_a(m0, 16 * kb, lane));
#pragma unroll
            for (int u = 0; u < kDig - s; ++u) mma_f16(S[s + u], ar, bw[u][2 * kb], bw[u][2 * kb + 1]);
          }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          long long hi, lo;
          level_parts<2>(S, e, hi, lo);
          part[q * 256 + (m0 + (lane >> 2) + 8 * (e >> 1)) * 8 + 2 * (lane & 3) + (e & 1)] = {hi, lo};
        }
      }
      __syncthreads();
      {
        const int r = tid >> 3, c = tid & 7, row = t * kTsRows + r;
        long long hi = 0, lo = 0;
        for (int q = 0; q < kt; ++q) {
          const longlong2 v = part[q * 256 + tid];
          hi += v.x;
          lo += v.y;
        }
        if (n0 + c < ncol) {
          double *cp = Cj + (long long)row * ldc + n0 + c;
          const int er = gr[r], eh = GH[n0 + c];
          double s = parts_value(hi, lo, er + eh);
          if (er >= 1025 || eh >= 1025) s = __longlong_as_double(0x7ff8000000000000LL);
          if (row < n) *cp = (beta == 0.0 ? 0.0 : beta * *cp) + alpha * s;
          else if (beta == 0.0) *cp = 0.0;
        }
      }
      if (n0 + 8 < ncol) __syncthreads();             // the partials have been read
    }
  }
}

}  // namespace

void launch_tsdots(const SubDesc *d_subs, int nsub, const double *A, int lda, long long sa,
                   int na, const double *B, int ldb, long long sb, int nb, double *Hpart,
                   int chunks, double *H, long long hs, cudaStream_t s,
                   const int *gate) {
  // One warp for each half of a 16 x 8 block of H, sixteen at most: all 32
  // columns a CTA can stage for up to 32 of A, 16 for up to 64, else eight.
  const int width = na <= 32 ? 32 : na <= 64 ? 16 : 8, groups = (nb + width - 1) / width;
  const bool small = 2 * ((na + 15) / 16) * ((std::min(nb, width) + 7) / 8) <= 8;
  auto run = [&](auto k, int warps, int sm) {
    (void)ensure_smem(k, sm);                // a failure surfaces as a launch error
    k<<<dim3(chunks, nsub, groups), 32 * warps, sm, s>>>(d_subs, A, lda, sa, na, B, ldb, sb, nb, width, Hpart, chunks, gate); GENEO_COUNT_LAUNCH();
  };
  if (A == B && lda == ldb && sa == sb && na == nb && na <= 8) {
    (void)ensure_smem(k_tsgram, kTgSmem);
    k_tsgram<<<dim3(chunks, nsub), kTsThreads, kTgSmem, s>>>(d_subs, A, lda, sa, na, Hpart, chunks, gate); GENEO_COUNT_LAUNCH();
    k_tsdots_reduce<<<nsub, 256, 0, s>>>(Hpart, chunks, na * nb, H, hs, gate); GENEO_COUNT_LAUNCH();
    return;
  }
  if (na <= 32) small ? run(k_tsdots<1, 8>, 8, tsdots_smem<1>()) : run(k_tsdots<1, 16>, 16, tsdots_smem<1>());
  else if (na <= 64) small ? run(k_tsdots<2, 8>, 8, tsdots_smem<2>()) : run(k_tsdots<2, 16>, 16, tsdots_smem<2>());
  else if (na <= 96) run(k_tsdots<3, 16>, 16, tsdots_smem<3>());
  else run(k_tsdots<4, 16>, 16, tsdots_smem<4>());
  k_tsdots_reduce<<<nsub, 256, 0, s>>>(Hpart, chunks, na * nb, H, hs, gate); GENEO_COUNT_LAUNCH();
}

void launch_tsgemm(const SubDesc *d_subs, int nsub, int npad, const double *A, int lda,
                   long long sa, int na, const double *H, int ldh, long long hs, double *C,
                   int ldc, long long sc, int nb, double alpha, double beta, cudaStream_t s,
                   const int *gate) {
  const dim3 g((npad / kTsRows + kTsTiles - 1) / kTsTiles, nsub, (nb + 31) / 32);
  auto run = [&](auto k, int sm) {
    (void)ensure_smem(k, sm);
    k<<<g, kTsThreads, sm, s>>>(d_subs, npad, A, lda, sa, na, H, ldh, hs, C, ldc, sc, nb, alpha, beta, gate); GENEO_COUNT_LAUNCH();
  };
  if (na <= 32) run(k_tsgemm<1>, tsgemm_smem<1>());
  else if (na <= 64) run(k_tsgemm<2>, tsgemm_smem<2>());
  else if (na <= 96) run(k_tsgemm<3>, tsgemm_smem<3>());
  else run(k_tsgemm<4>, tsgemm_smem<4>());
}

}  // namespace geneo
