// K2, FP64: the plain dense method's blocked Cholesky on the tensor cores.
//
// GB300 runs FP64 at 1.2 TFLOP/s, so the matrix products are taken on the FP16
// tensor cores by splitting (K. Ozaki, T. Ogita, S. Oishi, S. M. Rump,
// "Error-free transformations of matrix multiplication by using fast routines
// of matrix multiplication and its applications", Numer. Algorithms 59(1),
// 2012): every row of an operand is scaled by a power of two to 62-bit integers
// (entries within 2^-9 of the row's largest keep all their bits), written as
// eight balanced base-256 digits (|d| <= 128, exact in FP16), and the digit
// products of equal weight are summed in one FP32 accumulator:
//
//   sum_k a_k b_k = 256^14 sum_l D_l 256^-l,  D_l = sum_k sum_{i + j = l} a_ik b_jk
//
// for l = 0..7 (36 products).  The leading digit is at most 64, so |D_l| < 8 *
// 128 * 2^14 = 2^24 and the sums are exact whatever their order; the levels are
// combined in integers and rounded to FP64 once.  The other 28 digit products (l
// > 7) are left out: about 2^-57.5 of the product of the two rows' largest
// entries (rms, 128 normal entries), against 2^-53 of every partial sum in FP64
// arithmetic.  (Seven digits of 55 bits: backward errors 10 to 40% above the FP64
// products'.)  That is a bound by rows, not by entries: an entry whose terms are
// far below its rows' largest has its sum taken in FP64 where L is the result
// (entries; a solve refines its weighting, for which the bound by rows is
// enough), so that |Z - L L^T| stays a few units of |L| |L^T| entry by entry.  n = 300, six clouds
// in R^6 to R^20, t = 1 to 6: at most 2.3e-15 of |L| |L^T|, FP64 products 8.0e-15
// (by digits alone 0.03 at worst).
//
// Per tile column K: the diagonal tile (FP64, k_potrf_f64), the digits of
// inv(L_KK) and of the panel's tiles, the panel solve L_IK = A_IK inv(L_KK)^T,
// the digits of the solved panel and the trailing update C_IJ -= L_IK L_JK^T.
// n = 5001: 123 ms with FP64 products throughout, 15.8 ms this way (8.5 of
// them the 40 diagonal tiles); backward error 5e-16 -> 0.6e-16.  The sums in FP64
// cost nothing where the entries of Z are within a few decades; n = 4000: 11.4
// ms, N(0, I_10) at t = 6 19.8, N(0, I_6) at t = 6 36.5 (a third of the entries;
// FP64 products 87.9).
#include <cuda_fp16.h>

#include <algorithm>

#include "mag_internal.cuh"
#include "mag_tc.cuh"

namespace mag {

namespace {

// ---------------------------------------------------------- diagonal tile
// The elimination of [A; I] of k_potrf.cu in FP64, in four panels of 32
// columns, four columns at a time, by a cluster of eight CTAs: each holds one
// block of 32 rows, A's four (becoming L) and those of W = inv(L)^T.  Per panel
// the CTA of the diagonal block factors it and hands it to the others' shared
// memory, the blocks below it (and W's up to it) are solved, A's
// go round in the same way, and every CTA updates its remaining columns.  Bound:
// the FP64 pipe, 16 SM cycles a warp operation and 64 on one of its quarters:
// the panels' chain of pivots (about 30 us a panel), then the trailing updates
// (98,000 cycles on the busiest of eight CTAs, 555,000 on one).  214 us a tile;
// one CTA took 343, an elimination column by column about 1,000.
constexpr int PB = 32;
constexpr int NPB = TILE / PB;
constexpr int LDR = TILE + 2;
constexpr int LDW = PB + 2;
constexpr int P64_THREADS = 512;
constexpr int P64_CTAS = 2 * NPB;

struct Potrf64Smem {
  double R[PB * LDR];         // the CTA's rows
  double D[PB * LDW];         // the panel's diagonal block of L
  double X[NPB][PB * LDW];    // the panel's blocks of L below it, by row block
  double rinv[PB];            // 1 / L[c][c] of the panel
};

__device__ __forceinline__ void st_remote_f64(uint32_t cluster_addr, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(cluster_addr), "d"(v) : "memory");
}

// s = sqrt(p) and its reciprocal, p > 0: the FP32 seed, two Newton steps, s
// from p r by its exact residual, then r as the reciprocal of that s (both
// within 0.51 units and consistent: the column is scaled by 1 / L_jj).
__device__ __forceinline__ double rsqrt64(double p, double* sq) {
  // p scaled to FP32's range by an even power of two
  const int ex = (__double2hiint(p) >> 20) - 1023;
  const int h = ex >> 1;
  const double ps = __hiloint2double(__double2hiint(p) - h * (1 << 21), __double2loint(p));  // in [1, 4)
  double r = (double)rsqrtf((float)ps);
  const double hp = 0.5 * ps;
#pragma unroll
  for (int i = 0; i < 2; ++i) r = fma(r, fma(-hp * r, r, 0.5), r);
  double s = ps * r;
  s = fma(0.5 * r, fma(-s, s, ps), s);
  r = fma(r, fma(-s, r, 1.0), r);
  *sq = __hiloint2double(__double2hiint(s) + h * (1 << 20), __double2loint(s));
  return __hiloint2double(__double2hiint(r) - h * (1 << 20), __double2loint(r));
}

struct Pivot64 {
  double r0, r1, r2, r3, s0, s1, s2, s3, l10, l20, l30, l21, l31, l32;
  int bad;
};

__device__ __forceinline__ void pivot_factor64(const double* a, int j, Pivot64& q) {
  const unsigned full = 0xffffffffu;
  const double d00 = __shfl_sync(full, a[0], j), d10 = __shfl_sync(full, a[0], j + 1);
  const double d20 = __shfl_sync(full, a[0], j + 2), d30 = __shfl_sync(full, a[0], j + 3);
  const double d11 = __shfl_sync(full, a[1], j + 1), d21 = __shfl_sync(full, a[1], j + 2);
  const double d31 = __shfl_sync(full, a[1], j + 3), d22 = __shfl_sync(full, a[2], j + 2);
  const double d32 = __shfl_sync(full, a[2], j + 3), d33 = __shfl_sync(full, a[3], j + 3);
  // a pivot that is not positive (or below FP64's normal range) is reported
  // and replaced by 1, so that the kernel finishes on finite values
  constexpr double kMin = 2.2250738585072014e-308;
  const bool b0 = !(d00 >= kMin);
  q.r0 = rsqrt64(b0 ? 1.0 : d00, &q.s0);
  q.l10 = d10 * q.r0, q.l20 = d20 * q.r0, q.l30 = d30 * q.r0;
  const double p1 = fma(-q.l10, q.l10, d11);
  const bool b1 = !(p1 >= kMin);
  q.r1 = rsqrt64(b1 ? 1.0 : p1, &q.s1);
  q.l21 = fma(-q.l20, q.l10, d21) * q.r1, q.l31 = fma(-q.l30, q.l10, d31) * q.r1;
  const double p2 = fma(-q.l21, q.l21, fma(-q.l20, q.l20, d22));
  const bool b2 = !(p2 >= kMin);
  q.r2 = rsqrt64(b2 ? 1.0 : p2, &q.s2);
  q.l32 = fma(-q.l31, q.l21, fma(-q.l30, q.l20, d32)) * q.r2;
  const double p3 = fma(-q.l32, q.l32, fma(-q.l31, q.l31, fma(-q.l30, q.l30, d33)));
  const bool b3 = !(p3 >= kMin);
  q.r3 = rsqrt64(b3 ? 1.0 : p3, &q.s3);
  q.bad = (int)b0 | (int)b1 << 1 | (int)b2 << 2 | (int)b3 << 3;
}

// A panel's steps for a block of 32 rows (DIAG: the diagonal block's) by four
// warps, a row per lane: warp w owns column groups w and w + 4 of the eight.
// The owner of a group scales its four columns and writes them to the row; the
// others follow after a barrier of the four.  The owner of the next group
// updates that one first and leaves its other until it has written.  (An SM
// quarter issues a warp's FP64 operation in 64 cycles: a warp alone took 20 us
// for its 528, 28 with the pivots.)  own: this lane's 32 entries, Ld: the panel's
// diagonal block of L (row stride ld), rinv its reciprocals.
template <bool DIAG>
__device__ __forceinline__ void panel_rows64(double* own, const double* Ld, int ld, double* rinv, int w, int lane,
                                             int row, DevStatus* st) {
  double a[2][4];
#pragma unroll
  for (int s = 0; s < 2; ++s)
#pragma unroll
    for (int c = 0; c < 4; ++c) a[s][c] = own[16 * s + 4 * w + c];
  // slot s (group w + 4 s) -= group g's columns
  auto update = [&](double(&v)[4], int s, int g) {
    const int j = 4 * g;
    const double2 x01 = *reinterpret_cast<const double2*>(own + j), x23 = *reinterpret_cast<const double2*>(own + j + 2);
    const double* Lq = Ld + (16 * s + 4 * w) * ld + j;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const double2 v01 = *reinterpret_cast<const double2*>(Lq + c * ld);
      const double2 v23 = *reinterpret_cast<const double2*>(Lq + c * ld + 2);
      v[c] = fma(-x23.y, v23.y, fma(-x23.x, v23.x, fma(-x01.y, v01.y, fma(-x01.x, v01.x, v[c]))));
    }
  };
  // group g = w + 4 s: its columns
  auto eliminate = [&](double(&v)[4], int g) {
    const int j = 4 * g;
    Pivot64 q;
    q.bad = 0;
    if (DIAG) {
      pivot_factor64(v, j, q);
    } else {
      q.r0 = rinv[j], q.r1 = rinv[j + 1], q.r2 = rinv[j + 2], q.r3 = rinv[j + 3];
      const double* r1 = Ld + (j + 1) * ld + j;
      q.l10 = r1[0];
      q.l20 = r1[ld], q.l21 = r1[ld + 1];
      q.l30 = r1[2 * ld], q.l31 = r1[2 * ld + 1], q.l32 = r1[2 * ld + 2];
    }
    double x0 = v[0] * q.r0;
    double x1 = fma(-x0, q.l10, v[1]) * q.r1;
    double x2 = fma(-x1, q.l21, fma(-x0, q.l20, v[2])) * q.r2;
    double x3 = fma(-x2, q.l32, fma(-x1, q.l31, fma(-x0, q.l30, v[3]))) * q.r3;
    if (DIAG) {
      x0 = lane < j ? 0.0 : (lane == j ? q.s0 : x0);
      x1 = lane < j + 1 ? 0.0 : (lane == j + 1 ? q.s1 : x1);
      x2 = lane < j + 2 ? 0.0 : (lane == j + 2 ? q.s2 : x2);
      x3 = lane < j + 3 ? 0.0 : (lane == j + 3 ? q.s3 : x3);
      if (lane == 0) {
        rinv[j] = q.r0, rinv[j + 1] = q.r1, rinv[j + 2] = q.r2, rinv[j + 3] = q.r3;
        if (q.bad) {
          atomicOr(&st->flags, ST_NOTPD);
          atomicMin(&st->notpd_index, row + j + __ffs(q.bad));
        }
      }
    }
    own[j] = x0, own[j + 1] = x1, own[j + 2] = x2, own[j + 3] = x3;
  };
  auto meet = [] { asm volatile("bar.sync 1, 128;" ::: "memory"); };
  if (w == 0) eliminate(a[0], 0);
  meet();
#pragma unroll 1
  for (int g = 0; g < PB / 4 - 1; ++g) {
    const int next = g + 1;
    if (w == (next & 3)) {
      if (next < 4) {
        update(a[0], 0, g);
        eliminate(a[0], next);
      } else {
        update(a[1], 1, g);
        eliminate(a[1], next);
      }
    }
    if (w > g && w != next) update(a[0], 0, g);
    if (w + 4 > g && w + 4 != next) update(a[1], 1, g);
    meet();
  }
}

// 8 x 32 outputs: C -= P Q^T, K = 32 (P, C: rows of R; Q: a block of X).  The
// sums start from C: the partial sums shrink towards the Schur complement, where
// a sum taken apart rises to C's size and cancels (backward error 1.9e-16 for
// 0.5e-16 at 128 points of the unit cube).
__device__ __forceinline__ void trailing_job64(const double* P, const double* Q, double* C, int lane) {
  const double* p = P + (lane >> 3) * LDR;
  const double* q = Q + (lane & 7) * LDW;
  double* c = C + (lane >> 3) * LDR + (lane & 7);
  double acc[2][4];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = c[4 * i * LDR + 8 * j];
#pragma unroll 4
  for (int k = 0; k < PB; ++k) {
    double b[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) b[j] = q[8 * j * LDW + k];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const double a = -p[4 * i * LDR + k];
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = fma(a, b[j], acc[i][j]);
    }
  }
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) c[4 * i * LDR + 8 * j] = acc[i][j];
}

// The CTA's block of 32 x 32 (row stride LDR) into dst of every CTA of the cluster.
__device__ __forceinline__ void hand_round(const double* src, double* dst, int tid) {
  const uint32_t d = smem_u32(dst);
#pragma unroll
  for (int i = 0; i < PB * PB / P64_THREADS; ++i) {
    const int e = tid + i * P64_THREADS, r = e / PB, c = e % PB;
    const double v = src[r * LDR + c];
#pragma unroll
    for (int k = 0; k < P64_CTAS; ++k) st_remote_f64(map_to_rank(d + (r * LDW + c) * 8, k), v);
  }
}

__global__ void __cluster_dims__(P64_CTAS, 1, 1) __launch_bounds__(P64_THREADS, 1)
    k_potrf_f64(double* __restrict__ Z, double* __restrict__ Dinv, double* __restrict__ DinvT, int64_t K,
                DevStatus* st) {
  extern __shared__ __align__(16) unsigned char p64_smem[];
  Potrf64Smem& S = *reinterpret_cast<Potrf64Smem*>(p64_smem);
  const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
  const int rank = (int)blockIdx.x, blk = rank & (NPB - 1);
  const bool isW = rank >= NPB;
  // set by earlier kernels (this one sets none before the first cluster barrier): uniform over the cluster
  if (*(volatile int*)&st->flags & (ST_NOTPD | ST_NONFINITE | ST_DUPLICATE | ST_TIMEOUT)) return;
  double* tile = Z + tri_index(K, K) * TILE_ELEMS;
#pragma unroll
  for (int i = 0; i < PB * TILE / 2 / P64_THREADS; ++i) {
    const int e = tid + i * P64_THREADS, r = e >> 6, c = (e & 63) * 2;
    double2 v = make_double2(0.0, 0.0);
    if (isW) {
      if (c == blk * PB + (r & ~1)) (r & 1 ? v.y : v.x) = 1.0;
    } else if (c < (blk + 1) * PB) {
      v = *reinterpret_cast<const double2*>(tile + (blk * PB + r) * TILE + c);
    }
    *reinterpret_cast<double2*>(S.R + r * LDR + c) = v;
  }
  cluster_sync_all();
#pragma unroll 1
  for (int kb = 0; kb < NPB; ++kb) {
    const int o = kb * PB;
    if (rank == kb) {
      if (w < 4) panel_rows64<true>(S.R + lane * LDR + o, S.R + o, LDR, S.rinv, w, lane, (int)(K * TILE + o), st);
      __syncthreads();
      hand_round(S.R + o, S.D, tid);
      if (tid < PB) {
        const double v = S.rinv[tid];
        for (int k = 0; k < P64_CTAS; ++k)
          if (k != rank) st_remote_f64(map_to_rank(smem_u32(&S.rinv[tid]), k), v);
      }
    }
    cluster_sync_all();
    const bool mine = isW ? blk <= kb : blk > kb;
    if (mine && w < 4) panel_rows64<false>(S.R + lane * LDR + o, S.D, LDW, S.rinv, w, lane, 0, st);
    __syncthreads();
    if (mine && !isW) hand_round(S.R + o, S.X[blk], tid);
    cluster_sync_all();
    if (mine) {
      // A's blocks up to the diagonal, W's all: a quarter (8 rows) of a product a job
      const int last = isW ? NPB - 1 : blk;
      for (int job = w; job < 4 * (last - kb); job += P64_THREADS / 32) {
        const int jb = kb + 1 + (job >> 2);
        double* row = S.R + 8 * (job & 3) * LDR;
        trailing_job64(row + o, S.X[jb], row + jb * PB, lane);
      }
    }
    __syncthreads();
  }
  if (!isW) {
    for (int e = tid; e < PB * TILE; e += P64_THREADS) {
      const int r = e >> 7, c = e & 127;
      tile[(blk * PB + r) * TILE + c] = c <= blk * PB + r ? S.R[r * LDR + c] : 0.0;
    }
    return;
  }
  // W[c][r] = inv(L)[r][c], c = blk PB ..
  double* Y = Dinv + K * TILE_ELEMS + blk * PB;
  double* YT = DinvT + K * TILE_ELEMS + blk * PB * TILE;
  for (int e = tid; e < PB * TILE; e += P64_THREADS) {
    const int i = e >> 7, r = e & 127;
    YT[e] = r >= blk * PB + i ? S.R[i * LDR + r] : 0.0;
  }
  for (int e = tid; e < PB * TILE; e += P64_THREADS) {
    const int r = e >> 5, i = e & 31;
    Y[r * TILE + i] = r >= blk * PB + i ? S.R[i * LDR + r] : 0.0;
  }
}

// ----------------------------------------------------------------- digits
constexpr int NDIG = 8;
constexpr int64_t CHUNK_BYTES = 128 * 128;                     // 128 rows x 64 FP16 columns
constexpr int64_t DIGIT_BYTES = 2 * NDIG * CHUNK_BYTES;        // a tile's digits: [K chunk][digit][128 rows]
constexpr int64_t DIGIT_STRIDE = DIGIT_BYTES + 1024;           // then 128 row exponents and 128 row weights

// Digits of the FP64 tiles of column K: slot 0 from `first` (inv(L_KK) without
// its diagonal, when given), the following slots from tiles (I, K), I = K + 1
// ....  Row r of a tile is x = X 2^(e_r - 62), |X| < 2^62, X = sum_i d_i
// 256^(7 - i).  A row whose largest entry is below 2^-450 counts as zero.  A
// row's weight is the exponent that its errors are judged by (k_oz_gemm): e_r,
// nothing for a row of zeros, 64 more where the digits leave out the row.
constexpr int WEIGHT_NONE = -16384;
__global__ void __launch_bounds__(256) k_digits(const double* __restrict__ first, const double* __restrict__ Z,
                                                int64_t K, unsigned char* __restrict__ out, const DevStatus* st) {
  if (st->flags & (ST_NOTPD | ST_NONFINITE | ST_DUPLICATE | ST_TIMEOUT)) return;
  const int64_t slot = blockIdx.x, I = K + 1 + slot - (first ? 1 : 0);
  const double* src = first && slot == 0 ? first : Z + tri_index(I, K) * TILE_ELEMS;
  unsigned char* dst = out + slot * DIGIT_STRIDE;
  int* exps = reinterpret_cast<int*>(dst + DIGIT_BYTES);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll 2
  for (int r = warp; r < TILE; r += 8) {
    const double2 v01 = *reinterpret_cast<const double2*>(src + r * TILE + 4 * lane);
    const double2 v23 = *reinterpret_cast<const double2*>(src + r * TILE + 4 * lane + 2);
    unsigned long long b[4] = {
        (unsigned long long)__double_as_longlong(v01.x), (unsigned long long)__double_as_longlong(v01.y),
        (unsigned long long)__double_as_longlong(v23.x), (unsigned long long)__double_as_longlong(v23.y)};
    unsigned mx = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (first && slot == 0 && 4 * lane + q == r) b[q] = 0;
      mx = max(mx, (unsigned)(b[q] >> 52) & 0x7ffu);
    }
    mx = __reduce_max_sync(0xffffffffu, mx);
    const bool zero = mx < 1023 - 450;
    if (lane == 0) {
      exps[r] = zero ? 0 : (int)mx - 1022;
      exps[TILE + r] = mx == 0 ? WEIGHT_NONE : (int)mx - 1022 + (zero ? 64 : 0);
    }
    __half d[NDIG][4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int ex = (int)(b[q] >> 52) & 0x7ff, s = (int)mx - ex;
      long long X = 0;
      if (!zero && ex > 0 && s < 63) {
        X = (long long)(((b[q] & 0xfffffffffffffull) | 0x10000000000000ull) << 9);
        if (s > 0) X = (X + (1ll << (s - 1))) >> s;
        if (b[q] >> 63) X = -X;
      }
#pragma unroll
      for (int i = NDIG - 1; i > 0; --i) {
        const int g = (int)((unsigned)(X + 128) & 255u) - 128;
        X = (X - g) >> 8;
        d[i][q] = __int2half_rn(g);
      }
      d[0][q] = __int2half_rn((int)X);
    }
    const int chunk = lane >> 4, unit = (lane & 15) >> 1;
    unsigned char* p = dst + chunk * NDIG * CHUNK_BYTES + swizzled_unit(r, unit) + (lane & 1) * 8;
#pragma unroll
    for (int i = 0; i < NDIG; ++i) {
      uint2 u;
      const __half2 lo = __halves2half2(d[i][0], d[i][1]), hi = __halves2half2(d[i][2], d[i][3]);
      u.x = *reinterpret_cast<const uint32_t*>(&lo);
      u.y = *reinterpret_cast<const uint32_t*>(&hi);
      *reinterpret_cast<uint2*>(p + i * CHUNK_BYTES) = u;
    }
  }
}

// The least exponent among the entries of each half tile of Z (64 columns),
// rows and columns of the padding left out.
__global__ void __launch_bounds__(256) k_least_exponent(const double* __restrict__ Z, int64_t n, int* __restrict__ least) {
  __shared__ int part[8];
  const int64_t q = blockIdx.x >> 1;
  const int h = blockIdx.x & 1, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int64_t I, J;
  tri_coords(q, &I, &J);
  const int64_t col = J * TILE + 64 * h + 2 * lane;
  int e = 0x7ff;
#pragma unroll 4
  for (int r = warp; r < TILE; r += 8) {
    const double2 z = *reinterpret_cast<const double2*>(Z + q * TILE_ELEMS + r * TILE + 64 * h + 2 * lane);
    if (I * TILE + r < n) {
      if (col < n) e = min(e, (__double2hiint(z.x) >> 20) & 0x7ff);
      if (col + 1 < n) e = min(e, (__double2hiint(z.y) >> 20) & 0x7ff);
    }
  }
  e = __reduce_min_sync(0xffffffffu, e);
  if (lane == 0) part[warp] = e;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 1; k < 8; ++k) e = min(e, part[k]);
    least[blockIdx.x] = e - 1023;
  }
}

// ---------------------------------------------------------------- products
// 128 x 64 outputs (half h of a tile) of A B^T from the digits, K = 128 in two
// chunks of 64 columns: 128 KB of A's digits and 64 KB of B's in shared memory
// at a time, the eight levels in 8 x 64 TMEM columns.  ASSIGN: tile (I, K) of
// the panel, A = its own digits (slot 1 + i), B = inv(L_KK) without its
// diagonal (slot 0), whose part is one FP64 product an entry; else the trailing
// update of tile (I, J), A and B the panel's digits.
//
// What the digits drop is a fraction of the rows' largest entries max_a max_b,
// about 2^-57, while the factor's error is to stay a fraction of |L| |L^T| entry
// by entry, which is at least Z_ij.  Rows whose entries span many decades
// (points in few dimensions at large t) leave some entries below: where neither
// the half tile's least Z_ij nor |C_ij| (in the panel |a_ij inv_jj|) reaches
// 2^-8 max_a max_b, an entry's sum is taken in FP64, a warp each.  The test runs
// beside the products.  The panel's halves read all of a row of A there, so the
// two CTAs of a tile are then a cluster and write once both have read.
constexpr int OZ_THREADS = 256;
constexpr uint32_t OZ_TMEM = 512;
constexpr int OZ_SMEM = NDIG * (128 * 128 + 64 * 128);
constexpr int OZ_LD = 66;
constexpr int OZ_MARGIN = 8;

__device__ __forceinline__ void mma_f16_128x64(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t accumulate) {
  constexpr uint32_t idesc = (1u << 4) | ((uint32_t)(64 >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float* v) {
  uint32_t r[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ int exponent_of(double v) { return ((__double2hiint(v) >> 20) & 0x7ff) - 1023; }

// least: k_least_exponent's (null: every entry by digits); inv: inv(L_KK) (ASSIGN)
template <bool ASSIGN>
__global__ void __launch_bounds__(OZ_THREADS, 1)
    k_oz_gemm(double* __restrict__ Z, int64_t N, int64_t K, const unsigned char* __restrict__ digits,
              const int* __restrict__ least, const double* __restrict__ inv, DevStatus* st, uint64_t timeout_ns) {
  extern __shared__ __align__(1024) unsigned char oz_raw[];
  unsigned char* smem = (unsigned char*)(((uintptr_t)oz_raw + 1023) & ~(uintptr_t)1023);
  __shared__ __align__(8) uint64_t full_bar, done_bar[2];  // done_bar[c]: the products of chunk c
  __shared__ uint32_t tmem_base_sh;
  __shared__ int abort_flag;
  __shared__ int ea[128], eb[64], wa[128], wb[64];  // row exponents and weights
  __shared__ uint2 low[128];                        // a row's columns 2 l (x) and 2 l + 1 (y) that need FP64 sums
  __shared__ int skip, any_low;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) skip = (*(volatile int*)&st->flags & (ST_NOTPD | ST_NONFINITE | ST_DUPLICATE | ST_TIMEOUT)) != 0;
  __syncthreads();
  if (skip) {  // uniform across the CTA
    if (ASSIGN && least) cluster_sync_all();  // the other half's CTA may have gone on
    return;
  }
  const int h = blockIdx.x & 1;
  int64_t I, J;
  const unsigned char *da, *db;
  if (ASSIGN) {
    I = K + 1 + (blockIdx.x >> 1), J = K;
    da = digits + (1 + (int64_t)(blockIdx.x >> 1)) * DIGIT_STRIDE;
    db = digits;
  } else {
    int64_t i, j;
    tri_coords((int64_t)(blockIdx.x >> 1), &i, &j);
    I = K + 1 + i, J = K + 1 + j;
    da = digits + i * DIGIT_STRIDE;
    db = digits + j * DIGIT_STRIDE;
  }
  if (tid == 0) {
    abort_flag = 0;
    any_low = 0;
    mbar_init(&full_bar, 1);
    mbar_init(&done_bar[0], 1);
    mbar_init(&done_bar[1], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_sh)),
                 "r"(OZ_TMEM)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  const int* xa = reinterpret_cast<const int*>(da + DIGIT_BYTES);
  const int* xb = reinterpret_cast<const int*>(db + DIGIT_BYTES) + 64 * h;
  if (tid < 128)
    ea[tid] = xa[tid], wa[tid] = xa[TILE + tid], low[tid] = make_uint2(0, 0);
  else if (tid < 192)
    eb[tid - 128] = xb[tid - 128], wb[tid - 128] = xb[TILE + tid - 128];
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base_sh;
  const uint64_t deadline = globaltimer() + timeout_ns;
  const int64_t tile = tri_index(I, J);
  double* C = Z + tile * TILE_ELEMS + 64 * h;
  // the inverse's diagonal for this lane's columns 2 lane, 2 lane + 1
  double2 iv = make_double2(1.0, 1.0);
  if (ASSIGN) iv = make_double2(inv[(64 * h + 2 * lane) * (TILE + 1)], inv[(64 * h + 2 * lane + 1) * (TILE + 1)]);
  if (tid == 0) {
    bool ok = true;
    for (int c = 0; c < 2 && ok; ++c) {
      if (c > 0) ok = mbar_wait(&done_bar[0], 0, &abort_flag, deadline);  // chunk 0's operands have been read
      if (!ok) break;
      mbar_expect_tx(&full_bar, OZ_SMEM);
      for (int i = 0; i < NDIG; ++i) {
        bulk_load(smem + i * CHUNK_BYTES, da + (c * NDIG + i) * CHUNK_BYTES, CHUNK_BYTES, &full_bar);
        bulk_load(smem + NDIG * CHUNK_BYTES + i * 8192, db + (c * NDIG + i) * CHUNK_BYTES + h * 8192, 8192, &full_bar);
      }
      ok = mbar_wait(&full_bar, c, &abort_flag, deadline);
      if (!ok) {
        const uint64_t dl = globaltimer() + 200000000ull;  // let the loads land before the CTA ends
        while (!mbar_try_wait(&full_bar, c) && globaltimer() < dl) {
        }
        break;
      }
      tc_fence_after();
      for (int l = 0; l < NDIG; ++l)
        for (int i = 0; i <= l; ++i) {
          const uint32_t sa = smem_u32(smem + i * CHUNK_BYTES);
          const uint32_t sb = smem_u32(smem + NDIG * CHUNK_BYTES + (l - i) * 8192);
#pragma unroll
          for (int k = 0; k < 4; ++k)
            mma_f16_128x64(tmem + l * 64, smem_desc<128>(sa + 32 * k), smem_desc<128>(sb + 32 * k),
                           (c | i | k) != 0);
        }
      mma_commit(&done_bar[c]);
    }
  } else if (warp > 0 && least) {
    const int b0 = wb[2 * lane], b1 = wb[2 * lane + 1], bmax = __reduce_max_sync(0xffffffffu, max(b0, b1));
    const int zmin = least[2 * tile + h] + OZ_MARGIN;
    for (int r = warp - 1; r < TILE; r += OZ_THREADS / 32 - 1) {
      const int w = wa[r];
      if (w + bmax <= zmin) continue;  // uniform
      const double2 c = *reinterpret_cast<const double2*>(C + r * TILE + 2 * lane);
      const unsigned x = __ballot_sync(0xffffffffu, w + b0 > max(zmin, exponent_of(c.x) + exponent_of(iv.x) + OZ_MARGIN));
      const unsigned y = __ballot_sync(0xffffffffu, w + b1 > max(zmin, exponent_of(c.y) + exponent_of(iv.y) + OZ_MARGIN));
      if (lane == 0 && (x | y)) low[r] = make_uint2(x, y), *(volatile int*)&any_low = 1;
    }
  }
  __syncwarp();
  double2 old[16];  // rows warp + 8 i: on their way while the products run
#pragma unroll
  for (int i = 0; i < 16; ++i) old[i] = *reinterpret_cast<const double2*>(C + (warp + 8 * i) * TILE + 2 * lane);
  const bool waited = mbar_wait(&done_bar[1], 0, &abort_flag, deadline);
  const bool fine = __syncthreads_and(waited ? 1 : 0) != 0;  // one decision for the whole CTA
  tc_fence_after();
  double* stage = reinterpret_cast<double*>(smem);  // [128][OZ_LD], once the MMAs have read the operands
  if (fine) {
    const int r = 32 * (warp & 3) + lane, c0 = 32 * (warp >> 2);
    const uint32_t base = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)c0;
    const int er = ea[r] - 36 + 1023;
#pragma unroll 1
    for (int g = 0; g < 4; ++g) {
      float v[NDIG][8];
#pragma unroll
      for (int l = 0; l < NDIG; ++l) tmem_ld8(base + l * 64 + 8 * g, v[l]);
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
      for (int l = 0; l < NDIG; ++l)  // no use of the values moves above the wait
        asm volatile("" : "+f"(v[l][0]), "+f"(v[l][1]), "+f"(v[l][2]), "+f"(v[l][3]), "+f"(v[l][4]), "+f"(v[l][5]),
                          "+f"(v[l][6]), "+f"(v[l][7]));
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        // sum_l D_l 256^(7 - l) = t 2^32 + f, |t| < 2^46
        const long long lo = (long long)__float2int_rn(v[4][q]) * 16777216 +
                             ((long long)__float2int_rn(v[5][q]) * 65536 +
                              ((long long)__float2int_rn(v[6][q]) * 256 + __float2int_rn(v[7][q])));
        const long long t = (long long)__float2int_rn(v[0][q]) * 16777216 +
                            ((long long)__float2int_rn(v[1][q]) * 65536 +
                             ((long long)__float2int_rn(v[2][q]) * 256 + __float2int_rn(v[3][q]))) +
                            (lo >> 32);
        // the leading 62 bits or more: left-aligned by k <= 32
        const int k = min(__clzll((long long)(t ^ (t >> 63))) - 1, 32);
        const long long X = (long long)(((unsigned long long)t << k) | ((unsigned long long)(unsigned)lo << k >> 32));
        const int c = c0 + 8 * g + q;
        const int sc = er + eb[c] - k;  // positive: rows below 2^-450 are zero
        stage[r * OZ_LD + c] = __ll2double_rn(X) * __hiloint2double(sc << 20, 0);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (fine && any_low) {  // uniform
    const double* A = Z + tri_index(I, K) * TILE_ELEMS;
    const double* B = (ASSIGN ? inv : Z + tri_index(J, K) * TILE_ELEMS) + 64 * h * TILE;
    for (int r = warp; r < TILE; r += OZ_THREADS / 32) {
      const uint2 m = low[r];
      if (!(m.x | m.y)) continue;  // uniform
      const double2 a0 = reinterpret_cast<const double2*>(A + r * TILE)[lane];
      const double2 a1 = reinterpret_cast<const double2*>(A + r * TILE)[lane + 32];
      auto part = [&](int c) {  // this lane's columns 2 lane, 2 lane + 1 and the same beyond 64
        double2 b0 = reinterpret_cast<const double2*>(B + c * TILE)[lane];
        double2 b1 = reinterpret_cast<const double2*>(B + c * TILE)[lane + 32];
        if (ASSIGN) {  // the columns before the diagonal
          const int k = 64 * h + c - 2 * lane;
          b0 = make_double2(k > 0 ? b0.x : 0.0, k > 1 ? b0.y : 0.0);
          b1 = make_double2(k > 64 ? b1.x : 0.0, k > 65 ? b1.y : 0.0);
        }
        return fma(a1.y, b1.y, fma(a1.x, b1.x, fma(a0.y, b0.y, a0.x * b0.x)));
      };
#pragma unroll 1
      for (int p = 0; p < 2; ++p) {
        unsigned set = p ? m.y : m.x;
        auto next = [&] {
          const int c = 2 * (__ffs((int)set) - 1) + p;
          set &= set - 1;
          return c;
        };
        // four sums together share the reduction's last levels: 5.5 operations
        // of the FP64 pipe a sum, 9 apart
#pragma unroll 1
        while (__popc(set) >= 4) {
          const int c0 = next(), c1 = next(), c2 = next(), c3 = next();
          const double s0 = part(c0), s1 = part(c1), s2 = part(c2), s3 = part(c3);
          const bool up = (lane & 16) != 0, odd = (lane & 8) != 0;
          double u0 = (up ? s2 : s0) + __shfl_xor_sync(0xffffffffu, up ? s0 : s2, 16);
          double u1 = (up ? s3 : s1) + __shfl_xor_sync(0xffffffffu, up ? s1 : s3, 16);
          double u = (odd ? u1 : u0) + __shfl_xor_sync(0xffffffffu, odd ? u0 : u1, 8);
#pragma unroll
          for (int o = 4; o > 0; o >>= 1) u += __shfl_xor_sync(0xffffffffu, u, o);
          if ((lane & 7) == 0) stage[r * OZ_LD + (up ? (odd ? c3 : c2) : (odd ? c1 : c0))] = u;
        }
#pragma unroll 1
        while (set) {
          const int c = next();
          double u = part(c);
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) u += __shfl_xor_sync(0xffffffffu, u, o);
          if (lane == 0) stage[r * OZ_LD + c] = u;
        }
      }
      __syncwarp();  // the row's entries are read below by this warp
    }
  }
  if (ASSIGN && least) cluster_sync_all();
  if (fine) {
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const int r = warp + 8 * i;
      const double2 v = *reinterpret_cast<const double2*>(stage + r * OZ_LD + 2 * lane);
      double2 c = old[i];
      if (ASSIGN)
        c.x = fma(c.x, iv.x, v.x), c.y = fma(c.y, iv.y, v.y);
      else
        c.x -= v.x, c.y -= v.y;
      *reinterpret_cast<double2*>(C + r * TILE + 2 * lane) = c;
    }
  }
  if (tid == 0 && abort_flag) atomicOr(&st->flags, ST_TIMEOUT);
  tc_fence_after();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(OZ_TMEM) : "memory");
}

constexpr uint64_t kOzTimeout = 10000000000ull;

}  // namespace

// the digits of a panel and of an inverse, then the half tiles' least exponents
size_t factor64_scratch_bytes(int64_t N) {
  return (size_t)(N + 1) * DIGIT_STRIDE + 2 * (size_t)num_lower_tiles(N) * sizeof(int);
}
static int* least_of(void* scratch, int64_t N) {
  return reinterpret_cast<int*>(static_cast<unsigned char*>(scratch) + (N + 1) * DIGIT_STRIDE);
}

cudaError_t launch_factor64_begin(const double* Z, int64_t n, int64_t N, void* scratch, cudaStream_t s) {
  const int64_t tiles = num_lower_tiles(N);
  if (2 * tiles > 0x7fffffffLL) return cudaErrorInvalidValue;
  k_least_exponent<<<(unsigned)(2 * tiles), 256, 0, s>>>(Z, n, least_of(scratch, N));
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_potrf_f64(double* Z, double* Dinv, double* DinvT, int64_t K, DevStatus* st, cudaStream_t s) {
  cudaError_t e = cudaFuncSetAttribute(k_potrf_f64, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)sizeof(Potrf64Smem));
  if (e != cudaSuccess) return e;
  k_potrf_f64<<<P64_CTAS, P64_THREADS, sizeof(Potrf64Smem), s>>>(Z, Dinv, DinvT, K, st);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_factor64_panel(double* Z, const double* Dinv, int64_t K, int64_t N, void* scratch, bool entries,
                                  DevStatus* st, cudaStream_t s) {
  unsigned char* dg = static_cast<unsigned char*>(scratch);
  cudaError_t e;
  const int64_t below = N - K - 1;
  if (below <= 0) return cudaSuccess;
  const int smem = OZ_SMEM + 1024;
  e = cudaFuncSetAttribute(k_oz_gemm<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  k_digits<<<(unsigned)(below + 1), 256, 0, s>>>(Dinv + K * TILE_ELEMS, Z, K, dg, st);
  note_launch();
  cudaLaunchConfig_t c{};
  c.gridDim = dim3((unsigned)(2 * below)), c.blockDim = dim3(OZ_THREADS), c.dynamicSmemBytes = smem, c.stream = s;
  cudaLaunchAttribute pair[1];
  pair[0].id = cudaLaunchAttributeClusterDimension;
  pair[0].val.clusterDim.x = 2, pair[0].val.clusterDim.y = 1, pair[0].val.clusterDim.z = 1;
  c.attrs = pair, c.numAttrs = entries ? 1 : 0;
  e = cudaLaunchKernelEx(&c, k_oz_gemm<true>, Z, N, K, (const unsigned char*)dg,
                         entries ? (const int*)least_of(scratch, N) : nullptr, Dinv + K * TILE_ELEMS, st, kOzTimeout);
  if (e != cudaSuccess) return e;
  note_launch();
  k_digits<<<(unsigned)below, 256, 0, s>>>(nullptr, Z, K, dg, st);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_factor64_update(double* Z, int64_t K, int64_t N, void* scratch, bool entries, DevStatus* st,
                                   cudaStream_t s) {
  const int64_t below = N - K - 1, tiles = num_lower_tiles(below);
  if (below <= 0) return cudaSuccess;
  if (2 * tiles > 0x7fffffffLL) return cudaErrorInvalidValue;
  const int smem = OZ_SMEM + 1024;
  cudaError_t e = cudaFuncSetAttribute(k_oz_gemm<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  k_oz_gemm<false><<<(unsigned)(2 * tiles), OZ_THREADS, smem, s>>>(Z, N, K, static_cast<const unsigned char*>(scratch),
                                                                  entries ? least_of(scratch, N) : nullptr, nullptr, st,
                                                                  kOzTimeout);
  note_launch();
  return cudaGetLastError();
}

}  // namespace mag
