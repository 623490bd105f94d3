// K1: fused distance + exp generator of Z = exp[-t d] (Sec. 2), packed lower tiles.
//
// k_generate_q, k_dist_q + k_generate_from_dist and k_dense_q form the pairs in
// 64-bit fixed point from the quantized coordinates (mag_fx.cuh), without an FP64
// operation but for pairs too close for those.  k_generate, below, serves the
// points that admit no quantization (m > 512, a non-finite coordinate, every
// dimension constant, a scale beyond 2^+-400, exact_distances = 0, no memory for
// the copy):
//
// One CTA per lower tile (I, J).  Coordinates of the tile's 128 row points and
// 128 column points are staged in shared memory in chunks of MC coordinates;
// every pair difference x_jl - x_kl is taken in FP64 and squared/accumulated
// with FP64 FMAs (no ||x||^2 + ||y||^2 - 2 x^T y expansion, so close points do
// not cancel).  The FP32 tile (factor input) takes sqrt/exp in FP32 from the
// FP64 d^2; the FP64 tile (FP64 factor or stored residual) takes them in FP64.
//
// Thread layout of k_generate (512 threads): warp w handles tile rows w + 16 i (i < 8),
// lane l handles tile columns 4 l + q (q < 4), so each thread stores its four
// entries of a row with one 16-byte store (FP32: a float4; FP64: two
// double2) and a warp's stores cover one whole tile row.  The column points
// are staged in shared memory with column 4 l + q at position 32 q + l, so
// the distance loop's reads stay conflict free.
//
// Side outputs, all fused: full row sums of Z (for ||Z||inf and the Gershgorin
// bound used to choose the factor precision), min off-diagonal d^2 (the Sec. 1
// bound), and flags for non-finite coordinates and coincident points.
#include "mag_fx.cuh"
#include "mag_internal.cuh"
#include "mag_math.cuh"

namespace mag {

namespace {

constexpr int GEN_THREADS = 512;
constexpr int GEN_MC = 32;  // coordinates staged per chunk

__device__ inline void atomic_max_nonneg(unsigned long long* a, double v) {
  atomicMax(a, (unsigned long long)__double_as_longlong(v));
}

// Tiles of a slab layout (mag_internal.cuh: tile_index with column cap W)
// whose tile (0, 0) is the global tile (t0, t0); W >= the tile rows and
// t0 = 0 give the whole packed matrix.
template <bool WF, bool WD, bool ROWSUM, bool WDIST>
__global__ void __launch_bounds__(GEN_THREADS, 1)
    k_generate(const double* __restrict__ X, int64_t n, int m, double t, float* __restrict__ Zf,
               double* __restrict__ Zd, double* __restrict__ Dd, double* __restrict__ rowsum, DevStatus* st,
               int kind, double dcut, int64_t t0, int64_t W, double kc) {
  extern __shared__ double smem[];
  double* xr = smem;                   // [TILE][GEN_MC] row points (broadcast reads)
  double* xc = smem + TILE * GEN_MC;   // [GEN_MC][TILE] column points (conflict free)
  __shared__ double colpart[GEN_THREADS / 32][TILE];
  __shared__ unsigned long long warpmin[GEN_THREADS / 32];
  __shared__ __align__(16) double exptab[EXPT_SMEM];
  if (WD) load_exp_table(exptab);

  int64_t I, J;
  tile_coords((int64_t)blockIdx.x, W, &I, &J);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t row0 = (t0 + I) * TILE, col0 = (t0 + J) * TILE;

  double d2[8][4];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int q = 0; q < 4; ++q) d2[i][q] = 0.0;

  for (int l0 = 0; l0 < m; l0 += GEN_MC) {
    const int mc = min(GEN_MC, m - l0);
    for (int e = threadIdx.x; e < TILE * mc; e += GEN_THREADS) {
      const int r = e / mc, l = e - r * mc;
      const int64_t gr = row0 + r, gc = col0 + r;
      xr[r * GEN_MC + l] = gr < n ? X[gr * m + l0 + l] : 0.0;
      xc[l * TILE + 32 * (r & 3) + (r >> 2)] = gc < n ? X[gc * m + l0 + l] : 0.0;
    }
    __syncthreads();
    for (int l = 0; l < mc; ++l) {
      double a[8], b[4];
#pragma unroll
      for (int i = 0; i < 8; ++i) a[i] = xr[(warp + 16 * i) * GEN_MC + l];
#pragma unroll
      for (int q = 0; q < 4; ++q) b[q] = xc[l * TILE + 32 * q + lane];  // column 4 lane + q
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const double diff = a[i] - b[q];
          d2[i][q] = fma(diff, diff, d2[i][q]);
        }
    }
    __syncthreads();
  }

  const int64_t tile_off = tile_index(I, J, W) * TILE_ELEMS;
  // row/column partial sums of a thread cover 4 and 8 entries: FP32 is ample
  // for a norm, and keeps the FP64 pipe for the distances and the exponential
  float rs[8], cs[4];
#pragma unroll
  for (int i = 0; i < 8; ++i) rs[i] = 0.0f;
#pragma unroll
  for (int q = 0; q < 4; ++q) cs[q] = 0.0f;
  unsigned long long mind2b = 0x7ff0000000000000ull;  // +inf
  int flags = 0;
  const float tf = (float)t;
  // d > dcut = tiny_arg / t (from the host) on the bit patterns (d >= 0):
  // the FP64 pipe stays on the distances and the exponential
  const unsigned long long tiny_bits = (unsigned long long)__double_as_longlong(dcut);

#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int r = warp + 16 * i;
    const int64_t gr = row0 + r;
    float zfv[4];
    double zdv[4], ddv[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int c = 4 * lane + q;
      const int64_t gc = col0 + c;
      const double v = d2[i][q];
      double zd = 0.0, dd = 0.0;
      float zf = 0.0f;
      if (gr >= n || gc >= n || gr == gc) {
        zd = (gr == gc) ? 1.0 : 0.0;
        zf = (float)zd;
      } else {
        // v >= 0 or NaN: the checks and the minimum on the bit pattern (integer
        // pipe; non-negative doubles order like their bits)
        const unsigned long long vb = (unsigned long long)__double_as_longlong(v);
        if ((vb >> 52) >= 0x7ffull) flags |= ST_NONFINITE;
        else if (vb == 0ull) flags |= ST_DUPLICATE;
        else mind2b = vb < mind2b ? vb : mind2b;
        if (WD || WDIST) dd = sqrt_pos(v);
        if (WD && !kind && (unsigned long long)__double_as_longlong(dd) > tiny_bits) {
          zf = exp_neg_tiny_td(tf, t, dd);
          zd = f32_to_f64_nonneg(zf);
        } else {
          if (WD) zd = mat_entry(kind, t, kc, dd, exptab);
          if (WF)
            zf = WD ? (kind == MAT_DEFLATED ? __double2float_rn(zd) : f64_to_f32_nonneg(zd))
                    : (kind == MAT_EXP ? expf(-td_f32(tf, t, v))
                                       : (kind == MAT_SHIFTED_DIST ? 1.0f - td_f32(tf, t, v)
                                                                   : fmaf((float)kc, expm1f(-td_f32(tf, t, v)), 1.0f)));
        }
      }
      zfv[q] = zf;
      zdv[q] = zd;
      ddv[q] = dd;
      if (ROWSUM && gr < n && gc < n) {
        const float zs = WF ? zf : (float)zd;
        rs[i] += zs;
        cs[q] += zs;
      }
    }
    // the four entries of row r, columns 4 lane .. 4 lane + 3: 16-byte stores
    const int64_t e = tile_off + (int64_t)r * TILE + 4 * lane;
    if (WF) *reinterpret_cast<float4*>(Zf + e) = make_float4(zfv[0], zfv[1], zfv[2], zfv[3]);
    if (WD) {
      *reinterpret_cast<double2*>(Zd + e) = make_double2(zdv[0], zdv[1]);
      *reinterpret_cast<double2*>(Zd + e + 2) = make_double2(zdv[2], zdv[3]);
    }
    if (WDIST) {
      *reinterpret_cast<double2*>(Dd + e) = make_double2(ddv[0], ddv[1]);
      *reinterpret_cast<double2*>(Dd + e + 2) = make_double2(ddv[2], ddv[3]);
    }
  }

  if (flags) atomicOr(&st->flags, flags);
  // min d^2 over the CTA
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long other = __shfl_xor_sync(0xffffffffu, mind2b, o);
    mind2b = other < mind2b ? other : mind2b;
  }
  if (lane == 0) warpmin[warp] = mind2b;

  if (ROWSUM) {
    // row sums: an FP32 lane tree (a norm: depth 5 adds at most 5 roundings
    // to the 4-entry partials), one FP64 atomic per row
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      float v = rs[i];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      const int64_t gr = row0 + warp + 16 * i;
      if (lane == 0 && gr < n) atomicAdd(rowsum + gr, (double)v);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) colpart[warp][4 * lane + q] = (double)cs[q];
  }
  __syncthreads();
  if (ROWSUM && I != J && threadIdx.x < TILE) {
    double v = 0.0;
    for (int w = 0; w < GEN_THREADS / 32; ++w) v += colpart[w][threadIdx.x];
    const int64_t gc = col0 + threadIdx.x;
    if (gc < n) atomicAdd(rowsum + gc, v);
  }
  if (threadIdx.x == 0) {
    unsigned long long v = warpmin[0];
    for (int w = 1; w < GEN_THREADS / 32; ++w) v = warpmin[w] < v ? warpmin[w] : v;
    if (v < 0x7ff0000000000000ull) atomicMin(&st->min_d2_bits, v);
  }
}

// Z from stored FP64 distances (same layout): one CTA per lower tile, the
// exponential of mag_fx.cuh (EXP: Z = exp(-t d)) or FP64, 16-byte reads and
// stores (lane l: columns 4 l .. 4 l + 3).  Tiles of the padding get the
// identity, as in k_generate.
template <bool WF, bool WD, bool EXP>
__global__ void __launch_bounds__(256) k_generate_from_dist(const double* __restrict__ Dd, int64_t n, double t,
                                                            FxScale sc, float* __restrict__ Zf,
                                                            double* __restrict__ Zd, double* __restrict__ rowsum,
                                                            int kind, double dcut, double kc) {
  __shared__ __align__(16) double exptab[EXP ? 2 : 2 * EXPT_SIZE];
  __shared__ fx_u64 fxtab[EXP ? FX_TABLE_SIZE : 2];
  __shared__ float colpart[8][TILE];
  if (EXP)
    load_fx_table(fxtab);
  else
    load_exp_table_d(exptab);
  __syncthreads();
  int64_t I, J;
  tri_coords((int64_t)blockIdx.x, &I, &J);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t off = tri_index(I, J) * TILE_ELEMS;
  const float tf = (float)t;
  const unsigned long long tiny_bits = (unsigned long long)__double_as_longlong(dcut);
  // row/column partial sums in FP32 (a norm)
  float cs[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll 1
  for (int i = 0; i < 16; ++i) {
    const int r = warp * 16 + i;
    const int64_t gr = I * TILE + r;
    float rs = 0.0f;
    // lane: columns 4 lane .. 4 lane + 3 of row r, read and written with
    // 16-byte accesses
    const int64_t e0 = off + (int64_t)r * TILE + 4 * lane;
    const double2 d01 = *reinterpret_cast<const double2*>(Dd + e0);
    const double2 d23 = *reinterpret_cast<const double2*>(Dd + e0 + 2);
    const double dv[4] = {d01.x, d01.y, d23.x, d23.y};
    float zfv[4];
    double zdv[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int c = 4 * lane + q;
      const int64_t gc = J * TILE + c;
      double zd;
      float zf;
      if (gr >= n || gc >= n || gr == gc) {
        zd = (gr == gc) ? 1.0 : 0.0;
        zf = (float)zd;
        if (gr == gc && gr < n) rs += 1.0f;  // the diagonal counts in its row sum
      } else {
        const double d = dv[q];
        const unsigned long long db = (unsigned long long)__double_as_longlong(d);
        if (EXP && db > tiny_bits) {
          zf = exp_neg_tiny_td(tf, t, d);
          zd = f32_to_f64_nonneg(zf);
        } else {
          zd = EXP ? __longlong_as_double((long long)fx_exp_neg_d(db, sc.kg, sc.g, fxtab))
                   : mat_entry(kind, t, kc, d, exptab);
          zf = !EXP && kind == MAT_DEFLATED ? __double2float_rn(zd) : f64_to_f32_nonneg(zd);
        }
        rs += zf;
        cs[q] += zf;
      }
      zfv[q] = zf;
      zdv[q] = zd;
    }
    if (WF) *reinterpret_cast<float4*>(Zf + e0) = make_float4(zfv[0], zfv[1], zfv[2], zfv[3]);
    if (WD) {
      *reinterpret_cast<double2*>(Zd + e0) = make_double2(zdv[0], zdv[1]);
      *reinterpret_cast<double2*>(Zd + e0 + 2) = make_double2(zdv[2], zdv[3]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) rs += __shfl_xor_sync(0xffffffffu, rs, o);
    if (lane == 0 && gr < n) atomicAdd(rowsum + gr, (double)rs);
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) colpart[warp][4 * lane + q] = cs[q];
  __syncthreads();
  if (I != J && threadIdx.x < TILE) {
    double v = 0.0;
    for (int w = 0; w < 8; ++w) v += (double)colpart[w][threadIdx.x];
    const int64_t gc = J * TILE + threadIdx.x;
    if (gc < n) atomicAdd(rowsum + gc, v);
  }
}

// max_j ||x_j - x_0||^2 (FP64 differences) into aux_bits: 2 max_j ||x_j - x_0||
// bounds every pairwise distance (triangle inequality through x_0).
__global__ void k_far_from_first(const double* __restrict__ X, int64_t n, int m, DevStatus* st) {
  double v = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    double s2 = 0.0;
    for (int l = 0; l < m; ++l) {
      const double diff = X[i * m + l] - X[l];
      s2 = fma(diff, diff, s2);
    }
    v = fmax(v, s2);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  if ((threadIdx.x & 31) == 0) atomic_max_nonneg(&st->far_d2_bits, v);
}

__global__ void k_rowsum_max(const double* __restrict__ rowsum, int64_t n, DevStatus* st) {
  double v = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    v = fmax(v, rowsum[i] - 1.0);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  if ((threadIdx.x & 31) == 0) atomic_max_nonneg(&st->off_max_bits, fmax(v, 0.0));
}

// Pairs of quantized points that are too close for them (fx_close): d^2 from
// the FP64 differences, as k_generate, with the coincident-point flag.  A cloud
// with one point far away has nothing but such pairs: the dense Z of 4096 points
// then takes 2.66 ms in R^64 and 4.00 in R^100 (k_generate 2.72 and 3.99; 2.93 and
// 4.49 with 8-byte loads).
__device__ __noinline__ double close_square(const double* __restrict__ X, int64_t gr, int64_t gc, int m, int* flags,
                                            unsigned long long* mind2b) {
  double v = 0.0;
  const double *x = X + gr * m, *y = X + gc * m;
  if (!((m & 1) | ((uintptr_t)X & 15))) {  // 16-byte loads: a warp's are in 32 different lines
#pragma unroll 4
    for (int l = 0; l < m; l += 2) {
      const double2 a = *reinterpret_cast<const double2*>(x + l), b = *reinterpret_cast<const double2*>(y + l);
      const double d0 = a.x - b.x, d1 = a.y - b.y;
      v = fma(d1, d1, fma(d0, d0, v));
    }
  } else {
#pragma unroll 4
    for (int l = 0; l < m; ++l) {
      const double diff = x[l] - y[l];
      v = fma(diff, diff, v);
    }
  }
  const unsigned long long vb = (unsigned long long)__double_as_longlong(v);
  if (vb == 0ull) *flags |= ST_DUPLICATE;
  else *mind2b = vb < *mind2b ? vb : *mind2b;
  return v;
}

// A CTA's flags and min d^2 (mq: the least square of this thread's pairs that
// were not close, h = ~0 if none) into the status.
__device__ __forceinline__ void finish_min(unsigned long long mind2b, const FxSquare& mq, int e, int flags,
                                           unsigned long long* warpmin, DevStatus* st) {
  if (mq.h != ~0ull) {
    const unsigned long long b = fx_square_bits(mq, e);
    mind2b = b < mind2b ? b : mind2b;
  }
  if (flags) atomicOr(&st->flags, flags);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long other = __shfl_xor_sync(0xffffffffu, mind2b, o);
    mind2b = other < mind2b ? other : mind2b;
  }
  if ((threadIdx.x & 31) == 0) warpmin[threadIdx.x >> 5] = mind2b;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long v = warpmin[0];
    for (int w = 1; w < FX_THREADS / 32; ++w) v = warpmin[w] < v ? warpmin[w] : v;
    if (v < 0x7ff0000000000000ull) atomicMin(&st->min_d2_bits, v);
  }
}

// FP64 distances of the packed lower tiles from the quantized coordinates
// (mag_fx.cuh; pairs too close for them from the FP64 differences of X), with
// min d^2 and the coincident-point flag as k_generate: one CTA per tile.  Rows
// and columns of the padding get d = 0 (the generator from distances gives
// them the identity by index).
template <int KIND>
__global__ void __launch_bounds__(FX_THREADS, fx_ctas(KIND))
    k_dist_q(const fx_coord* __restrict__ Xq, const double* __restrict__ X, int64_t n, int m, int qe,
             double* __restrict__ Dd, DevStatus* st) {
  extern __shared__ __align__(16) unsigned char gen_smem[];
  __shared__ unsigned long long warpmin[FX_THREADS / 32];
  int64_t I, J;
  tri_coords((int64_t)blockIdx.x, &I, &J);
  const int lane = threadIdx.x & 31;
  const int64_t row0 = I * TILE, col0 = J * TILE;
  const int64_t tile_off = tri_index(I, J) * TILE_ELEMS;
  unsigned long long mind2b = 0x7ff0000000000000ull;  // +inf
  FxSquare mq{~0ull, ~0ull};
  int flags = 0;
  fx_tile_pairs<KIND>(Xq, n, m, row0, col0, reinterpret_cast<fx_coord*>(gen_smem), [&](int r, FxSquare(&q)[4]) {
    const int64_t gr = row0 + r;
    double ddv[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int64_t gc = col0 + 4 * lane + c;
      double dd = 0.0;
      if (gr < n && gc < n && gr != gc) {
        if (fx_close(q[c], m)) {
          dd = sqrt_pos(close_square(X, gr, gc, m, &flags, &mind2b));
        } else {
          if (q[c].h < mq.h || (q[c].h == mq.h && q[c].l < mq.l)) mq = q[c];
          const FxRoot rt = fx_root_start(q[c]);
          dd = __longlong_as_double((long long)fx_dist_bits(fx_root(rt), rt.j, qe));
        }
      }
      ddv[c] = dd;
    }
    const int64_t e = tile_off + (int64_t)r * TILE + 4 * lane;
    *reinterpret_cast<double2*>(Dd + e) = make_double2(ddv[0], ddv[1]);
    *reinterpret_cast<double2*>(Dd + e + 2) = make_double2(ddv[2], ddv[3]);
  }, (int)blockIdx.y, (int)gridDim.y);
  finish_min(mind2b, mq, qe, flags, warpmin, st);
}

// k_generate with the pair distances from the quantized coordinates and, for
// Z = exp(-t d) (EXP), the exponential of mag_fx.cuh from the unrounded
// distance: no FP64 operation but in the pairs too close for the quantized
// coordinates.  The same entries, checks and outputs in one pass (row sums
// when rowsum is given), tiles in the slab layout of k_generate.  Used where
// no distances are kept (a single t, the slabs of the out-of-core factor); a
// multi-t call keeps them with k_dist_q, then k_generate_from_dist.
template <int KIND, bool WF, bool WD, bool EXP>
__global__ void __launch_bounds__(FX_THREADS, fx_ctas(KIND))
    k_generate_q(const fx_coord* __restrict__ Xq, const double* __restrict__ X, int64_t n, int m, FxScale sc,
                 double t, float* __restrict__ Zf, double* __restrict__ Zd, double* __restrict__ rowsum,
                 DevStatus* st, int kind, float tiny, double kc, int64_t t0, int64_t W) {
  extern __shared__ __align__(16) unsigned char gen_smem[];
  __shared__ float colpart[FX_THREADS / 32][TILE];
  __shared__ unsigned long long warpmin[FX_THREADS / 32];
  __shared__ __align__(16) double exptab[EXP ? 2 : 2 * EXPT_SIZE];
  __shared__ fx_u64 fxtab[EXP ? FX_TABLE_SIZE : 2];
  if (EXP)
    load_fx_table(fxtab);
  else
    load_exp_table_d(exptab);
  int64_t I, J;
  tile_coords((int64_t)blockIdx.x, W, &I, &J);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t row0 = (t0 + I) * TILE, col0 = (t0 + J) * TILE;
  const int64_t tile_off = tile_index(I, J, W) * TILE_ELEMS;
  float cs[4] = {0.0f, 0.0f, 0.0f, 0.0f};
  unsigned long long mind2b = 0x7ff0000000000000ull;  // +inf
  FxSquare mq{~0ull, ~0ull};
  int flags = 0;
  fx_tile_pairs<KIND>(Xq, n, m, row0, col0, reinterpret_cast<fx_coord*>(gen_smem), [&](int r, FxSquare(&q)[4]) {
    const int64_t gr = row0 + r;
    float rs = 0.0f;
    float zfv[4];
    double zdv[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int64_t gc = col0 + 4 * lane + c;
      double zd = 0.0;
      float zf = 0.0f;
      if (gr >= n || gc >= n || gr == gc) {
        zd = (gr == gc) ? 1.0 : 0.0;
        zf = (float)zd;
      } else {
        fx_u64 s = 0, db = 0;
        int j = 0;
        if (fx_close(q[c], m)) {
          db = (fx_u64)__double_as_longlong(sqrt_pos(close_square(X, gr, gc, m, &flags, &mind2b)));
          if (EXP) zd = __longlong_as_double((long long)fx_exp_neg_d(db, sc.kg, sc.g, fxtab));
        } else {
          if (q[c].h < mq.h || (q[c].h == mq.h && q[c].l < mq.l)) mq = q[c];
          const FxRoot rt = fx_root_start(q[c]);
          // t d in FP32: beyond `tiny` the entry is evaluated on the FP32 pipe
          const float td = fx_float(fx_bits(rt.sf) + ((uint32_t)(rt.j - 63) << 23)) * sc.t63;
          if (EXP && td > tiny) {
            zf = exp_neg_tiny_f(td);
            zd = f32_to_f64_nonneg(zf);
          } else {
            s = fx_root(rt);
            j = rt.j;
            if (EXP)
              zd = __longlong_as_double((long long)fx_exp_neg(s, j - sc.e + sc.kg, sc.g, fxtab));
            else
              db = fx_dist_bits(s, j, sc.e);
          }
        }
        if (!EXP) zd = mat_entry(kind, t, kc, __longlong_as_double((long long)db), exptab);
        if (WF || !WD) zf = !EXP && kind == MAT_DEFLATED ? __double2float_rn(zd) : f64_to_f32_nonneg(zd);
      }
      zfv[c] = zf;
      zdv[c] = zd;
      if (gr < n && gc < n) {
        const float zs = WF ? zf : (float)zd;
        rs += zs;
        cs[c] += zs;
      }
    }
    const int64_t e = tile_off + (int64_t)r * TILE + 4 * lane;
    if (WF) *reinterpret_cast<float4*>(Zf + e) = make_float4(zfv[0], zfv[1], zfv[2], zfv[3]);
    if (WD) {
      *reinterpret_cast<double2*>(Zd + e) = make_double2(zdv[0], zdv[1]);
      *reinterpret_cast<double2*>(Zd + e + 2) = make_double2(zdv[2], zdv[3]);
    }
    // the row's sum: an FP32 lane tree, one FP64 atomic per row
    if (rowsum) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) rs += __shfl_xor_sync(0xffffffffu, rs, o);
      if (lane == 0 && gr < n) atomicAdd(rowsum + gr, (double)rs);
    }
  }, (int)blockIdx.y, (int)gridDim.y);
#pragma unroll
  for (int c = 0; c < 4; ++c) colpart[warp][4 * lane + c] = cs[c];
  finish_min(mind2b, mq, sc.e, flags, warpmin, st);  // synchronizes
  if (rowsum && I != J && threadIdx.x < TILE) {
    double v = 0.0;
    for (int w = 0; w < FX_THREADS / 32; ++w) v += (double)colpart[w][threadIdx.x];
    const int64_t gc = col0 + threadIdx.x;
    if (gc < n) atomicAdd(rowsum + gc, v);
  }
}

// Z = exp(-t d) as the dense n x n row-major matrix, both triangles, from the
// quantized coordinates: one CTA per lower tile writes it and its transpose
// (eight rows at a time through shared memory, 64 contiguous bytes per column
// in FP64), with the checks of k_generate.  In one pass; packed tiles first and
// a copy of them afterwards took twice the time.
template <int KIND, typename T>
__global__ void __launch_bounds__(FX_THREADS, fx_ctas(KIND))
    k_dense_q(const fx_coord* __restrict__ Xq, const double* __restrict__ X, int64_t n, int m, FxScale sc,
              T* __restrict__ Z, DevStatus* st) {
  extern __shared__ __align__(16) unsigned char gen_smem[];
  __shared__ unsigned long long warpmin[FX_THREADS / 32];
  __shared__ fx_u64 fxtab[FX_TABLE_SIZE];
  __shared__ T rows[2][FX_THREADS / 32][TILE + 1];  // two passes' rows, by the parity of the pass
  load_fx_table(fxtab);
  int64_t I, J;
  tri_coords((int64_t)blockIdx.x, &I, &J);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t row0 = I * TILE, col0 = J * TILE;
  unsigned long long mind2b = 0x7ff0000000000000ull;  // +inf
  FxSquare mq{~0ull, ~0ull};
  int flags = 0;
  fx_tile_pairs<KIND>(Xq, n, m, row0, col0, reinterpret_cast<fx_coord*>(gen_smem), [&](int r, FxSquare(&q)[4]) {
    const int64_t gr = row0 + r;
    const int pass = r >> 3;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int64_t gc = col0 + 4 * lane + c;
      double z = 1.0;
      if (gr < n && gc < n && gr != gc) {
        fx_u64 b;
        if (fx_close(q[c], m)) {
          const double d = sqrt_pos(close_square(X, gr, gc, m, &flags, &mind2b));
          b = fx_exp_neg_d((fx_u64)__double_as_longlong(d), sc.kg, sc.g, fxtab);
        } else {
          if (q[c].h < mq.h || (q[c].h == mq.h && q[c].l < mq.l)) mq = q[c];
          const FxRoot rt = fx_root_start(q[c]);
          b = fx_exp_neg(fx_root(rt), rt.j - sc.e + sc.kg, sc.g, fxtab);
        }
        z = __longlong_as_double((long long)b);
      }
      T v;
      if constexpr (sizeof(T) == 8)
        v = z;
      else
        v = f64_to_f32_nonneg(z);
      rows[pass & 1][warp][4 * lane + c] = v;
    }
    __syncthreads();  // every warp is on the same pass
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int64_t gc = col0 + lane + 32 * k;
      if (gr < n && gc < n) Z[gr * n + gc] = rows[pass & 1][warp][lane + 32 * k];
    }
    if (I != J) {  // the transpose: column (tid / 8) + 32 k, row tid % 8 of the pass
      const int rr = threadIdx.x & 7;
      const int64_t tr = row0 + 8 * pass + rr;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int c = (threadIdx.x >> 3) + 32 * k;
        if (tr < n && col0 + c < n) Z[(col0 + c) * n + tr] = rows[pass & 1][rr][c];
      }
    }
  });
  finish_min(mind2b, mq, sc.e, flags, warpmin, st);
}

// q = round(2^e (x - lo_l)) with x - lo_l taken exactly as s + err (TwoSum):
// round(2^e s) + round(2^e err), within one unit of 2^e (x - lo_l); stored as
// its limbs.
__global__ void k_quantize(const double* __restrict__ X, int64_t n, int m,
                           const unsigned long long* __restrict__ range, int e, fx_coord* __restrict__ Xq) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n * m) return;
  const int l = (int)(k % m);
  const double x = X[k], b = -ordered_value(range[2 * l]);
  const double s = x + b;
  const double bv = s - x;
  const double err = (x - (s - bv)) + (b - bv);
  const long long q = __double2ll_rn(ldexp(s, e)) + __double2ll_rn(ldexp(err, e));
  const int lb = fx_limb_of(m);
  Xq[k] = fx_coord{(int)(q & ((1ll << lb) - 1)), (int)(q >> lb)};
}

template <bool WF, bool WD, bool ROWSUM, bool WDIST = false>
cudaError_t launch_gen_t(const double* X, int64_t n, int m, double t, int64_t N, float* Zf,
                         double* Zd, double* rowsum, DevStatus* st, cudaStream_t s, double* Dd = nullptr,
                         int kind = 0, double tiny_arg = INFINITY, int64_t t0 = 0, int64_t W = -1, double kc = 0.0) {
  const size_t smem = 2 * (size_t)TILE * GEN_MC * sizeof(double);
  auto kern = k_generate<WF, WD, ROWSUM, WDIST>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  // N: tile rows of the (slab) matrix from global tile t0; W < 0: all columns
  if (W < 0) W = N;
  const int64_t tiles = num_slab_tiles(N, W);
  if (tiles > 0x7fffffffLL) return cudaErrorInvalidValue;
  // entries with d > tiny_arg / t leave the FP64 exponential
  const double dcut = tiny_arg / t;
  kern<<<(unsigned)tiles, GEN_THREADS, smem, s>>>(X, n, m, t, Zf, Zd, Dd, rowsum, st, kind, dcut, t0, W, kc);
  note_launch();
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_generate(const double* X, int64_t n, int m, double t, int64_t N, float* Zf,
                            double* Zd, double* rowsum, DevStatus* st, cudaStream_t s, int kind, double tiny_arg,
                            double kc) {
  if (Zf && Zd)
    return launch_gen_t<true, true, true>(X, n, m, t, N, Zf, Zd, rowsum, st, s, nullptr, kind, tiny_arg, 0, -1, kc);
  if (Zf) return launch_gen_t<true, false, true>(X, n, m, t, N, Zf, Zd, rowsum, st, s, nullptr, kind, INFINITY, 0, -1, kc);
  if (Zd)
    return launch_gen_t<false, true, true>(X, n, m, t, N, Zf, Zd, rowsum, st, s, nullptr, kind, tiny_arg, 0, -1, kc);
  return cudaErrorInvalidValue;
}

cudaError_t launch_generate_dist(const double* X, int64_t n, int m, double t, int64_t N, float* Zf,
                                 double* Zd, double* Dd, double* rowsum, DevStatus* st, cudaStream_t s,
                                 int kind, double tiny_arg, double kc) {
  if (Zf && Zd)
    return launch_gen_t<true, true, true, true>(X, n, m, t, N, Zf, Zd, rowsum, st, s, Dd, kind, tiny_arg, 0, -1, kc);
  if (Zf) return launch_gen_t<true, false, true, true>(X, n, m, t, N, Zf, Zd, rowsum, st, s, Dd, kind, INFINITY, 0, -1, kc);
  if (Zd)
    return launch_gen_t<false, true, true, true>(X, n, m, t, N, Zf, Zd, rowsum, st, s, Dd, kind, tiny_arg, 0, -1, kc);
  return cudaErrorInvalidValue;
}

namespace {

// CTAs a tile: a tile's 16 rows a warp take 45 us, so while all of a launch's
// CTAs are resident at once its rows are shared by two or four (n = 300, m = 6:
// 52 -> 19 us).
unsigned row_slices(int64_t tiles, int kind) {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return 1;
  const int64_t resident = (int64_t)sms * fx_ctas(kind);
  return 4 * tiles <= resident ? 4u : (2 * tiles <= resident ? 2u : 1u);
}

template <int KIND, bool WF, bool WD, bool EXP>
cudaError_t launch_gen_q(const fx_coord* Xq, const double* X, int64_t n, int m, const FxScale& sc, double t,
                         unsigned tiles, float* Zf, double* Zd, double* rowsum, DevStatus* st, cudaStream_t s,
                         int kind, float tiny, double kc, int64_t t0, int64_t W) {
  auto kern = k_generate_q<KIND, WF, WD, EXP>;
  const size_t smem = fx_tile_smem(m);
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FX_TILE_SMEM_MAX);
  if (e != cudaSuccess) return e;
  kern<<<dim3(tiles, row_slices(tiles, KIND)), FX_THREADS, smem, s>>>(Xq, X, n, m, sc, t, Zf, Zd, rowsum, st, kind, tiny, kc, t0, W);
  note_launch();
  return cudaGetLastError();
}

template <int KIND, bool EXP>
cudaError_t launch_gen_q_out(const fx_coord* Xq, const double* X, int64_t n, int m, const FxScale& sc, double t,
                             unsigned tiles, float* Zf, double* Zd, double* rowsum, DevStatus* st, cudaStream_t s,
                             int kind, float tiny, double kc, int64_t t0, int64_t W) {
  if (Zf && Zd)
    return launch_gen_q<KIND, true, true, EXP>(Xq, X, n, m, sc, t, tiles, Zf, Zd, rowsum, st, s, kind, tiny, kc, t0, W);
  if (Zf)  // FP32 tiles alone: rounded from the FP64 entries
    return launch_gen_q<KIND, true, false, EXP>(Xq, X, n, m, sc, t, tiles, Zf, Zd, rowsum, st, s, kind, tiny, kc, t0, W);
  if (Zd)
    return launch_gen_q<KIND, false, true, EXP>(Xq, X, n, m, sc, t, tiles, Zf, Zd, rowsum, st, s, kind, tiny, kc, t0, W);
  return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_generate_q(const void* Xq, const double* X, int64_t n, int m, int e, double t, int64_t N,
                              float* Zf, double* Zd, double* rowsum, DevStatus* st, cudaStream_t s, int kind,
                              double tiny_arg, double kc, int64_t t0, int64_t W) {
  if (m < 1 || m > FX_MAX_DIM) return cudaErrorInvalidValue;
  // N: tile rows of the (slab) matrix from global tile t0; W < 0: all columns
  if (W < 0) W = N;
  const int64_t tiles = num_slab_tiles(N, W);
  if (tiles > 0x7fffffffLL) return cudaErrorInvalidValue;
  const FxScale sc = fx_scale(t, e);
  const fx_coord* q = static_cast<const fx_coord*>(Xq);
  const unsigned g = (unsigned)tiles;
  const float ta = (float)tiny_arg;
#define MAG_GEN_Q(KIND_)                                                                                               \
  return kind == MAT_EXP                                                                                               \
             ? launch_gen_q_out<KIND_, true>(q, X, n, m, sc, t, g, Zf, Zd, rowsum, st, s, kind, ta, kc, t0, W)         \
             : launch_gen_q_out<KIND_, false>(q, X, n, m, sc, t, g, Zf, Zd, rowsum, st, s, kind, ta, kc, t0, W)
  switch (fx_kind(m)) {
    case 0: MAG_GEN_Q(0);
    case 1: MAG_GEN_Q(1);
    default: MAG_GEN_Q(2);
  }
#undef MAG_GEN_Q
}

template <int KIND, typename T>
static cudaError_t launch_dense_t(const fx_coord* Xq, const double* X, int64_t n, int m, const FxScale& sc, T* Z,
                                  unsigned tiles, DevStatus* st, cudaStream_t s) {
  auto kern = k_dense_q<KIND, T>;
  const size_t smem = fx_tile_smem(m);
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FX_TILE_SMEM_MAX);
  if (e != cudaSuccess) return e;
  kern<<<tiles, FX_THREADS, smem, s>>>(Xq, X, n, m, sc, Z, st);
  note_launch();
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_dense_q(const void* Xq, const double* X, int64_t n, int m, int e, double t, T* Z, DevStatus* st,
                           cudaStream_t s) {
  if (m < 1 || m > FX_MAX_DIM) return cudaErrorInvalidValue;
  const int64_t tiles = num_lower_tiles((n + TILE - 1) / TILE);
  if (tiles > 0x7fffffffLL) return cudaErrorInvalidValue;
  const FxScale sc = fx_scale(t, e);
  const fx_coord* q = static_cast<const fx_coord*>(Xq);
  switch (fx_kind(m)) {
    case 0: return launch_dense_t<0, T>(q, X, n, m, sc, Z, (unsigned)tiles, st, s);
    case 1: return launch_dense_t<1, T>(q, X, n, m, sc, Z, (unsigned)tiles, st, s);
    default: return launch_dense_t<2, T>(q, X, n, m, sc, Z, (unsigned)tiles, st, s);
  }
}
template cudaError_t launch_dense_q<float>(const void*, const double*, int64_t, int, int, double, float*, DevStatus*,
                                           cudaStream_t);
template cudaError_t launch_dense_q<double>(const void*, const double*, int64_t, int, int, double, double*,
                                            DevStatus*, cudaStream_t);

cudaError_t launch_quantize(const double* X, int64_t n, int m, const unsigned long long* range, int e, void* Xq,
                            cudaStream_t s) {
  const int64_t k = n * m;
  k_quantize<<<(unsigned)((k + 255) / 256), 256, 0, s>>>(X, n, m, range, e, static_cast<fx_coord*>(Xq));
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_dist_q(const void* Xq, const double* X, int64_t n, int m, int e, int64_t N, double* Dd,
                          DevStatus* st, cudaStream_t s) {
  if (m < 1 || m > FX_MAX_DIM) return cudaErrorInvalidValue;
  const size_t smem = fx_tile_smem(m);
  const int64_t tiles = num_lower_tiles(N);
  if (tiles > 0x7fffffffLL) return cudaErrorInvalidValue;
  const fx_coord* q = static_cast<const fx_coord*>(Xq);
  const int kd = fx_kind(m);
  auto kern = kd == 0 ? k_dist_q<0> : (kd == 1 ? k_dist_q<1> : k_dist_q<2>);
  cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FX_TILE_SMEM_MAX);
  if (err != cudaSuccess) return err;
  kern<<<dim3((unsigned)tiles, row_slices(tiles, kd)), FX_THREADS, smem, s>>>(q, X, n, m, e, Dd, st);
  note_launch();
  return cudaGetLastError();
}

namespace {

template <bool WF, bool WD>
void launch_from_dist(unsigned tiles, const double* Dd, int64_t n, double t, const FxScale& sc, float* Zf, double* Zd,
                      double* rowsum, cudaStream_t s, int kind, double dcut, double kc) {
  if (kind == MAT_EXP)
    k_generate_from_dist<WF, WD, true><<<tiles, 256, 0, s>>>(Dd, n, t, sc, Zf, Zd, rowsum, kind, dcut, kc);
  else
    k_generate_from_dist<WF, WD, false><<<tiles, 256, 0, s>>>(Dd, n, t, sc, Zf, Zd, rowsum, kind, dcut, kc);
}

}  // namespace

cudaError_t launch_generate_from_dist(const double* Dd, int64_t n, double t, int64_t N, float* Zf, double* Zd,
                                     double* rowsum, cudaStream_t s, int kind, double tiny_arg, double kc) {
  const unsigned tiles = (unsigned)num_lower_tiles(N);
  const double dcut = tiny_arg / t;
  const FxScale sc = fx_scale(t, 0);
  if (Zf && Zd)
    launch_from_dist<true, true>(tiles, Dd, n, t, sc, Zf, Zd, rowsum, s, kind, dcut, kc);
  else if (Zf)
    launch_from_dist<true, false>(tiles, Dd, n, t, sc, Zf, Zd, rowsum, s, kind, INFINITY, kc);
  else if (Zd)
    launch_from_dist<false, true>(tiles, Dd, n, t, sc, Zf, Zd, rowsum, s, kind, dcut, kc);
  else
    return cudaErrorInvalidValue;
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_generate_slab(const double* X, int64_t n, int m, double t, int64_t t0, int64_t W, float* Zf,
                                 DevStatus* st, cudaStream_t s, double tiny_arg, const void* Xq, int qe) {
  const int64_t N = (n + TILE - 1) / TILE;
  if (t0 < 0 || t0 >= N || W < 1) return cudaErrorInvalidValue;
  if (Xq)
    return launch_generate_q(Xq, X, n, m, qe, t, N - t0, Zf, nullptr, nullptr, st, s, MAT_EXP, tiny_arg, 0.0, t0, W);
  return launch_gen_t<true, false, false>(X, n, m, t, N - t0, Zf, nullptr, nullptr, st, s, nullptr, MAT_EXP,
                                          tiny_arg, t0, W);
}

cudaError_t launch_min_distance(const double* X, int64_t n, int m, DevStatus* st, cudaStream_t s) {
  const int64_t N = (n + TILE - 1) / TILE;
  return launch_gen_t<false, false, false>(X, n, m, 1.0, N, nullptr, nullptr, nullptr, st, s);
}

cudaError_t launch_far_from_first(const double* X, int64_t n, int m, DevStatus* st, cudaStream_t s) {
  int blocks = (int)((n + 255) / 256);
  if (blocks > 4096) blocks = 4096;
  k_far_from_first<<<blocks, 256, 0, s>>>(X, n, m, st);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_rowsum_max(const double* rowsum, int64_t n, DevStatus* st, cudaStream_t s) {
  int blocks = (int)((n + 255) / 256);
  if (blocks > 1024) blocks = 1024;
  k_rowsum_max<<<blocks, 256, 0, s>>>(rowsum, n, st);
  note_launch();
  return cudaGetLastError();
}

}  // namespace mag
