// K1, the bound alone: min_{j != k} d_jk^2 over all pairs, with the flags for
// coincident points and non-finite coordinates.
//
// GB300 runs FP64 at 1/64 of FP32, and nearly every pair is far from the
// minimum: the pairs are compared in FP32 and only those that could hold the
// minimum are evaluated in FP64, by the generator's own expression, so the
// result is the FP64 minimum bit for bit.
//
//   coordinates: a_l = (x_l - lo_l) 2^-E in FP32, E from the largest span, so
//     0 <= a_l <= 1 and each is within 2^-24 of its value;
//   pairs: |d32 - d| <= delta d + eps with delta = (m + 8) 2^-24 (rounding of
//     the differences, the squares and their sum) and eps = 1.05 sqrt(m) 2^-23
//     (the coordinates' rounding);
//   any pair's d32 bounds the minimum by d32 (1 + delta) + eps, so the
//     minimum's own d32 is at most (d32 (1 + delta) + eps) (1 + delta) + eps.
//
// A first launch takes the least d32 of the diagonal tiles; the main launch
// reads the least d32 known so far when a tile starts, and lowers it.  With
// N = n / 128 tiles a side the expected number of pairs evaluated in FP64 is
// about N; where a cloud's close pairs cannot be told apart in FP32 (spans of
// 2^20 times the closest distances, a lattice) more are, at worst all of them,
// at the FP64 rate.  Non-finite spans, no span at all or spans beyond 2^+-400
// send every pair there.
//
// One CTA per lower tile, 256 threads, 8 x 8 pairs a thread, four 16-byte
// shared-memory reads per 64 differences and FMAs.  Bound: FP32 issue (2 m + 1
// operations a pair).  A call at n = 30,000: m = 10 0.67 ms (17.1 ms with FP64
// differences for every pair); n = 60,000, m = 30 4.7 ms (194); a 28^3 lattice
// 0.28 ms (3.1), two clusters 1e9 of their closest distances apart, half of
// the pairs evaluated in FP64, 1.3 ms at n = 20,000 (2.6); n = 200 43 us (56).
#include "mag_internal.cuh"
#include "mag_math.cuh"

namespace mag {

namespace {

constexpr int MD_THREADS = 256;
constexpr int MD_MC = 32;  // dimensions staged per chunk

// Doubles in an order-preserving unsigned encoding (for atomic min / max).
__device__ __forceinline__ unsigned long long ordered_bits(double v) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  return (b >> 63) ? ~b : b | 0x8000000000000000ull;
}

// Starting values of the range and (if given) of the least d32^2.
__global__ void k_range_init(unsigned long long* range, int m, unsigned* best32) {
  for (int e = threadIdx.x; e < 2 * m; e += blockDim.x) range[e] = (e & 1) ? 0ull : ~0ull;
  if (threadIdx.x == 0) {
    range[2 * m] = 0ull;
    if (best32) *best32 = 0x7f800000u;
  }
}

// Per dimension min and max of X in the ordered encoding: range[2 l] (starts
// at ~0), range[2 l + 1] (starts at 0); range[2 m] = 1 if a coordinate is not
// finite.  A thread stays on one dimension (m <= 256: rows of whole points per
// CTA pass, consecutive threads on consecutive addresses).
__global__ void __launch_bounds__(256) k_range_ordered(const double* __restrict__ X, int64_t n, int m,
                                                       unsigned long long* __restrict__ range) {
  __shared__ unsigned long long slo[256], shi[256];
  const int t = threadIdx.x;
  bool bad = false;
  if (m <= 256) {
    const int per = 256 / m;  // points per CTA pass
    unsigned long long lo = ~0ull, hi = 0ull;
    if (t < per * m)
      for (int64_t i = (int64_t)blockIdx.x * per + t / m; i < n; i += (int64_t)gridDim.x * per) {
        const double v = X[i * m + t % m];
        if (!isfinite(v)) bad = true;
        const unsigned long long b = ordered_bits(v);
        lo = b < lo ? b : lo;
        hi = b > hi ? b : hi;
      }
    slo[t] = lo;
    shi[t] = hi;
    __syncthreads();
    if (t < m) {
      for (int k = t + m; k < per * m; k += m) {
        lo = slo[k] < lo ? slo[k] : lo;
        hi = shi[k] > hi ? shi[k] : hi;
      }
      atomicMin(range + 2 * t, lo);
      atomicMax(range + 2 * t + 1, hi);
    }
  } else {
    for (int l = t; l < m; l += 256) {
      unsigned long long lo = ~0ull, hi = 0ull;
      for (int64_t i = blockIdx.x; i < n; i += gridDim.x) {
        const double v = X[i * m + l];
        if (!isfinite(v)) bad = true;
        const unsigned long long b = ordered_bits(v);
        lo = b < lo ? b : lo;
        hi = b > hi ? b : hi;
      }
      atomicMin(range + 2 * l, lo);
      atomicMax(range + 2 * l + 1, hi);
    }
  }
  if (bad) range[2 * m] = 1ull;
}

// A[tile][l][r] = (x_l - lo_l) 2^-E of point r of each 128-point tile in FP32
// (NaN past n: such pairs compare false); one CTA per tile.  0 where the span
// admits no scale (every pair is then evaluated in FP64).
__global__ void __launch_bounds__(256) k_scale_points(const double* __restrict__ X, int64_t n, int m,
                                                      const unsigned long long* __restrict__ range,
                                                      float* __restrict__ A, DevStatus* st) {
  __shared__ double smax[8];
  const int t = threadIdx.x;
  double S = 0.0;
  for (int l = t; l < m; l += 256) S = fmax(S, ordered_value(range[2 * l + 1]) - ordered_value(range[2 * l]));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) S = fmax(S, __shfl_xor_sync(0xffffffffu, S, o));
  if ((t & 31) == 0) smax[t >> 5] = S;
  __syncthreads();
  for (int w = 0; w < 8; ++w) S = fmax(S, smax[w]);
  const bool finite = range[2 * m] == 0ull;
  if (!finite && blockIdx.x == 0 && t == 0) atomicOr(&st->flags, ST_NONFINITE);
  const int E = S > 0.0 && isfinite(S) ? ilogb(S) + 1 : 1000;
  const double scale = finite && E > -400 && E < 400 ? ldexp(1.0, -E) : 0.0;
  const int64_t row0 = (int64_t)blockIdx.x * TILE;
  float* out = A + row0 * m;
  for (int e = t; e < TILE * m; e += 256) {
    const int r = e / m, l = e - r * m;
    const int64_t g = row0 + r;
    float v = __int_as_float(0x7fc00000);
    if (g < n) v = scale > 0.0 ? (float)((X[g * m + l] - ordered_value(range[2 * l])) * scale) : 0.0f;
    out[l * TILE + r] = v;
  }
}

// Least d32^2 (bits; starts at +inf) over the tiles of the launch.  ALL: all
// lower tiles, with the FP64 evaluation of the pairs that could hold the
// minimum; else the diagonal tiles, FP32 only.
template <bool ALL>
__global__ void __launch_bounds__(MD_THREADS, 2)
    k_min_dist(const double* __restrict__ X, const float* __restrict__ A, int64_t n, int m,
               unsigned* __restrict__ best32, DevStatus* st) {
  __shared__ __align__(16) float ar[MD_MC * TILE], ac[MD_MC * TILE];
  __shared__ unsigned smin[MD_THREADS / 32];
  __shared__ float sthr;
  int64_t I = blockIdx.x, J = blockIdx.x;
  if (ALL) tri_coords((int64_t)blockIdx.x, &I, &J);
  const int t = threadIdx.x, tx = t & 15, ty = t >> 4;
  const unsigned known = *(volatile unsigned*)best32;
  if (ALL && t == 0) {
    const double delta = (m + 8) * 0x1p-24, eps = 1.05 * sqrt((double)m) * 0x1p-23;
    double d = sqrt((double)__uint_as_float(known));
    d = (d * (1.0 + delta) + eps) * (1.0 + delta) + eps;
    sthr = __double2float_ru(d * d);
  }
  // rows 4 ty + i and 64 + 4 ty + i (i < 4), columns 4 tx + j and 64 + 4 tx + j
  float d2[8][8];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) d2[i][j] = 0.0f;
  for (int l0 = 0; l0 < m; l0 += MD_MC) {
    const int mc = min(MD_MC, m - l0);
    __syncthreads();
    const float4* gr = reinterpret_cast<const float4*>(A + (I * m + l0) * TILE);
    const float4* gc = reinterpret_cast<const float4*>(A + (J * m + l0) * TILE);
    for (int e = t; e < mc * TILE / 4; e += MD_THREADS) {
      reinterpret_cast<float4*>(ar)[e] = gr[e];
      reinterpret_cast<float4*>(ac)[e] = gc[e];
    }
    __syncthreads();
#pragma unroll 2
    for (int l = 0; l < mc; ++l) {
      const float4 a0 = *reinterpret_cast<const float4*>(ar + l * TILE + 4 * ty);
      const float4 a1 = *reinterpret_cast<const float4*>(ar + l * TILE + 64 + 4 * ty);
      const float4 b0 = *reinterpret_cast<const float4*>(ac + l * TILE + 4 * tx);
      const float4 b1 = *reinterpret_cast<const float4*>(ac + l * TILE + 64 + 4 * tx);
      const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
      const float b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const float diff = a[i] - b[j];
          d2[i][j] = fmaf(diff, diff, d2[i][j]);
        }
    }
  }
  if (I == J) {  // pairs of a diagonal tile once, below its diagonal
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int r = (i >> 2) * 64 + 4 * ty + (i & 3), c = (j >> 2) * 64 + 4 * tx + (j & 3);
        if (c >= r) d2[i][j] = __int_as_float(0x7fc00000);
      }
  }
  float mn = INFINITY;
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) mn = fminf(mn, d2[i][j]);  // NaN (padding, the skipped half) is passed over
  unsigned long long cand = 0ull;
  const float thr = ALL ? sthr : 0.0f;
  if (ALL && mn <= thr) {
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < 8; ++j)
        if (d2[i][j] <= thr) cand |= 1ull << (8 * i + j);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
  if ((t & 31) == 0) smin[t >> 5] = __float_as_uint(mn);
  if (ALL && cand) {
    unsigned long long mind2b = 0x7ff0000000000000ull;
    int flags = 0;
    do {
      const int b = __ffsll((long long)cand) - 1, i = b >> 3, j = b & 7;
      cand &= cand - 1ull;
      const int64_t gr = I * TILE + (i >> 2) * 64 + 4 * ty + (i & 3), gc = J * TILE + (j >> 2) * 64 + 4 * tx + (j & 3);
      double v = 0.0;
      for (int l = 0; l < m; ++l) {
        const double diff = X[gr * m + l] - X[gc * m + l];
        v = fma(diff, diff, v);
      }
      const unsigned long long vb = (unsigned long long)__double_as_longlong(v);
      if ((vb >> 52) >= 0x7ffull) flags |= ST_NONFINITE;
      else if (vb == 0ull) flags |= ST_DUPLICATE;
      else mind2b = vb < mind2b ? vb : mind2b;
    } while (cand);
    if (flags) atomicOr(&st->flags, flags);
    if (mind2b < *(volatile unsigned long long*)&st->min_d2_bits) atomicMin(&st->min_d2_bits, mind2b);
  }
  __syncthreads();
  if (t == 0) {
    unsigned v = smin[0];
    for (int w = 1; w < MD_THREADS / 32; ++w) v = smin[w] < v ? smin[w] : v;
    if (v < known) atomicMin(best32, v);
  }
}

cudaError_t range_ordered(const double* X, int64_t n, int m, unsigned long long* range, unsigned* best32,
                          cudaStream_t s) {
  k_range_init<<<1, 256, 0, s>>>(range, m, best32);
  note_launch();
  const int64_t passes = (n * m + 255) / 256;
  k_range_ordered<<<(unsigned)(passes < 304 ? passes : 304), 256, 0, s>>>(X, n, m, range);
  note_launch();
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_range_ordered(const double* X, int64_t n, int m, unsigned long long* range, cudaStream_t s) {
  return range_ordered(X, n, m, range, nullptr, s);
}

size_t min_distance_scratch_bytes(int64_t n, int m) {
  const int64_t N = (n + TILE - 1) / TILE;
  return (size_t)(2 * m + 2) * sizeof(unsigned long long) + 256 + (size_t)N * TILE * m * sizeof(float);
}

cudaError_t launch_min_distance_filtered(const double* X, int64_t n, int m, void* scratch, DevStatus* st,
                                         cudaStream_t s) {
  const int64_t N = (n + TILE - 1) / TILE, tiles = num_lower_tiles(N);
  if (tiles > 0x7fffffffLL) return cudaErrorInvalidValue;
  unsigned long long* range = static_cast<unsigned long long*>(scratch);
  unsigned* best32 = reinterpret_cast<unsigned*>(range + 2 * m + 1);
  const size_t head = ((size_t)(2 * m + 2) * sizeof(unsigned long long) + 255) & ~(size_t)255;
  float* A = reinterpret_cast<float*>(static_cast<char*>(scratch) + head);
  cudaError_t e = range_ordered(X, n, m, range, best32, s);
  if (e != cudaSuccess) return e;
  k_scale_points<<<(unsigned)N, 256, 0, s>>>(X, n, m, range, A, st);
  note_launch();
  k_min_dist<false><<<(unsigned)N, MD_THREADS, 0, s>>>(X, A, n, m, best32, st);
  note_launch();
  k_min_dist<true><<<(unsigned)tiles, MD_THREADS, 0, s>>>(X, A, n, m, best32, st);
  note_launch();
  return cudaGetLastError();
}

}  // namespace mag
