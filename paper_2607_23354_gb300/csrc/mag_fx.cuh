// Distances and exponentials on the integer pipe.
//
// GB300 issues FP64 at 1/64 of the FP32 and integer rate, so an FP64 operation
// costs as much as 64 integer ones: exp(-t d) of a pair from its quantized
// coordinates (the exact d^2 of quantize_points) is formed here in 64-bit fixed
// point with a 32 x 32 -> 64-bit multiplier, about 230 instructions against the
// nine FP64 operations (and a hundred others) it replaces, and rounded to FP64
// once.
//
//   d^2   exact: coordinates as two limbs, q = hi 2^30 + lo, the differences
//         of both limbs, and three 64-bit sums (lo lo, hi lo, hi hi) of signed
//         32 x 32-bit products;
//   d     sqrt of the leading 64 bits: an FP32 reciprocal square root, then two
//         corrections s += (v - s^2) / (2 s) with the residual exact in 64-bit
//         integers and the quotient in FP32 (P. Markstein, "Computation of
//         elementary functions on the IBM RISC System/6000 processor", IBM J.
//         Res. Dev. 34(1), 1990, on integers); within 2^-62 relative;
//   exp   Tang's table method (P. T. P. Tang, ACM TOMS 15(2), 1989):
//         256 t d / ln 2 = N + f from one 64 x 64-bit product with the scaled t
//         (never rounded to FP64), exp(-t d) = 2^-(N >> 8) T[N mod 256] (1 - p),
//         p = r - r^2/2 + r^3/6 - r^4/24 + r^5/120, r = f ln2/256 < 2^-8.5, the
//         cubic and later terms in 32 bits.  Omitted terms and truncations stay
//         below 2^-57.5 relative, so the rounding to FP64 dominates: within
//         0.55 units in the last place (and t d 2^-11 for t's own rounding to
//         64 bits: 0.53 measured below t d = 64).
//
// The functions are host functions too: tests compare them with
// arbitrary-precision arithmetic on the CPU.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#include <cuda_runtime.h>
#define FX_HD __host__ __device__ __forceinline__
#else
#include <math.h>
#define FX_HD static inline
#endif

namespace mag {

#include "fx_table.inc"

typedef unsigned long long fx_u64;

constexpr int FX_MAX_DIM = 512;          // d^2 < 512 2^118 fits 128 bits

// Limbs by the dimension: a coordinate of fx_coord_bits(m) bits, q = hi 2^LB + lo
// with LB = fx_limb_of(m).  31 + 30 bits while four dimensions' products fit
// the 64-bit sums, 30 + 29 bits for 16 dimensions and, with the sums emptied
// every 16, any more.  The finer grid at m <= 4 is for the pairs too close for
// it (fx_close), which are common in few dimensions and cost their whole warp
// the FP64 differences: the generation of the 8-component cloud of 16,384 points
// in R^3 takes 2.35 ms with 59 bits, 1.64 with 61.
constexpr int FX_LOW_DIM = 4;
constexpr int FX_SPILL = 16;
FX_HD int fx_limb_of(int m) { return m <= FX_LOW_DIM ? 31 : 30; }
FX_HD int fx_coord_bits(int m) { return 2 * fx_limb_of(m) - 1; }

struct fx_coord {
  int lo, hi;
};

// t and the coordinates' scale 2^-e as the exponential takes them.
struct FxScale {
  fx_u64 g;     // 256 t / ln 2 = g 2^-63 2^kg, 2^63 <= g < 2^64
  int kg;
  int e;        // a quantized coordinate unit is 2^-e
  float t63;    // t 2^(63 - e) in FP32 (range test of the FP32 path)
};

// ------------------------------------------------------------- primitives
FX_HD uint32_t fx_mulhi(uint32_t a, uint32_t b) {
#ifdef __CUDA_ARCH__
  return __umulhi(a, b);
#else
  return (uint32_t)(((fx_u64)a * b) >> 32);
#endif
}
// upper 32 bits of (hi:lo) << s and lower 32 bits of (hi:lo) >> s, 0 <= s < 32
FX_HD uint32_t fx_shl(uint32_t lo, uint32_t hi, int s) {
#ifdef __CUDA_ARCH__
  return __funnelshift_l(lo, hi, s);
#else
  return (uint32_t)((((((fx_u64)hi) << 32) | lo) << s) >> 32);
#endif
}
FX_HD int fx_clz(uint32_t a) {
#ifdef __CUDA_ARCH__
  return __clz((int)a);
#else
  return a ? __builtin_clz(a) : 32;
#endif
}
FX_HD float fx_float(uint32_t b) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(b);
#else
  union { uint32_t u; float f; } x;
  x.u = b;
  return x.f;
#endif
}
FX_HD uint32_t fx_bits(float v) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(v);
#else
  union { uint32_t u; float f; } x;
  x.f = v;
  return x.u;
#endif
}
FX_HD float fx_rsqrt(float v) {
#ifdef __CUDA_ARCH__
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
  return r;
#else
  return 1.0f / sqrtf(v);
#endif
}
FX_HD uint32_t fx_hi(fx_u64 a) { return (uint32_t)(a >> 32); }
FX_HD uint32_t fx_lo(fx_u64 a) { return (uint32_t)a; }
FX_HD fx_u64 fx_make(uint32_t lo, uint32_t hi) { return ((fx_u64)hi << 32) | lo; }

// -------------------------------------------------------------- distances
// The three limb sums of a pair's d^2 (Bx signed).
struct FxSums {
  fx_u64 A, C;
  long long Bx;
};
FX_HD void fx_clear(FxSums& s) { s.A = 0, s.C = 0, s.Bx = 0; }
FX_HD void fx_accumulate(FxSums& s, fx_coord a, fx_coord b) {
  const int dl = a.lo - b.lo, dh = a.hi - b.hi;
  s.A += (fx_u64)((long long)dl * dl);
  s.Bx += (long long)dh * dl;
  s.C += (fx_u64)((long long)dh * dh);
}
// d^2 = (qh:ql) in units of 2^-2e
struct FxSquare {
  fx_u64 h, l;
};
FX_HD void fx_square_clear(FxSquare& q) { q.h = 0, q.l = 0; }
// q += C 2^(2 LB) + Bx 2^(LB + 1) + A
template <int LB>
FX_HD void fx_add(FxSquare& q, const FxSums& s) {
  fx_u64 l = q.l + s.A;
  fx_u64 h = q.h + (l < s.A ? 1 : 0);
  const fx_u64 bl = (fx_u64)s.Bx << (LB + 1);
  l += bl;
  h += (fx_u64)(s.Bx >> (63 - LB)) + (l < bl ? 1 : 0);
  const fx_u64 cl = s.C << (2 * LB);
  l += cl;
  h += (s.C >> (64 - 2 * LB)) + (l < cl ? 1 : 0);
  q.h = h, q.l = l;
}
// Pairs this close (d < sqrt(m) 2^(53-e)) take the FP64 differences.
FX_HD bool fx_close(const FxSquare& q, int m) { return q.h < ((fx_u64)m << 42); }

// d = s 2^-62 2^(j - e) with 2^62 <= s <= 2^63, of a pair that is not close; sf
// = the FP32 start value of s 2^-62 (relative error below 2^-21).
struct FxRoot {
  fx_u64 v;      // d^2's leading bits, v 2^-63 in [1, 2)
  int par, j;
  float y, sf;   // 1/sqrt, sqrt
};
FX_HD FxRoot fx_root_start(const FxSquare& q) {
  FxRoot r;
  const uint32_t w3 = fx_hi(q.h), w2 = fx_lo(q.h), w1 = fx_hi(q.l);
  const int lz = fx_clz(w3);  // < 32: not close, so q.h >= 2^42
  r.v = fx_make(fx_shl(w1, w2, lz), fx_shl(w2, w3, lz));
  r.par = (lz + 1) & 1;
  r.j = (127 - lz - r.par) >> 1;
  const float f = fx_float(((fx_hi(r.v) >> 8) & 0x7fffffu) | ((uint32_t)(127 + r.par) << 23));
  r.y = fx_rsqrt(f);
  r.sf = f * r.y;
  return r;
}
// FP32 to the nearest integer below 2^22 by the magic constant
FX_HD int fx_small_int(float v) { return (int)(fx_bits(v + 12582912.0f) - 0x4B400000u); }
FX_HD int fx_int(float v) {
#ifdef __CUDA_ARCH__
  return __float2int_rn(v);
#else
  return (int)lrintf(v);
#endif
}
FX_HD fx_u64 fx_root(const FxRoot& r) {
  const uint32_t s0 = fx_bits(r.sf + 2.0f) - 0x40000000u;  // sf 2^22
  const fx_u64 v61 = r.v >> (2 - r.par);                   // v 2^par scaled by 2^61
  const long long r0 = (long long)(v61 - (((fx_u64)s0 * s0) << 17));  // below 2^42.5
  const int c0 = fx_int((float)(int)(r0 >> 19) * r.y);
  const fx_u64 s1 = ((fx_u64)s0 << 21) + (long long)c0;    // scale 2^43, within 2^-42
  const uint32_t l = fx_lo(s1), h = fx_hi(s1);
  const fx_u64 sq = (fx_u64)l * l + ((fx_u64)(2u * h * l) << 32);  // s1^2 mod 2^64
  const long long r1 = (long long)((r.v << (23 + r.par)) - sq);    // scale 2^86, below 2^46
  const int c1 = fx_small_int((float)(int)((r1 + (1 << 23)) >> 24) * (0.5f * r.y));
  return (s1 << 19) + (long long)c1;                       // scale 2^62
}
// d as FP64 bits; s + half may reach 2^63: the carry moves the exponent
FX_HD fx_u64 fx_dist_bits(fx_u64 s, int j, int e) {
  return ((fx_u64)(uint32_t)(j - e + 1022) << 52) + ((s + 0x200u) >> 10);
}

// ------------------------------------------------------------ exponential
// a b for 64-bit a, b: the high 64 bits and the 32 below them.
FX_HD fx_u64 fx_mul(fx_u64 a, fx_u64 b, uint32_t* below) {
  const uint32_t al = fx_lo(a), ah = fx_hi(a), bl = fx_lo(b), bh = fx_hi(b);
  const fx_u64 t = (fx_u64)al * bh + fx_mulhi(al, bl);
  const fx_u64 u = (fx_u64)ah * bl + fx_lo(t);
  *below = fx_lo(u);
  return (fx_u64)ah * bh + fx_hi(t) + fx_hi(u);
}
// high 64 bits of a b, up to 2 units low
FX_HD fx_u64 fx_mul_low(fx_u64 a, fx_u64 b) {
  const uint32_t ah = fx_hi(a), bh = fx_hi(b);
  return (fx_u64)ah * bh + fx_mulhi(ah, fx_lo(b)) + fx_mulhi(fx_lo(a), bh);
}

// exp(-t d) = z 2^-63 2^-shift, z in (0.49, 1] 2^63, for d = dm 2^-62 2^kd (dm
// <= 2^63; normalized, 2^62 <= dm, for full accuracy), t as in FxScale (g,
// kg), k = kd + kg; T: the table.
FX_HD fx_u64 fx_exp_fixed(fx_u64 dm, int k, fx_u64 g, const fx_u64* T, int* shift) {
  uint32_t below;
  const fx_u64 H = fx_mul(dm, g, &below);  // 256 t d / ln 2 = H 2^(k - 61)
  const int q = k + 3;
  uint32_t N, fh, fl;
  if (q < 0) {
    const fx_u64 f = q > -64 ? H >> -q : 0;
    N = 0;
    fh = fx_hi(f), fl = fx_lo(f);
  } else {
    // past FP64's range (dm normalized: N >= 2^20): any large N
    N = q > 24 ? 0x100000u : fx_shl(fx_hi(H), 0u, q);
    fh = fx_shl(fx_lo(H), fx_hi(H), q & 31);
    fl = fx_shl(below, fx_lo(H), q & 31);
  }
  const fx_u64 R = fx_mul_low(fx_make(fl, fh), FX_LN2);              // r, scale 2^72
  const uint32_t Rh = fx_hi(R);                                      // 2^40
  const fx_u64 R2 = (fx_u64)Rh * Rh + 2ull * fx_mulhi(Rh, fx_lo(R)); // r^2, 2^80
  const uint32_t R2h = fx_hi(R2);                                    // 2^48
  const uint32_t W = 2863311531u - fx_mulhi(Rh, 2796203u) + fx_mulhi(R2h, 2185u);  // 1/6 - r/24 + r^2/120, 2^34
  // r^3, 2^57; the unit makes up for the three truncations on average
  const uint32_t R3 = (uint32_t)(((fx_u64)R2h * Rh) >> 31) + 1u;
  const fx_u64 p = R - (R2 >> 9) + (((fx_u64)R3 * W) >> 19);         // 1 - exp(-r), 2^72
  const fx_u64 t = T[N & (FX_TABLE_SIZE - 1)];
  *shift = (int)(N >> 8);
  return t - (fx_mul_low(t, p) >> 8);
}
// z 2^-63 2^-shift rounded to FP64 (z in (0.25, 1] 2^63), 0 below FP64's
// normal range
FX_HD fx_u64 fx_pack(fx_u64 z, int shift) {
  const uint32_t zh = fx_hi(z);
  const int s = (zh >> 31) ? 0 : ((zh >> 30) ? 1 : 2);
  const uint32_t mh = fx_shl(fx_lo(z), zh, s), ml = fx_lo(z) << s;
  const int ex = 1022 - s - shift;
  if (ex < 1) return 0;
  const fx_u64 m = (fx_make(ml, mh) >> 11) + ((ml >> 10) & 1u);
  return ((fx_u64)(uint32_t)ex << 52) + m;
}
// 1 / (s 2^-62) in units of 2^-63 for 2^62 <= s <= 2^63, from its FP32 value y
// (relative error below 2^-21): q0 = y, r = 1 - s q0 exact, q0 (1 + r + r^2);
// within 2^-59.
FX_HD fx_u64 fx_recip(fx_u64 s, float y) {
  const uint32_t q0 = fx_bits(y + 1.0f) - 0x3f800000u;  // y 2^23
  const long long r = -(long long)((s >> 2) * q0);      // 1 - s q0, scale 2^83 (mod 2^64)
  const int rh = (int)(r >> 32);
  const long long p = r + (long long)((fx_u64)((long long)rh * rh) >> 19);
  const long long hi = (long long)(int)(p >> 32) * (long long)q0;  // scale 2^74 above the low half
  return ((fx_u64)q0 << 40) + (fx_u64)(hi >> 11) + (((fx_u64)fx_lo((fx_u64)p) * q0) >> 43);
}
// z 2^-63 2^-shift rounded to FP64 for any z > 0 with its leading bit in the
// high word
FX_HD fx_u64 fx_pack_any(fx_u64 z, int shift) {
  const int s = fx_clz(fx_hi(z));
  const uint32_t mh = fx_shl(fx_lo(z), fx_hi(z), s), ml = fx_lo(z) << s;
  const int ex = 1022 - s - shift;
  if (ex < 1) return 0;
  return ((fx_u64)(uint32_t)ex << 52) + (fx_make(ml, mh) >> 11) + ((ml >> 10) & 1u);
}
// The same rounded to FP32 (z in (0.25, 1] 2^63): the conversion rounds 32 bits
// with the rest as a sticky bit, z's own error being far below it.  0 below
// 2^-125, where the exponent field would run out.
FX_HD float fx_float_of(fx_u64 z, int shift) {
  if (shift >= 124) return 0.0f;
#ifdef __CUDA_ARCH__
  const float f = __uint2float_rn(fx_hi(z) | 1u);
#else
  const float f = (float)(fx_hi(z) | 1u);
#endif
  return fx_float(fx_bits(f) - ((uint32_t)(31 + shift) << 23));
}
FX_HD fx_u64 fx_exp_neg(fx_u64 dm, int k, fx_u64 g, const fx_u64* T) {
  int shift;
  const fx_u64 z = fx_exp_fixed(dm, k, g, T, &shift);
  return fx_pack(z, shift);
}
// The same from FP64 d >= 0, finite.
FX_HD fx_u64 fx_exp_neg_d(fx_u64 dbits, int kg, fx_u64 g, const fx_u64* T) {
  const int ex = (int)(dbits >> 52);
  const fx_u64 frac = dbits & 0xfffffffffffffull;
  return fx_exp_neg((ex ? frac | 0x10000000000000ull : frac) << 10, (ex ? ex : 1) - 1023 + kg, g, T);
}
// d^2 = (h:l) 2^-2e rounded to FP64 (h > 0)
FX_HD fx_u64 fx_square_bits(const FxSquare& q, int e) {
  int lz = 0;
  fx_u64 h = q.h, l = q.l;
  while (!(h >> 63)) h = (h << 1) | (l >> 63), l <<= 1, ++lz;
  const fx_u64 rest = h & 0x7ffull;
  fx_u64 m = h >> 11;
  if ((rest >> 10) && ((rest & 0x3ffull) || l || (m & 1))) ++m;
  return ((fx_u64)(uint32_t)(127 - lz - 2 * e + 1022) << 52) + m;
}

// ------------------------------------------------------------------- host
// 256 t / ln 2 = g 2^-63 2^kg for t > 0: the product of t's significand with
// 128 bits of log2 e, rounded to 64.
inline void fx_scale_t(double t, fx_u64* g, int* kg) {
  union { double d; fx_u64 u; } x;
  x.d = t;
  int ex = (int)(x.u >> 52) & 0x7ff;
  fx_u64 m = x.u & 0xfffffffffffffull;
  if (ex == 0) {  // subnormal: normalize
    ex = 1;
    while (!(m >> 52)) m <<= 1, --ex;
  } else {
    m |= 1ull << 52;
  }
  m <<= 11;  // t = m 2^-63 2^(ex - 1023)
  // log2 e = LOG2E_HI 2^-63 + ..., in [1, 2): p in [2^126, 2^128)
  unsigned __int128 p = (unsigned __int128)m * FX_LOG2E_HI + (((unsigned __int128)m * FX_LOG2E_LO) >> 64);
  const int up = (int)(p >> 127);
  p += (unsigned __int128)1 << (up ? 63 : 62);  // far below a carry out: m is a multiple of 2^11
  const fx_u64 h = (fx_u64)(p >> (up ? 64 : 63));
  *g = h;
  *kg = ex - 1023 + 8 + up;
}
inline FxScale fx_scale(double t, int e) {
  FxScale s;
  fx_scale_t(t, &s.g, &s.kg);
  s.e = e;
  s.t63 = (float)ldexp(t, 63 - e);
  return s;
}

#ifdef __CUDACC__
// ----------------------------------------------------------------- kernels
static __device__ const fx_u64 kFxTable[FX_TABLE_SIZE] = {FX_TABLE_ENTRIES};

__device__ __forceinline__ void load_fx_table(fx_u64* tab) {
  for (int i = threadIdx.x; i < FX_TABLE_SIZE; i += blockDim.x) tab[i] = kFxTable[i];
}

// The pairs of one 128 x 128 tile (rows row0 .., columns col0 .. of the n
// quantized points Xq), THREADS threads (NW warps): f(r, q) is called once for
// every row r = warp + NW i of the tile with the squares q[4] of the lane's columns 4 lane ..
// 4 lane + 3.  KIND: 0 for m <= FX_LOW_DIM, 1 for m <= FX_SPILL, 2 beyond.
// Beyond FX_SPILL two rows are accumulated together, where the column reads
// would set the pace; below, one (they hide behind the finishing work).  smem:
// fx_tile_smem bytes.  slice of slices (1, 2 or 4): that part of the rows only.
constexpr int FX_THREADS = 256;
inline int fx_kind(int m) { return m <= FX_LOW_DIM ? 0 : (m <= FX_SPILL ? 1 : 2); }
// CTAs per SM the kernels over tiles are compiled for: one row at a time fits
// 80 registers, and three CTAs hide more of the multiplier's latency than two
// (n = 16,384, m = 8: 1.79 against 1.95 ms); two rows need 128.
constexpr int fx_ctas(int kind) { return kind < 2 ? 3 : 2; }
constexpr int FX_CHUNK = 32;  // dimensions staged at a time
// A kernel's limit on dynamic shared memory is the process's, not the call's: every
// launch sets it to what its largest m takes, so that a call from another thread
// cannot lower it between this one's setting and its launch.
constexpr size_t FX_TILE_SMEM_MAX = 2 * (size_t)128 * FX_CHUNK * sizeof(fx_coord);
inline size_t fx_tile_smem(int m) { return 2 * (size_t)128 * (m < FX_CHUNK ? m : FX_CHUNK) * sizeof(fx_coord); }

template <int KIND, int THREADS = FX_THREADS, class F>
__device__ __forceinline__ void fx_tile_pairs(const fx_coord* __restrict__ Xq, int64_t n, int m, int64_t row0,
                                              int64_t col0, fx_coord* smem, F&& f, int slice = 0, int slices = 1) {
  constexpr int R = KIND < 2 ? 1 : 2, LB = KIND == 0 ? 31 : 30, NW = THREADS / 32;
  const int mc = m < FX_CHUNK ? m : FX_CHUNK;
  fx_coord* xr = smem;              // [128][mc] row points (broadcast reads)
  fx_coord* xc = smem + 128 * mc;   // [mc][128]: column 4 l + q at 32 q + l (conflict free)
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  auto stage = [&](int l0, int cnt) {
    for (int e = threadIdx.x; e < 128 * cnt; e += THREADS) {
      const int r = e / cnt, l = e - r * cnt;
      const int64_t gr = row0 + r, gc = col0 + r;
      xr[r * mc + l] = gr < n ? Xq[gr * m + l0 + l] : fx_coord{0, 0};
      xc[l * 128 + 32 * (r & 3) + (r >> 2)] = gc < n ? Xq[gc * m + l0 + l] : fx_coord{0, 0};
    }
  };
  if (R == 1 || m <= FX_CHUNK) {
    stage(0, m);
    __syncthreads();
  }
#pragma unroll 1
  for (int i = 128 / NW * slice / slices; i < 128 / NW * (slice + 1) / slices; i += R) {
    FxSquare q[R][4];
    FxSums s[R][4];
#pragma unroll
    for (int k = 0; k < R; ++k)
#pragma unroll
      for (int c = 0; c < 4; ++c) fx_square_clear(q[k][c]), fx_clear(s[k][c]);
#pragma unroll 1
    for (int l0 = 0; l0 < m; l0 += FX_CHUNK) {
      const int cnt = m - l0 < mc ? m - l0 : mc;
      if (R > 1 && m > FX_CHUNK) {
        __syncthreads();
        stage(l0, cnt);
        __syncthreads();
      }
      const fx_coord* xrow = xr + (warp + NW * i) * mc;
#pragma unroll 1
      for (int la = 0; la < cnt; la += FX_SPILL) {
        const int lb = cnt - la < FX_SPILL ? cnt : la + FX_SPILL;
#pragma unroll 2
        for (int l = la; l < lb; ++l) {
          fx_coord b[4];
#pragma unroll
          for (int c = 0; c < 4; ++c) b[c] = xc[l * 128 + 32 * c + lane];
#pragma unroll
          for (int k = 0; k < R; ++k) {
            const fx_coord a = xrow[NW * k * mc + l];
#pragma unroll
            for (int c = 0; c < 4; ++c) fx_accumulate(s[k][c], a, b[c]);
          }
        }
#pragma unroll
        for (int k = 0; k < R; ++k)
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            fx_add<LB>(q[k][c], s[k][c]);
            if (R > 1) fx_clear(s[k][c]);
          }
      }
    }
#pragma unroll 1
    for (int k = 0; k < R; ++k) {
      f(warp + NW * (i + k), q[0]);
      if (R > 1) {
#pragma unroll
        for (int c = 0; c < 4; ++c) q[0][c] = q[R - 1][c];
      }
    }
  }
}
#endif  // __CUDACC__

}  // namespace mag
