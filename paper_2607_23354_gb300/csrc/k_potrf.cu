// K2 diagonal tile, FP32: L = chol(A) of one 128 x 128 tile, inv(L) and its
// transpose, by one CTA.  The tile sits on the factor's critical path (one
// call per tile column), so the kernel is built around its dependence chain,
// not around its 1.4 MFLOP.
//
// One elimination of the 256 x 128 matrix [A; I]: the column operations that
// turn A into L turn I into L^{-T}, so W = inv(L)^T needs no pass of its own.
// It runs in four panels of 32 columns.  In panel kb five 32-row blocks take
// part -- A's blocks kb..3 and W's blocks 0..kb (a block of W is zero before
// its own panel) -- each held by one warp, one row per lane in registers.
// Columns are eliminated four at a time: every lane of the diagonal warp
// forms the 4 x 4 Cholesky factor of the pivot block itself, scales its own
// four entries and publishes them with one 16-byte store; the other warps
// follow one pivot block behind on named barriers that the diagonal warp only
// arrives at.  The chain from one pivot block to the next stays in registers:
// the next block's old entries are fetched by shuffles ahead of time, its
// four rows of the new columns by sixteen more, and the four pivots take two
// rounds of reciprocal square roots (a pivot pair's second one from the 2 x 2
// determinant, beside the first).  The row registers rotate by four per pivot
// block, which keeps the body a short loop.
//
// The trailing update, C -= P Q^T with K = 32, runs on the tensor cores as
// mma.sync BF16 with each operand split into three BF16 parts (24 bits) and
// the six products down to 2^-18: FP32-class products, and 7 times fewer
// shared-memory wavefronts than register-tiled FP32 FMAs, which took 3,200
// cycles a panel against 1,400-1,900 and starved the panel's own loads beside
// them.  The splits are written once, by the warps that finish the rows.
// Eleven more warps take what the next panel does not need: the rest of the
// previous panel's trailing update and the write-out of finished columns.
//
// Bound: latency.  Of 32,000 cycles the chain of 32 pivot blocks takes
// 23,000 (about 430 a block, 700 where 16 or more columns remain: a 16-byte
// broadcast read returns to the registers at 32 bytes a cycle), the three
// trailing updates 5,500.  One lane scaling and publishing a column at a time,
// with warp-serial block inverses and register-tiled FP32 block products, took
// 107,000.  57 us a launch before, 22 now (event to event, alone); a solve of
// n = 16384 points in R^3 22.8 ms before, 17.2 with it alone.  Backward error of a tile's
// factor: 1.1e-7 of ||Z|| before, 0.7e-7 now (Z of [0,1]^8, t = 1).
#include <cuda_bf16.h>

#include "mag_internal.cuh"

namespace mag {

namespace {

constexpr int PB = 32;            // panel width, block edge
constexpr int NPB = TILE / PB;    // 4
constexpr int LDP = TILE + 4;     // row stride (floats): 16-byte aligned rows, 8 rows cover all banks
constexpr int LDS = 20;           // row stride of a split panel (32-bit pairs): fragment reads free of conflicts
constexpr int POTRF_THREADS = 512;
constexpr int PANEL_WARPS = NPB + 1;
constexpr int BG_WARPS = POTRF_THREADS / 32 - PANEL_WARPS;

struct PotrfSmem {
  float M[2 * TILE * LDP];          // rows 0..127: the tile, becoming L; rows 128 + c: W[c][r] = inv(L)[r][c]
  uint32_t split[2][3][TILE * LDS]; // a panel's rows below its diagonal block as BF16 pairs, by panel parity and part
  float rinv[TILE];                 // 1 / L[c][c]
};

__device__ __forceinline__ float rsqrt_ftz(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
// r ~ 1 / sqrt(p) improved by one Newton step; e (half the seed's relative
// error in p r^2) returned for the test of the seed
__device__ __forceinline__ float rsqrt_newton(float p, float r, float* e) {
  *e = fmaf(-0.5f * p * r, r, 0.5f);
  return fmaf(r, *e, r);
}
__device__ __forceinline__ void bar_sync(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void bar_arrive(int id, int threads) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// The 4 x 4 factor of one pivot block: reciprocal square roots of the pivots
// and the entries below the diagonal.
struct Pivot {
  float r0, r1, r2, r3, l10, l20, l30, l21, l31, l32;
  int bad;  // bit i: pivot i is not positive
};

// The factor with the second pivots' roots from the seeds s1, s3 (PAIRED: of the
// pairs' determinants) or from the pivots themselves.  True where both seeds are
// within 2^-11 of the pivots'.
template <bool PAIRED>
__device__ __forceinline__ bool pivot_steps(float d00, float d10, float d20, float d30, float d11, float d21, float d31,
                                            float d22, float d32, float d33, Pivot& q) {
  constexpr float kMinPivot = 1.17549435e-38f, kSeed = 0x1p-12f;
  float e0, e1, e2, e3;
  const float s0 = rsqrt_ftz(d00), s1 = PAIRED ? rsqrt_ftz(fmaf(d00, d11, -d10 * d10)) : 0.0f;
  q.r0 = rsqrt_newton(d00, s0, &e0);
  q.l10 = d10 * q.r0, q.l20 = d20 * q.r0, q.l30 = d30 * q.r0;
  const float p1 = fmaf(-q.l10, q.l10, d11);
  q.r1 = rsqrt_newton(p1, PAIRED ? (d00 * s0) * s1 : rsqrt_ftz(p1), &e1);
  q.l21 = fmaf(-q.l20, q.l10, d21) * q.r1, q.l31 = fmaf(-q.l30, q.l10, d31) * q.r1;
  const float p2 = fmaf(-q.l21, q.l21, fmaf(-q.l20, q.l20, d22));
  const float s32 = fmaf(-q.l31, q.l21, fmaf(-q.l30, q.l20, d32));
  const float s33 = fmaf(-q.l31, q.l31, fmaf(-q.l30, q.l30, d33));
  const float s2 = rsqrt_ftz(p2), s3 = PAIRED ? rsqrt_ftz(fmaf(p2, s33, -s32 * s32)) : 0.0f;
  q.r2 = rsqrt_newton(p2, s2, &e2);
  q.l32 = s32 * q.r2;
  const float p3 = fmaf(-q.l32, q.l32, s33);
  q.r3 = rsqrt_newton(p3, PAIRED ? (p2 * s2) * s3 : rsqrt_ftz(p3), &e3);
  q.bad = (int)!(d00 >= kMinPivot) | (int)!(p1 >= kMinPivot) << 1 | (int)!(p2 >= kMinPivot) << 2 |
          (int)!(p3 >= kMinPivot) << 3;
  return fabsf(e1) < kSeed && fabsf(e3) < kSeed;
}

// A pivot that is not positive, or below FP32's normal range, is reported;
// the entries after it are then meaningless (NaN or infinite) and the factor
// is dropped.  A pair's second pivot d11 - d10^2 / d00 is first approximated as
// 1 / sqrt = sqrt(d00) / sqrt(d00 d11 - d10^2), so that both roots start
// together, and a Newton step takes it to the pivot itself, the entry that is
// scaled and judged.  The two round apart: where the pivot has cancelled so far
// that they differ by 2^-11 or more (or in sign), the block starts again from the
// pivots.  The arguments are the same in every lane.
__device__ __forceinline__ void pivot_factor(float d00, float d10, float d20, float d30, float d11, float d21,
                                             float d31, float d22, float d32, float d33, Pivot& q) {
  if (!pivot_steps<true>(d00, d10, d20, d30, d11, d21, d31, d22, d32, d33, q))
    pivot_steps<false>(d00, d10, d20, d30, d11, d21, d31, d22, d32, d33, q);
}

// x - y z
__device__ __forceinline__ float fnma(float y, float z, float x) { return fmaf(-y, z, x); }

// a[c] <- a[c + 4] - x . L[row j + 4 + c][j .. j + 3] for c in [C0, C1):
// Lj points at row 0 of the panel's diagonal block, column j (broadcast
// reads).  Columns past the panel's end repeat rows 28 .. 31 and are never
// used.
template <int C0, int C1>
__device__ __forceinline__ void update_rotate(float* a, const float* Lj, int j, float x0, float x1, float x2,
                                              float x3) {
#pragma unroll
  for (int c4 = C0; c4 < C1; c4 += 4) {
    const float* Lq = Lj + min(j + 4 + c4, PB - 4) * LDP;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const float4 v = *reinterpret_cast<const float4*>(Lq + c * LDP);
      a[c4 + c] = fnma(x3, v.w, fnma(x2, v.z, fnma(x1, v.y, fnma(x0, v.x, a[c4 + c + 4]))));
    }
  }
}

// Two FP32 values as three BF16 pairs: x = p1 + p2 + p3 up to 2^-24 |x|.
__device__ __forceinline__ uint32_t bf16_pair(float lo, float hi) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}
__device__ __forceinline__ void split3(float x, float y, uint32_t& p1, uint32_t& p2, uint32_t& p3) {
  p1 = bf16_pair(x, y);
  x -= __uint_as_float(p1 << 16), y -= __uint_as_float(p1 & 0xffff0000u);
  p2 = bf16_pair(x, y);
  x -= __uint_as_float(p2 << 16), y -= __uint_as_float(p2 & 0xffff0000u);
  p3 = bf16_pair(x, y);
}

// GN pivot blocks from block g0 on with WIDTH columns left behind the first:
// the diagonal block's warp.  q: the first block's factor on entry, the next
// one's on return.
template <int GN, int WIDTH>
__device__ __forceinline__ void diag_steps(PotrfSmem& S, float* a, Pivot& q, int o, int g0, float* own, int lane,
                                           int64_t K, DevStatus* st) {
  const unsigned full = 0xffffffffu;
#pragma unroll 1
  for (int g = g0; g < g0 + GN; ++g) {
    const int j = 4 * g, jn = j + 4;
    // the next pivot block before this update (beyond the panel: unused)
    float d00 = __shfl_sync(full, a[4], jn), d10 = __shfl_sync(full, a[4], jn + 1);
    float d20 = __shfl_sync(full, a[4], jn + 2), d30 = __shfl_sync(full, a[4], jn + 3);
    float d11 = __shfl_sync(full, a[5], jn + 1), d21 = __shfl_sync(full, a[5], jn + 2);
    float d31 = __shfl_sync(full, a[5], jn + 3), d22 = __shfl_sync(full, a[6], jn + 2);
    float d32 = __shfl_sync(full, a[6], jn + 3), d33 = __shfl_sync(full, a[7], jn + 3);
    const float x0 = a[0] * q.r0;
    const float x1 = fnma(x0, q.l10, a[1]) * q.r1;
    const float x2 = fnma(x1, q.l21, fnma(x0, q.l20, a[2])) * q.r2;
    const float x3 = fnma(x2, q.l32, fnma(x1, q.l31, fnma(x0, q.l30, a[3]))) * q.r3;
    // entries above the diagonal are left as they come; nothing reads them
    *reinterpret_cast<float4*>(own + j) = make_float4(x0, x1, x2, x3);
    if (lane == 0) *reinterpret_cast<float4*>(S.rinv + o + j) = make_float4(q.r0, q.r1, q.r2, q.r3);
    __syncwarp();
    bar_arrive(1 + g, 32 * PANEL_WARPS);
    if (q.bad && lane == 0) {
      atomicOr(&st->flags, ST_NOTPD);
      atomicMin(&st->notpd_index, (int)(K * TILE + o + j) + __ffs(q.bad));
    }
    if (jn < PB) {
      // the new columns' rows jn .. jn + 3, to every lane
      float u[4][4];
#pragma unroll
      for (int c = 0; c < 4; ++c) u[c][0] = __shfl_sync(full, x0, jn + c);
#pragma unroll
      for (int c = 0; c < 4; ++c) u[c][1] = __shfl_sync(full, x1, jn + c);
#pragma unroll
      for (int c = 0; c < 4; ++c) u[c][2] = __shfl_sync(full, x2, jn + c);
#pragma unroll
      for (int c = 0; c < 4; ++c) u[c][3] = __shfl_sync(full, x3, jn + c);
      const float xs[4] = {x0, x1, x2, x3};
#pragma unroll
      for (int c = 0; c < 4; ++c) a[c] = a[c + 4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        d00 = fnma(u[0][i], u[0][i], d00), d10 = fnma(u[1][i], u[0][i], d10);
        d20 = fnma(u[2][i], u[0][i], d20), d30 = fnma(u[3][i], u[0][i], d30);
        d11 = fnma(u[1][i], u[1][i], d11), d21 = fnma(u[2][i], u[1][i], d21);
        d31 = fnma(u[3][i], u[1][i], d31), d22 = fnma(u[2][i], u[2][i], d22);
        d32 = fnma(u[3][i], u[2][i], d32), d33 = fnma(u[3][i], u[3][i], d33);
#pragma unroll
        for (int c = 0; c < 4; ++c) a[c] = fnma(xs[i], u[c][i], a[c]);
      }
      pivot_factor(d00, d10, d20, d30, d11, d21, d31, d22, d32, d33, q);
      update_rotate<4, WIDTH>(a, S.M + o * LDP + o + j, j, x0, x1, x2, x3);
    }
  }
}

// The same steps of a warp whose rows lie below the diagonal block (or in W):
// every finished row is also stored as its split parts (sp: this lane's row).
template <int GN, int WIDTH>
__device__ __forceinline__ void row_steps(PotrfSmem& S, float* a, int o, int g0, float* own, uint32_t* sp) {
#pragma unroll 1
  for (int g = g0; g < g0 + GN; ++g) {
    const int j = 4 * g;
    const float* Lj = S.M + o * LDP + o + j;  // the diagonal block's columns from j on
    bar_sync(1 + g, 32 * PANEL_WARPS);
    const float4 r = *reinterpret_cast<const float4*>(S.rinv + o + j);
    const float4 q1 = *reinterpret_cast<const float4*>(Lj + (j + 1) * LDP);
    const float4 q2 = *reinterpret_cast<const float4*>(Lj + (j + 2) * LDP);
    const float4 q3 = *reinterpret_cast<const float4*>(Lj + (j + 3) * LDP);
    const float x0 = a[0] * r.x;
    const float x1 = fnma(x0, q1.x, a[1]) * r.y;
    const float x2 = fnma(x1, q2.y, fnma(x0, q2.x, a[2])) * r.z;
    const float x3 = fnma(x2, q3.z, fnma(x1, q3.y, fnma(x0, q3.x, a[3]))) * r.w;
    *reinterpret_cast<float4*>(own + j) = make_float4(x0, x1, x2, x3);
    uint2 p1, p2, p3;
    split3(x0, x1, p1.x, p2.x, p3.x);
    split3(x2, x3, p1.y, p2.y, p3.y);
    *reinterpret_cast<uint2*>(sp + 2 * g) = p1;
    *reinterpret_cast<uint2*>(sp + TILE * LDS + 2 * g) = p2;
    *reinterpret_cast<uint2*>(sp + 2 * TILE * LDS + 2 * g) = p3;
    if (j + 4 < PB) update_rotate<0, WIDTH>(a, Lj, j, x0, x1, x2, x3);
  }
}

__device__ __forceinline__ void load_row(const float* own, float* a) {
#pragma unroll
  for (int c = 0; c < PB; c += 4) {
    const float4 v = *reinterpret_cast<const float4*>(own + c);
    a[c] = v.x, a[c + 1] = v.y, a[c + 2] = v.z, a[c + 3] = v.w;
  }
}

// d += a b, m16n8k16, BF16 operands (the PTX fragment layout).
__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// 16 x 16 outputs of the trailing update with panel kb: rows row0 .. + 15 of
// M, columns col0 .. + 15 (both multiples of 16; the split parts hold row r
// of M, r >= 32 (kb + 1), at r - 32 (kb + 1)).
__device__ __forceinline__ void trailing_job(PotrfSmem& S, int kb, int row0, int col0, int lane) {
  const int g = lane >> 2, t = lane & 3, base = (kb + 1) * PB;
  const uint32_t* sp = &S.split[kb & 1][0][0];
  const uint32_t* pa = sp + (row0 - base + g) * LDS + t;
  const uint32_t* pb = sp + (col0 - base + g) * LDS + t;
  // the leading products of each 16 columns and the small ones in
  // accumulators of their own, added with rounding to nearest at the end (the
  // tensor cores truncate a running sum)
  float lead[2][2][4], low[2][4];
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int i = 0; i < 4; ++i) lead[0][h][i] = lead[1][h][i] = low[h][i] = 0.0f;
#pragma unroll
  for (int k = 0; k < PB / 16; ++k) {
    uint32_t a[3][4], b[2][3][2];
#pragma unroll
    for (int p = 0; p < 3; ++p) {
      const uint32_t* q = pa + p * TILE * LDS + 8 * k;
      a[p][0] = q[0], a[p][1] = q[8 * LDS], a[p][2] = q[4], a[p][3] = q[8 * LDS + 4];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const uint32_t* r = pb + p * TILE * LDS + 8 * h * LDS + 8 * k;
        b[h][p][0] = r[0], b[h][p][1] = r[4];
      }
    }
    // smallest products first
#pragma unroll
    for (int s = 2; s >= 0; --s)
#pragma unroll
      for (int p = 0; p <= s; ++p)
#pragma unroll
        for (int h = 0; h < 2; ++h) mma_bf16(s ? low[h] : lead[k][h], a[p], b[h][s - p][0], b[h][s - p][1]);
  }
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      float2* c = reinterpret_cast<float2*>(S.M + (row0 + g + 8 * i) * LDP + col0 + 8 * h + 2 * t);
      float2 v = *c;
      v.x -= (lead[0][h][2 * i] + lead[1][h][2 * i]) + low[h][2 * i];
      v.y -= (lead[0][h][2 * i + 1] + lead[1][h][2 * i + 1]) + low[h][2 * i + 1];
      *c = v;
    }
}

// Write-outs, warp q of `of`.  Columns of block b: L's rows from block b on;
// inv(L)'s block row b and its transpose's block column b (from W).
__device__ __forceinline__ void write_l(const float* M, float* __restrict__ tile, int b, int q, int of, int lane) {
  // eight lanes a row (32 columns), four rows a pass
  const int c = b * PB + 4 * (lane & 7);
  for (int r = b * PB + 4 * q + (lane >> 3); r < TILE; r += 4 * of) {
    const float4 v = *reinterpret_cast<const float4*>(M + r * LDP + c);
    *reinterpret_cast<float4*>(tile + r * TILE + c) =
        make_float4(c <= r ? v.x : 0.0f, c + 1 <= r ? v.y : 0.0f, c + 2 <= r ? v.z : 0.0f, c + 3 <= r ? v.w : 0.0f);
  }
}
__device__ __forceinline__ void write_inv(const float* W, float* __restrict__ Y, float* __restrict__ YT, int b, int q,
                                          int of, int lane) {
  const int r = b * PB + 4 * (lane & 7);
  for (int c = 4 * (4 * q + (lane >> 3)); c < (b + 1) * PB; c += 16 * of) {
    float4 v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      v[i] = *reinterpret_cast<const float4*>(W + (c + i) * LDP + r);
      *reinterpret_cast<float4*>(YT + (c + i) * TILE + r) = v[i];
    }
    *reinterpret_cast<float4*>(Y + r * TILE + c) = make_float4(v[0].x, v[1].x, v[2].x, v[3].x);
    *reinterpret_cast<float4*>(Y + (r + 1) * TILE + c) = make_float4(v[0].y, v[1].y, v[2].y, v[3].y);
    *reinterpret_cast<float4*>(Y + (r + 2) * TILE + c) = make_float4(v[0].z, v[1].z, v[2].z, v[3].z);
    *reinterpret_cast<float4*>(Y + (r + 3) * TILE + c) = make_float4(v[0].w, v[1].w, v[2].w, v[3].w);
  }
}
// Zeros above the diagonal blocks (L, inv(L)) and below them (the transpose).
__device__ __forceinline__ void write_zeros(float* __restrict__ tile, float* __restrict__ Y, float* __restrict__ YT,
                                            int q, int of, int lane) {
  const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int r = q; r < TILE; r += of) {
    const int c = 4 * lane;
    if (c / PB > r / PB) {
      *reinterpret_cast<float4*>(tile + r * TILE + c) = z;
      *reinterpret_cast<float4*>(Y + r * TILE + c) = z;
    } else if (c / PB < r / PB) {
      *reinterpret_cast<float4*>(YT + r * TILE + c) = z;
    }
  }
}

// One tile: Y = inv(L), YT = inv(L)^T; K: the tile column (for the report of a
// pivot that is not positive).
__device__ __forceinline__ void potrf_tile(float* __restrict__ tile, float* __restrict__ Y, float* __restrict__ YT,
                                           int64_t K, DevStatus* st) {
  extern __shared__ __align__(16) unsigned char potrf_smem[];
  PotrfSmem& S = *reinterpret_cast<PotrfSmem*>(potrf_smem);
  float* W = S.M + TILE * LDP;
  const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
#pragma unroll
  for (int i = 0; i < TILE * TILE / 4 / POTRF_THREADS; ++i) {  // I's blocks on and above the diagonal
    const int e = tid + i * POTRF_THREADS, r = e >> 5, c = (e & 31) * 4;
    if (c / PB >= r / PB)
      *reinterpret_cast<float4*>(W + r * LDP + c) = make_float4(c == r ? 1.0f : 0.0f, c + 1 == r ? 1.0f : 0.0f,
                                                                c + 2 == r ? 1.0f : 0.0f, c + 3 == r ? 1.0f : 0.0f);
  }
  wait_previous();
  // set by earlier kernels of the stream: uniform across the CTA
  if (*(volatile int*)&st->flags & (ST_NOTPD | ST_NONFINITE | ST_DUPLICATE | ST_TIMEOUT)) return;
  // A's blocks on and below the diagonal
#pragma unroll
  for (int i = 0; i < TILE * TILE / 4 / POTRF_THREADS; ++i) {
    const int e = tid + i * POTRF_THREADS, r = e >> 5, c = (e & 31) * 4;
    if (c / PB <= r / PB)
      *reinterpret_cast<float4*>(S.M + r * LDP + c) = reinterpret_cast<const float4*>(tile)[e];
  }
  __syncthreads();

#pragma unroll 1
  for (int kb = 0; kb < NPB; ++kb) {
    const int o = kb * PB;
    if (kb == NPB - 1) launch_next();  // the panel solve's set-up takes as long as the rest of this
    // the panel's row blocks in M: A's kb .. 3, then W's 0 .. kb (M's blocks
    // 4 .. 4 + kb): blocks kb + pw.  Warps 1, 2, 3 and 5 follow the diagonal
    // warp, away from its scheduler.
    const int pw = w < NPB ? w : (w == NPB + 1 ? NPB : -1);
    if (w == 0) {
      float* own = S.M + (o + lane) * LDP + o;
      float a[PB];
      load_row(own, a);
      const unsigned full = 0xffffffffu;
      Pivot q;
      pivot_factor(__shfl_sync(full, a[0], 0), __shfl_sync(full, a[0], 1), __shfl_sync(full, a[0], 2),
                   __shfl_sync(full, a[0], 3), __shfl_sync(full, a[1], 1), __shfl_sync(full, a[1], 2),
                   __shfl_sync(full, a[1], 3), __shfl_sync(full, a[2], 2), __shfl_sync(full, a[2], 3),
                   __shfl_sync(full, a[3], 3), q);
      // 28 columns remain behind the first pivot block, 12 behind the fifth
      diag_steps<4, 28>(S, a, q, o, 0, own, lane, K, st);
      diag_steps<4, 12>(S, a, q, o, 4, own, lane, K, st);
    } else if (pw > 0) {
      float* own = S.M + (o + pw * PB + lane) * LDP + o;
      uint32_t* sp = &S.split[kb & 1][0][((pw - 1) * PB + lane) * LDS];
      float a[PB];
      load_row(own, a);
      row_steps<4, 28>(S, a, o, 0, own, sp);
      row_steps<4, 12>(S, a, o, 4, own, sp);
    } else {
      const int bw = w == NPB ? 0 : w - PANEL_WARPS;
      if (kb == 0) {
        write_zeros(tile, Y, YT, bw, BG_WARPS, lane);
      } else {
        const int p = kb - 1;  // the finished panel
        // its trailing update beyond the current panel: column blocks jb > kb
        // of A's row blocks jb .. 3 and W's 0 .. p
        int job = bw;
#pragma unroll 1
        for (int jb = kb + 1; jb < NPB; ++jb) {
          const int jobs = 4 * (NPB - jb + p + 1);
          for (; job < jobs; job += BG_WARPS)
            trailing_job(S, p, jb * PB + 16 * (job >> 1), jb * PB + 16 * (job & 1), lane);
          job -= jobs;
        }
        write_l(S.M, tile, p, bw, BG_WARPS, lane);
        write_inv(W, Y, YT, p, bw, BG_WARPS, lane);
      }
    }
    __syncthreads();
    if (kb < NPB - 1) {
      // the next panel's columns: its four row blocks A kb + 1 .. 3, W 0 .. kb
      trailing_job(S, kb, (kb + 1) * PB + 16 * (w >> 1), (kb + 1) * PB + 16 * (w & 1), lane);
      __syncthreads();
    }
  }
  write_l(S.M, tile, NPB - 1, w, POTRF_THREADS / 32, lane);
  write_inv(W, Y, YT, NPB - 1, w, POTRF_THREADS / 32, lane);
}

__global__ void __launch_bounds__(POTRF_THREADS, 1)
    k_potrf_f32(float* __restrict__ Z, float* __restrict__ Dinv, float* __restrict__ DinvT, int64_t K, DevStatus* st) {
  potrf_tile(Z + tri_index(K, K) * TILE_ELEMS, Dinv + K * TILE_ELEMS, DinvT + K * TILE_ELEMS, K, st);
}

// Diagonal tile K of each of a batch's problems (one CTA each).
__global__ void __launch_bounds__(POTRF_THREADS, 1)
    k_potrf_batch(const TiledProblem* __restrict__ probs, float* __restrict__ Z, float* __restrict__ Dinv,
                  float* __restrict__ DinvT, int64_t K, DevStatus* st) {
  const TiledProblem& P = probs[blockIdx.x];
  potrf_tile(Z + (P.tile0 + tri_index(K, K)) * TILE_ELEMS, Dinv + (P.diag0 + K) * TILE_ELEMS,
             DinvT + (P.diag0 + K) * TILE_ELEMS, K, st + blockIdx.x);
}

}  // namespace

cudaError_t launch_potrf_f32(float* Z, float* Dinv, float* DinvT, int64_t K, DevStatus* st, cudaStream_t s) {
  cudaError_t e = cudaFuncSetAttribute(k_potrf_f32, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)sizeof(PotrfSmem));
  if (e != cudaSuccess) return e;
  e = launch_after(k_potrf_f32, dim3(1), dim3(POTRF_THREADS), sizeof(PotrfSmem), s, Z, Dinv, DinvT, K, st);
  if (e != cudaSuccess) return e;
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_potrf_batch(const TiledProblem* probs, int count, float* Z, float* Dinv, float* DinvT, int64_t K,
                               DevStatus* st, cudaStream_t s) {
  cudaError_t e = cudaFuncSetAttribute(k_potrf_batch, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)sizeof(PotrfSmem));
  if (e != cudaSuccess) return e;
  k_potrf_batch<<<(unsigned)count, POTRF_THREADS, sizeof(PotrfSmem), s>>>(probs, Z, Dinv, DinvT, K, st);
  note_launch();
  return cudaGetLastError();
}

}  // namespace mag
