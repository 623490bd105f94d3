// K8, tiled: a batch's problems of more than one factor block (n <= 2048)
// through the tile kernels together.  A column of 128 x 128 tiles is one launch
// over all problems that still have it, so a launch's CTAs are the tiles of
// hundreds of problems, where one CTA per problem leaves a 2048-point problem
// 40 ms on one SM.  Problems are sorted by decreasing n: those with a tile
// column J are a prefix.
//
//   k_bt_range, k_bt_quantize  fixed-point coordinates of the clouds (mag_fx.cuh)
//   k_bt_generate  Z's tiles: a cloud's distances once, the exponential for each
//                  of its problems; FP32 for the factor, 60-bit fixed point for
//                  the residual
//   per column J   k_bt_update (left-looking: tile -= sum_k L_Ik L_Jk^T),
//                  k_potrf_batch, k_bt_panel (L_IJ = A_IJ inv(L_JJ)^T)
//   k_bt_solve     one CTA per problem: residual norms, the refinement's
//                  decisions and the two triangular sweeps in FP32
//   k_bt_residual  Z w per tile in integers
//
// The factor's products are three FP16 products of split operands with FP32
// accumulators, the leading and the small products apart, read out and added in
// FP32 every 128 columns.
//
// Bound: the generator by the integer pipe, the update by the operands' path
// into shared memory (128 KB a product, 1 us), the residual by memory.
#include <algorithm>

#include "mag_fx.cuh"
#include "mag_internal.cuh"
#include "mag_math.cuh"
#include "mag_tc.cuh"

namespace mag {

namespace {

__device__ __forceinline__ bool stopped(const DevStatus* st) {
  return (*(volatile const int*)&st->flags & (ST_NOTPD | ST_NONFINITE | ST_DUPLICATE | ST_TIMEOUT)) != 0;
}

// --------------------------------------------------------------- quantize
__device__ __forceinline__ unsigned long long ordered_of(double v) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  return (b >> 63) ? ~b : b | 0x8000000000000000ull;
}

// Per dimension of a cloud the largest ~x and x in the ordered encoding (range,
// zeroed before), BQ_PARTS CTAs a cloud; bit 1 of cloud_flags for a coordinate
// that is not finite.
constexpr int BQ_THREADS = 512, BQ_PARTS = 8;

__global__ void __launch_bounds__(BQ_THREADS) k_bt_range(const double* __restrict__ points,
                                                         const TiledCloud* __restrict__ clouds,
                                                         int* __restrict__ cloud_flags,
                                                         unsigned long long* __restrict__ range) {
  static_assert(FX_MAX_DIM <= BQ_THREADS, "a thread stays on one dimension");
  __shared__ unsigned long long part[2][BQ_THREADS];
  const TiledCloud C = clouds[blockIdx.x];
  const double* X = points + C.point_offset;
  const int t = threadIdx.x, m = C.m, per = BQ_THREADS / m, l = t % m;
  unsigned long long lo = 0, hi = 0;
  bool bad = false;
  if (t < per * m) {
#pragma unroll 4
    for (int i = (int)blockIdx.y * per + t / m; i < C.n; i += BQ_PARTS * per) {
      const double v = X[i * m + l];
      const unsigned long long b = ordered_of(v);
      bad |= ((unsigned)__double2hiint(v) & 0x7ff00000u) == 0x7ff00000u;
      lo = ~b > lo ? ~b : lo;
      hi = b > hi ? b : hi;
    }
  }
  part[0][t] = lo;
  part[1][t] = hi;
  if (__syncthreads_or(bad) && t == 0) atomicOr(cloud_flags + C.flag, 1);
  if (t < m) {
    for (int k = t + m; k < per * m; k += m) {
      lo = part[0][k] > lo ? part[0][k] : lo;
      hi = part[1][k] > hi ? part[1][k] : hi;
    }
    atomicMax(range + C.range_offset + 2 * t, lo);
    atomicMax(range + C.range_offset + 2 * t + 1, hi);
  }
}

// A cloud's scale exponent and coordinates (the unit and limits of the single
// solver's).  cloud_flags: 2 every point the same, 4 no coordinates; problems of
// a flagged cloud are then stopped by their status.
__global__ void __launch_bounds__(BQ_THREADS) k_bt_quantize(const double* __restrict__ points,
                                                            TiledCloud* __restrict__ clouds,
                                                            TiledProblem* __restrict__ probs,
                                                            int* __restrict__ cloud_flags,
                                                            const unsigned long long* __restrict__ range,
                                                            fx_coord* __restrict__ Xq, DevStatus* __restrict__ st) {
  __shared__ double lo_s[FX_MAX_DIM], warp_s[BQ_THREADS / 32];
  const TiledCloud C = clouds[blockIdx.x];
  const double* X = points + C.point_offset;
  const int t = threadIdx.x, m = C.m, n = C.n;
  const bool first = blockIdx.y == 0;
  const bool bad = (cloud_flags[C.flag] & 1) != 0;  // k_bt_range's
  double S = 0.0;
  if (t < m) {
    const double lo = ordered_value(~range[C.range_offset + 2 * t]);
    lo_s[t] = lo;
    S = ordered_value(range[C.range_offset + 2 * t + 1]) - lo;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) S = fmax(S, __shfl_xor_sync(0xffffffffu, S, o));
  if ((t & 31) == 0) warp_s[t >> 5] = S;
  __syncthreads();
  for (int k = 0; k < BQ_THREADS / 32; ++k) S = fmax(S, warp_s[k]);
  int f = 0, e = 0;
  if (bad) {
    f = 1;
  } else if (!(S > 0.0)) {
    f = 2 | 4;
  } else if (!isfinite(S)) {
    f = 4;
  } else {
    e = fx_coord_bits(m) - (ilogb(S) + 1);
    if (e < -400 || e > 400) f = 4;
  }
  if (first) {
    if (t == 0) {
      clouds[blockIdx.x].e = e;
      if (f) atomicOr(cloud_flags + C.flag, f);
    }
    for (int p = t; p < C.nprob; p += BQ_THREADS) {
      if (f)
        atomicOr(&st[C.prob[p]].flags, ST_NONFINITE);
      else
        probs[C.prob[p]].t63 = (float)ldexp(probs[C.prob[p]].t, 63 - e);
    }
  }
  if (f) return;
  const int lb = fx_limb_of(m);
  fx_coord* out = Xq + C.xq_offset;
  const double scale = ldexp(1.0, e);
#pragma unroll 2
  for (int k = (int)blockIdx.y * BQ_THREADS + t; k < n * m; k += BQ_PARTS * BQ_THREADS) {
    // x - lo exactly as s + err (TwoSum), both rounded on the grid
    const double x = X[k], b = -lo_s[k % m];
    const double s = x + b;
    const double bv = s - x;
    const double err = (x - (s - bv)) + (b - bv);
    const long long q = __double2ll_rn(s * scale) + __double2ll_rn(err * scale);
    out[k] = fx_coord{(int)(q & ((1ll << lb) - 1)), (int)(q >> lb)};
  }
}

// --------------------------------------------------------------- generate
__device__ __noinline__ double close_distance(const double* __restrict__ X, int64_t gr, int64_t gc, int m, int* dup) {
  double v = 0.0;
  for (int l = 0; l < m; ++l) {
    const double diff = X[gr * m + l] - X[gc * m + l];
    v = fma(diff, diff, v);
  }
  if (v == 0.0) *dup = 1;
  return sqrt(v);
}

// z 2^-63 2^-shift in units of 2^-60, at most 1, as two limbs of 30 bits in the
// halves of a word.
__device__ __forceinline__ fx_u64 fixed60(fx_u64 z, int shift) {
  if (shift > 60) return 0;
  const fx_u64 v = (z >> (shift + 3)) + ((z >> (shift + 2)) & 1);
  return fx_make(fx_lo(v) & 0x3fffffffu, (uint32_t)(v >> 30));
}

// One tile (I, J) of a cloud: the distances once, then every problem's entries.
// Entries below e^-46 take the FP32 exponential and count as zero in the
// residual (below its unit).
template <int KIND>
__global__ void __launch_bounds__(FX_THREADS, 2)
    k_bt_generate(const int2* __restrict__ tasks, const TiledCloud* __restrict__ clouds,
                  const TiledProblem* __restrict__ probs, const double* __restrict__ points,
                  const fx_coord* __restrict__ Xq, float* __restrict__ Zf, fx_u64* __restrict__ Zi,
                  int* __restrict__ cloud_flags) {
  extern __shared__ __align__(16) unsigned char bt_smem[];
  __shared__ fx_u64 fxtab[FX_TABLE_SIZE];
  const int2 task = tasks[blockIdx.x];
  const TiledCloud& C = clouds[task.x];
  if (cloud_flags[C.flag] & ~2) return;  // uniform; coincident points may be found while this runs
  load_fx_table(fxtab);
  const int I = task.y >> 8, J = task.y & 255, n = C.n, m = C.m, e = C.e, nprob = C.nprob;
  const int* plist = C.prob;
  const double* X = points + C.point_offset;
  const int lane = threadIdx.x & 31;
  const int row0 = I * TILE, col0 = J * TILE;
  int dup = 0;
  fx_tile_pairs<KIND>(Xq + C.xq_offset, n, m, row0, col0, reinterpret_cast<fx_coord*>(bt_smem),
                      [&](int r, FxSquare(&q)[4]) {
    const int gr = row0 + r;
    // per column: d = dm 2^-62 2^kd, and d in FP32 in units of 2^(e - 63)
    fx_u64 dm[4];
    int kd[4];
    float df[4];
    unsigned on = 0, unit = 0;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int gc = col0 + 4 * lane + c;
      dm[c] = 0, kd[c] = 0, df[c] = 0.0f;
      if (gr == gc) unit |= 1u << c;
      if (gr < n && gc < n && gr != gc) {
        on |= 1u << c;
        if (fx_close(q[c], m)) {
          const fx_u64 b = (fx_u64)__double_as_longlong(close_distance(X, gr, gc, m, &dup));
          const int ex = (int)(b >> 52);
          const fx_u64 frac = b & 0xfffffffffffffull;
          dm[c] = (ex ? frac | 0x10000000000000ull : frac) << 10;
          kd[c] = (ex ? ex : 1) - 1023;
        } else {
          const FxRoot rt = fx_root_start(q[c]);
          df[c] = fx_float(fx_bits(rt.sf) + ((uint32_t)(rt.j - 63) << 23));
          dm[c] = fx_root(rt);
          kd[c] = rt.j - e;
        }
      }
    }
#pragma unroll 1
    for (int p = 0; p < nprob; ++p) {
      const TiledProblem& P = probs[plist[p]];
      const fx_u64 g = P.g;
      const int kg = P.kg;
      const float t63 = P.t63;
      float zf[4];
      fx_u64 zi[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        zf[c] = (unit >> c & 1) ? 1.0f : 0.0f;
        zi[c] = 0;
        if (on >> c & 1) {
          const float td = df[c] * t63;
          if (td > (float)kTinyArg) {
            zf[c] = exp_neg_tiny_f(td);
          } else {
            int shift;
            const fx_u64 z = fx_exp_fixed(dm[c], kd[c] + kg, g, fxtab, &shift);
            zi[c] = fixed60(z, shift);
            zf[c] = fx_float_of(z, shift);
          }
        } else if ((unit >> c & 1) && gr < n) {
          zi[c] = 1ull << 62;  // 1
        }
      }
      const int64_t o = (P.tile0 + tri_index(I, J)) * TILE_ELEMS + r * TILE + 4 * lane;
      *reinterpret_cast<float4*>(Zf + o) = make_float4(zf[0], zf[1], zf[2], zf[3]);
      *reinterpret_cast<ulonglong2*>(Zi + o) = make_ulonglong2(zi[0], zi[1]);
      *reinterpret_cast<ulonglong2*>(Zi + o + 2) = make_ulonglong2(zi[2], zi[3]);
    }
  });
  if (dup) atomicOr(cloud_flags + C.flag, 2);
}

// A warp's 32 x 64 block of a tile between global memory (two rows of 256
// contiguous bytes a step) and its lanes' rows, through 8 KB of shared memory:
// 16-byte unit u of row r at unit u ^ (r & 15).  A lane reading or writing its
// own row of global memory touches 32 lines an instruction, 4 us a tile.
__device__ __forceinline__ void block_load(const float* __restrict__ C, float4* stage, int lane, float4 (&x)[16]) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    float4 t[8];
#pragma unroll
    for (int i = 0; i < 8; ++i)
      t[i] = reinterpret_cast<const float4*>(C + (16 * h + 2 * i + (lane >> 4)) * TILE)[lane & 15];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int r = 16 * h + 2 * i + (lane >> 4);
      stage[r * 16 + ((lane ^ r) & 15)] = t[i];
    }
  }
  __syncwarp();
#pragma unroll
  for (int q = 0; q < 16; ++q) x[q] = stage[lane * 16 + ((q ^ lane) & 15)];
}
__device__ __forceinline__ void block_store(float* __restrict__ C, float4* stage, int lane, const float4 (&x)[16]) {
#pragma unroll
  for (int q = 0; q < 16; ++q) stage[lane * 16 + ((q ^ lane) & 15)] = x[q];
  __syncwarp();
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const int r = 2 * i + (lane >> 4);
    reinterpret_cast<float4*>(C + r * TILE)[lane & 15] = stage[r * 16 + ((lane ^ r) & 15)];
  }
}

// ----------------------------------------------------------------- update
// Tile (I, J) -= sum_{k < J} L_Ik L_Jk^T, one CTA each.  The panel solve left
// every L tile as FP16 operands (hi and lo of 2^12 L, in the swizzled layout):
// 64 columns of both tiles are one stage of 64 KB.  The accumulators (leading
// products, small products) are double-buffered in TMEM: the epilogue adds a
// k's sums in FP32 while the next k's products run.
constexpr int BU_THREADS = 320;  // 8 epilogue warps, a loader, an MMA issuer
constexpr int BU_STAGES = 3;
constexpr uint32_t BU_HALF = 32768;  // one tile's 64 columns: hi 16 KB, lo 16 KB
constexpr int BU_SMEM = BU_STAGES * 2 * (int)BU_HALF + 1024;
constexpr int64_t OPER_BYTES = 65536;  // a tile's operands

__global__ void __launch_bounds__(BU_THREADS, 1)
    k_bt_update(const int2* __restrict__ tasks, int J, const TiledProblem* __restrict__ probs, float* __restrict__ Zf,
                const unsigned char* __restrict__ oper, DevStatus* __restrict__ sts, uint64_t timeout_ns) {
  extern __shared__ __align__(1024) unsigned char bu_raw[];
  unsigned char* smem = (unsigned char*)(((uintptr_t)bu_raw + 1023) & ~(uintptr_t)1023);
  __shared__ __align__(8) uint64_t full[BU_STAGES], empty[BU_STAGES], acc_full[2], acc_empty[2], c_read;
  __shared__ uint32_t tmem_base_sh;
  __shared__ int abort_flag, skip;
  const int2 task = tasks[blockIdx.x];
  const int p = task.x, I = task.y;
  DevStatus* st = sts + p;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) skip = stopped(st);
  __syncthreads();
  if (skip) return;  // uniform across the CTA
  const int64_t tile0 = probs[p].tile0;
  if (tid == 0) {
    abort_flag = 0;
    for (int i = 0; i < BU_STAGES; ++i) mbar_init(&full[i], 1), mbar_init(&empty[i], 1);
    for (int i = 0; i < 2; ++i) mbar_init(&acc_full[i], 1), mbar_init(&acc_empty[i], 8);
    mbar_init(&c_read, 8);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_sh)),
                 "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base_sh;
  const uint64_t deadline = globaltimer() + timeout_ns;
  const bool diag = I == J;
  const int steps = 2 * J;
  if (warp == 8) {
    if (lane == 0) {
      const unsigned char* a = oper + (tile0 + tri_index(I, 0)) * OPER_BYTES;
      const unsigned char* b = oper + (tile0 + tri_index(J, 0)) * OPER_BYTES;
      int s = 0;
      bool ok = true;
      for (; s < steps; ++s) {
        const int slot = s % BU_STAGES, use = s / BU_STAGES;
        // the last slot first holds the tile for the epilogue warps
        if ((use > 0 && !mbar_wait(&empty[slot], (use - 1) & 1, &abort_flag, deadline)) ||
            (s == BU_STAGES - 1 && !mbar_wait(&c_read, 0, &abort_flag, deadline))) {
          ok = false;
          break;
        }
        unsigned char* dst = smem + slot * 2 * BU_HALF;
        mbar_expect_tx(&full[slot], diag ? BU_HALF : 2 * BU_HALF);
        bulk_load(dst, a + (int64_t)s * BU_HALF, BU_HALF, &full[slot]);
        if (!diag) bulk_load(dst + BU_HALF, b + (int64_t)s * BU_HALF, BU_HALF, &full[slot]);
      }
      if (!ok) {  // let the loads in flight land before the CTA ends
        const uint64_t dl = globaltimer() + 200000000ull;
        for (int i = s > BU_STAGES ? s - BU_STAGES : 0; i < s; ++i)
          while (!mbar_try_wait(&full[i % BU_STAGES], (i / BU_STAGES) & 1) && globaltimer() < dl) {
          }
      }
    }
  } else if (warp == 9) {
    if (lane == 0) {
      for (int s = 0; s < steps; ++s) {
        const int slot = s % BU_STAGES, use = s / BU_STAGES, k = s >> 1;
        if ((s & 1) == 0 && k >= 2 && !mbar_wait(&acc_empty[k & 1], ((k >> 1) - 1) & 1, &abort_flag, deadline)) break;
        if (!mbar_wait(&full[slot], use & 1, &abort_flag, deadline)) break;
        tc_fence_after();
        const uint32_t lead = tmem + (k & 1) * 256, low = lead + 128;
        const uint32_t a = smem_u32(smem + slot * 2 * BU_HALF), b = diag ? a : a + BU_HALF;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const uint64_t ah = smem_desc<128>(a + 32 * q), al = smem_desc<128>(a + 16384 + 32 * q);
          const uint64_t bh = smem_desc<128>(b + 32 * q), bl = smem_desc<128>(b + 16384 + 32 * q);
          const uint32_t more = ((s & 1) | q) != 0;
          mma_f16_128x128(lead, ah, bh, more);
          mma_f16_128x128(low, ah, bl, more);
          mma_f16_128x128(low, al, bh, 1u);
        }
        mma_commit(&empty[slot]);
        if (s & 1) mma_commit(&acc_full[k & 1]);
      }
    }
  } else {
    const int r0 = 32 * (warp & 3), c0 = 64 * (warp >> 2);
    float* C = Zf + (tile0 + tri_index(I, J)) * TILE_ELEMS + r0 * TILE + c0;
    const uint32_t base = tmem + ((uint32_t)r0 << 16) + (uint32_t)c0;
    float4* stage = reinterpret_cast<float4*>(smem + (BU_STAGES - 1) * 2 * BU_HALF + warp * 8192);
    float4 sum[16];
    block_load(C, stage, lane, sum);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncwarp();
    if (lane == 0) mbar_arrive(&c_read);
    constexpr float kInv = 1.0f / (float)(1 << FP16_SCALE_LOG2) / (float)(1 << FP16_SCALE_LOG2);
    bool ok = true;
    for (int k = 0; k < J; ++k) {
      if (!mbar_wait(&acc_full[k & 1], (k >> 1) & 1, &abort_flag, deadline)) ok = false;
      ok = __all_sync(0xffffffffu, ok);  // the reads below are warp-wide
      if (!ok) break;
      tc_fence_after();
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float v[32], u[32];
        tmem_ld32(base + (k & 1) * 256 + 32 * h, v);
        tmem_ld32(base + (k & 1) * 256 + 128 + 32 * h, u);
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          float4& s = sum[8 * h + q];
          s.x = fmaf(-(v[4 * q] + u[4 * q]), kInv, s.x);
          s.y = fmaf(-(v[4 * q + 1] + u[4 * q + 1]), kInv, s.y);
          s.z = fmaf(-(v[4 * q + 2] + u[4 * q + 2]), kInv, s.z);
          s.w = fmaf(-(v[4 * q + 3] + u[4 * q + 3]), kInv, s.w);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&acc_empty[k & 1]);
    }
    if (ok) block_store(C, stage, lane, sum);  // every product has read its operands
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (tid == 0 && abort_flag) atomicOr(&st->flags, ST_TIMEOUT);
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
}

// ------------------------------------------------------------ panel solve
// L_IJ = A_IJ inv(L_JJ)^T for task.z consecutive tiles I = task.y .. of problem
// task.x, as k_trsm_tc; the tiles share the split inverse.  Writes L in FP32
// and as the update's operands.
constexpr int BP_THREADS = 256;
constexpr int BP_OP = 2 * 128 * 128;
constexpr int BP_SMEM = 4 * BP_OP + 1024;

__global__ void __launch_bounds__(BP_THREADS, 1)
    k_bt_panel(const int4* __restrict__ tasks, int J, const TiledProblem* __restrict__ probs, float* __restrict__ Zf,
               const float* __restrict__ Dinv, unsigned char* __restrict__ oper, DevStatus* __restrict__ sts,
               uint64_t timeout_ns) {
  extern __shared__ __align__(1024) unsigned char bp_raw[];
  unsigned char* smem = (unsigned char*)(((uintptr_t)bp_raw + 1023) & ~(uintptr_t)1023);
  unsigned char *b_hi = smem, *b_lo = smem + BP_OP, *a_hi = smem + 2 * BP_OP, *a_lo = smem + 3 * BP_OP;
  __shared__ int aexp[TILE], bexp[TILE];
  __shared__ __align__(8) uint64_t done_bar;
  __shared__ uint32_t tmem_base_sh;
  __shared__ int abort_flag, skip;
  const int4 task = tasks[blockIdx.x];
  DevStatus* st = sts + task.x;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) skip = stopped(st);
  __syncthreads();
  if (skip) return;  // uniform across the CTA
  if (tid == 0) {
    abort_flag = 0;
    mbar_init(&done_bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_sh)),
                 "r"(256u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  const int64_t tile0 = probs[task.x].tile0;
  float4 x[16];
  trsm_load(Dinv + (probs[task.x].diag0 + J) * TILE_ELEMS, x);
  trsm_split(x, b_hi, b_lo, bexp);
  trsm_load(Zf + (tile0 + tri_index(task.y, J)) * TILE_ELEMS, x);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base_sh;
  const uint64_t deadline = globaltimer() + timeout_ns;
  constexpr float kScale = (float)(1 << FP16_SCALE_LOG2);
  for (int i = 0; i < task.z; ++i) {
    const int64_t tile = tile0 + tri_index(task.y + i, J);
    trsm_split(x, a_hi, a_lo, aexp);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    if (tid == 0) {
      tc_fence_after();
#pragma unroll
      for (int c = 0; c < 2; ++c) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const uint32_t o = c * 16384 + k * 32;
          const uint64_t ah = smem_desc<128>(smem_u32(a_hi + o)), al = smem_desc<128>(smem_u32(a_lo + o));
          const uint64_t bh = smem_desc<128>(smem_u32(b_hi + o)), bl = smem_desc<128>(smem_u32(b_lo + o));
          mma_f16_128x128(tmem, ah, bh, (c | k) != 0);
          mma_f16_128x128(tmem + 128, ah, bl, (c | k) != 0);
          mma_f16_128x128(tmem + 128, al, bh, 1u);
        }
      }
      mma_commit(&done_bar);
    }
    if (i + 1 < task.z) trsm_load(Zf + (tile0 + tri_index(task.y + i + 1, J)) * TILE_ELEMS, x);
    const bool waited = mbar_wait(&done_bar, i & 1, &abort_flag, deadline);
    const bool ok = __syncthreads_and(waited ? 1 : 0) != 0;  // one decision for the whole CTA
    if (!ok) break;
    tc_fence_after();
    // TMEM lanes 32 (warp & 3) .. are the rows, warp >> 2 picks 64 columns: one K chunk
    const int r0 = 32 * (warp & 3), c0 = 64 * (warp >> 2);
    const float ra = pow2f(-aexp[r0 + lane]);
    float4* stage = reinterpret_cast<float4*>(a_hi + warp * 8192);  // the products have read A
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      float v[32], u[32];
      const uint32_t ta = tmem + ((uint32_t)r0 << 16) + (uint32_t)(c0 + 32 * j);
      tmem_ld32(ta, v);
      tmem_ld32(ta + 128, u);
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int c = c0 + 32 * j + 4 * q;
        stage[lane * 16 + (((8 * j + q) ^ lane) & 15)] =
            make_float4((v[4 * q] + u[4 * q]) * ra * pow2f(-bexp[c]), (v[4 * q + 1] + u[4 * q + 1]) * ra * pow2f(-bexp[c + 1]),
                        (v[4 * q + 2] + u[4 * q + 2]) * ra * pow2f(-bexp[c + 2]),
                        (v[4 * q + 3] + u[4 * q + 3]) * ra * pow2f(-bexp[c + 3]));
      }
    }
    __syncwarp();
    float* out = Zf + tile * TILE_ELEMS + r0 * TILE + c0;
    unsigned char* op = oper + tile * OPER_BYTES + (warp >> 2) * BU_HALF;
#pragma unroll 4
    for (int k = 0; k < 16; ++k) {
      const int r = 2 * k + (lane >> 4), q = lane & 15;
      const float4 o = stage[r * 16 + ((lane ^ r) & 15)];
      reinterpret_cast<float4*>(out + r * TILE)[q] = o;
      const float y[4] = {o.x * kScale, o.y * kScale, o.z * kScale, o.w * kScale};
      __align__(8) __half h[4], l[4];
#pragma unroll
      for (int x4 = 0; x4 < 4; ++x4) {
        h[x4] = __float2half_rn(y[x4]);
        l[x4] = __float2half_rn(y[x4] - __half2float(h[x4]));
      }
      const uint32_t off2 = swizzled_unit(r0 + r, q >> 1) + (q & 1) * 8;
      *reinterpret_cast<uint2*>(op + off2) = *reinterpret_cast<const uint2*>(h);
      *reinterpret_cast<uint2*>(op + 16384 + off2) = *reinterpret_cast<const uint2*>(l);
    }
    tc_fence_before();
    __syncthreads();  // the accumulators, A's operands and exponents are free
  }
  if (tid == 0 && abort_flag) atomicOr(&st->flags, ST_TIMEOUT);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(256u) : "memory");
}

// --------------------------------------------------------------- residual
// Z w of a tile in integers, exactly.  z = (zh 2^30 + zl) 2^-60; w = (wh 2^30 +
// wl) 2^(ew - 55), |w| < 2^ew, |wh| <= 2^25, -2^29 <= wl < 2^29.  A sum holds
//   V = 2^30 sum zh wh + sum (zh wl + zl wh) + 2^-30 sum zl wl, unit 2^(ew - 85),
// rounded down once per eight rows (column sums) or by a lane's row (row sums): at
// most 2^-71 of |w|'s largest entry, where an FP64 sum loses 2^-53 of itself at every step.  The FP64 pipe
// would take 16 cycles of an SM for 32 entries and a sum, the 32 x 32 -> 64-bit
// multiplier 2.  The parts of a lane's sums over eight rows (four columns) stay
// below 2^63.  Integer sums are the same in any order.
constexpr int BR_THREADS = 256;

struct Wide {
  long long hi;            // V = hi 2^32 + lo
  unsigned long long lo;
};
__device__ __forceinline__ void wide_add(Wide& a, long long hh, long long mid) {
  // hh 2^30 + mid
  const long long h = (hh >> 2) + (mid >> 32);
  const unsigned long long l = (((unsigned long long)hh << 30) & 0xffffffffull) + ((unsigned long long)mid & 0xffffffffull);
  a.hi += h;
  a.lo += l;
}

constexpr int BR_ROWS = 64, BR_SLOTS = 4;  // rows of a CTA, in slots of 16 KB
constexpr int BR_SMEM = BR_ROWS * TILE * 8;

// 64 rows of a tile (blockIdx.x & 1: which), all of them on their way into
// shared memory at once: three CTAs keep 192 KB of an SM's reads in flight (8
// 16-byte loads a thread in registers, two CTAs: 4.6 TB/s).  A lane takes
// columns 2 lane, 2 lane + 1 and the same beyond 64.  P, S: a tile's 128 row
// sums, then the column sums of either half.
template <bool FIRST>
__global__ void __launch_bounds__(BR_THREADS, 3)
    k_bt_residual(const int2* __restrict__ tasks, const TiledProblem* __restrict__ probs,
                  const TiledState* __restrict__ state, const fx_u64* __restrict__ Zi, const int2* __restrict__ W,
                  longlong2* __restrict__ P, unsigned* __restrict__ S, DevStatus* __restrict__ sts,
                  uint64_t timeout_ns) {
  extern __shared__ __align__(128) unsigned char br_smem[];
  __shared__ __align__(8) uint64_t bar[BR_SLOTS];
  __shared__ int abort_flag;
  const int2 task = tasks[blockIdx.x >> 1];
  if (state[task.x].done) return;  // uniform
  const int half = blockIdx.x & 1, I = task.y >> 8, J = task.y & 255;
  const int64_t tile = probs[task.x].tile0 + tri_index(I, J);
  const int2* w = W + probs[task.x].diag0 * TILE;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int k = 0; k < BR_SLOTS; ++k) mbar_init(&bar[k], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    const fx_u64* src = Zi + tile * TILE_ELEMS + half * BR_ROWS * TILE;
    for (int k = 0; k < BR_SLOTS; ++k) {
      mbar_expect_tx(&bar[k], BR_SMEM / BR_SLOTS);
      bulk_load(br_smem + k * (BR_SMEM / BR_SLOTS), src + k * (BR_ROWS / BR_SLOTS) * TILE, BR_SMEM / BR_SLOTS, &bar[k]);
    }
  }
  __syncthreads();
  const uint64_t deadline = globaltimer() + timeout_ns;
  longlong2* sums = P + tile * 3 * TILE;
  unsigned* zsums = S + tile * 3 * TILE;
  int2 wc[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) wc[c] = w[J * TILE + 2 * lane + 64 * (c >> 1) + (c & 1)];
  unsigned cz[4] = {0, 0, 0, 0};
  long long chh[4] = {0, 0, 0, 0}, cmid[4] = {0, 0, 0, 0}, cll[4] = {0, 0, 0, 0};
  bool ok = true;
#pragma unroll 1
  for (int k = 0; k < BR_SLOTS; ++k) {
    ok = ok && mbar_wait(&bar[k], 0, &abort_flag, deadline);
    ok = __all_sync(0xffffffffu, ok);
    if (!ok) break;
#pragma unroll
    for (int rr = 0; rr < 2; ++rr) {
      const int r = 16 * k + 2 * warp + rr, gr = half * BR_ROWS + r;
      const ulonglong2* zr = reinterpret_cast<const ulonglong2*>(br_smem) + r * (TILE / 2);
      const ulonglong2 v0 = zr[lane], v1 = zr[lane + 32];
      const int2 wr = w[I * TILE + gr];
      const fx_u64 e[4] = {v0.x, v0.y, v1.x, v1.y};
      long long hh = 0, mid = 0, ll = 0;
      unsigned zs = 0;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int zh = (int)fx_hi(e[c]), zl = (int)fx_lo(e[c]);
        hh += (long long)zh * wc[c].x;
        mid += (long long)zh * wc[c].y;
        mid += (long long)zl * wc[c].x;
        ll += (long long)zl * wc[c].y;
        chh[c] += (long long)zh * wr.x;
        cmid[c] += (long long)zh * wr.y;
        cmid[c] += (long long)zl * wr.x;
        cll[c] += (long long)zl * wr.y;
        if (FIRST) {
          zs += (unsigned)zh >> 6;
          cz[c] += (unsigned)zh >> 6;
        }
      }
      // the row's sum over the lanes, below 2^88, in 26-bit limbs from bit 14 up
      // (bits 0..13 of a lane's part, 2^-71 of |w|'s largest entry, are dropped)
      const long long m2 = mid + (ll >> 30);
      const long long vh = (hh >> 2) + (m2 >> 32);                        // bits 32 up
      const fx_u64 vl = (fx_u64)(((unsigned)hh & 3u) << 30) + (unsigned)m2;  // bits 0..32
      const long long up = vh + (long long)(vl >> 32);
      const unsigned s0 = __reduce_add_sync(0xffffffffu, __funnelshift_r((unsigned)vl, (unsigned)up, 14) & 0x3ffffffu);
      const unsigned s1 = __reduce_add_sync(0xffffffffu, (unsigned)(up >> 8) & 0x3ffffffu);
      const int s2 = __reduce_add_sync(0xffffffffu, (int)(up >> 34));
      if (lane == 0) {
        // hi 2^32 + lo of s0 2^14 + s1 2^40 + s2 2^66
        const fx_u64 a = (fx_u64)s0 << 14;
        sums[gr] = make_longlong2((long long)(a >> 32) + ((long long)s1 << 8) + (long long)s2 * (1ll << 34),
                                  (long long)(a & 0xffffffffull));
      }
      if (FIRST) {
        zs = __reduce_add_sync(0xffffffffu, zs);
        if (lane == 0) zsums[gr] = zs;
      }
    }
  }
  const bool fine = __syncthreads_and(ok ? 1 : 0) != 0;  // every row has been read
  if (!fine) {
    // every thread left a wait, so this CTA's loads may be in flight
    if (threadIdx.x == 0) {
      atomicOr(&sts[task.x].flags, ST_TIMEOUT);
      const uint64_t dl = globaltimer() + 200000000ull;
      for (int k = 0; k < BR_SLOTS; ++k)
        while (!mbar_try_wait(&bar[k], 0) && globaltimer() < dl) {
        }
    }
    return;
  }
  if (I == J) return;  // uniform: the whole tile's rows
  Wide* col = reinterpret_cast<Wide*>(br_smem);                                            // [warp][TILE]
  unsigned* colz = reinterpret_cast<unsigned*>(br_smem + BR_THREADS / 32 * TILE * sizeof(Wide));
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    Wide t;
    t.hi = 0, t.lo = 0;
    wide_add(t, chh[c], cmid[c] + (cll[c] >> 30));
    const int cc = 2 * lane + 64 * (c >> 1) + (c & 1);
    col[warp * TILE + cc] = t;
    if (FIRST) colz[warp * TILE + cc] = cz[c];
  }
  __syncthreads();
  if (threadIdx.x < TILE) {
    const int c = threadIdx.x;
    long long hi = 0;
    unsigned long long lo = 0;
    unsigned sz = 0;
#pragma unroll
    for (int k = 0; k < BR_THREADS / 32; ++k) {
      hi += col[k * TILE + c].hi;
      lo += col[k * TILE + c].lo;
      if (FIRST) sz += colz[k * TILE + c];
    }
    sums[(1 + half) * TILE + c] = make_longlong2(hi + (long long)(lo >> 32), (long long)(lo & 0xffffffffull));
    if (FIRST) zsums[(1 + half) * TILE + c] = sz;
  }
}

// ------------------------------------------------------------------ solve
// One CTA per problem.  FIRST: w = (L L^T)^-1 1.  Else r = 1 - Z w from the
// tiles' sums, the stopping rule of k_batch_solve, the results once it holds,
// or a correction.  Sweeps: left-looking, a warp per row of L (forward) or per
// row of L's tiles below, transposed (backward), eight rows' loads in flight;
// the diagonal tiles by their inverses.
constexpr int BS_THREADS = 512;
constexpr int BS_WARPS = BS_THREADS / 32;
static_assert(TILE / BS_WARPS == 8, "rows per warp");

struct BtSolveSmem {
  float v[BATCH_NMAX], t[TILE];
  float part[BS_WARPS][TILE];
  double red[3][BS_WARPS];
};

// t[r] = sum_c M[r][c] x[c] (+ add) for the tile's 128 rows; row r on warp r % 16
template <class F>
__device__ __forceinline__ void rows_dot(const float (&acc)[8], int warp, int lane, F&& out) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    float a = acc[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    if (lane == 0) out(warp + BS_WARPS * i, a);
  }
}
__device__ __forceinline__ void tile_rows(const float* __restrict__ M, float4 x, int warp, int lane, float (&acc)[8]) {
  float4 l[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) l[i] = reinterpret_cast<const float4*>(M + (warp + BS_WARPS * i) * TILE)[lane];
#pragma unroll
  for (int i = 0; i < 8; ++i) acc[i] += (l[i].x * x.x + l[i].y * x.y) + (l[i].z * x.z + l[i].w * x.w);
}

// x = (L L^T)^-1 v in place (S.v)
__device__ void bt_sweeps(BtSolveSmem& S, const float* __restrict__ L, const float* __restrict__ Y,
                          const float* __restrict__ YT, int N) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  for (int J = 0; J < N; ++J) {
    float acc[8] = {};
#pragma unroll 2
    for (int K = 0; K < J; ++K)
      tile_rows(L + tri_index(J, K) * TILE_ELEMS, reinterpret_cast<const float4*>(S.v + K * TILE)[lane], warp, lane, acc);
    rows_dot(acc, warp, lane, [&](int r, float a) { S.t[r] = S.v[J * TILE + r] - a; });
    __syncthreads();
    float d[8] = {};
    tile_rows(Y + (int64_t)J * TILE_ELEMS, reinterpret_cast<const float4*>(S.t)[lane], warp, lane, d);
    rows_dot(d, warp, lane, [&](int r, float a) { S.v[J * TILE + r] = a; });
    __syncthreads();
  }
  for (int J = N - 1; J >= 0; --J) {
    float4 acc = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll 1
    for (int I = J + 1; I < N; ++I) {
      const float* M = L + tri_index(I, J) * TILE_ELEMS;
      float4 l[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) l[i] = reinterpret_cast<const float4*>(M + (warp + BS_WARPS * i) * TILE)[lane];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float x = S.v[I * TILE + warp + BS_WARPS * i];
        acc.x = fmaf(l[i].x, x, acc.x), acc.y = fmaf(l[i].y, x, acc.y);
        acc.z = fmaf(l[i].z, x, acc.z), acc.w = fmaf(l[i].w, x, acc.w);
      }
    }
    reinterpret_cast<float4*>(S.part[warp])[lane] = acc;
    __syncthreads();
    if (tid < TILE) {
      float a = 0.0f;
#pragma unroll
      for (int k = 0; k < BS_WARPS; ++k) a += S.part[k][tid];
      S.t[tid] = S.v[J * TILE + tid] - a;
    }
    __syncthreads();
    float d[8] = {};
    tile_rows(YT + (int64_t)J * TILE_ELEMS, reinterpret_cast<const float4*>(S.t)[lane], warp, lane, d);
    rows_dot(d, warp, lane, [&](int r, float a) { S.v[J * TILE + r] = a; });
    __syncthreads();
  }
}

__device__ __forceinline__ void two_sum(double a, double b, double* s, double* e) {
  const double x = a + b;
  const double bv = x - a;
  *e = (a - (x - bv)) + (b - bv);
  *s = x;
}

template <bool FIRST>
__global__ void __launch_bounds__(BS_THREADS, 2)
    k_bt_solve(const TiledProblem* __restrict__ probs, TiledState* __restrict__ state, const float* __restrict__ Zf,
               const float* __restrict__ Dinv, const float* __restrict__ DinvT, const longlong2* __restrict__ P,
               const unsigned* __restrict__ Zs, double* __restrict__ w, int2* __restrict__ W,
               double* __restrict__ w_out, double* __restrict__ mag_out, int* __restrict__ status,
               const DevStatus* __restrict__ sts, const int* __restrict__ cloud_flags, int* __restrict__ remaining,
               double tol, int max_iter) {
  __shared__ __align__(16) BtSolveSmem S;
  const TiledProblem& pb = probs[blockIdx.x];
  TiledState& T = state[blockIdx.x];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n = pb.n, N = (n + TILE - 1) / TILE;
  double* wp = w + pb.diag0 * TILE;
  int2* Wp = W + pb.diag0 * TILE;
  if (FIRST) {
    const int cf = cloud_flags[pb.flag];
    if (cf || stopped(sts + blockIdx.x)) {  // uniform: earlier kernels' flags
      if (tid == 0) {
        status[pb.pid] = (cf & 1) ? MAG_BATCH_NONFINITE : ((cf & 2) ? MAG_BATCH_DUPLICATE : MAG_BATCH_NOTPD);
        mag_out[pb.pid] = 0.0;
        T.done = 1;
      }
      return;
    }
    for (int i = tid; i < N * TILE; i += BS_THREADS) S.v[i] = i < n ? 1.0f : 0.0f;
  } else {
    if (T.done) return;
    if (stopped(sts + blockIdx.x)) {  // a wait ran out
      __syncthreads();                // T.done has been read
      if (tid == 0) {
        status[pb.pid] = MAG_BATCH_NOCONV;
        mag_out[pb.pid] = 0.0;
        T.done = 1;
      }
      return;
    }
  }
  auto block_max = [&](double a, int k) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a = fmax(a, __shfl_xor_sync(0xffffffffu, a, o));
    if (lane == 0) S.red[k][warp] = a;
  };
  auto all_max = [&](int k) {
    double a = 0.0;
    for (int j = 0; j < BS_WARPS; ++j) a = fmax(a, S.red[k][j]);
    return a;
  };
  double rn = 1.0;
  if (!FIRST) {
    // rows of block I: the tiles (I, J <= I) by rows, (K > I, I) by columns
    const int ew = T.ew, it = T.it;
    double rmax = 0.0, wmax = 0.0, zmax = 0.0;
    double rv[BATCH_NMAX / BS_THREADS];
#pragma unroll
    for (int q = 0; q < BATCH_NMAX / BS_THREADS; ++q) {
      const int i = tid + q * BS_THREADS;
      rv[q] = 0.0;
      if (i < n) {
        const int I = i / TILE, r = i % TILE;
        long long hi = 0;
        unsigned long long lo = 0, zs = 0;  // Zs: row sums of Z in units of 2^-24, rounded down
        for (int K = 0; K < N; ++K) {
          // its rows of tile (I, K), or the two halves' columns of tile (K, I)
          const int64_t o = (pb.tile0 + (K <= I ? tri_index(I, K) : tri_index(K, I))) * 3 * TILE + (K <= I ? 0 : TILE) + r;
          const longlong2 a = P[o], b = K <= I ? make_longlong2(0, 0) : P[o + TILE];
          hi += a.x + b.x;
          lo += (unsigned long long)(a.y + b.y);
          if (it == 0) zs += Zs[o] + (K <= I ? 0u : Zs[o + TILE]);
        }
        // r = 1 - V 2^(ew - 85), the subtraction in integers where 1 is a multiple of the unit
        __int128 V = ((__int128)hi << 32) + (__int128)lo;
        double ri;
        if (ew <= 60 && ew >= -30) {
          V = ((__int128)1 << (85 - ew)) - V;
          const bool neg = V < 0;
          unsigned __int128 a = neg ? (unsigned __int128)-V : (unsigned __int128)V;
          const double m = (double)(unsigned long long)(a >> 64) * 18446744073709551616.0 + (double)(unsigned long long)a;
          ri = ldexp(neg ? -m : m, ew - 85);
        } else {
          const double m = (double)(long long)(V >> 64) * 18446744073709551616.0 + (double)(unsigned long long)V;
          ri = 1.0 - ldexp(m, ew - 85);
        }
        rv[q] = ri;
        rmax = fmax(rmax, ri == ri ? fabs(ri) : INFINITY);
        wmax = fmax(wmax, fabs(wp[i]));
        zmax = fmax(zmax, (double)zs * 5.9604644775390625e-8);  // 2^-24
      }
    }
    block_max(rmax, 0);
    block_max(zmax, 1);
    block_max(wmax, 2);
    __syncthreads();
    rn = all_max(0);
    const double zn = it == 0 ? all_max(1) : T.zn, wn = all_max(2), prev = T.prev;
    int slow = T.slow;
    const double rel = (zn > 0.0 && wn > 0.0) ? rn / (zn * wn) : INFINITY;
    int st = -1;
    if (rel <= tol) {
      st = MAG_BATCH_OK;
    } else if (it >= max_iter || !(rel < INFINITY) || (rel > 0.5 * prev && ++slow >= 2)) {
      st = MAG_BATCH_NOCONV;
    }
    __syncthreads();  // the state and the reductions have been read
    if (st >= 0) {
      double s = 0.0, c = 0.0;
      for (int i = tid; i < n; i += BS_THREADS) {
        const double wi = wp[i];
        w_out[pb.w_offset + i] = wi;
        double hi, lo;
        two_sum(s, wi, &hi, &lo);
        s = hi;
        c += lo;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        double hi, lo;
        const double other = __shfl_xor_sync(0xffffffffu, s, o);
        const double oc = __shfl_xor_sync(0xffffffffu, c, o);
        two_sum(s, other, &hi, &lo);
        s = hi;
        c += oc + lo;
      }
      if (lane == 0) S.red[0][warp] = s, S.red[1][warp] = c;
      __syncthreads();
      if (tid == 0) {
        double ss = 0.0, cc = 0.0;
        for (int k = 0; k < BS_WARPS; ++k) {
          double hi, lo;
          two_sum(ss, S.red[0][k], &hi, &lo);
          ss = hi;
          cc += S.red[1][k] + lo;
        }
        mag_out[pb.pid] = ss + cc;
        status[pb.pid] = st;
        T.done = 1;
      }
      return;
    }
    if (tid == 0) {
      T.slow = rel > 0.5 * prev ? slow : 0;
      T.prev = rel;
      T.it = it + 1;
      T.zn = zn;
    }
    const double inv = rn > 0.0 ? 1.0 / rn : 0.0;
#pragma unroll
    for (int q = 0; q < BATCH_NMAX / BS_THREADS; ++q) {
      const int i = tid + q * BS_THREADS;
      if (i < N * TILE) S.v[i] = (float)(rv[q] * inv);
    }
  }
  __syncthreads();
  bt_sweeps(S, Zf + pb.tile0 * TILE_ELEMS, Dinv + pb.diag0 * TILE_ELEMS, DinvT + pb.diag0 * TILE_ELEMS, N);
  // the new w and its integers for the next residual
  double wmax = 0.0;
  double wv[BATCH_NMAX / BS_THREADS];
  bool finite = true;
#pragma unroll
  for (int q = 0; q < BATCH_NMAX / BS_THREADS; ++q) {
    const int i = tid + q * BS_THREADS;
    wv[q] = 0.0;
    if (i < n) {
      wv[q] = FIRST ? (double)S.v[i] : wp[i] + rn * (double)S.v[i];
      wp[i] = wv[q];
      finite &= isfinite(wv[q]) != 0;
      wmax = fmax(wmax, fabs(wv[q]));
    }
  }
  block_max(finite ? wmax : INFINITY, 2);
  __syncthreads();
  wmax = all_max(2);
  if (!(wmax < INFINITY) || !(wmax > 1e-290)) {  // nothing to refine
    if (tid == 0) {
      status[pb.pid] = MAG_BATCH_NOCONV;
      mag_out[pb.pid] = 0.0;
      T.done = 1;
    }
    return;
  }
  const int ew = ilogb(wmax) + 1;
#pragma unroll
  for (int q = 0; q < BATCH_NMAX / BS_THREADS; ++q) {
    const int i = tid + q * BS_THREADS;
    if (i < N * TILE) {
      const long long a = __double2ll_rn(ldexp(wv[q], 55 - ew));
      const int hi = (int)((a + (1ll << 29)) >> 30);
      Wp[i] = make_int2(hi, (int)(a - ((long long)hi << 30)));
    }
  }
  if (tid == 0) {
    T.ew = ew;
    if (FIRST) {
      T.it = 0;
      T.slow = 0;
      T.prev = INFINITY;
      T.done = 0;
    }
    atomicAdd(remaining, 1);
  }
}

constexpr uint64_t kBtTimeout = 10000000000ull;

template <class K>
cudaError_t dynamic_smem(K kern, int bytes) {
  return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

}  // namespace

size_t tiled_coord_bytes() { return sizeof(fx_coord); }
void tiled_scale(double t, unsigned long long* g, int* kg) { fx_scale_t(t, g, kg); }
int tiled_kind(int m) { return fx_kind(m); }

cudaError_t launch_bt_quantize(const TiledBatch& B, const double* points, int clouds, cudaStream_t s) {
  const dim3 grid((unsigned)clouds, BQ_PARTS);
  k_bt_range<<<grid, BQ_THREADS, 0, s>>>(points, B.clouds, B.cloud_flags, B.range);
  note_launch();
  k_bt_quantize<<<grid, BQ_THREADS, 0, s>>>(points, B.clouds, B.probs, B.cloud_flags, B.range,
                                            static_cast<fx_coord*>(B.Xq), B.st);
  note_launch();
  return cudaGetLastError();
}

template <int KIND>
static cudaError_t launch_bt_generate_t(const TiledBatch& B, const double* points, const int2* tasks, int count,
                                        int mmax, cudaStream_t s) {
  const int smem = (int)fx_tile_smem(mmax);
  cudaError_t e = dynamic_smem(k_bt_generate<KIND>, (int)FX_TILE_SMEM_MAX);
  if (e != cudaSuccess) return e;
  k_bt_generate<KIND><<<(unsigned)count, FX_THREADS, smem, s>>>(tasks, B.clouds, B.probs, points,
                                                               static_cast<const fx_coord*>(B.Xq), B.Zf, B.Zi,
                                                               B.cloud_flags);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_bt_generate(const TiledBatch& B, const double* points, int kind, const int2* tasks, int count,
                               int mmax, cudaStream_t s) {
  if (count <= 0) return cudaSuccess;
  switch (kind) {
    case 0: return launch_bt_generate_t<0>(B, points, tasks, count, mmax, s);
    case 1: return launch_bt_generate_t<1>(B, points, tasks, count, mmax, s);
    default: return launch_bt_generate_t<2>(B, points, tasks, count, mmax, s);
  }
}

cudaError_t launch_bt_update(const TiledBatch& B, int J, const int2* tasks, int count, cudaStream_t s) {
  if (count <= 0 || J == 0) return cudaSuccess;
  cudaError_t e = dynamic_smem(k_bt_update, BU_SMEM);
  if (e != cudaSuccess) return e;
  k_bt_update<<<(unsigned)count, BU_THREADS, BU_SMEM, s>>>(tasks, J, B.probs, B.Zf, B.oper, B.st, kBtTimeout);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_bt_panel(const TiledBatch& B, int J, const int4* tasks, int count, cudaStream_t s) {
  if (count <= 0) return cudaSuccess;
  cudaError_t e = dynamic_smem(k_bt_panel, BP_SMEM);
  if (e != cudaSuccess) return e;
  k_bt_panel<<<(unsigned)count, BP_THREADS, BP_SMEM, s>>>(tasks, J, B.probs, B.Zf, B.Dinv, B.oper, B.st, kBtTimeout);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_bt_residual(const TiledBatch& B, bool first, const int2* tasks, int count, cudaStream_t s) {
  if (count <= 0) return cudaSuccess;
  auto kern = first ? k_bt_residual<true> : k_bt_residual<false>;
  cudaError_t e = dynamic_smem(kern, BR_SMEM);
  if (e != cudaSuccess) return e;
  kern<<<(unsigned)(2 * count), BR_THREADS, BR_SMEM, s>>>(tasks, B.probs, B.state, B.Zi, B.W, B.P, B.S, B.st, kBtTimeout);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_bt_solve(const TiledBatch& B, bool first, int count, double* w_out, double* mag_out, int* status,
                            double tol, int max_iter, cudaStream_t s) {
  if (count <= 0) return cudaSuccess;
  if (first)
    k_bt_solve<true><<<(unsigned)count, BS_THREADS, 0, s>>>(B.probs, B.state, B.Zf, B.Dinv, B.DinvT, B.P, B.S, B.w, B.W,
                                                            w_out, mag_out, status, B.st, B.cloud_flags, B.remaining, tol,
                                                            max_iter);
  else
    k_bt_solve<false><<<(unsigned)count, BS_THREADS, 0, s>>>(B.probs, B.state, B.Zf, B.Dinv, B.DinvT, B.P, B.S, B.w, B.W,
                                                             w_out, mag_out, status, B.st, B.cloud_flags, B.remaining, tol,
                                                            max_iter);
  note_launch();
  return cudaGetLastError();
}

}  // namespace mag
