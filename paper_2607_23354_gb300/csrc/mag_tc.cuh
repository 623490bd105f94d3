// Inline PTX shared by the tcgen05 kernels: mbarriers with bounded waits, the
// shared-memory matrix descriptor, MMA commit and TMEM loads.
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "mag_internal.cuh"

namespace mag {

// ------------------------------------------------------------ PTX wrappers
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ uint64_t globaltimer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait for the phase with `parity` to complete.  Returns false if the
// deadline passed (then raises the CTA abort flag) or another role aborted.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag,
                                          uint64_t deadline) {
  uint32_t it = 0;
  while (!mbar_try_wait(bar, parity)) {
    if ((++it & 255u) == 0) {
      if (*abort_flag) return false;
      if (globaltimer() > deadline) {
        *abort_flag = 1;
        return false;
      }
    }
  }
  return true;
}
__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
// Shared-memory matrix descriptor, K-major, version 1, base offset 0:
// 128-byte rows -> SWIZZLE_128B (layout 2), 8-row groups 1024 B apart;
// 64-byte rows  -> SWIZZLE_64B (layout 4), 8-row groups 512 B apart.
template <int CHUNK>
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);         // start address
  d |= (uint64_t)1 << 16;                           // leading byte offset (unused for swizzled K-major)
  d |= (uint64_t)((8 * CHUNK) >> 4) << 32;          // stride byte offset: 8 rows
  d |= (uint64_t)1 << 46;                           // descriptor version
  d |= (uint64_t)(CHUNK == 128 ? 2 : 4) << 61;      // SWIZZLE_128B / SWIZZLE_64B
  return d;
}
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                   smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float* v) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, "
      "%13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, "
      "[%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
        "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]),
        "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]),
        "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// ---------------------------------------------------------------- clusters
__device__ __forceinline__ uint32_t map_to_rank(uint32_t saddr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_remote_s64(uint32_t cluster_addr, int64_t v) {
  asm volatile("st.shared::cluster.s64 [%0], %1;" ::"r"(cluster_addr), "l"(v) : "memory");
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// A 128-row x 128-column FP16 operand in the layout the K-major SWIZZLE_128B
// descriptors read: two chunks of 64 columns (16 KB each), row r at byte 128 r of
// its chunk, 16-byte unit u (columns 8u .. 8u + 7 of the chunk) at unit
// u ^ (r & 7).  Within a chunk, then by the unit of the whole row (0 .. 15).
__device__ __forceinline__ uint32_t swizzled_unit(int r, int u) { return (uint32_t)(r * 128 + ((u ^ (r & 7)) << 4)); }
__device__ __forceinline__ uint32_t operand_unit(int r, int u16) {
  return (uint32_t)((u16 >> 3) * 16384) + swizzled_unit(r, u16 & 7);
}

// Untiled bulk copy to shared memory (16-byte aligned addresses, a multiple of
// 16 bytes), completing on `bar`.
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

// ------------------------------------------- FP32 tiles as FP16 operands
__device__ __forceinline__ float pow2f(int e) { return __uint_as_float((uint32_t)(e + 127) << 23); }

// Power-of-two exponent e with max |x| * 2^e in [2^13, 2^14): 0 for a row of
// zeros, subnormals or non-finite values.
__device__ __forceinline__ int row_scale_exp(float m) {
  const int ex = (int)((__float_as_uint(m) >> 23) & 0xffu);
  if (ex == 0 || ex == 255) return 0;
  const int e = 14 - (ex - 126);
  return e < -100 ? -100 : (e > 100 ? 100 : e);
}

// 128 x 128 FP32 tile (row-major) in registers: warp w holds rows
// 2 (w + 8 i) + (lane >> 4), i = 0..7, lane & 15 holds its columns
// 8 (lane & 15) .. + 7.
__device__ __forceinline__ void trsm_load(const float* __restrict__ src, float4 (&x)[16]) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int r = 2 * (warp + 8 * i) + (lane >> 4);
    const float4* p = reinterpret_cast<const float4*>(src + r * TILE + 8 * (lane & 15));
    x[2 * i] = __ldcg(p);
    x[2 * i + 1] = __ldcg(p + 1);
  }
}

// Split the register tile into scaled FP16 hi / lo operands and the row
// exponents.
__device__ __forceinline__ void trsm_split(const float4 (&x)[16], unsigned char* hi, unsigned char* lo, int* rexp) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int r = 2 * (warp + 8 * i) + (lane >> 4);
    const float4 a = x[2 * i], b = x[2 * i + 1];
    float m = fmaxf(fmaxf(fmaxf(fabsf(a.x), fabsf(a.y)), fmaxf(fabsf(a.z), fabsf(a.w))),
                    fmaxf(fmaxf(fabsf(b.x), fabsf(b.y)), fmaxf(fabsf(b.z), fabsf(b.w))));
#pragma unroll
    for (int o = 1; o < 16; o <<= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    const int e = row_scale_exp(m);
    const float sc = pow2f(e);
    const float v[8] = {a.x * sc, a.y * sc, a.z * sc, a.w * sc, b.x * sc, b.y * sc, b.z * sc, b.w * sc};
    __align__(16) __half h[8], l[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      h[q] = __float2half_rn(v[q]);
      l[q] = __float2half_rn(v[q] - __half2float(h[q]));
    }
    const uint32_t off = operand_unit(r, lane & 15);
    *reinterpret_cast<uint4*>(hi + off) = *reinterpret_cast<const uint4*>(h);
    *reinterpret_cast<uint4*>(lo + off) = *reinterpret_cast<const uint4*>(l);
    if ((lane & 15) == 0) rexp[r] = e;
  }
}

__device__ __forceinline__ void mma_f16_128x128(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t accumulate) {
  // D = F32, A = B = F16, both K-major, M = 128, N = 128
  constexpr uint32_t idesc = (1u << 4) | ((uint32_t)(128 >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
      : "memory");
}

}  // namespace mag
