// Device helpers of the kernels whose database operand lies in tensor memory (gemm_ts.cu, ring32.cu):
// MMAs with A in tensor memory, descriptors of 128-byte swizzled tiles, the residues of drained
// accumulators, ring positions and distributed shared memory.
#pragma once
#include "tcgen05.cuh"

namespace ipc {
namespace tc {

// Shared-memory matrix descriptor of a K-major tile in 128-byte swizzled rows: 8-row groups 1,024
// bytes apart, layout type SWIZZLE_128B (2 at bits 61-63).
__device__ __forceinline__ uint64_t sdesc128(uint32_t addr) {
  return static_cast<uint64_t>((addr & 0x3FFFFu) >> 4) | (1ull << 16) | (static_cast<uint64_t>(1024 >> 4) << 32) |
         (1ull << 46) | (2ull << 61);
}

__device__ __forceinline__ void umma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b, uint32_t idesc, bool accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(
          d_tmem),
      "r"(a_tmem), "l"(b), "r"(idesc), "r"(accumulate ? 1u : 0u)
      : "memory");
}

__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
      "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]),
      "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]),
      "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
      : "memory");
}

// Two fp32 lanes: a * b + c and a + b.
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t both(float x) {
  const uint64_t b = __float_as_uint(x);
  return b | (b << 32);
}

// The low 16 bits of STEP v, v whole numbers with |v| <= 2^24 as floats (two columns): v minus its
// nearest multiple of 2^16 / STEP, times STEP, plus 1.5 * 2^23 has them in its low mantissa bits.
// Every step is exact: v / (2^16 / STEP) rounds to a whole number below 2^16 + 1, the remainder is
// at most 2^15 / STEP in size, and sums within 2^15 of 1.5 * 2^23 have unit steps.
template <int STEP>
__device__ __forceinline__ uint32_t low16x2(uint32_t v0, uint32_t v1) {
  constexpr float M = 12582912.0f, P = 65536.0f / STEP;
  const uint64_t v = v0 | (static_cast<uint64_t>(v1) << 32);
  const uint64_t t = fma2(v, both(1.0f / P), both(M));
  const uint64_t h = fma2(t, both(1.0f), both(-M));
  const uint64_t r = fma2(h, both(-P), v);
  const uint64_t u = fma2(r, both(static_cast<float>(STEP)), both(M));
  return pack_lo16(static_cast<uint32_t>(u), static_cast<uint32_t>(u >> 32));
}
__device__ __forceinline__ bool named_sync_or(uint32_t id, uint32_t n, bool pred) {
  uint32_t r;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n bar.red.or.pred q, %2, %3, p;\n selp.u32 %0, 1, 0, q;\n}\n"
      : "=r"(r)
      : "r"(pred ? 1u : 0u), "r"(id), "r"(n)
      : "memory");
  return r != 0;
}
// Address of a shared-memory location of another CTA of the cluster.
__device__ __forceinline__ uint32_t mapa(uint32_t addr, uint32_t rank) {
  uint32_t d;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"(addr), "r"(rank));
  return d;
}
__device__ __forceinline__ uint4 ld_cluster128(uint32_t a) {
  uint4 v;
  asm volatile("ld.shared::cluster.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
  return v;
}
__device__ __forceinline__ uint32_t ld_cluster32(uint32_t a) {
  uint32_t v;
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;\n barrier.cluster.wait.acquire;" ::: "memory");
}

// Position in a ring whose size is known at run time.
struct Ring {
  uint32_t s = 0, ph = 0;
  __device__ __forceinline__ void next(uint32_t n) {
    if (++s == n) {
      s = 0;
      ph ^= 1u;
    }
  }
};

// Stage and phase parity of the G-th use of a ring of N stages.
template <uint32_t N>
__device__ __forceinline__ uint32_t turn_of(uint32_t G) { return G / N; }
template <uint32_t N>
__device__ __forceinline__ uint32_t stage_of(uint32_t G) { return G - turn_of<N>(G) * N; }
template <uint32_t N>
__device__ __forceinline__ uint32_t phase_of(uint32_t G) { return turn_of<N>(G) & 1u; }

}  // namespace tc
}  // namespace ipc
