// Shared device and host helpers of the GB300 iris uniqueness library.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>

#include "../../include/ipcheck.h"

namespace ipc {

// ---------------------------------------------------------------------------
// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11): ten rounds, each two
// 32x32->64 products with multipliers 0xD2511F53 / 0xCD9E8D57, the high halves
// XORed with the other counter words and the round key; the key advances by
// the Weyl increments 0x9E3779B9 / 0xBB67AE85 between rounds.
// ---------------------------------------------------------------------------
// The round keys of a seed. Kernels that draw many blocks take them as launch parameters: a round is
// then two wide products and two three-input xors with the key as a constant-bank operand, four
// instructions where advancing the key costs two more. Kernels that draw a few in their epilogue take the
// seed and advance the key: twenty keys derived there are kept in registers across the main loop (integer
// step of 8,000 rows x 248 columns: 9.46 against 9.16 ms).
struct PhiloxKey {
  uint32_t k[20];
};

__host__ __device__ inline PhiloxKey philox_key(uint64_t seed) {
  PhiloxKey key;
  for (int r = 0; r < 10; ++r) {
    key.k[2 * r] = static_cast<uint32_t>(seed) + static_cast<uint32_t>(r) * 0x9E3779B9u;
    key.k[2 * r + 1] = static_cast<uint32_t>(seed >> 32) + static_cast<uint32_t>(r) * 0xBB67AE85u;
  }
  return key;
}

__device__ __forceinline__ uint4 philox(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, const PhiloxKey& key) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint32_t hi0 = __umulhi(0xD2511F53u, c0), lo0 = 0xD2511F53u * c0;
    const uint32_t hi1 = __umulhi(0xCD9E8D57u, c2), lo1 = 0xCD9E8D57u * c2;
    c0 = hi1 ^ c1 ^ key.k[2 * r];
    c2 = hi0 ^ c3 ^ key.k[2 * r + 1];
    c1 = lo1;
    c3 = lo0;
  }
  return make_uint4(c0, c1, c2, c3);
}

__device__ __forceinline__ uint4 philox(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, uint64_t seed) {
  uint32_t k0 = static_cast<uint32_t>(seed), k1 = static_cast<uint32_t>(seed >> 32);
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint32_t hi0 = __umulhi(0xD2511F53u, c0), lo0 = 0xD2511F53u * c0;
    const uint32_t hi1 = __umulhi(0xCD9E8D57u, c2), lo1 = 0xCD9E8D57u * c2;
    c0 = hi1 ^ c1 ^ k0;
    c2 = hi0 ^ c3 ^ k1;
    c1 = lo1;
    c3 = lo0;
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
  return make_uint4(c0, c1, c2, c3);
}

__device__ __forceinline__ uint32_t word_of(const uint4& w, uint32_t i) {
  return i == 0 ? w.x : i == 1 ? w.y : i == 2 ? w.z : w.w;
}

// Device status bits (kernel gave up a bounded wait, bad launch argument seen on device).
constexpr uint32_t ST_WAIT_TIMEOUT = 1u;
constexpr uint32_t ST_BAD_ARGUMENT = 2u;

__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ void raise_status(uint32_t* status, uint32_t bits) {
  if (status) atomicOr(status, bits);
}

// ---------------------------------------------------------------------------
// Host side.
// ---------------------------------------------------------------------------
void set_error(const std::string& msg);            // thread-local last error for stage-level calls
int cuda_fail(cudaError_t e, const char* what);    // records and maps to IPC_ECUDA
uint32_t* status_ptr();                            // device status word of the current device
inline cudaStream_t as_stream(void* s) { return reinterpret_cast<cudaStream_t>(s); }

}  // namespace ipc

#define IPC_CUDA_TRY(expr)                                  \
  do {                                                      \
    cudaError_t e__ = (expr);                               \
    if (e__ != cudaSuccess) return ipc::cuda_fail(e__, #expr); \
  } while (0)
