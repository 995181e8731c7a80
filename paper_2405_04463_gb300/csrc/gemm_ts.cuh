// The tcgen05 ring GEMM over Z_2^16 (gemm_ts.cu) as the context, serving and stage-level calls use it.
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

namespace ipc {

constexpr uint32_t RING_GEMM_PASSES = 6;
constexpr uint64_t L2_QUERY_BYTES = 112ull << 20;  // query operands that stay in L2 beside the database

// One ring GEMM of a launch: z = [x[0] | x[1]] . b + zero share (segments = 2) or x[0] . b (segments = 1).
struct RingGemm {
  const int8_t *x_lo[2], *x_hi[2];  // limb planes [x_rows][l] of the K segments
  uint32_t segments;
  const uint16_t *b_lo, *b_hi;      // [n_pad][segments l] fp16 limbs
  uint64_t seed_own, seed_prev;
  uint32_t vec;
  uint16_t* z;                      // [n_cols][ldz]
};

// The form with both operands in shared memory (gemm_tc.cu): passes of equal segments, tiles of 256 columns.
int ring_gemm_ss_ready();
int ring_gemm_ss(uint32_t n_pass, const RingGemm* g, size_t x_rows, uint32_t n_cols, uint32_t n_pad, uint32_t l,
                 const uint32_t* col_tags, size_t ldz, uint64_t row0, const uint32_t* col_tiles,
                 const uint32_t* n_col_list, cudaStream_t stream);

// Loads every form of the kernel on this device (once). Loading one may wait for the work on the device, so
// contexts call this when they are made; without it the first launch does.
int ring_gemm_ts_ready();

// n_pass ring GEMMs over the same rows and columns, in as few launches as pay.
int ring_gemm_ts(uint32_t n_pass, const RingGemm* g, size_t x_rows, uint32_t n_cols, uint32_t n_pad, uint32_t l,
                 const uint32_t* col_tags, size_t ldz, uint64_t row0, cudaStream_t stream);

// The passes of a launch that pay for `cols` columns and K of `segments` (the longest pass's): n_pass, 3 or 1.
uint32_t ring_gemm_ts_passes(uint32_t n_pass, uint32_t segments, size_t x_rows, uint32_t cols, uint32_t l);

// The same with `per` passes in a launch. col_tiles (device, may be null): the column tiles of list_cols
// columns to compute, n_col_list (device) their count, walked by one CTA per SM.
int ring_gemm_ts_by(uint32_t per, uint32_t n_pass, const RingGemm* g, size_t x_rows, uint32_t n_cols, uint32_t n_pad,
                    uint32_t l, const uint32_t* col_tags, size_t ldz, uint64_t row0, uint32_t list_cols,
                    const uint32_t* col_tiles, const uint32_t* n_col_list, cudaStream_t stream);

}  // namespace ipc
