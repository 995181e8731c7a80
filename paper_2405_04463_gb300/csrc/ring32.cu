// A0-A3 over Z_{2^32} for the lifting variants (Sec. 5.1, Sec. 6.2): ConstLift computes ml,
// NoLift also the code dot product, over Z_{2^32}.
//
// A0: client sharing of the masked bits and mask bits read in Z_{2^32}.
// A1: four balanced int8 limbs per element, x = x0 + 2^8 x1 + 2^16 x2 + 2^24 x3 (mod 2^32), in
//     four resident int8 planes (the size of the u32 shares).
// A2: the query operand's four limbs as fp16 bit patterns (exact).
// A3 (gemm_tc32_kernel): the ring dot product on tcgen05 with fp32 TMEM accumulators, exact:
//     z = sum_s 2^(8s) S_s (mod 2^32),  S_s = sum over a + b = s of sum_k x_a[k] y_b[k],
//   ten limb products per k (1 + 2 + 3 + 4 for s = 0..3); products with a + b > 3 vanish mod
//   2^32. The database limbs are widened from int8 to fp16 on their way into tensor memory.
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <mutex>
#include <string>
#include <type_traits>

#include "gemm_ts.cuh"
#include "tcgen05_ts.cuh"

namespace ipc {
namespace {

using namespace tc;

// Balanced signed limbs of x mod 2^32, least significant first, each in [-128, 127].
__device__ __forceinline__ void limbs32(uint32_t x, int8_t (&o)[4]) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int v = static_cast<int8_t>(x & 0xFFu);
    o[i] = static_cast<int8_t>(v);
    x = (x - static_cast<uint32_t>(v)) >> 8;  // exact: x - v is 0 mod 256
  }
}

__device__ __forceinline__ uint16_t f16_of8(int8_t v) { return __half_as_ushort(__short2half_rn(v)); }

// A0 over Z_{2^32}: one thread per (row, 2 consecutive elements); one Philox call per vector
// gives both elements' x_0, x_1 (words 2e, 2e + 1).
__global__ void encode_share32_kernel(const uint64_t* __restrict__ code_bits, const uint64_t* __restrict__ mask_bits,
                                      uint32_t n, uint32_t l, const __grid_constant__ PhiloxKey key, uint32_t side, uint32_t idx0,
                                      uint32_t* __restrict__ code_sh, uint32_t* __restrict__ mask_sh) {
  const uint32_t pairs = l >> 1;
  const uint64_t tid = blockIdx.x * static_cast<uint64_t>(blockDim.x) + threadIdx.x;
  if (tid >= static_cast<uint64_t>(n) * pairs) return;
  const uint32_t r = static_cast<uint32_t>(tid / pairs), t = static_cast<uint32_t>(tid % pairs);
  const uint32_t nw = (l + 63) >> 6;
  const uint32_t b0 = t << 1;
  const uint32_t cw = static_cast<uint32_t>(code_bits[static_cast<uint64_t>(r) * nw + (b0 >> 6)] >> (b0 & 63)) & 3u;
  const uint32_t mw = static_cast<uint32_t>(mask_bits[static_cast<uint64_t>(r) * nw + (b0 >> 6)] >> (b0 & 63)) & 3u;
  const uint64_t plane = static_cast<uint64_t>(n) * l;
  const uint64_t at = static_cast<uint64_t>(r) * l + b0;
#pragma unroll
  for (uint32_t vec = 0; vec < 2; ++vec) {
    const uint4 w = philox(t, idx0 + r, (side << 8) | vec, IPC_D_SHARE32 << 24, key);
    uint32_t x0[2] = {w.x, w.z}, x1[2] = {w.y, w.w}, x2[2];
#pragma unroll
    for (uint32_t e = 0; e < 2; ++e) {
      const uint32_t cb = (cw >> e) & 1u, mb = (mw >> e) & 1u;
      const uint32_t val = vec == 0 ? (mb - 2u * (cb & mb)) : mb;  // T = -1, U = 0, F = +1 / mask bit
      x2[e] = val - x0[e] - x1[e];
    }
    uint32_t* dst = vec == 0 ? code_sh : mask_sh;
    *reinterpret_cast<uint2*>(dst + at) = make_uint2(x0[0], x0[1]);
    *reinterpret_cast<uint2*>(dst + plane + at) = make_uint2(x1[0], x1[1]);
    *reinterpret_cast<uint2*>(dst + 2 * plane + at) = make_uint2(x2[0], x2[1]);
  }
}

// A1 over Z_{2^32}: 4 elements per thread, one int8 limb plane per limb.
__global__ void split_limbs32_kernel(const uint32_t* __restrict__ x, size_t count, int8_t* __restrict__ o0,
                                     int8_t* __restrict__ o1, int8_t* __restrict__ o2, int8_t* __restrict__ o3) {
  const size_t i4 = (blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x) * 4;
  if (i4 >= count) return;
  int8_t* out[4] = {o0, o1, o2, o3};
  if (i4 + 4 <= count) {
    const uint4 v = *reinterpret_cast<const uint4*>(x + i4);
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
    uint32_t packed[4] = {0u, 0u, 0u, 0u};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      int8_t lb[4];
      limbs32(w[e], lb);
#pragma unroll
      for (int i = 0; i < 4; ++i) packed[i] |= static_cast<uint32_t>(static_cast<uint8_t>(lb[i])) << (8 * e);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) *reinterpret_cast<uint32_t*>(out[i] + i4) = packed[i];
  } else {
    for (size_t e = i4; e < count; ++e) {
      int8_t lb[4];
      limbs32(x[e], lb);
      for (int i = 0; i < 4; ++i) out[i][e] = lb[i];
    }
  }
}

// A2 over Z_{2^32}: party i's operand [rot(Y_i + Y_{i-1}) | rot(Y_i)] (K = 2l), or, for one
// segment, rot(Y_i) alone (K = l); four fp16 limb planes. Eight consecutive k of one row n per
// thread (l a multiple of 8, so a group stays in one half), one 16-byte store per plane.
__global__ void prep_query32_kernel(const uint32_t* __restrict__ y, uint64_t plane, uint32_t Q, ipc_geom g,
                                    uint32_t party, uint32_t segments, uint16_t* __restrict__ o0,
                                    uint16_t* __restrict__ o1, uint16_t* __restrict__ o2, uint16_t* __restrict__ o3,
                                    uint32_t n_pad) {
  const uint32_t l = g.rows * g.cols * g.cell, K = segments * l, groups = K / 8;
  const uint64_t tid = blockIdx.x * static_cast<uint64_t>(blockDim.x) + threadIdx.x;
  if (tid >= static_cast<uint64_t>(n_pad) * groups) return;
  const uint32_t n = static_cast<uint32_t>(tid / groups);
  const uint32_t k0 = static_cast<uint32_t>(tid % groups) * 8;
  uint32_t val[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
  if (n < Q * g.R) {
    const uint32_t q = n / g.R, rho = n % g.R;
    const int32_t shift = g.rot_lo + static_cast<int32_t>(rho);
    const bool sum = segments == 2 && k0 < l;  // first half of K = 2l: y_i + y_{i-1}
    const uint32_t kk = k0 < l ? k0 : k0 - l;
    uint32_t c = kk % g.cell;
    const uint32_t cidx = kk / g.cell;
    uint32_t j = cidx % g.cols, r = cidx / g.cols;
    int32_t jsi = (static_cast<int32_t>(j) - shift) % static_cast<int32_t>(g.cols);
    uint32_t js = static_cast<uint32_t>(jsi < 0 ? jsi + static_cast<int32_t>(g.cols) : jsi);
    const uint32_t prev = (party + 2) % 3;
    const uint32_t* yi = y + party * plane + static_cast<uint64_t>(q) * l;
    const uint32_t* yp = y + prev * plane + static_cast<uint64_t>(q) * l;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const uint32_t src = (r * g.cols + js) * g.cell + c;
      val[e] = sum ? yi[src] + yp[src] : yi[src];
      if (++c == g.cell) {
        c = 0;
        if (++js == g.cols) js = 0;
        if (++j == g.cols) {
          j = 0;
          ++r;
        }
      }
    }
  }
  uint32_t w[4][4];
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    int8_t a[4], b[4];
    limbs32(val[2 * v], a);
    limbs32(val[2 * v + 1], b);
#pragma unroll
    for (int i = 0; i < 4; ++i) w[i][v] = f16_of8(a[i]) | (static_cast<uint32_t>(f16_of8(b[i])) << 16);
  }
  uint16_t* out[4] = {o0, o1, o2, o3};
#pragma unroll
  for (int i = 0; i < 4; ++i) *reinterpret_cast<uint4*>(out[i] + tid * 8) = make_uint4(w[i][0], w[i][1], w[i][2], w[i][3]);
}

// ----------------------------------- A3 -----------------------------------
// One CTA per tile of 128 database rows x nw query columns (the launch's columns dealt out in 16-column units,
// so that tiles differ by one unit and none computes padding). With four balanced limbs per operand
// z = sum over s of 2^(8s) S_s, S_s the sum of the limb products x_a y_b, a + b = s (ten per k; products
// with a + b > 3 vanish mod 2^32). The database limbs are widened in registers and stored to tensor
// memory, as in the 16-bit kernel, and the query tiles of a stage lie one under the other in shared
// memory, so that one MMA of N = 2 nw multiplies a limb with two of them; its D is a pair of neighbouring
// accumulators [S_0 | S_1 | S_2 | S_3]:
//     H:  [S_2 | S_3] += x_0 [y_2 | y_3], x_1 [y_1 | y_2], x_2 [y_0 | y_1];  S_3 += x_3 y_0
//     Lo: [S_0 | S_1] += x_0 [y_0 | y_1];  S_1 += x_1 y_0
// Every accumulator starts at 0 and is drained while all partial sums are integers of at most 2^24: H
// every 256 k (S_3 gains at most 4 * 2^14 per k; only (S_2 + 2^8 S_3) mod 2^16 matters), Lo every 512 k.
// While H is drained the Lo products of the next stages run, and the other way round.
// Bound by the MMAs: 5 cycles per k and column, 64 B of query operand per cycle from shared memory. The
// earlier form kept both operands in shared memory, drained every 64 k and needed two passes over K for
// tiles of 256 columns, because four accumulators of that width do not fit the 512 TMEM columns; with A
// in tensor memory narrow MMAs run at the same rate, and 96 columns leave room for two widened k-blocks.
// 65,536 rows x 992 columns (K = 25,600): 20.9 ms against 22.7 ms; 30,000 x 496: 5.06 against 6.07 ms;
// 19,456 x 96 (a tile per SM): 0.59 against 1.60 ms; 1,000 x 31: 0.053 against 1.51 ms. Two warps that
// issue, one for H and one for Lo, take 5.95 ms at 30,000 x 496.
constexpr int TM = 128, KB = 32;
constexpr uint32_t KB_UNIT = 4;        // k-blocks in which K is counted out: 128 elements
constexpr uint32_t HP = 8, LP = 16;    // k-blocks between drains of H and of Lo
constexpr uint32_t LOFF = 4;           // Lo's drains fall at LOFF + i LP, away from H's
constexpr uint32_t KR = 64, KBR = 2;   // elements and k-blocks of a raw or query stage
constexpr uint32_t NQ = 3, MAX_NR = 4;
constexpr uint32_t RAW_TILE = TM * KR, RAW_STAGE = 4 * RAW_TILE;
constexpr uint32_t A_COLS = 64;        // TMEM columns of a widened k-block: four limbs of 16 (two fp16 a column)
constexpr uint32_t SMEM_MAX = 231424;
constexpr uint32_t MAX_TN = 96, MAX_SPLIT = 8;
constexpr uint32_t DW = 8, WW = 8, MAXG = 3, ISSUE_WARPS = 4, THREADS = (ISSUE_WARPS + DW + WW) * 32;
constexpr uint32_t NA3_TN = 80;        // up to here the 512 TMEM columns hold three widened k-blocks beside the accumulators
constexpr uint32_t MAX_NA = 3, NUM_BARS = 2 * NQ + 2 * MAX_NA + 2 * MAX_NR + 6;
static_assert(MAX_TN <= MAXG * 16 * (DW / 4) && WW == 4 * KBR, "a drain thread's columns; a widening group per k-block of a raw stage");

struct Maps32 {
  CUtensorMap b[2][4];  // query limbs [n_pad][K], fp16: boxes of tn columns, and of tn - 16
  CUtensorMap x[2][4];  // database limbs of the two K segments, [x_rows][l] int8
};

struct Tc32Params {
  uint32_t n_cols, x_rows;
  uint32_t tn;  // columns of the widest tiles; the others have 16 less
  uint32_t nr, n_ct, n_rt;
  uint32_t segs, kb_seg;  // K segments; k-blocks of one
  const uint32_t* col_tags;
  uint64_t seed_own, seed_prev;
  uint32_t vec;
  uint32_t* z;
  uint64_t ldz, row0;
  uint32_t* status;
};

// Warps: 0 query copies, 1 MMAs (one elected lane issues), 2 raw copies, 3 joins the query tiles' arrival to
// the widened stage's barrier, 4-11 drain (a TMEM lane quarter and half of the columns each), 12-19
// widening. A cluster's CTAs take parts of K (SPLIT) and join their sums through distributed shared memory.
// Every wait is bounded (2 s, or sooner once another role has failed); a failed CTA raises the status word,
// lets its copies and MMAs finish, frees its tensor memory and stores nothing.
template <uint32_t NA, bool SPLIT>
__device__ __forceinline__ void tc32_tile(const Maps32& maps, const Tc32Params& p, uint32_t q0, uint32_t d0, uint32_t nw,
                                          uint32_t rank, uint32_t n_rank) {
  constexpr uint32_t LEAD = NA, DT = DW * 32;
  static_assert(HP - LOFF >= LEAD && LOFF >= LEAD && LP % HP == 0 && NQ * KBR >= LEAD, "drains apart");
  extern __shared__ uint8_t smem_raw[];
  __shared__ uint32_t s_tmem;
  __shared__ uint32_t s_abort;
  const uint32_t q_tile = nw * 128, q_stage = 4 * q_tile;
  const uint32_t k_units = p.segs * p.kb_seg / KB_UNIT;
  const uint32_t kb0 = SPLIT ? k_units * rank / n_rank * KB_UNIT : 0;
  const uint32_t nst = (SPLIT ? k_units * (rank + 1) / n_rank : k_units) * KB_UNIT - kb0;  // stages: one k-block each
  // two segments are taken in turn, 128 elements each
  auto k_of = [&](uint32_t kb, uint32_t& seg) {
    const uint32_t u = kb / KB_UNIT;
    seg = p.segs == 2 ? u & 1u : 0u;
    return static_cast<int32_t>(((p.segs == 2 ? u >> 1 : u) * KB_UNIT + kb % KB_UNIT) * KB);
  };
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t qring = smem_addr(smem), rring = qring + NQ * q_stage, bars = rring + p.nr * RAW_STAGE;
  const uint32_t q_full = bars, q_empty = q_full + 8 * NQ, a_full = q_empty + 8 * NQ, a_empty = a_full + 8 * NA,
                 r_full = a_empty + 8 * NA, r_empty = r_full + 8 * MAX_NR, h_full = r_empty + 8 * MAX_NR,
                 h_empty = h_full + 8, l_full = h_full + 16, l_empty = h_full + 24, done_bar = h_full + 32;
  volatile uint32_t* abort = &s_abort;
  const uint32_t warp = __shfl_sync(0xFFFFFFFFu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (uint32_t s = 0; s < NQ; ++s) {
      mbar_init(q_full + 8 * s, 1);
      mbar_init(q_empty + 8 * s, 1);
    }
    for (uint32_t s = 0; s < NA; ++s) {
      mbar_init(a_full + 8 * s, WW / 2 + 1);
      mbar_init(a_empty + 8 * s, 1);
    }
    for (uint32_t s = 0; s < MAX_NR; ++s) {
      mbar_init(r_full + 8 * s, 1);
      mbar_init(r_empty + 8 * s, WW);
    }
    mbar_init(h_full, 1);
    mbar_init(h_empty, DW);
    mbar_init(l_full, 1);
    mbar_init(l_empty, DW);
    mbar_init(done_bar, 1);
    s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&s_tmem)), "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = s_tmem, tH = tmem + 2 * nw, tA = tmem + 4 * nw;
  auto all_wait = [&](uint32_t bar, uint32_t par) {
    return __all_sync(0xFFFFFFFFu, mbar_wait(bar, par, p.status, abort)) != 0;
  };
  // z = sum + r_i for four rows of a column, r_i = F(seed_own) - F(seed_prev) (App. C)
  auto put_z = [&](uint32_t col, uint32_t r0, const uint4& a) {
    if (col >= p.n_cols || r0 >= p.x_rows) return;
    const uint32_t req = p.col_tags[2 * col], tag = p.col_tags[2 * col + 1];
    const uint32_t grp = static_cast<uint32_t>((p.row0 + r0) >> 2), ctr3 = (IPC_D_ZA32 << 24) | p.vec;
    const uint4 fo = philox(grp, tag, req, ctr3, p.seed_own);
    const uint4 fp = philox(grp, tag, req, ctr3, p.seed_prev);
    const uint4 v = make_uint4(a.x + fo.x - fp.x, a.y + fo.y - fp.y, a.z + fo.z - fp.z, a.w + fo.w - fp.w);
    uint32_t* dst = p.z + static_cast<uint64_t>(col) * p.ldz + r0;
    if (r0 + 4 <= p.x_rows) {
      __stcs(reinterpret_cast<uint4*>(dst), v);  // streamed: z is read by a later kernel, not from L2
    } else {
      const uint32_t w[4] = {v.x, v.y, v.z, v.w};
      for (uint32_t e = 0; e < p.x_rows - r0; ++e) dst[e] = w[e];
    }
  };

  if (warp == 0) {
    // ---------------------------- query copies -----------------------------
    uint32_t issued = 0;
    for (uint32_t kb = kb0; kb < kb0 + nst; kb += KBR) {
      const uint32_t qs = stage_of<NQ>(issued);
      if (!all_wait(q_empty + 8 * qs, phase_of<NQ>(issued) ^ 1u)) break;
      if (elect_one()) {
        const uint32_t full = q_full + 8 * qs, base = qring + qs * q_stage;
        uint32_t seg;
        const int32_t k = k_of(kb, seg), kx = k + static_cast<int32_t>(seg * p.kb_seg * KB);
        mbar_expect_tx(full, q_stage);
#pragma unroll
        for (uint32_t t = 0; t < 4; ++t) tma_load(base + t * q_tile, &maps.b[nw != p.tn][t], kx, static_cast<int32_t>(q0), full);
      }
      __syncwarp();
      ++issued;
    }
    if (*abort) {
      // copies that may still be in flight land before the CTA leaves (bounded, no abort)
      for (uint32_t G = issued > NQ ? issued - NQ : 0; G < issued; ++G)
        mbar_wait(q_full + 8 * stage_of<NQ>(G), phase_of<NQ>(G), p.status, nullptr);
    }
  } else if (warp == 1) {
    // -------------------------------- MMA issuer --------------------------------
    const uint32_t id1 = (1u << 4) | ((nw >> 3) << 17) | (static_cast<uint32_t>(TM >> 4) << 24);
    const uint32_t id2 = (1u << 4) | ((nw >> 2) << 17) | (static_cast<uint32_t>(TM >> 4) << 24);
    auto wait_stage = [&](uint32_t G) { return all_wait(a_full + 8 * stage_of<NA>(G), phase_of<NA>(G)); };
    auto free_stage = [&](uint32_t G) {
      if (G % KBR == KBR - 1) umma_commit(q_empty + 8 * stage_of<NQ>(G / KBR));
      umma_commit(a_empty + 8 * stage_of<NA>(G));
    };
    auto issue_h = [&](uint32_t G, bool frees) {
      const uint32_t q = qring + stage_of<NQ>(G / KBR) * q_stage + (G % KBR) * 64u, a = tA + stage_of<NA>(G) * A_COLS;
      const bool opens = G % HP == 0;
      if (elect_one()) {
#pragma unroll
        for (uint32_t ks = 0; ks < KB / 16; ++ks) {
          const uint32_t b = q + 32u * ks, x = a + 8 * ks;
          umma_ts(tH, x, sdesc128(b + 2 * q_tile), id2, !(opens && ks == 0));  // x_0 [y_2 | y_3]
          umma_ts(tH, x + 16, sdesc128(b + q_tile), id2, true);                // x_1 [y_1 | y_2]
          umma_ts(tH, x + 32, sdesc128(b), id2, true);                         // x_2 [y_0 | y_1]
          umma_ts(tH + nw, x + 48, sdesc128(b), id1, true);                    // x_3 y_0
        }
        if ((G + 1) % HP == 0 || G + 1 == nst) umma_commit(h_full);
        if (frees) free_stage(G);
      }
      __syncwarp();
    };
    auto issue_l = [&](uint32_t G, bool frees) {
      const uint32_t q = qring + stage_of<NQ>(G / KBR) * q_stage + (G % KBR) * 64u, a = tA + stage_of<NA>(G) * A_COLS;
      const bool opens = G == 0 || G % LP == LOFF;
      if (elect_one()) {
#pragma unroll
        for (uint32_t ks = 0; ks < KB / 16; ++ks) {
          const uint32_t b = q + 32u * ks, x = a + 8 * ks;
          umma_ts(tmem, x, sdesc128(b), id2, !(opens && ks == 0));  // x_0 [y_0 | y_1]
          umma_ts(tmem + nw, x + 16, sdesc128(b), id1, true);       // x_1 y_0
        }
        if (frees) free_stage(G);
        if ((G + 1) % LP == LOFF || G + 1 == nst) umma_commit(l_full);
      }
      __syncwarp();
    };
    uint32_t h_per = 0, l_per = 0;
    bool ok = true;
    for (uint32_t s = 0; s < nst && ok;) {
      const bool h_opens = s % HP == 0, l_opens = s == 0 || s % LP == LOFF;
      const uint32_t lead = nst - s < LEAD ? nst - s : LEAD;
      if (h_opens && !l_opens) {
        // the Lo products of the next stages run while H is drained
        for (uint32_t j = 0; j < lead && ok; ++j) {
          if (!(ok = wait_stage(s + j))) break;
          fence_after();
          issue_l(s + j, false);
        }
        if (!ok || !(ok = all_wait(h_empty, (h_per++ & 1u) ^ 1u))) break;
        fence_after();
        for (uint32_t j = 0; j < lead; ++j) issue_h(s + j, true);
        s += lead;
      } else if (l_opens) {
        // the H products of the next stages run while Lo is drained (at s = 0 both begin)
        if (h_opens && !(ok = all_wait(h_empty, (h_per++ & 1u) ^ 1u))) break;
        for (uint32_t j = 0; j < lead && ok; ++j) {
          if (!(ok = wait_stage(s + j))) break;
          fence_after();
          issue_h(s + j, false);
        }
        if (!ok || !(ok = all_wait(l_empty, (l_per++ & 1u) ^ 1u))) break;
        fence_after();
        for (uint32_t j = 0; j < lead; ++j) issue_l(s + j, true);
        s += lead;
      } else {
        if (!(ok = wait_stage(s))) break;
        fence_after();
        issue_h(s, false);
        issue_l(s, true);
        ++s;
      }
    }
    // every MMA issued above completes before the tensor memory is freed
    if (elect_one()) umma_commit(done_bar);
    __syncwarp();
    mbar_wait(done_bar, 0, p.status, nullptr);
  } else if (warp == 2) {
    // ------------------------------- raw copies ---------------------------------
    Ring r;
    uint32_t issued = 0;
    for (uint32_t kb = kb0; kb < kb0 + nst; kb += KBR) {
      if (!all_wait(r_empty + 8 * r.s, r.ph ^ 1u)) break;
      if (elect_one()) {
        const uint32_t full = r_full + 8 * r.s, base = rring + r.s * RAW_STAGE;
        uint32_t seg;
        const int32_t kx = k_of(kb, seg);
        mbar_expect_tx(full, RAW_STAGE);
#pragma unroll
        for (uint32_t t = 0; t < 4; ++t)
          tma_load(base + t * RAW_TILE, &maps.x[seg][t], kx, static_cast<int32_t>(d0), full);
      }
      __syncwarp();
      ++issued;
      r.next(p.nr);
    }
    if (*abort) {
      for (uint32_t G = issued > p.nr ? issued - p.nr : 0; G < issued; ++G)
        mbar_wait(r_full + 8 * (G % p.nr), (G / p.nr) & 1u, p.status, nullptr);
    }
  } else if (warp == 3) {
    // a widened stage's full barrier also counts the arrival of its query tiles; a_empty keeps the turn
    for (uint32_t G = 0; G < nst; ++G) {
      if (G % KBR == 0 && !all_wait(q_full + 8 * stage_of<NQ>(G / KBR), phase_of<NQ>(G / KBR))) break;
      if (!all_wait(a_empty + 8 * stage_of<NA>(G), phase_of<NA>(G) ^ 1u)) break;
      if (lane == 0) mbar_arrive(a_full + 8 * stage_of<NA>(G));
    }
  } else if (warp >= ISSUE_WARPS + DW) {
    // -------------------------------- widening ----------------------------------
    // the first four warps take the even k-blocks (a raw stage's first), the others the odd ones
    const uint32_t kr = (warp - ISSUE_WARPS - DW) >> 2, row = 32 * (warp & 3u) + lane, x = (row >> 1) & 3u;
    const uint32_t lane_base = (32u * (warp & 3u)) << 16;
    // chunks 2 kr, 2 kr + 1 of the 64-byte swizzled row
    const uint32_t o0 = ((2 * kr) ^ x) * 16, o1 = ((2 * kr + 1) ^ x) * 16;
    Ring r;
    for (uint32_t G = kr; G < nst; G += KBR) {
      if (!all_wait(r_full + 8 * r.s, r.ph)) break;
      const uint32_t src = rring + r.s * RAW_STAGE + row * KR, dst = tA + lane_base + stage_of<NA>(G) * A_COLS;
      uint32_t w[32];
      auto widen = [&](uint32_t limb) {  // this row's 32 elements of limbs `limb` and `limb` + 1
        const uint32_t t0 = src + limb * RAW_TILE, t1 = t0 + RAW_TILE;
        const uint4 v[4] = {lds128(t0 + o0), lds128(t0 + o1), lds128(t1 + o0), lds128(t1 + o1)};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          uint4 c0, c1;
          widen16(v[e], c0, c1);
          w[8 * e] = c0.x, w[8 * e + 1] = c0.y, w[8 * e + 2] = c0.z, w[8 * e + 3] = c0.w;
          w[8 * e + 4] = c1.x, w[8 * e + 5] = c1.y, w[8 * e + 6] = c1.z, w[8 * e + 7] = c1.w;
        }
      };
      widen(0);
      if (!all_wait(a_empty + 8 * stage_of<NA>(G), phase_of<NA>(G) ^ 1u)) break;
      fence_after();
      tmem_st32(dst, w);
      widen(2);
      __syncwarp();
      if (lane == 0) mbar_arrive(r_empty + 8 * r.s);
      r.next(p.nr);
      tmem_st32(dst + 32, w);
      tmem_wait_st();
      fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(a_full + 8 * stage_of<NA>(G));
    }
  } else {
    // ----------------------------------- drain ----------------------------------
    const uint32_t half = (warp - ISSUE_WARPS) >> 2, span = (nw / 16 + 1) / 2 * 16, col0 = half * span;
    const uint32_t ng = col0 < nw ? ((nw - col0 < span ? nw - col0 : span) / 16) : 0;
    const uint32_t t0 = tmem + ((32u * (warp & 3u)) << 16) + col0;
    uint32_t acc[16 * MAXG];  // this row's sums of the warp's columns mod 2^32
#pragma unroll
    for (uint32_t k = 0; k < 16 * MAXG; ++k) acc[k] = 0;
    // one drain: the pair of accumulators at t, 16 columns of each at a time, to f; then the pair is released
    auto drain = [&](uint32_t full, uint32_t par, uint32_t t, uint32_t empty, auto&& f) {
      if (!all_wait(full, par)) return false;
      fence_after();
#pragma unroll
      for (uint32_t g = 0; g < MAXG; ++g) {
        if (g < ng) {
          uint32_t a[16], b[16];
          tmem_ld16(t + 16 * g, a);
          tmem_ld16(t + nw + 16 * g, b);
          tmem_wait_ld();
          if (g == ng - 1) {  // the last of this warp's columns is in registers
            fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(empty);
          }
          f(g, a, b);
        }
      }
      if (ng == 0 && lane == 0) mbar_arrive(empty);
      return true;
    };
    uint32_t h_per = 0, l_per = 0;
    bool ok = true;
    for (uint32_t s = 1; s <= nst && ok; ++s) {
      if (s % HP == 0 || s == nst)
        ok = drain(h_full, h_per++ & 1u, t0 + 2 * nw, h_empty, [&](uint32_t g, const uint32_t (&a)[16], const uint32_t (&b)[16]) {
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            const uint32_t u = add16x2(low16x2<1>(a[2 * k], a[2 * k + 1]), low16x2<256>(b[2 * k], b[2 * k + 1]));
            acc[16 * g + 2 * k] += u << 16;
            acc[16 * g + 2 * k + 1] += u & 0xFFFF0000u;
          }
        });
      if (ok && (s % LP == LOFF || s == nst))
        ok = drain(l_full, l_per++ & 1u, t0, l_empty, [&](uint32_t g, const uint32_t (&a)[16], const uint32_t (&b)[16]) {
#pragma unroll
          for (int k = 0; k < 16; ++k)
            acc[16 * g + k] += static_cast<uint32_t>(__float2int_rn(__uint_as_float(a[k]))) +
                               (static_cast<uint32_t>(__float2int_rn(__uint_as_float(b[k]))) << 8);
        });
    }
    // ---- epilogue: the sums through the (now idle) query ring, then four rows of a column at a time ----
    if (!named_sync_or(1, DT, *abort != 0)) {
      uint32_t* zs = reinterpret_cast<uint32_t*>(smem);  // [nw][TM]
      const uint32_t row = 32 * (warp & 3u) + lane;
#pragma unroll
      for (uint32_t k = 0; k < 16 * MAXG; ++k)
        if (k < 16 * ng) zs[(col0 + k) * TM + row] = acc[k];
      if (!SPLIT) {
        named_sync(1, DT);
        for (uint32_t it = threadIdx.x - ISSUE_WARPS * 32; it < nw * (TM / 4); it += DT)
          put_z(q0 + it / (TM / 4), d0 + 4 * (it % (TM / 4)), *reinterpret_cast<const uint4*>(zs + it * 4));
      }
    }
  }
  if (SPLIT) {
    // every thread of every CTA passes both cluster barriers, also after a failed wait
    __syncwarp();
    cluster_sync();
    if (warp >= ISSUE_WARPS && warp < ISSUE_WARPS + DW) {
      bool bad = false;
      for (uint32_t r = 0; r < n_rank; ++r) bad = bad || ld_cluster32(mapa(smem_addr(&s_abort), r)) != 0;
      if (!bad)
        for (uint32_t it = rank * DT + threadIdx.x - ISSUE_WARPS * 32; it < nw * (TM / 4); it += n_rank * DT) {
          uint4 v = make_uint4(0, 0, 0, 0);
          for (uint32_t r = 0; r < n_rank; ++r) {
            const uint4 o = ld_cluster128(mapa(qring + it * 16, r));
            v = make_uint4(v.x + o.x, v.y + o.y, v.z + o.z, v.w + o.w);
          }
          put_z(q0 + it / (TM / 4), d0 + 4 * (it % (TM / 4)), v);
        }
    }
    __syncwarp();
    cluster_sync();
  }
  fence_before();
  __syncthreads();
  if (warp == 0) {
    fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
  }
}

template <bool SPLIT>
__global__ void __launch_bounds__(THREADS, 1)
    gemm_tc32_kernel(const __grid_constant__ Maps32 maps, const __grid_constant__ Tc32Params p) {
  uint32_t rank = 0, n_rank = 1;
  if (SPLIT) {
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(n_rank));
  }
  // the tile, nw columns wide: the tiles with 16 columns more come first, and of each width bands of up to 8
  // column tiles, all row tiles of a band before the next. A band's tiles stream K in step and share the
  // database in L2; with both widths in a band they did not (65,536 x 992: 62.9 GB read for 25.3 so, 22.1 ms
  // for 20.9; x 496 11.9 for 10.8).
  constexpr uint32_t kBand = 8;
  uint32_t q0, d0, nw;
  {
    const uint32_t units = (p.n_cols + 15) / 16, base = units / p.n_ct, rem = units % p.n_ct;
    uint32_t lin = blockIdx.x / n_rank, first = 0, of = rem;
    if (lin >= rem * p.n_rt) {
      lin -= rem * p.n_rt;
      first = rem;
      of = p.n_ct - rem;
    }
    const uint32_t band = lin / (kBand * p.n_rt), c0 = band * kBand;
    const uint32_t width = of - c0 < kBand ? of - c0 : kBand;
    const uint32_t in_band = lin - band * kBand * p.n_rt, ct = first + c0 + in_band % width;
    q0 = 16 * (ct * base + (ct < rem ? ct : rem));
    nw = 16 * (base + (ct < rem ? 1 : 0));
    d0 = in_band / width * TM;
  }
  if (nw > NA3_TN)
    tc32_tile<2, SPLIT>(maps, p, q0, d0, nw, rank, n_rank);
  else
    tc32_tile<3, SPLIT>(maps, p, q0, d0, nw, rank, n_rank);
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

uint32_t cdiv(uint32_t a, uint32_t b) { return (a + b - 1) / b; }

// CTAs that run at once in clusters of k, by device (set with the kernels' attributes).
uint32_t g_at_once[64][MAX_SPLIT + 1];

cudaError_t ready() {
  const void* k[2] = {reinterpret_cast<const void*>(&gemm_tc32_kernel<false>),
                      reinterpret_cast<const void*>(&gemm_tc32_kernel<true>)};
  cudaError_t e = load_kernels({reinterpret_cast<const void*>(&prep_query32_kernel)});
  for (const void* f : k)
    if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_MAX);
  int dev = 0;
  if (e == cudaSuccess) e = cudaGetDevice(&dev);
  for (uint32_t s = 2; s <= MAX_SPLIT && e == cudaSuccess && dev >= 0 && dev < 64; ++s) {
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = s;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(s);
    cfg.blockDim = dim3(THREADS);
    cfg.dynamicSmemBytes = SMEM_MAX;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    e = cudaOccupancyMaxActiveClusters(&n, gemm_tc32_kernel<true>, &cfg);
    g_at_once[dev][s] = e == cudaSuccess ? static_cast<uint32_t>(n) * s : 0;
  }
  return e;
}

// Column tiles and parts of K with the shortest estimate. A tile of w columns takes 68 + 9.9 w cycles a k-block,
// a line through launches of the measured widths, and at least 650 (the raw copies and the widening). Its
// tiles have base 16-column units or one more. Few rounds of the chip end together where all tiles are equal;
// unequal ones fill half a round more than their number, but no round is shorter than the narrowest tile or
// longer than the widest. `together` launches fill each other's last rounds. Then the parts of K, each with a
// start and an end. Measured, tiles of two widths against equal ones with padding: 30,000 rows x 496 columns
// 5.06 ms against 5.34, 17,000 x 372 2.14 against 2.38, 8,000 x 1,240 3.30 against 3.40.
void pick_shape(uint32_t n_cols, uint32_t row_tiles, uint32_t kb_total, uint32_t together, uint32_t& n_ct, uint32_t& split) {
  int dev = 0;
  const uint32_t* at_once = cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < 64 ? g_at_once[dev] : nullptr;
  const double sms = sm_count_current();
  const uint32_t units = cdiv(n_cols, 16), least = cdiv(units, MAX_TN / 16);
  auto cycles = [](uint32_t w) { return std::max(650.0, 68 + 9.9 * 16 * w); };
  double best = 1e300;
  for (uint32_t t = least; t <= least + 3 && t <= units; ++t) {
    const uint32_t base = units / t, rem = units % t;
    const double ctas = static_cast<double>(t) * row_tiles * together, most = cycles(base + (rem > 0)),
                 mean = (rem * cycles(base + 1) + (t - rem) * cycles(base)) / t;
    for (uint32_t s = 1; s <= MAX_SPLIT && s <= kb_total / KB_UNIT; ++s) {
      if (s > 1 && (!at_once || at_once[s] == 0)) continue;
      const double rounds = ctas * s / (s == 1 ? sms : at_once[s]), whole = std::ceil(rounds);
      double tiles = (rounds + 0.5) * mean;
      if (rounds < 8) tiles = std::min(std::max(rem ? tiles : 0.0, whole * cycles(base)), whole * most);
      const double cost = tiles * kb_total / s + whole * (s == 1 ? 10000 : 14000);
      if (cost < best * 0.999) {
        best = cost;
        n_ct = t;
        split = s;
      }
    }
  }
}

int launch_tc32(const Maps32& m, const Tc32Params& p, uint32_t split, uint32_t smem, cudaStream_t stream) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(p.n_ct * p.n_rt * split);
  cfg.blockDim = dim3(THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute at[1];
  if (split > 1) {
    at[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
    at[cfg.numAttrs].val.clusterDim.x = split;
    at[cfg.numAttrs].val.clusterDim.y = at[cfg.numAttrs].val.clusterDim.z = 1;
    ++cfg.numAttrs;
  }
  cfg.attrs = at;
  IPC_CUDA_TRY(cudaLaunchKernelEx(&cfg, split > 1 ? gemm_tc32_kernel<true> : gemm_tc32_kernel<false>, m, p));
  return IPC_OK;
}

}  // namespace

// As ring_gemm_ts_ready.
int ring_gemm_tc32_ready() {
  static PerDevice attr;
  IPC_CUDA_TRY(attr.run(ready));
  return IPC_OK;
}

// Whether a chunk's Z_2^32 GEMMs run best one after another: over many rounds of the chip three launches' tiles
// drift until they no longer share what lies in L2, if that does not hold two query operands; over few, launches
// side by side fill each other's last rounds. Requests without lifting, sustained, in ms (side by side / in turn):
//     30,000 rows x   496 columns ( 9 rounds a launch)  29.6 /  30.5
//     30,000      x   992         (17)                  59.6 /  59.5
//     16,384      x 1,984         (18)                  66.2 /  63.6
//     65,536      x   744         (27)                  99.7 /  96.4
//     65,536      x   992         (37)                 129.9 / 125.9
bool ring_gemm_tc32_in_turn(uint32_t segments, size_t x_rows, uint32_t n_cols, uint32_t l) {
  const double rounds = static_cast<double>(cdiv(n_cols, MAX_TN)) * cdiv(static_cast<uint32_t>(x_rows), TM) / sm_count_current();
  return 2 * 8ull * segments * l * n_cols > L2_QUERY_BYTES && rounds >= 17;
}

// segments: 2 for K = 2l over [x[0..3] | x[4..7]] (ABY3 replicated sharing, x[4..7] the
// previous party's component), 1 for K = l over x[0..3] alone. K must be a multiple of 256. together: like
// launches in flight at the same time, this one among them.
int ring_gemm_tc32(uint32_t segments, const int8_t* const x[8], size_t x_rows, const uint16_t* const b[4],
                   uint32_t n_cols, uint32_t n_pad, uint32_t l, const uint32_t* col_tags, uint64_t seed_own,
                   uint64_t seed_prev, uint32_t vec, uint32_t* z, size_t ldz, uint64_t row0, uint32_t together,
                   cudaStream_t stream) {
  if (segments != 1 && segments != 2) {
    set_error("Z_2^32 ring GEMM: one or two K segments");
    return IPC_EINVAL;
  }
  if ((segments * l) % (8 * KB) != 0) {
    set_error("Z_2^32 ring GEMM: K must be a multiple of 256");
    return IPC_EINVAL;
  }
  if (n_pad % 128 != 0 || n_cols > n_pad || ldz % 4 != 0 || ldz < x_rows || !aligned16(z)) {
    set_error("Z_2^32 ring GEMM: n_pad % 128, n_cols <= n_pad, ldz % 4, ldz >= x_rows and a 16-byte aligned z");
    return IPC_EINVAL;
  }
  if (x_rows == 0 || n_cols == 0) return IPC_OK;
  if (x_rows > 65535ull * TM) {
    set_error("Z_2^32 ring GEMM: too many rows for one launch");
    return IPC_EINVAL;
  }
  if (const int rc = ring_gemm_tc32_ready()) return rc;
  Tc32Params p{};
  p.n_rt = static_cast<uint32_t>((x_rows + TM - 1) / TM);
  p.n_ct = 1;
  uint32_t split = 1;
  pick_shape(n_cols, p.n_rt, segments * l / KB, together, p.n_ct, split);
  p.tn = 16 * cdiv(cdiv(n_cols, 16), p.n_ct);
  const uint32_t q_stage = 4 * p.tn * 128;
  p.nr = std::min(MAX_NR, (SMEM_MAX - 1024 - 8 * NUM_BARS - NQ * q_stage) / RAW_STAGE);
  const uint32_t smem = 1024 + NQ * q_stage + p.nr * RAW_STAGE + 8 * NUM_BARS;
  Maps32 m;
  int rc;
  for (int i = 0; i < 4; ++i) {
    if ((rc = make_map_f16k64(&m.b[0][i], b[i], static_cast<uint64_t>(segments) * l, n_pad, p.tn)) ||
        (rc = make_map_f16k64(&m.b[1][i], b[i], static_cast<uint64_t>(segments) * l, n_pad, std::max(16u, p.tn - 16))) ||
        (rc = make_map_raw(&m.x[0][i], x[i], l, x_rows, KR, TM)) ||
        (rc = make_map_raw(&m.x[1][i], x[segments == 2 ? 4 + i : i], l, x_rows, KR, TM)))
      return rc;
  }
  p.n_cols = n_cols;
  p.x_rows = static_cast<uint32_t>(x_rows);
  p.segs = segments;
  p.kb_seg = l / KB;
  p.col_tags = col_tags;
  p.seed_own = seed_own;
  p.seed_prev = seed_prev;
  p.vec = vec;
  p.z = z;
  p.ldz = ldz;
  p.row0 = row0;
  p.status = status_ptr();
  return launch_tc32(m, p, split, smem, stream);
}

int prep_query32(const uint32_t* y, uint64_t y_plane, uint32_t Q, const ipc_geom* g, uint32_t party,
                 uint32_t segments, uint16_t* const b[4], uint32_t n_pad, cudaStream_t stream) {
  const uint64_t l = g ? static_cast<uint64_t>(g->rows) * g->cols * g->cell : 0;
  if (!g || l == 0 || g->R == 0 || g->R > 31 || party > 2 || (segments != 1 && segments != 2) || !y || !b || !b[0] ||
      !b[1] || !b[2] || !b[3] || Q == 0 || static_cast<uint64_t>(Q) * g->R > n_pad) {
    set_error("Z_2^32 query operand: bad geometry, party, segments, pointers or n_pad < Q*R");
    return IPC_EINVAL;
  }
  for (int i = 0; i < 4; ++i)
    if (reinterpret_cast<uintptr_t>(b[i]) & 15u) {
      set_error("Z_2^32 query operand: limb planes must be 16-byte aligned");
      return IPC_EINVAL;
    }
  const uint64_t threads = static_cast<uint64_t>(n_pad) * segments * l / 8;
  const uint32_t bs = 256;
  prep_query32_kernel<<<static_cast<unsigned>((threads + bs - 1) / bs), bs, 0, stream>>>(
      y, y_plane, Q, *g, party, segments, b[0], b[1], b[2], b[3], n_pad);
  IPC_CUDA_TRY(cudaGetLastError());
  return IPC_OK;
}

}  // namespace ipc

using namespace ipc;

extern "C" int ipc_encode_share32(const uint64_t* code_bits, const uint64_t* mask_bits, uint32_t n, uint32_t l,
                                  uint64_t client_seed, uint32_t side, uint32_t idx0, uint32_t* code_sh,
                                  uint32_t* mask_sh, void* stream) {
  if (l == 0 || l % 2 != 0 || !code_bits || !mask_bits || !code_sh || !mask_sh) {
    set_error("ipc_encode_share32: l must be a positive even number and pointers non-null");
    return IPC_EINVAL;
  }
  if (n == 0) return IPC_OK;
  const uint64_t total = static_cast<uint64_t>(n) * (l / 2);
  const uint32_t bs = 256;
  encode_share32_kernel<<<static_cast<unsigned>((total + bs - 1) / bs), bs, 0, static_cast<cudaStream_t>(stream)>>>(
      code_bits, mask_bits, n, l, philox_key(client_seed), side, idx0, code_sh, mask_sh);
  IPC_CUDA_TRY(cudaGetLastError());
  return IPC_OK;
}

extern "C" int ipc_split_limbs32(const uint32_t* x, size_t count, int8_t* const limbs[4], void* stream) {
  if (!x || !limbs || !limbs[0] || !limbs[1] || !limbs[2] || !limbs[3]) {
    set_error("ipc_split_limbs32: null pointer");
    return IPC_EINVAL;
  }
  if (!aligned16(x)) {
    set_error("ipc_split_limbs32: x must be 16-byte aligned");
    return IPC_EINVAL;
  }
  for (int i = 0; i < 4; ++i)
    if (reinterpret_cast<uintptr_t>(limbs[i]) & 3u) {
      set_error("ipc_split_limbs32: limb planes must be 4-byte aligned");
      return IPC_EINVAL;
    }
  if (count == 0) return IPC_OK;
  const size_t threads = (count + 3) / 4;
  const uint32_t bs = 256;
  split_limbs32_kernel<<<static_cast<unsigned>((threads + bs - 1) / bs), bs, 0, static_cast<cudaStream_t>(stream)>>>(
      x, count, limbs[0], limbs[1], limbs[2], limbs[3]);
  IPC_CUDA_TRY(cudaGetLastError());
  return IPC_OK;
}

extern "C" int ipc_prep_query32_f16(const uint32_t* y, uint32_t Q, const ipc_geom* g, uint32_t party,
                                    uint32_t segments, uint16_t* const b[4], uint32_t n_pad, void* stream) {
  const uint64_t l = g ? static_cast<uint64_t>(g->rows) * g->cols * g->cell : 0;
  return prep_query32(y, Q * l, Q, g, party, segments, b, n_pad, static_cast<cudaStream_t>(stream));
}

extern "C" int ipc_ring_gemm_tc32(uint32_t segments, const int8_t* const x[8], size_t x_rows,
                                  const uint16_t* const b[4], uint32_t n_cols, uint32_t n_pad, uint32_t l,
                                  const uint32_t* col_tags, uint64_t seed_own, uint64_t seed_prev, uint32_t vec,
                                  uint32_t* z, size_t ldz, uint64_t row0, void* stream) {
  if (!x || !b || !col_tags || !z) {
    set_error("ipc_ring_gemm_tc32: null pointer");
    return IPC_EINVAL;
  }
  for (int i = 0; i < 4; ++i)
    if (!x[i] || !b[i] || (segments == 2 && !x[4 + i]) || !aligned16(x[i]) || !aligned16(b[i]) ||
        (segments == 2 && !aligned16(x[4 + i]))) {
      set_error("ipc_ring_gemm_tc32: limb planes must be non-null and 16-byte aligned");
      return IPC_EINVAL;
    }
  if (x_rows > IPC_MAX_GEMM_ROWS) {
    set_error("ipc_ring_gemm_tc32: x_rows above IPC_MAX_GEMM_ROWS");
    return IPC_EINVAL;
  }
  if (l % 16 != 0) {
    set_error("ipc_ring_gemm_tc32: l must be a multiple of 16");
    return IPC_EINVAL;
  }
  return ring_gemm_tc32(segments, x, x_rows, b, n_cols, n_pad, l, col_tags, seed_own, seed_prev, vec, z, ldz, row0, 1,
                        static_cast<cudaStream_t>(stream));
}
