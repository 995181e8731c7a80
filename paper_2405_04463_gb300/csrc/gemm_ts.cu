// A3 on the 5th-generation tensor cores: tcgen05.mma (kind::f16) with the database operand in tensor
// memory (A from TMEM) and the query operand in shared memory, fp16 operands carrying the balanced
// int8 limbs, fp32 accumulators.
//
// The ring product is the three limb products of Sec. 6.1:
//     z = L + 256 C + r  (mod 2^16),  L = sum lo*lo',  C = sum (lo*hi' + hi*lo').
// sm_103a has no integer tcgen05 kind, but the arithmetic is exact on the f16 kind:
//   * every limb is an integer in [-128, 127], exactly an fp16 value, and every product an integer
//     with |p| <= 2^14, exact in fp32;
//   * an accumulator starts at 0 (the first MMA of a period overwrites it) and is drained after at most
//     1,024 products (C every 512 k, two products per k; L every 1,024 k), so every partial sum, in any
//     order or grouping, is an integer of at most 2^24 in size, which fp32 holds exactly.
//
// The database stays resident as int8 limb planes (the size of its u16 shares). TMA brings raw int8
// tiles into shared memory; widening warps read one row per thread, make fp16 pairs in registers and
// store them to tensor memory, where the MMAs read them. Neither the widened tile nor the A operand of
// the MMAs passes through shared memory. That was the bound of the form with both operands in shared
// memory: per k-block of 32 and 256 columns it moved 6 x 12 KB of MMA operands, 40 KB of copies, 8 KB of
// raw reads and 16 KB of widened writes, 1,088 cycles at 128 B per cycle against 768 of the tensor pipe,
// and ran at 1,090. Here 208 columns move 40 KB + 35 KB + 8 KB, 650 cycles against 624.
// MMAs with A in tensor memory also run at N / 2 cycles down to N = 32 (64 cycles at least with A in
// shared memory), so a tile is as wide as its columns: the width is a launch parameter.
//
// Measured (one ring GEMM of l = 12,800, K = 25,600, CUDA events, both forms in turn in one process):
//   65,536 rows x 992 columns: 5.6-5.8 ms against 6.3-6.6 ms (power cap; 5.4 against 6.1 ms cold);
//   100,000 rows x 31 columns: 0.87 ms against 2.57 ms (the database bytes at 5.9 TB/s);
//   1,000 rows x 4 columns: 0.023 ms against 0.43 ms (K split over a cluster);
//   19,456 rows (one tile per SM): 64 / 128 / 160 / 208 columns 0.17 / 0.25 / 0.31 / 0.37 ms against 0.44-0.48.
//
// Roles (one CTA per tile of 128 database rows x tn query columns, 16 warps):
//   warp 0         query copies: tn x 64 fp16 lo and hi tiles, 128-byte swizzle.
//   warp 1         MMAs. The whole warp runs the loop and one elected lane issues: MMAs take uniform
//                  registers, and issued from a lane's own branch each cost tens of cycles more (a
//                  k-block took 1,270 cycles so).
//   warp 2         raw copies: 128 rows x 64 or 128 int8 of both planes.
//   warp 3         arrives on a stage's full barrier when its query tiles have landed, so that the MMA
//                  warp has one barrier per stage to look at (two waits a k-block cost 20 % at 208 columns).
//   4 or 8 warps   drain: a thread owns one TMEM lane (database row) and up to 112 or 160 columns, their
//                  running sums kept mod 2^16 two to a register.
//   8 or 4 warps   widening, four warps (a TMEM lane quarter each) per k-block.
// TMEM: L in columns [0, tn), C in [tn, 2 tn), then NA widened stages.
// While C is drained the MMA warp runs the L products of the next stages, and the other way round; the
// two accumulators' periods are shifted against each other so that their drains do not meet.
//
// A launch holds up to six passes (ring GEMMs of one chunk: their own operands, zero shares and z) and
// takes one tile per CTA, or walks a device-side list of column tiles with one CTA per SM. Where the
// tiles do not fill the chip, the CTAs of a cluster take parts of K and join their sums through
// distributed shared memory.
// Every mbarrier wait is bounded (2 s, or sooner once another role has failed); a failed CTA raises the
// status word, lets its copies and MMAs finish, frees its tensor memory and stores nothing.
#include <algorithm>
#include <cmath>

#include "gemm_ts.cuh"
#include "tcgen05_ts.cuh"

namespace ipc {
namespace {

using namespace tc;

constexpr int TM = 128;               // database rows per tile (MMA M = TMEM lanes)
constexpr int KB = 32;                // elements of K in a k-block
constexpr uint32_t KB_UNIT = 4;       // k-blocks in which K is counted out: 128 elements, the granule of l
constexpr uint32_t CP = 16, LP = 32;  // k-blocks between drains of C (512 k) and of L (1,024 k)
constexpr int ISSUE_WARPS = 4;
constexpr uint32_t MAX_NR = 8;        // raw stages at most
constexpr uint32_t SMEM_MAX = 231424;  // dynamic shared memory, leaving room for the static words
constexpr uint32_t A_COLS = 32;       // TMEM columns of a widened k-block: lo 16, hi 16 (two fp16 a column)
constexpr double LAUNCH_ROUNDS = 32;  // of the chip, of a launch whose passes' query operands don't fit the L2
constexpr uint32_t MAX_TN = 208;      // 2 x 208 accumulator columns leave three widened k-blocks

struct TsPass {
  uint16_t* z;
  uint64_t seed_own, seed_prev;
  uint32_t vec, x0, x1;  // x0, x1: map pairs of the first and second K segment's database planes
  uint32_t segs;         // K segments: 2 (replicated sharing) or 1
};
struct TsParams {
  uint32_t n_cols, x_rows;
  uint32_t tn;                 // query columns per tile, a multiple of 16
  uint32_t nr;                 // raw stages
  uint32_t kb_seg;             // k-blocks of a K segment, l / KB
  uint32_t n_col_tiles, n_row_tiles, n_pass;
  uint32_t pass_inner;         // the passes of a tile are neighbours (else all tiles of a pass come first)
  const uint32_t* col_tiles;
  const uint32_t* n_col_list;
  const uint32_t* col_tags;
  uint64_t ldz, row0;
  uint32_t* status;
  TsPass pass[RING_GEMM_PASSES];
};
struct TsMaps {
  CUtensorMap q[RING_GEMM_PASSES][2];
  CUtensorMap x[RING_GEMM_PASSES][2];
};

// Stages one accumulator runs ahead while the other is drained, and the stage (of L's period) at which
// L's drains fall, away from those of C.
template <int KBS>
struct Sched;
template <>
struct Sched<1> {
  static constexpr uint32_t LEAD = 3, LOFF = 8;
};
template <>
struct Sched<2> {
  static constexpr uint32_t LEAD = 2, LOFF = 4;
};
template <>
struct Sched<4> {
  static constexpr uint32_t LEAD = 2, LOFF = 6;
};

// KBS: k-blocks of a widened stage; KQ: of a query stage; KR: elements of K of a raw stage; NA, NQ:
// widened and query stages; DW, WW: drain and widening warps; MAXG: 16-column groups of a drain thread.
// PAIR: both limb products of lo in one MMA, its B the lo and hi query tiles one under the other
// (N = 2 tn) and its D [L | C]; two such accumulator pairs take turns, so no drain is waited for. At
// 32 columns the MMA warp needs 40-50 cycles to issue an MMA of 16, and this saves one in three:
// 100,000 rows x 62 columns 0.88 ms against 1.04 ms, 93 columns 1.32 against 1.49 ms.
// LISTED: also built for lists of column tiles, whose widths are 64, 128 and 208.
template <int KBS_, int KQ_, int KR_, uint32_t NA_, uint32_t NQ_, int DW_, int WW_, int MAXG_, bool LISTED_, bool PAIR_ = false>
struct Cfg {
  static constexpr bool PAIR = PAIR_, LISTED = LISTED_;
  static constexpr uint32_t KBS = KBS_, KQ = KQ_, KR = KR_, NA = NA_, NQ = NQ_, DW = DW_, WW = WW_, MAXG = MAXG_;
  static constexpr uint32_t THREADS = (ISSUE_WARPS + DW + WW) * 32;
  static constexpr uint32_t RAW_STAGE = 2 * TM * KR;  // lo and hi tiles
  static constexpr uint32_t NUM_BARS = 2 * NQ + 2 * NA + 2 * MAX_NR + 6;
  static constexpr uint32_t q_stage(uint32_t tn) { return KQ * 2 * tn * KB * 2; }
  // the widest tile: its accumulators and widened stages fit the 512 TMEM columns
  static constexpr uint32_t TN_TMEM = (512 - NA * KBS * A_COLS) / (PAIR ? 4 : 2), TN_DRAIN = MAXG * 16 * (DW / 4);
  static constexpr uint32_t TN = TN_TMEM < TN_DRAIN ? TN_TMEM : TN_DRAIN;
  static constexpr uint32_t raw_stages(uint32_t tn) {
    const uint32_t n = (SMEM_MAX - 1024 - 8 * NUM_BARS - NQ * q_stage(tn)) / RAW_STAGE;
    return n < MAX_NR ? n : MAX_NR;
  }
  static constexpr uint32_t smem(uint32_t tn, uint32_t nr) { return 1024 + NQ * q_stage(tn) + nr * RAW_STAGE + 8 * NUM_BARS; }
  static_assert((KR == 64 || KR == 128) && KQ % KBS == 0 && KQ % 2 == 0 && KB_UNIT % KQ == 0, "stages");
  static_assert(KBS % (WW / 4) == 0 && (KR / KB) % (WW / 4) == 0, "a widening group takes whole k-blocks");
};
// By tile width. Narrow tiles are bound by the database bytes and by the MMA warp's pace per stage: long
// stages and eight widening warps. From 129 columns on TMEM leaves room for shorter stages only.
using Cfg64 = Cfg<4, 4, 128, 2, 4, 4, 8, 4, true, true>;
using Cfg96 = Cfg<2, 2, 128, 2, 4, 4, 8, 6, false, true>;
using Cfg128 = Cfg<2, 2, 128, 4, 4, 4, 8, 8, true>;
using Cfg160 = Cfg<2, 2, 128, 3, 3, 4, 8, 10, false>;
using Cfg192 = Cfg<1, 2, 64, 3, 3, 8, 4, 6, false>;
using Cfg208 = Cfg<1, 2, 64, 3, 3, 8, 4, 7, true>;
static_assert(Cfg64::TN >= 64 && Cfg96::TN >= 96 && Cfg128::TN >= 128 && Cfg160::TN >= 160 && Cfg192::TN >= 192 && Cfg208::TN >= MAX_TN, "");
static_assert(Cfg64::raw_stages(64) >= 2 && Cfg96::raw_stages(96) >= 2 && Cfg128::raw_stages(128) >= 2 && Cfg160::raw_stages(160) >= 2 &&
                  Cfg192::raw_stages(192) >= 2 && Cfg208::raw_stages(208) >= 2,
              "raw copies run ahead of the widening");

template <class F, bool LIST, bool SPLIT>
__global__ void __launch_bounds__(F::THREADS, 1)
    gemm_ts_kernel(const __grid_constant__ TsMaps maps, const __grid_constant__ TsParams p) {
  constexpr uint32_t KBS = F::KBS, KQ = F::KQ, KR = F::KR, NA = F::NA, NQ = F::NQ, DW = F::DW, WW = F::WW, MAXG = F::MAXG;
  constexpr uint32_t RAW_STAGE = F::RAW_STAGE, DT = DW * 32;
  constexpr uint32_t WG = WW / 4;    // widening groups of four warps (one per TMEM lane quarter)
  constexpr uint32_t SPQ = KQ / KBS;  // widened stages per query stage
  constexpr uint32_t KBR = KR / KB;   // k-blocks of a raw stage
  constexpr uint32_t CPS = CP / KBS, LPS = LP / KBS, LOFF = Sched<KBS>::LOFF;
  constexpr uint32_t LEAD = Sched<KBS>::LEAD < NA ? Sched<KBS>::LEAD : NA;
  static_assert(LEAD <= NQ * SPQ && LOFF < LPS && LOFF % CPS >= LEAD && CPS - LOFF % CPS >= LEAD, "drains apart");
  extern __shared__ uint8_t smem_raw[];
  __shared__ uint32_t s_tmem;
  __shared__ uint32_t s_abort;
  const uint32_t tn = p.tn, q_half = tn * 128, q_blk = 2 * q_half, q_stage = KQ / 2 * q_blk;
  uint32_t my_items = 1, n_ct = p.n_col_tiles;
  if (LIST) {
    n_ct = *p.n_col_list;
    const uint32_t n_items = n_ct * p.n_row_tiles * p.n_pass;
    my_items = n_items > blockIdx.x ? (n_items - blockIdx.x + gridDim.x - 1) / gridDim.x : 0;
    if (my_items == 0) return;  // uniform for the CTA, before any barrier or allocation
  }
  uint32_t rank = 0, n_rank = 1;
  if (SPLIT) {
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(n_rank));
  }

  // Item i of this CTA: pass, first query column and database row, columns of the tile. Tiles walk
  // bands of up to kBand column tiles, all row tiles of a band before the next: the tiles in flight at
  // once cover about 19 row tiles x 8 column tiles, so that database tiles are read by a band's CTAs
  // together and the band's query tiles stay in L2 while the rows stream past.
  constexpr uint32_t kBand = 8;
  auto coords = [&](uint32_t i, uint32_t& q0, uint32_t& d0, uint32_t& ps, uint32_t& nw) {
    const uint32_t n_rt = p.n_row_tiles;
    uint32_t lin = SPLIT ? blockIdx.x / n_rank : blockIdx.x + i * gridDim.x;
    ps = 0;
    if (p.n_pass > 1) {
      if (p.pass_inner) {
        ps = lin % p.n_pass;
        lin /= p.n_pass;
      } else {
        ps = lin / (n_ct * n_rt);
        lin -= ps * n_ct * n_rt;
      }
    }
    const uint32_t band = lin / (kBand * n_rt), c0 = band * kBand;
    const uint32_t width = n_ct - c0 < kBand ? n_ct - c0 : kBand;
    const uint32_t in_band = lin - band * kBand * n_rt;
    const uint32_t ct = c0 + in_band % width;
    if (LIST) {
      q0 = p.col_tiles[ct] * tn;
      nw = tn;
    } else {
      // the 16-column units of n_cols dealt out evenly: no tile computes more than its share of padding
      const uint32_t units = (p.n_cols + 15) / 16, base = units / n_ct, rem = units % n_ct;
      q0 = 16 * (ct * base + (ct < rem ? ct : rem));
      nw = 16 * (base + (ct < rem ? 1 : 0));
    }
    d0 = (in_band / width) * TM;
  };

  // this CTA's k-blocks of every item: all, or its share of K (a list's passes have equal K)
  uint32_t kb0 = 0, nkb, segs;
  {
    uint32_t q0, d0, ps, nw;
    coords(0, q0, d0, ps, nw);
    segs = p.pass[ps].segs;
    const uint32_t units = segs * p.kb_seg / KB_UNIT;
    if (SPLIT) kb0 = units * rank / n_rank * KB_UNIT;
    nkb = (SPLIT ? units * (rank + 1) / n_rank : units) * KB_UNIT - kb0;
  }
  const uint32_t nst = nkb / KBS;
  // Two segments are taken in turn, 128 elements each: the parties that share a component then read
  // the same part of it at about the same time, from L2.
  auto k_of = [&](uint32_t kb, uint32_t& seg) {
    const uint32_t u = kb / KB_UNIT;
    seg = segs == 2 ? u & 1u : 0u;
    return static_cast<int32_t>(((segs == 2 ? u >> 1 : u) * KB_UNIT + kb % KB_UNIT) * KB);
  };

  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t qring = smem_addr(smem), rring = qring + NQ * q_stage, bars = rring + p.nr * RAW_STAGE;
  const uint32_t q_full = bars, q_empty = q_full + 8 * NQ, a_full = q_empty + 8 * NQ,
                 a_empty = a_full + 8 * NA, r_full = a_empty + 8 * NA, r_empty = r_full + 8 * MAX_NR,
                 c_full = r_empty + 8 * MAX_NR, c_empty = c_full + 8, l_full = c_full + 16, l_empty = c_full + 24,
                 done_bar = c_full + 32, epi_done = c_full + 40;
  volatile uint32_t* abort = &s_abort;
  const uint32_t warp = __shfl_sync(0xFFFFFFFFu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (uint32_t s = 0; s < NQ; ++s) {
      mbar_init(q_full + 8 * s, 1);
      mbar_init(q_empty + 8 * s, 1);
    }
    for (uint32_t s = 0; s < NA; ++s) {
      mbar_init(a_full + 8 * s, WW + 1);
      mbar_init(a_empty + 8 * s, 1);
    }
    for (uint32_t s = 0; s < MAX_NR; ++s) {
      mbar_init(r_full + 8 * s, 1);
      mbar_init(r_empty + 8 * s, WW);
    }
    mbar_init(c_full, 1);
    mbar_init(c_empty, DW);
    mbar_init(l_full, 1);
    mbar_init(l_empty, DW);
    mbar_init(done_bar, 1);
    mbar_init(epi_done, DW);
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
  const uint32_t tmem = s_tmem;
  // PAIR: accumulator pair b at 2 tn b, its full and empty barriers in c_full, c_empty (b = 0) and l_full, l_empty
  const uint32_t tL = tmem, tC = tmem + tn, tA = tmem + (F::PAIR ? 4 : 2) * tn;
  // a wait by the whole warp, which stays converged
  auto all_wait = [&](uint32_t bar, uint32_t par) {
    return __all_sync(0xFFFFFFFFu, mbar_wait(bar, par, p.status, abort)) != 0;
  };

  // Adds the zero shares r_i = F(seed_own) - F(seed_prev) (App. C) of 8 rows of a column, one Philox
  // block per seed, and writes their z.
  auto put_z = [&](const TsPass& P, uint32_t col, uint32_t r0, const uint4& sum) {
    if (col >= p.n_cols || r0 >= p.x_rows) return;
    const uint32_t req = p.col_tags[2 * col], tag = p.col_tags[2 * col + 1];
    const uint32_t grp = static_cast<uint32_t>((p.row0 + r0) >> 3), ctr3 = (IPC_D_ZA << 24) | P.vec;
    const uint4 fo = philox(grp, tag, req, ctr3, P.seed_own);
    const uint4 fq = philox(grp, tag, req, ctr3, P.seed_prev);
    auto add = [](uint32_t a, uint32_t o, uint32_t f) { return add16x2(a, sub16x2(o, f)); };
    const uint4 v = make_uint4(add(sum.x, fo.x, fq.x), add(sum.y, fo.y, fq.y), add(sum.z, fo.z, fq.z),
                               add(sum.w, fo.w, fq.w));
    uint16_t* dst = P.z + static_cast<uint64_t>(col) * p.ldz + r0;
    if (r0 + 8 <= p.x_rows) {
      __stcs(reinterpret_cast<uint4*>(dst), v);  // streamed: z is read by a later kernel, not from L2
    } else {
      const uint32_t w[4] = {v.x, v.y, v.z, v.w};
      for (uint32_t e = 0; e < p.x_rows - r0; ++e) dst[e] = static_cast<uint16_t>(w[e >> 1] >> (16 * (e & 1)));
    }
  };

  if (warp == 0) {
    // ---------------------------- query copies -----------------------------
    uint32_t issued = 0;
    bool ok = true;
    for (uint32_t i = 0; i < my_items && ok; ++i) {
      uint32_t q0, d0, ps, nw;
      coords(i, q0, d0, ps, nw);
      if (i > 0 && !all_wait(epi_done, (i - 1) & 1u)) break;
      const CUtensorMap *mlo = &maps.q[ps][0], *mhi = &maps.q[ps][1];
      for (uint32_t kb = kb0; kb < kb0 + nkb; kb += KQ) {
        const uint32_t qs = stage_of<NQ>(issued);
        if (!(ok = all_wait(q_empty + 8 * qs, phase_of<NQ>(issued) ^ 1u))) break;
        const uint32_t full = q_full + 8 * qs, base = qring + qs * q_stage;
        if (elect_one()) {
          mbar_expect_tx(full, q_stage);
#pragma unroll
          for (uint32_t j = 0; j < KQ / 2; ++j) {
            uint32_t seg;
            const int32_t k = k_of(kb + 2 * j, seg), kx = k + static_cast<int32_t>(seg * p.kb_seg * KB);
            tma_load(base + j * q_blk, mlo, kx, static_cast<int32_t>(q0), full);
            tma_load(base + j * q_blk + q_half, mhi, kx, static_cast<int32_t>(q0), full);
          }
        }
        __syncwarp();
        ++issued;
      }
    }
    if (*abort) {
      // copies that may still be in flight land before the CTA leaves (bounded, no abort)
      for (uint32_t G = issued > NQ ? issued - NQ : 0; G < issued; ++G)
        mbar_wait(q_full + 8 * stage_of<NQ>(G), phase_of<NQ>(G), p.status, nullptr);
    }
  } else if (warp == 1) {
    // -------------------------------- MMA issuer --------------------------------
    // kind::f16: D f32 (bits 4-5 = 1), A and B f16, K-major, N >> 3 at bits 17-22, M >> 4 at bits 24-28
    uint32_t idesc = 0;
    uint32_t c_per = 0, l_per = 0;
    // one barrier tells of both operands of stage G
    auto wait_stage = [&](uint32_t G) { return all_wait(a_full + 8 * stage_of<NA>(G), phase_of<NA>(G)); };
    // C products of stage s; `frees`: its L products are issued already
    auto issue_c = [&](uint32_t s, uint32_t G, bool frees) {
      const uint32_t qs = stage_of<NQ>(G / SPQ), as = stage_of<NA>(G), t0 = G % SPQ * (2 * KBS);
      const uint32_t qb = qring + qs * q_stage, ab = tA + as * (KBS * A_COLS);
      if (elect_one()) {
        bool acc = s % CPS != 0;
#pragma unroll
        for (uint32_t t = 0; t < 2 * KBS; ++t) {  // 16 elements of K each
          const uint32_t b = qb + ((t0 + t) >> 2) * q_blk + ((t0 + t) & 3u) * 32u, a = ab + (t >> 1) * A_COLS + (t & 1u) * 8u;
          umma_ts(tC, a, sdesc128(b + q_half), idesc, acc);  // lo * hi'
          umma_ts(tC, a + 16, sdesc128(b), idesc, true);     // hi * lo'
          acc = true;
        }
        if ((s + 1) % CPS == 0 || s + 1 == nst) umma_commit(c_full);
        if (frees) {
          if (G % SPQ == SPQ - 1) umma_commit(q_empty + 8 * qs);
          umma_commit(a_empty + 8 * as);
        }
      }
      __syncwarp();
    };
    auto issue_l = [&](uint32_t s, uint32_t G, bool frees) {
      const uint32_t qs = stage_of<NQ>(G / SPQ), as = stage_of<NA>(G), t0 = G % SPQ * (2 * KBS);
      const uint32_t qb = qring + qs * q_stage, ab = tA + as * (KBS * A_COLS);
      if (elect_one()) {
        bool acc = !(s == 0 || s % LPS == LOFF);
#pragma unroll
        for (uint32_t t = 0; t < 2 * KBS; ++t) {
          const uint32_t b = qb + ((t0 + t) >> 2) * q_blk + ((t0 + t) & 3u) * 32u, a = ab + (t >> 1) * A_COLS + (t & 1u) * 8u;
          umma_ts(tL, a, sdesc128(b), idesc, acc);  // lo * lo'
          acc = true;
        }
        if (frees) {
          if (G % SPQ == SPQ - 1) umma_commit(q_empty + 8 * qs);
          umma_commit(a_empty + 8 * as);
        }
        if ((s + 1) % LPS == LOFF || s + 1 == nst) umma_commit(l_full);
      }
      __syncwarp();
    };
    bool ok = true;
    for (uint32_t i = 0; i < my_items && ok; ++i) {
      uint32_t q0, d0, ps, nw;
      coords(i, q0, d0, ps, nw);
      idesc = (1u << 4) | ((nw >> 3) << 17) | (static_cast<uint32_t>(TM >> 4) << 24);
      bool seen = false;
      if constexpr (F::PAIR) {
        const uint32_t idesc1 = (1u << 4) | ((tn >> 3) << 17) | (static_cast<uint32_t>(TM >> 4) << 24);
        const uint32_t idesc2 = (1u << 4) | ((tn >> 2) << 17) | (static_cast<uint32_t>(TM >> 4) << 24);
        for (uint32_t s = 0; s < nst; ++s) {
          const bool opens = s % CPS == 0;
          if (opens) {
            if (!(ok = all_wait(c_per & 1u ? l_empty : c_empty, ((c_per >> 1) & 1u) ^ 1u))) break;
            ++c_per;
          }
          const uint32_t G = i * nst + s, qs = stage_of<NQ>(G / SPQ), as = stage_of<NA>(G);
          const uint32_t full = c_per & 1u ? c_full : l_full, d = tmem + ((c_per - 1) & 1u) * 2 * tn;
          if (!seen && !(ok = wait_stage(G))) break;
          fence_after();
          const bool next = s + 1 < nst && mbar_try(a_full + 8 * stage_of<NA>(G + 1), phase_of<NA>(G + 1));
          const uint32_t qb = qring + qs * q_stage, ab = tA + as * (KBS * A_COLS), t0 = G % SPQ * (2 * KBS);
          if (elect_one()) {
#pragma unroll
            for (uint32_t t = 0; t < 2 * KBS; ++t) {
              const uint32_t b = qb + ((t0 + t) >> 2) * q_blk + ((t0 + t) & 3u) * 32u, a = ab + (t >> 1) * A_COLS + (t & 1u) * 8u;
              umma_ts(d, a, sdesc128(b), idesc2, !(opens && t == 0));  // lo * [lo' | hi']
              umma_ts(d + tn, a + 16, sdesc128(b), idesc1, true);      // hi * lo'
            }
            if (G % SPQ == SPQ - 1) umma_commit(q_empty + 8 * qs);
            umma_commit(a_empty + 8 * as);
            if ((s + 1) % CPS == 0 || s + 1 == nst) umma_commit(full);
          }
          __syncwarp();
          seen = __all_sync(0xFFFFFFFFu, next) != 0;
        }
      }
      for (uint32_t s = F::PAIR ? nst : 0; s < nst && ok;) {
        const bool c_opens = s % CPS == 0, l_opens = s == 0 || s % LPS == LOFF;
        const uint32_t lead = nst - s < LEAD ? nst - s : LEAD, G = i * nst + s;
        if (c_opens && !l_opens) {
          // the L products of the next stages run while C is drained
          for (uint32_t j = 0; j < lead && ok; ++j) {
            if (!(ok = wait_stage(G + j))) break;
            fence_after();
            issue_l(s + j, G + j, false);
          }
          if (!ok || !(ok = all_wait(c_empty, (c_per++ & 1u) ^ 1u))) break;
          fence_after();
          for (uint32_t j = 0; j < lead; ++j) issue_c(s + j, G + j, true);
          s += lead;
        } else if (l_opens) {
          // the C products of the next stages run while L is drained (at s = 0 both begin an item)
          if (c_opens) {
            if (!(ok = all_wait(c_empty, (c_per++ & 1u) ^ 1u))) break;
          }
          for (uint32_t j = 0; j < lead && ok; ++j) {
            if (!(ok = wait_stage(G + j))) break;
            fence_after();
            issue_c(s + j, G + j, false);
          }
          if (!ok || !(ok = all_wait(l_empty, (l_per++ & 1u) ^ 1u))) break;
          fence_after();
          for (uint32_t j = 0; j < lead; ++j) issue_l(s + j, G + j, true);
          s += lead;
        } else {
          // the look at the next stage's barrier is under way while this stage's MMAs are issued
          if (!seen && !(ok = wait_stage(G))) break;
          fence_after();
          const bool next = KBS > 1 && s + 1 < nst && mbar_try(a_full + 8 * stage_of<NA>(G + 1), phase_of<NA>(G + 1));
          issue_c(s, G, false);
          issue_l(s, G, true);
          seen = __all_sync(0xFFFFFFFFu, next) != 0;
          ++s;
          continue;
        }
        seen = false;
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
    bool ok = true;
    for (uint32_t i = 0; i < my_items && ok; ++i) {
      uint32_t q0, d0, ps, nw;
      coords(i, q0, d0, ps, nw);
      const TsPass& P = p.pass[ps];
      for (uint32_t kb = kb0; kb < kb0 + nkb; kb += KBR) {
        if (!(ok = all_wait(r_empty + 8 * r.s, r.ph ^ 1u))) break;
        uint32_t seg;
        const int32_t kx = k_of(kb, seg);
        const uint32_t xi = seg ? P.x1 : P.x0, full = r_full + 8 * r.s, base = rring + r.s * RAW_STAGE;
        if (elect_one()) {
          mbar_expect_tx(full, RAW_STAGE);
          tma_load(base, &maps.x[xi][0], kx, static_cast<int32_t>(d0), full);
          tma_load(base + RAW_STAGE / 2, &maps.x[xi][1], kx, static_cast<int32_t>(d0), full);
        }
        __syncwarp();
        ++issued;
        r.next(p.nr);
      }
    }
    if (*abort) {
      for (uint32_t G = issued > p.nr ? issued - p.nr : 0; G < issued; ++G)
        mbar_wait(r_full + 8 * (G % p.nr), (G / p.nr) & 1u, p.status, nullptr);
    }
  } else if (warp == 3) {
    // a stage's full barrier also counts the arrival of its query tiles, so that the MMA warp, whose
    // waits cost it issue time, has one barrier to look at; a_empty keeps this warp in the right turn
    const uint32_t total = my_items * nst;
    for (uint32_t G = 0; G < total; ++G) {
      if (G % SPQ == 0 && !all_wait(q_full + 8 * stage_of<NQ>(G / SPQ), phase_of<NQ>(G / SPQ))) break;
      if (!all_wait(a_empty + 8 * stage_of<NA>(G), phase_of<NA>(G) ^ 1u)) break;
      if (lane == 0) mbar_arrive(a_full + 8 * stage_of<NA>(G));
    }
  } else if (warp >= ISSUE_WARPS + DW) {
    // -------------------------------- widening ----------------------------------
    const uint32_t g = (warp - ISSUE_WARPS - DW) >> 2, row = 32 * (warp & 3u) + lane;
    const uint32_t lane_base = (32u * (warp & 3u)) << 16;
    Ring r;
    const uint32_t total = my_items * nst;
    bool ok = true;
    for (uint32_t G = 0; G < total && ok; ++G) {
      const uint32_t as = stage_of<NA>(G), aph = phase_of<NA>(G);
      const uint32_t dst = tA + lane_base + as * (KBS * A_COLS);
#pragma unroll
      for (uint32_t jj = 0; jj < KBS / WG; ++jj) {
        // k-block jb of the stage, kr of its raw stage: 32 bytes of this row of each plane, chunks
        // 2 kr and 2 kr + 1 of the swizzled row
        const uint32_t jb = jj * WG + g, kr = (G * KBS + jb) % KBR;
        if (kr == g && !(ok = all_wait(r_full + 8 * r.s, r.ph))) break;
        const uint32_t src = rring + r.s * RAW_STAGE + row * KR, x = KR == 64 ? (row >> 1) & 3u : row & 7u;
        const uint32_t o0 = ((2 * kr) ^ x) * 16, o1 = ((2 * kr + 1) ^ x) * 16;
        const uint4 l0 = lds128(src + o0), l1 = lds128(src + o1);
        const uint4 h0 = lds128(src + RAW_STAGE / 2 + o0), h1 = lds128(src + RAW_STAGE / 2 + o1);
        uint32_t w[32];
        auto put = [&](int at, uint4 v) {
          uint4 c0, c1;
          widen16(v, c0, c1);
          w[at] = c0.x, w[at + 1] = c0.y, w[at + 2] = c0.z, w[at + 3] = c0.w;
          w[at + 4] = c1.x, w[at + 5] = c1.y, w[at + 6] = c1.z, w[at + 7] = c1.w;
        };
        put(0, l0);
        put(8, l1);
        put(16, h0);
        put(24, h1);
        if (kr + WG >= KBR) {  // this group's last k-block of the raw stage: its bytes are in registers
          __syncwarp();
          if (lane == 0) mbar_arrive(r_empty + 8 * r.s);
          r.next(p.nr);
        }
        if (jj == 0) {
          if (!(ok = all_wait(a_empty + 8 * as, aph ^ 1u))) break;
          fence_after();
        }
        tmem_st32(dst + jb * A_COLS, w);
      }
      if (!ok) break;
      tmem_wait_st();
      fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(a_full + 8 * as);
    }
  } else if (warp >= ISSUE_WARPS) {
    // ----------------------------------- drain ----------------------------------
    const uint32_t dw = warp - ISSUE_WARPS, h = dw >> 2;
    const uint32_t lane_base = (32u * (warp & 3u)) << 16;
    uint32_t c_per = 0, l_per = 0;
    bool ok = true;
    for (uint32_t i = 0; i < my_items && ok; ++i) {
      uint32_t q0, d0, ps, nw;
      coords(i, q0, d0, ps, nw);
      const uint32_t span = ((nw / 16 + DW / 4 - 1) / (DW / 4)) * 16;  // columns per drain warp of a quarter
      const uint32_t col0 = h * span, ng = col0 < nw ? ((nw - col0 < span ? nw - col0 : span) / 16) : 0;
      // z2[k]: the running sums (mod 2^16) of columns 2k and 2k + 1 of this thread's span
      uint32_t z2[8 * MAXG];
#pragma unroll
      for (int k = 0; k < 8 * MAXG; ++k) z2[k] = 0;
      auto drain = [&](uint32_t full, uint32_t par, uint32_t taddr, uint32_t empty, bool is_c) {
        if (!all_wait(full, par)) return false;
        fence_after();
#pragma unroll
        for (uint32_t gr = 0; gr < MAXG; ++gr) {
          if (gr < ng) {
            uint32_t v[16];
            tmem_ld16(taddr + lane_base + col0 + 16 * gr, v);
            tmem_wait_ld();
            if (gr == ng - 1) {  // the last of this warp's columns is in registers
              fence_before();
              __syncwarp();
              if (lane == 0) mbar_arrive(empty);
            }
#pragma unroll
            for (int k = 0; k < 8; ++k)
              z2[8 * gr + k] = add16x2(z2[8 * gr + k], is_c ? low16x2<256>(v[2 * k], v[2 * k + 1])
                                                             : low16x2<1>(v[2 * k], v[2 * k + 1]));
          }
        }
        if (ng == 0 && lane == 0) mbar_arrive(empty);
        return true;
      };
      if constexpr (F::PAIR) {
        for (uint32_t s = 0; s < nst; s += CPS, ++c_per) {
          const uint32_t b = c_per & 1u, d = tmem + lane_base + b * 2 * tn + col0;
          if (!(ok = all_wait(b ? l_full : c_full, (c_per >> 1) & 1u))) break;
          fence_after();
#pragma unroll
          for (uint32_t gr = 0; gr < MAXG; ++gr) {
            if (gr < ng) {
              uint32_t u[16], v[16];
              tmem_ld16(d + 16 * gr, u);
              tmem_ld16(d + tn + 16 * gr, v);
              tmem_wait_ld();
              if (gr == ng - 1) {  // the last of this warp's columns is in registers
                fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(b ? l_empty : c_empty);
              }
#pragma unroll
              for (int k = 0; k < 8; ++k)
                z2[8 * gr + k] = add16x2(z2[8 * gr + k], add16x2(low16x2<1>(u[2 * k], u[2 * k + 1]),
                                                                 low16x2<256>(v[2 * k], v[2 * k + 1])));
            }
          }
          if (ng == 0 && lane == 0) mbar_arrive(b ? l_empty : c_empty);
        }
      }
      for (uint32_t s = F::PAIR ? nst + 1 : 1; s <= nst && ok; ++s) {
        if (s % CPS == 0 || s == nst) ok = drain(c_full, c_per++ & 1u, tC, c_empty, true);
        if (ok && (s % LPS == LOFF || s == nst)) ok = drain(l_full, l_per++ & 1u, tL, l_empty, false);
      }
      // ---- epilogue ----
      if (named_sync_or(1, DT, *abort != 0)) break;
      uint16_t* zs = reinterpret_cast<uint16_t*>(smem);  // [tn][TM]
      const uint32_t row = 32 * (warp & 3u) + lane;
#pragma unroll
      for (uint32_t k = 0; k < 8 * MAXG; ++k)
        if (k < 8 * ng) {
          zs[(col0 + 2 * k) * TM + row] = static_cast<uint16_t>(z2[k]);
          zs[(col0 + 2 * k + 1) * TM + row] = static_cast<uint16_t>(z2[k] >> 16);
        }
      if (SPLIT) break;  // the partial sums are joined below
      named_sync(1, DT);
      for (uint32_t it = threadIdx.x - ISSUE_WARPS * 32; it < nw * (TM / 8); it += DT)
        put_z(p.pass[ps], q0 + it / (TM / 8), d0 + 8 * (it % (TM / 8)), *reinterpret_cast<const uint4*>(zs + it * 8));
      fence_proxy_async();  // the next item's query copies overwrite zs through the async proxy
      __syncwarp();
      if (lane == 0) mbar_arrive(epi_done);
    }
  }
  if (SPLIT) {
    // every thread of every CTA passes both cluster barriers, also after a failed wait
    __syncwarp();
    cluster_sync();
    if (warp >= ISSUE_WARPS && warp < ISSUE_WARPS + DW) {
      bool bad = false;
      for (uint32_t r = 0; r < n_rank; ++r) bad = bad || ld_cluster32(mapa(smem_addr(&s_abort), r)) != 0;
      if (!bad) {
        uint32_t q0, d0, ps, nw;
        coords(0, q0, d0, ps, nw);
        for (uint32_t it = rank * DT + threadIdx.x - ISSUE_WARPS * 32; it < nw * (TM / 8); it += n_rank * DT) {
          uint4 v = make_uint4(0, 0, 0, 0);
          for (uint32_t r = 0; r < n_rank; ++r) {
            const uint4 o = ld_cluster128(mapa(qring + it * 16, r));
            v = make_uint4(add16x2(v.x, o.x), add16x2(v.y, o.y), add16x2(v.z, o.z), add16x2(v.w, o.w));
          }
          put_z(p.pass[ps], q0 + it / (TM / 8), d0 + 8 * (it % (TM / 8)), v);
        }
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


// Loads every form of the kernel, so that a first call of any shape readies all of them: later calls may
// be captured into graphs.
template <class F>
cudaError_t ready() {
  cudaError_t e = cudaSuccess;
  auto set = [&](const void* k) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_MAX);
  };
  set(reinterpret_cast<const void*>(&gemm_ts_kernel<F, false, false>));
  set(reinterpret_cast<const void*>(&gemm_ts_kernel<F, false, true>));
  if constexpr (F::LISTED) set(reinterpret_cast<const void*>(&gemm_ts_kernel<F, true, false>));
  return e;
}

// CTAs that run at once in clusters of k (one a SM; clusters do not reach every SM), by device.
constexpr uint32_t MAX_SPLIT = 8;
uint32_t g_at_once[64][MAX_SPLIT + 1];

cudaError_t clusters_at_once(uint32_t k) {
  int dev = 0, n = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || dev < 0 || dev >= 64) return e;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(k);
  cfg.blockDim = dim3(Cfg208::THREADS);
  cfg.dynamicSmemBytes = SMEM_MAX;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = k;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  e = cudaOccupancyMaxActiveClusters(&n, gemm_ts_kernel<Cfg208, false, true>, &cfg);
  g_at_once[dev][k] = e == cudaSuccess ? static_cast<uint32_t>(n) * k : 0;
  return e;
}

template <class F>
int launch_ts(const TsMaps& m, TsParams& p, uint32_t ctas, uint32_t split, cudaStream_t stream) {
  p.nr = F::raw_stages(p.tn);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(ctas);
  cfg.blockDim = dim3(F::THREADS);
  cfg.dynamicSmemBytes = F::smem(p.tn, p.nr);
  cfg.stream = stream;
  cudaLaunchAttribute at[1];
  if (split > 1) {
    at[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
    at[cfg.numAttrs].val.clusterDim.x = split;
    at[cfg.numAttrs].val.clusterDim.y = at[cfg.numAttrs].val.clusterDim.z = 1;
    ++cfg.numAttrs;
  }
  cfg.attrs = at;
  auto* kernel = split > 1 ? gemm_ts_kernel<F, false, true> : gemm_ts_kernel<F, false, false>;
  if constexpr (F::LISTED) {
    if (p.col_tiles) kernel = gemm_ts_kernel<F, true, false>;
  } else if (p.col_tiles) {
    set_error("tcgen05 ring GEMM: no form for listed tiles of this width");
    return IPC_EINVAL;
  }
  IPC_CUDA_TRY(cudaLaunchKernelEx(&cfg, kernel, m, p));
  return IPC_OK;
}

uint32_t cdiv(uint32_t a, uint32_t b) { return (a + b - 1) / b; }

// Column tiles per row tile and the parts of K (a cluster's CTAs): the pair with the shortest estimate
//     rounds of the chip x (k-blocks of a CTA x (250 + 2.45 tile columns) + a tile's start and end)
// in units of 0.55 ns. The cost of a k-block is a line through launches of whole rounds (181 ns at 32 columns,
// 212 at 64, 315 at 128, 358 at 160, 415 at 208). A few rounds count whole; over many, other launches and
// drifting tiles fill the last one.
// At 1,000 rows x 4 columns splitting K by 8 gives 0.023 ms against 0.15 ms unsplit, at 1,000 x 279 0.042
// against 0.085 ms with a guess of nine SMs in ten for clusters; 9,973 x 217 takes two tiles of 112 by 2
// (0.31 ms; unsplit 0.40), 40,000 x 279 two tiles of 144 (0.67 ms; three of 96: 0.73).
double pick_shape(uint32_t n_cols, uint32_t row_tiles, uint32_t n_pass, uint32_t kb_total, uint32_t sms, uint32_t& n_ct,
                  uint32_t& split) {
  int dev = 0;
  const uint32_t* at_once = cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < 64 ? g_at_once[dev] : nullptr;
  const uint32_t units = cdiv(n_cols, 16), least = cdiv(units, MAX_TN / 16);
  double best = 1e300;
  for (uint32_t t = least; t <= least + 2 && t <= units; ++t) {
    const double kb_cycles = 250 + 2.45 * 16 * cdiv(units, t), ctas = static_cast<double>(n_pass) * t * row_tiles;
    for (uint32_t s = 1; s <= MAX_SPLIT && s <= kb_total / KB_UNIT; ++s) {
      if (s > 1 && (!at_once || at_once[s] == 0)) continue;
      const double rounds = ctas * s / (s == 1 ? sms : at_once[s]);
      const double cost = (rounds < 4 ? std::ceil(rounds) : rounds + 0.5) * (kb_cycles * kb_total / s + (s == 1 ? 10000 : 14000));
      if (cost < best * 0.999) {
        best = cost;
        n_ct = t;
        split = s;
      }
    }
  }
  return best;
}

// The estimate of the form with both operands in shared memory, whose tiles are 256 columns wide and take 1,030
// of these units a k-block (572 ns): less than two tiles of 128 (1,127). So it pays from 241 to 256 columns,
// and around 500 where it saves a round. A request of 248 columns, sustained: 65,536 rows of Galois-ring shares
// 5.64 ms with tiles of 128 and 5.42 ms so, replicated 10.63 and 10.34 ms; 8,000 x 496 Galois 1.41 and 1.36 ms.
// 4 % must be gained to leave the estimates' errors behind.
double ss_cost(uint32_t n_cols, uint32_t row_tiles, uint32_t n_pass, uint32_t kb_total, uint32_t sms) {
  const double rounds = static_cast<double>(n_pass) * cdiv(n_cols, 256) * row_tiles / sms;
  return (rounds < 8 ? std::ceil(rounds) : rounds + 0.5) * (1030.0 * kb_total + 10000) / 0.96;
}

int ring_gemm_ts_group(uint32_t n_pass, const RingGemm* g, size_t x_rows, uint32_t n_cols, uint32_t n_pad, uint32_t l,
                 const uint32_t* col_tags, size_t ldz, uint64_t row0, uint32_t list_cols, const uint32_t* col_tiles,
                 const uint32_t* n_col_list, cudaStream_t stream) {
  uint32_t kb_most = 0;
  bool equal = true;
  for (uint32_t i = 0; i < n_pass; ++i) {
    equal = equal && g[i].segments == g[0].segments;
    if (g[i].segments != 1 && g[i].segments != 2) {
      set_error("tcgen05 ring GEMM: one or two K segments");
      return IPC_EINVAL;
    }
    if (g[i].segments * l % 256 != 0) {
      set_error("tcgen05 ring GEMM: K must be a multiple of 256");
      return IPC_EINVAL;
    }
    if (col_tiles && g[i].segments != g[0].segments) {
      set_error("tcgen05 ring GEMM: the passes over a list of column tiles have equal K");
      return IPC_EINVAL;
    }
    kb_most = std::max(kb_most, g[i].segments * l / KB);
  }
  if (const int rc = ring_gemm_ts_ready()) return rc;
  TsParams p{};
  TsMaps m;
  const uint32_t sms = static_cast<uint32_t>(sm_count_current());
  uint32_t split = 1;
  p.n_row_tiles = cdiv(static_cast<uint32_t>(x_rows), TM);
  if (col_tiles) {
    // 256 columns: their own kernel, as two tiles of 128 they cost 10 % more
    if (list_cols == 256)
      return ring_gemm_ss(n_pass, g, x_rows, n_cols, n_pad, l, col_tags, ldz, row0, col_tiles, n_col_list, stream);
    p.tn = list_cols;
  } else {
    p.n_col_tiles = 1;
    const double cost = pick_shape(n_cols, p.n_row_tiles, n_pass, kb_most, sms, p.n_col_tiles, split);
    if (equal && ss_cost(n_cols, p.n_row_tiles, n_pass, kb_most, sms) < cost)
      return ring_gemm_ss(n_pass, g, x_rows, n_cols, n_pad, l, col_tags, ldz, row0, nullptr, nullptr, stream);
    p.tn = 16 * cdiv(cdiv(n_cols, 16), p.n_col_tiles);
  }
  const uint32_t raw_cols = p.tn <= 64    ? Cfg64::KR
                            : p.tn <= 96  ? Cfg96::KR
                            : p.tn <= 128 ? Cfg128::KR
                            : p.tn <= 160 ? Cfg160::KR
                            : p.tn <= 192 ? Cfg192::KR
                                          : Cfg208::KR;
  int rc;
  uint32_t nx = 0;
  const int8_t* seen[RING_GEMM_PASSES][2];
  auto x_map = [&](const int8_t* lo, const int8_t* hi, uint32_t& at) {
    for (at = 0; at < nx; ++at)
      if (seen[at][0] == lo && seen[at][1] == hi) return static_cast<int>(IPC_OK);
    if (nx == RING_GEMM_PASSES) {
      set_error("tcgen05 ring GEMM: too many database planes in one launch");
      return static_cast<int>(IPC_EINVAL);
    }
    seen[nx][0] = lo;
    seen[nx][1] = hi;
    ++nx;
    if (int e = make_map_raw(&m.x[at][0], lo, l, x_rows, raw_cols, TM)) return e;
    return make_map_raw(&m.x[at][1], hi, l, x_rows, raw_cols, TM);
  };
  bool two = true;
  for (uint32_t i = 0; i < n_pass; ++i) {
    TsPass& P = p.pass[i];
    P.z = g[i].z;
    P.seed_own = g[i].seed_own;
    P.seed_prev = g[i].seed_prev;
    P.vec = g[i].vec;
    P.segs = g[i].segments;
    two = two && P.segs == 2;
    if ((rc = x_map(g[i].x_lo[0], g[i].x_hi[0], P.x0))) return rc;
    P.x1 = P.x0;
    if (P.segs == 2 && (rc = x_map(g[i].x_lo[1], g[i].x_hi[1], P.x1))) return rc;
    const uint64_t K = static_cast<uint64_t>(P.segs) * l;
    if ((rc = make_map_f16k64(&m.q[i][0], g[i].b_lo, K, n_pad, p.tn)) ||
        (rc = make_map_f16k64(&m.q[i][1], g[i].b_hi, K, n_pad, p.tn)))
      return rc;
  }
  p.kb_seg = l / KB;
  p.n_cols = n_cols;
  p.x_rows = static_cast<uint32_t>(x_rows);
  p.n_pass = n_pass;
  // Side by side the passes of a row tile share its components in L2; that pays where the database's
  // bytes bound the launch. Wider tiles are bound by the MMAs and go pass by pass.
  p.pass_inner = two && p.tn <= 64;
  p.col_tiles = col_tiles;
  p.n_col_list = n_col_list;
  p.col_tags = col_tags;
  p.ldz = ldz;
  p.row0 = row0;
  p.status = status_ptr();
  const uint32_t ctas = col_tiles ? sms : n_pass * p.n_col_tiles * p.n_row_tiles * split;
  if (p.tn <= 64) return launch_ts<Cfg64>(m, p, ctas, split, stream);
  if (p.tn <= 96) return launch_ts<Cfg96>(m, p, ctas, split, stream);
  if (p.tn <= 128) return launch_ts<Cfg128>(m, p, ctas, split, stream);
  if (p.tn <= 160) return launch_ts<Cfg160>(m, p, ctas, split, stream);
  if (p.tn <= 192) return launch_ts<Cfg192>(m, p, ctas, split, stream);
  return launch_ts<Cfg208>(m, p, ctas, split, stream);
}

}  // namespace

int ring_gemm_ts_ready() {
  if (const int rc = ring_gemm_ss_ready()) return rc;
  static PerDevice attr;
  IPC_CUDA_TRY(attr.run([] {
    cudaError_t e = ready<Cfg64>();
    if (e == cudaSuccess) e = ready<Cfg96>();
    if (e == cudaSuccess) e = ready<Cfg128>();
    if (e == cudaSuccess) e = ready<Cfg160>();
    if (e == cudaSuccess) e = ready<Cfg192>();
    if (e == cudaSuccess) e = ready<Cfg208>();
    for (uint32_t k = 2; k <= MAX_SPLIT && e == cudaSuccess; ++k) e = clusters_at_once(k);
    return e;
  }));
  return IPC_OK;
}

// The passes of a launch follow one another, so that two passes' query operands are in use at once. As long
// as those fit the L2 together all passes run in one launch, which fills the chip best (three passes of
// 51 MB, 30,000 x 496: 4.1 ms against 4.6 ms as three launches). Else tiles drift apart over the rounds of a
// launch (waves of one tile per SM) until every one reads its query tiles from DRAM, while every launch
// leaves its last round partly empty: up to 32 rounds all six passes go together, or else a vector's three,
// or else each alone. Replicated sharing, a request sustained, in ms (six launches / two / one):
//     16,384 rows x   992 columns ( 4.2 rounds a pass)  9.97 /  9.43 /  9.46
//     16,384      x 1,984         ( 8.4)               19.22 / 18.96 / 19.98
//     40,000      x   992         (10.3)               23.15 / 22.69 / 23.92
//     65,536      x   992         (17)                 36.58 / 38.45 / 40.13
// Galois-ring shares (K half as long) differ by less than 1 % from 8 rounds a pass on, and 2,000 x 1,984
// takes 1.80 / 1.57 / 1.48 ms.
uint32_t ring_gemm_ts_passes(uint32_t n_pass, uint32_t segments, size_t x_rows, uint32_t cols, uint32_t l) {
  const uint64_t bytes = 4ull * segments * l * cols;
  const double rounds = static_cast<double>(cdiv(cols, MAX_TN)) * cdiv(static_cast<uint32_t>(x_rows), TM) / sm_count_current();
  if (2 * bytes <= L2_QUERY_BYTES || n_pass * rounds <= LAUNCH_ROUNDS) return n_pass;
  return 3 * rounds <= LAUNCH_ROUNDS ? 3 : 1;
}

int ring_gemm_ts_by(uint32_t per, uint32_t n_pass, const RingGemm* g, size_t x_rows, uint32_t n_cols, uint32_t n_pad,
                    uint32_t l, const uint32_t* col_tags, size_t ldz, uint64_t row0, uint32_t list_cols,
                    const uint32_t* col_tiles, const uint32_t* n_col_list, cudaStream_t stream) {
  if (n_pass == 0 || n_pass > RING_GEMM_PASSES || per == 0) {
    set_error("tcgen05 ring GEMM: one to six passes");
    return IPC_EINVAL;
  }
  for (uint32_t first = 0; first < n_pass; first += per) {
    const int rc = ring_gemm_ts_group(std::min(per, n_pass - first), g + first, x_rows, n_cols, n_pad, l, col_tags, ldz,
                                      row0, list_cols, col_tiles, n_col_list, stream);
    if (rc) return rc;
  }
  return IPC_OK;
}

int ring_gemm_ts(uint32_t n_pass, const RingGemm* g, size_t x_rows, uint32_t n_cols, uint32_t n_pad, uint32_t l,
                 const uint32_t* col_tags, size_t ldz, uint64_t row0, cudaStream_t stream) {
  uint32_t segments = 0;
  for (uint32_t i = 0; i < n_pass && i < RING_GEMM_PASSES; ++i) segments = std::max(segments, g[i].segments);
  return ring_gemm_ts_by(ring_gemm_ts_passes(n_pass, segments, x_rows, n_cols, l), n_pass, g, x_rows, n_cols, n_pad, l,
                         col_tags, ldz, row0, 0, nullptr, nullptr, stream);
}

int ring_gemm_tc_variant(uint32_t tile_cols, uint32_t segments, const int8_t* const x_lo[2],
                         const int8_t* const x_hi[2], size_t x_rows, const uint16_t* b_lo, const uint16_t* b_hi,
                         uint32_t n_cols, uint32_t n_pad, uint32_t l, const uint32_t* col_tags, uint64_t seed_own,
                         uint64_t seed_prev, uint32_t vec, uint16_t* z, size_t ldz, uint64_t row0,
                         const uint32_t* col_tiles, const uint32_t* n_col_list, cudaStream_t stream) {
  const RingGemm g{{x_lo[0], x_lo[1]}, {x_hi[0], x_hi[1]}, segments, b_lo, b_hi, seed_own, seed_prev, vec, z};
  return ring_gemm_ts_by(1, 1, &g, x_rows, n_cols, n_pad, l, col_tags, ldz, row0, tile_cols, col_tiles, n_col_list, stream);
}

int ring_gemm_tc(const int8_t* const x_lo[2], const int8_t* const x_hi[2], size_t x_rows, const uint16_t* b_lo,
                 const uint16_t* b_hi, uint32_t n_cols, uint32_t n_pad, uint32_t l, const uint32_t* col_tags,
                 uint64_t seed_own, uint64_t seed_prev, uint32_t vec, uint16_t* z, size_t ldz, uint64_t row0,
                 cudaStream_t stream) {
  return ring_gemm_tc_variant(256, 2, x_lo, x_hi, x_rows, b_lo, b_hi, n_cols, n_pad, l, col_tags, seed_own,
                              seed_prev, vec, z, ldz, row0, nullptr, nullptr, stream);
}

}  // namespace ipc
