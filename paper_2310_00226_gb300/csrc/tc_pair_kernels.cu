// tcgen05 split-precision mode product with one MMA per pair of SMs
// (cta_group::2), for one problem or for a group of independent problems in
// one persistent launch.  The arithmetic is that of tc_kernels.cu (the same
// MMAs in the same K order: results are bit-identical); see the comment at
// the kernel for the division of work between the two CTAs of a pair.
#include "tc_common.cuh"

#include <algorithm>

namespace sem3d {

namespace {

using namespace tcx;

// ---------------------------------------------------------------- CTA-pair kernel
//
// The same mode product with one MMA per pair of SMs (tcgen05 cta_group::2):
// a cluster of 2 CTAs owns a 256-row x bn-output tile (bn <= 256, see
// tile_outputs).  CTA r of the pair stages its own 128 rows of A and rows
// [r bn/2, (r + 1) bn/2) of the W tile, so a stage holds 32 KB per CTA instead
// of 48 KB (6 stages fit where 4 did) and each SM loads half of W without
// multicast.  The leader CTA
// (rank 0) issues M = 256 MMAs that read A and W from both CTAs' shared memory
// at the same offsets and accumulate rows 128 r .. 128 r + 127 of the tile in
// CTA r's tensor memory.  Both CTAs' TMA loads complete on the leader's "full"
// barrier (armed by the leader with the pair's bytes); MMA completion arrives
// on the "empty" and "tfull" barriers of both CTAs (commit multicast); the
// epilogue warps of both CTAs release a TMEM buffer on the leader's "tempty"
// barrier.  Pairs of clusters pack every SM (clusters of 4 leave SMs idle on
// GPCs whose SM count is not a multiple of 4).
//
// Epilogue warps: as the one-CTA kernel, but 16 for the division pass, whose
// epilogue (a reciprocal and a shuffle per value) otherwise outlasts the
// loads: n = 511 in parity order 207 -> 186 us.  Their staging buffers take
// the place of one operand stage.  16 warps are worth nothing to the other
// split outputs.
__host__ __device__ constexpr int pair_epi(int mode) { return mode == OUT_DIV_SPLIT ? 16 : epi_warps(mode); }
__host__ __device__ constexpr int pair_threads(int mode) { return 64 + 32 * pair_epi(mode); }
__host__ __device__ constexpr int pair_stages(int mode) { return mode == OUT_DIV_SPLIT ? 5 : 6; }
constexpr int P_B_TILE_BYTES = (BN / 2) * BK * 2;  // 8 KB: this CTA's half of W
constexpr int P_STAGE_BYTES = 2 * A_TILE_BYTES + 2 * P_B_TILE_BYTES;  // 32 KB
__host__ __device__ constexpr int pair_smem_bytes(int pass, int mode) {
  return pair_stages(mode) * P_STAGE_BYTES + 1024 /*align*/ + 256 /*barriers*/ +
         (pass == 0 ? pair_epi(mode) * XSTAGE_BYTES : 0);
}

__device__ __forceinline__ void mma_bf16_pair(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                              uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}\n"
      ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// One pair tile handed to the kernel body: the problem's arguments and tensor
// maps, and the tile's (pair of flattened M tiles, N tile) within that problem.
struct PairTile {
  const TcArgs* a;
  const CUtensorMap *Ah, *Al, *Bh, *Bl;
  int mp, nt;
};

// Tile source of a launch for one problem: the kernel's own parameters.
struct OneProblem {
  const CUtensorMap *Ah, *Al, *Bh, *Bl;
  const TcArgs* a;
  int total;
  __device__ __forceinline__ void at(int pt, int& /*cursor*/, PairTile& t) const {
    t.a = a; t.Ah = Ah; t.Al = Al; t.Bh = Bh; t.Bl = Bl;
    t.mp = pt / a->n_tiles;
    t.nt = pt - t.mp * a->n_tiles;
  }
};

// Tile source of a grouped launch: problem q owns pair tiles [tile0, tile0 +
// its count) of the launch (prefix offsets, ascending).  Each thread walks its
// tiles in ascending order, so its cursor into the table only moves forward.
struct ProblemGroup {
  const TcGroupEntry* tab;
  int count, total;
  __device__ __forceinline__ void at(int pt, int& cursor, PairTile& t) const {
    while (cursor + 1 < count && tab[cursor + 1].tile0 <= pt) ++cursor;
    const TcGroupEntry& e = tab[cursor];
    t.a = &e.a; t.Ah = &e.A_hi; t.Al = &e.A_lo; t.Bh = &e.B_hi; t.Bl = &e.B_lo;
    const int local = pt - e.tile0;
    t.mp = local / e.a.n_tiles;
    t.nt = local - t.mp * e.a.n_tiles;
  }
};

template <int PASS, int MODE, int NP, class Src>
__device__ __forceinline__ void pair_body(const Src& src, int* err, int stall) {
  constexpr int P_STAGES = pair_stages(MODE);
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + P_STAGES * P_STAGE_BYTES);
  // bars: full[P_STAGES], empty[P_STAGES], tfull[2], tempty[2], drain[1]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * P_STAGES + 5);
  const uint32_t bar0 = smem_u32(bars);
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (P_STAGES + s); };
  auto tfull_bar = [&](int b) { return bar0 + 8u * (2 * P_STAGES + b); };
  auto tempty_bar = [&](int b) { return bar0 + 8u * (2 * P_STAGES + 2 + b); };
  const uint32_t drain_bar = bar0 + 8u * (2 * P_STAGES + 4);
  constexpr uint16_t kPair = 3;  // both CTAs of the pair

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr bool a_mn = (PASS != 0);
  const int rank = (int)cluster_ctarank();
  const int pid = blockIdx.x >> 1, npairs = gridDim.x >> 1;

  pdl_trigger();
  if (threadIdx.x == 0) {
    for (int s = 0; s < P_STAGES; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(tfull_bar(b), 1); mbar_init(tempty_bar(b), 2 * pair_epi(MODE)); }
    mbar_init(drain_bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();  // both CTAs' barriers are initialised before any cross-CTA signal
  pdl_wait();
  tc_fence_after();
  const uint32_t tmem_base = *reinterpret_cast<volatile uint32_t*>(tmem_slot);

  // Pair tile pt -> (problem, M pair mp, N tile nt); this CTA's flattened M
  // tile is 2 mp + rank, i.e. M tile mt of batch b (past the problem's last
  // one, TMA reads zeros and nothing is stored).
  const int total_pt = src.total;
  PairTile t;
  if (warp == 0 && lane == 0) {
    // ------------------------------------------------ TMA producer (each CTA)
    const uint32_t full_leader0 = mapa_shared(full_bar(0), 0);
    int it = 0, cursor = 0;
    bool ok = true;
    for (int pt = pid; pt < total_pt && ok && !stall; pt += npairs) {
      src.at(pt, cursor, t);
      const int mf = 2 * t.mp + rank;
      const int b = PASS == 1 ? mf / t.a->m_tiles : 0;
      const int m0 = (mf - b * t.a->m_tiles) * BM, bn = t.a->bn, n0 = t.nt * bn + rank * (bn / 2);
      const int k_blocks = t.a->k_blocks;
      for (int kb = 0; kb < k_blocks; ++kb, ++it) {
        const int s = it % P_STAGES;
        const uint32_t par = ((it / P_STAGES) & 1) ^ 1;
        if (!mbar_wait(empty_bar(s), par, err, KERN_SPLIT_PAIR | WAIT_PRODUCER)) { ok = false; break; }
        const uint32_t st = smem_u32(smem + s * P_STAGE_BYTES);
        const uint32_t a_hi = st, a_lo = st + A_TILE_BYTES;
        const uint32_t b_hi = st + 2 * A_TILE_BYTES, b_lo = b_hi + P_B_TILE_BYTES;
        const uint32_t fb = full_leader0 + 8u * s;  // the leader's full barrier of stage s
        if (rank == 0)
          mbar_arrive_expect_tx(full_bar(s), (NP == 3 ? 4 : 2) * A_TILE_BYTES + (NP == 3 ? 2 : 1) * bn * (BK * 2));
        const int k0 = kb * BK;
        if (PASS == 0) {
          tma_load_2d_pair(a_hi, t.Ah, fb, k0, m0);
          if (NP == 3) tma_load_2d_pair(a_lo, t.Al, fb, k0, m0);
        } else if (PASS == 1) {
          tma_load_3d_pair(a_hi, t.Ah, fb, m0, k0, b);
          tma_load_3d_pair(a_hi + A_TILE_BYTES / 2, t.Ah, fb, m0 + 64, k0, b);
          if (NP == 3) {
            tma_load_3d_pair(a_lo, t.Al, fb, m0, k0, b);
            tma_load_3d_pair(a_lo + A_TILE_BYTES / 2, t.Al, fb, m0 + 64, k0, b);
          }
        } else {
          tma_load_2d_pair(a_hi, t.Ah, fb, m0, k0);
          tma_load_2d_pair(a_hi + A_TILE_BYTES / 2, t.Ah, fb, m0 + 64, k0);
          if (NP == 3) {
            tma_load_2d_pair(a_lo, t.Al, fb, m0, k0);
            tma_load_2d_pair(a_lo + A_TILE_BYTES / 2, t.Al, fb, m0 + 64, k0);
          }
        }
        tma_load_2d_pair(b_hi, t.Bh, fb, k0, n0);
        if (NP == 3) tma_load_2d_pair(b_lo, t.Bl, fb, k0, n0);
      }
    }
    // Drain: the last fill of each stage has landed (leader: its full barrier
    // counts both CTAs' bytes) and the MMAs reading it have completed (both:
    // the commit arrived on this CTA's empty barrier), so no copy, MMA read or
    // remote arrival targets this CTA after it exits.
    const int armed = it;
    for (int q = (armed > P_STAGES ? armed - P_STAGES : 0); q < armed; ++q) {
      if (rank == 0) mbar_wait(full_bar(q % P_STAGES), (q / P_STAGES) & 1, nullptr);
      mbar_wait(empty_bar(q % P_STAGES), (q / P_STAGES) & 1, nullptr);
    }
  } else if (warp == 1 && lane == 0 && rank == 0) {
    // ------------------------------------------------ MMA issuer (leader CTA only)
    constexpr uint32_t a_lbo = a_mn ? 4096u : 16u, a_sbo = a_mn ? 1024u : 512u, a_kstep = a_mn ? 2048u : 32u;
    constexpr uint32_t a_layout = a_mn ? LAYOUT_SW128 : LAYOUT_SW64;
    int it = 0, cc = 0, cursor = 0;
    bool ok = true;
    for (int pt = pid; pt < total_pt && ok; pt += npairs, ++cc) {
      src.at(pt, cursor, t);
      const int k_blocks = t.a->k_blocks;
      const uint32_t idesc = make_idesc(2 * BM, t.a->bn, a_mn, 0);
      const int buf = cc & 1;
      if (!mbar_wait_cluster(tempty_bar(buf), ((cc >> 1) & 1) ^ 1, err, KERN_SPLIT_PAIR | WAIT_MMA_TMEM)) {
        ok = false;
        break;
      }
      tc_fence_after();
      const uint32_t tmem_d = tmem_base + (uint32_t)(buf * BN);
      for (int kb = 0; kb < k_blocks; ++kb, ++it) {
        const int s = it % P_STAGES;
        if (!mbar_wait(full_bar(s), (it / P_STAGES) & 1, err, KERN_SPLIT_PAIR | WAIT_MMA_FULL)) { ok = false; break; }
        tc_fence_after();
        const uint32_t st = smem_u32(smem + s * P_STAGE_BYTES);
        const uint32_t a_hi = st, a_lo = st + A_TILE_BYTES;
        const uint32_t b_hi = st + 2 * A_TILE_BYTES, b_lo = b_hi + P_B_TILE_BYTES;
#pragma unroll
        for (int k16 = 0; k16 < BK / 16; ++k16) {
          const uint64_t dah = smem_desc(a_hi + k16 * a_kstep, a_lbo, a_sbo, a_layout);
          const uint64_t dal = smem_desc(a_lo + k16 * a_kstep, a_lbo, a_sbo, a_layout);
          const uint64_t dbh = smem_desc(b_hi + k16 * 32u, 16u, 512u, LAYOUT_SW64);
          const uint64_t dbl = smem_desc(b_lo + k16 * 32u, 16u, 512u, LAYOUT_SW64);
          const uint32_t acc = (kb | k16) ? 1u : 0u;
          mma_bf16_pair(tmem_d, dah, dbh, idesc, acc);
          if (NP == 3) {
            mma_bf16_pair(tmem_d, dah, dbl, idesc, 1u);
            mma_bf16_pair(tmem_d, dal, dbh, idesc, 1u);
          }
        }
        mma_commit_pair_mc(empty_bar(s), kPair);  // the stage is free in both CTAs once these finish
      }
      if (!ok) break;
      mma_commit_pair_mc(tfull_bar(buf), kPair);  // accumulator ready for both CTAs' epilogues
    }
    mma_commit_pair_mc(drain_bar, 1);  // every pair MMA issued so far has completed
    mbar_wait(drain_bar, 0, nullptr);
  } else if (warp >= 2) {
    // ------------------------------------------------ epilogue (each CTA, its own 128 rows)
    const int quad = warp & 3;
    const int slice = (warp - 2) >> 2;
    uint8_t* xstage = PASS == 0 ? smem + P_STAGES * P_STAGE_BYTES + 256 + (warp - 2) * XSTAGE_BYTES : nullptr;
    constexpr int SLICES = pair_epi(MODE) / 4;  // warps per lane quadrant; they take 32-output chunks in turn
    const uint32_t tempty_leader0 = mapa_shared(tempty_bar(0), 0);
    float vmax = 0.f;
    int cc = 0, cursor = 0;
    for (int pt = pid; pt < total_pt; pt += npairs, ++cc) {
      src.at(pt, cursor, t);
      const TcArgs& a = *t.a;
      const int mf = 2 * t.mp + rank;
      const int b = PASS == 1 ? mf / a.m_tiles : 0;
      const int row = (mf - b * a.m_tiles) * BM + quad * 32 + lane;
      const bool any = mf < a.m_tiles * a.batches;
      const uint32_t lane_addr = tmem_base + ((uint32_t)(quad * 32) << 16);
      const int buf = cc & 1;
      if (!mbar_wait(tfull_bar(buf), (cc >> 1) & 1, err, KERN_SPLIT_PAIR | WAIT_EPILOGUE)) break;
      tc_fence_after();
      // this warp's chunks of the tile (warp-uniform); the accumulator goes back
      // once the last one is in registers, before it is converted and stored
      const int cols = any ? min(a.bn, a.nout - t.nt * a.bn) : 0;
      if (slice * 32 >= cols) {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_remote(tempty_leader0 + 8u * buf);
      }
#pragma unroll 1
      for (int ch = slice; ch * 32 < cols; ch += SLICES) {
        float v[32];
        tmem_ld32(lane_addr + (uint32_t)(buf * BN + ch * 32), v);
        if ((ch + SLICES) * 32 >= cols) {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_remote(tempty_leader0 + 8u * buf);
        }
        epilogue_chunk<PASS, MODE, NP, 0>(a, row, t.nt * a.bn + ch * 32, b, v, 1.f, 1.f, vmax, xstage);
      }
    }
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();  // no copy, MMA or arrival of the pair targets this CTA any more
  tc_fence_after();
  if (warp == 1) {
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS));
  }
}

template <int PASS, int MODE, int NP>
__global__ void __launch_bounds__(pair_threads(MODE), 1)
    mode_product_bf16x3_pair_kernel(const __grid_constant__ CUtensorMap tmA_hi,
                                    const __grid_constant__ CUtensorMap tmA_lo,
                                    const __grid_constant__ CUtensorMap tmB_hi,
                                    const __grid_constant__ CUtensorMap tmB_lo, const __grid_constant__ TcArgs a) {
  const OneProblem src{&tmA_hi, &tmA_lo, &tmB_hi, &tmB_lo, &a, (a.m_tiles * a.batches + 1) / 2 * a.n_tiles};
  pair_body<PASS, MODE, NP>(src, a.err, a.stall);
}

// The same pass for many problems in one persistent launch (grouped batched
// solve): pair tiles of all problems form one queue, problem q's tiles
// starting at tab[q].tile0; each problem brings its own tensor maps and
// epilogue arguments in the device table (64-byte aligned).
template <int PASS, int MODE, int NP>
__global__ void __launch_bounds__(pair_threads(MODE), 1)
    mode_product_bf16x3_pair_group_kernel(const TcGroupEntry* __restrict__ tab, int count, int total, int* err,
                                          int stall) {
  const ProblemGroup src{tab, count, total};
  pair_body<PASS, MODE, NP>(src, err, stall);
}

// One pass in parity order: its two blocks as a group of two problems, kept
// in the kernel's parameters.
struct FoldPass {
  TcGroupEntry e[2];
};

template <int PASS, int MODE>
__global__ void __launch_bounds__(pair_threads(MODE), 1)
    mode_product_fold_kernel(const __grid_constant__ FoldPass f, int total, int* err, int stall) {
  const ProblemGroup src{f.e, 2, total};
  pair_body<PASS, MODE, 3>(src, err, stall);
}

// CTA-pair launch: clusters of 2, one pair per pair of SMs, persistent over
// pair tiles.
// `resident`: the kernel's co-resident clusters of 2 CTAs, asked for once per device.
template <class Kern, class... Args>
cudaError_t launch_pairs(Kern kern, PerDevice& resident, int pass, int mode, long long work_pairs,
                         int num_sms, cudaStream_t s, const Args&... args) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.blockDim = dim3(pair_threads(mode));
  cfg.dynamicSmemBytes = pair_smem_bytes(pass, mode);
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int max_pairs = 0;
  cfg.gridDim = dim3(2 * (num_sms / 2));
  const cudaError_t e = on_device(resident, [&](int& n) {
    cudaError_t q = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, pair_smem_bytes(pass, mode));
    if (q == cudaSuccess) q = cudaOccupancyMaxActiveClusters(&n, kern, &cfg);
    return q == cudaSuccess && n < 1 ? cudaErrorInvalidConfiguration : q;
  }, &max_pairs);
  if (e != cudaSuccess) return e;
  const long long pairs = work_pairs < max_pairs ? work_pairs : max_pairs;
  cfg.gridDim = dim3((unsigned)(2 * pairs));
  cfg.stream = s;
  attr[1] = pdl_attribute();
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

template <int PASS, int MODE, int NP>
cudaError_t launch_tc_pair(const CUtensorMap& a0, const CUtensorMap& a1, const CUtensorMap& b0, const CUtensorMap& b1,
                           const TcArgs& a, long long work_pairs, int num_sms, cudaStream_t s) {
  static PerDevice resident;
  return launch_pairs(mode_product_bf16x3_pair_kernel<PASS, MODE, NP>, resident, PASS, MODE, work_pairs, num_sms, s,
                      a0, a1, b0, b1, a);
}

template <int PASS, int MODE>
cudaError_t launch_fold_pass(const FoldPass& f, int total, int* err, int stall, int num_sms, cudaStream_t s) {
  static PerDevice resident;
  return launch_pairs(mode_product_fold_kernel<PASS, MODE>, resident, PASS, MODE, total, num_sms, s, f, total, err,
                      stall);
}

template <int PASS>
cudaError_t launch_tc_pair_mode(int mode, int nprod, const CUtensorMap& a0, const CUtensorMap& a1,
                                const CUtensorMap& b0, const CUtensorMap& b1, const TcArgs& a, long long work,
                                int num_sms, cudaStream_t s) {
  if (nprod == 1) {
    switch (mode) {
      case OUT_SPLIT: return launch_tc_pair<PASS, OUT_SPLIT, 1>(a0, a1, b0, b1, a, work, num_sms, s);
      case OUT_DIV_SPLIT: return launch_tc_pair<PASS, OUT_DIV_SPLIT, 1>(a0, a1, b0, b1, a, work, num_sms, s);
      case OUT_F64: return launch_tc_pair<PASS, OUT_F64, 1>(a0, a1, b0, b1, a, work, num_sms, s);
      case OUT_F64_ACCUM: return launch_tc_pair<PASS, OUT_F64_ACCUM, 1>(a0, a1, b0, b1, a, work, num_sms, s);
      default: return cudaErrorInvalidValue;
    }
  }
  switch (mode) {
    case OUT_SPLIT: return launch_tc_pair<PASS, OUT_SPLIT, 3>(a0, a1, b0, b1, a, work, num_sms, s);
    case OUT_DIV_SPLIT: return launch_tc_pair<PASS, OUT_DIV_SPLIT, 3>(a0, a1, b0, b1, a, work, num_sms, s);
    case OUT_F64: return launch_tc_pair<PASS, OUT_F64, 3>(a0, a1, b0, b1, a, work, num_sms, s);
    case OUT_F64_ACCUM: return launch_tc_pair<PASS, OUT_F64_ACCUM, 3>(a0, a1, b0, b1, a, work, num_sms, s);
    default:
      if constexpr (PASS == 2) {
        if (mode == OUT_DF_STORE) return launch_tc_pair<PASS, OUT_DF_STORE, 3>(a0, a1, b0, b1, a, work, num_sms, s);
        if (mode == OUT_DF_ACCUM) return launch_tc_pair<PASS, OUT_DF_ACCUM, 3>(a0, a1, b0, b1, a, work, num_sms, s);
        return launch_tc_pair<PASS, OUT_DF_ACCUM_F64, 3>(a0, a1, b0, b1, a, work, num_sms, s);
      }
      return cudaErrorInvalidValue;
  }
}

// Grouped launch: the same pass of `count` problems, one persistent launch.
template <int PASS, int MODE, int NP>
cudaError_t launch_pair_group_t(const TcGroupEntry* tab, int count, int total, int* err, int stall, int num_sms,
                                cudaStream_t s) {
  static PerDevice resident;
  return launch_pairs(mode_product_bf16x3_pair_group_kernel<PASS, MODE, NP>, resident, PASS, MODE, total, num_sms, s,
                      tab, count, total, err, stall);
}

cudaError_t launch_pair_group(int axis, int mode, int nprod, const TcGroupEntry* tab, int count, int total, int* err,
                              int stall, int num_sms, cudaStream_t s) {
  // The modes a grouped solve uses: forward z, y (split), x (division); backward
  // x, y (split) and z (split, FP64 store / accumulate, double-FP32 modes).
  if (nprod == 3) {
    if (axis == 0 && mode == OUT_SPLIT) return launch_pair_group_t<0, OUT_SPLIT, 3>(tab, count, total, err, stall, num_sms, s);
    if (axis == 0 && mode == OUT_DIV_SPLIT) return launch_pair_group_t<0, OUT_DIV_SPLIT, 3>(tab, count, total, err, stall, num_sms, s);
    if (axis == 1 && mode == OUT_SPLIT) return launch_pair_group_t<1, OUT_SPLIT, 3>(tab, count, total, err, stall, num_sms, s);
    if (axis == 2 && mode == OUT_SPLIT) return launch_pair_group_t<2, OUT_SPLIT, 3>(tab, count, total, err, stall, num_sms, s);
    if (axis == 2 && mode == OUT_F32) return launch_pair_group_t<2, OUT_F32, 3>(tab, count, total, err, stall, num_sms, s);
    if (axis == 2 && mode == OUT_F64) return launch_pair_group_t<2, OUT_F64, 3>(tab, count, total, err, stall, num_sms, s);
    if (axis == 2 && mode == OUT_F64_ACCUM) return launch_pair_group_t<2, OUT_F64_ACCUM, 3>(tab, count, total, err, stall, num_sms, s);
    if (axis == 2 && mode == OUT_DF_STORE) return launch_pair_group_t<2, OUT_DF_STORE, 3>(tab, count, total, err, stall, num_sms, s);
    if (axis == 2 && mode == OUT_DF_ACCUM) return launch_pair_group_t<2, OUT_DF_ACCUM, 3>(tab, count, total, err, stall, num_sms, s);
    if (axis == 2 && mode == OUT_DF_ACCUM_F64) return launch_pair_group_t<2, OUT_DF_ACCUM_F64, 3>(tab, count, total, err, stall, num_sms, s);
  } else if (nprod == 1) {
    if (axis == 0 && mode == OUT_SPLIT) return launch_pair_group_t<0, OUT_SPLIT, 1>(tab, count, total, err, stall, num_sms, s);
    if (axis == 0 && mode == OUT_DIV_SPLIT) return launch_pair_group_t<0, OUT_DIV_SPLIT, 1>(tab, count, total, err, stall, num_sms, s);
    if (axis == 1 && mode == OUT_SPLIT) return launch_pair_group_t<1, OUT_SPLIT, 1>(tab, count, total, err, stall, num_sms, s);
    if (axis == 2 && mode == OUT_SPLIT) return launch_pair_group_t<2, OUT_SPLIT, 1>(tab, count, total, err, stall, num_sms, s);
    if (axis == 2 && mode == OUT_F64) return launch_pair_group_t<2, OUT_F64, 1>(tab, count, total, err, stall, num_sms, s);
    if (axis == 2 && mode == OUT_F64_ACCUM) return launch_pair_group_t<2, OUT_F64_ACCUM, 1>(tab, count, total, err, stall, num_sms, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

// Two entries per problem: a parity-order problem queues its two blocks.
size_t tc_group_table_bytes(int count) { return ((size_t)count * 2 * sizeof(TcGroupEntry) + 255) & ~size_t(255); }

cudaError_t launch_mode_product_bf16x3_grouped(int count, const TcGroupItem* items, int axis, int which, int epi,
                                               int nprod, int* err_flag, void* dev_table, void* host_table,
                                               size_t table_bytes, int num_sms, cudaStream_t s) {
  if (count < 1 || !items || tc_group_table_bytes(count) > table_bytes) return cudaErrorInvalidValue;
  if ((reinterpret_cast<uintptr_t>(dev_table) | reinterpret_cast<uintptr_t>(host_table)) & 63)
    return cudaErrorInvalidValue;
  TcGroupEntry* tab = static_cast<TcGroupEntry*>(host_table);
  long long total = 0;
  int mode = -1, entries = 0;
  for (int q = 0; q < count; ++q) {
    const TcGroupItem& it = items[q];
    if (it.fold && nprod != 3) return cudaErrorInvalidValue;
    for (int par = 0; par < (it.fold ? 2 : 1); ++par) {
      PassSetup ps;
      cudaError_t e = it.fold ? prepare_parity_pass(*it.fold, it.c, axis, it.ax, which, par, it.in, it.out, it.out32,
                                                    epi, err_flag, ps)
                              : prepare_pass(*it.g, axis, *it.W, which, it.in, it.out, it.out64, epi, it.lamx, it.lamy,
                                             it.lamz, err_flag, it.df, nprod, nullptr, true, ps);
      if (e != cudaSuccess) return e;
      if (mode >= 0 && ps.mode != mode) return cudaErrorInvalidValue;  // one epilogue mode per launch
      mode = ps.mode;
      TcGroupEntry& en = tab[entries++];
      en.A_hi = ps.mAh; en.A_lo = ps.mAl; en.B_hi = ps.mBh; en.B_lo = ps.mBl;
      en.a = ps.a;
      en.tile0 = (int)total;
      total += pair_tiles(ps.a);
      if (total >= (1LL << 31)) return cudaErrorInvalidValue;
    }
  }
  cudaError_t e = cudaMemcpyAsync(dev_table, host_table, (size_t)entries * sizeof(TcGroupEntry), cudaMemcpyHostToDevice, s);
  if (e != cudaSuccess) return e;
  if (total == 0) return cudaSuccess;
  return launch_pair_group(axis, mode, nprod, static_cast<const TcGroupEntry*>(dev_table), entries, (int)total, err_flag,
                           tc_take_stall(), num_sms, s);
}

cudaError_t launch_mode_product_fold(const FoldGeom& g, float c, int axis, const DevAxis* ax, int which, TcBuffers in,
                                     TcBuffers out, float* out32, int epi, int* err_flag, int num_sms, cudaStream_t s) {
  FoldPass f;
  long long total = 0;
  int mode = 0;
  for (int par = 0; par < 2; ++par) {
    PassSetup ps;
    const cudaError_t e = prepare_parity_pass(g, c, axis, ax, which, par, in, out, out32, epi, err_flag, ps);
    if (e != cudaSuccess) return e;
    TcGroupEntry& en = f.e[par];
    en.A_hi = ps.mAh; en.A_lo = ps.mAl; en.B_hi = ps.mBh; en.B_lo = ps.mBl;
    en.a = ps.a;
    en.tile0 = (int)total;
    total += pair_tiles(ps.a);
    mode = ps.mode;
  }
  if (total >= (1LL << 31)) return cudaErrorInvalidValue;
  const int stall = tc_take_stall(), t = (int)total;
  if (axis == 0 && mode == OUT_SPLIT) return launch_fold_pass<0, OUT_SPLIT>(f, t, err_flag, stall, num_sms, s);
  if (axis == 0 && mode == OUT_DIV_SPLIT) return launch_fold_pass<0, OUT_DIV_SPLIT>(f, t, err_flag, stall, num_sms, s);
  if (axis == 1 && mode == OUT_SPLIT) return launch_fold_pass<1, OUT_SPLIT>(f, t, err_flag, stall, num_sms, s);
  if (axis == 2 && mode == OUT_SPLIT) return launch_fold_pass<2, OUT_SPLIT>(f, t, err_flag, stall, num_sms, s);
  if (axis == 2 && mode == OUT_F32) return launch_fold_pass<2, OUT_F32>(f, t, err_flag, stall, num_sms, s);
  return cudaErrorInvalidValue;
}

namespace tcx {

cudaError_t launch_pair_pass(int axis, int nprod, const PassSetup& ps, long long work_pairs, int num_sms,
                             cudaStream_t s) {
  if (axis == 0) return launch_tc_pair_mode<0>(ps.mode, nprod, ps.mAh, ps.mAl, ps.mBh, ps.mBl, ps.a, work_pairs, num_sms, s);
  if (axis == 1) return launch_tc_pair_mode<1>(ps.mode, nprod, ps.mAh, ps.mAl, ps.mBh, ps.mBl, ps.a, work_pairs, num_sms, s);
  return launch_tc_pair_mode<2>(ps.mode, nprod, ps.mAh, ps.mAl, ps.mBh, ps.mBl, ps.a, work_pairs, num_sms, s);
}

}  // namespace tcx

}  // namespace sem3d
