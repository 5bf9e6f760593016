// FP32 CUDA-core mode product (the SEM3D_FP32 tier): FFMA with FP32 operands
// and accumulation, no tensor cores.  Same strided formulation as the FP64
// DMMA kernel (Section 2.4, Eq. 11-13: one Kronecker factor at a time, no
// transposes): C[row, o] = sum_t A[row, t] * W[o, t], rows enumerated by two
// loops (p < R1 stride s1, q < R2 stride s2), axis stride sm.
//
// Bound by the shared-memory reads that feed the FP32 pipe, at two blocks of
// 126 registers a thread (n = 383: pipe 53% busy, shared memory 70%; n = 767 with
// full matrices 46 of 74 TF/s).  A CTA of 256 threads computes a BM x BN
// output tile; each thread owns TM rows (in pairs of neighbours, so that a
// packed f32x2 multiply-add serves two rows; the packed form has the scalar
// one's lane rate for half the issue slots, which leaves room for the shared-
// memory reads) x TN outputs.  Lanes run along the contiguous index of the
// pass's output: along the outputs for x, along the rows for y and z.  K
// advances in chunks of 16 staged in shared memory, with one buffer (load,
// sync, compute, sync) or two (the next chunk's global loads are in flight in
// registers while the current chunk is multiplied).  Which of the
// configurations runs is decided per pass shape and form of W by measuring
// them (f32_autotune), since the best one depends on n and on the number of rows: a
// 63-wide output axis wastes half of a 128-wide tile, while large passes want
// the larger register tiles.
//
// Refined solves (two sweeps or more: errors of 1e-15 to 1e-14, as with the full
// matrices; 8 right-hand sides each at n = 63 .. 599) use the parity blocks of T^{-1} and T (Axis1D::par):
// half the multiply-adds.  Forward, half sums and differences of a line are
// formed on load; backward, the epilogue writes E + O and E - O to mirrored
// nodes.  Bare solves, one sweep and the Cahn-Hilliard step keep the full
// matrices.  Eight uneven problems (n = 63..255), 18 grouped passes: 8.2 ms
// (scalar, full matrices, lanes along the outputs in every pass) -> 4.3 ms.
#include <algorithm>
#include <map>
#include <mutex>
#include <tuple>
#include <type_traits>

#include "sem3d_internal.h"
#include "tc_ptx.cuh"

namespace sem3d {

namespace {

struct F32Pass {
  const void* in;         // float or double (first pass of a solve)
  void* out;              // float, or double for the last pass
  const float* W;         // n x n row-major, or the even block (ne x ne) and then the odd one (no x no)
  long long s1, s2, sm;
  int R1, R2, n, ne, no;
  int epi;                // EPI_STORE / EPI_DIV (x pass only) / EPI_ACCUM (double output only)
  int cfg;                // configuration index (F32Cfg below)
  int nx, ny;
  const double *lamx, *lamy, *lamz;
  double c;
};

template <int BM_, int BN_, int TM_, int TN_, int STAGES_>
struct F32Cfg {
  static constexpr int BM = BM_, BN = BN_, BK = 16, TM = TM_, TN = TN_, STAGES = STAGES_;
  static constexpr int TX = BN / TN, TY = BM / TM;  // threads along outputs / rows
  static_assert(TX * TY == 256, "256 threads");
  static_assert(TM % 4 == 0 && TN % 4 == 0, "pairs of rows and outputs in either parity");
  static constexpr int A_LD = BM + 2;  // padded rows of the staged tiles: 8-byte reads, conflict-free writes
  static constexpr int SMEM_FLOATS = STAGES * BK * (A_LD + BN + 2);
};

// How a pass uses W: the full matrix, or its parity blocks from nodes to modes
// (even modes first) or from modes to nodes.
enum : int { W_FULL = 0, W_FWD = 1, W_BWD = 2 };

// Configurations: tile shape x {two stages, one stage}.  Indexes 0..2 are the
// double-buffered ones (the grouped launch uses those).
using Cfg0 = F32Cfg<128, 128, 8, 8, 2>;
using Cfg1 = F32Cfg<128, 64, 8, 4, 2>;
using Cfg2 = F32Cfg<64, 64, 4, 4, 2>;
using Cfg3 = F32Cfg<128, 128, 8, 8, 1>;
using Cfg4 = F32Cfg<128, 64, 8, 4, 1>;
using Cfg5 = F32Cfg<64, 64, 4, 4, 1>;
constexpr int F32_NCFG = 6;
constexpr int F32_SMEM_MAX = Cfg0::SMEM_FLOATS;  // the largest

__host__ __device__ constexpr int cfg_bm(int c) { return (c % 3 == 2) ? 64 : 128; }
__host__ __device__ constexpr int cfg_bn(int c) { return (c % 3 == 0) ? 128 : 64; }

typedef unsigned long long f2;  // two FP32 numbers

__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f2 dup2(float a) {
  f2 r;
  asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(a));
  return r;
}
__device__ __forceinline__ void unpack2(f2 v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }

__device__ __forceinline__ float to_f32(float x) { return x; }
__device__ __forceinline__ float to_f32(double x) { return f64_to_f32_rn(x); }  // off the FP64 pipe

// FP32 -> FP64 off the FP64 pipe (subnormals, which f32_to_f64 flushes, by the hardware).
__device__ __forceinline__ double to_f64(float x) {
  return (__float_as_uint(x) & 0x7F800000u) ? f32_to_f64(x) : (double)x;
}

// Offset of row `row` of the pass (rows = R1 * R2 in all).
__device__ __forceinline__ long long row_offset(const F32Pass& p, long long rows, long long row) {
  if (rows <= 0xFFFFFFFFLL) {
    const unsigned int q = (unsigned int)row / (unsigned int)p.R1;
    return ((unsigned int)row - q * (unsigned int)p.R1) * p.s1 + q * p.s2;
  }
  return (row % p.R1) * p.s1 + (row / p.R1) * p.s2;
}

// One BM x BN output tile (row tile bx, output tile by) of pass p.  With parity
// blocks the tile is BN/2 outputs of either parity and a chunk 8 + 8 of K.
template <class C, typename TIN, typename TOUT, bool KCONTIG, int MODE>
__device__ __forceinline__ void f32_tile(const F32Pass& p, long long bx, int by, float* smem) {
  constexpr int NP = MODE == W_FULL ? 1 : 2;                      // parities
  constexpr int BK = C::BK / NP, BN = C::BN / NP, TN = C::TN / NP;  // of one parity
  constexpr int TG = C::TM / 2;                                   // row pairs per thread
  constexpr int W_LD = BN + 2, LA = C::BM * BK / 256, LW = NP * BN * BK / 256;
  float* As = smem;                                     // [STAGES][NP][BK][A_LD]
  float* Ws = smem + C::STAGES * C::BK * C::A_LD;       // [STAGES][NP][BK][W_LD]
  const int tid = threadIdx.x;
  const int tx = KCONTIG ? tid % C::TX : tid / C::TY, ty = KCONTIG ? tid / C::TX : tid % C::TY;
  // this thread's rows 2 ty + 2 TY g + {0, 1} and outputs (per parity)
  auto out_of = [&](int c) { return KCONTIG ? 2 * tx + 2 * C::TX * (c >> 1) + (c & 1) : tx * TN + c; };
  const long long rows = (long long)p.R1 * p.R2;
  const long long row0 = bx * C::BM;
  const int o0 = by * BN, kmax = MODE == W_FULL ? p.n : p.ne;
  const TIN* in = static_cast<const TIN*>(p.in);

  f2 acc[NP][TG][TN];
#pragma unroll
  for (int q = 0; q < NP; ++q)
#pragma unroll
    for (int g = 0; g < TG; ++g)
#pragma unroll
      for (int c = 0; c < TN; ++c) acc[q][g][c] = 0ull;

  // The rows this thread loads are the same in every K chunk: decode them once.
  const TIN* abase[LA];
#pragma unroll
  for (int it = 0; it < LA; ++it) {
    const int e = tid + it * 256;
    const long long row = row0 + (KCONTIG ? e / BK : e % C::BM);
    abase[it] = row < rows ? in + row_offset(p, rows, row) : nullptr;
  }
  // Raw loads of the next chunk: converted, and added or subtracted, when they
  // are stored, after the current chunk's multiply-adds.
  TIN ra[LA][NP];
  float rw[LW];
  auto load = [&](int t0) {
#pragma unroll
    for (int it = 0; it < LA; ++it) {
      const int e = tid + it * 256;
      const int t = t0 + (KCONTIG ? e % BK : e / C::BM);
      const bool ok = abase[it] && t < kmax;
      ra[it][0] = ok ? abase[it][(long long)t * p.sm] : TIN(0);
      if constexpr (MODE != W_FULL)  // the middle node of an odd n (t = no) has no partner
        ra[it][NP - 1] =
            ok && t < p.no ? abase[it][(long long)(MODE == W_FWD ? p.n - 1 - t : p.ne + t) * p.sm] : TIN(0);
    }
#pragma unroll
    for (int it = 0; it < LW; ++it) {
      const int e = tid + it * 256;
      const int kk = e % BK, o = o0 + (e / BK) % BN, q = NP == 1 ? 0 : e / (BK * BN);
      const int t = t0 + kk, m = MODE == W_FULL ? p.n : q == 0 ? p.ne : p.no;
      rw[it] = (o < m && t < m) ? __ldg(p.W + (q == 0 ? 0 : (long long)p.ne * p.ne) + (long long)o * m + t) : 0.f;
    }
  };
  auto store = [&](int st, int t0) {
    float* a = As + st * C::BK * C::A_LD;
    float* w = Ws + st * NP * BK * W_LD;
#pragma unroll
    for (int it = 0; it < LA; ++it) {
      const int e = tid + it * 256;
      const int kk = KCONTIG ? e % BK : e / C::BM, r = KCONTIG ? e / BK : e % C::BM;
      float u = to_f32(ra[it][0]);
      if constexpr (MODE != W_FULL) {
        float v = to_f32(ra[it][NP - 1]);
        if (sizeof(TIN) == 8) {  // a right-hand side: halved, so that no sum of a mirrored pair overflows
          u *= 0.5f;
          v *= 0.5f;
        }
        if (MODE == W_FWD) {
          const float d = t0 + kk < p.no ? u - v : 0.f;
          u = u + v;
          v = d;
        }
        a[(BK + kk) * C::A_LD + r] = v;
      }
      a[kk * C::A_LD + r] = u;
    }
#pragma unroll
    for (int it = 0; it < LW; ++it) {
      const int e = tid + it * 256;
      const int q = NP == 1 ? 0 : e / (BK * BN);
      w[(q * BK + e % BK) * W_LD + (e / BK) % BN] = rw[it];
    }
  };
  auto compute = [&](int st) {
    const float* a = As + st * C::BK * C::A_LD + 2 * ty;
    const float* w = Ws + st * NP * BK * W_LD;
#pragma unroll
    for (int kk = 0; kk < BK; ++kk)
#pragma unroll
      for (int q = 0; q < NP; ++q) {
        f2 av[TG];
        float bv[TN];
#pragma unroll
        for (int g = 0; g < TG; ++g)
          av[g] = *reinterpret_cast<const f2*>(a + (q * BK + kk) * C::A_LD + 2 * C::TY * g);
#pragma unroll
        for (int c = 0; c < TN; c += 2) {
          const float2 v = *reinterpret_cast<const float2*>(w + (q * BK + kk) * W_LD + out_of(c));
          bv[c] = v.x; bv[c + 1] = v.y;
        }
#pragma unroll
        for (int c = 0; c < TN; ++c) {
          const f2 b = dup2(bv[c]);
#pragma unroll
          for (int g = 0; g < TG; ++g) acc[q][g][c] = fma2(av[g], b, acc[q][g][c]);
        }
      }
  };

  const int nch = (kmax + BK - 1) / BK;
  load(0);
  store(0, 0);
  __syncthreads();
  for (int ch = 0; ch < nch; ++ch) {
    if (C::STAGES == 2) {
      // The other buffer was last read in the previous chunk, before the
      // barrier that ended it: it can be refilled while this one is used.
      const int cur = ch & 1;
      if (ch + 1 < nch) load((ch + 1) * BK);
      compute(cur);
      if (ch + 1 < nch) store(cur ^ 1, (ch + 1) * BK);
      __syncthreads();
    } else {
      compute(0);
      __syncthreads();
      if (ch + 1 < nch) {
        load((ch + 1) * BK);
        store(0, (ch + 1) * BK);
        __syncthreads();
      }
    }
  }
  TOUT* out = static_cast<TOUT*>(p.out);
#pragma unroll
  for (int g = 0; g < TG; ++g)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const long long row = row0 + 2 * ty + 2 * C::TY * g + h;
      if (row >= rows) continue;
      TOUT* dst = out + row_offset(p, rows, row);
      double ly = 0.0, lz = 0.0;
      if (KCONTIG && p.epi == EPI_DIV) {  // x pass: row = (j, l)
        const unsigned int l = (unsigned int)row / (unsigned int)p.ny;  // R1 = ny nz is an int
        ly = p.lamy[(unsigned int)row - l * (unsigned int)p.ny];
        lz = p.lamz[l];
      }
      // the row's values and where they go (at < 0: outside), then all reads of
      // an accumulating pass before the first write
      float v[NP][TN];
      int at[NP][TN];
#pragma unroll
      for (int c = 0; c < TN; ++c) {
        const int o = o0 + out_of(c);
#pragma unroll
        for (int q = 0; q < NP; ++q) {
          float x, y;
          unpack2(acc[q][g][c], x, y);
          v[q][c] = h ? y : x;
        }
        if constexpr (MODE == W_FULL) {
          at[0][c] = o < p.n ? o : -1;
          if (KCONTIG && p.epi == EPI_DIV && o < p.n) v[0][c] = v[0][c] / (float)(p.lamx[o] + ly + lz + p.c);
        } else {
          const bool pair = o < p.no;  // else the middle of an odd n
          at[0][c] = o < p.ne ? o : -1;
          at[NP - 1][c] = !pair ? -1 : MODE == W_FWD ? p.ne + o : p.n - 1 - o;
          if (MODE == W_BWD) {
            const float e = v[0][c], d = pair ? v[NP - 1][c] : 0.f;
            v[0][c] = e + d;
            v[NP - 1][c] = e - d;
          } else if (KCONTIG && p.epi == EPI_DIV) {
            const double d = ly + lz + p.c;
            // of halved right-hand sides
            if (o < p.ne) v[0][c] = v[0][c] / (0.5f * f64_to_f32_rn(p.lamx[o] + d));
            if (pair) v[NP - 1][c] = v[NP - 1][c] / (0.5f * f64_to_f32_rn(p.lamx[p.ne + o] + d));
          }
        }
      }
      if constexpr (sizeof(TOUT) == 8) {
        double old[NP][TN];
#pragma unroll
        for (int q = 0; q < NP; ++q)
#pragma unroll
          for (int c = 0; c < TN; ++c)
            old[q][c] = p.epi == EPI_ACCUM && at[q][c] >= 0 ? dst[(long long)at[q][c] * p.sm] : 0.0;
#pragma unroll
        for (int q = 0; q < NP; ++q)
#pragma unroll
          for (int c = 0; c < TN; ++c)
            if (at[q][c] >= 0)
              dst[(long long)at[q][c] * p.sm] = p.epi == EPI_ACCUM ? old[q][c] + to_f64(v[q][c]) : to_f64(v[q][c]);
      } else {
#pragma unroll
        for (int q = 0; q < NP; ++q)
#pragma unroll
          for (int c = 0; c < TN; ++c)
            if (at[q][c] >= 0) dst[(long long)at[q][c] * p.sm] = v[q][c];
      }
    }
}

template <int CFG>
struct CfgOf;
template <> struct CfgOf<0> { using T = Cfg0; };
template <> struct CfgOf<1> { using T = Cfg1; };
template <> struct CfgOf<2> { using T = Cfg2; };
template <> struct CfgOf<3> { using T = Cfg3; };
template <> struct CfgOf<4> { using T = Cfg4; };
template <> struct CfgOf<5> { using T = Cfg5; };

template <int CFG, typename TIN, typename TOUT, bool KCONTIG, int MODE>
__global__ void __launch_bounds__(256, 2) mode_product_f32_kernel(F32Pass p) {
  pdl_trigger();
  pdl_wait();
  __shared__ __align__(16) float smem[CfgOf<CFG>::T::SMEM_FLOATS];
  f32_tile<typename CfgOf<CFG>::T, TIN, TOUT, KCONTIG, MODE>(p, blockIdx.x, blockIdx.y, smem);
}

// Grouped launch: one pass (the same axis and operand types) of many
// independent problems in a single grid.  Block b belongs to the problem q
// with block_begin[q] <= b < block_begin[q+1]; its tiles are numbered row
// tile fastest, with that problem's own (double-buffered) configuration.
struct F32Group {
  int count;
  const F32Pass* passes;
  const long long* block_begin;  // count + 1 entries
};

template <typename TIN, typename TOUT, bool KCONTIG, int MODE>
__global__ void __launch_bounds__(256, 2) mode_product_f32_grouped_kernel(F32Group g) {
  __shared__ __align__(16) float smem[F32_SMEM_MAX];
  __shared__ int prob;
  if (threadIdx.x == 0) {
    int q = 0;
    while (q + 1 < g.count && g.block_begin[q + 1] <= (long long)blockIdx.x) ++q;
    prob = q;
  }
  __syncthreads();
  const F32Pass p = g.passes[prob];
  const long long lb = (long long)blockIdx.x - g.block_begin[prob];
  const long long rows = (long long)p.R1 * p.R2;
  const int cfg = p.cfg % 3;
  const long long rt = (rows + cfg_bm(cfg) - 1) / cfg_bm(cfg);
  if (cfg == 0) f32_tile<Cfg0, TIN, TOUT, KCONTIG, MODE>(p, lb % rt, (int)(lb / rt), smem);
  else if (cfg == 1) f32_tile<Cfg1, TIN, TOUT, KCONTIG, MODE>(p, lb % rt, (int)(lb / rt), smem);
  else f32_tile<Cfg2, TIN, TOUT, KCONTIG, MODE>(p, lb % rt, (int)(lb / rt), smem);
}

// Outputs of the tile grid: the parity blocks' tiles take half of BN of either.
long long out_tiles(const F32Pass& p, int cfg, int mode) {
  const int bn = mode == W_FULL ? cfg_bn(cfg) : cfg_bn(cfg) / 2, m = mode == W_FULL ? p.n : p.ne;
  return (m + bn - 1) / bn;
}

template <int CFG, typename TIN, typename TOUT, int MODE>
cudaError_t launch_cfg(const F32Pass& p, bool kcontig, cudaStream_t s) {
  const long long rows = (long long)p.R1 * p.R2;
  const long long bx = (rows + cfg_bm(CFG) - 1) / cfg_bm(CFG);
  if (bx >= (1LL << 31)) return cudaErrorInvalidValue;
  dim3 grid((unsigned)bx, (unsigned)out_tiles(p, CFG, MODE));
  if constexpr (sizeof(TIN) + sizeof(TOUT) == 8) {
    if (kcontig) return launch_pdl(mode_product_f32_kernel<CFG, TIN, TOUT, true, MODE>, grid, dim3(256), 0, s, p);
  }
  if (kcontig) return cudaErrorInvalidValue;  // FP64 operands: the z passes' only
  return launch_pdl(mode_product_f32_kernel<CFG, TIN, TOUT, false, MODE>, grid, dim3(256), 0, s, p);
}

template <typename TIN, typename TOUT, int MODE>
cudaError_t launch_f32(const F32Pass& p, bool kcontig, cudaStream_t s) {
  switch (p.cfg) {
    case 0: return launch_cfg<0, TIN, TOUT, MODE>(p, kcontig, s);
    case 1: return launch_cfg<1, TIN, TOUT, MODE>(p, kcontig, s);
    case 2: return launch_cfg<2, TIN, TOUT, MODE>(p, kcontig, s);
    case 3: return launch_cfg<3, TIN, TOUT, MODE>(p, kcontig, s);
    case 4: return launch_cfg<4, TIN, TOUT, MODE>(p, kcontig, s);
    default: return launch_cfg<5, TIN, TOUT, MODE>(p, kcontig, s);
  }
}

template <typename TIN, typename TOUT, int MODE>
cudaError_t launch_f32_grouped(const F32Group& grp, long long blocks, bool kcontig, cudaStream_t s) {
  if constexpr (sizeof(TIN) + sizeof(TOUT) == 8) {
    if (kcontig) {
      mode_product_f32_grouped_kernel<TIN, TOUT, true, MODE><<<(unsigned)blocks, 256, 0, s>>>(grp);
      return cudaGetLastError();
    }
  }
  if (kcontig) return cudaErrorInvalidValue;  // FP64 operands: the z passes' only
  mode_product_f32_grouped_kernel<TIN, TOUT, false, MODE><<<(unsigned)blocks, 256, 0, s>>>(grp);
  return cudaGetLastError();
}

// FP64 input belongs to the first (forward) pass of a solve, FP64 output to
// the last (backward) one; `run` is called with the operand types and mode.
template <class Run>
cudaError_t dispatch_f32(bool in_f64, bool out_f64, int mode, Run run) {
  if (mode == W_FWD) {
    if (out_f64) return cudaErrorInvalidValue;
    return in_f64 ? run(double(), float(), std::integral_constant<int, W_FWD>()) : run(float(), float(), std::integral_constant<int, W_FWD>());
  }
  if (mode == W_BWD) {
    if (in_f64) return cudaErrorInvalidValue;
    return out_f64 ? run(float(), double(), std::integral_constant<int, W_BWD>()) : run(float(), float(), std::integral_constant<int, W_BWD>());
  }
  if (in_f64 && out_f64) return cudaErrorInvalidValue;
  if (in_f64) return run(double(), float(), std::integral_constant<int, W_FULL>());
  if (out_f64) return run(float(), double(), std::integral_constant<int, W_FULL>());
  return run(float(), float(), std::integral_constant<int, W_FULL>());
}

// ---------------------------------------------------------------- autotuner
// Pass shape and form (full matrices or parity blocks) -> configuration, filled
// by f32_autotune from measurements.  Each form is measured for itself: the
// tiles of the blocks hold half the outputs of either parity, and a choice
// made for one costs the other up to 45% (63x255x127 bare: 244 us with the
// blocks' choice, 169 with its own; 127^3 194 and 145).  Rows are capped at the
// tuning size: beyond a few waves of tiles the ranking no longer changes with
// the row count.
constexpr long long TUNE_ROWS = 65536;
using TuneKey = std::tuple<int, int, long long, int>;  // (K contiguous, n, min(rows, TUNE_ROWS), parity)
std::mutex g_tune_mu;
std::map<TuneKey, int> g_tune;

TuneKey tune_key(bool kcontig, int n, long long rows, bool parity) {
  return TuneKey{kcontig ? 1 : 0, n, rows < TUNE_ROWS ? rows : TUNE_ROWS, parity ? 1 : 0};
}

// A form that has not been measured takes the other's choice.
int tuned_cfg(bool kcontig, int n, long long rows, bool parity) {
  std::lock_guard<std::mutex> lk(g_tune_mu);
  auto it = g_tune.find(tune_key(kcontig, n, rows, parity));
  if (it == g_tune.end()) it = g_tune.find(tune_key(kcontig, n, rows, !parity));
  return it == g_tune.end() ? 0 : it->second;
}

// The pass along `axis` with T^{-1} (which = 0) or T; `parity`: by its blocks.
F32Pass make_pass(const Geom& g, int axis, const DevAxis* ax, int which, bool parity, const void* in, void* out, int epi,
                  bool* kcontig) {
  F32Pass p{};
  p.in = in;
  p.out = out;
  p.W = parity ? ax[axis].Wpf[which] : ax[axis].Wf[which];
  p.n = ax[axis].n;
  p.ne = ax[axis].ne;
  p.no = ax[axis].no;
  p.epi = epi;
  p.nx = g.nx;
  p.ny = g.ny;
  p.lamx = parity ? ax[0].lam_par : ax[0].lam;
  p.lamy = parity ? ax[1].lam_par : ax[1].lam;
  p.lamz = parity ? ax[2].lam_par : ax[2].lam;
  p.c = g.c;
  const long long nxy = (long long)g.nx * g.ny;
  *kcontig = false;
  if (axis == 0) {
    p.R1 = g.ny * g.nz; p.R2 = 1; p.s1 = g.nx; p.s2 = 0; p.sm = 1; *kcontig = true;
  } else if (axis == 1) {
    p.R1 = g.nx; p.R2 = g.nz; p.s1 = 1; p.s2 = nxy; p.sm = g.nx;
  } else {
    p.R1 = (int)nxy; p.R2 = 1; p.s1 = 1; p.s2 = 0; p.sm = nxy;
  }
  p.cfg = tuned_cfg(*kcontig, p.n, (long long)p.R1 * p.R2, parity);
  return p;
}

// EPI_DIV is the x pass's (rows are (j, l) lines), EPI_ACCUM the FP64 output's.
bool epi_ok(int axis, int epi, bool out_f64) {
  return (epi != EPI_DIV || axis == 0) && (epi != EPI_ACCUM || out_f64);
}

}  // namespace

cudaError_t f32_autotune(const Geom& g, const DevAxis* ax, bool parity) {
  // The three pass shapes of this grid, each timed on a synthetic forward pass
  // of the form asked for with the same K extent, output length and access
  // pattern and min(rows, TUNE_ROWS) rows, on scratch buffers of this device.
  struct Shape { bool kcontig; int n; long long rows; };
  const Shape shapes[3] = {{true, g.nx, (long long)g.ny * g.nz},
                           {false, g.ny, (long long)g.nx * g.nz},
                           {false, g.nz, (long long)g.nx * g.ny}};
  std::vector<int> todo;
  {
    std::lock_guard<std::mutex> lk(g_tune_mu);
    for (int a = 0; a < 3; ++a)
      if (!g_tune.count(tune_key(shapes[a].kcontig, shapes[a].n, shapes[a].rows, parity))) todo.push_back(a);
  }
  if (todo.empty()) return cudaSuccess;
  size_t need = 0;
  for (int a : todo) {
    const long long r = shapes[a].rows < TUNE_ROWS ? shapes[a].rows : TUNE_ROWS;
    need = std::max(need, (size_t)r * shapes[a].n * sizeof(float));
  }
  float *in = nullptr, *out = nullptr;
  cudaStream_t s = nullptr;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  cudaError_t err = cudaMalloc(&in, need);
  if (err == cudaSuccess) err = cudaMalloc(&out, need);
  if (err == cudaSuccess) err = cudaMemset(in, 0, need);
  if (err == cudaSuccess) err = cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
  if (err == cudaSuccess) err = cudaEventCreate(&e0);
  if (err == cudaSuccess) err = cudaEventCreate(&e1);
  for (size_t q = 0; q < todo.size() && err == cudaSuccess; ++q) {
    const Shape& sh = shapes[todo[q]];
    const long long r = sh.rows < TUNE_ROWS ? sh.rows : TUNE_ROWS;
    F32Pass p{};
    p.in = in; p.out = out; p.W = parity ? ax[todo[q]].Wpf[0] : ax[todo[q]].Wf[0]; p.epi = EPI_STORE; p.n = sh.n;
    p.ne = ax[todo[q]].ne; p.no = ax[todo[q]].no;
    p.R1 = (int)r; p.R2 = 1; p.s2 = 0;
    if (sh.kcontig) { p.s1 = sh.n; p.sm = 1; }
    else { p.s1 = 1; p.sm = r; }
    int best = 0;
    float best_ms = 0.f;
    auto pass = [&] {
      return parity ? launch_f32<float, float, W_FWD>(p, sh.kcontig, s) : launch_f32<float, float, W_FULL>(p, sh.kcontig, s);
    };
    for (int c = 0; c < F32_NCFG && err == cudaSuccess; ++c) {
      p.cfg = c;
      err = pass();  // warm-up
      if (err == cudaSuccess) err = cudaEventRecord(e0, s);
      for (int rep = 0; rep < 3 && err == cudaSuccess; ++rep) err = pass();
      if (err == cudaSuccess) err = cudaEventRecord(e1, s);
      if (err == cudaSuccess) err = cudaEventSynchronize(e1);
      float ms = 0.f;
      if (err == cudaSuccess) err = cudaEventElapsedTime(&ms, e0, e1);
      if (err == cudaSuccess && (c == 0 || ms < best_ms)) { best = c; best_ms = ms; }
    }
    if (err == cudaSuccess) {
      std::lock_guard<std::mutex> lk(g_tune_mu);
      g_tune[tune_key(sh.kcontig, sh.n, sh.rows, parity)] = best;
    }
  }
  if (e0) cudaEventDestroy(e0);
  if (e1) cudaEventDestroy(e1);
  if (s) cudaStreamDestroy(s);
  if (in) cudaFree(in);
  if (out) cudaFree(out);
  return err;
}

void f32_set_config(int axis, const Geom& g, int cfg) {
  const bool kc = axis == 0;
  const int n = axis == 0 ? g.nx : (axis == 1 ? g.ny : g.nz);
  const long long rows = axis == 0 ? (long long)g.ny * g.nz : (axis == 1 ? (long long)g.nx * g.nz : (long long)g.nx * g.ny);
  std::lock_guard<std::mutex> lk(g_tune_mu);
  for (bool parity : {false, true}) g_tune[tune_key(kc, n, rows, parity)] = cfg;
}

int f32_config(int axis, const Geom& g, bool parity) {
  if (axis == 0) return tuned_cfg(true, g.nx, (long long)g.ny * g.nz, parity);
  if (axis == 1) return tuned_cfg(false, g.ny, (long long)g.nx * g.nz, parity);
  return tuned_cfg(false, g.nz, (long long)g.nx * g.ny, parity);
}

cudaError_t launch_mode_product_f32_grouped(int count, const Geom* geoms, int axis, const DevAxis* const* ax, int which,
                                            bool parity, const void* const* in, bool in_f64, void* const* out,
                                            bool out_f64, int epi, void* dev_table, size_t table_bytes,
                                            void* host_table, cudaStream_t s) {
  // Table layout: count passes, then count + 1 block offsets.
  const size_t need = (size_t)count * sizeof(F32Pass) + (size_t)(count + 1) * sizeof(long long);
  if (count < 1 || need > table_bytes || !epi_ok(axis, epi, out_f64)) return cudaErrorInvalidValue;
  const int mode = !parity ? W_FULL : which == 0 ? W_FWD : W_BWD;
  F32Pass* passes = static_cast<F32Pass*>(host_table);
  long long* begin = reinterpret_cast<long long*>(static_cast<char*>(host_table) + (size_t)count * sizeof(F32Pass));
  bool kcontig = false;
  begin[0] = 0;
  for (int q = 0; q < count; ++q) {
    passes[q] = make_pass(geoms[q], axis, ax[q], which, parity, in[q], out[q], epi, &kcontig);
    passes[q].cfg %= 3;  // the grouped kernel holds the double-buffered shapes
    const long long rows = (long long)passes[q].R1 * passes[q].R2;
    const int c = passes[q].cfg;
    begin[q + 1] = begin[q] + ((rows + cfg_bm(c) - 1) / cfg_bm(c)) * out_tiles(passes[q], c, mode);
  }
  if (begin[count] >= (1LL << 31)) return cudaErrorInvalidValue;
  cudaError_t e = cudaMemcpyAsync(dev_table, host_table, need, cudaMemcpyHostToDevice, s);
  if (e != cudaSuccess) return e;
  F32Group grp{count, static_cast<const F32Pass*>(dev_table),
               reinterpret_cast<const long long*>(static_cast<const char*>(dev_table) + (size_t)count * sizeof(F32Pass))};
  return dispatch_f32(in_f64, out_f64, mode, [&](auto ti, auto to, auto m) {
    return launch_f32_grouped<decltype(ti), decltype(to), decltype(m)::value>(grp, begin[count], kcontig, s);
  });
}

cudaError_t launch_mode_product_f32(const Geom& g, int axis, const DevAxis* ax, int which, bool parity, const void* in,
                                    bool in_f64, void* out, bool out_f64, int epi, cudaStream_t s) {
  if (!epi_ok(axis, epi, out_f64)) return cudaErrorInvalidValue;
  bool kcontig = false;
  const F32Pass p = make_pass(g, axis, ax, which, parity, in, out, epi, &kcontig);
  return dispatch_f32(in_f64, out_f64, !parity ? W_FULL : which == 0 ? W_FWD : W_BWD, [&](auto ti, auto to, auto m) {
    return launch_f32<decltype(ti), decltype(to), decltype(m)::value>(p, kcontig, s);
  });
}

}  // namespace sem3d
