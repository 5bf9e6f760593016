// FP64 kernels: the plain-FP64 mode product (mma.sync DMMA), the banded
// FP64 operator / residual, and the FP64 -> split-bf16 conversion.
#include "sem3d_internal.h"

namespace sem3d {

namespace {

// ------------------------------------------------------------------ DMMA GEMM
//
// A mode product along one axis is a GEMM C[row, o] = sum_t A[row, t] W[o, t]
// where `row` enumerates the grid lines along that axis.  Rows are described
// by two loops (p < R1 with stride s1, q < R2 with stride s2) and the axis
// index has stride sm, so the same kernel serves x, y and z without
// transposes (Section 2.4, Eq. 11: the paper's tensorprod / pagemtimes).
//
// The FP64 pipe bounds it (1.05 TF/s on this GPU, reached at n = 255), so W is
// taken in its parity blocks (Axis1D::par), which halves the multiply-adds:
// forward, the A tiles are the half sums and half differences of a line,
// formed as they are loaded, and the outputs are the modes, even ones first;
// backward, the A tiles are the two halves of the modes and the epilogue
// writes E + O and E - O to the mirrored nodes.  A CTA computes BM rows x
// (32 even + 32 odd) outputs in K chunks of 16 + 16; the next chunk's loads
// are in flight while the current one is multiplied.  8 warps, each owning
// BM/2 rows x (8 even + 8 odd) outputs, i.e. BM/16 x 2 fragments of
// mma.m8n8k4.f64.  Measured per pass: n = 255 8.0 ms (full matrices) -> 4.0;
// n = 63 88 us (full matrices, 64-row tiles) -> 25.

constexpr int F64_BN = 32, F64_BK = 16;  // outputs and K of one parity per CTA and chunk

struct F64Pass {
  const double* in;
  double* out;
  const double* W;        // even block (ne x ne row-major), then the odd one (no x no)
  long long s1, s2, sm;   // strides of p, q and the axis index
  int R1, R2, n, ne, no;  // row loops and axis length
  int epi;
  int nx, ny;             // to decode (i, j, l) for the division epilogue
  const double *lamx, *lamy, *lamz;  // mode order (even modes first)
  double c;
};

// Half of x off the FP64 pipe, which bounds the passes: one off the exponent; below 2^-1021 the magnitude's
// bits shifted, the last one dropped; infinities and NaN as they are.
__device__ __forceinline__ double half_of(double x) {
  const unsigned int h = (unsigned int)__double2hiint(x), w = (unsigned int)__double2loint(x);
  const unsigned int m = h & 0x7FFFFFFFu, sign = h & 0x80000000u;
  const bool tiny = m < 0x00200000u;
  const unsigned int hi = tiny ? m >> 1 : m < 0x7FF00000u ? m - 0x00100000u : m;
  return __hiloint2double((int)(sign | hi), (int)(tiny ? __funnelshift_r(w, m, 1) : w));
}

template <bool KCONTIG, bool FWD, bool HALF, int BM>
__global__ void __launch_bounds__(256) mode_product_f64_kernel(F64Pass p) {
  constexpr int AF = BM / 16;                    // fragments of 8 rows per warp
  constexpr int LA = BM * F64_BK / 256;          // (even, odd) A pairs loaded per thread and chunk
  constexpr int LW = 2 * F64_BN * F64_BK / 256;  // W entries loaded per thread and chunk
  __shared__ double As[2][F64_BK][BM + 1];       // [parity]
  __shared__ double Bs[2][F64_BK][F64_BN + 1];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const long long rows = (long long)p.R1 * p.R2;
  const long long row0 = (long long)blockIdx.x * BM;
  const int o0 = blockIdx.y * F64_BN;
  const int wr = (warp & 1) * (BM / 2), wc = (warp >> 1) * 8;

  // (no pdl_trigger: blocks set up early would share the SMs that idle in this
  // pass, and with them one FP64 pipe, in their own: 63^3 315 -> 480 us)
  // The rows this thread loads are the same in every chunk.
  const double* abase[LA];
#pragma unroll
  for (int it = 0; it < LA; ++it) {
    const int e = tid + it * 256;
    const long long row = row0 + (KCONTIG ? e / F64_BK : e % BM);
    abase[it] = row < rows ? p.in + (row % p.R1) * p.s1 + (row / p.R1) * p.s2 : nullptr;
  }
  double ra[LA][2], rw[LW];
  auto load = [&](int t0) {
#pragma unroll
    for (int it = 0; it < LA; ++it) {
      const int e = tid + it * 256;
      const int t = t0 + (KCONTIG ? e % F64_BK : e / BM);
      double u = 0.0, v = 0.0;
      if (abase[it] && t < p.ne) {
        u = abase[it][(long long)t * p.sm];
        if (t < p.no) v = abase[it][(long long)(FWD ? p.n - 1 - t : p.ne + t) * p.sm];
      }
      // the middle node of an odd n (t = no) has no partner: v = 0 and the
      // odd block has no such column
      ra[it][0] = FWD && !HALF ? u + v : u;
      ra[it][1] = FWD && !HALF ? (t < p.no ? u - v : 0.0) : v;
    }
#pragma unroll
    for (int it = 0; it < LW; ++it) {
      const int e = tid + it * 256;
      const int kk = e % F64_BK, o = o0 + (e / F64_BK) % F64_BN, par = e / (F64_BK * F64_BN);
      const int t = t0 + kk, m = par == 0 ? p.ne : p.no;
      rw[it] = (o < m && t < m) ? __ldg(p.W + (par == 0 ? 0 : (long long)p.ne * p.ne) + (long long)o * m + t) : 0.0;
    }
  };
  auto store = [&](int t0) {
#pragma unroll
    for (int it = 0; it < LA; ++it) {
      const int e = tid + it * 256;
      const int kk = KCONTIG ? e % F64_BK : e / BM, r = KCONTIG ? e / F64_BK : e % BM;
      if (HALF) {  // no sum of a mirrored pair overflows (here: the loads stay in flight)
        const double u = half_of(ra[it][0]), v = half_of(ra[it][1]);
        As[0][kk][r] = u + v;
        As[1][kk][r] = t0 + kk < p.no ? u - v : 0.0;
      } else {
        As[0][kk][r] = ra[it][0];
        As[1][kk][r] = ra[it][1];
      }
    }
#pragma unroll
    for (int it = 0; it < LW; ++it) {
      const int e = tid + it * 256;
      Bs[e / (F64_BK * F64_BN)][e % F64_BK][(e / F64_BK) % F64_BN] = rw[it];
    }
  };

  double acc[AF][2][2];  // [fragment][parity][column]
#pragma unroll
  for (int a = 0; a < AF; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) acc[a][b][0] = acc[a][b][1] = 0.0;

  pdl_wait();
  load(0);
  for (int t0 = 0; t0 < p.ne; t0 += F64_BK) {
    store(t0);
    __syncthreads();
    if (t0 + F64_BK < p.ne) load(t0 + F64_BK);
#pragma unroll
    for (int k4 = 0; k4 < F64_BK; k4 += 4) {
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        const double bfr = Bs[b][k4 + (lane & 3)][wc + (lane >> 2)];
#pragma unroll
        for (int a = 0; a < AF; ++a) {
          const double afr = As[b][k4 + (lane & 3)][wr + a * 8 + (lane >> 2)];
          asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0,%1}, {%2}, {%3}, {%0,%1};\n"
                       : "+d"(acc[a][b][0]), "+d"(acc[a][b][1])
                       : "d"(afr), "d"(bfr));
        }
      }
    }
    __syncthreads();
  }
  // Epilogue: fragment a holds rows wr + a*8 + lane/4, outputs
  // wc + 2*(lane%4) + {0,1} of both parities.
  auto put = [&](long long base, int o, double v) {
    const long long idx = base + (long long)o * p.sm;
    if (FWD && KCONTIG && p.epi == EPI_DIV) {
      const long long i = idx % p.nx, jl = idx / p.nx;
      const long long j = jl % p.ny, l = jl / p.ny;
      p.out[idx] = v / half_of(p.lamx[i] + p.lamy[j] + p.lamz[l] + p.c);  // of halved right-hand sides
    } else if (p.epi == EPI_ACCUM) {
      p.out[idx] += v;
    } else {
      p.out[idx] = v;
    }
  };
#pragma unroll
  for (int a = 0; a < AF; ++a) {
    const long long row = row0 + wr + a * 8 + (lane >> 2);
    if (row >= rows) continue;
    const long long base = (row % p.R1) * p.s1 + (row / p.R1) * p.s2;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int o = o0 + wc + 2 * (lane & 3) + h;
      if (o >= p.ne) continue;
      const double e = acc[a][0][h], d = acc[a][1][h];
      if (o >= p.no) {  // the middle of an odd n
        put(base, o, e);
      } else if (FWD) {
        put(base, o, e);
        put(base, p.ne + o, d);
      } else {
        put(base, o, e + d);
        put(base, p.n - 1 - o, e - d);
      }
    }
  }
}

template <bool KCONTIG, bool FWD, bool HALF = false>
cudaError_t launch_f64(const F64Pass& p, int num_sms, cudaStream_t s) {
  // Rows per CTA: the CTAs of an SM share its FP64 pipe, so a pass takes as
  // long as the SM with the most rows; the largest tile within that minimum.
  // (n = 63: 125 tiles of 32 rows, one per SM at most, instead of 62 of 64.)
  const long long rows = (long long)p.R1 * p.R2;
  const long long nt = (p.ne + F64_BN - 1) / F64_BN;
  int best = 64;
  long long best_cost = 0;
  for (int bm : {64, 32, 16}) {
    const long long blocks = (rows + bm - 1) / bm * nt;
    const long long cost = (blocks + num_sms - 1) / num_sms * bm;
    if (bm == 64 || cost < best_cost) { best = bm; best_cost = cost; }
  }
  const long long bx = (rows + best - 1) / best;
  if (bx >= (1LL << 31)) return cudaErrorInvalidValue;
  const dim3 grid((unsigned)bx, (unsigned)nt);
  if (best == 64) return launch_pdl(mode_product_f64_kernel<KCONTIG, FWD, HALF, 64>, grid, dim3(256), 0, s, p);
  if (best == 32) return launch_pdl(mode_product_f64_kernel<KCONTIG, FWD, HALF, 32>, grid, dim3(256), 0, s, p);
  return launch_pdl(mode_product_f64_kernel<KCONTIG, FWD, HALF, 16>, grid, dim3(256), 0, s, p);
}

// ------------------------------------------------------------------ stencil
//
// (H_x (+) H_y (+) H_z) u with the banded H = M^{-1} S of each axis
// (Eq. 12): row i of H couples the nodes of the one or two elements that
// contain node i, stored as H[i][i+d], d in [-k, k].  One thread per node.

struct StencilArgs {
  const double* u;
  const double* f;
  double* out64;
  __nv_bfloat16* hi;
  __nv_bfloat16* lo;
  const double *Hx, *Hy, *Hz;
  const int *lox, *hix, *loy, *hiy, *loz, *hiz;
  int nx, ny, nz, k, Px, mode;
  double c;
  float* out32;        // mode 3: FP32 residual at pitch Px; with st, max |r| -> slot 0 (element kernels)
  F16State* st;
};

__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xFFFFFFFFu, v, o));
  return v;
}

__global__ void __launch_bounds__(256) stencil_kernel(StencilArgs a) {
  const long long N = (long long)a.nx * a.ny * a.nz;
  const int bw = 2 * a.k + 1;
  for (long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x; idx < N;
       idx += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(idx % a.nx);
    const long long jl = idx / a.nx;
    const int j = (int)(jl % a.ny), l = (int)(jl / a.ny);
    const double* u = a.u;
    double s = a.c * u[idx];
    // x: the band of row i (lanes of a warp sit on different rows of H_x).
    {
      const double* h = a.Hx + (long long)i * bw;
      const long long base = idx - i;
      for (int t = a.lox[i]; t <= a.hix[i]; ++t) s += h[t - i + a.k] * u[base + t];
    }
    // y
    {
      const double* h = a.Hy + (long long)j * bw;
      const long long base = idx - (long long)j * a.nx;
      for (int t = a.loy[j]; t <= a.hiy[j]; ++t) s += h[t - j + a.k] * u[base + (long long)t * a.nx];
    }
    // z
    {
      const double* h = a.Hz + (long long)l * bw;
      const long long pl = (long long)a.nx * a.ny;
      const long long base = idx - (long long)l * pl;
      for (int t = a.loz[l]; t <= a.hiz[l]; ++t) s += h[t - l + a.k] * u[base + (long long)t * pl];
    }
    if (a.mode == 0) {
      a.out64[idx] = s;
    } else {
      const double r = a.f[idx] - s;
      if (a.mode == 1) {
        a.out64[idx] = r;
      } else if (a.mode == 3) {
        a.out32[(long long)i + (long long)a.Px * jl] = (float)r;
      } else {
        const float rf = (float)r;
        const __nv_bfloat16 h16 = __float2bfloat16_rn(rf);
        const __nv_bfloat16 l16 = __float2bfloat16_rn(rf - __bfloat162float(h16));
        const long long o = (long long)i + (long long)a.Px * jl;
        a.hi[o] = h16;
        a.lo[o] = l16;
      }
    }
  }
}

// Element-wise variant of the same operator for a uniform mesh and
// 1 <= K <= 8, bound by the FP64 pipe.  Along x, one thread owns the K global nodes g = ex*K + q
// (q = 0..K-1) of element ex: node q = 0 is the vertex shared with element
// ex-1 (row of 2K+1 entries), q > 0 are the element's other nodes (K+1
// entries each).  The thread keeps the 2K+1 node values of elements ex-1 and
// ex in registers, and every thread runs the same fully unrolled loops, so
// the lanes of a warp never wait on each other's band lengths.  The rows of
// H depend only on q (table Hq, x table with c added on its diagonal).  The
// y and z bands are uniform across a warp (its lanes share j and l).
// Work per node: k+2 FMAs per axis on average (6 at k = 4), accumulated from
// f in residual modes.
// With Neumann data (NEU) every global node is an unknown, and a boundary row is
// the vertex row applied to values mirrored at the boundary (its stiffness and
// mass are half an inner vertex's, so its entries are twice the one-sided
// ones: the same numbers, halved and doubled exactly).  The last node of a
// line has an element of its own.  (321x161x241, k = 5: 679 us with a thread per
// node and per-row band tables -> 477.)
template <int K, int MODE, bool NEU>
__global__ void __launch_bounds__(256) stencil_elem_kernel(StencilArgs a, const double* __restrict__ Hqx,
                                                           const double* __restrict__ Hqy,
                                                           const double* __restrict__ Hqz, int nex) {
  constexpr int BW = 2 * K + 1, OFF = NEU ? 0 : 1;  // unknown index = global node - OFF
  const long long lines = (long long)a.ny * a.nz;
  const long long total = (long long)nex * lines;
  const long long plane = (long long)a.nx * a.ny;
  float rmax = 0.f;  // MODE 3: max |r| of this thread's nodes
  // unknown `i` of an axis of n nodes, mirrored at a Neumann boundary
  auto mirror = [](int i, int n) { return NEU ? (i < 0 ? -i : i >= n ? 2 * (n - 1) - i : i) : i; };
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    const int ex = (int)(t % nex);
    const long long jl = t / nex;
    const int j = (int)(jl % a.ny), l = (int)(jl / a.ny);
    const long long line = jl * a.nx;
    const int i0 = ex * K - OFF;  // unknown index of node q = 0 (g = ex*K)
    auto own = [&](int i) { return NEU ? i < a.nx : i >= 0; };  // a node of this thread's that exists
    // x window: global nodes (ex-1)K .. (ex+1)K -> unknowns i0-K .. i0+K
    double w[BW];
#pragma unroll
    for (int d = 0; d < BW; ++d) {
      const int i = mirror(i0 - K + d, a.nx);
      w[d] = (i >= 0 && i < a.nx) ? __ldg(a.u + line + i) : 0.0;
    }
    double acc[K];
#pragma unroll
    for (int q = 0; q < K; ++q) {
      const int i = i0 + q;
      acc[q] = (MODE != 0 && own(i)) ? __ldg(a.f + line + i) : 0.0;
    }
    // x part
#pragma unroll
    for (int q = 0; q < K; ++q) {
      const int dlo = (q == 0) ? -K : -q, dhi = (q == 0) ? K : K - q;
#pragma unroll
      for (int d = dlo; d <= dhi; ++d) {
        const double hv = __ldg(Hqx + q * BW + d + K);
        if (MODE == 0) acc[q] += hv * w[K + q + d];
        else acc[q] -= hv * w[K + q + d];
      }
    }
    // y part: row j of H_y, local index qy = (j+OFF) % K
    {
      const int qy = (j + OFF) % K;
      const int dlo = (qy == 0) ? -K : -qy, dhi = (qy == 0) ? K : K - qy;
      for (int d = dlo; d <= dhi; ++d) {
        const int jj = mirror(j + d, a.ny);
        if (jj < 0 || jj >= a.ny) continue;
        const double hv = __ldg(Hqy + qy * BW + d + K);
        const double* src = a.u + ((long long)l * a.ny + jj) * a.nx;
#pragma unroll
        for (int q = 0; q < K; ++q) {
          const int i = i0 + q;
          const double uv = own(i) ? __ldg(src + i) : 0.0;
          if (MODE == 0) acc[q] += hv * uv;
          else acc[q] -= hv * uv;
        }
      }
    }
    // z part
    {
      const int qz = (l + OFF) % K;
      const int dlo = (qz == 0) ? -K : -qz, dhi = (qz == 0) ? K : K - qz;
      for (int d = dlo; d <= dhi; ++d) {
        const int ll = mirror(l + d, a.nz);
        if (ll < 0 || ll >= a.nz) continue;
        const double hv = __ldg(Hqz + qz * BW + d + K);
        const double* src = a.u + (long long)ll * plane + (long long)j * a.nx;
#pragma unroll
        for (int q = 0; q < K; ++q) {
          const int i = i0 + q;
          const double uv = own(i) ? __ldg(src + i) : 0.0;
          if (MODE == 0) acc[q] += hv * uv;
          else acc[q] -= hv * uv;
        }
      }
    }
    if (MODE == 3) {
#pragma unroll
      for (int q = 0; q < K; ++q) {
        const int i = i0 + q;
        if (!own(i)) continue;
        const float rf = (float)acc[q];
        a.out32[(long long)i + (long long)a.Px * jl] = rf;
        rmax = fmaxf(rmax, fabsf(rf));
      }
      continue;
    }
#pragma unroll
    for (int q = 0; q < K; ++q) {
      const int i = i0 + q;
      if (!own(i)) continue;
      if (MODE != 2) {
        a.out64[line + i] = acc[q];
      } else {
        const float rf = (float)acc[q];
        const __nv_bfloat16 h16 = __float2bfloat16_rn(rf);
        const __nv_bfloat16 l16 = __float2bfloat16_rn(rf - __bfloat162float(h16));
        const long long o = (long long)i + (long long)a.Px * jl;
        a.hi[o] = h16;
        a.lo[o] = l16;
      }
    }
  }
  if (MODE == 3 && a.st) {  // every lane of the warp gets here (after the loop)
    rmax = warp_max(rmax);
    if ((threadIdx.x & 31) == 0 && rmax > 0.f) atomicMax(&a.st->maxbits[0], __float_as_uint(rmax));
  }
}

template <int K, bool NEU>
cudaError_t launch_elem(const StencilArgs& a, const DevAxis* ax, int mode, cudaStream_t s) {
  const int nex = NEU ? (a.nx - 1) / K + 1 : (a.nx + 1) / K;
  const long long total = (long long)nex * a.ny * a.nz;
  long long b = (total + 255) / 256;
  // One thread per work item (no grid-stride wrap): blocks are issued in
  // order, so the resident set sweeps the grid plane by plane and the z
  // neighbours of a plane are still in L2 when they are read again.
  if (b > 0x7FFFFFFFLL) b = 0x7FFFFFFFLL;
  const int grid = (int)(b < 1 ? 1 : b);
  const double *hx = ax[0].Hq, *hy = ax[1].Hq, *hz = ax[2].Hq;
  if (mode == 0) stencil_elem_kernel<K, 0, NEU><<<grid, 256, 0, s>>>(a, hx, hy, hz, nex);
  else if (mode == 1) stencil_elem_kernel<K, 1, NEU><<<grid, 256, 0, s>>>(a, hx, hy, hz, nex);
  else if (mode == 2) stencil_elem_kernel<K, 2, NEU><<<grid, 256, 0, s>>>(a, hx, hy, hz, nex);
  else stencil_elem_kernel<K, 3, NEU><<<grid, 256, 0, s>>>(a, hx, hy, hz, nex);
  return cudaGetLastError();
}

// Zero the pad columns i in [nx, Px) of a split array (the stencil writes
// only i < nx).
__global__ void zero_pads_kernel(__nv_bfloat16* hi, __nv_bfloat16* lo, int nx, int Px, long long lines) {
  const int w = Px - nx;
  const long long total = lines * w;
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    const long long line = e / w;
    const long long o = line * Px + nx + (e % w);
    hi[o] = __float2bfloat16_rn(0.f);
    lo[o] = __float2bfloat16_rn(0.f);
  }
}

// FP64 (dense, pitch nx) -> bf16 hi + lo (pitch Px, zero pads):
// hi = bf16(x), lo = bf16(x - hi), x rounded to FP32 first.  A group of
// 2^shift lanes (a warp, or fewer where a line has fewer chunks of 4) walks a
// (j, l) line; a lane converts 4 consecutive entries and writes them as one
// 8-byte store per array (rows of pitch Px, a multiple of 16, are aligned).
// With emax set, the largest biased FP64 exponent of the input also goes to
// *emax (the fixed-point residual's scale of f); the slot is read before the
// atomic, which most warps then skip.  A block per line before, most of it idle
// on short lines: 63^3 7.2 -> 5.7 us, 321x161x241 41 -> 29 us (5.1 TB/s).
__global__ void __launch_bounds__(256) split_kernel(const double* in, __nv_bfloat16* hi, __nv_bfloat16* lo, int nx,
                                                    int Px, long long lines, int shift, int* emax) {
  const int chunks = Px >> 2, group = 1 << shift;
  const int c0 = threadIdx.x & (group - 1);
  unsigned int m = 0;
  for (long long line = ((long long)blockIdx.x * 256 + threadIdx.x) >> shift; line < lines;
       line += (long long)gridDim.x * 256 >> shift) {
    const double* row = in + line * nx;
    uint2* hrow = reinterpret_cast<uint2*>(hi + line * Px);
    uint2* lrow = reinterpret_cast<uint2*>(lo + line * Px);
#pragma unroll 2
    for (int c = c0; c < chunks; c += group) {
      uint32_t hw[2], lw[2];
#pragma unroll
      for (int p = 0; p < 4; p += 2) {
        const int i = 4 * c + p;
        const double d0 = i < nx ? row[i] : 0.0, d1 = i + 1 < nx ? row[i + 1] : 0.0;
        m = max(m, max((unsigned int)(__double_as_longlong(d0) >> 52) & 0x7FFu,
                       (unsigned int)(__double_as_longlong(d1) >> 52) & 0x7FFu));
        const float x0 = f64_to_f32_rn(d0), x1 = f64_to_f32_rn(d1);
        const __nv_bfloat16 h0 = __float2bfloat16_rn(x0), h1 = __float2bfloat16_rn(x1);
        const __nv_bfloat16 l0 = __float2bfloat16_rn(x0 - __bfloat162float(h0));
        const __nv_bfloat16 l1 = __float2bfloat16_rn(x1 - __bfloat162float(h1));
        hw[p / 2] = (uint32_t)__bfloat16_as_ushort(h0) | ((uint32_t)__bfloat16_as_ushort(h1) << 16);
        lw[p / 2] = (uint32_t)__bfloat16_as_ushort(l0) | ((uint32_t)__bfloat16_as_ushort(l1) << 16);
      }
      hrow[c] = make_uint2(hw[0], hw[1]);
      lrow[c] = make_uint2(lw[0], lw[1]);
    }
  }
  if (emax) {  // every lane of the block gets here
    m = __reduce_max_sync(0xFFFFFFFFu, m);
    if ((threadIdx.x & 31) == 0 && (int)m > __ldcg(emax)) atomicMax(emax, (int)m);
  }
}

// Grid of a streaming (grid-stride) kernel: enough blocks to fill the GPU a
// few times over; each thread then walks the arrays in order.
int grid_for(long long work, int per_block) {
  long long b = (work + per_block - 1) / per_block;
  if (b > 152LL * 32) b = 152LL * 32;
  if (b < 1) b = 1;
  return (int)b;
}

}  // namespace

cudaError_t launch_mode_product_f64(const Geom& g, int axis, const DevAxis* ax, int which, const double* in,
                                    double* out, int epi, int num_sms, cudaStream_t s) {
  F64Pass p{};
  p.in = in;
  p.out = out;
  p.W = ax[axis].par[which];
  p.n = ax[axis].n;
  p.ne = ax[axis].ne;
  p.no = ax[axis].no;
  p.epi = epi;
  p.nx = g.nx;
  p.ny = g.ny;
  p.lamx = ax[0].lam_par;
  p.lamy = ax[1].lam_par;
  p.lamz = ax[2].lam_par;
  p.c = g.c;
  const long long nxy = (long long)g.nx * g.ny;
  bool kcontig = false;
  if (axis == 0) {         // rows = (j,l) lines, t = i contiguous
    p.R1 = g.ny * g.nz; p.R2 = 1; p.s1 = g.nx; p.s2 = 0; p.sm = 1; kcontig = true;
  } else if (axis == 1) {  // rows = (i, l), t = j
    p.R1 = g.nx; p.R2 = g.nz; p.s1 = 1; p.s2 = nxy; p.sm = g.nx;
  } else {                 // rows = (i,j) plane, t = l
    p.R1 = (int)nxy; p.R2 = 1; p.s1 = 1; p.s2 = 0; p.sm = nxy;
  }
  if (epi == EPI_DIV && (axis != 0 || which != 0)) return cudaErrorInvalidValue;
  if (epi == EPI_HALF) {  // the first pass of a solve
    if (kcontig || which != 0) return cudaErrorInvalidValue;
    return launch_f64<false, true, true>(p, num_sms, s);
  }
  if (which == 0) return kcontig ? launch_f64<true, true>(p, num_sms, s) : launch_f64<false, true>(p, num_sms, s);
  return kcontig ? launch_f64<true, false>(p, num_sms, s) : launch_f64<false, false>(p, num_sms, s);
}

namespace {

StencilArgs stencil_args(const Geom& g, int k, const DevAxis* ax, const double* u, const double* f, int mode) {
  StencilArgs a{};
  a.u = u; a.f = f;
  a.Hx = ax[0].Hband; a.Hy = ax[1].Hband; a.Hz = ax[2].Hband;
  a.lox = ax[0].band_lo; a.hix = ax[0].band_hi;
  a.loy = ax[1].band_lo; a.hiy = ax[1].band_hi;
  a.loz = ax[2].band_lo; a.hiz = ax[2].band_hi;
  a.nx = g.nx; a.ny = g.ny; a.nz = g.nz; a.k = k; a.Px = g.Px; a.mode = mode; a.c = g.c;
  return a;
}

cudaError_t launch_stencil_any(const StencilArgs& a, const Geom& g, const DevAxis* ax, cudaStream_t s) {
  const long long N = (long long)g.nx * g.ny * g.nz;
  const bool neu = g.bc != 0;
  switch (a.k) {
    case 1: return neu ? launch_elem<1, true>(a, ax, a.mode, s) : launch_elem<1, false>(a, ax, a.mode, s);
    case 2: return neu ? launch_elem<2, true>(a, ax, a.mode, s) : launch_elem<2, false>(a, ax, a.mode, s);
    case 3: return neu ? launch_elem<3, true>(a, ax, a.mode, s) : launch_elem<3, false>(a, ax, a.mode, s);
    case 4: return neu ? launch_elem<4, true>(a, ax, a.mode, s) : launch_elem<4, false>(a, ax, a.mode, s);
    case 5: return neu ? launch_elem<5, true>(a, ax, a.mode, s) : launch_elem<5, false>(a, ax, a.mode, s);
    case 6: return neu ? launch_elem<6, true>(a, ax, a.mode, s) : launch_elem<6, false>(a, ax, a.mode, s);
    case 7: return neu ? launch_elem<7, true>(a, ax, a.mode, s) : launch_elem<7, false>(a, ax, a.mode, s);
    case 8: return neu ? launch_elem<8, true>(a, ax, a.mode, s) : launch_elem<8, false>(a, ax, a.mode, s);
    default:  // higher degrees: one thread per node, per-row band ranges
      stencil_kernel<<<(int)((N + 255) / 256 < 0x7FFFFFFF ? (N + 255) / 256 : 0x7FFFFFFF), 256, 0, s>>>(a);
      return cudaGetLastError();
  }
}

}  // namespace

cudaError_t launch_stencil(const Geom& g, int k, const DevAxis* ax, const double* u, const double* f, double* out64,
                           __nv_bfloat16* out_hi, __nv_bfloat16* out_lo, int mode, cudaStream_t s) {
  StencilArgs a = stencil_args(g, k, ax, u, f, mode);
  a.out64 = out64; a.hi = out_hi; a.lo = out_lo;
  const cudaError_t e = launch_stencil_any(a, g, ax, s);
  if (e != cudaSuccess || mode != 2 || g.Px == g.nx) return e;
  const long long lines = (long long)g.ny * g.nz;
  zero_pads_kernel<<<grid_for(lines * (g.Px - g.nx), 256), 256, 0, s>>>(out_hi, out_lo, g.nx, g.Px, lines);
  return cudaGetLastError();
}

cudaError_t launch_stencil_f32out(const Geom& g, int k, const DevAxis* ax, const double* u, const double* f,
                                  float* out32, F16State* st, cudaStream_t s) {
  if (st && (k < 1 || k > 8 || g.bc != 0)) return cudaErrorInvalidValue;
  StencilArgs a = stencil_args(g, k, ax, u, f, 3);
  a.out32 = out32; a.st = st;
  return launch_stencil_any(a, g, ax, s);
}

// ------------------------------------------------------------------ F16X3 split
__global__ void __launch_bounds__(256) absmax_f64_kernel(const double* in, long long N, F16State* st) {
  float m = 0.f;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x)
    m = fmaxf(m, (float)fabs(in[i]));
  m = warp_max(m);
  if ((threadIdx.x & 31) == 0 && m > 0.f) atomicMax(&st->maxbits[0], __float_as_uint(m));
}

// hi + lo = fp16 split of x * 2^e, e from slot 0's max (largest |x 2^e| near
// 2^15 < 65504); fp16 subnormals keep the absolute error below 2^-24 of 2^e.
template <bool IN64>
__global__ void __launch_bounds__(256) split_f16_kernel(const void* in, __half* hi, __half* lo, int nx, int Px,
                                                        long long lines, F16State* st) {
  const float mx = __uint_as_float(st->maxbits[0]);
  int e = 0;
  if (mx > 0.f && isfinite(mx)) {
    e = ilogbf(32768.f / mx);
    e = e < -120 ? -120 : (e > 120 ? 120 : e);
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) st->e[0] = e;
  const float sc = __int_as_float((e + 127) << 23);
  const long long total = lines * Px;
  for (long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (long long)gridDim.x * blockDim.x) {
    const long long line = idx / Px;
    const int i = (int)(idx - line * Px);
    float x = 0.f;
    if (i < nx) x = IN64 ? f64_to_f32_rn(static_cast<const double*>(in)[line * nx + i]) : static_cast<const float*>(in)[idx];
    x *= sc;
    const __half h = __float2half_rn(x);
    hi[idx] = h;
    lo[idx] = __float2half_rn(x - __half2float(h));
  }
}

cudaError_t launch_absmax_f64(const Geom& g, const double* in, F16State* st, cudaStream_t s) {
  const long long N = (long long)g.nx * g.ny * g.nz;
  absmax_f64_kernel<<<grid_for(N, 256), 256, 0, s>>>(in, N, st);
  return cudaGetLastError();
}

cudaError_t launch_split_f16(const Geom& g, const void* in, bool in_f64, __half* hi, __half* lo, F16State* st,
                             cudaStream_t s) {
  const long long lines = (long long)g.ny * g.nz;
  if (in_f64) split_f16_kernel<true><<<grid_for(lines * g.Px, 256), 256, 0, s>>>(in, hi, lo, g.nx, g.Px, lines, st);
  else split_f16_kernel<false><<<grid_for(lines * g.Px, 256), 256, 0, s>>>(in, hi, lo, g.nx, g.Px, lines, st);
  return cudaGetLastError();
}

cudaError_t launch_split(const Geom& g, const double* in, __nv_bfloat16* hi, __nv_bfloat16* lo, cudaStream_t s,
                         int* emax) {
  const long long lines = (long long)g.ny * g.nz;
  int shift = 2;
  while (shift < 5 && (1 << shift) < (g.Px >> 2)) ++shift;
  long long blocks = ((lines << shift) + 255) / 256;
  if (blocks > 152LL * 16) blocks = 152LL * 16;
  if (blocks < 1) blocks = 1;
  split_kernel<<<(int)blocks, 256, 0, s>>>(in, hi, lo, g.nx, g.Px, lines, shift, emax);
  return cudaGetLastError();
}

}  // namespace sem3d
