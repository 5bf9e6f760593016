// Pointwise kernels of the Cahn-Hilliard BDF2 step (Section 3.5, Eqs. 19-20).
//
// With -Lap -> H3 = T3 diag(L) T3^{-1} (L = lambda_x,i + lambda_y,j +
// lambda_z,l), one step is
//   phi_{n+1} = T3 [ (T3^{-1} phi_hat - dt m L * T3^{-1} g)
//                    / (a + dt m (eps L^2 + (S/eps) L)) ]
// phi_hat = 2 phi_n - phi_{n-1}/2, g = (F'(phi_bar) - S phi_bar)/eps,
// phi_bar = 2 phi_n - phi_{n-1}, F'(phi) = phi^3 - phi, a = 3/2.  The two
// forward transforms and the backward one are the solver's mode products;
// these kernels do the pointwise parts (prep before, combine in between).
#include "sem3d_internal.h"

namespace sem3d {

namespace {

constexpr int CH_THREADS = 256;

int ch_grid(long long n) {
  long long b = (n + CH_THREADS - 1) / CH_THREADS;
  if (b > 152LL * 32) b = 152LL * 32;
  return (int)(b < 1 ? 1 : b);
}

__device__ __forceinline__ void split2f(float v, __nv_bfloat16& h, __nv_bfloat16& l) {
  h = __float2bfloat16_rn(v);
  l = __float2bfloat16_rn(v - __bfloat162float(h));
}

// FP64 / FP32 inputs: phi_hat and g at pitch nx.
template <typename T>
__global__ void __launch_bounds__(CH_THREADS) ch_prep_kernel(const double* phi_n, const double* phi_nm1, T* ghat,
                                                             T* g, long long N, ChParams c) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x) {
    const double pn = phi_n[i], pm = phi_nm1[i];
    const double bar = 2.0 * pn - pm;
    ghat[i] = (T)(2.0 * pn - 0.5 * pm);
    g[i] = (T)((bar * bar * bar - bar - c.S * bar) / c.eps);
  }
}

// Four values split into bf16 hi + lo, packed for one 8-byte store each.
__device__ __forceinline__ void split4(const float (&v)[4], uint2& h, uint2& l) {
  __nv_bfloat16 hh[4], ll[4];
#pragma unroll
  for (int p = 0; p < 4; ++p) split2f(v[p], hh[p], ll[p]);
  auto pack = [](__nv_bfloat16 a, __nv_bfloat16 b) {
    return (uint32_t)__bfloat16_as_ushort(a) | ((uint32_t)__bfloat16_as_ushort(b) << 16);
  };
  h = make_uint2(pack(hh[0], hh[1]), pack(hh[2], hh[3]));
  l = make_uint2(pack(ll[0], ll[1]), pack(ll[2], ll[3]));
}

// Split-bf16 inputs (pitch Px, zero pads), FP32 arithmetic.  Threads walk the
// nodes in order, a thread takes 4 consecutive ones of a line: the bf16 arrays are then
// written (and, below, read) 8 bytes at a time.  Bound by HBM (24 B per node);
// n = 511, one node a thread and 2-byte stores -> this: 749 -> 463 us.
__global__ void __launch_bounds__(CH_THREADS) ch_prep_split_kernel(const double* __restrict__ phi_n,
                                                                   const double* __restrict__ phi_nm1,
                                                                   __nv_bfloat16* gh_hi, __nv_bfloat16* gh_lo,
                                                                   __nv_bfloat16* g_hi, __nv_bfloat16* g_lo, int nx,
                                                                   int Px, long long lines, ChParams c) {
  const float S = (float)c.S, inv_eps = (float)(1.0 / c.eps);
  const int chunks = Px >> 2;
  const long long total = lines * chunks;
  for (long long w = (long long)blockIdx.x * blockDim.x + threadIdx.x; w < total;
       w += (long long)gridDim.x * blockDim.x) {
    const long long line = w / chunks;
    const int i0 = (int)(w - line * chunks) * 4;
    const double* pn_row = phi_n + line * nx + i0;
    const double* pm_row = phi_nm1 + line * nx + i0;
    double dn[4], dm[4];
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      dn[p] = i0 + p < nx ? __ldg(pn_row + p) : 0.0;
      dm[p] = i0 + p < nx ? __ldg(pm_row + p) : 0.0;
    }
    float gh[4], gg[4];
#pragma unroll
    for (int p = 0; p < 4; ++p) {  // zero beyond the line, as its inputs are
      const float pn = f64_to_f32_rn(dn[p]), pm = f64_to_f32_rn(dm[p]);
      const float bar = 2.f * pn - pm;
      gh[p] = 2.f * pn - 0.5f * pm;
      gg[p] = (bar * bar * bar - bar - S * bar) * inv_eps;
      if (i0 + p >= nx) gh[p] = gg[p] = 0.f;
    }
    const long long o = line * Px + i0;
    uint2 h, l;
    split4(gh, h, l);
    *reinterpret_cast<uint2*>(gh_hi + o) = h;
    *reinterpret_cast<uint2*>(gh_lo + o) = l;
    split4(gg, h, l);
    *reinterpret_cast<uint2*>(g_hi + o) = h;
    *reinterpret_cast<uint2*>(g_lo + o) = l;
  }
}

template <typename T>
__global__ void __launch_bounds__(CH_THREADS) ch_combine_kernel(const T* a1, const T* a2, T* out, const double* lx,
                                                                const double* ly, const double* lz, int nx, int ny,
                                                                long long N, ChParams c) {
  for (long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x; idx < N;
       idx += (long long)gridDim.x * blockDim.x) {
    const long long i = idx % nx, jl = idx / nx;
    const double L = lx[i] + ly[jl % ny] + lz[jl / ny];
    const double num = (double)a1[idx] - c.dt * c.m * L * (double)a2[idx];
    const double den = 1.5 + c.dt * c.m * (c.eps * L * L + (c.S / c.eps) * L);
    out[idx] = (T)(num / den);
  }
}

// As ch_prep_split_kernel (12 B per node): n = 511 458 -> 283 us.
__global__ void __launch_bounds__(CH_THREADS) ch_combine_split_kernel(
    const __nv_bfloat16* __restrict__ a1h, const __nv_bfloat16* __restrict__ a1l,
    const __nv_bfloat16* __restrict__ a2h, const __nv_bfloat16* __restrict__ a2l, __nv_bfloat16* oh, __nv_bfloat16* ol,
    const float* __restrict__ lx, const float* __restrict__ ly, const float* __restrict__ lz, int nx, int ny, int Px,
    long long lines, ChParams c) {
  const float dtm = (float)(c.dt * c.m), eps = (float)c.eps, s_eps = (float)(c.S / c.eps);
  const int chunks = Px >> 2;
  const long long total = lines * chunks;
  auto ld4 = [](const __nv_bfloat16* p, float (&v)[4]) {
    const uint2 r = __ldg(reinterpret_cast<const uint2*>(p));
    v[0] = __uint_as_float(r.x << 16); v[1] = __uint_as_float(r.x & 0xFFFF0000u);
    v[2] = __uint_as_float(r.y << 16); v[3] = __uint_as_float(r.y & 0xFFFF0000u);
  };
  for (long long w = (long long)blockIdx.x * blockDim.x + threadIdx.x; w < total;
       w += (long long)gridDim.x * blockDim.x) {
    const long long line = w / chunks;
    const int i0 = (int)(w - line * chunks) * 4;
    const float lyz = __ldg(ly + (int)(line % ny)) + __ldg(lz + (int)(line / ny));
    const long long o = line * Px + i0;
    float h1[4], l1[4], h2[4], l2[4], v[4];
    ld4(a1h + o, h1);
    ld4(a1l + o, l1);
    ld4(a2h + o, h2);
    ld4(a2l + o, l2);
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      v[p] = 0.f;
      if (i0 + p < nx) {
        const float L = __ldg(lx + i0 + p) + lyz;
        const float x1 = h1[p] + l1[p];
        const float x2 = h2[p] + l2[p];
        v[p] = (x1 - dtm * L * x2) / (1.5f + dtm * (eps * L * L + s_eps * L));
      }
    }
    uint2 h, l;
    split4(v, h, l);
    *reinterpret_cast<uint2*>(oh + o) = h;
    *reinterpret_cast<uint2*>(ol + o) = l;
  }
}

}  // namespace

cudaError_t launch_ch_prep(int tier, const Geom& g, const double* phi_n, const double* phi_nm1, void* ghat, void* gg,
                           TcBuffers sh, TcBuffers sg, const ChParams& c, cudaStream_t s) {
  const long long N = (long long)g.nx * g.ny * g.nz;
  if (tier == SEM3D_FP64) {
    ch_prep_kernel<double><<<ch_grid(N), CH_THREADS, 0, s>>>(phi_n, phi_nm1, static_cast<double*>(ghat),
                                                               static_cast<double*>(gg), N, c);
  } else if (tier == SEM3D_FP32) {
    ch_prep_kernel<float><<<ch_grid(N), CH_THREADS, 0, s>>>(phi_n, phi_nm1, static_cast<float*>(ghat),
                                                              static_cast<float*>(gg), N, c);
  } else {
    const long long lines = (long long)g.ny * g.nz;
    ch_prep_split_kernel<<<ch_grid(lines * (g.Px / 4)), CH_THREADS, 0, s>>>(phi_n, phi_nm1, sh.hi, sh.lo, sg.hi, sg.lo, g.nx,
                                                                  g.Px, lines, c);
  }
  return cudaGetLastError();
}

cudaError_t launch_ch_combine(int tier, const Geom& g, const DevAxis* ax, const void* a1, const void* a2, void* out,
                              TcBuffers s1, TcBuffers s2, TcBuffers so, const ChParams& c, cudaStream_t s) {
  const long long N = (long long)g.nx * g.ny * g.nz;
  if (tier == SEM3D_FP64) {
    ch_combine_kernel<double><<<ch_grid(N), CH_THREADS, 0, s>>>(
        static_cast<const double*>(a1), static_cast<const double*>(a2), static_cast<double*>(out),
        ax[0].lam_par, ax[1].lam_par, ax[2].lam_par, g.nx, g.ny, N, c);  // FP64 transforms order the modes by parity
  } else if (tier == SEM3D_FP32) {
    ch_combine_kernel<float><<<ch_grid(N), CH_THREADS, 0, s>>>(
        static_cast<const float*>(a1), static_cast<const float*>(a2), static_cast<float*>(out), ax[0].lam,
        ax[1].lam, ax[2].lam, g.nx, g.ny, N, c);
  } else {
    const long long lines = (long long)g.ny * g.nz;
    ch_combine_split_kernel<<<ch_grid(lines * (g.Px / 4)), CH_THREADS, 0, s>>>(
        s1.hi, s1.lo, s2.hi, s2.lo, so.hi, so.lo, ax[0].lamf, ax[1].lamf, ax[2].lamf, g.nx, g.ny, g.Px, lines, c);
  }
  return cudaGetLastError();
}

}  // namespace sem3d
