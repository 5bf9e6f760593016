// Low-precision copies of an axis's eigenbasis, made on the device at plan
// set-up from the FP64 matrices (n^2 entries, ten arrays each).  Bound by the
// FP64 upload.  A plan on axes already diagonalised, with the conversions on
// the host and one allocation per array -> now: n = 63 1.1 -> 0.33 ms, 255
// 10.0 -> 0.37 ms, 999 140 -> 0.6 ms; 449x320x383 19 -> 0.8 ms.
#include "sem3d_internal.h"

namespace sem3d {

namespace {

__device__ __forceinline__ void split_bf16(float x, __nv_bfloat16& hi, __nv_bfloat16& lo) {
  hi = __float2bfloat16_rn(x);
  lo = __float2bfloat16_rn(x - __bfloat162float(hi));
}

struct AxisCopies {
  const double* w[2];    // T^{-1}, T
  const double* par[2];  // their parity blocks
  float *f32[2], *pf32[2], *t32[2];
  __half *h16[2], *l16[2];
  __nv_bfloat16 *hi[2], *lo[2], *phi[2], *plo[2];
  double sc16[2];        // 2^eW16
  int n, Kp, ne, no;
};

// Blocks of 256 over the n x Kp entries of one matrix (blockIdx.y = 0: T^{-1},
// 1: T), pad columns included.
__global__ void __launch_bounds__(256) axis_copies_kernel(AxisCopies a) {
  const int q = blockIdx.y;
  const long long e = (long long)blockIdx.x * 256 + threadIdx.x;
  if (e < (long long)a.n * a.Kp) {
    const int o = (int)(e / a.Kp), t = (int)(e % a.Kp);
    const bool in = t < a.n;
    const double x = in ? a.w[q][(long long)o * a.n + t] : 0.0;
    const float f = (float)x;
    if (in) a.f32[q][(long long)o * a.n + t] = f;
    a.t32[q][e] = tf32_round(f);
    split_bf16(f, a.hi[q][e], a.lo[q][e]);
    const float s = (float)(x * a.sc16[q]);
    const __half h = __float2half_rn(s);
    a.h16[q][e] = h;
    a.l16[q][e] = __float2half_rn(s - __half2float(h));
  }
  const int pe = pad16(a.ne), po = pad16(a.no);
  const long long even = (long long)a.ne * pe;
  if (e < even + (long long)a.no * po) {
    const bool odd = e >= even;
    const long long r = odd ? e - even : e;
    const int p = odd ? po : pe, m = odd ? a.no : a.ne;
    const int o = (int)(r / p), t = (int)(r % p);
    const long long at = (odd ? (long long)a.ne * a.ne : 0) + (long long)o * m + t;
    const float x = t < m ? (float)a.par[q][at] : 0.f;
    if (t < m) a.pf32[q][at] = x;
    split_bf16(x, a.phi[q][e], a.plo[q][e]);
  }
}

}  // namespace

cudaError_t launch_axis_copies(const DevAxis& D, const double* const w[2], cudaStream_t s) {
  AxisCopies a{};
  a.n = D.n; a.Kp = D.Kp; a.ne = D.ne; a.no = D.no;
  for (int q = 0; q < 2; ++q) {
    a.w[q] = w[q];
    a.par[q] = D.par[q];
    a.f32[q] = D.Wf[q]; a.pf32[q] = D.Wpf[q]; a.t32[q] = D.Wt32[q];
    a.h16[q] = D.W16_hi[q]; a.l16[q] = D.W16_lo[q];
    a.hi[q] = D.W_hi[q]; a.lo[q] = D.W_lo[q];
    a.phi[q] = D.Wp_hi[q]; a.plo[q] = D.Wp_lo[q];
    a.sc16[q] = ldexp(1.0, D.eW16[q]);
  }
  const long long work = (long long)D.n * D.Kp;  // the parity blocks hold fewer entries
  axis_copies_kernel<<<dim3((unsigned)((work + 255) / 256), 2), 256, 0, s>>>(a);
  return cudaGetLastError();
}

}  // namespace sem3d
