// Parity form of the split tier's working arrays (see Axis1D::par for the
// 1D statement).  Folding every axis of the right-hand side once turns each of
// the six tensor-core passes into two independent products with matrices of
// half the size, on half the contracted axis each: half the tensor work, the
// same bytes, and no other change to the passes (the solve is then eight
// independent problems, one per combination of parities).
//   fold   : right-hand side (FP64) or residual (FP32), in node order ->
//            split-bf16 array in parity order, the sums over the 8 mirror
//            images of a node taken in FP32;
//   unfold : the correction (FP32, parity order, written by the last pass) ->
//            added to the solution at the 8 mirror images of a node.
// A thread takes the 8 mirror images of one node (fold: of two neighbours, so
// that the bf16 outputs go out in pairs).  Every stream is read and written in
// runs of whole lines, forwards or backwards.  A sum of 8 values may exceed
// FP32's range where the values do not: right-hand sides from 2^110 on, found by
// the exponent that the fold records, are folded again at 2^-8, their residuals
// and corrections scaled to match (powers of two: the same digits).  (Folding
// everything at 1/8 would cost the other end of the range: the low bf16 part of
// values below 1e-25.)  For all others that is one launch, 3 us, whose blocks
// return at once.  Both kernels are bound by HBM, the updates of the
// double-FP32 pair by too few warps waiting for it (48 to 80 registers): at
// n = 999 fold 1.9 ms from FP64 (12 B per node, 6.3 TB/s) and 1.14 ms from FP32
// (8 B, 7.0), unfold 2.85 ms into FP64 (20 B, 7.0), 1.6 ms into the pair (8 B,
// 5.0), 2.9 ms added to it (16 B, 5.6), 4.0 ms from the pair into FP64 (20 B, 5.0).
#include <algorithm>

#include "tc_common.cuh"

namespace sem3d {

namespace {

using namespace tcx;

__device__ __forceinline__ float to_f32(double x) { return f64_to_f32_rn(x); }
__device__ __forceinline__ float to_f32(float x) { return x; }

// Largest biased FP64 exponent of a block's values -> *emax.  The slot is read
// before the atomic: it stops growing after the first blocks, and an atomic
// per warp on one address cost 2-5 ms at n = 999.  Called by whole blocks.
__device__ __forceinline__ void block_max_exp(unsigned int m, int* emax) {
  __shared__ unsigned int top;
  if (threadIdx.x == 0) top = 0;
  __syncthreads();
  m = __reduce_max_sync(0xFFFFFFFFu, m);
  if ((threadIdx.x & 31) == 0 && m > top) atomicMax(&top, m);
  __syncthreads();
  if (threadIdx.x == 0 && (int)top > __ldcg(emax)) atomicMax(emax, (int)top);
}

__device__ __forceinline__ unsigned int exp_of(double x) {
  return (unsigned int)(__double_as_longlong(x) >> 52) & 0x7FFu;
}
__device__ __forceinline__ unsigned int exp_of(float) { return 0; }

// Right-hand sides whose largest biased FP64 exponent is at least this are scaled.
constexpr int kFoldBig = 1023 + 110;
constexpr float kFoldDown = 1.f / 256, kFoldUp = 256.f;

// FOLD_F: f, its largest exponent to *fexp; FOLD_BIG: f at kFoldDown if its
// exponent calls for it (else nothing); FOLD_R: a residual, scaled as f was.
enum : int { FOLD_F, FOLD_BIG, FOLD_R };

template <int WHAT, typename TIN>
__device__ __forceinline__ void fold_nodes(const TIN* __restrict__ in, int pitch, __nv_bfloat16* __restrict__ hi,
                                           __nv_bfloat16* __restrict__ lo, const FoldGeom& g, long long idx, float sc,
                                           unsigned int& m) {
  const unsigned int cp = (unsigned int)g.Pe >> 1;
  const int c = (int)(idx % cp);
  const long long jl = idx / cp;
  const int j = (int)(jl % g.ne[1]), l = (int)(jl / g.ne[1]);
  const bool my = j < g.no[1], mz = l < g.no[2];  // has a mirror image along y / z
  const int i0 = 2 * c;
  // the lines (j,l), (j',l), (j,l'), (j',l'): values at i and at its mirror
  // image (all loads issued before the conversions), then x-even / x-odd parts
  TIN ra[4][2], rb[4][2];
  float e[4][2], o[4][2];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const bool ok = (!(q & 1) || my) && (!(q & 2) || mz);
    const int jq = (q & 1) ? g.ny - 1 - j : j, lq = (q & 2) ? g.nz - 1 - l : l;
    const TIN* row = in + ((long long)lq * g.ny + jq) * pitch;
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      const int i = i0 + p;
      ra[q][p] = (ok && i < g.ne[0]) ? __ldg(row + i) : TIN(0);
      rb[q][p] = (ok && i < g.no[0]) ? __ldg(row + g.nx - 1 - i) : TIN(0);
    }
  }
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      if (WHAT == FOLD_F) m = max(m, max(exp_of(ra[q][p]), exp_of(rb[q][p])));
      float a = to_f32(ra[q][p]), b = to_f32(rb[q][p]);
      if (WHAT != FOLD_F) { a *= sc; b *= sc; }
      e[q][p] = a + b;
      o[q][p] = i0 + p < g.no[0] ? a - b : 0.f;
    }
#pragma unroll
  for (int x = 0; x < 2; ++x) {
    if (x == 1 && i0 >= g.Po) break;
    float v[4][2];  // (y even, z even), (y odd, z even), (y even, z odd), (y odd, z odd)
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      const float a0 = x ? o[0][p] : e[0][p], a1 = x ? o[1][p] : e[1][p];
      const float a2 = x ? o[2][p] : e[2][p], a3 = x ? o[3][p] : e[3][p];
      const float s0 = a0 + a1, d0 = a0 - a1, s1 = a2 + a3, d1 = a2 - a3;
      v[0][p] = s0 + s1; v[1][p] = d0 + d1; v[2][p] = s0 - s1; v[3][p] = d0 - d1;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (((q & 1) && !my) || ((q & 2) && !mz)) continue;
      const long long row = (long long)((q & 2) ? g.ne[2] + l : l) * g.ny + ((q & 1) ? g.ne[1] + j : j);
      const long long at = row * g.Px + (x ? g.Pe : 0) + i0;
      uint32_t h, w;
      split_pair(v[q][0], v[q][1], h, w);
      *reinterpret_cast<uint32_t*>(hi + at) = h;
      *reinterpret_cast<uint32_t*>(lo + at) = w;
    }
  }
}

template <int WHAT, typename TIN>
__global__ void __launch_bounds__(256) fold_split_kernel(const TIN* __restrict__ in, int pitch,
                                                         __nv_bfloat16* __restrict__ hi,
                                                         __nv_bfloat16* __restrict__ lo, FoldGeom g, int* fexp) {
  const long long total = (long long)((unsigned int)g.Pe >> 1) * g.ne[1] * g.ne[2];
  long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  unsigned int m = 0;
  if (WHAT == FOLD_BIG) {  // a few blocks
    if (*fexp < kFoldBig) return;
    for (; idx < total; idx += (long long)gridDim.x * blockDim.x)
      fold_nodes<WHAT>(in, pitch, hi, lo, g, idx, kFoldDown, m);
  } else {
    const float sc = WHAT == FOLD_R && __ldg(fexp) >= kFoldBig ? kFoldDown : 1.f;
    if (idx < total) fold_nodes<WHAT>(in, pitch, hi, lo, g, idx, sc, m);
    if (WHAT == FOLD_F) block_max_exp(m, fexp);
  }
}

// What the correction is added to.  DF_*: the solution as a double-FP32 pair
// at pitch PxDf (zero pads); LOZ: its low parts are zero, and read as such.
enum : int { UP_F64 = 0, UP_F64_ACC, UP_DF, UP_DF_ACC, UP_DF_ACC_LOZ, UP_DF_F64, UP_DF_F64_LOZ };

template <int MODE>
__global__ void __launch_bounds__(256) unfold_update_kernel(const float* __restrict__ delta, FoldGeom g, double* u,
                                                            float* dhi, float* dlo, int PxDf,
                                                            const int* __restrict__ fexp,
                                                            int* emax) {
  constexpr bool df = MODE >= UP_DF, reads = MODE != UP_F64 && MODE != UP_DF;
  constexpr bool loz = MODE == UP_DF_ACC_LOZ || MODE == UP_DF_F64_LOZ;
  const float up = __ldg(fexp) >= kFoldBig ? kFoldUp : 1.f;
  const long long total = (long long)g.Pe * g.ne[1] * g.ne[2];
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  unsigned int m = 0;
  if (idx < total) {
    const int i = (int)(idx % g.Pe);
    const long long jl = idx / g.Pe;
    const int j = (int)(jl % g.ne[1]), l = (int)(jl / g.ne[1]);
    const bool in = i < g.ne[0], mx = i < g.no[0], my = j < g.no[1], mz = l < g.no[2];
    // line q of the 4 mirror images along y and z; node 2q: i, node 2q+1: its mirror image along x
    bool ok[8];
    long long line[4];
    float v[8];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const bool ex = (!(q & 1) || my) && (!(q & 2) || mz);
      line[q] = (long long)((q & 2) ? g.nz - 1 - l : l) * g.ny + ((q & 1) ? g.ny - 1 - j : j);
      ok[2 * q] = ex && in;
      ok[2 * q + 1] = ex && mx;
      const long long src = ((long long)((q & 2) ? g.ne[2] + l : l) * g.ny + ((q & 1) ? g.ne[1] + j : j)) * g.Px;
      const float e = ok[2 * q] ? __ldg(delta + src + i) : 0.f;
      const float o = ok[2 * q + 1] ? __ldg(delta + src + g.Pe + i) : 0.f;
      v[2 * q] = e + o;
      v[2 * q + 1] = e - o;
    }
#pragma unroll
    for (int x = 0; x < 2; ++x) {
      const float a = v[x], b = v[2 + x], c = v[4 + x], d = v[6 + x];
      const float s0 = a + b, d0 = a - b, s1 = c + d, d1 = c - d;
      v[x] = s0 + s1; v[2 + x] = d0 + d1; v[4 + x] = s0 - s1; v[6 + x] = d0 - d1;
    }
    float oh[8], ol[8];
    double od[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int at = (q & 1) ? g.nx - 1 - i : i;
      if (reads && df) {
        oh[q] = ok[q] ? dhi[line[q >> 1] * PxDf + at] : 0.f;
        ol[q] = (ok[q] && !loz) ? dlo[line[q >> 1] * PxDf + at] : 0.f;
      } else if (reads) {
        od[q] = ok[q] ? u[line[q >> 1] * g.nx + at] : 0.0;
      }
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      if (!ok[q]) continue;
      v[q] *= up;  // here, where the reads above are on their way
      const int at = (q & 1) ? g.nx - 1 - i : i;
      const long long d = line[q >> 1] * PxDf + at, w = line[q >> 1] * g.nx + at;
      if (MODE == UP_F64 || MODE == UP_F64_ACC) {
        const double r = reads ? od[q] + f32_to_f64(v[q]) : f32_to_f64(v[q]);
        u[w] = r;
        m = max(m, exp_of(r));
      } else if (MODE == UP_DF) {
        dhi[d] = v[q];
        if (dlo) dlo[d] = 0.f;
      } else {
        // (oh + ol) + v: two-sum of the leading parts, then renormalise
        const float sum = oh[q] + v[q];
        const float bb = sum - oh[q];
        const float err = (oh[q] - (sum - bb)) + (v[q] - bb);
        const float t = ol[q] + err;
        const float nh = sum + t;
        const float nl = t - (nh - sum);
        if (MODE == UP_DF_ACC || MODE == UP_DF_ACC_LOZ) {
          dhi[d] = nh;
          dlo[d] = nl;
        } else {
          const double r = f32_to_f64(nh) + f32_to_f64(nl);
          u[w] = r;
          m = max(m, exp_of(r));
        }
      }
    }
    // the pad columns of the double-FP32 solution stay zero (the residual reads
    // them as boundary values)
    if ((MODE == UP_DF || MODE == UP_DF_ACC_LOZ) && g.nx + i < PxDf) {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        if (((q & 1) && !my) || ((q & 2) && !mz)) continue;
        if (MODE == UP_DF) dhi[line[q] * PxDf + g.nx + i] = 0.f;
        if (dlo) dlo[line[q] * PxDf + g.nx + i] = 0.f;
      }
    }
  }
  if (emax) block_max_exp(m, emax);
}

}  // namespace

FoldGeom fold_geom(const Geom& g) {
  FoldGeom f{};
  f.nx = g.nx; f.ny = g.ny; f.nz = g.nz;
  const int n3[3] = {g.nx, g.ny, g.nz};
  for (int a = 0; a < 3; ++a) { f.no[a] = n3[a] / 2; f.ne[a] = n3[a] - f.no[a]; }
  f.Pe = pad16(f.ne[0]);
  f.Po = pad16(f.no[0]);
  f.Px = f.Pe + f.Po;
  return f;
}

cudaError_t launch_fold(const FoldGeom& g, const double* f64, const float* f32, int pitch, TcBuffers out, int* fexp,
                        int num_sms, cudaStream_t s) {
  const long long total = (long long)(g.Pe / 2) * g.ne[1] * g.ne[2], blocks = (total + 255) / 256;
  if (blocks >= (1LL << 31)) return cudaErrorInvalidValue;
  const unsigned b = (unsigned)blocks, few = (unsigned)std::min<long long>(blocks, 8LL * num_sms);
  if (f32) {
    fold_split_kernel<FOLD_R><<<b, 256, 0, s>>>(f32, pitch, out.hi, out.lo, g, fexp);
    return cudaGetLastError();
  }
  const cudaError_t e = cudaMemsetAsync(fexp, 0, sizeof(int), s);
  if (e != cudaSuccess) return e;
  fold_split_kernel<FOLD_F><<<b, 256, 0, s>>>(f64, pitch, out.hi, out.lo, g, fexp);
  fold_split_kernel<FOLD_BIG><<<few, 256, 0, s>>>(f64, pitch, out.hi, out.lo, g, fexp);
  return cudaGetLastError();
}

cudaError_t launch_unfold(const FoldGeom& g, const float* delta, int epi, bool lo_zero, double* u, DfBuffers df,
                          int PxDf, const int* fexp, int* emax, cudaStream_t s) {
  const long long total = (long long)g.Pe * g.ne[1] * g.ne[2], blocks = (total + 255) / 256;
  if (blocks >= (1LL << 31)) return cudaErrorInvalidValue;
  const unsigned b = (unsigned)blocks;
  auto run = [&](auto kern) { kern<<<b, 256, 0, s>>>(delta, g, u, df.hi, df.lo, PxDf, fexp, emax); };
  switch (epi) {
    case EPI_STORE: run(unfold_update_kernel<UP_F64>); break;
    case EPI_ACCUM: run(unfold_update_kernel<UP_F64_ACC>); break;
    case EPI_DF_STORE: run(unfold_update_kernel<UP_DF>); break;
    case EPI_DF_ACCUM: lo_zero ? run(unfold_update_kernel<UP_DF_ACC_LOZ>) : run(unfold_update_kernel<UP_DF_ACC>); break;
    case EPI_DF_ACCUM_F64: lo_zero ? run(unfold_update_kernel<UP_DF_F64_LOZ>) : run(unfold_update_kernel<UP_DF_F64>); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

}  // namespace sem3d
