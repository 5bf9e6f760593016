// Refinement residual r = f - (c + H_x (+) H_y (+) H_z) u (Eq. 12) in
// double-FP32 arithmetic: u = uh + ul and the rows of H = ch + cl are pairs of
// FP32 numbers (about 48 significant bits; EXACT, where every residual of a
// solve is in this arithmetic: with a third FP32 term, which makes the rows
// exact).  Products use the FMA error-free transformation, sums the two-sum of
// the leading parts.  FP32 runs at ~70x the FP64 rate on this GPU, so a
// refinement sweep whose only job is to bring the error down to what the
// final FP64-accurate sweep removes can use it.
//
// Two kernels, both bound by their FP32 operations (12 a term, k + 2 terms per
// axis and node, beside 20 bytes of HBM per node):
//  - k in {1, 2, 4}: a warp per line, a lane per 4 nodes, whose x rows are known
//    at compile time because 4 % k == 0 (stencil_df4_kernel); the nodes in pairs
//    in packed f32x2 instructions and the loads of a row's lines together:
//    n = 255, k = 4 178 -> 157 us with u's low half zero, 194 -> 180 else;
//  - other k: blocks of 8 lines x 64 nodes marching along z (stencil_df_kernel).
//    Every plane is staged once in shared memory (cp.async, two planes ahead),
//    adds its z terms to the running sums of its element's k + 1 planes, and
//    serves its own y and x terms; two nodes per lane in packed f32x2
//    instructions (124 lanes per clock and SM, as scalar ones, for half the
//    issue slots).  A lane's x row is not known at compile time: all 2k + 1
//    offsets enter, with zeros outside the node's band.  A thread per element
//    and line, which this replaces, read its neighbours at a stride of k and
//    waited on L1: 449x320x383, k = 3 1.02 -> 0.60 ms; 383^3, k = 6 1.16 -> 0.88.
//    At k = 4 it takes 11.7 ms at n = 999, more than the vector kernel.
// Tried: summing onto an offset that dominates every term, so that a fast
// two-sum suffices (6 operations a term, n = 999 8.2 ms): its noise, relative to
// the largest sum on the grid, is some 80 times the two-sum's and took the
// normwise backward error of the refined solution from 2.5e-16 to 1.1e-15.
#include "sem3d_internal.h"

namespace sem3d {

namespace {

typedef unsigned long long f2;  // two FP32 numbers

__device__ __forceinline__ f2 pack2(float a, float b) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(f2 v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ f2 as2(const float2& v) { return *reinterpret_cast<const f2*>(&v); }
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 sub2(f2 a, f2 b) {
  f2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
// -a as a multiply-add: a sign flip is two integer instructions
__device__ __forceinline__ f2 neg2(f2 a) { return fma2(a, 0xBF800000BF800000ull, 0x8000000080000000ull); }

// Exact split of an FP64 value into hi (first 24 significant bits, truncated)
// and lo (the next 24, rounded) with integer operations only.  |x| < 2^-126
// gives (0, 0); 2^-126 <= |x| < 2^-74 gives lo = 0; Inf and NaN give NaN.
__device__ __forceinline__ void f64_to_df(double x, float& hi, float& lo) {
  const unsigned int h = (unsigned int)__double2hiint(x), w = (unsigned int)__double2loint(x);
  const unsigned int sign = h & 0x80000000u, ex = (h >> 20) & 0x7FFu;
  // rebiased exponent and leading 23 fraction bits (the bits shifted out drop out of the difference)
  const unsigned int m = __funnelshift_l(w, h, 3) - (896u << 23);
  const float scale = __uint_as_float(((m & 0x7F800000u) - (52u << 23)));
  hi = __uint_as_float(ex < 897u ? sign : ex > 1150u ? 0x7FC00000u : sign | m);
  lo = ex < 949u ? 0.f : __uint_as_float(__float_as_uint(__uint2float_rn(w & 0x1FFFFFFFu) * scale) | sign);
}

// The negated rows of H per axis and local index q, entry q (2k+1) + d + k, as
// FP32 terms; a kernel parameter.
template <int K>
struct DfCoef {
  float h[K * (2 * K + 1)], l[K * (2 * K + 1)], l2[K * (2 * K + 1)];  // x
  float2 yh[K * (2 * K + 1)], yl[K * (2 * K + 1)], yl2[K * (2 * K + 1)];  // y and z: each twice, for
  float2 zh[K * (2 * K + 1)], zl[K * (2 * K + 1)], zl2[K * (2 * K + 1)];  // the packed operations
};

struct DfArgs {
  const float* uh;
  const float* ul;
  const double* f;
  __nv_bfloat16* hi;
  __nv_bfloat16* lo;
  float* out32;        // if set: FP32 residual at pitch Px; with st, max |r| -> its slot 0
  F16State* st;
  int nx, ny, nz, Px;
  int seg;             // z elements per block
};

// One term of the running sum: (S, Sl) += (nh + nl [+ nl2]) (uh + ul).
template <bool EXACT, bool LO0>
__device__ __forceinline__ void df_term(f2& S, f2& Sl, f2 nh, f2 nl, f2 nl2, f2 uh, f2 ul) {
  const f2 p = mul2(nh, uh);
  f2 t = fma2(nh, uh, neg2(p));
  if (EXACT) t = fma2(nl2, uh, t);
  t = fma2(nl, uh, t);
  if (!LO0) t = fma2(nh, ul, t);
  const f2 s = add2(S, p);
  const f2 bb = sub2(s, S);
  const f2 err = add2(sub2(S, sub2(s, bb)), sub2(p, bb));
  S = s;
  Sl = add2(Sl, add2(err, t));
}

constexpr int DF_LINES = 8, DF_NODES = 64, DF_STAGES = 3;  // block tile: lines x nodes per line; planes in flight

// Staged part of a plane: the block's lines and k more on either side, 4 or 8
// more nodes at either end of a line (16-byte copies; zero outside the grid).
template <int K>
struct DfTile {
  static constexpr int HX = K <= 4 ? 4 : 8, LW = DF_NODES + 2 * HX, NL = DF_LINES + 2 * K;
  static constexpr int FLOATS = NL * LW;
  // a stage: hi [, lo] of the tile, then f of the block's own lines
  static constexpr int F_BYTES = DF_LINES * DF_NODES * 8;
  __host__ __device__ static constexpr int stage_bytes(bool lo0) { return (lo0 ? 1 : 2) * FLOATS * 4 + F_BYTES; }
};

__device__ __forceinline__ void cp_async8(double* dst, const double* src, bool in) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src),
               "r"(in ? 8 : 0)
               : "memory");
}
__device__ __forceinline__ void cp_async16(float* dst, const float* src, bool in) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src),
               "r"(in ? 16 : 0)
               : "memory");
}

template <int K, bool EXACT, bool LO0>
__global__ void __launch_bounds__(256, K <= 6 ? 3 : 2) stencil_df_kernel(DfArgs a, const __grid_constant__ DfCoef<K> cf) {
  using T = DfTile<K>;
  constexpr int BW = 2 * K + 1;
  constexpr int PM = (K + 1) / 2;            // aligned pairs on either side of a lane's pair along x
  constexpr int STAGE = T::stage_bytes(LO0);
  extern __shared__ __align__(16) unsigned char tiles[];  // [stage]: hi, lo [NL][LW], f [lines][nodes]
  __shared__ float2 xh[BW][K], xl[BW][K], xl2[EXACT ? BW : 1][EXACT ? K : 1];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int x0 = blockIdx.x * DF_NODES, j0 = blockIdx.y * DF_LINES;
  const int i0 = x0 + 2 * lane, j = j0 + warp;
  for (int e = threadIdx.x; e < BW * K; e += 256) {  // x rows of the pair (i, i+1) whose first node has local index q
    const int d = e / K, q = e % K, q1 = (q + 1) % K;
    xh[d][q] = make_float2(cf.h[q * BW + d], cf.h[q1 * BW + d]);
    xl[d][q] = make_float2(cf.l[q * BW + d], cf.l[q1 * BW + d]);
    if (EXACT) xl2[d][q] = make_float2(cf.l2[q * BW + d], cf.l2[q1 * BW + d]);
  }
  const long long plane = (long long)a.ny * a.Px;
  const int nez = (a.nz + 1) / K;
  const int e0 = blockIdx.z * a.seg, e1 = min(e0 + a.seg, nez);
  // Planes are numbered by their global node g = l + 1; this block stages the
  // planes g0 .. g1 (boundary planes 0 and nz + 1 come in as zeros).
  const int g0 = e0 * K, g1 = e1 * K;
  constexpr int CHUNKS = T::NL * (T::LW / 4), PER = (CHUNKS + 255) / 256;  // 16-byte copies per plane and thread
  int src[PER], dst[PER];  // offsets in a plane (-1: outside) and in a staged plane (-1: none)
#pragma unroll
  for (int n = 0; n < PER; ++n) {
    const int c = threadIdx.x + n * 256, r = c / (T::LW / 4), q = c - r * (T::LW / 4);
    const int jr = j0 - K + r, x = x0 - T::HX + 4 * q;
    dst[n] = c < CHUNKS ? r * T::LW + 4 * q : -1;
    src[n] = jr >= 0 && jr < a.ny && x >= 0 && x < a.Px ? jr * a.Px + x : -1;
  }
  auto stage_plane = [&](int g) {
    if (g <= g1) {
      float* t = reinterpret_cast<float*>(tiles + ((g - g0) % DF_STAGES) * STAGE);
      const bool inz = g >= 1 && g <= a.nz;
      const long long at = inz ? (g - 1) * plane : 0;
#pragma unroll
      for (int n = 0; n < PER; ++n) {
        if (dst[n] < 0) continue;
        const bool in = inz && src[n] >= 0;
        const long long from = at + (in ? src[n] : 0);
        cp_async16(t + dst[n], a.uh + from, in);
        if (!LO0) cp_async16(t + T::FLOATS + dst[n], a.ul + from, in);
      }
      double* tf = reinterpret_cast<double*>(t + (LO0 ? 1 : 2) * T::FLOATS) + warp * DF_NODES + lane;
#pragma unroll
      for (int n = 0; n < 2; ++n) {
        const bool in = inz && j < a.ny && x0 + lane + 32 * n < a.nx;
        cp_async8(tf + 32 * n, in ? a.f + ((long long)(g - 1) * a.ny + j) * a.nx + x0 + lane + 32 * n : a.f, in);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  float rmax = 0.f;
  const bool active = j < a.ny && i0 < a.Px;  // inactive threads only stage
  const int qx = (i0 + 1) % K, qy = (j + 1) % K;
  const long long col = (long long)j * a.Px + i0;
  auto zterm = [&](f2& S, f2& Sl, int q, int d, f2 uh, f2 ul) {  // z row of local index q, offset d (compile time)
    const int c = q * BW + d + K;
    df_term<EXACT, LO0>(S, Sl, as2(cf.zh[c]), as2(cf.zl[c]), EXACT ? as2(cf.zl2[c]) : 0ull, uh, ul);
  };
  // x and y terms of the staged plane g for this lane's two nodes; ch, cl: their values
  auto xy_terms = [&](int g, f2& S, f2& Sl, f2& uh, f2& ul) {
    const float* th = reinterpret_cast<const float*>(tiles + ((g - g0) % DF_STAGES) * STAGE) + (warp + K) * T::LW +
                      T::HX + 2 * lane;
    const float* tl = th + T::FLOATS;
    auto lds = [](const float* p) { return *reinterpret_cast<const f2*>(p); };
    uh = lds(th);
    ul = LO0 ? 0ull : lds(tl);
    // y: the element's lines (at a vertex line the element above's, then the
    // one below's); lines outside the grid are staged as zeros
    auto yterm = [&](int d, const float* h, const float* l, int c) {
      df_term<EXACT, LO0>(S, Sl, as2(cf.yh[c]), as2(cf.yl[c]), EXACT ? as2(cf.yl2[c]) : 0ull, lds(h + d * T::LW),
                          LO0 ? 0ull : lds(l + d * T::LW));
    };
    {
      const float *h = th - qy * T::LW, *l = tl - qy * T::LW;
      const int c = qy * BW + K - qy;
#pragma unroll
      for (int t = 0; t <= K; ++t) yterm(t, h, l, c + t);
      if (qy == 0) {
#pragma unroll
        for (int t = -K; t < 0; ++t) yterm(t, th, tl, t + K);
      }
    }
    // x: aligned pairs around the lane's own; an odd offset takes one value of each of two
    f2 ph[2 * PM + 1], pl[LO0 ? 1 : 2 * PM + 1];
#pragma unroll
    for (int m = -PM; m <= PM; ++m) {
      ph[PM + m] = m == 0 ? uh : lds(th + 2 * m);
      if (!LO0) pl[PM + m] = m == 0 ? ul : lds(tl + 2 * m);
    }
    auto shifted = [&](const f2* p, int d) -> f2 {  // values at d, d + 1
      if (((d + 2 * PM) & 1) == 0) return p[(d + 2 * PM) / 2];
      float a0, a1, b0, b1;
      unpack2(p[(d + 2 * PM) / 2], a0, a1);
      unpack2(p[(d + 2 * PM) / 2 + 1], b0, b1);
      return pack2(a1, b0);
    };
#pragma unroll
    for (int d = -K; d <= K; ++d) {
      const f2 ch = as2(xh[d + K][qx]), cl = as2(xl[d + K][qx]);
      const f2 cl2 = EXACT ? as2(xl2[EXACT ? d + K : 0][EXACT ? qx : 0]) : 0ull;
      df_term<EXACT, LO0>(S, Sl, ch, cl, cl2, shifted(ph, d), LO0 ? 0ull : shifted(pl, d));
    }
  };
  // f of plane l: high parts kept for the end, low parts into Sl
  const bool in0 = i0 < a.nx, in1 = i0 + 1 < a.nx;
  auto take_f = [&](int g, f2& fh, f2& Sl) {
    const unsigned char* t = tiles + ((g - g0) % DF_STAGES) * STAGE + (STAGE - T::F_BYTES);
    const double2 v = reinterpret_cast<const double2*>(t)[warp * (DF_NODES / 2) + lane];
    float h0, l0, h1, l1;
    f64_to_df(v.x, h0, l0);
    f64_to_df(v.y, h1, l1);
    fh = pack2(h0, h1);
    Sl = add2(Sl, pack2(l0, l1));
  };
  auto finish = [&](int l, f2 fh, f2 S, f2 Sl) {  // r = f + S + Sl
    const f2 s = add2(fh, S);
    const f2 bb = sub2(s, fh);
    const f2 err = add2(sub2(fh, sub2(s, bb)), sub2(S, bb));
    float r0, r1;
    unpack2(add2(s, add2(err, Sl)), r0, r1);
    r0 = in0 ? r0 : 0.f;  // pads stay zero
    r1 = in1 ? r1 : 0.f;
    const long long row = l * plane + col;
    if (a.out32) {
      *reinterpret_cast<float2*>(a.out32 + row) = make_float2(r0, r1);
      rmax = fmaxf(rmax, fmaxf(fabsf(r0), fabsf(r1)));
    } else {
      const __nv_bfloat16 h0 = __float2bfloat16_rn(r0), h1 = __float2bfloat16_rn(r1);
      const __nv_bfloat16 l0 = __float2bfloat16_rn(r0 - __bfloat162float(h0));
      const __nv_bfloat16 l1 = __float2bfloat16_rn(r1 - __bfloat162float(h1));
      *reinterpret_cast<__nv_bfloat162*>(a.hi + row) = __nv_bfloat162(h0, h1);
      *reinterpret_cast<__nv_bfloat162*>(a.lo + row) = __nv_bfloat162(l0, l1);
    }
  };
  // Sums of an element's planes t = 0 .. K (its two vertices and the nodes
  // between); every plane adds its z terms to all of them when it arrives.
  f2 S[K + 1], Sl[K + 1], F[K + 1], vh = 0ull, vl = 0ull;  // vh, vl: this lane's nodes in the element's left vertex plane
  stage_plane(g0);
  stage_plane(g0 + 1);
  // Wait for plane g, stage g + 2 into the buffer that g - 1 was read from.
  auto next_plane = [&](int g) {
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();
    stage_plane(g + 2);
  };
  // The segment's first vertex plane: the element before it adds its z terms
  S[K] = 0ull;
  Sl[K] = 0ull;
  if (active) {
#pragma unroll
    for (int t = 0; t < K; ++t) {
      const int g = g0 - K + t;
      if (g < 1) continue;
      const f2 uh = __ldg(reinterpret_cast<const f2*>(a.uh + (g - 1) * plane + col));
      const f2 ul = LO0 ? 0ull : __ldg(reinterpret_cast<const f2*>(a.ul + (g - 1) * plane + col));
      zterm(S[K], Sl[K], 0, t - K, uh, ul);
    }
  }
  next_plane(g0);
  F[K] = 0ull;
  if (active && g0 >= 1) {
    take_f(g0, F[K], Sl[K]);
    xy_terms(g0, S[K], Sl[K], vh, vl);
    zterm(S[K], Sl[K], 0, 0, vh, vl);
  }
#pragma unroll 1
  for (int e = e0; e < e1; ++e) {
    S[0] = S[K];
    Sl[0] = Sl[K];
    F[0] = F[K];
    // the left vertex's terms in the element's other planes
#pragma unroll
    for (int t = 1; t <= K; ++t) {
      S[t] = 0ull;
      Sl[t] = 0ull;
      zterm(S[t], Sl[t], t % K, -t, vh, vl);
    }
#pragma unroll
    for (int t = 1; t <= K; ++t) {
      const int g = e * K + t;
      next_plane(g);
      F[t] = 0ull;
      if (active && g <= a.nz) {
        take_f(g, F[t], Sl[t]);
        xy_terms(g, S[t], Sl[t], vh, vl);
#pragma unroll
        for (int u = 0; u <= K; ++u) zterm(S[u], Sl[u], u % K, t - u, vh, vl);
      }
    }
    if (active) {
#pragma unroll
      for (int t = 0; t < K; ++t)
        if (e * K + t >= 1) finish(e * K + t - 1, F[t], S[t], Sl[t]);
    }
  }
  if (a.out32 && a.st) {
    __syncwarp();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) rmax = fmaxf(rmax, __shfl_xor_sync(0xFFFFFFFFu, rmax, o));
    if (lane == 0 && rmax > 0.f) atomicMax(&a.st->maxbits[0], __float_as_uint(rmax));
  }
}

// Launch one instantiation; its shared memory may exceed the default limit.
template <int K, bool EXACT, bool LO0>
cudaError_t run_df(const DfArgs& a, const DfCoef<K>& cf, dim3 grid, cudaStream_t s) {
  auto kern = stencil_df_kernel<K, EXACT, LO0>;
  constexpr int smem = DF_STAGES * DfTile<K>::stage_bytes(LO0);
  if (smem > 40 * 1024) {
    static PerDevice ready;
    const cudaError_t e = on_device(ready, [&](int& set) {
      set = 1;
      return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    });
    if (e != cudaSuccess) return e;
  }
  kern<<<grid, 256, smem, s>>>(a, cf);
  return cudaGetLastError();
}

template <int K>
cudaError_t launch_df(DfArgs a, const DevAxis* ax, bool exact, bool lo_zero, int num_sms, cudaStream_t s) {
  DfCoef<K> cf{};
  for (int w = 0; w < 3; ++w)
    for (int e = 0; e < K * (2 * K + 1); ++e) {
      const float h = -ax[w].Hq_hi_host[e], l = -ax[w].Hq_lo_host[e], l2 = -ax[w].Hq_lo2_host[e];
      if (w == 0) { cf.h[e] = h; cf.l[e] = l; cf.l2[e] = l2; }
      if (w == 1) { cf.yh[e] = make_float2(h, h); cf.yl[e] = make_float2(l, l); cf.yl2[e] = make_float2(l2, l2); }
      if (w == 2) { cf.zh[e] = make_float2(h, h); cf.zl[e] = make_float2(l, l); cf.zl2[e] = make_float2(l2, l2); }
    }
  // Blocks of 8 lines x 64 nodes marching over `seg` z elements: long enough
  // that the k planes read ahead of a segment cost little, short enough for a
  // few blocks per SM.
  const int nez = (a.nz + 1) / K;
  const long long tiles = (long long)((a.Px + DF_NODES - 1) / DF_NODES) * ((a.ny + DF_LINES - 1) / DF_LINES);
  const long long want = (8LL * num_sms + tiles - 1) / tiles;  // segments
  int seg = (int)((nez + want - 1) / want);
  seg = seg < 1 ? 1 : seg > 16 ? 16 : seg;
  if ((nez + seg - 1) / seg > 65535) seg = (nez + 65534) / 65535;
  a.seg = seg;
  const dim3 grid((unsigned)((a.Px + DF_NODES - 1) / DF_NODES), (unsigned)((a.ny + DF_LINES - 1) / DF_LINES),
                  (unsigned)((nez + seg - 1) / seg));
  if (grid.y > 65535) return cudaErrorInvalidValue;
  if (exact) return lo_zero ? run_df<K, true, true>(a, cf, grid, s) : run_df<K, true, false>(a, cf, grid, s);
  return lo_zero ? run_df<K, false, true>(a, cf, grid, s) : run_df<K, false, false>(a, cf, grid, s);
}

// One term of one node's running sum: (S, Sl) += (nh + nl [+ nl2]) (uh + ul),
// dropping nl ul and nl2 ul; the third coefficient term enters only when EXACT
// (else the 48-bit nh + nl).  LO0: ul is zero (the solution right after the
// first solve), and nh ul, exactly 0 there, is not formed (the same result).
template <bool EXACT, bool LO0>
__device__ __forceinline__ void df_add_prod(float& S, float& Sl, float nh, float nl, float uh, float ul, float nl2) {
  const float p = nh * uh;
  float t = fmaf(nh, uh, -p);
  if (EXACT) t = fmaf(nl2, uh, t);
  t = fmaf(nl, uh, t);
  if (!LO0) t = fmaf(nh, ul, t);
  const float s = S + p;
  const float bb = s - S;
  const float err = (S - (s - bb)) + (p - bb);
  S = s;
  Sl = Sl + (err + t);
}

// Negated rows of H for the vector residual (k <= 4), as kernel parameters.
// x: entry [P][m] holds what node m of a lane's 12-node window contributes to
// the lane's nodes 2P and 2P + 1 (read at compile-time offsets); y and z: the
// rows per local index, each entry twice (read at warp-uniform offsets).
struct Df4Coef {
  float2 xh[2][12], xl[2][12], xl2[2][12];     // l2: third terms (used when EXACT)
  float2 h[2][4 * 9], l[2][4 * 9], l2[2][4 * 9];
};

// Window nodes (4 + p + d) in the band of the row at position p of a lane's 4.
__host__ __device__ constexpr int df4_lo(int K, int p) { return 4 + p - ((p + 1) % K == 0 ? K : (p + 1) % K); }
__host__ __device__ constexpr int df4_hi(int K, int p) { return 4 + p + K - (p + 1) % K; }

// Double-FP32 residual for k in {1, 2, 4}.  A lane handles the 4 consecutive
// nodes i = 4c .. 4c+3 of one (j, l) line -- one float4 of each of u_hi and
// u_lo, whose rows (pitch Px, a multiple of 16) are 16-byte aligned and whose
// pad columns are zero -- and a warp handles one line, its lanes striding over
// the line's Px/4 chunks.  Since 4 % k == 0, node 4c+p has the local index
// (p+1) % k for every c: each position's x row of H is known at compile time
// and only its band is summed.  The y and z rows depend on the warp's (j, l).
template <int K, bool EXACT, bool LO0>
__global__ void __launch_bounds__(256, 4) stencil_df4_kernel(DfArgs a, const __grid_constant__ Df4Coef cf) {
  constexpr int BW = 2 * K + 1;
  const int lane = threadIdx.x & 31;
  const long long lines = (long long)a.ny * a.nz;
  const int chunks = a.Px >> 2;
  const long long splane = (long long)a.ny * chunks;  // float4 per z-plane
  const float4* UH = reinterpret_cast<const float4*>(a.uh);
  const float4* UL = reinterpret_cast<const float4*>(a.ul);
  float rmax = 0.f;
  for (long long line = (long long)blockIdx.x * 8 + (threadIdx.x >> 5); line < lines;
       line += (long long)gridDim.x * 8) {  // warp-uniform
    const int j = (int)(line % a.ny), l = (int)(line / a.ny);
    const int qy = (j + 1) % K, qz = (l + 1) % K;
    const long long row4 = line * chunks;
    const double* frow = a.f + line * a.nx;
    for (int c = lane; c < chunks; c += 32) {
      const int i0 = 4 * c;
      f2 S[2], Sl[2];  // running sums of the node pairs (0, 1) and (2, 3)
#pragma unroll
      for (int P = 0; P < 2; ++P) {
        float h[2] = {0.f, 0.f}, l[2] = {0.f, 0.f};
#pragma unroll
        for (int e = 0; e < 2; ++e)
          if (i0 + 2 * P + e < a.nx) f64_to_df(__ldg(frow + i0 + 2 * P + e), h[e], l[e]);
        S[P] = pack2(h[0], h[1]);
        Sl[P] = pack2(l[0], l[1]);
      }
      // x: nodes i0-4 .. i0+7 (the neighbouring chunks; zero outside the line)
      float wh[12], wl[12];
      {
        const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 ph = c > 0 ? __ldg(UH + row4 + c - 1) : z4, pl = (c > 0 && !LO0) ? __ldg(UL + row4 + c - 1) : z4;
        const float4 ch = __ldg(UH + row4 + c), cl = LO0 ? z4 : __ldg(UL + row4 + c);
        const float4 nh = c + 1 < chunks ? __ldg(UH + row4 + c + 1) : z4;
        const float4 nl = (c + 1 < chunks && !LO0) ? __ldg(UL + row4 + c + 1) : z4;
        wh[0] = ph.x; wh[1] = ph.y; wh[2] = ph.z; wh[3] = ph.w; wh[4] = ch.x; wh[5] = ch.y;
        wh[6] = ch.z; wh[7] = ch.w; wh[8] = nh.x; wh[9] = nh.y; wh[10] = nh.z; wh[11] = nh.w;
        wl[0] = pl.x; wl[1] = pl.y; wl[2] = pl.z; wl[3] = pl.w; wl[4] = cl.x; wl[5] = cl.y;
        wl[6] = cl.z; wl[7] = cl.w; wl[8] = nl.x; wl[9] = nl.y; wl[10] = nl.z; wl[11] = nl.w;
      }
#pragma unroll
      for (int m = 0; m < 12; ++m) {
#pragma unroll
        for (int P = 0; P < 2; ++P) {
          const bool in0 = m >= df4_lo(K, 2 * P) && m <= df4_hi(K, 2 * P);  // compile-time after unrolling
          const bool in1 = m >= df4_lo(K, 2 * P + 1) && m <= df4_hi(K, 2 * P + 1);
          const float2 nh = cf.xh[P][m], nl = cf.xl[P][m], n2 = EXACT ? cf.xl2[P][m] : make_float2(0.f, 0.f);
          if (in0 && in1) {
            df_term<EXACT, LO0>(S[P], Sl[P], as2(nh), as2(nl), as2(n2), pack2(wh[m], wh[m]),
                                LO0 ? 0ull : pack2(wl[m], wl[m]));
          } else if (in0 || in1) {
            float s0, s1, l0, l1;
            unpack2(S[P], s0, s1);
            unpack2(Sl[P], l0, l1);
            if (in0) df_add_prod<EXACT, LO0>(s0, l0, nh.x, nl.x, wh[m], wl[m], n2.x);
            else df_add_prod<EXACT, LO0>(s1, l1, nh.y, nl.y, wh[m], wl[m], n2.y);
            S[P] = pack2(s0, s1);
            Sl[P] = pack2(l0, l1);
          }
        }
      }
      // y and z: the rows of the neighbouring lines, in order of their offset: at
      // a vertex (q = 0) the k before it, then the k + 1 of the element.  The
      // latter's loads depend on no branch and go out together, lines outside
      // the grid counting as zeros, except where both halves of five lines
      // would not fit the registers (n = 511, k = 4: 1.37 ms with a branch at
      // every offset, 1.43 without; with one half 1.23 and 1.17).
      auto rows = [&](int w, int q, int pos, int n, long long pitch) {
        auto load = [&](const float4* U, int d) {
          return pos + d >= 0 && pos + d < n ? __ldg(reinterpret_cast<const ulonglong2*>(U + row4 + d * pitch + c))
                                             : make_ulonglong2(0, 0);
        };
        auto term = [&](int at, ulonglong2 vh, ulonglong2 vl) {
          const f2 nh = as2(cf.h[w][at]), nl = as2(cf.l[w][at]), n2 = EXACT ? as2(cf.l2[w][at]) : 0ull;
          df_term<EXACT, LO0>(S[0], Sl[0], nh, nl, n2, vh.x, vl.x);
          df_term<EXACT, LO0>(S[1], Sl[1], nh, nl, n2, vh.y, vl.y);
        };
        if constexpr (K == 4 && !LO0) {
#pragma unroll
          for (int d = -K; d <= K; ++d) {  // warp-uniform conditions
            if (d < (q == 0 ? -K : -q) || d > (q == 0 ? K : K - q) || pos + d < 0 || pos + d >= n) continue;
            term(q * BW + d + K, load(UH, d), load(UL, d));
          }
        } else {
          if (q == 0) {  // warp-uniform
#pragma unroll
            for (int d = -K; d < 0; ++d) term(d + K, load(UH, d), LO0 ? make_ulonglong2(0, 0) : load(UL, d));
          }
#pragma unroll
          for (int t = 0; t <= K; ++t)
            term(q * (BW - 1) + K + t, load(UH, t - q), LO0 ? make_ulonglong2(0, 0) : load(UL, t - q));
        }
      };
      rows(0, qy, j, a.ny, chunks);
      rows(1, qz, l, a.nz, splane);
      float ah[4], al[4];
      unpack2(S[0], ah[0], ah[1]);
      unpack2(S[1], ah[2], ah[3]);
      unpack2(Sl[0], al[0], al[1]);
      unpack2(Sl[1], al[2], al[3]);
      float r[4];
#pragma unroll
      for (int p = 0; p < 4; ++p) r[p] = (i0 + p < a.nx) ? ah[p] + al[p] : 0.f;  // pads stay zero
      const long long o = line * a.Px + i0;
      if (a.out32) {
        *reinterpret_cast<float4*>(a.out32 + o) = make_float4(r[0], r[1], r[2], r[3]);
#pragma unroll
        for (int p = 0; p < 4; ++p) rmax = fmaxf(rmax, fabsf(r[p]));
      } else {
        uint32_t hw[2], lw[2];
#pragma unroll
        for (int p = 0; p < 4; p += 2) {
          const __nv_bfloat16 h0 = __float2bfloat16_rn(r[p]), h1 = __float2bfloat16_rn(r[p + 1]);
          const __nv_bfloat16 l0 = __float2bfloat16_rn(r[p] - __bfloat162float(h0));
          const __nv_bfloat16 l1 = __float2bfloat16_rn(r[p + 1] - __bfloat162float(h1));
          hw[p / 2] = (uint32_t)__bfloat16_as_ushort(h0) | ((uint32_t)__bfloat16_as_ushort(h1) << 16);
          lw[p / 2] = (uint32_t)__bfloat16_as_ushort(l0) | ((uint32_t)__bfloat16_as_ushort(l1) << 16);
        }
        *reinterpret_cast<uint2*>(a.hi + o) = make_uint2(hw[0], hw[1]);
        *reinterpret_cast<uint2*>(a.lo + o) = make_uint2(lw[0], lw[1]);
      }
    }
  }
  if (a.out32 && a.st) {  // every lane of the warp gets here
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) rmax = fmaxf(rmax, __shfl_xor_sync(0xFFFFFFFFu, rmax, o));
    if ((threadIdx.x & 31) == 0 && rmax > 0.f) atomicMax(&a.st->maxbits[0], __float_as_uint(rmax));
  }
}

template <int K>
cudaError_t launch_df4(const DfArgs& a, const DevAxis* ax, bool exact, bool lo_zero, cudaStream_t s) {
  Df4Coef cf{};
  constexpr int BW = 2 * K + 1;
  for (int m = 0; m < 12; ++m)
    for (int p = 0; p < 4; ++p) {
      if (m < df4_lo(K, p) || m > df4_hi(K, p)) continue;
      const int e = (p + 1) % K * BW + m - 4 - p + K;
      const float h = -ax[0].Hq_hi_host[e], l = -ax[0].Hq_lo_host[e], l2 = -ax[0].Hq_lo2_host[e];
      float2 *ph = &cf.xh[p / 2][m], *pl = &cf.xl[p / 2][m], *p2 = &cf.xl2[p / 2][m];
      if (p % 2 == 0) { ph->x = h; pl->x = l; p2->x = l2; }
      else { ph->y = h; pl->y = l; p2->y = l2; }
    }
  for (int w = 0; w < 2; ++w)
    for (int e = 0; e < K * BW; ++e) {
      const float h = -ax[w + 1].Hq_hi_host[e], l = -ax[w + 1].Hq_lo_host[e], l2 = -ax[w + 1].Hq_lo2_host[e];
      cf.h[w][e] = make_float2(h, h);
      cf.l[w][e] = make_float2(l, l);
      cf.l2[w][e] = make_float2(l2, l2);
    }
  // One block per 8 consecutive lines and no grid stride: the resident blocks
  // then sweep the grid plane by plane, so the rows 1..K planes away that a
  // warp reads were read moments earlier by other warps and are still in L2.
  const long long lines = (long long)a.ny * a.nz;
  long long blocks = (lines + 7) / 8;
  if (blocks > 0x7FFFFFFFLL) blocks = 0x7FFFFFFFLL;
  const unsigned g = (unsigned)(blocks < 1 ? 1 : blocks);
  if (exact) {
    if (lo_zero) stencil_df4_kernel<K, true, true><<<g, 256, 0, s>>>(a, cf);
    else stencil_df4_kernel<K, true, false><<<g, 256, 0, s>>>(a, cf);
  } else {
    if (lo_zero) stencil_df4_kernel<K, false, true><<<g, 256, 0, s>>>(a, cf);
    else stencil_df4_kernel<K, false, false><<<g, 256, 0, s>>>(a, cf);
  }
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_stencil_df(const Geom& g, int k, const DevAxis* ax, DfBuffers u, const double* f,
                              __nv_bfloat16* out_hi, __nv_bfloat16* out_lo, int num_sms, cudaStream_t s, float* out32,
                              F16State* st, bool exact_coef, bool lo_zero) {
  if (g.bc != 0) return cudaErrorInvalidValue;  // element-pattern rows (Dirichlet) only
  DfArgs a{};
  a.uh = u.hi; a.ul = u.lo; a.f = f; a.hi = out_hi; a.lo = out_lo;
  a.out32 = out32; a.st = st;
  a.nx = g.nx; a.ny = g.ny; a.nz = g.nz; a.Px = g.Px;
  switch (k) {
    case 1: return launch_df4<1>(a, ax, exact_coef, lo_zero, s);
    case 2: return launch_df4<2>(a, ax, exact_coef, lo_zero, s);
    case 4: return launch_df4<4>(a, ax, exact_coef, lo_zero, s);
    case 3: return launch_df<3>(a, ax, exact_coef, lo_zero, num_sms, s);
    case 5: return launch_df<5>(a, ax, exact_coef, lo_zero, num_sms, s);
    case 6: return launch_df<6>(a, ax, exact_coef, lo_zero, num_sms, s);
    case 7: return launch_df<7>(a, ax, exact_coef, lo_zero, num_sms, s);
    case 8: return launch_df<8>(a, ax, exact_coef, lo_zero, num_sms, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace sem3d
