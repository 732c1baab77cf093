// gp_argle.cuh -- the flows of the imaginary-time preparation, and its float32 steps.
//
// Between two steps the field is phi(kx, ky, z) (with NV = 3 also d_z phi in that form): a step is
//   y   inverse transforms of phi and of i k~_y phi (and of d_z phi)
//   x   inverse transforms of d_y phi (d_z phi), i k~_x phi and phi; rest; its forward transform
//   y   forward
//   z   forward, the combination with F phi, inverse transforms of the new phi (and of i k~_z phi)
// NV = 0, 2, 3: the velocity components that the flow has (none; TG: x and y; ABC).  A derivative
// commutes with the transforms along the other axes, so each component needs its own path only
// from its axis on: 6, 9 or 12 one-dimensional transforms a step, where the components' own
// three-dimensional inverse transforms took 15, plus three pointwise passes.  Where phi itself is
// wanted (the last step, a renormalisation, a convergence check) the last z sweep writes it to phi,
// whose y and x transforms follow.  GB300, 128^3, 20 TG steps and the energy: 3.30 ms so before, now 1.61 ms;
// ABC 3.42 and 2.04, no flow at 96^3 2.61 and 0.83.  Bound by latency at 16 warps per SM (the fields stay in L2).
#pragma once
#include "gp_reduce.cuh"
#include "gp_sweep.cuh"

namespace gp {

enum { FLOW_NONE = 0, FLOW_TG = 1, FLOW_ABC = 2 };

struct Flow {
  int kind;
  double A, B, C;
};

// component J of the velocity at grid point (ix, iy, iz) from the tables, in the precision S of the tables
template <int J, typename S>
__device__ __forceinline__ S flow_comp(const Flow& f, const S* __restrict__ tab, int ix, int iy, int iz, int n) {
  const S* s1 = tab;
  const S* c1 = tab + n;
  if (f.kind == FLOW_NONE) return S(0);
  if (f.kind == FLOW_TG) {
    if constexpr (J == 0) return s1[ix] * c1[iy] * c1[iz];
    else if constexpr (J == 1) return -c1[ix] * s1[iy] * c1[iz];
    else return S(0);
  }
  S v = S(0);
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const S* sk = tab + 2 * k * n;
    const S* ck = sk + n;
    if constexpr (J == 0) v += (S)f.B * ck[iy] + (S)f.C * sk[iz];
    else if constexpr (J == 1) v += (S)f.C * ck[iz] + (S)f.A * sk[ix];
    else v += (S)f.A * ck[ix] + (S)f.B * sk[iy];
  }
  return v;
}
template <typename S>
__device__ __forceinline__ void flow_tab(const Flow& f, const S* __restrict__ tab, int ix, int iy, int iz, int n, S* v) {
  v[0] = flow_comp<0>(f, tab, ix, iy, iz, n);
  v[1] = flow_comp<1>(f, tab, ix, iy, iz, n);
  v[2] = flow_comp<2>(f, tab, ix, iy, iz, n);
}

struct ArgleStep {
  float2* f;                 // the field's mixed form
  float2* gy;                // d_y phi, d_z phi
  float2* gz;
  float2* ph;                // F phi
  float2* dst;               // z: where the mixed form goes (f or the user's field)
  const tw_t<float>* tw_fwd;
  const tw_t<float>* tw_inv;
  const float* tab;
  Flow flow;
  float q, beta;             // 1 / (4 alpha), beta
  float hd, dtau;            // dtau alpha / 2, dtau
};
// the launches of one length (instantiated in gp_inst_*.cu)
template <int L> struct ArgleLaunch {
  static cudaError_t y(const ArgleStep& a, int nv, cudaStream_t s);
  static cudaError_t x(const ArgleStep& a, int nv, cudaStream_t s);
  static cudaError_t z(const ArgleStep& a, bool combine, bool gz, cudaStream_t s);
};

template <int L> __host__ __device__ constexpr int argle_threads(bool contig) {
  return (contig ? contig_batch<float, L>() : strided_batch<float, L>()) * (L / Plan<L>::E);
}
// x: 16 warps per SM; 8 where a thread holds more than 16 points twice
template <int L> __host__ __device__ constexpr int argle_min_ctas(bool contig) {
  if (contig) return (Plan<L>::E > 16 ? 256 : 512) / argle_threads<L>(true) > 16 ? 16 : (Plan<L>::E > 16 ? 256 : 512) / argle_threads<L>(true);
  return rcapped<float, L>() ? rcap_blocks<float, L>(false) : (argle_threads<L>(false) > 256 ? 1 : 512 / argle_threads<L>(false) > 16 ? 16 : 512 / argle_threads<L>(false));
}
// v <- i k~ v, v at the positions that a forward transform leaves
template <int L, int E> __device__ __forceinline__ void times_ik(float2 (&v)[E], int t) {
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const float k = (float)wavenumber_d(out_pos<L, false>(e, t), L);
    v[e] = float2{-k * v[e].y, k * v[e].x};
  }
}

template <int L, int NV>
__global__ void __launch_bounds__(argle_threads<L>(false), argle_min_ctas<L>(false)) k_argle_y(const ArgleStep a) {
  constexpr int E = Plan<L>::E, B = strided_batch<float, L>();
  constexpr KConst inv_l = kconst(1.0 / L);
  extern __shared__ __align__(16) unsigned char smraw[];
  float2* sm = reinterpret_cast<float2*>(smraw);
  const int p = threadIdx.x % B, t = threadIdx.x / B, tile = blockIdx.x;
  const long base = (tile % (L / B)) * B + p + (long)(tile / (L / B)) * ((long)L * L), st = L;
  LayStrided lay{B};
  float2 v[E];
  // one pass per result: d_y phi, (d_z phi,) phi; a loop, so that the transform's code is there once
#pragma unroll 1
  for (int q = 0; q < NV; ++q) {
    const float2* src = NV == 3 && q == 1 ? a.gz : a.f;
    float2* dst = q == 0 ? a.gy : (NV == 3 && q == 1 ? a.gz : a.f);
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = src[base + out_pos<L, false>(e, t) * st];
    if (q == 0) times_ik<L>(v, t);
    __syncthreads();   // the exchanges of the pass before
    fft_regs<float, L, B, LayStrided, true>(v, t, p, sm, lay, a.tw_inv);
#pragma unroll
    for (int e = 0; e < E; ++e) dst[base + in_pos<L, false>(e, t) * st] = kscale(v[e], inv_l);
  }
}

template <int L, int NV>
__global__ void __launch_bounds__(argle_threads<L>(true), argle_min_ctas<L>(true)) k_argle_x(const ArgleStep a) {
  constexpr int E = Plan<L>::E, TP = L / E, B = contig_batch<float, L>();
  constexpr KConst inv_l = kconst(1.0 / L);
  constexpr bool WARP_X = TP <= 32;
  extern __shared__ __align__(16) unsigned char smraw[];
  float2* sm = reinterpret_cast<float2*>(smraw);
  const int p = threadIdx.x / TP, t = threadIdx.x % TP;
  const int row = blockIdx.x * B + p, iy = row % L, iz = row / L;
  const long base = (long)row * L;
  LayContig<L> lay;
  float2 v[E];
  [[maybe_unused]] float2 g[E];   // v . grad phi
  if constexpr (NV > 0) {
#pragma unroll
    for (int e = 0; e < E; ++e) g[e] = float2{0.0f, 0.0f};
  }
  // one pass per inverse transform: d_x phi, d_y phi, (d_z phi,) phi
#pragma unroll 1
  for (int q = NV > 0 ? 0 : NV; q <= NV; ++q) {
    const float2* src = q == 1 && NV > 0 ? a.gy : (q == 2 && NV == 3 ? a.gz : a.f);
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = src[base + out_pos<L, false>(e, t)];
    if (NV > 0 && q == 0) times_ik<L>(v, t);
    xsync<WARP_X>();   // the exchanges of the pass before
    fft_regs<float, L, B, LayContig<L>, true, WARP_X>(v, t, p, sm, lay, a.tw_inv);
    if constexpr (NV > 0) {
      if (q < NV) {
#pragma unroll
        for (int e = 0; e < E; ++e) {
          const int ix = in_pos<L, false>(e, t);
          const float w = q == 0 ? flow_comp<0>(a.flow, a.tab, ix, iy, iz, L)
                                 : (q == 1 ? flow_comp<1>(a.flow, a.tab, ix, iy, iz, L) : flow_comp<2>(a.flow, a.tab, ix, iy, iz, L));
          g[e] = float2{fmaf(w, v[e].x, g[e].x), fmaf(w, v[e].y, g[e].y)};
        }
      }
    }
  }
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const float2 f = kscale(v[e], inv_l);
    float c = a.beta * (1.0f - (f.x * f.x + f.y * f.y));
    if constexpr (NV > 0) {
      float w[3];
      flow_tab<float>(a.flow, a.tab, in_pos<L, false>(e, t), iy, iz, L, w);
      c -= a.q * (w[0] * w[0] + w[1] * w[1] + w[2] * w[2]);
      const float2 d = kscale(g[e], inv_l);
      v[e] = float2{d.y + c * f.x, -d.x + c * f.y};   // -i v . grad phi + c phi
    } else {
      v[e] = float2{c * f.x, c * f.y};
    }
  }
  xsync<WARP_X>();
  fft_regs<float, L, B, LayContig<L>, false, WARP_X>(v, t, p, sm, lay, a.tw_fwd);
#pragma unroll
  for (int e = 0; e < E; ++e) a.f[base + out_pos<L, false>(e, t)] = v[e];
}

// COMBINE: F phi <- [(1 - a) F phi + dtau F rest] / (1 + a) first, a = dtau alpha |k|^2 / 2; GZ: d_z phi is wanted
template <int L, bool COMBINE, bool GZ>
__global__ void __launch_bounds__(argle_threads<L>(false), argle_min_ctas<L>(false)) k_argle_z(const ArgleStep a) {
  constexpr int E = Plan<L>::E, B = strided_batch<float, L>();
  constexpr KConst inv_l = kconst(1.0 / L);
  extern __shared__ __align__(16) unsigned char smraw[];
  float2* sm = reinterpret_cast<float2*>(smraw);
  const int p = threadIdx.x % B, t = threadIdx.x / B, tile = blockIdx.x;
  const int ix = (tile % (L / B)) * B + p, iy = tile / (L / B);
  const long base = ix + (long)iy * L, st = (long)L * L;
  LayStrided lay{B};
  float2 v[E];
  if constexpr (COMBINE) {
    const int kx = wavenumber(ix, L), ky = wavenumber(iy, L);
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = a.f[base + in_pos<L, false>(e, t) * st];
    fft_regs<float, L, B, LayStrided, false>(v, t, p, sm, lay, a.tw_fwd);
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int pos = out_pos<L, false>(e, t), kz = wavenumber(pos, L);
      const float d = a.hd * (float)(kx * kx + ky * ky + kz * kz);
      const float num = 1.0f - d, den = 1.0f / (1.0f + d);
      const float2 x = a.ph[base + pos * st];
      v[e] = float2{(num * x.x + a.dtau * v[e].x) * den, (num * x.y + a.dtau * v[e].y) * den};
      a.ph[base + pos * st] = v[e];
    }
    __syncthreads();   // the exchanges
  } else {
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = a.ph[base + out_pos<L, false>(e, t) * st];
  }
#pragma unroll 1
  for (int q = GZ ? 0 : 1; q < 2; ++q) {   // d_z phi, phi
    if (GZ && q == 0) times_ik<L>(v, t);
    fft_regs<float, L, B, LayStrided, true>(v, t, p, sm, lay, a.tw_inv);
    float2* dst = q == 0 ? a.gz : a.dst;
#pragma unroll
    for (int e = 0; e < E; ++e) dst[base + in_pos<L, false>(e, t) * st] = kscale(v[e], inv_l);
    if (q == 0) {
      __syncthreads();   // the exchanges
#pragma unroll
      for (int e = 0; e < E; ++e) v[e] = a.ph[base + out_pos<L, false>(e, t) * st];   // this thread's own values
    }
  }
}

template <int L> static cudaError_t argle_launch(void (*k)(ArgleStep), const ArgleStep& a, bool contig, cudaStream_t s) {
  constexpr int BS = strided_batch<float, L>(), BC = contig_batch<float, L>();
  const size_t sm = sizeof(float2) * (contig ? (size_t)contig_pitch<L>() * BC : (size_t)L * BS);
  const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  k<<<contig ? L * L / BC : L * (L / BS), argle_threads<L>(contig), sm, s>>>(a);
  return cudaGetLastError();
}
template <int L> cudaError_t ArgleLaunch<L>::y(const ArgleStep& a, int nv, cudaStream_t s) {
  return argle_launch<L>(nv == 3 ? k_argle_y<L, 3> : k_argle_y<L, 2>, a, false, s);
}
template <int L> cudaError_t ArgleLaunch<L>::x(const ArgleStep& a, int nv, cudaStream_t s) {
  return argle_launch<L>(nv == 3 ? k_argle_x<L, 3> : nv == 2 ? k_argle_x<L, 2> : k_argle_x<L, 0>, a, true, s);
}
template <int L> cudaError_t ArgleLaunch<L>::z(const ArgleStep& a, bool combine, bool gz, cudaStream_t s) {
  if (combine) return argle_launch<L>(gz ? k_argle_z<L, true, true> : k_argle_z<L, true, false>, a, false, s);
  return argle_launch<L>(gz ? k_argle_z<L, false, true> : k_argle_z<L, false, false>, a, false, s);
}

}  // namespace gp
