// gp_deriv.cuh -- spectral first derivatives of float32 fields, one axis per kernel.
//
// d_j psi = F^-1 i k~_j F psi involves the transform along axis j only: the other two cancel.  One
// kernel per axis reads the field, transforms its pencils forward, multiplies by i k~ (the Nyquist
// mode zeroed) and transforms back -- 2 one-dimensional transforms and 16 bytes per point, where
// going through the three-dimensional spectrum takes 3 + 3 transforms per component (12 sweeps and a
// k-space pass for a gradient, 96 bytes per point more) and rounds more often.  What is done with
// the derivative happens in the same kernel (EPI): pointwise work, sums over the axis' spectrum, and
// the first forward transform of the result along the same axis.
//
// A CTA walks tiles of pencils of one axis (gp_sweep.cuh's tiles and transforms).  The next tile is
// copied to shared memory (cp.async) while the current one is worked on, and stays there for the
// pointwise work; the exchanges between radix passes use a buffer of their own.  Bound by latency and
// instruction issue at 16 warps per SM (128 registers a thread; 12 at 96 and 192, see deriv_ahead): GB300, 256^3, the diagnostics' three
// kernels (3 or 4 transforms and 20 to 28 bytes per point each) 0.15, 0.15 and 0.22 ms.
#pragma once
#include <type_traits>

#include "gp_reduce.cuh"
#include "gp_sweep.cuh"

namespace gp {

struct DerivArgs {
  const float2* in;
  const tw_t<float>* tw_fwd;
  const tw_t<float>* tw_inv;
};

// EPI: a struct with
//   static constexpr int AXIS;      the axis of the derivative
//   static constexpr bool MODES;    mode() is wanted
//   static constexpr bool PRE;      pre() is wanted: a value of the point, read ahead of the inverse transform
//   static constexpr int POST;      0: put() takes the point's value; 1: its forward transform along the axis;
//                                   2: the same, and put2() that of second()
//   using State = ...;              per-thread state, default-constructed
//   void mode(State&, int k, int kd, float2 F)   a mode of this axis: wavenumber, Nyquist-zeroed one, value
//   float pre(long i)
//   float2 point(State&, long i, float2 f, float2 g, float pre)   f: the field, g: its derivative, at i
//   float2 second(float2 f)
//   void put(long i, float2 v), put2(long i, float2 v)
//   void finish(State&)             at the end, by every thread of the block
template <int L, bool CONTIG> __host__ __device__ constexpr int deriv_batch() {
  return CONTIG ? contig_batch<float, L>() : strided_batch<float, L>();
}
template <int L, bool CONTIG> __host__ __device__ constexpr int deriv_threads() { return deriv_batch<L, CONTIG>() * (L / Plan<L>::E); }
// CTAs per SM that the registers must allow (16 warps per SM)
template <int L, bool CONTIG> __host__ __device__ constexpr int deriv_min_ctas() {
  return 512 / deriv_threads<L, CONTIG>() > 16 ? 16 : 512 / deriv_threads<L, CONTIG>();
}
template <int L, bool CONTIG> __host__ __device__ constexpr int deriv_exchange() {   // elements
  return (CONTIG ? contig_pitch<L>() : L) * deriv_batch<L, CONTIG>();
}
// two tiles of look-ahead up to 256 points; beyond, one tile at a time, read directly.  With those CTAs they fit in
// shared memory, but for the lengths of 24 elements a thread: 96 and 192 hold three quarters of them (192 three CTAs of
// 74 to 77 KB, 96 three of 77 KB for x and six of 37 KB for y and z), 12 warps per SM
template <int L> __host__ __device__ constexpr bool deriv_ahead() { return L >= 32 && L <= 256; }
template <int L, bool CONTIG> __host__ __device__ constexpr size_t deriv_smem() {
  return sizeof(float2) * ((size_t)deriv_exchange<L, CONTIG>() + (deriv_ahead<L>() ? 2 * (size_t)deriv_batch<L, CONTIG>() * L : 0));
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}

template <int L, class EPI>
__global__ void __launch_bounds__((deriv_threads<L, EPI::AXIS == 0>()), (deriv_min_ctas<L, EPI::AXIS == 0>()))
    k_deriv(const DerivArgs a, int tiles, const EPI epi) {
  constexpr bool CONTIG = EPI::AXIS == 0, AHEAD = deriv_ahead<L>();
  constexpr int E = Plan<L>::E, TP = L / E, B = deriv_batch<L, CONTIG>(), NT = deriv_threads<L, CONTIG>();
  constexpr KConst inv_l = kconst(1.0 / L);
  constexpr bool WARP_X = CONTIG && TP <= 32;
  extern __shared__ __align__(16) unsigned char smraw[];
  float2* const tile_buf = reinterpret_cast<float2*>(smraw);                   // AHEAD: [2][pos][pencil] or [2][row][x]
  float2* const sm = tile_buf + (AHEAD ? 2 * B * L : 0);                       // exchanges
  const int p = CONTIG ? threadIdx.x / TP : threadIdx.x % B, t = CONTIG ? threadIdx.x % TP : threadIdx.x / B;
  using Lay = std::conditional_t<CONTIG, LayContig<L>, LayStrided>;
  Lay lay;
  if constexpr (!CONTIG) lay.B = B;
  // element (pencil 0, position 0) of a tile, and the step along the pencil
  auto origin = [&](int tile) -> long {
    if constexpr (CONTIG) return (long)tile * B * L;
    else return (tile % (L / B)) * B + (long)(tile / (L / B)) * (EPI::AXIS == 1 ? (long)L * L : (long)L);
  };
  constexpr long step = CONTIG ? 1 : (EPI::AXIS == 1 ? (long)L : (long)L * L);
  auto fetch = [&](int tile, int b) {   // the tile into buffer b, 16 bytes at a time
    if constexpr (AHEAD) {
      const float2* src = a.in + origin(tile);
      float2* dst = tile_buf + b * B * L;
      if constexpr (CONTIG) {
        for (int q = threadIdx.x; q < B * L / 2; q += NT) cp_async16(dst + 2 * q, src + 2 * q);
      } else {
        for (int q = threadIdx.x; q < B * L / 2; q += NT) {
          const int pos = q / (B / 2), c = q % (B / 2);
          cp_async16(dst + pos * B + 2 * c, src + pos * step + 2 * c);
        }
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  typename EPI::State st{};
  if (AHEAD && (int)blockIdx.x < tiles) fetch(blockIdx.x, 0);
  int b = 0;
  for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x, b ^= 1) {
    const long base = origin(tile) + (CONTIG ? (long)p * L : (long)p);
    float2 v[E];
    if constexpr (AHEAD) {
      if (tile + (int)gridDim.x < tiles) {
        fetch(tile + gridDim.x, b ^ 1);   // its last readers are past the barrier at the end of the loop
        asm volatile("cp.async.wait_group 1;" ::: "memory");
      } else {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
      }
      __syncthreads();
    }
    auto field = [&](int pos) -> float2 {
      if constexpr (AHEAD) return tile_buf[b * B * L + (CONTIG ? p * L + pos : pos * B + p)];
      else return a.in[base + pos * step];
    };
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = field(in_pos<L, false>(e, t));
    xsync<WARP_X>();   // the previous tile's exchanges
    fft_regs<float, L, B, Lay, false, WARP_X>(v, t, p, sm, lay, a.tw_fwd);
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int i = out_pos<L, false>(e, t), kd = wavenumber_d(i, L);
      if constexpr (EPI::MODES) epi.mode(st, wavenumber(i, L), kd, v[e]);
      const float f = (float)kd;
      v[e] = float2{-f * v[e].y, f * v[e].x};
    }
    [[maybe_unused]] float pv[E];
    if constexpr (EPI::PRE) {
#pragma unroll
      for (int e = 0; e < E; ++e) pv[e] = epi.pre(base + in_pos<L, false>(e, t) * step);
    }
    xsync<WARP_X>();
    fft_regs<float, L, B, Lay, true, WARP_X>(v, t, p, sm, lay, a.tw_inv);
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int pos = in_pos<L, false>(e, t);
      const long i = base + pos * step;
      float pe = 0.0f;
      if constexpr (EPI::PRE) pe = pv[e];
      v[e] = epi.point(st, i, field(pos), kscale(v[e], inv_l), pe);
      if constexpr (EPI::POST == 0) epi.put(i, v[e]);
    }
    if constexpr (EPI::POST > 0) {
      xsync<WARP_X>();
      fft_regs<float, L, B, Lay, false, WARP_X>(v, t, p, sm, lay, a.tw_fwd);
#pragma unroll
      for (int e = 0; e < E; ++e) epi.put(base + out_pos<L, false>(e, t) * step, v[e]);
    }
    if constexpr (EPI::POST > 1) {
#pragma unroll
      for (int e = 0; e < E; ++e) v[e] = epi.second(field(in_pos<L, false>(e, t)));
      xsync<WARP_X>();
      fft_regs<float, L, B, Lay, false, WARP_X>(v, t, p, sm, lay, a.tw_fwd);
#pragma unroll
      for (int e = 0; e < E; ++e) epi.put2(base + out_pos<L, false>(e, t) * step, v[e]);
    }
    if constexpr (AHEAD) __syncthreads();   // the tile's buffer is free again
  }
  epi.finish(st);
}

// most blocks of a derivative kernel (the same for every length and axis, so that per-block sums can
// be sized without knowing the kernel); small fields have fewer tiles
constexpr int DERIV_BLOCKS = 152 * 4;

template <int L, class EPI> cudaError_t deriv_launch(const DerivArgs& a, const EPI& epi, cudaStream_t s) {
  constexpr bool CONTIG = EPI::AXIS == 0;
  constexpr size_t smem = deriv_smem<L, CONTIG>();
  static const cudaError_t attr = cudaFuncSetAttribute(k_deriv<L, EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (attr != cudaSuccess) return attr;
  const int tiles = L * L / deriv_batch<L, CONTIG>();
  // as many as the registers allow at once, DERIV_BLOCKS at most (at 192 the last quarter runs after the others)
  int blocks = 152 * deriv_min_ctas<L, CONTIG>();
  if (blocks > DERIV_BLOCKS) blocks = DERIV_BLOCKS;
  k_deriv<L, EPI><<<tiles < blocks ? tiles : blocks, deriv_threads<L, CONTIG>(), smem, s>>>(a, tiles, epi);
  return cudaGetLastError();
}
template <class EPI> cudaError_t deriv(int n, const DerivArgs& a, const EPI& epi, cudaStream_t s) {
  switch (n) {
#define GP_CASE(L) case L: return deriv_launch<L, EPI>(a, epi, s);
    GP_CASE(8) GP_CASE(12) GP_CASE(16) GP_CASE(24) GP_CASE(32) GP_CASE(48) GP_CASE(64) GP_CASE(96) GP_CASE(128)
    GP_CASE(192) GP_CASE(256) GP_CASE(512) GP_CASE(1024)
#undef GP_CASE
    default: return cudaErrorInvalidValue;
  }
}

// what most EPIs leave out
struct DerivEpi {
  static constexpr bool MODES = false, PRE = false;
  static constexpr int POST = 0;
  struct State {};
  template <class S> __device__ __forceinline__ void mode(S&, int, int, float2) const {}
  __device__ __forceinline__ float pre(long) const { return 0.0f; }
  __device__ __forceinline__ float2 second(float2 f) const { return f; }
  __device__ __forceinline__ void put2(long, float2) const {}
  template <class S> __device__ __forceinline__ void finish(S&) const {}
};

}  // namespace gp
