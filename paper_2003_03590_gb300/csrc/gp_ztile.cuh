// gp_ztile.cuh -- persistent float32 z sweeps of 1024 points, tiles of 16 pencils.
//
// A z-pencil's elements lie one z-plane (8 MB) apart, and z tiles move at a fixed number of row pieces per
// second, loads or stores, whatever the pieces' length up to 128 bytes: 1024^3 takes 6.84 ms with 64-byte rows
// (8 pencils, what a ring of stages has room for), 8.4 ms when a store covers 32-byte pieces of eight rows, 3.58 ms
// with 128-byte rows (copy only).  So a tile has 16 pencils, 128 KB.  There is one landing buffer; the tile is held in
// registers (512 threads, 32 points each) and stored from them, 16 lanes to a row, and the next tile lands while
// this one is transformed.  The exchange between the two radix-32 passes goes through 68 KB beside the landing buffer, real
// parts first and then imaginary parts (both at once need 132 KB); the first one of inverse-N-forward goes through the
// landing buffer itself, which leaves the copy half of that tile's time (5.69 -> 5.44 ms).
// GB300, 1024^3, us per launch, ring of 64-byte-row stages / one tile per CTA / this kernel: forward 6840 / 4900 / 3470,
// N-forward 6840 / 5180 / 4020, inverse-N 6840 / 5870 / 3940, inverse-N-forward 6840 / 7790 / 5440.  One transform is bound
// by the copies; with two the block barriers keep the warps in step and instruction issue is the limit.
#pragma once
#include "gp_tma.cuh"

namespace gp {

// Lengths whose z sweeps run here.
template <int L> __host__ __device__ constexpr bool ztile_ok() { return L == 1024; }

template <int L> struct ZTile {
  static constexpr int B = 16;                           // pencils of a tile
  static constexpr int E = Plan<L>::E, TP = L / E;
  static constexpr int NT = B * TP;
  static constexpr int RB = 8 * B, BOX = 256;            // bytes of a row, rows of a copy
  // floats of a pencil's exchange: position pos at pos + pos / 32.  Writes (32 t + k) and reads (t + 32 r) of a
  // warp touch t and t + 1 (t even) of 16 pencils: 2 p + t modulo 32.
  static constexpr int PITCH = L + L / 32 + 2;
  static constexpr int LAND = L * RB, XCH = B * PITCH * 4;
  static constexpr size_t SMEM = LAND + XCH + 64 + 1024;   // alignment of the landing buffer
  static_assert(E == 32 && TP == 32 && PITCH % 32 == 2, "two passes of radix 32");
};

template <int L, int OP> __global__ void __launch_bounds__(ZTile<L>::NT, 1) k_ztile(const __grid_constant__ TmaSweepArgs a) {
  using G = ZTile<L>;
  constexpr int E = G::E;
  constexpr KConst inv_l = kconst(1.0 / L);
  extern __shared__ __align__(128) unsigned char smraw[];
  const uint32_t raw = smem_u32(smraw), pad = ((raw + 1023u) & ~1023u) - raw;
  uint64_t* full = reinterpret_cast<uint64_t*>(smraw + pad + G::LAND + G::XCH);
  int* taken = reinterpret_cast<int*>(full + 1);         // warps that are done with the landing buffer, counted on over the tiles
  const int tid = threadIdx.x, lane = tid & 31, p = tid % G::B, t = tid / G::B;
  // the copy's swizzle: 16-byte chunk c of row r at c ^ (r & 7)
  const uint32_t land = raw + pad + (uint32_t)t * G::RB + ((((uint32_t)p >> 1) ^ (uint32_t)(t & 7)) << 4) + (p & 1) * 8;
  float* const xch = reinterpret_cast<float*>(smraw + pad + G::LAND) + p * G::PITCH;
  constexpr int per_field = (L / G::B) * L;
  const int total = per_field * a.count;
  auto issue = [&](int tile) {
    const int f = tile / per_field, r = tile - f * per_field;
    mbar_expect_tx(full, (unsigned)G::LAND);
#pragma unroll
    for (int k = 0; k < L / G::BOX; ++k)
      tma_load_3d(smraw + pad + (size_t)k * G::BOX * G::RB, &a.map[f], full, (r % (L / G::B)) * G::B, r / (L / G::B), k * G::BOX);
  };
  if (tid == 0) {
    mbar_init(full, 1);
    *taken = 0;
    fence_mbar_init();
    if ((int)blockIdx.x < total) issue(blockIdx.x);
  }
  __syncthreads();
  float2 v[E];
  // the last warp to be done with the landing buffer starts the copy of the next tile
  auto taken_part = [&](int it, int tile) {
    fence_async_smem();
    __syncwarp();
    if (lane == 0) {
      __threadfence_block();
      const int n = atomicAdd(taken, 1);
      if (n == G::NT / 32 * (it + 1) - 1 && tile + (int)gridDim.x < total) {
        __threadfence_block();
        issue(tile + gridDim.x);
      }
    }
    __syncwarp();
  };
  // IN_LAND: the exchange goes through the landing buffer, position pos of pencil p at row pos
  auto transform = [&](auto inv, auto in_land) {
    constexpr bool INV = decltype(inv)::value;
    static_assert(radix_of<L, INV>(0) == 32 && Plan<L>::NP == 2, "two passes of radix 32");
    const float4* tw = INV ? a.tw_inv : a.tw_fwd;
    pass_compute<float, L, 1, LayStrided, INV, 0>(v, t, tw);
    if constexpr (decltype(in_land)::value) {
      float2* const x = reinterpret_cast<float2*>(smraw + pad) + p;
      __syncthreads();
#pragma unroll
      for (int e = 0; e < E; ++e) x[(32 * t + e) * G::B] = v[e];
      __syncthreads();
#pragma unroll
      for (int e = 0; e < E; ++e) v[e] = x[(t + 32 * e) * G::B];
    } else {
#pragma unroll
      for (int e = 0; e < E; ++e) xch[33 * t + e] = v[e].x;
      __syncthreads();
#pragma unroll
      for (int e = 0; e < E; ++e) v[e].x = xch[t + 33 * e];
      __syncthreads();
#pragma unroll
      for (int e = 0; e < E; ++e) xch[33 * t + e] = v[e].y;
      __syncthreads();
#pragma unroll
      for (int e = 0; e < E; ++e) v[e].y = xch[t + 33 * e];
    }
    pass_compute<float, L, 1, LayStrided, INV, 1>(v, t, tw);
  };
  int it = 0;
  for (int tile = blockIdx.x; tile < total; tile += gridDim.x, ++it) {
    bool ok = mbar_wait_bounded(full, (unsigned)it & 1u);
    if (!__syncthreads_and(ok)) {   // one decision; also the end of the exchange before
      if (tid == 0) atomicExch(a.status, 1);
      mbar_wait_bounded(full, (unsigned)it & 1u);   // a copy in flight lands before the shared memory goes away
      break;
    }
#pragma unroll
    for (int e = 0; e < E; ++e) {
      asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v[e].x), "=f"(v[e].y) : "r"(land + e * (uint32_t)(G::TP * G::RB)));
    }
    if constexpr (OP != OP_INV_N_FWD) taken_part(it, tile);
    if constexpr (OP == OP_N_FWD) nonlinear_all<E>(v, a.nl_coef, a.nl_shift);
    if constexpr (OP == OP_FWD || OP == OP_N_FWD) transform(std::false_type{}, std::false_type{});
    if constexpr (OP == OP_INV || OP == OP_INV_N || OP == OP_INV_N_FWD) {
      transform(std::true_type{}, std::bool_constant<OP == OP_INV_N_FWD>{});
      if constexpr (OP == OP_INV_N_FWD) taken_part(it, tile);
      if (a.scale_inv) {
#pragma unroll
        for (int e = 0; e < E; ++e) v[e] = kscale(v[e], inv_l);
      }
      if constexpr (OP != OP_INV) nonlinear_all<E>(v, a.nl_coef, a.nl_shift);
    }
    if constexpr (OP == OP_INV_N_FWD) transform(std::false_type{}, std::false_type{});
    const int f = tile / per_field, r = tile - f * per_field;
    float2* g = a.psi[f] + (size_t)(r / (L / G::B)) * L + (r % (L / G::B)) * G::B + p + (size_t)t * L * L;
#pragma unroll
    for (int e = 0; e < E; ++e) g[(size_t)e * G::TP * L * L] = v[e];
  }
}

template <int L> struct ZTileLaunch {
  template <int OP> static cudaError_t run(const TmaSweepArgs& a, cudaStream_t s) {
    static const cudaError_t attr =
        cudaFuncSetAttribute(k_ztile<L, OP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ZTile<L>::SMEM);
    if (attr != cudaSuccess) return attr;
    const int tiles = (L / ZTile<L>::B) * L * a.count, sms = TmaLaunch<L>::sms();
    k_ztile<L, OP><<<tiles < sms ? tiles : sms, ZTile<L>::NT, ZTile<L>::SMEM, s>>>(a);
    return cudaGetLastError();
  }
  static cudaError_t launch(const TmaSweepArgs& a, cudaStream_t s) {
    switch (a.op) {
#define GP_R(OPV) case OPV: return run<OPV>(a, s);
      GP_STRIDED_OPS(GP_R)
#undef GP_R
      default: return cudaErrorInvalidValue;
    }
  }
};

}  // namespace gp
