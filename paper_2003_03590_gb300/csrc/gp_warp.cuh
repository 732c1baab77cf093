// gp_warp.cuh -- persistent float32 sweeps in which a pencil never leaves its warp.
//
// The transforms, flows and tiles are those of gp_sweep.cuh (the results are the same bit for bit).
// What differs is who waits for whom: TP = L / E lanes of one warp hold a pencil (32 / TP pencils per
// warp), its exchange between the two radix passes goes through the warp's own part of the stage, in
// place, and the only synchronisation inside a tile is __syncwarp.  A stage changes hands by
// mbarriers: `full` (the copy has landed), `empty` (every warp of the tile has written its result),
// `freed` (the store has read it); a loader and a storer warp do the copies.  With block barriers
// around every exchange (four per transform) the warps of a CTA ran in lock-step and waited for the
// slowest, and the copies were issued by a compute thread.
//
// y/z tiles (B consecutive x of L rows).  The tile is copied by TMA with the swizzle of its row
// length: 16-byte chunk c of row r at chunk c ^ (r & 7) (128-byte rows) or c ^ ((r >> 1) & 3) (64-byte
// rows).  A half-warp's 16 accesses are 8 consecutive rows of the two pencils of one chunk: with the
// swizzle they cover all 32 banks once.  The exchange keeps that: Stockham position pos = R0 j + k of
// the first pass (radix R0, butterfly j, output k) is kept in row R0 j + (k ^ (j & 7)), so writes
// (fixed k, 8 consecutive j) and reads (fixed j, 8 consecutive k) both touch 8 rows that differ modulo
// 8.  The exclusive-or only reaches address bits that the tile's base leaves zero: an access is one
// XOR on a per-thread base plus an immediate.
//
// x tiles (B rows).  The rows are copied one by one (bulk copies) to a pitch of pitch() elements; a
// row's exchange uses the padded layout pos + pos / R0 inside its own row.
#pragma once
#include <type_traits>

#include "gp_tma.cuh"
#include "gp_ztile.cuh"

namespace gp {

// Lengths with this engine (two passes, power-of-two radices of at least 8; from 256 on, where it is
// the faster one: GB300, one launch, before -> now: 256^3 z inverse-N-forward 70 -> 66 us, fused plane
// kernel 147.8 -> 143.6 us; 512^3 z inverse-N-forward 603 -> 530 us, N-forward 410 -> 375 us; 1024^3 y
// 2930 -> 2650 us; at 64 and 128 points the per-sweep ensemble was 1% slower with it).
template <int L> __host__ __device__ constexpr bool warp_ok() { return L >= 256; }
// its y sweeps: not at 512, where the block kernel of gp_tma.cuh streams at 94% of the copy rate
// (336 us against 364)
template <int L> __host__ __device__ constexpr bool warp_axis(int axis) { return warp_ok<L>() && !(L == 512 && axis == 1); }
// pencils of a z tile: from 256 points on 16 (128-byte rows).  A z-pencil's elements lie one z-plane apart and a
// copy of z tiles runs at a fixed number of rows per second (512^3: 64-byte rows 675 us, 128-byte
// rows 361 us, 256-byte rows 338 us; 1024^3: 7157, 3581, 2786 us); at 1024 a stage of 16 pencils is
// 128 KB and the z sweeps have a kernel of their own (gp_ztile.cuh).
constexpr int WARP_Z_PENCILS = 16;

__device__ __forceinline__ float2 lds2(uint32_t a) {
  float2 v;
  asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a));
  return v;
}
__device__ __forceinline__ void sts2(uint32_t a, float2 v) {
  asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.x), "f"(v.y));
}

// ---------------------------------------------------------------- addresses of a thread's elements
// y/z tiles: B pencils, rows of RB = 8 B bytes.  at(): shared address of the tile, aligned to 1 KB.
template <int L, int B> struct WarpStrided {
  static constexpr int RB = 8 * B;
  static constexpr int TP = L / Plan<L>::E;
  static_assert(TP % 8 == 0 && (B == 16 || B == 8), "swizzle period of 8 rows");
  static constexpr int PW = 32 / TP;            // pencils per warp
  int t, p;                                     // lane's place along the pencil, its pencil
  uint32_t row0;                                // offset of (row t & 7, pencil p) in the tile
  uint32_t nat;                                 // shared address of (row t, pencil p)
  uint32_t wr;                                  // shared address of (row t & 7, pencil p)
  static __host__ __device__ __forceinline__ constexpr uint32_t swz(uint32_t r) {
    return (B == 16 ? (r & 7) : ((r >> 1) & 3)) << 4;
  }
  // what adding q (exclusive-or) to the low three bits of a row does to an address
  static __host__ __device__ __forceinline__ constexpr uint32_t mask(uint32_t q) { return ((q & 7) * RB) ^ swz(q & 7); }
  __device__ __forceinline__ WarpStrided(int w, int lane) {
    if constexpr (PW == 1) {
      t = lane;
      p = w;
    } else {
      t = (lane >> 1) % TP;
      p = 2 * (w * (PW / 2) + (lane >> 1) / TP) + (lane & 1);
    }
    const uint32_t t7 = t & 7;
    row0 = t7 * RB + ((((uint32_t)p >> 1) << 4) ^ swz(t7)) + (p & 1) * 8;
    nat = wr = 0;
  }
  __device__ __forceinline__ void at(uint32_t st) {
    wr = st + row0;
    nat = wr + (uint32_t)(t & ~7) * RB;
  }
  __device__ __forceinline__ uint32_t natural(int c) const { return nat + (uint32_t)c * RB; }   // row t + c, c % 8 == 0
  template <int R0> __device__ __forceinline__ uint32_t ex_write(int b, int k) const {
    return ((wr + (uint32_t)(R0 * t) * RB) ^ mask(k)) + (uint32_t)(b * TP * R0 + (k & ~7)) * RB;
  }
  template <int R0> __device__ __forceinline__ uint32_t ex_read(int b, int r) const {
    return (nat ^ mask(r)) + (uint32_t)(R0 * r + b * TP) * RB;
  }
};

// x tiles: rows of pitch() elements
template <int L> struct WarpContig {
  static constexpr int TP = L / Plan<L>::E;
  static constexpr int PW = 32 / TP;
  static __host__ __device__ constexpr int pitch() { return L + L / 16; }   // 16-byte multiple
  int t, p;
  uint32_t nat, row;
  __device__ __forceinline__ WarpContig(int w, int lane) {
    t = lane % TP;
    p = w * PW + lane / TP;
    nat = row = 0;
  }
  __device__ __forceinline__ void at(uint32_t st) {
    row = st + (uint32_t)(p * pitch()) * 8;
    nat = row + 8 * t;
  }
  __device__ __forceinline__ uint32_t natural(int c) const { return nat + 8 * c; }
  // element pos + pos / R0 for pos = R0 (t + b TP) + k (write) and pos = R0 r + t + b TP (read, t + b TP < R0)
  template <int R0> __device__ __forceinline__ uint32_t ex_write(int b, int k) const {
    return row + 8u * (uint32_t)((R0 + 1) * t) + 8u * (b * TP * (R0 + 1) + k);
  }
  template <int R0> __device__ __forceinline__ uint32_t ex_read(int b, int r) const {
    return nat + 8u * ((R0 + 1) * r + b * TP);
  }
};

// ---------------------------------------------------------------- transform of a warp's pencils
template <int L, bool INV, class Acc, bool TW_SH>
__device__ __forceinline__ void fft_warp(float2* v, const Acc& A, const float4* __restrict__ tw) {
  constexpr int E = Plan<L>::E, R0 = radix_of<L, INV>(0), R1 = radix_of<L, INV>(1);
  static_assert(Plan<L>::NP == 2, "two passes");
  pass_compute<float, L, 1, Acc, INV, 0, TW_SH>(v, A.t, tw);
#pragma unroll
  for (int b = 0; b < E / R0; ++b)
#pragma unroll
    for (int k = 0; k < R0; ++k) sts2(A.template ex_write<R0>(b, k), v[b * R0 + k]);
  __syncwarp();
#pragma unroll
  for (int b = 0; b < E / R1; ++b)
#pragma unroll
    for (int r = 0; r < R1; ++r) v[b * R1 + r] = lds2(A.template ex_read<R0>(b, r));
  __syncwarp();
  pass_compute<float, L, 1, Acc, INV, 1, TW_SH>(v, A.t, tw);
}

// One operation on a warp's pencils of a tile in shared memory (sweep_op_body's counterpart).
// (i1, i2): the row's other two grid indices (OP_FWD_K_INV only).
template <int OP, int L, class Acc, bool TW_SH>
__device__ __forceinline__ void warp_op(const SweepArgs<float>& a, const Acc& A, int i1, int i2) {
  constexpr int E = Plan<L>::E, TP = L / E;
  constexpr KConst inv_l = kconst(1.0 / L);
  constexpr bool IN_INV = OP == OP_INV || OP == OP_INV_N || OP == OP_INV_N_FWD;
  constexpr bool OUT_INV = OP == OP_INV || OP == OP_INV_N || OP == OP_FWD_K_INV;
  [[maybe_unused]] float4 eo{};
  if constexpr (OP == OP_FWD_K_INV) eo = __ldg(a.ek2 + i2 * L + i1);   // its latency under the transform
  float2 v[E];
  constexpr int RI = radix_of<L, IN_INV>(0);
#pragma unroll
  for (int e = 0; e < E; ++e) v[e] = lds2(A.natural((e / RI) * TP + (e % RI) * (L / RI)));
  __syncwarp();   // the exchange overwrites what other lanes have read
  if constexpr (OP == OP_N_FWD) nonlinear_all<E>(v, a.nl_coef, a.nl_shift);
  if constexpr (OP == OP_FWD || OP == OP_N_FWD || OP == OP_FWD_K_INV) fft_warp<L, false, Acc, TW_SH>(v, A, a.tw_fwd);
  if constexpr (IN_INV) {
    fft_warp<L, true, Acc, TW_SH>(v, A, a.tw_inv);
    if (a.scale_inv) {
#pragma unroll
      for (int e = 0; e < E; ++e) v[e] = kscale(v[e], inv_l);
    }
    if constexpr (OP != OP_INV) nonlinear_all<E>(v, a.nl_coef, a.nl_shift);
  }
  if constexpr (OP == OP_INV_N_FWD) fft_warp<L, false, Acc, TW_SH>(v, A, a.tw_fwd);
  if constexpr (OP == OP_FWD_K_INV) {
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = twmul_k(twmul_k(v[e], __ldg(a.ekx + out_pos<L, false>(e, A.t))), eo);
    fft_warp<L, true, Acc, TW_SH>(v, A, a.tw_inv);
  }
  constexpr int RO = radix_of<L, OUT_INV>(1);   // registers of the last pass (out_pos)
#pragma unroll
  for (int e = 0; e < E; ++e) sts2(A.natural((e / RO) * TP + (e % RO) * (L / RO)), v[e]);
}

// ---------------------------------------------------------------- copies
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, unsigned bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ void bulk_store(void* dst, uint32_t src, unsigned bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_load_hint(uint32_t dst, const void* src, unsigned bytes, uint64_t* bar, uint64_t pol) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(dst),
      "l"(src), "r"(bytes), "r"(smem_u32(bar)), "l"(pol)
      : "memory");
}
__device__ __forceinline__ void bulk_store_hint(void* dst, uint32_t src, unsigned bytes, uint64_t pol) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group.L2::cache_hint [%0], [%1], %2, %3;" ::"l"(dst), "r"(src),
               "r"(bytes), "l"(pol)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// ---------------------------------------------------------------- persistent sweep
// Geometry of one sweep kernel: S stages of one tile, NG groups of NW compute warps (group g takes
// the CTA's tiles g, g + NG, ...), one loader and one storer warp.
template <int L, bool CONTIG, int B, int S_, int NG_> struct WarpSweep {
  static constexpr int S = S_, NG = NG_;
  static constexpr int TP = L / Plan<L>::E;
  static constexpr int NW = B * TP / 32;                 // warps per tile
  static constexpr int NCT = NG * NW * 32;                 // compute threads
  static constexpr int NT = NCT + 64;
  static constexpr int STAGE = ((CONTIG ? B * WarpContig<L>::pitch() : B * L) * 8 + 1023) / 1024 * 1024;   // bytes
  static constexpr int BOX = L > 256 ? 256 : L;
  static constexpr int NBOX = L / BOX;
  static constexpr bool TWS = L <= 256;
  static constexpr int TWF = tw_size<L, false>(), TWI = tw_size<L, true>();
  static constexpr size_t TWB = TWS ? (size_t)(TWF + TWI) * 16 : 0;
  static constexpr size_t SMEM = (size_t)S * STAGE + 3 * 64 + 64 + TWB + 1024;   // barriers, counts, twiddles, alignment
  static_assert(B * TP % 32 == 0 && S <= 8, "whole warps per tile");
};

template <int L, int OP, bool CONTIG, int B, int S, int NG, int MINB>
__global__ void __launch_bounds__(WarpSweep<L, CONTIG, B, S, NG>::NT, MINB) k_warp_sweep(const __grid_constant__ TmaSweepArgs a) {
  using G = WarpSweep<L, CONTIG, B, S, NG>;
  extern __shared__ __align__(128) unsigned char smraw[];
  const uint32_t raw = smem_u32(smraw);
  const uint32_t pad = ((raw + 1023u) & ~1023u) - raw;
  const uint32_t buf = raw + pad;
  uint64_t* full = reinterpret_cast<uint64_t*>(smraw + pad + (size_t)S * G::STAGE);   // the stage's copy landed
  uint64_t* empty = full + 8;                                                         // its result is written
  uint64_t* freed = full + 16;                                                        // its store has read it
  volatile int* issued = reinterpret_cast<volatile int*>(full + 24);                  // loads issued per stage
  float4* tws = reinterpret_cast<float4*>(full + 32);
  const int tid = threadIdx.x;
  constexpr int per_field = CONTIG ? L * L / B : (L / B) * L;
  const int total = per_field * a.count;
  const int mine = total > (int)blockIdx.x ? (total - blockIdx.x + gridDim.x - 1) / gridDim.x : 0;   // tiles of this CTA
  if (tid == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], G::NW);
      mbar_init(&freed[s], 1);
      issued[s] = 0;
    }
    fence_mbar_init();
  }
  if constexpr (G::TWS) {
    for (int i = tid; i < G::TWF; i += blockDim.x) tws[i] = a.tw_fwd[i];
    for (int i = tid; i < G::TWI; i += blockDim.x) tws[G::TWF + i] = a.tw_inv[i];
  }
  __syncthreads();

  if (tid >= G::NCT) {
    if ((tid - G::NCT) % 32 != 0) return;
    auto copy = [&](int it, bool load) {
      const int tile = blockIdx.x + it * gridDim.x, s = it % S;
      const int f = tile / per_field, r = tile - f * per_field;
      const uint32_t st = buf + (uint32_t)s * G::STAGE;
      if constexpr (CONTIG) {
        float2* g = a.psi[f] + (size_t)r * B * L;
#pragma unroll
        for (int q = 0; q < B; ++q) {
          const uint32_t row = st + (uint32_t)(q * WarpContig<L>::pitch()) * 8;
          if (load) bulk_load(row, g + (size_t)q * L, L * 8, &full[s]);
          else bulk_store(g + (size_t)q * L, row, L * 8);
        }
      } else {
        const int x0 = (r % (L / B)) * B, c = r / (L / B);
#pragma unroll
        for (int k = 0; k < G::NBOX; ++k) {
          unsigned char* p = smraw + pad + (size_t)s * G::STAGE + (size_t)k * G::BOX * B * 8;
          const int c1 = a.axis == 1 ? k * G::BOX : c, c2 = a.axis == 1 ? c : k * G::BOX;
          if (load) tma_load_3d(p, &a.map[f], &full[s], x0, c1, c2);
          else tma_store_3d(&a.map[f], p, x0, c1, c2);
        }
      }
    };
    auto wait = [&](uint64_t* bar, unsigned parity) { return mbar_wait_bounded(bar, parity); };
    if (tid == G::NCT) {
      // loader: tile it goes into stage it % S once the storer has freed it
      int it = 0;
      for (; it < mine; ++it) {
        const int s = it % S;
        if (it >= S && !wait(&freed[s], (unsigned)(it / S - 1) & 1u)) {
          atomicExch(a.status, 1);
          break;
        }
        mbar_expect_tx(&full[s], (unsigned)(B * L) * 8u);
        copy(it, true);
        if constexpr (NG > 1) count_issued(issued + s);
      }
      // loads in flight land before the CTA's shared memory goes away, also when a wait gave up
      for (int q = it > S ? it - S : 0; q < it; ++q) wait(&full[q % S], (unsigned)(q / S) & 1u);
    } else {
      // storer
      for (int it = 0; it < mine; ++it) {
        const int s = it % S;
        if (!wait(&empty[s], (unsigned)(it / S) & 1u)) {
          atomicExch(a.status, 1);
          break;
        }
        copy(it, false);
        bulk_commit();
        if (it + S < mine) {
          bulk_wait_read0();
          mbar_arrive(&freed[s]);
        }
      }
      bulk_wait_all();
    }
    return;
  }

  SweepArgs<float> sa{};
  sa.tw_fwd = G::TWS ? tws : a.tw_fwd;
  sa.tw_inv = G::TWS ? tws + G::TWF : a.tw_inv;
  sa.ekx = a.ekx;
  sa.ek2 = a.ek2;
  sa.nl_coef = a.nl_coef;
  sa.nl_shift = a.nl_shift;
  sa.scale_inv = a.scale_inv;
  const int wid = tid >> 5, lane = tid & 31, grp = wid / G::NW;
  using Acc = std::conditional_t<CONTIG, WarpContig<L>, WarpStrided<L, CONTIG ? 16 : B>>;
  Acc A(wid % G::NW, lane);
  for (int it = grp; it < mine; it += NG) {
    const int s = it % S;
    const bool ok = NG > 1 ? stage_wait(&full[s], issued + s, it, S) : mbar_wait_bounded(&full[s], (unsigned)(it / S) & 1u);
    if (!__all_sync(0xffffffffu, ok)) {
      if (lane == 0) atomicExch(a.status, 1);
      break;
    }
    A.at(buf + (uint32_t)s * G::STAGE);
    int i1 = 0, i2 = 0;
    if constexpr (CONTIG) {
      const int tile = blockIdx.x + it * gridDim.x;
      const int row = (tile % per_field) * B + A.p;
      i1 = row % L;
      i2 = row / L;
    }
    warp_op<OP, L, Acc, G::TWS>(sa, A, i1, i2);
    fence_async_smem();
    __syncwarp();
    if (lane == 0) mbar_arrive(&empty[s]);
  }
}

// ---------------------------------------------------------------- configurations and launch
// Tiles and stages per length and axis: (pencils B, stages S, compute groups NG, CTAs per SM MINB the
// registers must allow) of a kind's configurations 0, 1 and 2 (the sweep variants TMA, TMA_2STAGE and
// TMA_GROUPS; see WarpLaunch).
struct WarpCfg { int B, S, NG, MINB; };
template <int L> __host__ __device__ constexpr WarpCfg warp_cfg(int axis, int v) {
  if (L == 256) return axis != 0 && v == 1 ? WarpCfg{16, 2, 1, 3} : WarpCfg{16, 3, 1, 2};
  if (L == 512) {
    if (axis == 2) return v == 1 ? WarpCfg{16, 2, 1, 1} : (v == 2 ? WarpCfg{16, 3, 1, 1} : WarpCfg{16, 3, 2, 1});
    return v == 2 ? WarpCfg{8, 3, 2, 2} : WarpCfg{8, 6, 4, 1};   // x
  }
  if (axis == 0) return v == 2 ? WarpCfg{4, 3, 2, 2} : WarpCfg{4, 6, 4, 1};
  return v == 1 ? WarpCfg{8, 2, 1, 1} : (v == 2 ? WarpCfg{8, 3, 2, 1} : WarpCfg{8, 3, 1, 1});   // y
}

template <int L> struct WarpLaunch {
  template <int AXIS, int V, int OP> static constexpr auto kernel() {
    constexpr WarpCfg c = warp_cfg<L>(AXIS, V);
    return k_warp_sweep<L, OP, AXIS == 0, c.B, c.S, c.NG, c.MINB>;
  }
  template <int AXIS, int V> using Geo =
      WarpSweep<L, AXIS == 0, warp_cfg<L>(AXIS, V).B, warp_cfg<L>(AXIS, V).S, warp_cfg<L>(AXIS, V).NG>;
  static constexpr int NV = L >= 512 ? 3 : 2;   // configurations of a y or z sweep
  template <int AXIS, int V, int OP> static int query() {
    int nb = 0;
    cudaFuncSetAttribute(kernel<AXIS, V, OP>(), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Geo<AXIS, V>::SMEM);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kernel<AXIS, V, OP>(), Geo<AXIS, V>::NT, Geo<AXIS, V>::SMEM);
    return nb;
  }
  // CTAs per SM of every kernel of this length, queried together on the first launch of the length
  // (which is never inside a stream capture: a step's first sweeps run directly)
  struct Occ { int n[3][3][8]; };
  template <int AXIS, int V> static void fill(Occ& o) {
    if constexpr (AXIS == 0) {
#define GP_Q(OPV) o.n[AXIS][V][OPV] = query<AXIS, V, OPV>();
      GP_CONTIG_OPS(GP_Q)
    } else {
      GP_STRIDED_OPS(GP_Q)
#undef GP_Q
    }
  }
  static const Occ& occ() {
    static const Occ o = [] {
      Occ q{};
      fill<0, 0>(q);
      if constexpr (warp_axis<L>(1)) fill<1, 0>(q), fill<1, 1>(q);
      if constexpr (!ztile_ok<L>()) fill<2, 0>(q), fill<2, 1>(q);
      if constexpr (NV > 2 && warp_axis<L>(1)) fill<1, 2>(q);
      if constexpr (NV > 2) fill<0, 2>(q);
      if constexpr (NV > 2 && !ztile_ok<L>()) fill<2, 2>(q);
      return q;
    }();
    return o;
  }
  template <int AXIS, int V, int OP> static cudaError_t run(const TmaSweepArgs& a, int cap, cudaStream_t s) {
    constexpr WarpCfg c = warp_cfg<L>(AXIS, V);
    int per = occ().n[AXIS][V][OP];
    if (per < 1) return cudaErrorInvalidConfiguration;
    if (cap > 0 && cap < per) per = cap;
    const int tiles = (L / c.B) * L * a.count;
    int grid = TmaLaunch<L>::sms() * per;
    if (grid > tiles) grid = tiles;
    kernel<AXIS, V, OP>()<<<grid, Geo<AXIS, V>::NT, Geo<AXIS, V>::SMEM, s>>>(a);
    return cudaGetLastError();
  }
  template <int AXIS, int V> static cudaError_t run_op(const TmaSweepArgs& a, int cap, cudaStream_t s) {
#define GP_R(OPV) case OPV: return run<AXIS, V, OPV>(a, cap, s);
    if constexpr (AXIS == 0) {
      switch (a.op) { GP_CONTIG_OPS(GP_R) default: return cudaErrorInvalidValue; }
    } else {
      switch (a.op) { GP_STRIDED_OPS(GP_R) default: return cudaErrorInvalidValue; }
    }
#undef GP_R
  }
  static cudaError_t launch(const TmaSweepArgs& a, int cap, int stages, int groups, cudaStream_t s) {
    if constexpr (ztile_ok<L>()) {
      if (a.axis == 2 && (groups == 1 || groups == 2)) return ZTileLaunch<L>::launch(a, s);   // whatever the variant
    }
    if constexpr (!warp_axis<L>(1)) {
      if (a.axis == 1 && groups == 1) return TmaLaunch<L>::launch(a, cap, stages, 1, s);
    }
    if (groups == 2) {
      if constexpr (NV > 2) {
        if (a.axis == 0) return run_op<0, 2>(a, cap, s);
        if constexpr (!ztile_ok<L>()) {
          if (a.axis == 2) return run_op<2, 2>(a, cap, s);
        }
        if constexpr (warp_axis<L>(1)) return run_op<1, 2>(a, cap, s);
        else return TmaLaunch<L>::launch(a, cap, 3, 1, s);
      }
    }
    if (groups != 1) return cudaErrorInvalidValue;
    if (a.axis == 0) return run_op<0, 0>(a, cap, s);
    if constexpr (!ztile_ok<L>()) {
      if (a.axis == 2) return stages == 2 ? run_op<2, 1>(a, cap, s) : run_op<2, 0>(a, cap, s);
    }
    if constexpr (warp_axis<L>(1)) return stages == 2 ? run_op<1, 1>(a, cap, s) : run_op<1, 0>(a, cap, s);
    else return cudaErrorInvalidValue;
  }
};

}  // namespace gp
