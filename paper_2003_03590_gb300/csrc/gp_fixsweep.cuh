// gp_fixsweep.cuh -- the sweeps of float64 fields: the operations and tiles of gp_sweep.cuh with the
// arithmetic of gp_fix.cuh.  A tile's pencils are read as float64, brought to the pencil's fixed-point
// scale, transformed (register radix passes with exchanges through shared memory), and written back
// as float64; between an inverse and a forward transform the flows are applied in fixed point too.
//
// What bounds it: the issue of integer instructions (224 per point for a forward transform of 256 points
// with its conversions, 45-58% of the issue slots used).  256^3 on GB300, one sweep: forward transform
// 0.73 ms in float64, 0.22 ms now (its memory traffic takes 0.08 ms); inverse, N, forward 0.53 ms,
// forward, K, inverse 0.43 ms (in float64 as separate passes 2.4 and 1.9 ms).  With the conversions in
// integer instructions too a forward transform took 0.38 ms.
// A tile holds 16 pencils (y/z; 8 at 1024) or as many rows as 256 threads transform; 128 registers a
// thread for the lengths with 16 elements per thread or fewer, so that two CTAs share an SM.
#pragma once
#include "gp_fix.cuh"
#include "gp_sweep.cuh"

namespace gp {

struct FixArgs {
  double2* psi[GP_MAXB];   // device fields, N^3 each, [z][y][x]; field blockIdx.y
  int count;
  const ufix2* tw_fwd;     // Stockham twiddles of both directions
  const ufix2* tw_inv;
  const ufix2* ek;         // exp(-i alpha s k^2) by grid index, N entries, then the products of two, index i2 * N + i1
  const ufix2* dir;        // the 256 directions of gp_fix.cuh's fnonlinear
  NlFix nl;
  int op, axis;
  int bad;                 // 1: the flow's phase is not finite; no kernel is launched, sweep() writes NaN
  int scale_inv;           // 1: inverse ops multiply by 1/N; 0: normalisation done with K (1/N^3)
};

__device__ __forceinline__ ufix2 ldg_u2(const ufix2* q) {
  const ulonglong2 v = __ldg(reinterpret_cast<const ulonglong2*>(q));
  return ufix2{v.x, v.y};
}

// powers of two and of three in a length, and log2
template <int L> __host__ __device__ constexpr int pow2_of() { return L % 2 == 0 ? 1 + pow2_of<(L % 2 == 0 ? L / 2 : 1)>() : 0; }
template <> __host__ __device__ constexpr int pow2_of<1>() { return 0; }

// 2^d as a float for d <= 0 (0 below 2^-120)
__device__ __forceinline__ float pow2f(int d) { return d < -120 ? 0.0f : __int_as_float((127 + d) << 23); }

// the scale of a pencil that holds an infinity or a NaN
constexpr int FIX_NOT_FINITE = -100000;
// The scale of this thread's pencil: the largest s with 2^s sum |z_i| <= 2^62, from each thread's sum
// f 2^e.  The same on every thread of the pencil and on every call.  red: 2 TP B words (y/z tiles).
template <int TP, int B, bool CONTIG> __device__ __forceinline__ int pencil_scale(int e, float f, int t, int p, int* red) {
  int em = e;
  float sum;
  if constexpr (CONTIG) {
#pragma unroll
    for (int o = TP / 2; o > 0; o >>= 1) em = max(em, __shfl_xor_sync(0xffffffffu, em, o));
    sum = f * pow2f(e - em);
#pragma unroll
    for (int o = TP / 2; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  } else if constexpr (TP == 1) {
    sum = f;
  } else {
    float* rf = reinterpret_cast<float*>(red + TP * B);
    __syncthreads();                 // an earlier use of red
    red[t * B + p] = e;
    rf[t * B + p] = f;
    __syncthreads();
#pragma unroll
    for (int q = 0; q < TP; ++q) em = max(em, red[q * B + p]);
    sum = 0.0f;
#pragma unroll
    for (int q = 0; q < TP; ++q) sum += rf[q * B + p] * pow2f(red[q * B + p] - em);
  }
  const int k = (int)(__float_as_uint(sum * 1.0002f + 1e-30f) >> 23) - 126;   // sum < 2^k
  return em >= 1024 ? FIX_NOT_FINITE : 62 - k - em;
}

// largest exponent field and bound of the sum of moduli (relative to it) of E float64 values, from the
// high words: their 20 mantissa bits give an upper bound within 2^-20
template <int E> __device__ __forceinline__ void sum_of_doubles(const cfix* v, int& ref, float& f) {
  int m = 1 << 20;
#pragma unroll
  for (int e = 0; e < E; ++e) m = max(m, max((int)(v[e].x >> 32) & 0x7fffffff, (int)(v[e].y >> 32) & 0x7fffffff));
  ref = m >> 20;
  const int off = (ref - 127) << 20;
  f = 0.0f;
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int a = max(((int)(v[e].x >> 32) & 0x7fffffff) - off, 0), b = max(((int)(v[e].y >> 32) & 0x7fffffff) - off, 0);
    f += mod_bound(__int_as_float((a << 3) | 7), __int_as_float((b << 3) | 7));
  }
}
// bound of the sum of moduli of E fixed-point values, in units of 2^32
template <int E> __device__ __forceinline__ float sum_of_fixed(const cfix* v) {
  float f = 0.0f;
#pragma unroll
  for (int e = 0; e < E; ++e)
    f += mod_bound((float)(abs((int)(v[e].x >> 32)) + 1), (float)(abs((int)(v[e].y >> 32)) + 1));
  return f;
}

// Conversions of E values.  The hardware's float64 <-> int64 conversions (they use the float64 pipe,
// which nothing else here needs) with the scale added to the exponent field; for scales near the ends
// of the float64 range the integer routines of gp_fix.cuh.
static __device__ __noinline__ long long to_fix_slow(long long bits, int s) { return to_fix((unsigned long long)bits, s); }
static __device__ __noinline__ long long from_fix_slow(long long v, int s) { return (long long)from_fix(v, s); }
constexpr int FIX_FAST = 900;
__device__ __forceinline__ long long to_fix_fast(long long bits, int s) {
  const int hi = (int)(bits >> 32), e = (hi >> 20) & 0x7ff;
  const double d = __hiloint2double(e + s > 0 ? hi + (s << 20) : 0, (int)bits);   // |d| 2^s < 2^62
  return __double2ll_rn(d);
}
__device__ __forceinline__ long long from_fix_fast(long long v, int s) {
  const double d = __ll2double_rn(v);
  const int hi = __double2hiint(d);
  return __double_as_longlong(__hiloint2double(hi != 0 ? hi - (s << 20) : 0, __double2loint(d)));
}
template <int E> __device__ __forceinline__ void to_fix_all(cfix* v, int s) {
  if (s > -FIX_FAST && s < FIX_FAST) {
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = cfix{to_fix_fast(v[e].x, s), to_fix_fast(v[e].y, s)};
  } else {
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = cfix{to_fix_slow(v[e].x, s), to_fix_slow(v[e].y, s)};
  }
}
template <int E> __device__ __forceinline__ void from_fix_all(cfix* v, int s) {
  if (s > -FIX_FAST && s < FIX_FAST) {
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = cfix{from_fix_fast(v[e].x, s), from_fix_fast(v[e].y, s)};
  } else {
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = cfix{from_fix_slow(v[e].x, s), from_fix_slow(v[e].y, s)};
  }
}

// ---------------------------------------------------------------- transform
template <int L, bool INV, int I> __device__ __forceinline__ void fix_pass(cfix* v, int t, const ufix2* __restrict__ tw) {
  constexpr int R = radix_of<L, INV>(I), NS = span_of<L, INV>(I), E = Plan<L>::E, TP = L / E;
#pragma unroll
  for (int b = 0; b < E / R; ++b) {
    if constexpr (NS > 1) {
      const ufix2* q = tw + tw_offset<L, INV>(I) + (t + b * TP) % NS;
#pragma unroll
      for (int r = 1; r < R; ++r) v[b * R + r] = ftwmul(v[b * R + r], ldg_u2(q + (r - 1) * NS));
    }
    fdft<R, INV>(v + b * R);
  }
}
template <int L, bool INV, int I, class Lay> __device__ __forceinline__ void fix_store(const cfix* v, int t, int p, cfix* sm, const Lay& lay) {
  constexpr int R = radix_of<L, INV>(I), NS = span_of<L, INV>(I), E = Plan<L>::E, TP = L / E;
#pragma unroll
  for (int b = 0; b < E / R; ++b) {
    const int j = t + b * TP, d = (j / NS) * NS * R + (j % NS);
#pragma unroll
    for (int r = 0; r < R; ++r)
      *reinterpret_cast<longlong2*>(sm + lay.template at<INV, I>(p, d + r * NS)) = make_longlong2(v[b * R + r].x, v[b * R + r].y);
  }
}
template <int L, bool INV, int I, class Lay> __device__ __forceinline__ void fix_load(cfix* v, int t, int p, const cfix* sm, const Lay& lay) {
  constexpr int R = radix_of<L, INV>(I), E = Plan<L>::E, TP = L / E;
#pragma unroll
  for (int b = 0; b < E / R; ++b)
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const longlong2 q = *reinterpret_cast<const longlong2*>(sm + lay.template at<INV, I - 1>(p, t + b * TP + r * (L / R)));
      v[b * R + r] = cfix{q.x, q.y};
    }
}
template <int L, bool INV, bool WARP_X, class Lay>
__device__ __forceinline__ void fix_fft(cfix* v, int t, int p, cfix* sm, const Lay& lay, const ufix2* __restrict__ tw) {
  constexpr int NP = Plan<L>::NP;
  fix_pass<L, INV, 0>(v, t, tw);
  if constexpr (NP > 1) {
    xsync<WARP_X>();   // an earlier exchange's reads
    fix_store<L, INV, 0>(v, t, p, sm, lay);
    xsync<WARP_X>();
    fix_load<L, INV, 1>(v, t, p, sm, lay);
    fix_pass<L, INV, 1>(v, t, tw);
  }
  if constexpr (NP > 2) {
    xsync<WARP_X>();
    fix_store<L, INV, 1>(v, t, p, sm, lay);
    xsync<WARP_X>();
    fix_load<L, INV, 2>(v, t, p, sm, lay);
    fix_pass<L, INV, 2>(v, t, tw);
  }
}

// ---------------------------------------------------------------- one tile
template <int OP, int L, int B, bool CONTIG, class Lay, class GetAddr>
__device__ __forceinline__ void fix_op(const FixArgs& a, int t, int p, cfix* sm, int* red, const Lay& lay, const GetAddr& addr,
                                       int i1, int i2) {
  constexpr int E = Plan<L>::E, TP = L / E;
  constexpr bool WARP_X = CONTIG;
  constexpr bool IN_INV = OP == OP_INV || OP == OP_INV_N || OP == OP_INV_N_FWD;
  constexpr bool OUT_INV = OP == OP_INV || OP == OP_INV_N || OP == OP_FWD_K_INV;
  constexpr bool N3 = L % 3 == 0;
  cfix v[E];
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const longlong2 q = *reinterpret_cast<const longlong2*>(addr(in_pos<L, IN_INV>(e, t)));
    v[e] = cfix{q.x, q.y};
  }
  int ref, s;
  float f;
  sum_of_doubles<E>(v, ref, f);
  s = pencil_scale<TP, B, CONTIG>(ref - 1023, f, t, p, red);
  // N on values at this thread's own scale st (pointwise: no headroom is needed), then the pencil's
  auto flow = [&](int st) {
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = fnonlinear(v[e], 2 * st + a.nl.q - 126, a.nl.m, a.nl.tc, a.nl.neg, a.dir);
  };
  auto to_scale = [&](int r) {
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = cfix{rescale1(v[e].x, r), rescale1(v[e].y, r)};
  };
  const bool bad = s == FIX_NOT_FINITE;   // every value of the pencil becomes NaN
  if (bad) s = 0;
  {
    const int s0 = OP == OP_N_FWD ? 1084 - ref : s;
    to_fix_all<E>(v, s0);
    if constexpr (OP == OP_N_FWD) {
      flow(s0);
      to_scale(s0 - s);
    }
  }
  if constexpr (OP == OP_FWD || OP == OP_N_FWD || OP == OP_FWD_K_INV) fix_fft<L, false, WARP_X>(v, t, p, sm, lay, a.tw_fwd);
  if constexpr (IN_INV) {
    fix_fft<L, true, WARP_X>(v, t, p, sm, lay, a.tw_inv);
    if (a.scale_inv) {   // 1/L: the power of two by the scale, 1/3 = (2/3)/2 by a product
      if constexpr (N3) {
#pragma unroll
        for (int e = 0; e < E; ++e) v[e] = cfix{fmulc(v[e].x, FIX_23), fmulc(v[e].y, FIX_23)};
      }
      s += pow2_of<L>() + (N3 ? 1 : 0);
    }
  }
  if constexpr (OP == OP_INV_N || OP == OP_INV_N_FWD) {
    unsigned m = 0;
#pragma unroll
    for (int e = 0; e < E; ++e) m |= (unsigned)abs((int)(v[e].x >> 32)) | (unsigned)abs((int)(v[e].y >> 32));
    const int h = max(0, __clz(m + 1) - 2);   // |components| 2^h < 2^62 (the high words are rounded down)
    to_scale(-h);
    s += h;
    flow(s);
  }
  if constexpr (OP == OP_INV_N_FWD) {
    const int sn = pencil_scale<TP, B, CONTIG>(32 - s, sum_of_fixed<E>(v), t, p, red);
    to_scale(s - sn);
    s = sn;
    fix_fft<L, false, WARP_X>(v, t, p, sm, lay, a.tw_fwd);
  }
  if constexpr (OP == OP_FWD_K_INV) {
    const ufix2 eo = ldg_u2(a.ek + L + i2 * L + i1);   // carries (16/27) for lengths 3 2^k
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = ftwmul(ftwmul(v[e], ldg_u2(a.ek + out_pos<L, false>(e, t))), eo);
    const int sn = pencil_scale<TP, B, CONTIG>(32 - s, sum_of_fixed<E>(v), t, p, red);
    to_scale(s - sn);
    s = sn + 3 * pow2_of<L>() + (N3 ? 4 : 0);          // 1/N^3
    fix_fft<L, true, WARP_X>(v, t, p, sm, lay, a.tw_inv);
  }
  from_fix_all<E>(v, s);
  if (bad) {
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = cfix{0x7ff8000000000000ll, 0x7ff8000000000000ll};
  }
#pragma unroll
  for (int e = 0; e < E; ++e)
    *reinterpret_cast<longlong2*>(addr(out_pos<L, OUT_INV>(e, t))) = make_longlong2(v[e].x, v[e].y);
}

template <int L> __host__ __device__ constexpr int fix_min_ctas() { return Plan<L>::E <= 16 ? 2 : 1; }

template <int L, int OP>
__global__ void __launch_bounds__(strided_batch<double, L>() * (L / Plan<L>::E), fix_min_ctas<L>()) k_fix_strided(const __grid_constant__ FixArgs a) {
  extern __shared__ __align__(16) unsigned char smraw[];
  constexpr int B = strided_batch<double, L>(), TP = L / Plan<L>::E;
  cfix* sm = reinterpret_cast<cfix*>(smraw);
  int* red = reinterpret_cast<int*>(smraw + sizeof(cfix) * (size_t)L * B);
  const int tid = threadIdx.x, p = tid % B, t = tid / B;
  const long st = (a.axis == 1) ? (long)L : (long)L * L;
  const long sc = (a.axis == 1) ? (long)L * L : (long)L;
  const int tile = blockIdx.x, x0 = (tile % (L / B)) * B, c = tile / (L / B);
  double2* base = a.psi[blockIdx.y] + x0 + p + (long)c * sc;
  auto addr = [&](int pos) { return base + (long)pos * st; };
  LayStrided lay{B};
  fix_op<OP, L, B, false>(a, t, p, sm, red, lay, addr, 0, 0);
}
template <int L, int OP>
__global__ void __launch_bounds__(contig_batch<double, L>() * (L / Plan<L>::E), fix_min_ctas<L>()) k_fix_contig(const __grid_constant__ FixArgs a) {
  extern __shared__ __align__(16) unsigned char smraw[];
  constexpr int B = contig_batch<double, L>(), TP = L / Plan<L>::E;
  static_assert(TP <= 32, "a row's threads lie in one warp");
  cfix* sm = reinterpret_cast<cfix*>(smraw);
  const int p = threadIdx.x / TP, t = threadIdx.x % TP;
  const long row = (long)blockIdx.x * B + p;
  double2* base = a.psi[blockIdx.y] + row * L;
  auto addr = [&](int pos) { return base + pos; };
  LayContig<L> lay;
  fix_op<OP, L, B, true>(a, t, p, sm, nullptr, lay, addr, (int)(row % L), (int)(row / L));
}

template <int L> struct FixLaunch {
  static constexpr int TP = L / Plan<L>::E;
  static constexpr int BS = strided_batch<double, L>(), BC = contig_batch<double, L>();
  static constexpr size_t smem_strided() { return sizeof(cfix) * (size_t)L * BS + 8 * (size_t)TP * BS; }
  static constexpr size_t smem_contig() { return sizeof(cfix) * (size_t)contig_pitch<L>() * BC; }
  // the shared-memory limit of every kernel, set together on the first launch of this length (never
  // inside a stream capture: a step's first sweeps run directly)
  static bool set_attributes() {
    static const bool done = [] {
#define GP_ATTR_C(OPV) cudaFuncSetAttribute(k_fix_contig<L, OPV>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_contig());
#define GP_ATTR_S(OPV) cudaFuncSetAttribute(k_fix_strided<L, OPV>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_strided());
      GP_CONTIG_OPS(GP_ATTR_C)
      GP_STRIDED_OPS(GP_ATTR_S)
#undef GP_ATTR_C
#undef GP_ATTR_S
      return true;
    }();
    return done;
  }
  static cudaError_t launch(const FixArgs& a, cudaStream_t s) {
    set_attributes();
    const dim3 gc((unsigned)((long)L * L / BC), (unsigned)a.count), gs((unsigned)((L / BS) * L), (unsigned)a.count);
#define GP_OP_CASE_C(OPV) \
  case OPV: k_fix_contig<L, OPV><<<gc, BC * TP, smem_contig(), s>>>(a); break;
#define GP_OP_CASE_S(OPV) \
  case OPV: k_fix_strided<L, OPV><<<gs, BS * TP, smem_strided(), s>>>(a); break;
    if (a.axis == 0) {
      switch (a.op) { GP_CONTIG_OPS(GP_OP_CASE_C) default: return cudaErrorInvalidValue; }
    } else {
      switch (a.op) { GP_STRIDED_OPS(GP_OP_CASE_S) default: return cudaErrorInvalidValue; }
    }
#undef GP_OP_CASE_C
#undef GP_OP_CASE_S
    return cudaGetLastError();
  }
};

}  // namespace gp
