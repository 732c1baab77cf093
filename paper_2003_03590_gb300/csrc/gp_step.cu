// gp_step.cu -- the Strang split step (Sec. 4.3, eq:adi_looptime) as a schedule of HBM sweeps.
//
// float32 fields (fused): the field stays in a mixed representation between
// sweeps -- physical along x and y, Fourier along z -- so each step is four
// sweeps, every one a full read and write of the field:
//   z: inverse z, N(dt), forward z        y: forward y
//   x: forward x, K(dt), inverse x        y: inverse y
// The half-step nonlinear flows of consecutive NKN steps merge into N(dt)
// (N preserves |psi|, so N(a) N(b) = N(a + b)); the first and last sweeps of a
// call carry N(dt/2).  The KNK order is the same cycle with K(dt/2) at the two
// ends: KNK^m = K(h) N(h) [NKN]^(m-1) N(h) K(h).
// Fields of identical shape and parameters are advanced by the same launches
// (blockIdx.y selects the field), and the repeating four-sweep cycle is
// captured once in a CUDA graph and replayed.
//
// float64 fields run the same four-sweep cycle with the sweeps of gp_fixsweep.cuh.  (One kernel per
// sub-flow and axis, with unmerged half steps, took 9 or 15 launches and two N per step.)
#include <cmath>
#include <cstdio>
#include <string>
#include <vector>

#include "gp_internal.h"

namespace gp {

static long long tune_key(int n, int axis, int op) { return (long long)n * 64 + axis * 8 + op; }

int sweep_variant(gp_plan* p, int n, int axis, int op) {
  if (!p->use_tma || !tma_supported(n)) return VARIANT_PLAIN;
  const long long k = tune_key(n, axis, op);
  for (const auto& e : p->tune)
    if (e.first == k) return e.second;
  return VARIANT_DEFAULT;
}

// The kernel of a sweep kind unless one was chosen for the plan, by the length.  Measured on GB300, us per
// launch of one field (the batched steps order the same way):
//   y, x, y as the fused plane kernel / as three sweeps: 32^3 27 / 15, 64^3 29 / 15, 96^3 37 / 23, 128^3
//     39 / 30, 192^3 103 / 82, 256^3 144 / 153, 512^3 1600 / 1160, 1024^3 11500 / 9240: fused where its
//     planes both fill the GPU and are few enough to stay in L2, which is 256;
//   x sweeps (forward, K, inverse), TMA / one tile per CTA: 128^3 16.9 / 14.5, 192^3 45.6 / 41.5, 256^3 71 / 64,
//     512^3 526 / 491, 1024^3 4440 / 4100: rows are contiguous, direct loads lose nothing;
//   y and z up to 128 points: one step of 24 fields of 64^3 75 us with TMA kernels, 69 without, of 16 fields
//     of 96^3 251 / 242, of 8 fields of 128^3 220 / 203 (a CTA has few tiles to pipeline); at 192 two
//     stages: z inverse-N-forward 45.6 / 37.8 / 37.3 (three stages / one tile per CTA / two stages);
//   z at 1024, TMA / one tile per CTA: forward 3470 / 4900, inverse-N-forward 5440 / 7790.
int default_variant(int n, int axis, int op) {
  if (op == OP_PLANE) return n == 256 ? VARIANT_TMA : VARIANT_PLAIN;
  if (axis == 0 || n <= 128) return VARIANT_PLAIN;
  if (n == 192) return VARIANT_TMA_2STAGE;
  return VARIANT_TMA;
}
int kernel_variant(gp_plan* p, int n, int axis, int op) {
  const int v = sweep_variant(p, n, axis, op);
  if (v != VARIANT_DEFAULT) return v;
  if (op == OP_PLANE && p->plane_skip > 0) return VARIANT_TMA;   // gp_plan_test_timeout tests the fused kernel
  return default_variant(n, axis, op);
}

// forward y, x (forward, K, inverse) and inverse y of a step as one fused plane-kernel launch
bool plane_on(gp_plan* p, int n) {
  return kernel_variant(p, n, 1, OP_PLANE) != VARIANT_PLAIN;
}

gp_status ensure_plane_sync(gp_plan* p, size_t ints) {
  if (p->plane_sync_ints >= ints) return GP_OK;
  if (p->plane_sync) {
    GP_CUDA(p, p->stream ? cudaStreamSynchronize(p->stream) : cudaDeviceSynchronize());
    cudaFree(p->plane_sync);
    p->plane_sync = nullptr;
    p->plane_sync_ints = 0;
    // captured graphs hold the old counters' address: drop them
    if (p->cycle_graph) {
      cudaGraphExecDestroy(p->cycle_graph);
      p->cycle_graph = nullptr;
    }
    if (p->run_graph) {
      cudaGraphExecDestroy(p->run_graph);
      p->run_graph = nullptr;
    }
    p->cycle_key.clear();
    p->run_key.clear();
    p->last_key.clear();
  }
  if (cudaMalloc(&p->plane_sync, ints * sizeof(int)) != cudaSuccess) {
    p->plane_sync = nullptr;
    return fail(p, GP_ERR_OOM, "plane kernel counters");
  }
  p->plane_sync_ints = ints;
  return GP_OK;
}

cudaError_t launch_sweep_variant(gp_plan* p, int n, const SweepArgs<float>& a, void* const* psi, int variant,
                                 cudaStream_t s) {
  if (a.op == OP_PLANE) {
    if (variant != VARIANT_PLAIN) {
      const int skip = p->plane_skip;
      p->plane_skip = 0;
      return tma_plane(n, a, psi, p->plane_sync, p->flag + 1, s, variant == VARIANT_TMA_2STAGE ? 2 : 3, skip,
                       variant == VARIANT_TMA_ONE ? 1 : 0, variant == VARIANT_TMA_GROUPS ? 2 : 1);
    }
    SweepArgs<float> b = a;
    const int ops[3][2] = {{1, OP_FWD}, {0, OP_FWD_K_INV}, {1, OP_INV}};
    for (const auto& o : ops) {
      b.axis = o[0];
      b.op = o[1];
      cudaError_t e = launch_sweep_variant(p, n, b, psi, kernel_variant(p, n, b.axis, b.op), s);
      if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
  }
  if (variant == VARIANT_PLAIN) return sweep(n, a, s);
  if (variant == VARIANT_TMA_2STAGE && a.axis != 0) return tma_sweep(n, a, psi, p->flag + 1, s, 0, 2);
  if (variant == VARIANT_TMA_GROUPS) return tma_sweep(n, a, psi, p->flag + 1, s, 0, 3, 2);
  return tma_sweep(n, a, psi, p->flag + 1, s, variant == VARIANT_TMA_ONE ? 1 : 0);
}

// one axis' transform of `count` float32 fields in one launch
cudaError_t fft1_many(gp_plan* p, FieldPlan& F, cpx<float>* const* xs, int count, int axis, bool inverse, cudaStream_t s) {
  SweepArgs<float> a{};
  a.count = count;
  void* ptrs[GP_MAXB];
  for (int k = 0; k < count; ++k) ptrs[k] = a.psi[k] = xs[k];
  a.tw_fwd = (const tw_t<float>*)F.t32.tw_fwd;
  a.tw_inv = (const tw_t<float>*)F.t32.tw_inv;
  a.op = inverse ? OP_INV : OP_FWD;
  a.scale_inv = 1;
  a.axis = axis;
  return launch_sweep_variant(p, F.n, a, ptrs, kernel_variant(p, F.n, a.axis, a.op), s);
}
// 3D transforms of `count` float32 fields of one plan length, one launch per axis for all of
// them, through the kernel variants chosen for the forward and inverse y/z sweeps (x: the default, plain)
cudaError_t fft3_many(gp_plan* p, FieldPlan& F, cpx<float>* const* xs, int count, bool inverse, cudaStream_t s) {
  const int order_f[3] = {0, 1, 2}, order_i[3] = {2, 1, 0};
  for (int i = 0; i < 3; ++i) {
    cudaError_t e = fft1_many(p, F, xs, count, inverse ? order_i[i] : order_f[i], inverse, s);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

namespace {

struct Group {
  std::vector<int> fields;
  int n = 0;
  bool fp64 = false;
  int split = 0;
};

struct Item {
  int group;
  int axis;
  int op;
  double s_nl;  // time of the nonlinear flow
  double s_k;   // time of the kinetic flow
};

bool same_shape(const gp_field_params& a, const gp_field_params& b, const FieldPlan& fa, const FieldPlan& fb) {
  return a.n == b.n && a.precision == b.precision && a.split == b.split && a.dt == b.dt &&
         a.nonlin_minus_one == b.nonlin_minus_one && fa.alpha == fb.alpha && fa.beta == fb.beta;
}

// whether two float64 fields of the plan share memory
bool f64_shared(gp_plan* p, void* const* psi) {
  for (size_t i = 0; i < p->f.size(); ++i)
    for (size_t j = 0; j < i && p->f[i].fp64; ++j) {
      if (!p->f[j].fp64) continue;
      const uintptr_t a = (uintptr_t)psi[i], b = (uintptr_t)psi[j];
      if (a < b + (size_t)p->f[j].npts * sizeof(double2) && b < a + (size_t)p->f[i].npts * sizeof(double2)) return true;
    }
  return false;
}

// f64: float64 fields too
std::vector<Group> make_groups(gp_plan* p, bool f64) {
  std::vector<Group> g;
  for (int i = 0; i < (int)p->f.size(); ++i) {
    if (p->f[i].fp64 && !f64) continue;
    bool placed = false;
    for (auto& G : g) {
      const int j = G.fields[0];
      if ((int)G.fields.size() < GP_MAXB && same_shape(p->f[i].prm, p->f[j].prm, p->f[i], p->f[j])) {
        G.fields.push_back(i);
        placed = true;
        break;
      }
    }
    if (!placed) {
      Group G;
      G.fields.push_back(i);
      G.n = p->f[i].n;
      G.fp64 = p->f[i].fp64;
      G.split = p->f[i].prm.split;
      g.push_back(G);
    }
  }
  return g;
}

gp_status launch_item(gp_plan* p, const Group& G, const Item& it, void* const* psi, cudaStream_t s) {
  FieldPlan& F = p->f[G.fields[0]];
  if (G.fp64) {
    const void* kt = nullptr;
    if (it.op == OP_FWD_K_INV && !(kt = ktable(p, G.fields[0], it.s_k, true)))
      return fail(p, GP_ERR_OOM, "kinetic table allocation");
    FixArgs a = fix_args(F, kt);
    a.count = (int)G.fields.size();
    for (int k = 0; k < a.count; ++k) a.psi[k] = (double2*)psi[G.fields[k]];
    a.op = it.op;
    a.axis = it.axis;
    a.nl = nl_fix(F.beta * it.s_nl, F.prm.nonlin_minus_one ? 1.0 : 0.0);
    if (!std::isfinite(F.beta * it.s_nl)) a.bad = 1;
    GP_CUDA(p, sweep(G.n, a, s));
    p->launches += 1;
    return GP_OK;
  }
  SweepArgs<float> a{};
  a.count = (int)G.fields.size();
  for (int k = 0; k < a.count; ++k) a.psi[k] = (cpx<float>*)psi[G.fields[k]];
  a.tw_fwd = (const tw_t<float>*)F.t32.tw_fwd;
  a.tw_inv = (const tw_t<float>*)F.t32.tw_inv;
  a.op = it.op;
  a.axis = it.axis;
  a.nl_coef = (float)(F.beta * it.s_nl);
  a.nl_shift = F.prm.nonlin_minus_one ? 1.0f : 0.0f;
  if (it.op == OP_FWD_K_INV || it.op == OP_PLANE) {
    const float4* kt = (const float4*)ktable(p, G.fields[0], it.s_k, false);
    if (!kt) return fail(p, GP_ERR_OOM, "kinetic table allocation");
    a.ekx = kt;
    a.ek2 = kt + G.n;   // includes the whole inverse normalisation 1/N^3
  }
  a.scale_inv = 0;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  if (p->prof) {
    static const char* opn[] = {"", "fwd", "inv", "inv_n_fwd", "n_fwd", "inv_n", "fwd_k_inv", "fwd_k_inv"};
    const bool tma = kernel_variant(p, G.n, it.axis, it.op) != VARIANT_PLAIN;
    std::string name = it.op == OP_PLANE ? std::string("k_tma_plane<") + std::to_string(G.n) + ">:y_fwd_x_fwd_k_inv_y_inv:xy"
                       : std::string(tma ? tma_kernel_name(G.n, it.axis) : plain_kernel_name(G.n, it.axis)) + std::to_string(G.n) + ">:" + opn[it.op] + ":" + "xyz"[it.axis];
    int kind = -1;
    for (int q = 0; q < (int)p->kinds.size(); ++q)
      if (p->kinds[q] == name) kind = q;
    if (kind < 0) {
      kind = (int)p->kinds.size();
      p->kinds.push_back(name);
    }
    GP_CUDA(p, cudaEventCreate(&e0));
    GP_CUDA(p, cudaEventCreate(&e1));
    GP_CUDA(p, cudaEventRecord(e0, s));
    p->ev_pool.push_back(e0);
    p->ev_pool.push_back(e1);
    p->ev_kind.push_back(kind);
  }
  void* ptrs[GP_MAXB];
  for (int k = 0; k < a.count; ++k) ptrs[k] = psi[G.fields[k]];
  cudaError_t e = launch_sweep_variant(p, G.n, a, ptrs, kernel_variant(p, G.n, it.axis, it.op), s);
  if (e != cudaSuccess) return cuda_fail(p, e, "sweep launch");
  if (p->prof) GP_CUDA(p, cudaEventRecord(e1, s));
  p->launches += 1;
  return GP_OK;
}

// the sweeps that carry K(sk): forward y, x (forward, K, inverse), inverse y -- three launches,
// or one of the fused plane kernel
void k_block(std::vector<Item>& v, int g, double sk, bool plane) {
  if (plane) {
    v.push_back({g, 1, OP_PLANE, 0.0, sk});
    return;
  }
  v.push_back({g, 1, OP_FWD, 0.0, 0.0});
  v.push_back({g, 0, OP_FWD_K_INV, 0.0, sk});
  v.push_back({g, 1, OP_INV, 0.0, 0.0});
}

gp_status run_items(gp_plan* p, const std::vector<Group>& groups, const std::vector<Item>& items, void* const* psi,
                    cudaStream_t s) {
  for (const Item& it : items) {
    gp_status st = launch_item(p, groups[it.group], it, psi, s);
    if (st != GP_OK) return st;
  }
  return GP_OK;
}

bool bad_ptr(const void* q) { return q == nullptr || ((uintptr_t)q & 15) != 0; }

// Record a sequence of item lists (each repeated) into one executable graph on a private stream.
gp_status capture(gp_plan* p, const std::vector<Group>& groups,
                  const std::vector<std::pair<const std::vector<Item>*, int>>& seq, void* const* psi,
                  cudaGraphExec_t* out) {
  cudaStream_t cap;
  GP_CUDA(p, cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking));
  cudaGraph_t graph = nullptr;
  gp_status st = GP_OK;
  cudaError_t e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
  if (e == cudaSuccess) {
    const long long before = p->launches;
    for (const auto& part : seq)
      for (int r = 0; r < part.second && st == GP_OK; ++r) st = run_items(p, groups, *part.first, psi, cap);
    p->launches = before;
    cudaError_t e2 = cudaStreamEndCapture(cap, &graph);
    if (st == GP_OK && e2 != cudaSuccess) st = cuda_fail(p, e2, "cudaStreamEndCapture");
  } else {
    st = cuda_fail(p, e, "cudaStreamBeginCapture");
  }
  cudaStreamDestroy(cap);
  if (st != GP_OK) {
    if (graph) cudaGraphDestroy(graph);
    return st;
  }
  e = cudaGraphInstantiate(out, graph, 0);
  cudaGraphDestroy(graph);
  if (e != cudaSuccess) {
    *out = nullptr;
    return cuda_fail(p, e, "cudaGraphInstantiate");
  }
  return GP_OK;
}

}  // namespace

// A whole NKN run of every field in one persistent launch (gp_ensemble.cu), captured in a graph
// with the counters' reset and replayed for a repeated call with the same fields and step count.
static bool fused_batch_ok(gp_plan* p) {
  if (!p->fused_batch || (int)p->f.size() > GP_ENS_MAXF) return false;
  for (const auto& F : p->f)
    if (F.fp64 || F.prm.split != GP_SPLIT_NKN || !ensemble_supported(F.n)) return false;
  return true;
}

static gp_status fused_batch_steps(gp_plan* p, void* const* psi, int nsteps) {
  std::vector<int> fields;
  for (int i = 0; i < (int)p->f.size(); ++i) {
    fields.push_back(i);
    if (!ktable(p, i, p->f[i].prm.dt, false)) return fail(p, GP_ERR_OOM, "kinetic table allocation");
  }
  gp_status st = ensure_plane_sync(p, ensemble_sync_ints(nsteps, (int)fields.size()));
  if (st != GP_OK) return st;
  cudaStream_t s = p->stream;
  if (p->plane_skip > 0) {   // gp_plan_test_timeout: one direct launch that skips leading tiles
    const int skip = p->plane_skip;
    p->plane_skip = 0;
    GP_CUDA(p, ensemble_run(p, fields, psi, nsteps, p->plane_sync, s, skip));
    p->launches += 1;
    return GP_OK;
  }
  std::vector<void*> key(psi, psi + p->f.size());
  key.push_back(nullptr);   // marks a fused-run graph
  if (p->prof) {
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    GP_CUDA(p, cudaEventCreate(&e0));
    GP_CUDA(p, cudaEventCreate(&e1));
    p->ev_pool.push_back(e0);
    p->ev_pool.push_back(e1);
    const std::string name = "k_ensemble_run:nkn_run:xyz";
    int kind = -1;
    for (int q = 0; q < (int)p->kinds.size(); ++q)
      if (p->kinds[q] == name) kind = q;
    if (kind < 0) {
      kind = (int)p->kinds.size();
      p->kinds.push_back(name);
    }
    p->ev_kind.push_back(kind);
    GP_CUDA(p, cudaEventRecord(e0, s));
    GP_CUDA(p, ensemble_run(p, fields, psi, nsteps, p->plane_sync, s));
    GP_CUDA(p, cudaEventRecord(e1, s));
    p->launches += 1;
    return GP_OK;
  }
  if (!(p->run_graph && p->run_key == key && p->run_steps == nsteps)) {
    GP_CUDA(p, ensemble_run(p, fields, psi, nsteps, p->plane_sync, s));   // first call: direct (sets attributes)
    p->launches += 1;
    cudaStream_t cap;
    GP_CUDA(p, cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking));
    cudaGraph_t graph = nullptr;
    cudaError_t e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
      e = ensemble_run(p, fields, psi, nsteps, p->plane_sync, cap);
      cudaError_t e2 = cudaStreamEndCapture(cap, &graph);
      if (e == cudaSuccess) e = e2;
    }
    cudaStreamDestroy(cap);
    if (e != cudaSuccess) {
      if (graph) cudaGraphDestroy(graph);
      return cuda_fail(p, e, "fused run capture");
    }
    cudaGraphExec_t g = nullptr;
    e = cudaGraphInstantiate(&g, graph, 0);
    cudaGraphDestroy(graph);
    if (e != cudaSuccess) return cuda_fail(p, e, "cudaGraphInstantiate");
    if (p->run_graph) cudaGraphExecDestroy(p->run_graph);
    p->run_graph = g;
    p->run_key = key;
    p->run_steps = nsteps;
    return GP_OK;
  }
  GP_CUDA(p, cudaGraphLaunch(p->run_graph, s));
  p->launches += 1;
  return GP_OK;
}

gp_status step_all(gp_plan* p, void* const* psi, int nsteps) {
  if (nsteps == 0) return GP_OK;
  if (fused_batch_ok(p)) return fused_batch_steps(p, psi, nsteps);
  // float64 fields that share memory are advanced one after the other, in the plan's order: the fields
  // of one launch, and the groups that take turns in the cycle, must not touch each other
  const bool in_turn = f64_shared(p, psi);
  if (in_turn) {
    for (int i = 0; i < (int)p->f.size(); ++i)   // tables first: no field changes if one cannot be had
      if (p->f[i].fp64 && (!ktable(p, i, p->f[i].prm.dt, true) || !ktable(p, i, 0.5 * p->f[i].prm.dt, true)))
        return fail(p, GP_ERR_OOM, "kinetic table allocation");
    for (int i = 0; i < (int)p->f.size(); ++i) {
      if (!p->f[i].fp64) continue;
      gp_status st = step_field(p, i, psi[i], nsteps);
      if (st != GP_OK) return st;
    }
  }
  std::vector<Group> groups = make_groups(p, !in_turn);
  if (groups.empty()) return GP_OK;
  cudaStream_t s = p->stream;
  for (int g = 0; g < (int)groups.size(); ++g) {
    const Group& G = groups[g];
    // tables are created before any capture starts
    const FieldPlan& F = p->f[G.fields[0]];
    if (!ktable(p, G.fields[0], F.prm.dt, G.fp64) || !ktable(p, G.fields[0], 0.5 * F.prm.dt, G.fp64))
      return fail(p, GP_ERR_OOM, "kinetic table allocation");
    if (!G.fp64 && plane_on(p, G.n)) {
      gp_status st = ensure_plane_sync(p, plane_sync_ints(G.n, (int)G.fields.size()));
      if (st != GP_OK) return st;
    }
  }

  std::vector<Item> pro, cyc, tail, epi;
  for (int g = 0; g < (int)groups.size(); ++g) {
    const Group& G = groups[g];
    const double dt = p->f[G.fields[0]].prm.dt, h = 0.5 * dt;
    const bool pl = !G.fp64 && plane_on(p, G.n);
    if (G.split == GP_SPLIT_NKN) {
      pro.push_back({g, 2, OP_N_FWD, h, 0.0});
      k_block(pro, g, dt, pl);
      epi.push_back({g, 2, OP_INV_N, h, 0.0});
    } else {
      pro.push_back({g, 2, OP_FWD, 0.0, 0.0});
      k_block(pro, g, h, pl);
      tail.push_back({g, 2, OP_INV_N_FWD, dt, 0.0});
      k_block(tail, g, h, pl);
      epi.push_back({g, 2, OP_INV, 0.0, 0.0});
    }
    cyc.push_back({g, 2, OP_INV_N_FWD, dt, 0.0});
    k_block(cyc, g, dt, pl);
  }
  const int ncycles = nsteps - 1;

  // in a caller's stream capture only kernels are launched: making a graph inside it is not allowed
  cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;
  GP_CUDA(p, cudaStreamIsCapturing(s, &capturing));
  const bool direct = p->prof || capturing != cudaStreamCaptureStatusNone;

  std::vector<void*> key(psi, psi + p->f.size());
  const long long whole = (long long)pro.size() + (long long)ncycles * (long long)cyc.size() + (long long)tail.size() +
                          (long long)epi.size();
  // a call repeated with the same fields and step count replays one graph of the whole run
  if (!direct && whole <= 8192 && p->run_graph && p->run_key == key && p->run_steps == nsteps) {
    GP_CUDA(p, cudaGraphLaunch(p->run_graph, s));
    p->launches += whole;
    return GP_OK;
  }
  if (!direct && whole <= 8192 && p->last_key == key && p->last_steps == nsteps) {
    std::vector<std::pair<const std::vector<Item>*, int>> seq = {{&pro, 1}, {&cyc, ncycles}, {&tail, 1}, {&epi, 1}};
    cudaGraphExec_t g = nullptr;
    gp_status st = capture(p, groups, seq, psi, &g);
    if (st != GP_OK) return st;
    if (p->run_graph) cudaGraphExecDestroy(p->run_graph);
    p->run_graph = g;
    p->run_key = key;
    p->run_steps = nsteps;
    GP_CUDA(p, cudaGraphLaunch(p->run_graph, s));
    p->launches += whole;
    return GP_OK;
  }
  if (capturing == cudaStreamCaptureStatusNone) {
    p->last_key = key;
    p->last_steps = nsteps;
  }

  gp_status st = run_items(p, groups, pro, psi, s);
  if (st != GP_OK) return st;
  if (ncycles >= 4 && !direct) {
    // capture the cycle once per set of field pointers, then replay it
    if (!p->cycle_graph || p->cycle_key != key) {
      if (p->cycle_graph) {
        cudaGraphExecDestroy(p->cycle_graph);
        p->cycle_graph = nullptr;
      }
      std::vector<std::pair<const std::vector<Item>*, int>> seq = {{&cyc, 1}};
      st = capture(p, groups, seq, psi, &p->cycle_graph);
      if (st != GP_OK) return st;
      p->cycle_key = key;
    }
    for (int c = 0; c < ncycles; ++c) GP_CUDA(p, cudaGraphLaunch(p->cycle_graph, s));
    p->launches += (long long)ncycles * (long long)cyc.size();
  } else {
    for (int c = 0; c < ncycles; ++c) {
      st = run_items(p, groups, cyc, psi, s);
      if (st != GP_OK) return st;
    }
  }
  st = run_items(p, groups, tail, psi, s);
  if (st != GP_OK) return st;
  return run_items(p, groups, epi, psi, s);
}

gp_status kinetic_block(gp_plan* p, int field, void* psi, double sk) {
  FieldPlan& F = p->f[field];
  Group G;
  G.fields.push_back(field);
  G.n = F.n;
  G.fp64 = F.fp64;
  std::vector<void*> ptrs(p->f.size(), nullptr);
  ptrs[field] = psi;
  const bool pl = !G.fp64 && plane_on(p, G.n);
  if (pl) {
    gp_status st = ensure_plane_sync(p, plane_sync_ints(G.n, 1));
    if (st != GP_OK) return st;
  }
  std::vector<Item> items;
  k_block(items, 0, sk, pl);
  return run_items(p, {G}, items, ptrs.data(), p->stream);
}

gp_status step_field(gp_plan* p, int field, void* psi, int nsteps) {
  // a one-field view of the plan (used by the adjoint's recomputation)
  std::vector<void*> ptrs(p->f.size(), nullptr);
  ptrs[field] = psi;
  FieldPlan& F = p->f[field];
  if (nsteps == 0) return GP_OK;
  Group G;
  G.fields.push_back(field);
  G.n = F.n;
  G.fp64 = F.fp64;
  G.split = F.prm.split;
  std::vector<Group> groups{G};
  const double dt = F.prm.dt, h = 0.5 * dt;
  const bool pl = !G.fp64 && plane_on(p, G.n);
  if (pl) {
    gp_status st = ensure_plane_sync(p, plane_sync_ints(G.n, 1));
    if (st != GP_OK) return st;
  }
  std::vector<Item> items;
  if (G.split == GP_SPLIT_NKN) {
    items.push_back({0, 2, OP_N_FWD, h, 0.0});
    k_block(items, 0, dt, pl);
    for (int c = 0; c < nsteps - 1; ++c) {
      items.push_back({0, 2, OP_INV_N_FWD, dt, 0.0});
      k_block(items, 0, dt, pl);
    }
    items.push_back({0, 2, OP_INV_N, h, 0.0});
  } else {
    items.push_back({0, 2, OP_FWD, 0.0, 0.0});
    k_block(items, 0, h, pl);
    for (int c = 0; c < nsteps; ++c) {
      items.push_back({0, 2, OP_INV_N_FWD, dt, 0.0});
      k_block(items, 0, c == nsteps - 1 ? h : dt, pl);
    }
    items.push_back({0, 2, OP_INV, 0.0, 0.0});
  }
  return run_items(p, groups, items, ptrs.data(), p->stream);
}

}  // namespace gp

using namespace gp;

extern "C" {

gp_status gp_step(gp_plan* p, void* const* psi, int nsteps) {
  if (!p) return GP_ERR_INVALID_ARG;
  if (!psi || nsteps < 0) return fail(p, GP_ERR_INVALID_ARG, "gp_step: null field list or negative nsteps");
  for (size_t i = 0; i < p->f.size(); ++i)
    if (bad_ptr(psi[i])) return fail(p, GP_ERR_INVALID_ARG, "gp_step: field pointer null or not 16-byte aligned");
  return step_all(p, psi, nsteps);
}

gp_status gp_step_host(gp_plan* p, void* const* psi_host, int nsteps) {
  if (!p) return GP_ERR_INVALID_ARG;
  if (!psi_host || nsteps < 0) return fail(p, GP_ERR_INVALID_ARG, "gp_step_host: null field list or negative nsteps");
  std::vector<void*> dev(p->f.size());
  for (size_t i = 0; i < p->f.size(); ++i) {
    FieldPlan& F = p->f[i];
    if (!psi_host[i]) return fail(p, GP_ERR_INVALID_ARG, "gp_step_host: null host field");
    const size_t bytes = (size_t)F.npts * (F.fp64 ? 16 : 8);
    if (!F.host_buf) GP_CUDA(p, cudaMalloc(&F.host_buf, bytes));
    dev[i] = F.host_buf;
    GP_CUDA(p, cudaMemcpyAsync(F.host_buf, psi_host[i], bytes, cudaMemcpyHostToDevice, p->stream));
  }
  gp_status st = step_all(p, dev.data(), nsteps);
  if (st != GP_OK) return st;
  for (size_t i = 0; i < p->f.size(); ++i) {
    FieldPlan& F = p->f[i];
    const size_t bytes = (size_t)F.npts * (F.fp64 ? 16 : 8);
    GP_CUDA(p, cudaMemcpyAsync(psi_host[i], F.host_buf, bytes, cudaMemcpyDeviceToHost, p->stream));
  }
  return check_status(p);
}

}  // extern "C"

extern "C" {

gp_status gp_profile(gp_plan* p, int enable) {
  if (!p) return GP_ERR_INVALID_ARG;
  if (enable) {
    GP_CUDA(p, p->stream ? cudaStreamSynchronize(p->stream) : cudaDeviceSynchronize());
    for (cudaEvent_t e : p->ev_pool) cudaEventDestroy(e);
    p->ev_pool.clear();
    p->ev_kind.clear();
    p->kinds.clear();
  }
  p->prof = enable != 0;
  return GP_OK;
}

int gp_profile_read(gp_plan* p, int max_kinds, char* names, long long* launches, double* ms) {
  if (!p || max_kinds < 0 || (max_kinds > 0 && (!names || !launches || !ms))) return -1;
  if ((p->stream ? cudaStreamSynchronize(p->stream) : cudaDeviceSynchronize()) != cudaSuccess) return -1;
  const int nk = (int)p->kinds.size();
  std::vector<double> tot(nk, 0.0);
  std::vector<long long> cnt(nk, 0);
  for (size_t i = 0; i < p->ev_kind.size(); ++i) {
    float t = 0.f;
    if (cudaEventElapsedTime(&t, p->ev_pool[2 * i], p->ev_pool[2 * i + 1]) != cudaSuccess) return -1;
    tot[p->ev_kind[i]] += t;
    cnt[p->ev_kind[i]] += 1;
  }
  const int nout = nk < max_kinds ? nk : max_kinds;
  for (int q = 0; q < nout; ++q) {
    std::snprintf(names + 64 * q, 64, "%s", p->kinds[q].c_str());
    launches[q] = cnt[q];
    ms[q] = tot[q];
  }
  return nout;
}

long long gp_launch_count(const gp_plan* p) { return p ? p->launches : -1; }

}  // extern "C"
