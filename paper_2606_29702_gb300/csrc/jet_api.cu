// Host side of libjet: plan creation (closure of the needed multi-indices,
// choice of the compiled channel set, tiling, workspace), call orchestration
// and the batched-ensemble work list.  See include/jet.h for the contract.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <map>
#include <set>
#include <string>
#include <vector>

#include "../../include/jet.h"
#include "jet_capture.h"
#include "jet_closures_gen.h"
#include "jet_internal.h"
#include "jet_plan.h"
#include "jet_tc.h"

using namespace jet;

namespace {

thread_local std::string g_err;

jet_status fail(jet_status st, const char* fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof(buf), fmt, ap);
  va_end(ap);
  g_err = buf;
  return st;
}

jet_status cuda_fail(cudaError_t e, const char* what) {
  cudaGetLastError();  // reported here: a caller's next check of its own calls does not find it
  return fail(e == cudaErrorMemoryAllocation ? JET_ERR_OOM : JET_ERR_CUDA, "%s: %s", what, cudaGetErrorString(e));
}

#define CK(expr)                                   \
  do {                                             \
    cudaError_t e_ = (expr);                       \
    if (e_ != cudaSuccess) return cuda_fail(e_, #expr); \
  } while (0)

using Alpha = std::vector<int>;  // orders per coordinate, length d

cudaError_t simt_launch(int cls, bool fp64, const SimtArgs& a, int grid, size_t smem, cudaStream_t s) {
  switch (cls) {
#define CASE(id, cl) \
  case id:           \
    return simt_launch_id<id>(fp64, a, grid, smem, s);
    JET_FOR_EACH_CLASS(CASE)
#undef CASE
  }
  return cudaErrorInvalidValue;
}

cudaError_t simt_occupancy(int cls, bool fp64, int ru, int threads, size_t smem, int* blocks) {
  switch (cls) {
#define CASE(id, cl) \
  case id:           \
    return simt_max_active_id<id>(fp64, ru, threads, smem, blocks);
    JET_FOR_EACH_CLASS(CASE)
#undef CASE
  }
  return cudaErrorInvalidValue;
}

cudaError_t debug_act(int cls, int kind, long long n, const double* z, const double* v, double* out, cudaStream_t s) {
  switch (cls) {
#define CASE(id, cl) \
  case id:           \
    return debug_activation_id<id>(kind, n, z, v, out, s);
    JET_FOR_EACH_CLASS(CASE)
#undef CASE
  }
  return cudaErrorInvalidValue;
}

}  // namespace

void jet::set_last_error(const char* msg) { g_err = msg; }

void jet::plan_prof_begin(jet_plan_s* p, cudaStream_t s) {
  if (!p->profiling) return;
  cudaEvent_t a, b;
  cudaEventCreate(&a);
  cudaEventCreate(&b);
  cudaEventRecord(a, s);
  p->prof.push_back({a, b});
}

void jet::plan_prof_end(jet_plan_s* p, cudaStream_t s) {
  if (!p->profiling || p->prof.empty()) return;
  cudaEventRecord(p->prof.back().second, s);
}

// Record an event pair around the dominant kernel of a call when profiling.
struct ProfScope {
  jet_plan_s* p;
  cudaStream_t s;
  ProfScope(jet_plan_s* p_, cudaStream_t s_) : p(p_), s(s_) { jet::plan_prof_begin(p, s); }
  ~ProfScope() { jet::plan_prof_end(p, s); }
};

namespace {

void free_plan_ws(jet_plan_s* p) {
  for (auto& e : p->prof) {
    cudaEventDestroy(e.first);
    cudaEventDestroy(e.second);
  }
  p->prof.clear();
  cudaFree(p->ws);
  cudaFree(p->store);
  p->ws = p->Wt = p->scratch = p->store = nullptr;
  p->grad_slices = p->loss_slices = nullptr;
  p->wsums = nullptr;
  if (p->tcp) tc_plan_destroy(p->tcp);
  p->tcp = nullptr;
}

bool alpha_leq(const Alpha& a, const Alpha& b) {
  for (size_t i = 0; i < a.size(); ++i)
    if (a[i] > b[i]) return false;
  return true;
}

// all multi-indices below a (componentwise), including a and 0
void below(const Alpha& a, std::set<Alpha>& out) {
  Alpha cur(a.size(), 0);
  while (true) {
    out.insert(cur);
    size_t i = 0;
    while (i < a.size()) {
      if (cur[i] < a[i]) {
        ++cur[i];
        break;
      }
      cur[i] = 0;
      ++i;
    }
    if (i == a.size()) break;
  }
}

size_t simt_tile_smem(const jet_plan_s* p, int P, int threads) {
  const int pitch = simt_pitch(p->C, P, p->wmax, threads, p->elem);
  return simt_smem_bytes(p->C, P, pitch, p->wmax, p->n_out, p->d, p->elem);
}

// most points per tile that `ctas` CTAs of `threads` per SM can hold, at most
// one item of the jet GEMMs per thread (FP64: two), in whole groups of points
int simt_most_points(const jet_plan_s* p, int ru, int threads, int ctas) {
  const int step = p->P0 ? p->P0 : 2;
  int P = std::max(step, threads * std::max(ru, 2) / p->wmax / step * step);
  while (P > step && (simt_tile_smem(p, P, threads) + kSimtCtaBytes) * ctas > kSimtSmBytes) P -= step;
  return P;
}

// CTA shape and largest tile of a SIMT plan.  FP32 runs two CTAs of 256 threads
// per SM (one CTA's barriers and elementwise phases overlap the other's GEMMs)
// unless shared memory then takes more than an eighth of the points in flight
// per SM that one CTA of 512 holds (256-wide layers).  Channel sets of 10 or
// more run one CTA of 256 threads with all registers.  (One CTA of 512 at width
// 64: 2->64x5->1 1.41 ms against 1.33 ms, forward pass of 2->64x6->3 at 10000
// points 93 against 83 us, composite loss 276 against 301 us.)  FP64 is bound by
// its two lanes per SM, not by the tile.
void simt_shape(jet_plan_s* p, int p8) {
  p->threads = kSimtThreads;
  p->P0 = p->fp64 ? 0 : p8 ? 8 * p8 : simt_group_points(p->wmax);
  if (p8) {
    p->P = 8 * p8;
    p->P_fixed = true;
    return;
  }
  const bool wide = !p->fp64 && p->C >= 10;
  p->P = simt_most_points(p, p->ru, kSimtThreads, wide ? 1 : 2);
  if (p->fp64 || wide) return;
  const int one = simt_most_points(p, p->ru, 2 * kSimtThreads, 1);
  if (7 * one > 8 * 2 * p->P) {
    p->P = one;
    p->threads = 2 * kSimtThreads;
  }
}

// Points per tile of one call on N points: the tile that leaves the busiest SM
// the least work, counted in GEMM warps per tile plus kTileWarps for what a
// tile costs whatever its size (its barriers and latencies).  FP32 warps count
// in fours, one per scheduler of the SM: six warps take as long as eight.
constexpr double kTileWarps = 2.0;
double simt_tile_cost(const jet_plan_s* p, int P) {
  int warps = (p->wmax / p->ru * P + 31) / 32;
  if (!p->fp64) warps = (warps + 3) / 4 * 4;
  return warps + kTileWarps;
}
int simt_call_points(const jet_plan_s* p, long long N) {
  if (p->P_fixed) return p->P;
  const int step = p->P0 ? p->P0 : 2;
  // the z-jet store holds whole tiles: near its capacity, tiles that end within it
  const bool stored = p->store && N <= p->store_max_points;
  int best = 0;
  double best_cost = 0.0;
  for (int P = p->P; P >= step; P -= step) {
    const long long tiles = (N + P - 1) / P, per_sm = (tiles + p->sms - 1) / p->sms;
    if (stored && tiles * P > p->store_max_points) continue;
    const double cost = (double)per_sm * simt_tile_cost(p, P);
    if (best == 0 || cost < best_cost) {
      best = P;
      best_cost = cost;
    }
  }
  return best;
}

// Most chunks that FP32 sums are kept for.  With FP32 sums a call's chunks are
// whole groups of P0 points, N and the plan alone fix them, and a tile takes up to
// P / P0 groups of one chunk: every sum is formed in the same order whatever the
// tile.  The count is part of the rounding of every gradient, not a residency: it
// is that of a kernel with three jet buffers (2 per SM where two of its CTAs fit,
// else 1; 1 for channel sets of 10 or more), kept so that gradients stay as they
// are.  The present kernel may hold two CTAs where it gives one (large tile
// overrides), and leaves the second slots empty then.
int simt_sum_chunks(const jet_plan_s* p) {
  const int P = p->P0, S0 = simt_swap(p->C, P) ? p->C + 1 : p->C;
  int pitch = S0 * P;
  while (pitch % 32 != 4) ++pitch;
  const size_t smem = (3 * (size_t)p->wmax * pitch + 2 * (size_t)p->n_out * p->C * P + (size_t)P * p->d) * 4 + 512;
  const int per_sm = p->C >= 10 ? 1 : (int)std::min<size_t>(2, kSimtSmBytes / (smem + 1024));
  return p->sms * std::max(1, per_sm);
}
void simt_sum_tiling(const jet_plan_s* p, DevInstance& I) {
  I.unit = p->P0;
  I.n_tiles = (I.N + I.unit - 1) / I.unit;
  const long long most = std::max<long long>(1, std::min<long long>(I.n_tiles, p->sum_chunks));
  I.tiles_per_chunk = (int)((I.n_tiles + most - 1) / most);
  I.chunk_rem = 0;
  I.n_chunks = (int)((I.n_tiles + I.tiles_per_chunk - 1) / I.tiles_per_chunk);
  if (p->P_fixed || p->store) {
    I.P = p->P0;
    return;
  }
  // groups per tile: least time of the busiest SM; whole runs of kWaccTiles
  // groups where a chunk takes several
  const long long per_sm = (I.n_chunks + p->sms - 1) / p->sms;
  const bool runs = p->C >= 7 && I.tiles_per_chunk > kWaccTiles;
  double best_cost = 0.0;
  I.P = p->P0;
  for (int V = p->P / p->P0; V >= 1; --V) {
    if (runs && kWaccTiles % V) continue;
    const double cost = (double)per_sm * ((I.tiles_per_chunk + V - 1) / V) * simt_tile_cost(p, V * p->P0);
    if (best_cost == 0.0 || cost < best_cost) {
      I.P = V * p->P0;
      best_cost = cost;
    }
  }
}

}  // namespace

extern "C" {

const char* jet_last_error(void) { return g_err.c_str(); }

const char* jet_version(void) { return "libjet 0.1 (sm_103a)"; }

}  // extern "C"

// Plan creation for one residual (n_specs = 1, grouped = false: the loss is
// the mean over all N points) or for a composite loss of n_specs terms, each
// over its own block of points (grouped = true).
static jet_status plan_create(jet_plan_t* out, int n_specs, const jet_residual_spec* const* specs,
                              const double* weights, const int32_t* paired, bool grouped, int32_t d_in,
                              int32_t n_layers, const int32_t* widths, int32_t n_needed, const jet_chan* needed,
                              jet_precision prec, size_t mem_budget_bytes, int32_t flags) {
  if (!out) return fail(JET_ERR_INVALID, "out is NULL");
  *out = nullptr;
  if (!specs || !widths || (n_needed > 0 && !needed)) return fail(JET_ERR_INVALID, "NULL spec, widths or needed");
  for (int g = 0; g < n_specs; ++g)
    if (!specs[g]) return fail(JET_ERR_INVALID, "NULL residual spec of loss term %d", g);
  if (d_in < 1 || d_in > 3) return fail(JET_ERR_INVALID, "d_in must be 1..3 (got %d)", d_in);
  if (n_layers < 2 || n_layers > kMaxLayers) return fail(JET_ERR_INVALID, "n_layers must be 2..%d", kMaxLayers);
  if (widths[0] != d_in) return fail(JET_ERR_INVALID, "widths[0] (%d) != d_in (%d)", widths[0], d_in);
  const int n_out = widths[n_layers];
  if (n_out < 1 || n_out > kMaxOut) return fail(JET_ERR_INVALID, "n_out must be 1..%d", kMaxOut);
  for (int l = 1; l < n_layers; ++l)
    if (widths[l] < 4 || widths[l] > 256 || widths[l] % 4)
      return fail(JET_ERR_UNSUPPORTED, "hidden width %d: must be a multiple of 4 in [4, 256]", widths[l]);
  if (prec < JET_FP64 || prec > JET_BF16X3) return fail(JET_ERR_INVALID, "unknown precision %d", (int)prec);
  for (int g = 0; g < n_specs; ++g) {
    const jet_residual_spec* spec = specs[g];
    if (spec->n_res < 1 || spec->n_res > kMaxRes || !spec->n_mono || !spec->mono)
      return fail(JET_ERR_INVALID, "residual spec: n_res must be 1..%d with n_mono and mono set", kMaxRes);
  }

  // ---- channel closure (Sec. 2.2: required states plus their lower-order chain)
  std::set<Alpha> need;
  for (int i = 0; i < n_needed; ++i) {
    Alpha a(d_in);
    for (int j = 0; j < d_in; ++j) a[j] = needed[i].alpha[j];
    for (int j = d_in; j < 4; ++j)
      if (needed[i].alpha[j]) return fail(JET_ERR_INVALID, "needed[%d] differentiates a coordinate >= d_in", i);
    need.insert(a);
  }
  need.insert(Alpha(d_in, 0));
  std::set<Alpha> closure;
  for (const Alpha& a : need) below(a, closure);
  if (!(flags & JET_FLAG_AUTO_CLOSE) && closure.size() != need.size())
    return fail(JET_ERR_NOT_CLOSED, "needed multi-indices are not downward closed (%zu given, closure has %zu)",
                need.size(), closure.size());
  // every spec factor must be carried
  int n_terms = 0;
  for (int g = 0; g < n_specs; ++g) {
    const jet_residual_spec* spec = specs[g];
    for (int c = 0; c < spec->n_res; ++c) {
      if (spec->n_mono[c] < 0 || (spec->n_mono[c] > 0 && !spec->mono[c]))
        return fail(JET_ERR_INVALID, "residual component %d: bad monomial list", c);
      n_terms += spec->n_mono[c];
    }
  }
  if (n_terms > kMaxTerms) return fail(JET_ERR_UNSUPPORTED, "%d monomials > %d", n_terms, kMaxTerms);
  for (int g = 0; g < n_specs; ++g) {
    const jet_residual_spec* spec = specs[g];
    for (int c = 0; c < spec->n_res; ++c)
      for (int m = 0; m < spec->n_mono[c]; ++m) {
        const jet_monomial& mo = spec->mono[c][m];
        if (mo.n_fac < 0 || mo.n_fac > 4) return fail(JET_ERR_INVALID, "monomial with %d factors", mo.n_fac);
        for (int f = 0; f < mo.n_fac; ++f) {
          const int o = mo.fac[f].out & ~JET_PAIR_SECOND;
          if ((mo.fac[f].out & JET_PAIR_SECOND) && !(paired && paired[g]))
            return fail(JET_ERR_INVALID, "JET_PAIR_SECOND in a term that is not paired");
          if (o < 0 || o >= n_out) return fail(JET_ERR_INVALID, "monomial factor output %d out of range", o);
          Alpha a(d_in);
          for (int j = 0; j < d_in; ++j) a[j] = mo.fac[f].alpha[j];
          for (int j = d_in; j < 4; ++j)
            if (mo.fac[f].alpha[j]) return fail(JET_ERR_INVALID, "a residual factor differentiates a coordinate >= d_in");
          if (!closure.count(a)) return fail(JET_ERR_INVALID, "residual uses a multi-index that is not in needed");
        }
      }
  }
  // ---- smallest compiled channel set containing the closure
  int best = -1;
  for (int k = 0; k < kNumClasses; ++k) {
    const ClassInfo& ci = kClassInfo[k];
    if (ci.d != d_in) continue;
    std::set<Alpha> have;
    for (int c = 0; c < ci.C; ++c) {
      Alpha a(d_in);
      for (int j = 0; j < d_in; ++j) a[j] = ci.alpha[c][j];
      have.insert(a);
    }
    bool ok = true;
    for (const Alpha& a : closure) ok = ok && have.count(a);
    if (ok && (best < 0 || ci.C < kClassInfo[best].C)) best = k;
  }
  if (best < 0) return fail(JET_ERR_UNSUPPORTED, "no compiled channel set in %d coordinates contains the closure", d_in);

  jet_plan_s* p = new jet_plan_s();
  cudaGetDevice(&p->device);
  p->d = d_in;
  p->L = n_layers;
  p->n_out = n_out;
  p->n_res = 0;
  for (int g = 0; g < n_specs; ++g) p->n_res = std::max(p->n_res, (int)specs[g]->n_res);
  p->widths.assign(widths, widths + n_layers + 1);
  p->cls = best;
  p->C = kClassInfo[best].C;
  p->prec = prec;
  p->fp64 = prec == JET_FP64;
  p->tc = prec >= JET_TF32;
  p->elem = p->fp64 ? 8 : 4;
  p->has_source = false;
  for (int g = 0; g < n_specs; ++g) p->has_source = p->has_source || specs[g]->has_source != 0;
  auto chan_index = [&](const jet_chan& ch) {
    const ClassInfo& ci = kClassInfo[best];
    for (int c = 0; c < ci.C; ++c) {
      bool eq = true;
      for (int j = 0; j < d_in; ++j) eq = eq && ci.alpha[c][j] == ch.alpha[j];
      if (eq) return c;
    }
    return -1;
  };
  for (int g = 0; g < n_specs; ++g) {
    const jet_residual_spec* spec = specs[g];
    DevGroup G;
    memset(&G, 0, sizeof(G));
    G.t0 = (int)p->terms.size();
    for (int c = 0; c < spec->n_res; ++c)
      for (int m = 0; m < spec->n_mono[c]; ++m) {
        const jet_monomial& mo = spec->mono[c][m];
        DevTerm t;
        t.coef = mo.coef;
        t.comp = c;
        t.nfac = mo.n_fac;
        t.pmask = 0;
        for (int f = 0; f < 4; ++f) t.fac[f] = 0;
        for (int f = 0; f < mo.n_fac; ++f) {
          t.fac[f] = (mo.fac[f].out & ~JET_PAIR_SECOND) * p->C + chan_index(mo.fac[f]);
          if (mo.fac[f].out & JET_PAIR_SECOND) t.pmask |= 1 << f;
        }
        p->terms.push_back(t);
      }
    G.t1 = (int)p->terms.size();
    G.n_res = spec->n_res;
    G.paired = paired && paired[g] ? 1 : 0;
    G.has_source = spec->has_source != 0;
    G.scale = weights ? weights[g] : 1.0;  // the term's weight; divided by its residual count per call
    p->groups.push_back(G);
  }
  p->n_groups = grouped ? n_specs : 0;
  long long off = 0;
  for (int l = 0; l < n_layers; ++l) {
    p->off_W.push_back(off);
    off += (long long)widths[l] * widths[l + 1];
    p->off_b.push_back(off);
    off += widths[l + 1];
  }
  p->n_params = off;

  // ---- tiling and occupancy of the fused SIMT kernel
  for (int l = 1; l < n_layers; ++l) p->wmax = std::max(p->wmax, widths[l]);
  p->ru = simt_units(widths, n_layers, p->fp64);
  simt_shape(p, JET_FLAG_TILE_GET(flags));
  p->smem = simt_tile_smem(p, p->P, p->threads);
  cudaDeviceProp prop;
  cudaError_t e = cudaGetDeviceProperties(&prop, p->device);
  if (e != cudaSuccess) {
    delete p;
    return cuda_fail(e, "cudaGetDeviceProperties");
  }
  int per_sm = 0;
  if (!p->tc) {
    p->sms = prop.multiProcessorCount;
    e = simt_occupancy(p->cls, p->fp64, p->ru, p->threads, p->smem, &per_sm);
    if (e != cudaSuccess || per_sm < 1) {
      delete p;
      return e != cudaSuccess ? cuda_fail(e, "occupancy") : fail(JET_ERR_UNSUPPORTED, "SIMT tile does not fit one SM");
    }
    per_sm = std::min(per_sm, 2);  // as measured; more CTAs would only add gradient slices
    p->grid = prop.multiProcessorCount * per_sm;
    p->ctas_per_sm = per_sm;
  }

  // ---- workspace
  long long jet_elems = 0;  // hidden z-jets of one tile
  for (int l = 1; l < n_layers; ++l) jet_elems += (long long)p->C * p->P * widths[l];
  if (!p->tc) {
    // FP32 forms whose per-chunk FP64 slices would not stay in L2 sum the
    // hidden-layer weights of a chunk in FP32; otherwise per-tile FP64 adds into
    // L2-resident slices are the cheaper of the two
    const int chunks = p->fp64 ? p->grid : std::max(p->grid, simt_sum_chunks(p));
    const bool slices_fit =
        p->fp64 || (double)simt_sum_chunks(p) * p->n_params * sizeof(double) <= kSimtSliceL2Bytes;
    p->wsums_stride = slices_fit ? 0 : simt_wacc_elems(widths, n_layers, p->fp64);
    p->sum_chunks = p->wsums_stride ? simt_sum_chunks(p) : 0;
    p->scratch_stride = jet_elems;
    const size_t b_ws = (size_t)chunks * p->wsums_stride * sizeof(float);
    size_t b_wt = (size_t)weight_ws_elems(p->n_params) * p->elem;
    size_t b_gs = (size_t)chunks * p->n_params * sizeof(double);
    size_t b_ls = (size_t)chunks * sizeof(double);
    size_t b_sc = (size_t)p->grid * p->scratch_stride * p->elem;
    Arena arena;
    arena.add(&p->Wt, b_wt);
    arena.add(&p->grad_slices, b_gs);
    arena.add(&p->loss_slices, b_ls);
    arena.add(&p->scratch, b_sc);
    arena.add(&p->wsums, b_ws);
    e = arena.alloc(&p->ws);
    p->ws_bytes = b_wt + b_gs + b_ls + b_sc + b_ws;
    if (e == cudaSuccess && (flags & JET_FLAG_STORE) && mem_budget_bytes > 0) {
      // as many points as the budget holds, in the smallest tiles of a call
      const int step = p->P_fixed ? p->P : p->P0 ? p->P0 : 2;
      const size_t per_step = (size_t)(jet_elems / p->P) * step * p->elem;
      const long long steps = (long long)(mem_budget_bytes / per_step);
      if (steps > 0) {
        p->store_max_points = steps * step;
        e = cudaMalloc(&p->store, steps * per_step);
        p->ws_bytes += steps * per_step;
      }
    }
    if (e != cudaSuccess) {
      free_plan_ws(p);
      delete p;
      return cuda_fail(e, "workspace allocation");
    }
  } else {
    jet_status st = tc_plan_create(p, &p->tcp, prop, mem_budget_bytes, flags);
    if (st != JET_OK) {
      free_plan_ws(p);
      delete p;
      return st;
    }
  }
  *out = p;
  return JET_OK;
}

extern "C" {

jet_status jet_plan_create(jet_plan_t* out, const jet_residual_spec* spec, int32_t d_in, int32_t n_layers,
                           const int32_t* widths, int32_t n_needed, const jet_chan* needed, jet_precision prec,
                           size_t mem_budget_bytes, int32_t flags) {
  if (!spec) {
    if (out) *out = nullptr;
    return fail(JET_ERR_INVALID, "NULL spec, widths or needed");
  }
  return plan_create(out, 1, &spec, nullptr, nullptr, false, d_in, n_layers, widths, n_needed, needed, prec,
                     mem_budget_bytes, flags);
}

jet_status jet_plan_create_loss(jet_plan_t* out, int32_t n_terms, const jet_loss_term* terms, int32_t d_in,
                                int32_t n_layers, const int32_t* widths, int32_t n_needed, const jet_chan* needed,
                                jet_precision prec, size_t mem_budget_bytes, int32_t flags) {
  if (out) *out = nullptr;
  if (!terms || n_terms < 1 || n_terms > kMaxGroups)
    return fail(JET_ERR_INVALID, "a composite loss takes 1..%d terms", kMaxGroups);
  std::vector<const jet_residual_spec*> specs(n_terms);
  std::vector<double> weights(n_terms);
  std::vector<int32_t> paired(n_terms);
  for (int g = 0; g < n_terms; ++g) {
    specs[g] = terms[g].spec;
    weights[g] = terms[g].weight;
    paired[g] = terms[g].paired ? 1 : 0;
    if (!(terms[g].weight >= 0.0)) return fail(JET_ERR_INVALID, "loss term %d: weight must be >= 0", g);
  }
  return plan_create(out, n_terms, specs.data(), weights.data(), paired.data(), true, d_in, n_layers, widths,
                     n_needed, needed, prec, mem_budget_bytes, flags);
}

jet_status jet_plan_set_term_points(jet_plan_t p, const int64_t* counts) {
  if (!p || !counts) return fail(JET_ERR_INVALID, "NULL plan or counts");
  if (p->n_groups == 0) return fail(JET_ERR_INVALID, "the plan has one residual over all points (no loss terms)");
  long long start = 0;
  for (int g = 0; g < p->n_groups; ++g) {
    if (counts[g] < 0) return fail(JET_ERR_INVALID, "loss term %d: negative point count", g);
    if (p->groups[g].paired && ((start | counts[g]) & 1))
      return fail(JET_ERR_INVALID, "paired loss term %d must start at an even point index and hold whole pairs", g);
    start += counts[g];
  }
  p->group_counts.assign(counts, counts + p->n_groups);
  return JET_OK;
}

jet_status jet_plan_get_info(jet_plan_t p, jet_plan_info* info) {
  if (!p || !info) return fail(JET_ERR_INVALID, "NULL plan or info");
  memset(info, 0, sizeof(*info));
  info->d_in = p->d;
  info->n_out = p->n_out;
  info->n_layers = p->L;
  info->n_channels = p->C;
  info->closure_class = p->cls;
  snprintf(info->class_name, sizeof(info->class_name), "%s", kClassInfo[p->cls].name);
  info->n_params = p->n_params;
  info->precision = p->prec;
  info->store_mode = p->store != nullptr;
  info->store_max_points = p->store_max_points;
  info->tile_points = p->tc ? tc_tile_points(p->tcp) : p->P;
  info->grid_ctas = p->tc ? tc_grid(p->tcp) : p->grid;
  info->workspace_bytes = p->tc ? tc_workspace_bytes(p->tcp) : p->ws_bytes;
  info->ctas_per_sm = p->tc ? tc_ctas_per_sm(p->tcp) : p->ctas_per_sm;
  info->cta_threads = p->tc ? tc_threads(p->tcp) : p->threads;
  info->wgrad_chunk_fp32 = p->tc ? tc_wgrad_chunk_fp32(p->tcp) : (p->wsums ? 1 : 0);
  return JET_OK;
}

jet_status jet_plan_profile(jet_plan_t p, int32_t enable) {
  if (!p) return fail(JET_ERR_INVALID, "NULL plan");
  p->profiling = enable != 0;
  return JET_OK;
}

jet_status jet_plan_profile_read(jet_plan_t p, int64_t* launches, double* total_ms) {
  if (!p || !launches || !total_ms) return fail(JET_ERR_INVALID, "NULL argument");
  double tot = 0.0;
  for (auto& e : p->prof) {
    cudaError_t err = cudaEventSynchronize(e.second);
    float ms = 0.f;
    if (err == cudaSuccess) err = cudaEventElapsedTime(&ms, e.first, e.second);
    if (err != cudaSuccess) return cuda_fail(err, "profile events");
    tot += ms;
  }
  *launches = (int64_t)p->prof.size();
  *total_ms = tot;
  for (auto& e : p->prof) {
    cudaEventDestroy(e.first);
    cudaEventDestroy(e.second);
  }
  p->prof.clear();
  return JET_OK;
}

jet_status jet_plan_destroy(jet_plan_t p) {
  if (!p) return JET_OK;
  free_plan_ws(p);
  delete p;
  return JET_OK;
}

}  // extern "C"

namespace {

// Fill the per-call instance descriptor of the SIMT kernel, for CTAs of
// `threads` with ru units per GEMM thread: the call's own tiles and chunks
// (want_grad: those of its FP32 sums, if it keeps any; a forward pass without a
// z-jet store takes any), or (batches) tiles of P points in `chunks` chunks.
void fill_instance(const jet_plan_s* p, const void* params, const void* X, long long N, const void* source,
                   void* r_out, bool want_grad, int ru, int threads, int P, int chunks, DevInstance& I) {
  memset(&I, 0, sizeof(I));
  I.L = p->L;
  I.d = p->d;
  I.n_out = p->n_out;
  I.n_res = p->n_res;
  for (int l = 0; l <= p->L; ++l) I.widths[l] = p->widths[l];
  for (int l = 0; l < p->L; ++l) {
    I.off_W[l] = p->off_W[l];
    I.off_b[l] = p->off_b[l];
  }
  I.n_params = p->n_params;
  I.params = params;
  I.Wt = p->Wt;
  I.X = X;
  I.source = source;
  I.r_out = r_out;
  I.N = N;
  I.inv_N = N > 0 ? 1.0 / (double)N : 0.0;
  I.n_terms = (int)p->terms.size();
  for (int m = 0; m < I.n_terms; ++m) I.terms[m] = p->terms[m];
  if (p->n_groups > 0) {
    I.inv_N = 1.0;  // each term's mean is in its scale
    I.n_groups = fill_groups(p, I.groups);
  }
  if (P > 0) {
    I.P = P;
    simt_set_chunks(I, chunks);
  } else if (p->sum_chunks && (want_grad || p->store)) {
    simt_sum_tiling(p, I);
  } else {
    I.P = simt_call_points(p, N);
    simt_set_chunks(I, p->grid);
  }
  I.P0 = p->fp64 ? I.P : p->P0;
  I.swap = p->fp64 ? 0 : simt_swap(p->C, I.P0);
  I.wr = simt_wgrad_rows(ru, p->wmax, I.P / I.P0, threads, p->fp64);
  I.pitch = simt_pitch(p->C, I.P, p->wmax, threads, p->elem);
  I.chunk_base = 0;
  I.grad_slices = p->grad_slices;
  I.loss_slices = p->loss_slices;
  I.store = nullptr;
  for (int l = 1; l < p->L; ++l) I.store_tile_stride += (long long)p->C * I.P * p->widths[l];
  simt_set_sums(I, p->C, p->wsums, p->wsums_stride);
}

jet_status check_call(const jet_plan_s* p, const void* params, const void* X, long long N, const void* source) {
  if (!p) return fail(JET_ERR_INVALID, "NULL plan");
  if (N < 0) return fail(JET_ERR_INVALID, "N < 0");
  if (p->n_groups > 0) {
    if ((int)p->group_counts.size() != p->n_groups)
      return fail(JET_ERR_INVALID, "a composite-loss plan needs jet_plan_set_term_points before its calls");
    long long tot = 0;
    for (long long c : p->group_counts) tot += c;
    if (tot != N) return fail(JET_ERR_INVALID, "N (%lld) differs from the loss terms' points (%lld)", N, tot);
  }
  if (!params) return fail(JET_ERR_INVALID, "NULL params");
  if (N > 0 && !X) return fail(JET_ERR_INVALID, "NULL X");
  if (p->has_source && N > 0 && !source) return fail(JET_ERR_INVALID, "the residual has a source: pass it");
  if (!p->has_source && source) return fail(JET_ERR_INVALID, "the residual has no source term");
  return JET_OK;
}

jet_status run_simt(jet_plan_s* p, int mode, const DevInstance& I, cudaStream_t s) {
  SimtArgs a;
  memset(&a, 0, sizeof(a));
  a.mode = mode;
  a.n_inst = 1;
  a.insts = nullptr;
  a.inst0 = I;
  a.n_items = I.n_chunks;
  a.item_inst = nullptr;
  a.scratch = p->scratch;
  a.scratch_stride = p->scratch_stride;
  a.ru = p->ru;
  a.threads = p->threads;
  a.carveout = simt_carveout(p->smem, p->ctas_per_sm);
  int grid = std::min(p->grid, I.n_chunks);
  ProfScope prof(p, s);
  CK(simt_launch(p->cls, p->fp64, a, grid, p->smem, s));
  return JET_OK;
}

ReduceJob make_job(const DevInstance& I, void* grad_out, double* loss_out, bool with_grad) {
  ReduceJob j;
  memset(&j, 0, sizeof(j));
  j.grad_slices = I.grad_slices;
  j.loss_slices = I.loss_slices;
  j.n_chunks = I.n_chunks;
  j.n_slice = I.n_slice;
  j.n_params = with_grad ? I.n_params : 0;
  if (with_grad && I.wsums && I.wsums_direct) {
    j.hid = HID_SIMT;
    j.L = I.L;
    for (int l = 0; l <= I.L; ++l) j.widths[l] = I.widths[l];
    j.n_hid = (int)I.wsums_stride;
    j.subs = 1;
    j.wr = I.wr;
    j.hid_sums = I.wsums;
    j.hid_stride = I.wsums_stride;
  }
  j.inv_N = I.inv_N;
  j.grad_out = grad_out;
  j.loss_out = loss_out;
  return j;
}

}  // namespace

extern "C" {

jet_status jet_forward_residual(jet_plan_t p, const void* params, const void* X, int64_t N, const void* source,
                                void* r_out, double* loss_out, jet_stream_t stream) {
  jet_status st = check_call(p, params, X, N, source);
  if (st != JET_OK) return st;
  cudaStream_t s = (cudaStream_t)stream;
  if (p->tc) return tc_forward(p, p->tcp, params, X, N, source, r_out, loss_out, s);
  if (N == 0) {
    if (loss_out) CK(cudaMemsetAsync(loss_out, 0, sizeof(double), s));
    return JET_OK;
  }
  DevInstance I;
  fill_instance(p, params, X, N, source, r_out, false, p->ru, p->threads, 0, 0, I);
  const bool store = p->store && N <= p->store_max_points;
  const unsigned long long capture = p->store ? stream_capture_id(s) : 0;
  if (store) I.store = p->store;
  if (store && capture) CK(p->st_graphs.add(s));
  CK(launch_transpose_weights(I, p->fp64, p->Wt, s));
  st = run_simt(p, MODE_FWD, I, s);
  if (st != JET_OK) return st;
  ReduceJob j = make_job(I, nullptr, loss_out, false);
  if (loss_out) CK(launch_reduce(&j, nullptr, 1, p->fp64, false, 1, 0.f, s));
  p->st_valid = store;
  p->st_capture = capture;
  p->st_params = params;
  p->st_X = X;
  p->st_src = source;
  p->st_N = N;
  return JET_OK;
}

jet_status jet_backward_params(jet_plan_t p, const void* params, const void* X, int64_t N, const void* source,
                               void* grad_out, void* r_out, double* loss_out, jet_stream_t stream) {
  jet_status st = check_call(p, params, X, N, source);
  if (st != JET_OK) return st;
  if (!grad_out) return fail(JET_ERR_INVALID, "NULL grad_out");
  cudaStream_t s = (cudaStream_t)stream;
  if (p->tc) return tc_backward(p, p->tcp, params, X, N, source, grad_out, r_out, loss_out, s);
  if (N == 0) {
    CK(cudaMemsetAsync(grad_out, 0, p->n_params * p->elem, s));
    if (loss_out) CK(cudaMemsetAsync(loss_out, 0, sizeof(double), s));
    return JET_OK;
  }
  DevInstance I;
  fill_instance(p, params, X, N, source, r_out, true, p->ru, p->threads, 0, 0, I);
  // a captured forward pass fills the store for its own graph's backward only, and
  // while a graph writes the store no eager call relies on it
  const unsigned long long capture = p->st_valid ? stream_capture_id(s) : 0;
  const bool from_store = p->st_valid && p->st_params == params && p->st_X == X && p->st_N == N &&
                          p->st_src == source && p->st_capture == capture && (capture || !p->st_graphs.live());
  if (from_store) I.store = p->store;
  CK(launch_transpose_weights(I, p->fp64, p->Wt, s));
  st = run_simt(p, from_store ? MODE_BWD_STORE : MODE_FWD_BWD, I, s);
  if (st != JET_OK) return st;
  ReduceJob j = make_job(I, grad_out, loss_out, true);
  CK(launch_reduce(&j, nullptr, 1, p->fp64, false, 1, 0.f, s));
  return JET_OK;
}

}  // extern "C"

// Adam step t = `step`, or *step_ctr + 1 (then incremented) with a device counter
static jet_status train_step(jet_plan_t p, void* params, void* adam_m, void* adam_v, int64_t step,
                             long long* step_ctr, float lr, const void* X, int64_t N, const void* source,
                             double* loss_out, cudaStream_t s) {
  jet_status st = check_call(p, params, X, N, source);
  if (st != JET_OK) return st;
  if (!adam_m || !adam_v) return fail(JET_ERR_INVALID, "NULL Adam state");
  if (N < 1) return fail(JET_ERR_INVALID, "train step needs N >= 1");
  p->st_valid = false;  // params change in place
  if (p->tc) return tc_train_step(p, p->tcp, params, adam_m, adam_v, step, step_ctr, lr, X, N, source, loss_out, s);
  DevInstance I;
  fill_instance(p, params, X, N, source, nullptr, true, p->ru, p->threads, 0, 0, I);
  CK(launch_transpose_weights(I, p->fp64, p->Wt, s));
  st = run_simt(p, MODE_FWD_BWD, I, s);
  if (st != JET_OK) return st;
  ReduceJob j = make_job(I, nullptr, loss_out, true);
  j.params = params;
  j.m = adam_m;
  j.v = adam_v;
  CK(launch_reduce(&j, nullptr, 1, p->fp64, true, step, lr, s, step_ctr));
  return JET_OK;
}

extern "C" {

jet_status jet_train_step(jet_plan_t p, void* params, void* adam_m, void* adam_v, int64_t step, float lr,
                          const void* X, int64_t N, const void* source, double* loss_out, jet_stream_t stream) {
  if (step < 1) return fail(JET_ERR_INVALID, "step must be >= 1");
  return train_step(p, params, adam_m, adam_v, step, nullptr, lr, X, N, source, loss_out, (cudaStream_t)stream);
}

jet_status jet_train_step_dev(jet_plan_t p, void* params, void* adam_m, void* adam_v, int64_t* step_counter,
                              float lr, const void* X, int64_t N, const void* source, double* loss_out,
                              jet_stream_t stream) {
  if (!step_counter) return fail(JET_ERR_INVALID, "NULL step counter");
  return train_step(p, params, adam_m, adam_v, 1, reinterpret_cast<long long*>(step_counter), lr, X, N, source,
                    loss_out, (cudaStream_t)stream);
}

jet_status jet_debug_activation(jet_plan_t p, int32_t kind, int64_t n, const double* z, const double* v, double* out,
                                jet_stream_t stream) {
  if (!p || !z || !out || (kind != 0 && !v)) return fail(JET_ERR_INVALID, "NULL argument");
  if (kind < 0 || kind > 2) return fail(JET_ERR_INVALID, "kind must be 0, 1 or 2");
  CK(debug_act(p->cls, kind, n, z, v, out, (cudaStream_t)stream));
  return JET_OK;
}

}  // extern "C"

// ------------------------------------------------------------------ batches

constexpr int kSimtBatchChunks = 16;  // least bound of a member's chunks
constexpr int kSimtBatchItems = 3;    // work items per CTA that the list aims at

struct jet_batch_s {
  std::vector<jet_plan_t> plans;
  int cls = -1;
  bool fp64 = false;
  bool tc = false;
  int grid = 0;
  size_t smem = 0;
  int ru = 0, ctas_per_sm = 0;
  std::vector<int> P;  // points per tile of every member
  int max_chunks_per_inst = kSimtBatchChunks;
  // device workspace
  DevInstance* d_insts = nullptr;
  int* d_item_inst = nullptr;
  int* d_next = nullptr;  // the kernel's item counter
  ReduceJob* d_jobs = nullptr;
  // FP64 slices and FP32 weight-gradient sums of a call's chunks, cut out per call
  // (batch_pool_bytes); loss sums [max_items]
  char* pool = nullptr;
  size_t pool_bytes = 0;
  double* loss_slices = nullptr;
  void* Wt = nullptr;
  void* scratch = nullptr;
  long long scratch_stride = 0;
  float* run_sums = nullptr;  // FP32 sums of a CTA's running chunk, of members whose chunks take several runs
  std::vector<long long> wt_off;
  // the call's descriptors and work list, and their pinned staging (eager calls)
  std::vector<DevInstance> insts;
  std::vector<int> items;
  DevInstance* h_insts = nullptr;
  int* h_item_inst = nullptr;
  ReduceJob* h_jobs = nullptr;
  int max_items = 0;
  TcBatch* tcb = nullptr;
  // the pinned staging buffers are rewritten by the next call only after the
  // uploads of this one have read them
  cudaEvent_t copied = nullptr;
  CaptureStore captured;  // descriptors of captured calls
};

namespace {

void free_batch(jet_batch_s* b) {
  cudaFree(b->d_insts);
  cudaFree(b->d_item_inst);
  cudaFree(b->d_next);
  cudaFree(b->d_jobs);
  cudaFree(b->pool);
  cudaFree(b->loss_slices);
  cudaFree(b->Wt);
  cudaFree(b->scratch);
  cudaFree(b->run_sums);
  cudaFreeHost(b->h_insts);
  cudaFreeHost(b->h_item_inst);
  cudaFreeHost(b->h_jobs);
  if (b->tcb) tc_batch_destroy(b->tcb);
  if (b->copied) cudaEventDestroy(b->copied);
}

// Most bytes a chunk of a plan takes in the pool: its FP64 slice, beside FP32 sums
// that the reduction reads or (channel sets of 7 or more, chunks of several runs)
// with every parameter.
size_t batch_chunk_bytes(const jet_plan_s* p) {
  const size_t all = (size_t)p->n_params * sizeof(double);
  if (!p->wsums) return all;
  const size_t direct = (size_t)(p->n_params - p->wsums_stride) * sizeof(double) + (size_t)p->wsums_stride * sizeof(float);
  return p->C < 7 ? direct : std::max(all, direct);
}

// Bytes that the chunks of any call fit: the work list gives every member one
// chunk and shares about kSimtBatchItems per CTA more among them by cost, at most
// max_chunks each, so the largest members may hold nearly all of them.  (Sized by
// max_chunks for every member, nine 3->256x8->1 FP32 networks took 12.4 GB; 4 GB so.)
size_t batch_pool_bytes(const std::vector<jet_plan_t>& plans, int grid, int max_chunks) {
  std::vector<size_t> per;
  for (const jet_plan_s* p : plans) per.push_back(batch_chunk_bytes(p));
  std::sort(per.rbegin(), per.rend());
  size_t total = 0;
  long long extra = (long long)kSimtBatchItems * grid;
  for (size_t b : per) {
    const long long k = std::min<long long>(max_chunks - 1, extra);
    extra -= k;
    total += (size_t)(1 + k) * b + 2 * 256;  // alignment of its two parts
  }
  return total;
}

// Build the per-call descriptors and work list: every instance is split into
// chunks of point tiles; items are ordered by estimated cost, largest first, and
// pulled by the persistent CTAs in that order.
jet_status batch_prepare(jet_batch_s* b, const void* const* params, const void* const* X, const int64_t* N,
                         const void* const* source, void* const* r_out) {
  const int n = (int)b->plans.size();
  auto tile_cost = [&](int i) {
    const jet_plan_s* p = b->plans[i];
    double c = 64.0;
    for (int l = 2; l < p->L; ++l) c += (double)p->widths[l - 1] * p->widths[l];
    return c * p->C * b->P[i];
  };
  double total_cost = 0.0;
  for (int i = 0; i < n; ++i) {
    jet_status st = check_call(b->plans[i], params[i], X[i], N[i], source ? source[i] : nullptr);
    if (st != JET_OK) return st;
    total_cost += tile_cost(i) * (double)((N[i] + b->P[i] - 1) / b->P[i]);
  }
  const double target = total_cost / ((double)kSimtBatchItems * b->grid);  // items of equal cost
  std::vector<std::pair<double, int>> cost;  // (cost, item) for ordering
  std::vector<int> item_inst;
  int chunk_base = 0;
  size_t pool_off = 0;
  auto take = [&](size_t bytes) {
    char* at = b->pool + pool_off;
    pool_off += (bytes + 255) / 256 * 256;
    return at;
  };
  b->insts.resize(n);
  for (int i = 0; i < n; ++i) {
    jet_plan_s* p = b->plans[i];
    DevInstance& I = b->insts[i];
    const long long tiles = (N[i] + b->P[i] - 1) / b->P[i];
    const double per_tile = tile_cost(i);
    const long long share = tiles > 0 ? (long long)(per_tile * (double)tiles / target + 0.5) : 0;
    const long long want = std::min<long long>(b->max_chunks_per_inst, std::max<long long>(1, share));
    fill_instance(p, params[i], X[i], N[i], source ? source[i] : nullptr, r_out ? r_out[i] : nullptr, true, b->ru,
                  kSimtThreads, b->P[i], (int)want, I);
    I.Wt = (char*)b->Wt + b->wt_off[i] * p->elem;
    simt_set_sums(I, p->C, p->wsums ? b->run_sums : nullptr, p->wsums_stride);
    I.grad_slices = reinterpret_cast<double*>(take((size_t)I.n_chunks * I.n_slice * sizeof(double)));
    if (I.wsums_direct) I.wsums = reinterpret_cast<float*>(take((size_t)I.n_chunks * I.wsums_stride * sizeof(float)));
    I.loss_slices = b->loss_slices + (long long)i * b->max_chunks_per_inst;
    I.chunk_base = chunk_base;
    for (int c = 0; c < I.n_chunks; ++c) {
      const long long nt = I.tiles_per_chunk + (c < I.chunk_rem ? 1 : 0);
      cost.push_back({per_tile * (double)nt, chunk_base + c});
      item_inst.push_back(i);
    }
    chunk_base += I.n_chunks;
  }
  if (chunk_base > b->max_items || pool_off > b->pool_bytes) return fail(JET_ERR_INVALID, "internal: work list overflow");
  std::vector<int> order(chunk_base);
  for (int k = 0; k < chunk_base; ++k) order[k] = k;
  std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return cost[x].first > cost[y].first; });
  // the kernel walks items in list order; item ids keep their instance chunk
  // numbering through chunk_base, so list position k maps to item order[k]; the
  // instance lookup table of the items follows
  b->items.assign(order.begin(), order.end());
  b->items.insert(b->items.end(), item_inst.begin(), item_inst.end());
  return JET_OK;
}

}  // namespace

extern "C" {

jet_status jet_batch_create(jet_batch_t* out, int32_t n, const jet_plan_t* plans, int32_t flags) {
  (void)flags;
  if (!out || n < 1 || !plans) return fail(JET_ERR_INVALID, "bad batch arguments");
  *out = nullptr;
  for (int i = 0; i < n; ++i)
    if (!plans[i]) return fail(JET_ERR_INVALID, "plan %d is NULL", i);
  const bool tc = plans[0]->tc;
  for (int i = 1; i < n; ++i) {
    if (plans[i]->tc != tc || plans[i]->fp64 != plans[0]->fp64)
      return fail(JET_ERR_UNSUPPORTED, "batch plans must share the precision family");
    if (plans[i]->cls != plans[0]->cls) return fail(JET_ERR_UNSUPPORTED, "batch plans must share the channel set");
  }
  jet_batch_s* b = new jet_batch_s();
  b->plans.assign(plans, plans + n);
  b->cls = plans[0]->cls;
  b->fp64 = plans[0]->fp64;
  b->tc = tc;
  if (tc) {
    jet_status st = tc_batch_create(b->plans, &b->tcb);
    if (st != JET_OK) {
      delete b;
      return st;
    }
    *out = b;
    return JET_OK;
  }
  // members share the launch: CTAs of kSimtThreads, the units per thread that
  // every member's widths allow, two CTAs per SM where the tiles let them
  b->ru = plans[0]->ru;
  for (int i = 1; i < n; ++i) b->ru = std::min(b->ru, plans[i]->ru);
  size_t smem = 0;
  for (int i = 0; i < n; ++i) {
    int P = plans[i]->P;
    if (!plans[i]->P_fixed)
      P = std::min(P, simt_most_points(plans[i], b->ru, kSimtThreads, !b->fp64 && plans[i]->C >= 10 ? 1 : 2));
    b->P.push_back(P);
    smem = std::max(smem, simt_tile_smem(plans[i], P, kSimtThreads));
  }
  b->smem = smem;
  int per_sm = 0, dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceProp prop;
  cudaError_t e = cudaGetDeviceProperties(&prop, dev);
  if (e == cudaSuccess) e = simt_occupancy(b->cls, b->fp64, b->ru, kSimtThreads, smem, &per_sm);
  if (e != cudaSuccess || per_sm < 1) {
    delete b;
    return e != cudaSuccess ? cuda_fail(e, "batch occupancy") : fail(JET_ERR_UNSUPPORTED, "batch tile does not fit");
  }
  b->ctas_per_sm = std::min(per_sm, 2);
  b->grid = prop.multiProcessorCount * b->ctas_per_sm;
  // the work list holds about three items per CTA, shared by cost: a member may
  // take several times its share (with 16 FP32 members a fixed 16 chunks left the
  // largest member's chunks running alone: 11.0 ms against 3.8 ms)
  b->max_chunks_per_inst = std::min(256, std::max(kSimtBatchChunks, 8 * b->grid / n));
  long long scr = 0, wt = 0, runs = 0;
  for (int i = 0; i < n; ++i) {
    scr = std::max(scr, plans[i]->scratch_stride);
    runs = std::max(runs, plans[i]->wsums_stride);
    b->wt_off.push_back(wt);
    wt += weight_ws_elems(plans[i]->n_params);
  }
  b->scratch_stride = scr;
  b->max_items = n * b->max_chunks_per_inst;
  const size_t elem = b->fp64 ? 8 : 4;
  e = cudaMalloc((void**)&b->d_insts, sizeof(DevInstance) * n);
  if (e == cudaSuccess) e = cudaMalloc((void**)&b->d_item_inst, sizeof(int) * 2 * b->max_items);
  if (e == cudaSuccess) e = cudaMalloc((void**)&b->d_next, sizeof(int));
  if (e == cudaSuccess) e = cudaMalloc((void**)&b->d_jobs, sizeof(ReduceJob) * n);
  if (e == cudaSuccess) e = cudaMalloc((void**)&b->loss_slices, sizeof(double) * b->max_items);
  if (e == cudaSuccess && runs) e = cudaMalloc((void**)&b->run_sums, sizeof(float) * b->grid * (size_t)runs);
  if (e == cudaSuccess) e = cudaMalloc(&b->Wt, elem * std::max<long long>(wt, 1));
  if (e == cudaSuccess) e = cudaMalloc(&b->scratch, elem * (size_t)b->grid * std::max<long long>(scr, 1));
  if (e == cudaSuccess) e = cudaMallocHost((void**)&b->h_insts, sizeof(DevInstance) * n);
  if (e == cudaSuccess) e = cudaMallocHost((void**)&b->h_item_inst, sizeof(int) * 2 * b->max_items);
  if (e == cudaSuccess) e = cudaMallocHost((void**)&b->h_jobs, sizeof(ReduceJob) * n);
  // the pool last: where it does not fit, one for the least bound of chunks
  while (e == cudaSuccess) {
    b->pool_bytes = batch_pool_bytes(b->plans, b->grid, b->max_chunks_per_inst);
    e = cudaMalloc((void**)&b->pool, b->pool_bytes);
    if (e != cudaErrorMemoryAllocation || b->max_chunks_per_inst == kSimtBatchChunks) break;
    cudaGetLastError();
    b->max_chunks_per_inst = kSimtBatchChunks;
    e = cudaSuccess;
  }
  if (e != cudaSuccess) {
    free_batch(b);
    delete b;
    return cuda_fail(e, "batch workspace");
  }
  *out = b;
  return JET_OK;
}

static jet_status batch_run(jet_batch_t b, const void* const* params, void* const* adam_m, void* const* adam_v,
                            int64_t step, long long* step_ctr, float lr, const void* const* X, const int64_t* N,
                            const void* const* source, void* const* grad_out, double* loss_out, bool adam,
                            cudaStream_t s) {
  const int n = (int)b->plans.size();
  jet_status st = batch_prepare(b, params, X, N, source, nullptr);
  if (st != JET_OK) return st;
  const int n_items = (int)b->items.size() / 2;
  std::vector<ReduceJob> jobs(n);
  for (int i = 0; i < n; ++i) {
    jobs[i] = make_job(b->insts[i], adam ? nullptr : grad_out[i], loss_out ? loss_out + i : nullptr, true);
    if (adam) {
      jobs[i].params = (void*)params[i];
      jobs[i].m = adam_m[i];
      jobs[i].v = adam_v[i];
    }
  }
  const DevInstance* d_insts = b->d_insts;
  const int* d_items = b->d_item_inst;
  const ReduceJob* d_jobs = b->d_jobs;
  const size_t b_insts = sizeof(DevInstance) * n, b_items = sizeof(int) * b->items.size(), b_jobs = sizeof(ReduceJob) * n;
  if (stream_is_capturing(s)) {
    const void* src[3] = {b->insts.data(), b->items.data(), jobs.data()};
    const size_t bytes[3] = {b_insts, b_items, b_jobs};
    char* dst[3];
    CK(b->captured.put(s, 3, src, bytes, dst));
    d_insts = reinterpret_cast<const DevInstance*>(dst[0]);
    d_items = reinterpret_cast<const int*>(dst[1]);
    d_jobs = reinterpret_cast<const ReduceJob*>(dst[2]);
  } else {
    if (b->copied) CK(cudaEventSynchronize(b->copied));
    else CK(cudaEventCreateWithFlags(&b->copied, cudaEventDisableTiming));
    memcpy(b->h_insts, b->insts.data(), b_insts);
    memcpy(b->h_item_inst, b->items.data(), b_items);
    memcpy(b->h_jobs, jobs.data(), b_jobs);
    CK(cudaMemcpyAsync(b->d_insts, b->h_insts, b_insts, cudaMemcpyHostToDevice, s));
    CK(cudaMemcpyAsync(b->d_item_inst, b->h_item_inst, b_items, cudaMemcpyHostToDevice, s));
    CK(cudaMemcpyAsync(b->d_jobs, b->h_jobs, b_jobs, cudaMemcpyHostToDevice, s));
    CK(cudaEventRecord(b->copied, s));
  }
  for (int i = 0; i < n; ++i) CK(launch_transpose_weights(b->insts[i], b->fp64, (void*)b->insts[i].Wt, s));
  SimtArgs a;
  memset(&a, 0, sizeof(a));
  a.mode = MODE_FWD_BWD;
  a.n_inst = n;
  a.insts = d_insts;
  a.n_items = n_items;
  a.item_inst = d_items;
  a.scratch = b->scratch;
  a.scratch_stride = b->scratch_stride;
  a.item_next = b->d_next;
  a.ru = b->ru;
  a.threads = kSimtThreads;
  a.carveout = simt_carveout(b->smem, b->ctas_per_sm);
  if (n_items > 0) {  // none: every member is empty
    CK(cudaMemsetAsync(b->d_next, 0, sizeof(int), s));
    CK(simt_launch(b->cls, b->fp64, a, std::min(b->grid, n_items), b->smem, s));
  }
  CK(launch_reduce(jobs.data(), d_jobs, n, b->fp64, adam, step, lr, s, step_ctr));
  return JET_OK;
}

jet_status jet_batch_backward(jet_batch_t b, const void* const* params, const void* const* X, const int64_t* N,
                              const void* const* source, void* const* grad_out, double* loss_out,
                              jet_stream_t stream) {
  if (!b || !params || !X || !N || !grad_out) return fail(JET_ERR_INVALID, "NULL batch argument");
  if (b->tc) return tc_batch_run(b->tcb, b->plans, params, nullptr, nullptr, 0, nullptr, 0.f, X, N, source,
                                 grad_out, loss_out, false, (cudaStream_t)stream);
  return batch_run(b, params, nullptr, nullptr, 0, nullptr, 0.f, X, N, source, grad_out, loss_out, false,
                   (cudaStream_t)stream);
}

static jet_status batch_train(jet_batch_t b, void* const* params, void* const* adam_m, void* const* adam_v,
                              int64_t step, long long* step_ctr, float lr, const void* const* X, const int64_t* N,
                              const void* const* source, double* loss_out, cudaStream_t s) {
  if (!b || !params || !adam_m || !adam_v || !X || !N) return fail(JET_ERR_INVALID, "NULL batch argument");
  if (b->tc) return tc_batch_run(b->tcb, b->plans, (const void* const*)params, adam_m, adam_v, step, step_ctr, lr,
                                 X, N, source, nullptr, loss_out, true, s);
  return batch_run(b, (const void* const*)params, adam_m, adam_v, step, step_ctr, lr, X, N, source, nullptr,
                   loss_out, true, s);
}

jet_status jet_batch_train_step(jet_batch_t b, void* const* params, void* const* adam_m, void* const* adam_v,
                                int64_t step, float lr, const void* const* X, const int64_t* N,
                                const void* const* source, double* loss_out, jet_stream_t stream) {
  if (step < 1) return fail(JET_ERR_INVALID, "step must be >= 1");
  return batch_train(b, params, adam_m, adam_v, step, nullptr, lr, X, N, source, loss_out, (cudaStream_t)stream);
}

jet_status jet_batch_train_step_dev(jet_batch_t b, void* const* params, void* const* adam_m, void* const* adam_v,
                                    int64_t* step_counter, float lr, const void* const* X, const int64_t* N,
                                    const void* const* source, double* loss_out, jet_stream_t stream) {
  if (!step_counter) return fail(JET_ERR_INVALID, "NULL step counter");
  return batch_train(b, params, adam_m, adam_v, 1, reinterpret_cast<long long*>(step_counter), lr, X, N, source,
                     loss_out, (cudaStream_t)stream);
}

jet_status jet_debug_batch_timeout(jet_batch_t b, int32_t code) {
  if (!b || code == 0) return fail(JET_ERR_INVALID, "NULL batch or code 0");
  if (!b->tc) return fail(JET_ERR_UNSUPPORTED, "only the tensor-core forms wait");
  tc_batch_set_timeout(b->tcb, code);
  return JET_OK;
}

jet_status jet_batch_destroy(jet_batch_t b) {
  if (!b) return JET_OK;
  free_batch(b);
  delete b;
  return JET_OK;
}

}  // extern "C"
