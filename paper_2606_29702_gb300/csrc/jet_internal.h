// Internal structures shared by the host orchestration (jet_api.cu) and the
// kernels.  Not part of the public ABI.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace jet {

constexpr int kMaxLayers = 16;   // weight layers
constexpr int kMaxTerms = 32;    // residual monomials over all components
constexpr int kMaxRes = 4;
constexpr int kMaxOut = 4;
constexpr int kMaxC = 16;

// One residual monomial: coef * prod fac, fac = o * C + channel index; bit f
// of pmask: factor f is read at the second point of a pair (paired loss terms).
struct DevTerm {
  double coef;
  int comp;
  int nfac;
  int fac[4];
  int pmask;
};

// One term of a composite loss (Sec. 3.1.1: weighted IC, BC and PDE terms over
// their own blocks of the concatenated points): the points [start, start +
// count), its monomials [t0, t1), scale = weight / (residuals of the term).
// A paired term has one residual per consecutive pair of points, evaluated at
// the pair's first point.
constexpr int kMaxGroups = 4;
struct DevGroup {
  long long start, count;
  double scale;
  int t0, t1;
  int n_res, paired, has_source;
};

// Kernel modes
enum : int {
  MODE_FWD = 0,        // residual + loss (+ z-jet store when store != null)
  MODE_FWD_BWD = 1,    // residual + loss + gradient, hidden jets recomputed per tile
  MODE_BWD_STORE = 2,  // gradient from a z-jet store written by MODE_FWD
};

// Everything a kernel needs to know about one PINN instance for one call.
struct alignas(16) DevInstance {
  int L;               // weight layers
  int d, n_out, n_res;
  int widths[kMaxLayers + 1];
  long long off_W[kMaxLayers];  // offsets (elements) into the packed params
  long long off_b[kMaxLayers];
  long long n_params;
  const void* params;  // packed, value type T
  const void* Wt;      // weight workspace, value type T: the packed parameters
                       // with every W^l transposed, then (at weight_copy_offset)
                       // a 16-byte-aligned copy of the packed parameters
  const void* X;       // [N][d]
  const void* source;  // [N][n_res] or null
  void* r_out;         // [N][n_res] or null
  long long N;
  double inv_N;
  int n_terms;
  DevTerm terms[kMaxTerms];
  // composite loss (0: one residual over all points, mean over N)
  int n_groups;
  DevGroup groups[kMaxGroups];
  // tiling
  int P;               // points per tile
  int P0;              // FP32 SIMT forms: points per weight-gradient group (P = V * P0); FP64: P
  int swap;            // odd points keep their channels in swapped pairs (simt_swap)
  int wr;              // rows of a weight-gradient item
  int unit;            // points per unit of the chunk partition (P or P0)
  int pitch;           // smem row pitch (elements) of a jet buffer, >= C * P
  long long n_tiles;    // partition units
  int tiles_per_chunk;  // units of every chunk; the first chunk_rem chunks take one more
  int chunk_rem;
  int n_chunks;
  int chunk_base;      // first work-item index of this instance
  // outputs of the chunk reduction (FP64): [n_chunks][n_slice], [n_chunks].
  // A slice holds every parameter (n_slice = n_params), or, with FP32 chunk sums
  // of the hidden-layer weights (wsums_direct), the others only (SliceMap)
  double* grad_slices;
  double* loss_slices;
  int n_slice;
  int goff_b[kMaxLayers];  // offsets of b^l and W^L in a slice (W^1 is first)
  int goff_WL;
  // z-jet store for MODE_FWD / MODE_BWD_STORE: per tile, per hidden layer,
  // [w][C * P] (as the shared-memory rows); null if not stored
  void* store;
  long long store_tile_stride;  // elements per tile
  // FP32 forms: FP32 sums of the hidden-layer weight gradients (simt_wacc_elems
  // floats, in the item order of the weight gradient), or null: FP64 adds per
  // tile.  wsums_direct: of each chunk, and the reduction reads them; else of each
  // CTA's running chunk, which adds them to its slice after every kWaccTiles tiles
  float* wsums;
  long long wsums_stride;
  int wsums_direct;
};

// Layout of an FP64 slice without the hidden-layer weights: W^1, b^1, b^2 ..
// b^{L-1}, W^L, b^L.  Fills the offsets and returns the slice's elements.
inline int slice_map(const int* widths, int L, int* goff_b, int* goff_WL) {
  int n = widths[0] * widths[1];
  for (int l = 1; l < L; ++l) {
    goff_b[l - 1] = n;
    n += widths[l];
  }
  *goff_WL = n;
  n += widths[L - 1] * widths[L];
  goff_b[L - 1] = n;
  return n + widths[L];
}

// Per-launch arguments of the fused SIMT kernel.
struct SimtArgs {
  int mode;
  int n_inst;
  const DevInstance* insts;   // device array (batched) or null
  DevInstance inst0;          // single-instance launches pass it by value
  int n_items;                // total work items (instance, chunk)
  int ru;                     // units per thread of the jet GEMMs (simt_units)
  int threads;                // CTA size
  int carveout;               // percent of the SM's 228 KB kept as shared memory (simt_carveout)
  const int* item_inst;       // [n_items] instance of each item (batched) or null
  void* scratch;              // per-CTA z-jet scratch
  long long scratch_stride;   // elements per CTA slot
  // batches: counter of the items taken after each CTA's first (zeroed before
  // the launch), so that a CTA that finishes takes the next item of the
  // cost-ordered list; null: a fixed stride
  int* item_next;
};

constexpr int kSimtThreads = 256;  // CTA of the no-alloc path and of batches
constexpr int kSimtRed = 128;      // doubles of the SIMT kernels' reduction area
// Weights of a jet GEMM pass through shared memory in two row slabs: 4 KB each
// up to width 64 (a 64 x 64 FP32 layer takes four), where two CTAs of 32 points
// then fit an SM with six channels (with 8 KB 2->64x5->1 FP32 takes 1.385 against
// 1.331 ms); 8 KB up to width 128; 16 KB above (a 256 x 256 layer takes 16; with 8
// KB its barriers cost 4% when it was set, while 3->256x8->1 now takes 9.86 ms with
// 8 KB and 10.14 ms with 16).
__host__ __device__ inline int simt_slab_elems(int wmax, size_t elem) {
  const int cap = (wmax <= 64 ? 4096 : wmax <= 128 ? 8192 : 16384) / (int)elem, need = wmax * wmax;
  return need < cap ? need : cap;
}
// FP64 form: adjacent lanes that share a weight-gradient item (4 x 4), each
// summing every NS-th vector of jet columns: as many as fill the CTA.
__host__ __device__ inline int simt_wgrad_slices(int items, int threads) {
  int ns = 1;
  while (ns < 8 && items * ns * 2 <= threads) ns *= 2;
  return ns;
}
// FP32 forms: the FP32 sums of a weight gradient run over groups of P0 points in
// two chains, the even and the odd columns of a point stride of S0 = C or C | 1,
// whatever the tile: tiles of V groups leave every sum as a tile of one group
// forms it, and the rounding of a gradient does not depend on the tile.
inline int simt_group_points(int wmax) { return 4 * (256 / wmax > 0 ? 256 / wmax : 1); }
// Where S0 = C | 1 != C (C even), the even columns of an odd point are its odd
// channels: such points keep their channels in swapped pairs, so that column
// parity is chain parity at the dense stride C too.
inline int simt_swap(int C, int P0) {
  const int lanes = P0 < 32 ? P0 : 32;
  return C % 2 == 0 && (C & -C) * lanes > 32 ? 1 : 0;
}
// Row pitch (elements) of a SIMT jet buffer of C * P columns.  The weight
// gradient's 16-byte loads walk 8 rows per quarter warp (FP64: 8 / NS rows x NS
// vectors): the pitch in 16-byte units is odd (NS modulo 2 NS), so that they hit
// distinct banks.
inline int simt_pitch(int C, int P, int wmax, int threads, size_t elem) {
  const int v = 16 / (int)elem;
  const int ns = elem == 4 ? 1 : simt_wgrad_slices((wmax / 4) * (wmax / 4), threads);
  int p = (C * P + v - 1) / v * v;
  while ((p / v) % (2 * ns) != ns) p += v;
  return p;
}
// Consecutive units per thread of the SIMT jet GEMMs.  FP64 takes one: its pipe
// costs a warp the same however many lanes work, and single units fill the
// warps of narrow layers (20 units x 8 points: 5 warps of 5, not 2.5 of 3).
inline int simt_units(const int* widths, int L, bool fp64) {
  if (fp64) return 1;
  for (int l = 1; l < L; ++l)
    if (widths[l] % 8) return 4;
  return 8;
}
// Rows of a weight-gradient item (x 4 columns): 4, fewer where that leaves threads
// without one (4 for all: sixteen FP32 networks of widths 32 to 128 3.88 against
// 3.82 ms; 8 rows read a quarter fewer words per FMA, but their 32 packed sums
// spilled: 2->64x5->1, C = 6, 1.37 against 1.32 ms when tried).
inline int simt_wgrad_rows(int ru, int wmax, int V, int threads, bool fp64) {
  const bool few = (long long)(wmax / 4) * (wmax / 4) * (V > 1 ? 2 : 1) < threads;
  return fp64 || !few ? 4 : ru == 8 ? 2 : 1;
}
constexpr int kWaccTiles = 64;     // tiles per FP32 weight-gradient run (channel sets of 7 or more)
// share of L2 the per-chunk FP64 gradient slices may take before the kernels
// accumulate a chunk's weight gradients in FP32 instead of adding per tile
constexpr double kSimtSliceL2Bytes = 48.0 * 1024 * 1024;
// FP32 forms: elements of a chunk's FP32 weight-gradient sums, one float per
// weight of every hidden-to-hidden layer W^l (l = 2 .. L-1, [w_l][w_{l-1}])
inline long long simt_wacc_elems(const int* widths, int L, bool fp64) {
  if (fp64) return 0;
  long long e = 0;
  for (int l = 2; l <= L - 1; ++l) e += (long long)widths[l] * widths[l - 1];
  return e;
}
// elements of the SIMT weight workspace: transposed copy, then aligned copy
__host__ __device__ inline long long weight_copy_offset(long long n_params) { return (n_params + 3) & ~3LL; }
__host__ __device__ inline long long weight_ws_elems(long long n_params) { return 2 * weight_copy_offset(n_params); }
// Dynamic shared memory of the fused SIMT kernel: two jet buffers
// [wmax][pitch], two weight slabs, output jets and adjoints [n_out*C][P], tile
// points [P][d], and a small reduction area.
inline size_t simt_smem_bytes(int C, int P, int pitch, int wmax, int n_out, int d, size_t elem) {
  size_t e = 2 * (size_t)wmax * pitch + 2 * (size_t)simt_slab_elems(wmax, elem) + 2 * (size_t)n_out * C * P +
             (size_t)P * d;
  size_t bytes = (e * elem + 15) / 16 * 16;
  return bytes + kSimtRed * sizeof(double);
}
// shared memory an SM spends on a CTA besides the dynamic part: the kernel's
// static arrays (the instance descriptor and the item index) and the reserve
constexpr size_t kSimtSmBytes = 228 * 1024;
constexpr size_t kSimtCtaBytes = sizeof(DevInstance) + 16 + 1024;
// Carve-out that holds `ctas` resident CTAs; the rest of the SM's 256 KB stays
// L1 (sixteen FP32 networks 3.92 ms with all of it shared memory, 3.82 ms with what
// two CTAs need; 2->64x6->1 composite loss at 12101 points 304 and 301 us).
inline int simt_carveout(size_t smem, int ctas) {
  const size_t pct = ((smem + kSimtCtaBytes) * ctas * 100 + kSimtSmBytes - 1) / kSimtSmBytes;
  return pct > 100 ? 100 : (int)pct;
}
// the chunks of a call: its units (tiles) over n_chunks CTAs or work items.  No
// points (an empty member of a batch): no chunk, so every sum over them is zero.
inline void simt_set_chunks(DevInstance& I, long long n_chunks) {
  I.unit = I.P;
  I.n_tiles = (I.N + I.unit - 1) / I.unit;
  if (n_chunks < 1) n_chunks = 1;
  if (n_chunks > I.n_tiles) n_chunks = I.n_tiles;
  I.n_chunks = (int)n_chunks;
  if (n_chunks == 0) {
    I.tiles_per_chunk = I.chunk_rem = 0;
    return;
  }
  I.tiles_per_chunk = (int)(I.n_tiles / n_chunks);
  I.chunk_rem = (int)(I.n_tiles % n_chunks);
}

// Where a call's weight-gradient sums go (after simt_set_chunks).  With FP32 sums
// the reduction reads them, unless a chunk of a wide channel set has more tiles
// than one run.
inline void simt_set_sums(DevInstance& I, int C, float* wsums, long long stride) {
  I.wsums = wsums;
  I.wsums_stride = stride;
  I.wsums_direct = wsums && (C < 7 || (I.tiles_per_chunk + (I.chunk_rem > 0 ? 1 : 0)) * (I.unit / I.P0) <= kWaccTiles) ? 1 : 0;
  if (I.wsums_direct) {
    I.n_slice = slice_map(I.widths, I.L, I.goff_b, &I.goff_WL);
  } else {
    I.n_slice = (int)I.n_params;
    for (int l = 0; l < I.L; ++l) I.goff_b[l] = (int)I.off_b[l];
    I.goff_WL = (int)I.off_W[I.L - 1];
  }
}

// Reductions and elementwise kernels (jet_reduce.cu)
// One reduction job per instance: grad[p] = sum_c slices[c][p] in FP64 (fixed
// order), loss = inv_N * sum_c loss_slices[c]; optionally fused with Adam.
// Where the hidden-layer weight gradients of a job are.
enum : int {
  HID_SLICES = 0,  // in the FP64 slices, with all other parameters
  HID_SIMT = 1,    // FP32 sums per chunk, in the item order of the SIMT weight gradient
  HID_TC = 2,      // FP32 sums per chunk and sub-tile, [k / 4][u][4] per layer (tensor-core kernel)
  HID_DONE = 3,    // one FP64 sum each, in parameter order (weight-gradient GEMM)
};
struct ReduceJob {
  const double* grad_slices;  // [n_chunks][n_slice]
  const double* loss_slices;
  int n_chunks;
  int n_slice;
  long long n_params;
  int hid;            // HID_*
  int L;              // for hid != HID_SLICES: the network's layers and widths,
  int widths[kMaxLayers + 1];
  int n_hid;          // its hidden-layer weights,
  int subs;           // HID_TC: sub-tiles summed in FP32 per chunk
  int wr;             // HID_SIMT: rows of a weight-gradient item
  const void* hid_sums;       // float [n_chunks][hid_stride], or HID_DONE double [n_hid]
  long long hid_stride;
  double inv_N;
  void* grad_out;     // value type T or null
  double* loss_out;   // or null
  void* params;       // Adam: updated in place (value type T)
  void* m;
  void* v;
};
cudaError_t launch_transpose_weights(const DevInstance& in, bool fp64, void* Wt, cudaStream_t s);
// jobs: host array (copied by value when n == 1); dev_jobs: the same on the
// device when n > 1.  Adam takes step t = `step`, or *step_ctr + 1 with a device
// counter, which the call then increments on the stream.
cudaError_t launch_reduce(const ReduceJob* jobs, const ReduceJob* dev_jobs, int n, bool fp64, bool adam,
                          long long step, float lr, cudaStream_t s, long long* step_ctr = nullptr);

}  // namespace jet

namespace jet {
// Sets the thread-local message returned by jet_last_error() (jet_api.cu).
void set_last_error(const char* msg);

// Per-class entry points, one explicit specialisation per instantiation unit.
template <int ID> cudaError_t simt_launch_id(bool fp64, const SimtArgs& a, int grid, size_t smem, cudaStream_t s);
template <int ID> cudaError_t simt_max_active_id(bool fp64, int ru, int threads, size_t smem, int* blocks);
template <int ID> cudaError_t debug_activation_id(int kind, long long n, const double* z, const double* v,
                                                  double* out, cudaStream_t s);
}  // namespace jet
