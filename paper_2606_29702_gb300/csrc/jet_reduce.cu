// Weight transposition (plus an aligned copy of the parameters), deterministic FP64 gradient/loss reduction over the
// chunk slices, and the fused full-batch Adam update (Sec. 3.1.1).
#include <cmath>

#include "jet_f64.cuh"
#include "jet_internal.h"
#include "jet_pdl.cuh"

namespace jet {

template <class T>
__global__ void transpose_weights_kernel(const __grid_constant__ DevInstance I, T* Wt) {
  dependency_wait();
  const T* P = reinterpret_cast<const T*>(I.params);
  T* Wc = Wt + weight_copy_offset(I.n_params);
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < I.n_params;
       e += (long long)gridDim.x * blockDim.x) {
    Wc[e] = P[e];
    for (int l = 0; l < I.L; ++l) {
      const long long off = I.off_W[l];
      const int fi = I.widths[l], fo = I.widths[l + 1];
      if (e >= off && e < off + (long long)fi * fo) {
        const long long r = e - off;
        const int o = (int)(r / fi), i = (int)(r % fi);
        Wt[off + (long long)i * fo + o] = P[e];
        break;
      }
    }
  }
}

cudaError_t launch_transpose_weights(const DevInstance& in, bool fp64, void* Wt, cudaStream_t s) {
  int grid = (int)((in.n_params + 255) / 256);
  if (grid > 2048) grid = 2048;
  if (grid < 1) grid = 1;
  if (fp64) return launch_dependent(&transpose_weights_kernel<double>, grid, 256, 0, s, in, reinterpret_cast<double*>(Wt));
  return launch_dependent(&transpose_weights_kernel<float>, grid, 256, 0, s, in, reinterpret_cast<float*>(Wt));
}

// Adam (Kingma & Ba 2015) with beta1 = 0.9, beta2 = 0.999, eps = 1e-8; the
// paper fixes only the learning rate (1e-3).  The update runs in the value
// type of the parameters (FP32 for the FP32 and BF16 forms); the gradient it
// takes is the FP64 sum over chunks.
// The 1-based step t is `step`, or *step_ctr + 1 when the counter lives in
// device memory; the bias corrections 1 - beta^t = -expm1(t ln beta) are
// formed on the device in both cases (ln beta from the host), so the two give
// identical updates for the same t.
struct AdamConst {
  double lr, beta1, beta2, eps;
  double ln_beta1, ln_beta2;
  float lr_f, beta1_f, beta2_f, eps_f;
  long long step;
  const long long* step_ctr;
};

// Element i of a job's gradient: the hidden-layer weights first, in the order
// their sums are stored, then the elements of the FP64 slices (consecutive i are
// consecutive addresses in every chunk).  param: its parameter; off: its offset
// in a chunk's sums (hidden) or slice; sub: floats between sub-tiles.
struct GradElem {
  long long param;
  long long off;
  int sub;
  bool hidden;
};
__device__ __forceinline__ GradElem grad_elem(const ReduceJob& J, long long i) {
  if (J.hid == HID_SLICES) return {i, i, 0, false};
  const int* w = J.widths;
  if (i < J.n_hid) {
    int e = (int)i, l = 2;
    long long base = (long long)w[0] * w[1] + w[1], off = 0;  // parameter offset of W^l, sums' offset of the layer
    for (; e >= w[l] * w[l - 1]; ++l) {
      e -= w[l] * w[l - 1];
      base += (long long)w[l] * w[l - 1] + w[l];
      off += (long long)w[l] * w[l - 1] * J.subs;
    }
    const int wi = w[l - 1];
    int u, k;
    if (J.hid == HID_SIMT) {
      const int nkb = wi / 4, it = e / (4 * J.wr), kb = it % nkb;
      u = it / nkb * J.wr + (e >> 2) % J.wr;
      k = kb + (e & 3) * nkb;
    } else if (J.hid == HID_TC) {
      u = (e >> 2) % wi;  // equal widths
      k = e / (4 * wi) * 4 + (e & 3);
    } else {
      u = e / wi;
      k = e - u * wi;
    }
    return {base + (long long)u * wi + k, off + e, w[l] * wi, true};
  }
  const long long j = i - J.n_hid;
  int r = (int)j;
  long long p = 0;
  int n = w[0] * w[1] + w[1];  // W^1, b^1
  for (int l = 2; l < J.L && r >= n; ++l) {  // b^l
    r -= n;
    p += n + (long long)w[l] * w[l - 1];
    n = w[l];
  }
  if (r >= n) {  // W^L, b^L
    r -= n;
    p += n;
  }
  return {p + r, j, 0, false};
}

// A block's 8 warps form 8 / G groups; a group takes 32 consecutive elements
// (lanes over elements, so every chunk's row is read coalesced), its G warps sum
// every G-th chunk in FP64 with eight loads in flight, and the first adds the G
// partials in a fixed order: deterministic.  Bound by the FP64 adds, which run
// at 2 a clock per SM.  G = 8 fills the GPU where there are few parameters and
// many chunks; G = 1 spares the adds of the partials where there are many
// parameters (a step of 64 BF16 networks 6.26 ms with G = 8, 5.91 ms so), except
// for the few elements of many chunks' slices beside FP32 sums, whose serial
// chains would be the tail.  The fused kernels leave their FP32 sums to this
// kernel: a flush of every chunk into FP64 slices took 16% of the composite loss
// 2->64x6->1 FP32 and a fifth of 3->256x8->1 FP32 when it went.
constexpr int kRedWarps = 8;

// warps per group for the FP32 (or finished) hidden-layer sums and for the
// elements of the FP64 slices
__host__ __device__ inline int red_g_hidden(bool many) { return many ? 1 : kRedWarps; }
__host__ __device__ inline int red_g_slices(const ReduceJob& J, bool many) {
  return many && (J.hid == HID_SLICES || J.n_chunks <= 16) ? 1 : kRedWarps;
}
__host__ __device__ inline long long red_hidden(const ReduceJob& J) { return J.hid == HID_SLICES ? 0 : J.n_hid; }
__host__ __device__ inline long long red_blocks(long long elems, int g) {
  const int per = 32 * kRedWarps / g;
  return (elems + per - 1) / per;
}

// sum over the chunks (every G-th from `first`) of one element
template <int G>
__device__ __forceinline__ double chunk_sum(const ReduceJob& J, const GradElem& el, int first) {
  const int gc = J.n_chunks;
  double g = 0.0;
  int c = first;
  if (el.hidden && J.hid == HID_DONE) {
    if (first == 0) g = reinterpret_cast<const double*>(J.hid_sums)[el.off];
  } else if (el.hidden) {
    const float* src = reinterpret_cast<const float*>(J.hid_sums) + el.off + c * J.hid_stride;
    const long long step = G * J.hid_stride;
    for (; c + 7 * G < gc; c += 8 * G, src += 8 * step) {
      float v[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j] = __ldcg(src + j * step);
      for (int q = 1; q < J.subs; ++q)
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] += __ldcg(src + j * step + (long long)q * el.sub);
#pragma unroll
      for (int j = 0; j < 8; ++j) g += widen(v[j]);
    }
#pragma unroll 2
    for (; c < gc; c += G, src += step) {
      float v = __ldcg(src);
      for (int q = 1; q < J.subs; ++q) v += __ldcg(src + (long long)q * el.sub);
      g += widen(v);
    }
  } else {
    const double* src = J.grad_slices + el.off;
    for (; c + 7 * G < gc; c += 8 * G) {
      double v[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j] = src[(long long)(c + j * G) * J.n_slice];
#pragma unroll
      for (int j = 0; j < 8; ++j) g += v[j];
    }
    for (; c < gc; c += G) g += src[(long long)c * J.n_slice];
  }
  return g;
}

struct BiasCorr {
  double c1, c2;
};

// elements [i0, i0 + 32 * kRedWarps / G) of the job, below `end`
template <class T, bool ADAM, int G>
__device__ __forceinline__ void reduce_elems(const ReduceJob& J, const AdamConst& ac, const BiasCorr& bc,
                                             long long i0, long long end, double (*part)[32]) {
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  const long long i = i0 + wp / G * 32 + lane;
  double g = 0.0;
  long long p = 0;
  if (i < end) {
    const GradElem el = grad_elem(J, i);
    p = el.param;
    g = chunk_sum<G>(J, el, wp % G);
  }
  if (G > 1) {
    part[wp][lane] = g;
    __syncthreads();
  }
  if (wp % G != 0 || i >= end) return;
#pragma unroll
  for (int w = 1; w < G; ++w) g += part[wp + w][lane];
  if (J.grad_out) reinterpret_cast<T*>(J.grad_out)[p] = (T)g;
  if (ADAM) {
    T* th = reinterpret_cast<T*>(J.params);
    T* m = reinterpret_cast<T*>(J.m);
    T* v = reinterpret_cast<T*>(J.v);
    if constexpr (sizeof(T) == 4) {
      const float bc1_f = (float)bc.c1, bc2_f = (float)bc.c2;
      const float gf = (float)g;
      const float mm = ac.beta1_f * m[p] + (1.0f - ac.beta1_f) * gf;
      const float vv = ac.beta2_f * v[p] + (1.0f - ac.beta2_f) * gf * gf;
      m[p] = mm;
      v[p] = vv;
      th[p] = th[p] - ac.lr_f * (mm / bc1_f) / (sqrtf(vv / bc2_f) + ac.eps_f);
    } else {
      const double mm = ac.beta1 * (double)m[p] + (1.0 - ac.beta1) * g;
      const double vv = ac.beta2 * (double)v[p] + (1.0 - ac.beta2) * g * g;
      m[p] = (T)mm;
      v[p] = (T)vv;
      const double mhat = mm / bc.c1, vhat = vv / bc.c2;
      th[p] = (T)((double)th[p] - ac.lr * mhat / (sqrt(vhat) + ac.eps));
    }
  }
}

// Blocks of a job: the hidden-layer sums, then the elements of the slices.  The
// chunk losses are summed by all threads of its first block in a fixed tree:
// one thread adding 304 of them one after another took 22 us (forward pass at
// 10000 points), the tree 4 us.
template <class T, bool ADAM>
__global__ void __launch_bounds__(32 * kRedWarps) reduce_kernel(const __grid_constant__ ReduceJob job0,
                                                                const ReduceJob* jobs, bool many, AdamConst ac) {
  dependency_wait();
  const ReduceJob& J = jobs ? jobs[blockIdx.y] : job0;
  // the grid covers the largest job: blocks past this job's have nothing to do
  // (block 0 stays: it writes the loss, also of loss-only jobs)
  const long long nh = red_hidden(J);
  const int gh = red_g_hidden(many), gs = red_g_slices(J, many);
  const long long bh = red_blocks(nh, gh), b = blockIdx.x;
  const bool hidden = b < bh;
  const long long i0 = hidden ? b * (32 * kRedWarps / gh) : nh + (b - bh) * (32 * kRedWarps / gs);
  const long long end = hidden ? nh : J.n_params;
  if (b > 0 && i0 >= end) return;
  __shared__ double part[kRedWarps][32];
  // bias corrections: one thread per block, one expm1 each (FP32 for the
  // FP32 update; FP64 arithmetic is slow on this GPU)
  __shared__ BiasCorr bc_s;
  if (ADAM) {
    if (threadIdx.x == 0) {
      const long long t = ac.step_ctr ? *ac.step_ctr + 1 : ac.step;
      if (sizeof(T) == 4) {
        bc_s.c1 = (double)-expm1f((float)((double)t * ac.ln_beta1));
        bc_s.c2 = (double)-expm1f((float)((double)t * ac.ln_beta2));
      } else {
        bc_s.c1 = -expm1((double)t * ac.ln_beta1);
        bc_s.c2 = -expm1((double)t * ac.ln_beta2);
      }
    }
    __syncthreads();
  }
  const BiasCorr bc = ADAM ? bc_s : BiasCorr{1.0, 1.0};
  if (i0 < end) {
    if ((hidden ? gh : gs) == 1) reduce_elems<T, ADAM, 1>(J, ac, bc, i0, end, part);
    else reduce_elems<T, ADAM, kRedWarps>(J, ac, bc, i0, end, part);
  }
  if (b == 0 && J.loss_out) {
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    double s = 0.0;
    for (int c = threadIdx.x; c < J.n_chunks; c += 32 * kRedWarps) s += J.loss_slices[c];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    __syncthreads();  // part's readers are done
    if (lane == 0) part[wp][0] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
      s = 0.0;
#pragma unroll
      for (int w = 0; w < kRedWarps; ++w) s += part[w][0];
      *J.loss_out = s * J.inv_N;
    }
  }
}

// the device step counter advances once the update that read it is done
__global__ void adam_advance_kernel(long long* step_ctr) {
  dependency_wait();
  *step_ctr += 1;
}

cudaError_t launch_reduce(const ReduceJob* jobs, const ReduceJob* dev_jobs, int n, bool fp64, bool adam,
                          long long step, float lr, cudaStream_t s, long long* step_ctr) {
  AdamConst ac;
  ac.lr = lr;
  ac.beta1 = 0.9;
  ac.beta2 = 0.999;
  ac.eps = 1e-8;
  ac.ln_beta1 = std::log(ac.beta1);
  ac.ln_beta2 = std::log(ac.beta2);
  ac.lr_f = lr;
  ac.beta1_f = 0.9f;
  ac.beta2_f = 0.999f;
  ac.eps_f = 1e-8f;
  ac.step = step < 1 ? 1 : step;
  ac.step_ctr = adam ? step_ctr : nullptr;
  // G = 1 once a warp per 32 parameters is 64 warps on each of 152 SMs and more
  // (with few it is slower: 2->64x5->1 FP32, 304 chunks, 1.342 ms against 1.331 ms).
  // A constant, so that the order of a sum does not follow the device.
  long long params = 0, gx = 1;
  for (int i = 0; i < n; ++i) params += jobs[i].n_params;
  const bool many = params >= 32LL * 64 * 152;
  for (int i = 0; i < n; ++i) {
    const long long nh = red_hidden(jobs[i]);
    const long long blocks = red_blocks(nh, red_g_hidden(many)) +
                             red_blocks(jobs[i].n_params > nh ? jobs[i].n_params - nh : 0, red_g_slices(jobs[i], many));
    gx = blocks > gx ? blocks : gx;
  }
  const dim3 grid((unsigned)gx, (unsigned)n);
  const ReduceJob* dj = n == 1 ? nullptr : dev_jobs;
  const int threads = 32 * kRedWarps;
  cudaError_t e;
  if (fp64) {
    e = launch_dependent(adam ? &reduce_kernel<double, true> : &reduce_kernel<double, false>, grid, threads, 0, s, jobs[0], dj, many, ac);
  } else {
    e = launch_dependent(adam ? &reduce_kernel<float, true> : &reduce_kernel<float, false>, grid, threads, 0, s, jobs[0], dj, many, ac);
  }
  if (e == cudaSuccess && adam && step_ctr) e = launch_dependent(&adam_advance_kernel, 1, 1, 0, s, step_ctr);
  return e;
}

}  // namespace jet
