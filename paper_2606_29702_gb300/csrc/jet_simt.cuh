// Fused SIMT partial-jet kernel (FP64 and plain FP32 forms).
//
// One persistent launch walks a list of work items (instance, chunk of point
// tiles).  For every tile of P collocation points a CTA runs, on chip:
//
//   forward   layer 1 seed (z^1_0 = W^1 x + b^1, z^1_{e_i} = W^1[:, i], higher
//             channels 0), then for every hidden layer the jet GEMM
//             Z^l = W^l A^{l-1} over all C channels with the bias on the value
//             channel only (Eq. 1-3, Sec. 2.2 "fused GEMM"), and the closed-
//             form tanh jet composition in registers (Eq. 2-3 recursion);
//   output    linear output layer on every channel, residual monomials,
//             loss partial (FP64);
//   backward  residual adjoint ub = (2 r / N) dr/du, output-layer adjoint,
//             then for l = L-1 .. 1: activation-jet adjoint (transpose of the
//             composition), weight gradient sum_cols Zb A^T, bias gradient on
//             the value channel, data gradient W^T Zb.
//
// Jets live in shared memory as [unit][point-major column] rows: column =
// n * C + alpha (FP32: in swapped channel pairs at odd points where I.swap says so;
// columns past C * P stay zero).  In the jet GEMMs a thread owns
// one point and RU consecutive units with every channel, so the composition
// and its adjoint are thread-local; the layer's weights pass through shared
// memory in row slabs.  The hidden z-jets of a tile are written to a per-CTA
// global scratch slot (or to a full-size store) as [unit][alpha * P + n] in the
// forward and read back in the backward, with tanh z in place of the value
// channel (the activation rule and its adjoint read z_0 only through tanh z_0):
// the memory of the backward is bounded by the number of CTAs, not by N.
// Gradient partial sums go to a per-(instance, chunk) FP64 slice; every slice
// element is added by one thread, group of points after group in the order of the
// tiles (fire-and-forget FP64 adds), so the final FP64 reduction is
// deterministic.  With a thread per group of a tile the biases, W^1 and W^L had
// no order: gradients whose sums cancel moved in the fourth digit; one thread per
// element costs at most 1% (2->64x5->1 FP32 1.319 -> 1.331 ms, 16 FP32 networks
// 3.80 -> 3.82 ms, 2->64x6->1 composite loss 304 -> 301 us).
//
// What bounds it: the FP32 pipe and shared-memory reads in the jet GEMMs
// (about 80% of the time), the FP64 pipe in the FP64 form.  Against the form
// with three jet buffers, 4 units per thread, weights read through L1, one
// lane per weight-gradient item and tiles that did not depend on N:
// 3->256x8->1 FP32 at N = 16385 19.29 -> 10.14 ms, 2->64x5->1 (C = 6) FP32 at
// 65536 1.769 -> 1.331 ms, 2->20x4->1 FP64 at 1000 343 -> 77 us.
#pragma once

#include <type_traits>

#include "jet_closures_gen.h"
#include "jet_f2.cuh"
#include "jet_f64.cuh"
#include "jet_groups.cuh"
#include "jet_internal.h"
#include "jet_pdl.cuh"

namespace jet {

template <class T> struct Vec;
template <> struct Vec<float> { static constexpr int N = 4; using type = float4; };
template <> struct Vec<double> { static constexpr int N = 2; using type = double2; };

template <class T> __device__ __forceinline__ T dev_tanh(T z);
template <> __device__ __forceinline__ float dev_tanh<float>(float z) { return tanhf(z); }
template <> __device__ __forceinline__ double dev_tanh<double>(double z) { return tanh(z); }

// p[k] = tanh^(k)(z) for k < NP, as polynomials of a = tanh z and s = 1 - a^2.
template <class T, int NP>
__device__ __forceinline__ void tanh_polys(T a, T* p) {
  const T a2 = a * a;
  const T s = T(1) - a2;
  p[0] = a;
  if (NP > 1) p[1] = s;
  if (NP > 2) p[2] = T(-2) * a * s;
  if (NP > 3) p[3] = s * (T(6) * a2 - T(2));
  if (NP > 4) p[4] = T(8) * a * s * (T(2) - T(3) * a2);
  if (NP > 5) p[5] = T(8) * s * (T(15) * a2 * a2 - T(15) * a2 + T(2));
}

template <class T, int NP>
__device__ __forceinline__ void tanh_derivs(T z, T* p) {
  tanh_polys<T, NP>(dev_tanh<T>(z), p);
}

// tanh_polys of two values in a packed pair
template <int NP>
__device__ __forceinline__ void tanh_polys_pair(f2 a, f2* p) {
  const f2 a2 = a * a;
  const f2 s = jfma(f2(-1.0f), a2, f2(1.0f));
  p[0] = a;
  if (NP > 1) p[1] = s;
  if (NP > 2) p[2] = f2(-2.0f) * a * s;
  if (NP > 3) p[3] = s * jfma(f2(6.0f), a2, f2(-2.0f));
  if (NP > 4) p[4] = f2(8.0f) * a * s * jfma(f2(-3.0f), a2, f2(2.0f));
  if (NP > 5) p[5] = f2(8.0f) * s * jfma(a2, jfma(f2(15.0f), a2, f2(-15.0f)), f2(2.0f));
}

template <class T>
__device__ __forceinline__ void vload(const T* p, T* out) {
  using V = typename Vec<T>::type;
  V v = *reinterpret_cast<const V*>(p);
  const T* q = reinterpret_cast<const T*>(&v);
#pragma unroll
  for (int j = 0; j < Vec<T>::N; ++j) out[j] = q[j];
}

// the C channels of one (unit, point) in a jet row: 16-byte accesses where the
// element count divides, else 8-byte or scalar ones (rows start on 16 bytes)
template <class T, int C>
__device__ __forceinline__ void load_chan(const T* p, T* v) {
  if constexpr (sizeof(T) == 4 && C % 4 != 0 && C % 2 == 0) {
#pragma unroll
    for (int c = 0; c < C; c += 2) {
      const float2 t = *reinterpret_cast<const float2*>(p + c);
      v[c] = t.x;
      v[c + 1] = t.y;
    }
  } else if constexpr (C % Vec<T>::N == 0) {
#pragma unroll
    for (int c = 0; c < C; c += Vec<T>::N) vload<T>(p + c, v + c);
  } else {
#pragma unroll
    for (int c = 0; c < C; ++c) v[c] = p[c];
  }
}
template <class T, int C>
__device__ __forceinline__ void store_chan(T* p, const T* v) {
  if constexpr (sizeof(T) == 4 && C % 4 == 0) {
#pragma unroll
    for (int c = 0; c < C; c += 4) *reinterpret_cast<float4*>(p + c) = make_float4(v[c], v[c + 1], v[c + 2], v[c + 3]);
  } else if constexpr (sizeof(T) == 4 && C % 2 == 0) {
#pragma unroll
    for (int c = 0; c < C; c += 2) *reinterpret_cast<float2*>(p + c) = make_float2(v[c], v[c + 1]);
  } else if constexpr (sizeof(T) == 8 && C % 2 == 0) {
#pragma unroll
    for (int c = 0; c < C; c += 2) *reinterpret_cast<double2*>(p + c) = make_double2(v[c], v[c + 1]);
  } else {
#pragma unroll
    for (int c = 0; c < C; ++c) p[c] = v[c];
  }
}

// 16 bytes from global to shared memory, asynchronously
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait0() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// p[0..3] += (a, b, c, d) in global memory as one fire-and-forget FP32
// vector reduction (16-byte aligned; no value comes back, so nothing waits)
__device__ __forceinline__ void red_add_v4(float* p, float a, float b, float c, float d) {
  asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
}

// The FP32 weight-gradient sums of a chunk, [item][WR][4] per layer as the items
// of SimtTile::wgrad, zeroed and added to the FP64 slice where a chunk is longer
// than one run (functions of their own, called once per run: inlined they would
// cost the tile's registers)
static __device__ __noinline__ void simt_wacc_zero(float* acc, const DevInstance& I) {
  long long n4 = 0;
  for (int l = 2; l < I.L; ++l) n4 += (long long)I.widths[l] * I.widths[l - 1] / 4;
  for (long long i = threadIdx.x; i < n4; i += blockDim.x)
    reinterpret_cast<float4*>(acc)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
}
// accumulator -> FP64 slice (consecutive threads read consecutive floats;
// eight loads in flight before their adds)
static __device__ __noinline__ void simt_wacc_flush(const float* a, const DevInstance& I, double* g) {
  const int NT = blockDim.x, WR = I.wr;
  for (int l = 2; l <= I.L - 1; ++l) {
    const int wo = I.widths[l], wi = I.widths[l - 1], nkb = wi / 4, n = wo * wi;
    double* gW = g + I.off_W[l - 1];
    for (int e0 = threadIdx.x; e0 < n; e0 += 8 * NT) {
      float v[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j] = e0 + j * NT < n ? __ldcg(a + e0 + j * NT) : 0.f;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int e = e0 + j * NT;
        if (e >= n) break;
        const int it = e / (4 * WR), r = (e >> 2) % WR, s = e & 3;
        const int kb = it % nkb, ub = it / nkb;
        atomicAdd(gW + (ub * WR + r) * wi + kb + s * nkb, widen(v[j]));
      }
    }
    a += n;
  }
}

template <class Cls, class T, int RU_>
struct SimtTile {
  static constexpr int C = Cls::C;
  static constexpr int NP = Cls::NP;
  static constexpr int TP = Vec<T>::N;
  static constexpr bool F32 = sizeof(T) == 4;
  static constexpr int RU = RU_;  // consecutive units per thread of the jet GEMMs
  static constexpr int EU = TP;   // consecutive units per thread of the elementwise phases
  // k steps of the jet GEMMs unrolled together: two where the sums and four
  // steps' operands would exceed the registers, else four (3->256x8->1, C = 7 at
  // 512 threads, 12.8 ms with four and 11.8 ms with two when it was set; with the
  // sums of the weight gradient in registers 9.94 and 10.14 ms)
  static constexpr int UK = C >= 7 ? 2 : 4;

  const DevInstance& I;
  const SimtArgs& A;
  const int NT;  // threads of the CTA
  T *B0, *B1;  // jet buffers [wmax][pitch]
  T* WS;     // two weight slabs
  T* UO;     // output jets [n_out*C][P]
  T* UB;     // output adjoints [n_out*C][P]
  T* XS;     // tile points [P][d]
  double* RED;
  int P, pitch, wmax;
  int P0, V;    // points per weight-gradient group, groups per tile
  bool swap;    // odd points keep their channels in swapped pairs
  int slab;     // elements of a weight slab
  int wst = 0;  // slab that holds, or waits for, the next GEMM's first rows
  const T* params;
  const T* Wt;  // transposed weights [in][out] per layer
  const T* Wc;  // aligned copy of the packed parameters
  // FP32 forms: the chunk's hidden-layer weight gradients add up in FP32
  // (fire-and-forget vector reductions; every element belongs to one thread,
  // which adds the tiles in program order).  Null: FP64 adds per tile.
  float* wacc_base = nullptr;
  bool wacc_first = false;  // the running tile stores its sums instead of adding them

  __device__ SimtTile(const DevInstance& I_, const SimtArgs& A_, unsigned char* smem, int chunk)
      : I(I_), A(A_), NT(blockDim.x) {
    P = I.P;
    pitch = I.pitch;
    P0 = I.P0;
    V = P / P0;
    swap = F32 && C % 2 == 0 && I.swap;
    wmax = 0;
    for (int l = 1; l < I.L; ++l) wmax = max(wmax, I.widths[l]);
    slab = simt_slab_elems(wmax, sizeof(T));
    T* base = reinterpret_cast<T*>(smem);
    const size_t be = (size_t)wmax * pitch;
    B0 = base;
    B1 = base + be;
    WS = base + 2 * be;
    UO = WS + 2 * slab;
    UB = UO + (size_t)I.n_out * C * P;
    XS = UB + (size_t)I.n_out * C * P;
    size_t off = (size_t)(XS - base) + (size_t)P * I.d;
    off = (off * sizeof(T) + 15) / 16 * 16;
    RED = reinterpret_cast<double*>(smem + off);
    params = reinterpret_cast<const T*>(I.params);
    Wt = reinterpret_cast<const T*>(I.Wt);
    Wc = Wt + weight_copy_offset(I.n_params);
    if (F32 && I.wsums) wacc_base = I.wsums + (long long)(I.wsums_direct ? chunk : (int)blockIdx.x) * I.wsums_stride;
  }

  // a point's channels in a jet row: exchange of channel pairs (see I.swap)
  __device__ __forceinline__ bool odd(int n) const { return swap && (n & 1); }
  static __device__ __forceinline__ void swap_pairs(T* v) {
#pragma unroll
    for (int c = 0; c + 1 < C; c += 2) {
      const T t = v[c];
      v[c] = v[c + 1];
      v[c + 1] = t;
    }
  }
  __device__ __forceinline__ void load_point(const T* row, int n, T* v) const {
    load_chan<T, C>(row + n * C, v);
    if (odd(n)) swap_pairs(v);
  }
  __device__ __forceinline__ void store_point(T* row, int n, T* v) const {
    if (odd(n)) swap_pairs(v);
    store_chan<T, C>(row + n * C, v);
  }

  // accumulator of W^l (l = 2..L-1): [item][wr][4] per thread item of wgrad
  __device__ float* wacc(int l) const {
    long long off = 0;
    for (int k = 2; k < l; ++k) off += (long long)I.widths[k] * I.widths[k - 1];
    return wacc_base + off;
  }
  __device__ const T* W(int l) const { return params + I.off_W[l - 1]; }   // l = 1..L
  __device__ const T* bias(int l) const { return params + I.off_b[l - 1]; }

  // hidden layer z-jet location for tile t, hidden layer l (1..L-1)
  __device__ T* zjet(long long tile, int l, bool to_store) const {
    long long off = 0;
    for (int k = 1; k < l; ++k) off += (long long)C * P * I.widths[k];
    if (to_store) return reinterpret_cast<T*>(I.store) + tile * I.store_tile_stride + off;
    return reinterpret_cast<T*>(A.scratch) + (long long)blockIdx.x * A.scratch_stride + off;
  }

  // ---------------------------------------------------------------- weights
  // The weight rows [K][wo] of one jet GEMM: W^l transposed (forward) or W^l
  // (data gradient), both 16-byte aligned in the weight workspace.
  struct Rows {
    const T* p;
    int K, wo;
  };
  __device__ Rows fwd_rows(int l) const { return {Wt + I.off_W[l - 1], I.widths[l - 1], I.widths[l]}; }
  __device__ Rows bwd_rows(int l) const { return {Wc + I.off_W[l - 1], I.widths[l], I.widths[l - 1]}; }
  __device__ int slab_rows(const Rows& w) const { return min(w.K, slab / w.wo); }
  // copy rows [k0, k0 + slab_rows) into slab `st` (asynchronously)
  __device__ void issue(const Rows& w, int k0, int st) const {
    const int n16 = min(slab_rows(w), w.K - k0) * w.wo / TP;
    const T* src = w.p + (long long)k0 * w.wo;
    T* dst = WS + st * slab;
    for (int i = threadIdx.x; i < n16; i += NT) cp_async16(dst + i * TP, src + i * TP);
    cp_async_commit();
  }

  // D[u][n] = sum_k rows[k][u] in[k][n] for all channels; thread item = (point
  // n, RU consecutive units u0), a point's channels as one vector load and the
  // RU weights as broadcast vector loads from the slab, 2 RU C flops per k; FP32
  // units accumulate in packed pairs.  done(n, u0, acc) takes an item's sums.
  // rows' first slab is in flight in slab wst on entry (and its barrier also
  // orders the phases before this one); on exit next's first slab is.  The FP32
  // pipe needs four FMAs per word read from shared memory, which bounds the
  // item's shape: with RU = 8 and C = 6 a warp reads 14 words per 48 FMAs.
  // One layer of 64 -> 64 units at C = 6 in a loop of its own, as a share of the
  // FP32 peak: 49% with RU = 4 and weights read through L1, 61% with RU = 8,
  // 69% with RU = 8 and weights in shared memory (C = 4: 43, 51 and 69%).
  struct Acc {
    typename std::conditional<F32, f2, T>::type v[F32 ? RU / 2 : RU][C];
  };
  template <class Done>
  __device__ __forceinline__ void gemm(const Rows& w, const Rows& next, const T* in, Done done) {
    const int items = (w.wo / RU) * P, rps = slab_rows(w);
    for (int it0 = 0; it0 < items; it0 += NT) {
      const int it = it0 + threadIdx.x;
      const bool act = it < items, last_pass = it0 + NT >= items;
      const int n = act ? it % P : 0, u0 = act ? (it / P) * RU : 0;
      Acc acc;
#pragma unroll
      for (int r = 0; r < (F32 ? RU / 2 : RU); ++r)
#pragma unroll
        for (int c = 0; c < C; ++c) acc.v[r][c] = 0.f;
      const T* ap = in + n * C;
      for (int k0 = 0; k0 < w.K; k0 += rps) {
        cp_async_wait0();
        __syncthreads();
        if (k0 + rps < w.K) issue(w, k0 + rps, wst ^ 1);
        else if (!last_pass) issue(w, 0, wst ^ 1);
        else if (next.p) issue(next, 0, wst ^ 1);
        const T* wp = WS + wst * slab + u0;
        wst ^= 1;
        if (!act) continue;
        const int kn = min(rps, w.K - k0);
#pragma unroll(UK)
        for (int k = 0; k < kn; ++k, ap += pitch, wp += w.wo) {
          T wv[RU], av[C];
          if constexpr (RU % TP == 0) {
#pragma unroll
            for (int r = 0; r < RU; r += TP) vload<T>(wp + r, wv + r);
          } else {
#pragma unroll
            for (int r = 0; r < RU; ++r) wv[r] = wp[r];
          }
          load_chan<T, C>(ap, av);
          if constexpr (F32) {
#pragma unroll
            for (int c = 0; c < C; ++c)
#pragma unroll
              for (int r = 0; r < RU / 2; ++r)
                acc.v[r][c] = jfma(f2(wv[2 * r], wv[2 * r + 1]), f2(av[c]), acc.v[r][c]);
          } else {
#pragma unroll
            for (int r = 0; r < RU; ++r)
#pragma unroll
              for (int c = 0; c < C; ++c) acc.v[r][c] = fma(wv[r], av[c], acc.v[r][c]);
          }
        }
      }
      if (!act) continue;
      if constexpr (F32 && C % 2 == 0) {
        if (odd(n)) {
#pragma unroll
          for (int r = 0; r < RU / 2; ++r)
#pragma unroll
            for (int c = 0; c < C; c += 2) {
              const f2 t = acc.v[r][c];
              acc.v[r][c] = acc.v[r][c + 1];
              acc.v[r][c + 1] = t;
            }
        }
      }
      done(n, u0, acc);
    }
  }

  // ---------------------------------------------------------------- forward
  __device__ void layer1(T* out, T* zdst) {
    const int w = I.widths[1], d = I.d, CP = C * P;
    const T* W1 = W(1);
    const T* b1 = bias(1);
    for (int it = threadIdx.x; it < (w / EU) * P; it += NT) {
      const int n = it % P, u0 = (it / P) * EU;
      T x[3];
#pragma unroll
      for (int i = 0; i < 3; ++i) x[i] = i < d ? XS[n * d + i] : T(0);
#pragma unroll
      for (int r = 0; r < EU; ++r) {
        const int u = u0 + r;
        T wrow[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) wrow[i] = i < d ? W1[u * d + i] : T(0);
        T z[C], p[NP], a[C];
#pragma unroll
        for (int c = 0; c < C; ++c) z[c] = T(0);
        T v = b1[u];
#pragma unroll
        for (int i = 0; i < 3; ++i) v += wrow[i] * x[i];
        z[0] = v;
#pragma unroll
        for (int i = 0; i < Cls::D; ++i) {
          const int fo = Cls::first_order(i);
          if (fo >= 0) z[fo] = wrow[i];
        }
        tanh_derivs<T, NP>(z[0], p);
        Cls::compose(z, p, a);
        store_point(out + u * pitch, n, a);
        if (zdst) {
          __stcg(zdst + (long long)u * CP + n, p[0]);
#pragma unroll
          for (int c = 1; c < C; ++c) __stcg(zdst + (long long)u * CP + c * P + n, z[c]);
        }
      }
    }
  }

  // Z^l = W^l A^{l-1} (+ b on channel 0), then a^l = compose(z^l)
  __device__ void hidden_fwd(int l, const T* in, T* out, T* zdst, const Rows& next) {
    const int CP = C * P;
    const T* bl = bias(l);
    gemm(fwd_rows(l), next, in, [&](int n, int u0, const Acc& acc) {
      if constexpr (F32) {
#pragma unroll
        for (int r = 0; r < RU; r += 2) {
          const int u = u0 + r;
          f2 z[C], p[NP], a[C];
#pragma unroll
          for (int c = 0; c < C; ++c) z[c] = acc.v[r / 2][c];
          z[0] = z[0] + f2(bl[u], bl[u + 1]);
          tanh_polys_pair<NP>(f2(tanhf(z[0].v.x), tanhf(z[0].v.y)), p);
          Cls::compose(z, p, a);
          T lo[C], hi[C];
#pragma unroll
          for (int c = 0; c < C; ++c) {
            lo[c] = a[c].v.x;
            hi[c] = a[c].v.y;
          }
          store_point(out + u * pitch, n, lo);
          store_point(out + (u + 1) * pitch, n, hi);
          if (zdst) {
            z[0] = p[0];
#pragma unroll
            for (int c = 0; c < C; ++c) {
              __stcg(zdst + (long long)u * CP + c * P + n, z[c].v.x);
              __stcg(zdst + (long long)(u + 1) * CP + c * P + n, z[c].v.y);
            }
          }
        }
      } else {
#pragma unroll
        for (int r = 0; r < RU; ++r) {
          const int u = u0 + r;
          T z[C], p[NP], a[C];
#pragma unroll
          for (int c = 0; c < C; ++c) z[c] = acc.v[r][c];
          z[0] += bl[u];
          tanh_derivs<T, NP>(z[0], p);
          Cls::compose(z, p, a);
          store_point(out + u * pitch, n, a);
          if (zdst) {
            __stcg(zdst + (long long)u * CP + n, p[0]);
#pragma unroll
            for (int c = 1; c < C; ++c) __stcg(zdst + (long long)u * CP + c * P + n, z[c]);
          }
        }
      }
    });
  }

  // a^l = compose(z^l) from a stored z-jet [w][C*P] (tanh z in channel 0)
  __device__ void compose_from(int l, const T* zsrc, T* out) {
    const int w = I.widths[l], CP = C * P;
    for (int it = threadIdx.x; it < (w / EU) * P; it += NT) {
      const int n = it % P, u0 = (it / P) * EU;
      // all loads first, so that they are in flight together
      T zz[EU][C];
#pragma unroll
      for (int r = 0; r < EU; ++r)
#pragma unroll
        for (int c = 0; c < C; ++c) zz[r][c] = __ldcg(zsrc + (long long)(u0 + r) * CP + c * P + n);
      if constexpr (F32) {
#pragma unroll
        for (int r = 0; r < EU; r += 2) {
          f2 z[C], p[NP], a[C];
#pragma unroll
          for (int c = 0; c < C; ++c) z[c] = f2(zz[r][c], zz[r + 1][c]);
          tanh_polys_pair<NP>(z[0], p);
          Cls::compose(z, p, a);
          T lo[C], hi[C];
#pragma unroll
          for (int c = 0; c < C; ++c) {
            lo[c] = a[c].v.x;
            hi[c] = a[c].v.y;
          }
          store_point(out + (u0 + r) * pitch, n, lo);
          store_point(out + (u0 + r + 1) * pitch, n, hi);
        }
      } else {
#pragma unroll
        for (int r = 0; r < EU; ++r) {
          T p[NP], a[C];
          tanh_polys<T, NP>(zz[r][0], p);
          Cls::compose(zz[r], p, a);
          store_point(out + (u0 + r) * pitch, n, a);
        }
      }
    }
  }

  // u_{o,alpha} = W^L a^{L-1}_alpha (+ b^L on the value channel); lanes walk
  // the row's columns n * C + alpha
  __device__ void output_layer(const T* in) {
    const int L = I.L, wi = I.widths[L - 1], no = I.n_out;
    const T* WL = W(L);
    const T* bL = bias(L);
    const int ncol = C * P;
    for (int it = threadIdx.x; it < no * ncol; it += NT) {
      const int o = it / ncol, col = it - o * ncol;
      const int n = col / C, c = (col - n * C) ^ (odd(n) ? 1 : 0);
      const T* ap = in + col;
      T s = c == 0 ? bL[o] : T(0);
#pragma unroll 4
      for (int k = 0; k < wi; ++k) s = fma(WL[o * wi + k], ap[k * pitch], s);
      UO[o * ncol + c * P + n] = s;
    }
  }

  // Residual r_c = sum of the monomials - source, the loss partial and (bwd)
  // UB = dL/du.  When the monomial values fit the UB area and 2 r / N the
  // reduction area: three parallel passes, (point, monomial) products, per
  // point sums, per (point, output channel) adjoints, each keeping the
  // operands and order of a per-point loop over the monomials (which is the
  // fallback).
  __device__ double residual(long long n0, int nvalid, bool bwd) {
    const int ncol = C * P, nt = I.n_terms;
    double loss = 0.0;
    const T* src = reinterpret_cast<const T*>(I.source);
    T* rout = reinterpret_cast<T*>(I.r_out);
    if (I.n_groups > 0) {  // composite loss: every term over its own points
      if (bwd)
        for (int i = threadIdx.x; i < I.n_out * ncol; i += NT) UB[i] = T(0);
      __syncthreads();
      return grouped_residual<T>(I.terms, I.groups, I.n_groups, I.n_res, UO, UB, P, n0, nvalid, src, rout, bwd,
                                 threadIdx.x, NT);
    }
    const T two_over_n = T(2.0 * I.inv_N);
    const bool parallel = nt <= I.n_out * C && I.n_res * P * (int)sizeof(T) <= kSimtRed * (int)sizeof(double);
    if (!parallel) {
      if (bwd)
        for (int i = threadIdx.x; i < I.n_out * ncol; i += NT) UB[i] = T(0);
      __syncthreads();
      for (int n = threadIdx.x; n < nvalid; n += NT) {
        T r[kMaxRes];
#pragma unroll
        for (int c = 0; c < kMaxRes; ++c) r[c] = c < I.n_res && src ? -src[(n0 + n) * I.n_res + c] : T(0);
        for (int m = 0; m < nt; ++m) {
          const DevTerm& tm = I.terms[m];
          T prod = T(tm.coef);
          for (int f = 0; f < tm.nfac; ++f) prod *= UO[tm.fac[f] * P + n];
#pragma unroll
          for (int c = 0; c < kMaxRes; ++c)
            if (c == tm.comp) r[c] += prod;
        }
#pragma unroll
        for (int c = 0; c < kMaxRes; ++c) {
          if (c >= I.n_res) break;
          if (rout) rout[(n0 + n) * I.n_res + c] = r[c];
          loss += (double)r[c] * (double)r[c];
        }
        if (bwd)
          for (int m = 0; m < nt; ++m) {
            const DevTerm& tm = I.terms[m];
            T rc = T(0);
#pragma unroll
            for (int c = 0; c < kMaxRes; ++c)
              if (c == tm.comp) rc = r[c];
            const T g = two_over_n * rc * T(tm.coef);
            for (int f = 0; f < tm.nfac; ++f) {
              T prod = g;
              for (int h = 0; h < tm.nfac; ++h)
                if (h != f) prod *= UO[tm.fac[h] * P + n];
              UB[tm.fac[f] * P + n] += prod;
            }
          }
      }
      return loss;
    }
    T* prodm = UB;                         // [n_terms][P]
    T* rg = reinterpret_cast<T*>(RED);     // [n_res][P]: 2 r / N
    for (int i = threadIdx.x; i < nt * nvalid; i += NT) {
      const int m = i / nvalid, n = i - m * nvalid;
      const DevTerm& tm = I.terms[m];
      T prod = T(tm.coef);
      for (int f = 0; f < tm.nfac; ++f) prod *= UO[tm.fac[f] * P + n];
      prodm[m * P + n] = prod;
    }
    __syncthreads();
    for (int n = threadIdx.x; n < nvalid; n += NT) {
      T r[kMaxRes];
#pragma unroll
      for (int c = 0; c < kMaxRes; ++c) r[c] = c < I.n_res && src ? -src[(n0 + n) * I.n_res + c] : T(0);
      for (int m = 0; m < nt; ++m) {
        const int cm = I.terms[m].comp;
        const T v = prodm[m * P + n];
#pragma unroll
        for (int c = 0; c < kMaxRes; ++c)
          if (c == cm) r[c] += v;
      }
#pragma unroll
      for (int c = 0; c < kMaxRes; ++c) {
        if (c >= I.n_res) break;
        if (rout) rout[(n0 + n) * I.n_res + c] = r[c];
        loss += (double)r[c] * (double)r[c];
        rg[c * P + n] = two_over_n * r[c];
      }
    }
    __syncthreads();  // the products in UB are consumed
    if (!bwd) return loss;
    for (int i = threadIdx.x; i < I.n_out * ncol; i += NT) {
      const int k = i / P, n = i - k * P;
      T acc = T(0);
      if (n < nvalid)
        for (int m = 0; m < nt; ++m) {
          const DevTerm& tm = I.terms[m];
          for (int f = 0; f < tm.nfac; ++f) {
            if (tm.fac[f] != k) continue;
            T prod = rg[tm.comp * P + n] * T(tm.coef);
            for (int h = 0; h < tm.nfac; ++h)
              if (h != f) prod *= UO[tm.fac[h] * P + n];
            acc += prod;
          }
        }
      UB[i] = acc;
    }
    return loss;
  }

  // ---------------------------------------------------------------- backward
  // Abar^{L-1} = W^L^T ub; dW^L = sum_cols ub a^{L-1}^T; db^L = sum_n ub_0
  __device__ void output_bwd(const T* a_last, T* abar, double* g) {
    const int L = I.L, wi = I.widths[L - 1], no = I.n_out;
    const T* WL = W(L);
    const int ncol = C * P;
    // Abar[k][n*C + c], one (unit, point) per item with all channels
    for (int it = threadIdx.x; it < wi * P; it += NT) {
      const int n = it % P, k = it / P;
      T s[C];
#pragma unroll
      for (int c = 0; c < C; ++c) s[c] = T(0);
      for (int o = 0; o < no; ++o) {
        const T w = WL[o * wi + k];
#pragma unroll
        for (int c = 0; c < C; ++c) s[c] = fma(w, UB[o * ncol + c * P + n], s[c]);
      }
      store_point(abar + k * pitch, n, s);
    }
    // dW^L[o][k], the groups of points one after another: four lanes share a sum,
    // each taking a quarter of a group's points; the partials combine by shuffles
    // in a fixed order (the loop runs whole warps: every lane reaches the shuffles)
    const int items = 4 * no * wi, items_w = (items + 31) & ~31;
    for (int it = threadIdx.x; it < items_w; it += NT) {
      const bool act = it < items;
      const int part = it & 3, ok = act ? it >> 2 : 0, o = ok / wi, k = ok - o * wi;
      for (int n0 = 0; n0 < P; n0 += P0) {
        T s = T(0);
        if (act)
          for (int n = n0 + part; n < n0 + P0; n += 4) {
            T av[C];
            load_point(a_last + k * pitch, n, av);
#pragma unroll
            for (int c = 0; c < C; ++c) s = fma(UB[o * ncol + c * P + n], av[c], s);
          }
        s += __shfl_xor_sync(0xffffffffu, s, 1);
        s += __shfl_xor_sync(0xffffffffu, s, 2);
        if (act && part == 0) atomicAdd(g + I.goff_WL + o * wi + k, widen(s));
      }
    }
    for (int o = NT - 1 - threadIdx.x; o < no; o += NT)  // db^L, by the last threads
      for (int n0 = 0; n0 < P; n0 += P0) {
        T s = T(0);
#pragma unroll 8
        for (int n = n0; n < n0 + P0; ++n) s += UB[o * ncol + n];
        atomicAdd(g + I.goff_b[L - 1] + o, widen(s));
      }
  }

  // Zbar^l = (d compose / dz)^T Abar^l per (unit, point), in place in `bar`;
  // z^l (tanh z in channel 0) from zsrc
  __device__ void act_adjoint(int l, const T* zsrc, T* bar) {
    const int w = I.widths[l], CP = C * P;
    for (int it = threadIdx.x; it < (w / EU) * P; it += NT) {
      const int n = it % P, u0 = (it / P) * EU;
      // all global loads first, so that they overlap
      T zz[EU][C];
#pragma unroll
      for (int r = 0; r < EU; ++r)
#pragma unroll
        for (int c = 0; c < C; ++c) zz[r][c] = __ldcg(zsrc + (long long)(u0 + r) * CP + c * P + n);
      if constexpr (F32) {
        // FP32: units (r, r+1) in packed pairs
#pragma unroll
        for (int r = 0; r < EU; r += 2) {
          T* b0 = bar + (u0 + r) * pitch;
          T* b1 = b0 + pitch;
          f2 z[C], p[NP], ab[C], zb[C];
          T lo[C], hi[C];
          load_point(b0, n, lo);
          load_point(b1, n, hi);
#pragma unroll
          for (int c = 0; c < C; ++c) {
            z[c] = f2(zz[r][c], zz[r + 1][c]);
            ab[c] = f2(lo[c], hi[c]);
          }
          tanh_polys_pair<NP>(z[0], p);
          Cls::adjoint(z, p, ab, zb);
#pragma unroll
          for (int c = 0; c < C; ++c) {
            lo[c] = zb[c].v.x;
            hi[c] = zb[c].v.y;
          }
          store_point(b0, n, lo);
          store_point(b1, n, hi);
        }
      } else {
#pragma unroll
        for (int r = 0; r < EU; ++r) {
          T* b0 = bar + (u0 + r) * pitch + n * C;
          T p[NP], ab[C], zb[C];
          load_chan<T, C>(b0, ab);
          tanh_polys<T, NP>(zz[r][0], p);
          Cls::adjoint(zz[r], p, ab, zb);
          store_chan<T, C>(b0, zb);
        }
      }
    }
  }

  // dW^l[u][k] += sum_cols Zbar[u][col] A[k][col]; db^l[u] += sum_n Zbar[u][n].
  // Thread item: WR rows u and 4 columns k (rows kb + s * nkb of A).
  __device__ void wgrad(int l, const T* zbar, const T* aprev, double* g) {
    if constexpr (!F32) {
      wgrad64(l, zbar, aprev, g);
    } else {
      // several groups added to the chunk's FP32 sums by one thread: the sums
      // wait in registers, one load and one store per tile instead of a vector
      // reduction per group (3->256x8->1, three groups a tile: 10.74 -> 10.14 ms)
      const int items = I.widths[l] / 4 * (I.widths[l - 1] / 4);
      if (I.wr == 4 && wacc_base && V > 1 && (V % 2 || items * 2 > NT)) wgrad32<4, true>(l, zbar, aprev, g);
      else if (I.wr == 4) wgrad32<4, false>(l, zbar, aprev, g);
      else wgrad32<(RU == 8 ? 2 : 1), false>(l, zbar, aprev, g);
    }
    // a thread per bias, its groups one after another
    const int wo = I.widths[l];
    double* gb = g + I.goff_b[l - 1];
    for (int u = threadIdx.x; u < wo; u += NT) {
      const T* zp = zbar + u * pitch;
      for (int n0 = 0; n0 < P; n0 += P0) {
        T s = T(0);
#pragma unroll 8
        for (int n = n0; n < n0 + P0; ++n) s += zp[n * C + (odd(n) ? 1 : 0)];
        atomicAdd(gb + u, widen(s));
      }
    }
  }

  // FP32: the groups of points one after another, their even and odd columns in
  // the two halves of a packed pair (the 16-byte loads deliver the pairs), summed
  // at the end of the group.  Where the items leave half the CTA idle, the two
  // halves of a warp take an item's even and odd groups and then swap half
  // their blocks, so that every element is added by one thread, group after group.
  template <int WR, bool HELD>
  __device__ __forceinline__ void wgrad32(int l, const T* zbar, const T* aprev, double* g) {
    const int wo = I.widths[l], wi = I.widths[l - 1];
    const int nkb = wi / 4, items = (wo / WR) * nkb, gcol = P0 * C;
    const bool two = !HELD && WR >= 2 && V % 2 == 0 && items * 2 <= NT;
    double* gW = g + I.off_W[l - 1];
    const int lane = threadIdx.x & 31, sl = two ? lane >> 4 : 0;
    const int work_w = ((two ? 2 * items : items) + 31) & ~31;  // whole warps: every lane reaches the shuffles
    for (int it = threadIdx.x; it < work_w; it += NT) {
      const int item = two ? (it >> 5) * 16 + (lane & 15) : it;
      const bool act = item < items;
      const int kb = act ? item % nkb : 0, ub = act ? item / nkb : 0;
      const T* zp = zbar + ub * WR * pitch;
      const T* app = aprev + kb * pitch;
      float* const sums = HELD && act ? wacc(l) + (long long)item * (WR * 4) : nullptr;
      T run[WR * 4];
      if constexpr (HELD) {
#pragma unroll
        for (int e = 0; e < WR * 4; e += 4) {
          float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
          if (act && !wacc_first) t = __ldcg(reinterpret_cast<const float4*>(sums + e));
          run[e] = t.x;
          run[e + 1] = t.y;
          run[e + 2] = t.z;
          run[e + 3] = t.w;
        }
      }
      for (int v0 = 0; v0 < V; v0 += two ? 2 : 1) {
        const int c0 = (v0 + sl) * gcol, c1 = act ? c0 + gcol : c0;
        f2 ap2[WR][4];
#pragma unroll
        for (int r = 0; r < WR; ++r)
#pragma unroll
          for (int s = 0; s < 4; ++s) ap2[r][s] = f2(0.f);
        for (int col = c0; col < c1; col += TP) {
          T av[4][TP];
#pragma unroll
          for (int s = 0; s < 4; ++s) vload<T>(app + s * nkb * pitch + col, av[s]);
          T zv[WR][TP];
#pragma unroll
          for (int r = 0; r < WR; ++r) vload<T>(zp + r * pitch + col, zv[r]);
#pragma unroll
          for (int r = 0; r < WR; ++r)
#pragma unroll
            for (int s = 0; s < 4; ++s)
#pragma unroll
              for (int j = 0; j < TP; j += 2)
                ap2[r][s] = jfma(f2(zv[r][j], zv[r][j + 1]), f2(av[s][j], av[s][j + 1]), ap2[r][s]);
        }
        T acc[WR * 4];
#pragma unroll
        for (int r = 0; r < WR; ++r)
#pragma unroll
          for (int s = 0; s < 4; ++s) acc[r * 4 + s] = ap2[r][s].v.x + ap2[r][s].v.y;
        const bool first = wacc_first && v0 == 0;
        if (!HELD && two) {
          constexpr int H = WR * 2;  // this thread's half of the block
#pragma unroll
          for (int e = 0; e < H; e += 4) {
            T lo[4], hi[4];  // four elements: group v0, group v0 + 1
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const int k = (e + j) % (WR * 2);
              const T got = __shfl_xor_sync(0xffffffffu, sl ? acc[k] : acc[k + H], 16);
              lo[j] = sl ? got : acc[k];
              hi[j] = sl ? acc[k + H] : got;
            }
            if (act) {
              add4<WR>(l, item, sl * H + e, lo, first, gW, ub, kb, nkb, wi);
              add4<WR>(l, item, sl * H + e, hi, false, gW, ub, kb, nkb, wi);
            }
          }
        } else if (HELD) {
#pragma unroll
          for (int e = 0; e < WR * 4; ++e) run[e] += acc[e];
        } else if (act) {
#pragma unroll
          for (int e = 0; e < WR * 4; e += 4) add4<WR>(l, item, e, acc + e, first, gW, ub, kb, nkb, wi);
        }
      }
      if (HELD && act)
#pragma unroll
        for (int e = 0; e < WR * 4; e += 4)
          __stcg(reinterpret_cast<float4*>(sums + e), make_float4(run[e], run[e + 1], run[e + 2], run[e + 3]));
    }
  }

  // one row of an item's block (from element e on) to the chunk's FP32 sums or
  // the FP64 slice: fire-and-forget adds, one thread per element and in order,
  // so the sums stay deterministic
  template <int WR>
  __device__ __forceinline__ void add4(int l, int item, int e, const T* v, bool first, double* gW, int ub, int kb,
                                       int nkb, int wi) {
    if (wacc_base) {
      float* a = wacc(l) + (long long)item * (WR * 4) + e;
      if (first) __stcg(reinterpret_cast<float4*>(a), make_float4(v[0], v[1], v[2], v[3]));
      else red_add_v4(a, v[0], v[1], v[2], v[3]);
      return;
    }
    double* d = gW + (ub * WR + (e >> 2)) * wi + kb;
#pragma unroll
    for (int s = 0; s < 4; ++s) atomicAdd(d + s * nkb, widen(v[s]));
  }

  // FP64: NS adjacent lanes share an item, each taking every NS-th vector of
  // columns, so that narrow layers fill the CTA (a 20 x 20 layer has 25 items);
  // their sums combine by halves, each lane ending with its own 1 / NS of the block.
  __device__ __forceinline__ void wgrad64(int l, const T* zbar, const T* aprev, double* g) {
    constexpr int WR = 4;
    const int wo = I.widths[l], wi = I.widths[l - 1];
    const int ncol = (C * P + TP - 1) / TP * TP;  // zero columns up to a whole vector
    const int nkb = wi / 4, items = (wo / WR) * nkb;
    const int NS = simt_wgrad_slices(items, NT);
    double* gW = g + I.off_W[l - 1];
    const int work = items * NS, work_w = (work + 31) & ~31;
    for (int it = threadIdx.x; it < work_w; it += NT) {
      const bool act = it < work;
      const int sl = it & (NS - 1), item = act ? it / NS : 0;
      const int kb = item % nkb, ub = item / nkb;
      T acc[WR * 4];
      const T* zp = zbar + ub * WR * pitch;
      const T* app = aprev + kb * pitch;
#pragma unroll
      for (int e = 0; e < WR * 4; ++e) acc[e] = T(0);
      for (int col = act ? sl * TP : ncol; col < ncol; col += NS * TP) {
        T zv[WR][TP], av[4][TP];
#pragma unroll
        for (int r = 0; r < WR; ++r) vload<T>(zp + r * pitch + col, zv[r]);
#pragma unroll
        for (int s = 0; s < 4; ++s) vload<T>(app + s * nkb * pitch + col, av[s]);
#pragma unroll
        for (int r = 0; r < WR; ++r)
#pragma unroll
          for (int s = 0; s < 4; ++s)
#pragma unroll
            for (int j = 0; j < TP; ++j) acc[r * 4 + s] = fma(zv[r][j], av[s][j], acc[r * 4 + s]);
      }
      // combine the NS lanes: at each step a lane keeps one half of its block
      // and sends the other to its partner
      int base = 0, n = WR * 4;
#pragma unroll
      for (int m = 1; m < 8; m <<= 1) {
        const int h = WR * 4 / 2 / m;
        if (m >= NS) break;
        const bool up = (it & m) != 0;
#pragma unroll
        for (int e = 0; e < h; ++e) {
          const T send = up ? acc[e] : acc[e + h], keep = up ? acc[e + h] : acc[e];
          acc[e] = keep + __shfl_xor_sync(0xffffffffu, send, m);
        }
        base += up ? h : 0;
        n = h;
      }
      if (!act) continue;
#pragma unroll
      for (int e = 0; e < WR * 4; ++e)
        if (e < n) {
          const int r = (base + e) >> 2, s = (base + e) & 3;
          atomicAdd(gW + (ub * WR + r) * wi + kb + s * nkb, (double)acc[e]);
        }
    }
  }

  // Abar^{l-1}[k][col] = sum_u W^l[u][k] Zbar^l[u][col]
  __device__ void dgrad(int l, const T* zbar, T* abar, const Rows& next) {
    gemm(bwd_rows(l), next, zbar, [&](int n, int k0, const Acc& acc) {
      if constexpr (F32) {
#pragma unroll
        for (int r = 0; r < RU; r += 2) {
          T lo[C], hi[C];
#pragma unroll
          for (int c = 0; c < C; ++c) {
            lo[c] = acc.v[r / 2][c].v.x;
            hi[c] = acc.v[r / 2][c].v.y;
          }
          store_point(abar + (k0 + r) * pitch, n, lo);
          store_point(abar + (k0 + r + 1) * pitch, n, hi);
        }
      } else {
#pragma unroll
        for (int r = 0; r < RU; ++r) store_chan<T, C>(abar + (k0 + r) * pitch + n * C, acc.v[r]);
      }
    });
  }

  // dW^1[u][i] += sum_n Zbar_0[u][n] x_i[n] + Zbar_{e_i}[u][n]; db^1[u] += sum_n Zbar_0[u][n];
  // a thread per unit, its groups of points one after another
  __device__ void layer1_bwd(const T* zbar, double* g) {
    const int w = I.widths[1], d = I.d;
    double* gW = g;
    double* gb = g + I.goff_b[0];
    for (int u = threadIdx.x; u < w; u += NT) {
      const T* zp = zbar + u * pitch;
      for (int n0 = 0; n0 < P; n0 += P0) {
        T sb = T(0), sw[3] = {T(0), T(0), T(0)};
#pragma unroll 4
        for (int n = n0; n < n0 + P0; ++n) {
          const T z0 = zp[n * C + (odd(n) ? 1 : 0)];
          sb += z0;
#pragma unroll
          for (int i = 0; i < 3; ++i)
            if (i < d) sw[i] = fma(z0, XS[n * d + i], sw[i]);
        }
#pragma unroll
        for (int i = 0; i < Cls::D; ++i) {
          const int fo = Cls::first_order(i);
          if (fo >= 0 && i < d) {
#pragma unroll 4
            for (int n = n0; n < n0 + P0; ++n) sw[i] += zp[n * C + (odd(n) ? fo ^ 1 : fo)];
          }
        }
#pragma unroll
        for (int i = 0; i < 3; ++i)
          if (i < d) atomicAdd(gW + u * d + i, widen(sw[i]));
        atomicAdd(gb + u, widen(sb));
      }
    }
  }

  // ---------------------------------------------------------------- driver
  // the first jet GEMM of a tile (p null: the network has none)
  __device__ Rows first_rows() const {
    if (I.L < 3) return {nullptr, 0, 0};
    return A.mode == MODE_BWD_STORE ? bwd_rows(I.L - 1) : fwd_rows(2);
  }

  // the tile of the points [n0, min(n0 + P, n1)); its first GEMM's first weight
  // slab is in flight on entry, and the next tile's on exit (more: there is one)
  __device__ double tile(long long n0, long long n1, double* g, bool more) {
    const int mode = A.mode;
    const long long rem = n1 - n0, t = n0 / P;  // t: the tile's place in the z-jet store
    const int nvalid = rem < (long long)P ? (int)rem : P;
    const int d = I.d;
    const T* X = reinterpret_cast<const T*>(I.X);
    for (int i = threadIdx.x; i < P * d; i += NT) {
      const int n = i / d;
      XS[i] = n < nvalid ? X[(n0 + n) * d + (i % d)] : T(0);
    }
    __syncthreads();
    const bool use_store = (mode == MODE_BWD_STORE) || (mode == MODE_FWD && I.store != nullptr);
    const bool write_z = (mode == MODE_FWD_BWD) || (mode == MODE_FWD && I.store != nullptr);
    const bool bwd = mode != MODE_FWD;
    const int L = I.L;
    const Rows none{nullptr, 0, 0}, first = more ? first_rows() : none;
    T *y = B0, *x = B1;  // y: the newest layer's jets
    if (mode != MODE_BWD_STORE) {
      layer1(y, write_z ? zjet(t, 1, use_store) : nullptr);
      for (int l = 2; l <= L - 1; ++l) {
        const Rows next = l < L - 1 ? fwd_rows(l + 1) : bwd ? bwd_rows(l) : first;
        hidden_fwd(l, y, x, write_z ? zjet(t, l, use_store) : nullptr, next);
        T* tmp = x;
        x = y;
        y = tmp;
      }
    } else {
      compose_from(L - 1, zjet(t, L - 1, true), y);
    }
    __syncthreads();
    output_layer(y);
    __syncthreads();
    double loss = residual(n0, nvalid, bwd);
    __syncthreads();
    if (!bwd) return loss;
    // x: Abar^l, then Zbar^l in place; y: A^{l-1}, then Abar^{l-1}
    output_bwd(y, x, g);
    __syncthreads();
    const bool from_store = mode == MODE_BWD_STORE;
    for (int l = L - 1; l >= 1; --l) {
      act_adjoint(l, zjet(t, l, from_store), x);
      if (l >= 2) compose_from(l - 1, zjet(t, l - 1, from_store), y);
      __syncthreads();
      if (l >= 2) {
        wgrad(l, x, y, g);
        dgrad(l, x, y, l > 2 ? bwd_rows(l - 1) : first);  // its first barrier ends the weight gradient's reads of y
        T* tmp = x;
        x = y;
        y = tmp;
      } else {
        layer1_bwd(x, g);
      }
      __syncthreads();
    }
    return loss;
  }
};

template <class Cls, class T, int RU>
__device__ __forceinline__ void simt_body(const SimtArgs& args) {
  extern __shared__ __align__(16) unsigned char smem[];
  dependency_wait();
  __shared__ int k_s;
  // the running item's descriptor: read in every phase, through shared memory
  // rather than a pointer that may be param or global space, which cost
  // registers that spilled (2->64x5->1, C = 6: 1.44 ms with it, 1.33 ms without;
  // 3->256x8->1 11.5 and 10.1 ms)
  __shared__ DevInstance inst_s;
  const int NT = blockDim.x;
  for (int k = blockIdx.x; k < args.n_items;) {
    // batched launches walk a cost-ordered list: position k -> item id, and
    // item id -> instance (second half of item_inst)
    const int item = args.item_inst ? args.item_inst[k] : k;
    const DevInstance* src = args.insts ? args.insts + args.item_inst[args.n_items + item] : &args.inst0;
    for (int i = threadIdx.x; i < (int)(sizeof(DevInstance) / 16); i += NT)
      reinterpret_cast<uint4*>(&inst_s)[i] = reinterpret_cast<const uint4*>(src)[i];
    __syncthreads();
    const DevInstance& I = inst_s;
    const int chunk = item - I.chunk_base;
    SimtTile<Cls, T, RU> S(I, args, smem, chunk);
    // columns past C * P are never written: zero them (and everything else)
    // once per item so that the weight-gradient sums over whole vectors see
    // zeros there
    for (int i = threadIdx.x; i < 2 * S.wmax * S.pitch; i += NT) S.B0[i] = T(0);
    const auto first = S.first_rows();
    if (first.p) S.issue(first, 0, 0);
    const bool bwd = args.mode != MODE_FWD;
    double* g = bwd ? I.grad_slices + (long long)chunk * I.n_slice : nullptr;
    if (bwd)
      for (int i = threadIdx.x; i < I.n_slice; i += NT) g[i] = 0.0;
    double loss = 0.0;
    // points of the chunk: the first chunk_rem chunks take one unit more than the rest
    const long long u0 = (long long)chunk * I.tiles_per_chunk + min(chunk, I.chunk_rem);
    const long long u1 = u0 + I.tiles_per_chunk + (chunk < I.chunk_rem ? 1 : 0);
    const long long s0 = u0 * I.unit, s1 = min(u1 * I.unit, I.N);
    // FP32 sums in runs of at most kWaccTiles groups (wide channel sets): the FP32
    // rounding of a weight's sum stays below kWaccTiles * 2^-24 of its magnitudes
    // at any N.  The reduction reads the sums of a single run.
    const bool runs = bwd && S.wacc_base != nullptr && !I.wsums_direct;
    if (runs) simt_wacc_zero(S.wacc_base, I);
    __syncthreads();
    int groups = 0;  // of the running FP32 run
    for (long long n = s0; n < s1; n += S.P) {
      const bool more = n + S.P < s1;
      S.wacc_first = n == s0 && I.wsums_direct;
      loss += S.tile(n, s1, g, more);
      __syncthreads();
      groups += S.V;
      if (runs && (!more || groups + S.V > kWaccTiles)) {
        __threadfence();
        __syncthreads();
        simt_wacc_flush(S.wacc_base, I, g);
        groups = 0;
        if (more) {
          __syncthreads();
          simt_wacc_zero(S.wacc_base, I);
          __syncthreads();
        }
      }
    }
    // block reduction of the loss partial (fixed order)
    for (int o = 16; o > 0; o >>= 1) loss += __shfl_down_sync(0xffffffffu, loss, o);
    if ((threadIdx.x & 31) == 0) S.RED[threadIdx.x >> 5] = loss;
    __syncthreads();
    if (threadIdx.x == 0) {
      double s = 0.0;
      for (int w = 0; w < NT / 32; ++w) s += S.RED[w];
      I.loss_slices[chunk] = s;
    }
    // the next item: from the shared counter, or a fixed stride
    if (args.item_next) {
      if (threadIdx.x == 0) k_s = (int)gridDim.x + atomicAdd(args.item_next, 1);
      __syncthreads();
      k = k_s;
    } else {
      k += gridDim.x;
    }
    __syncthreads();
  }
}

// Launch bounds: up to 512 threads (one CTA per SM, or two of 256) and so at
// most 128 registers, except where the tiles need one CTA of 256 threads with
// all registers (FP32 channel sets of 10 or more).  FP64 runs two CTAs of 256
// where their tiles fit: one CTA's elementwise phases overlap the other's GEMMs
// (with one of 160 registers 3->64x3->2 took 27.4 ms at 40000 points and
// 3->256x2->1 10.7 ms at 4096, with two 24.3 and 10.1 ms).
template <class Cls, class T>
constexpr int simt_max_threads() {
  return sizeof(T) == 8 || Cls::C >= 10 ? 256 : 512;
}
template <class Cls, class T>
constexpr int simt_min_ctas() {
  return sizeof(T) == 8 ? 2 : 1;
}
template <class Cls, class T, int RU>
__global__ void __launch_bounds__(simt_max_threads<Cls, T>(), simt_min_ctas<Cls, T>())
    simt_kernel(const __grid_constant__ SimtArgs args) {
  simt_body<Cls, T, RU>(args);
}

// the kernel for ru units per thread of the jet GEMMs: FP32 8 (every hidden
// width a multiple of 8) or 4, FP64 1
template <class Cls, class T>
constexpr auto simt_entry(int ru) {
  if constexpr (sizeof(T) == 8) return &simt_kernel<Cls, T, 1>;
  else return ru == 8 ? &simt_kernel<Cls, T, 8> : &simt_kernel<Cls, T, 4>;
}

// Elementwise activation rule on [n][C] FP64 jets (verification hook, Eq. 15).
template <class Cls>
__global__ void debug_activation_kernel(int kind, long long n, const double* z, const double* v, double* out) {
  constexpr int C = Cls::C;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    double zz[C], vv[C], oo[C], p[Cls::NP];
    for (int c = 0; c < C; ++c) {
      zz[c] = z[i * C + c];
      vv[c] = v ? v[i * C + c] : 0.0;
    }
    tanh_derivs<double, Cls::NP>(zz[0], p);
    if (kind == 0) Cls::compose(zz, p, oo);
    else if (kind == 1) Cls::tangent(zz, p, vv, oo);
    else Cls::adjoint(zz, p, vv, oo);
    for (int c = 0; c < C; ++c) out[i * C + c] = oo[c];
  }
}

}  // namespace jet
