// Generated by gen_closures.py -- do not edit.
// Per-closure jet algebra: Faa di Bruno activation composition (Eq. 2-3 and
// their higher-order recursion, Sec. 2.2), its tangent and its adjoint.
#pragma once

namespace jet {

// fused multiply-add of the jet algebra; a packed type adds its own overload
__device__ __forceinline__ float jfma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double jfma(double a, double b, double c) { return fma(a, b, c); }

// d1o4: d=1, channels 0 1 2 3 4
struct Cls_d1o4 {
  static constexpr int D = 1;
  static constexpr int C = 5;
  static constexpr int MAXORD = 4;
  static constexpr int NP = 6;  // p[0..MAXORD+1]
  // channel index of the first-order channel e_i (-1 if absent)
  static __host__ __device__ constexpr int first_order(int i) { return i == 0 ? 1 : -1; }
  // first channel index of the highest derivative order
  static constexpr int TOP_BEGIN = 4;
  template <class T> static __device__ __forceinline__ void compose(const T* z, const T* p, T* a) {
    a[0] = p[0];
    a[1] = p[1]*z[1];
    a[2] = jfma(z[2], p[1], p[2]*z[1]*z[1]);
    a[3] = jfma(z[3], p[1], jfma(z[2], T(3)*p[2]*z[1], p[3]*z[1]*z[1]*z[1]));
    a[4] = jfma(z[4], p[1], jfma(z[2], T(3)*p[2]*z[2], jfma(z[3], T(4)*p[2]*z[1], jfma(z[2], T(6)*p[3]*z[1]*z[1], p[4]*z[1]*z[1]*z[1]*z[1]))));
  }
  template <class T> static __device__ __forceinline__ void tangent(const T* z, const T* p, const T* v, T* da) {
    da[0] = p[1]*v[0];
    da[1] = jfma(v[1], p[1], p[2]*z[1]*v[0]);
    da[2] = jfma(v[2], p[1], jfma(v[1], T(2)*p[2]*z[1], jfma(z[2], p[2], p[3]*z[1]*z[1])*v[0]));
    da[3] = jfma(v[3], p[1], jfma(v[2], T(3)*p[2]*z[1], jfma(v[1], jfma(z[2], T(3)*p[2], T(3)*p[3]*z[1]*z[1]), jfma(z[3], p[2], jfma(z[2], T(3)*p[3]*z[1], p[4]*z[1]*z[1]*z[1]))*v[0])));
    da[4] = jfma(v[4], p[1], jfma(v[3], T(4)*p[2]*z[1], jfma(v[2], jfma(z[2], T(6)*p[2], T(6)*p[3]*z[1]*z[1]), jfma(v[1], jfma(z[3], T(4)*p[2], jfma(z[2], T(12)*p[3]*z[1], T(4)*p[4]*z[1]*z[1]*z[1])), jfma(z[4], p[2], jfma(z[2], T(3)*p[3]*z[2], jfma(z[3], T(4)*p[3]*z[1], jfma(z[2], T(6)*p[4]*z[1]*z[1], p[5]*z[1]*z[1]*z[1]*z[1]))))*v[0]))));
  }
  template <class T> static __device__ __forceinline__ void adjoint(const T* z, const T* p, const T* ab, T* zb) {
    zb[0] = jfma(ab[4], jfma(z[4], p[2], jfma(z[2], T(3)*p[3]*z[2], jfma(z[3], T(4)*p[3]*z[1], jfma(z[2], T(6)*p[4]*z[1]*z[1], p[5]*z[1]*z[1]*z[1]*z[1])))), jfma(ab[3], jfma(z[3], p[2], jfma(z[2], T(3)*p[3]*z[1], p[4]*z[1]*z[1]*z[1])), jfma(ab[2], jfma(z[2], p[2], p[3]*z[1]*z[1]), jfma(ab[1], p[2]*z[1], p[1]*ab[0]))));
    zb[1] = jfma(ab[4], jfma(z[3], T(4)*p[2], jfma(z[2], T(12)*p[3]*z[1], T(4)*p[4]*z[1]*z[1]*z[1])), jfma(ab[3], jfma(z[2], T(3)*p[2], T(3)*p[3]*z[1]*z[1]), jfma(ab[2], T(2)*p[2]*z[1], p[1]*ab[1])));
    zb[2] = jfma(ab[4], jfma(z[2], T(6)*p[2], T(6)*p[3]*z[1]*z[1]), jfma(ab[3], T(3)*p[2]*z[1], p[1]*ab[2]));
    zb[3] = jfma(ab[4], T(4)*p[2]*z[1], p[1]*ab[3]);
    zb[4] = p[1]*ab[4];
  }
  template <class T> static __device__ __forceinline__ void adjoint_conv(const T* z, const T* p, const T* ab, T* zb) {
    T c[5];
    c[0] = p[1];
    c[1] = p[2]*z[1];
    c[2] = jfma(z[2], p[2], p[3]*z[1]*z[1]);
    c[3] = jfma(z[3], p[2], jfma(z[2], T(3)*p[3]*z[1], p[4]*z[1]*z[1]*z[1]));
    c[4] = jfma(z[4], p[2], jfma(z[2], T(3)*p[3]*z[2], jfma(z[3], T(4)*p[3]*z[1], jfma(z[2], T(6)*p[4]*z[1]*z[1], p[5]*z[1]*z[1]*z[1]*z[1]))));
    zb[0] = jfma(ab[4], c[4], jfma(ab[3], c[3], jfma(ab[2], c[2], jfma(ab[1], c[1], c[0]*ab[0]))));
    zb[1] = jfma(ab[4], T(4)*c[3], jfma(ab[3], T(3)*c[2], jfma(ab[2], T(2)*c[1], c[0]*ab[1])));
    zb[2] = jfma(ab[4], T(6)*c[2], jfma(ab[3], T(3)*c[1], c[0]*ab[2]));
    zb[3] = jfma(ab[4], T(4)*c[1], c[0]*ab[3]);
    zb[4] = c[0]*ab[4];
  }
};

// d2o2: d=2, channels 00 10 01 20 11 02
struct Cls_d2o2 {
  static constexpr int D = 2;
  static constexpr int C = 6;
  static constexpr int MAXORD = 2;
  static constexpr int NP = 4;  // p[0..MAXORD+1]
  // channel index of the first-order channel e_i (-1 if absent)
  static __host__ __device__ constexpr int first_order(int i) { return i == 0 ? 1 : i == 1 ? 2 : -1; }
  // first channel index of the highest derivative order
  static constexpr int TOP_BEGIN = 3;
  template <class T> static __device__ __forceinline__ void compose(const T* z, const T* p, T* a) {
    a[0] = p[0];
    a[1] = p[1]*z[1];
    a[2] = p[1]*z[2];
    a[3] = jfma(z[3], p[1], p[2]*z[1]*z[1]);
    a[4] = jfma(z[4], p[1], p[2]*z[1]*z[2]);
    a[5] = jfma(z[5], p[1], p[2]*z[2]*z[2]);
  }
  template <class T> static __device__ __forceinline__ void tangent(const T* z, const T* p, const T* v, T* da) {
    da[0] = p[1]*v[0];
    da[1] = jfma(v[1], p[1], p[2]*z[1]*v[0]);
    da[2] = jfma(v[2], p[1], p[2]*z[2]*v[0]);
    da[3] = jfma(v[3], p[1], jfma(v[1], T(2)*p[2]*z[1], jfma(z[3], p[2], p[3]*z[1]*z[1])*v[0]));
    da[4] = jfma(v[4], p[1], jfma(v[2], p[2]*z[1], jfma(v[1], p[2]*z[2], jfma(z[4], p[2], p[3]*z[1]*z[2])*v[0])));
    da[5] = jfma(v[5], p[1], jfma(v[2], T(2)*p[2]*z[2], jfma(z[5], p[2], p[3]*z[2]*z[2])*v[0]));
  }
  template <class T> static __device__ __forceinline__ void adjoint(const T* z, const T* p, const T* ab, T* zb) {
    zb[0] = jfma(ab[5], jfma(z[5], p[2], p[3]*z[2]*z[2]), jfma(ab[4], jfma(z[4], p[2], p[3]*z[1]*z[2]), jfma(ab[3], jfma(z[3], p[2], p[3]*z[1]*z[1]), jfma(ab[2], p[2]*z[2], jfma(ab[1], p[2]*z[1], p[1]*ab[0])))));
    zb[1] = jfma(ab[4], p[2]*z[2], jfma(ab[3], T(2)*p[2]*z[1], p[1]*ab[1]));
    zb[2] = jfma(ab[5], T(2)*p[2]*z[2], jfma(ab[4], p[2]*z[1], p[1]*ab[2]));
    zb[3] = p[1]*ab[3];
    zb[4] = p[1]*ab[4];
    zb[5] = p[1]*ab[5];
  }
  template <class T> static __device__ __forceinline__ void adjoint_conv(const T* z, const T* p, const T* ab, T* zb) {
    T c[6];
    c[0] = p[1];
    c[1] = p[2]*z[1];
    c[2] = p[2]*z[2];
    c[3] = jfma(z[3], p[2], p[3]*z[1]*z[1]);
    c[4] = jfma(z[4], p[2], p[3]*z[1]*z[2]);
    c[5] = jfma(z[5], p[2], p[3]*z[2]*z[2]);
    zb[0] = jfma(ab[5], c[5], jfma(ab[4], c[4], jfma(ab[3], c[3], jfma(ab[2], c[2], jfma(ab[1], c[1], c[0]*ab[0])))));
    zb[1] = jfma(ab[4], c[2], jfma(ab[3], T(2)*c[1], c[0]*ab[1]));
    zb[2] = jfma(ab[5], T(2)*c[2], jfma(ab[4], c[1], c[0]*ab[2]));
    zb[3] = c[0]*ab[3];
    zb[4] = c[0]*ab[4];
    zb[5] = c[0]*ab[5];
  }
};

// d3o2: d=3, channels 000 100 010 001 200 110 101 020 011 002
struct Cls_d3o2 {
  static constexpr int D = 3;
  static constexpr int C = 10;
  static constexpr int MAXORD = 2;
  static constexpr int NP = 4;  // p[0..MAXORD+1]
  // channel index of the first-order channel e_i (-1 if absent)
  static __host__ __device__ constexpr int first_order(int i) { return i == 0 ? 1 : i == 1 ? 2 : i == 2 ? 3 : -1; }
  // first channel index of the highest derivative order
  static constexpr int TOP_BEGIN = 4;
  template <class T> static __device__ __forceinline__ void compose(const T* z, const T* p, T* a) {
    a[0] = p[0];
    a[1] = p[1]*z[1];
    a[2] = p[1]*z[2];
    a[3] = p[1]*z[3];
    a[4] = jfma(z[4], p[1], p[2]*z[1]*z[1]);
    a[5] = jfma(z[5], p[1], p[2]*z[1]*z[2]);
    a[6] = jfma(z[6], p[1], p[2]*z[1]*z[3]);
    a[7] = jfma(z[7], p[1], p[2]*z[2]*z[2]);
    a[8] = jfma(z[8], p[1], p[2]*z[2]*z[3]);
    a[9] = jfma(z[9], p[1], p[2]*z[3]*z[3]);
  }
  template <class T> static __device__ __forceinline__ void tangent(const T* z, const T* p, const T* v, T* da) {
    da[0] = p[1]*v[0];
    da[1] = jfma(v[1], p[1], p[2]*z[1]*v[0]);
    da[2] = jfma(v[2], p[1], p[2]*z[2]*v[0]);
    da[3] = jfma(v[3], p[1], p[2]*z[3]*v[0]);
    da[4] = jfma(v[4], p[1], jfma(v[1], T(2)*p[2]*z[1], jfma(z[4], p[2], p[3]*z[1]*z[1])*v[0]));
    da[5] = jfma(v[5], p[1], jfma(v[2], p[2]*z[1], jfma(v[1], p[2]*z[2], jfma(z[5], p[2], p[3]*z[1]*z[2])*v[0])));
    da[6] = jfma(v[6], p[1], jfma(v[3], p[2]*z[1], jfma(v[1], p[2]*z[3], jfma(z[6], p[2], p[3]*z[1]*z[3])*v[0])));
    da[7] = jfma(v[7], p[1], jfma(v[2], T(2)*p[2]*z[2], jfma(z[7], p[2], p[3]*z[2]*z[2])*v[0]));
    da[8] = jfma(v[8], p[1], jfma(v[3], p[2]*z[2], jfma(v[2], p[2]*z[3], jfma(z[8], p[2], p[3]*z[2]*z[3])*v[0])));
    da[9] = jfma(v[9], p[1], jfma(v[3], T(2)*p[2]*z[3], jfma(z[9], p[2], p[3]*z[3]*z[3])*v[0]));
  }
  template <class T> static __device__ __forceinline__ void adjoint(const T* z, const T* p, const T* ab, T* zb) {
    zb[0] = jfma(ab[9], jfma(z[9], p[2], p[3]*z[3]*z[3]), jfma(ab[8], jfma(z[8], p[2], p[3]*z[2]*z[3]), jfma(ab[7], jfma(z[7], p[2], p[3]*z[2]*z[2]), jfma(ab[6], jfma(z[6], p[2], p[3]*z[1]*z[3]), jfma(ab[5], jfma(z[5], p[2], p[3]*z[1]*z[2]), jfma(ab[4], jfma(z[4], p[2], p[3]*z[1]*z[1]), jfma(ab[3], p[2]*z[3], jfma(ab[2], p[2]*z[2], jfma(ab[1], p[2]*z[1], p[1]*ab[0])))))))));
    zb[1] = jfma(ab[6], p[2]*z[3], jfma(ab[5], p[2]*z[2], jfma(ab[4], T(2)*p[2]*z[1], p[1]*ab[1])));
    zb[2] = jfma(ab[8], p[2]*z[3], jfma(ab[7], T(2)*p[2]*z[2], jfma(ab[5], p[2]*z[1], p[1]*ab[2])));
    zb[3] = jfma(ab[9], T(2)*p[2]*z[3], jfma(ab[8], p[2]*z[2], jfma(ab[6], p[2]*z[1], p[1]*ab[3])));
    zb[4] = p[1]*ab[4];
    zb[5] = p[1]*ab[5];
    zb[6] = p[1]*ab[6];
    zb[7] = p[1]*ab[7];
    zb[8] = p[1]*ab[8];
    zb[9] = p[1]*ab[9];
  }
  template <class T> static __device__ __forceinline__ void adjoint_conv(const T* z, const T* p, const T* ab, T* zb) {
    T c[10];
    c[0] = p[1];
    c[1] = p[2]*z[1];
    c[2] = p[2]*z[2];
    c[3] = p[2]*z[3];
    c[4] = jfma(z[4], p[2], p[3]*z[1]*z[1]);
    c[5] = jfma(z[5], p[2], p[3]*z[1]*z[2]);
    c[6] = jfma(z[6], p[2], p[3]*z[1]*z[3]);
    c[7] = jfma(z[7], p[2], p[3]*z[2]*z[2]);
    c[8] = jfma(z[8], p[2], p[3]*z[2]*z[3]);
    c[9] = jfma(z[9], p[2], p[3]*z[3]*z[3]);
    zb[0] = jfma(ab[9], c[9], jfma(ab[8], c[8], jfma(ab[7], c[7], jfma(ab[6], c[6], jfma(ab[5], c[5], jfma(ab[4], c[4], jfma(ab[3], c[3], jfma(ab[2], c[2], jfma(ab[1], c[1], c[0]*ab[0])))))))));
    zb[1] = jfma(ab[6], c[3], jfma(ab[5], c[2], jfma(ab[4], T(2)*c[1], c[0]*ab[1])));
    zb[2] = jfma(ab[8], c[3], jfma(ab[7], T(2)*c[2], jfma(ab[5], c[1], c[0]*ab[2])));
    zb[3] = jfma(ab[9], T(2)*c[3], jfma(ab[8], c[2], jfma(ab[6], c[1], c[0]*ab[3])));
    zb[4] = c[0]*ab[4];
    zb[5] = c[0]*ab[5];
    zb[6] = c[0]*ab[6];
    zb[7] = c[0]*ab[7];
    zb[8] = c[0]*ab[8];
    zb[9] = c[0]*ab[9];
  }
};

// burgers: d=2, channels 00 10 01 20
struct Cls_burgers {
  static constexpr int D = 2;
  static constexpr int C = 4;
  static constexpr int MAXORD = 2;
  static constexpr int NP = 4;  // p[0..MAXORD+1]
  // channel index of the first-order channel e_i (-1 if absent)
  static __host__ __device__ constexpr int first_order(int i) { return i == 0 ? 1 : i == 1 ? 2 : -1; }
  // first channel index of the highest derivative order
  static constexpr int TOP_BEGIN = 3;
  template <class T> static __device__ __forceinline__ void compose(const T* z, const T* p, T* a) {
    a[0] = p[0];
    a[1] = p[1]*z[1];
    a[2] = p[1]*z[2];
    a[3] = jfma(z[3], p[1], p[2]*z[1]*z[1]);
  }
  template <class T> static __device__ __forceinline__ void tangent(const T* z, const T* p, const T* v, T* da) {
    da[0] = p[1]*v[0];
    da[1] = jfma(v[1], p[1], p[2]*z[1]*v[0]);
    da[2] = jfma(v[2], p[1], p[2]*z[2]*v[0]);
    da[3] = jfma(v[3], p[1], jfma(v[1], T(2)*p[2]*z[1], jfma(z[3], p[2], p[3]*z[1]*z[1])*v[0]));
  }
  template <class T> static __device__ __forceinline__ void adjoint(const T* z, const T* p, const T* ab, T* zb) {
    zb[0] = jfma(ab[3], jfma(z[3], p[2], p[3]*z[1]*z[1]), jfma(ab[2], p[2]*z[2], jfma(ab[1], p[2]*z[1], p[1]*ab[0])));
    zb[1] = jfma(ab[3], T(2)*p[2]*z[1], p[1]*ab[1]);
    zb[2] = p[1]*ab[2];
    zb[3] = p[1]*ab[3];
  }
  template <class T> static __device__ __forceinline__ void adjoint_conv(const T* z, const T* p, const T* ab, T* zb) {
    T c[4];
    c[0] = p[1];
    c[1] = p[2]*z[1];
    c[2] = p[2]*z[2];
    c[3] = jfma(z[3], p[2], p[3]*z[1]*z[1]);
    zb[0] = jfma(ab[3], c[3], jfma(ab[2], c[2], jfma(ab[1], c[1], c[0]*ab[0])));
    zb[1] = jfma(ab[3], T(2)*c[1], c[0]*ab[1]);
    zb[2] = c[0]*ab[2];
    zb[3] = c[0]*ab[3];
  }
};

// ks: d=2, channels 00 10 01 20 30 40
struct Cls_ks {
  static constexpr int D = 2;
  static constexpr int C = 6;
  static constexpr int MAXORD = 4;
  static constexpr int NP = 6;  // p[0..MAXORD+1]
  // channel index of the first-order channel e_i (-1 if absent)
  static __host__ __device__ constexpr int first_order(int i) { return i == 0 ? 1 : i == 1 ? 2 : -1; }
  // first channel index of the highest derivative order
  static constexpr int TOP_BEGIN = 5;
  template <class T> static __device__ __forceinline__ void compose(const T* z, const T* p, T* a) {
    a[0] = p[0];
    a[1] = p[1]*z[1];
    a[2] = p[1]*z[2];
    a[3] = jfma(z[3], p[1], p[2]*z[1]*z[1]);
    a[4] = jfma(z[4], p[1], jfma(z[3], T(3)*p[2]*z[1], p[3]*z[1]*z[1]*z[1]));
    a[5] = jfma(z[5], p[1], jfma(z[3], T(3)*p[2]*z[3], jfma(z[4], T(4)*p[2]*z[1], jfma(z[3], T(6)*p[3]*z[1]*z[1], p[4]*z[1]*z[1]*z[1]*z[1]))));
  }
  template <class T> static __device__ __forceinline__ void tangent(const T* z, const T* p, const T* v, T* da) {
    da[0] = p[1]*v[0];
    da[1] = jfma(v[1], p[1], p[2]*z[1]*v[0]);
    da[2] = jfma(v[2], p[1], p[2]*z[2]*v[0]);
    da[3] = jfma(v[3], p[1], jfma(v[1], T(2)*p[2]*z[1], jfma(z[3], p[2], p[3]*z[1]*z[1])*v[0]));
    da[4] = jfma(v[4], p[1], jfma(v[3], T(3)*p[2]*z[1], jfma(v[1], jfma(z[3], T(3)*p[2], T(3)*p[3]*z[1]*z[1]), jfma(z[4], p[2], jfma(z[3], T(3)*p[3]*z[1], p[4]*z[1]*z[1]*z[1]))*v[0])));
    da[5] = jfma(v[5], p[1], jfma(v[4], T(4)*p[2]*z[1], jfma(v[3], jfma(z[3], T(6)*p[2], T(6)*p[3]*z[1]*z[1]), jfma(v[1], jfma(z[4], T(4)*p[2], jfma(z[3], T(12)*p[3]*z[1], T(4)*p[4]*z[1]*z[1]*z[1])), jfma(z[5], p[2], jfma(z[3], T(3)*p[3]*z[3], jfma(z[4], T(4)*p[3]*z[1], jfma(z[3], T(6)*p[4]*z[1]*z[1], p[5]*z[1]*z[1]*z[1]*z[1]))))*v[0]))));
  }
  template <class T> static __device__ __forceinline__ void adjoint(const T* z, const T* p, const T* ab, T* zb) {
    zb[0] = jfma(ab[5], jfma(z[5], p[2], jfma(z[3], T(3)*p[3]*z[3], jfma(z[4], T(4)*p[3]*z[1], jfma(z[3], T(6)*p[4]*z[1]*z[1], p[5]*z[1]*z[1]*z[1]*z[1])))), jfma(ab[4], jfma(z[4], p[2], jfma(z[3], T(3)*p[3]*z[1], p[4]*z[1]*z[1]*z[1])), jfma(ab[3], jfma(z[3], p[2], p[3]*z[1]*z[1]), jfma(ab[2], p[2]*z[2], jfma(ab[1], p[2]*z[1], p[1]*ab[0])))));
    zb[1] = jfma(ab[5], jfma(z[4], T(4)*p[2], jfma(z[3], T(12)*p[3]*z[1], T(4)*p[4]*z[1]*z[1]*z[1])), jfma(ab[4], jfma(z[3], T(3)*p[2], T(3)*p[3]*z[1]*z[1]), jfma(ab[3], T(2)*p[2]*z[1], p[1]*ab[1])));
    zb[2] = p[1]*ab[2];
    zb[3] = jfma(ab[5], jfma(z[3], T(6)*p[2], T(6)*p[3]*z[1]*z[1]), jfma(ab[4], T(3)*p[2]*z[1], p[1]*ab[3]));
    zb[4] = jfma(ab[5], T(4)*p[2]*z[1], p[1]*ab[4]);
    zb[5] = p[1]*ab[5];
  }
  template <class T> static __device__ __forceinline__ void adjoint_conv(const T* z, const T* p, const T* ab, T* zb) {
    T c[6];
    c[0] = p[1];
    c[1] = p[2]*z[1];
    c[2] = p[2]*z[2];
    c[3] = jfma(z[3], p[2], p[3]*z[1]*z[1]);
    c[4] = jfma(z[4], p[2], jfma(z[3], T(3)*p[3]*z[1], p[4]*z[1]*z[1]*z[1]));
    c[5] = jfma(z[5], p[2], jfma(z[3], T(3)*p[3]*z[3], jfma(z[4], T(4)*p[3]*z[1], jfma(z[3], T(6)*p[4]*z[1]*z[1], p[5]*z[1]*z[1]*z[1]*z[1]))));
    zb[0] = jfma(ab[5], c[5], jfma(ab[4], c[4], jfma(ab[3], c[3], jfma(ab[2], c[2], jfma(ab[1], c[1], c[0]*ab[0])))));
    zb[1] = jfma(ab[5], T(4)*c[4], jfma(ab[4], T(3)*c[3], jfma(ab[3], T(2)*c[1], c[0]*ab[1])));
    zb[2] = c[0]*ab[2];
    zb[3] = jfma(ab[5], T(6)*c[3], jfma(ab[4], T(3)*c[1], c[0]*ab[3]));
    zb[4] = jfma(ab[5], T(4)*c[1], c[0]*ab[4]);
    zb[5] = c[0]*ab[5];
  }
};

// helmholtz: d=3, channels 000 100 010 001 200 020 002
struct Cls_helmholtz {
  static constexpr int D = 3;
  static constexpr int C = 7;
  static constexpr int MAXORD = 2;
  static constexpr int NP = 4;  // p[0..MAXORD+1]
  // channel index of the first-order channel e_i (-1 if absent)
  static __host__ __device__ constexpr int first_order(int i) { return i == 0 ? 1 : i == 1 ? 2 : i == 2 ? 3 : -1; }
  // first channel index of the highest derivative order
  static constexpr int TOP_BEGIN = 4;
  template <class T> static __device__ __forceinline__ void compose(const T* z, const T* p, T* a) {
    a[0] = p[0];
    a[1] = p[1]*z[1];
    a[2] = p[1]*z[2];
    a[3] = p[1]*z[3];
    a[4] = jfma(z[4], p[1], p[2]*z[1]*z[1]);
    a[5] = jfma(z[5], p[1], p[2]*z[2]*z[2]);
    a[6] = jfma(z[6], p[1], p[2]*z[3]*z[3]);
  }
  template <class T> static __device__ __forceinline__ void tangent(const T* z, const T* p, const T* v, T* da) {
    da[0] = p[1]*v[0];
    da[1] = jfma(v[1], p[1], p[2]*z[1]*v[0]);
    da[2] = jfma(v[2], p[1], p[2]*z[2]*v[0]);
    da[3] = jfma(v[3], p[1], p[2]*z[3]*v[0]);
    da[4] = jfma(v[4], p[1], jfma(v[1], T(2)*p[2]*z[1], jfma(z[4], p[2], p[3]*z[1]*z[1])*v[0]));
    da[5] = jfma(v[5], p[1], jfma(v[2], T(2)*p[2]*z[2], jfma(z[5], p[2], p[3]*z[2]*z[2])*v[0]));
    da[6] = jfma(v[6], p[1], jfma(v[3], T(2)*p[2]*z[3], jfma(z[6], p[2], p[3]*z[3]*z[3])*v[0]));
  }
  template <class T> static __device__ __forceinline__ void adjoint(const T* z, const T* p, const T* ab, T* zb) {
    zb[0] = jfma(ab[6], jfma(z[6], p[2], p[3]*z[3]*z[3]), jfma(ab[5], jfma(z[5], p[2], p[3]*z[2]*z[2]), jfma(ab[4], jfma(z[4], p[2], p[3]*z[1]*z[1]), jfma(ab[3], p[2]*z[3], jfma(ab[2], p[2]*z[2], jfma(ab[1], p[2]*z[1], p[1]*ab[0]))))));
    zb[1] = jfma(ab[4], T(2)*p[2]*z[1], p[1]*ab[1]);
    zb[2] = jfma(ab[5], T(2)*p[2]*z[2], p[1]*ab[2]);
    zb[3] = jfma(ab[6], T(2)*p[2]*z[3], p[1]*ab[3]);
    zb[4] = p[1]*ab[4];
    zb[5] = p[1]*ab[5];
    zb[6] = p[1]*ab[6];
  }
  template <class T> static __device__ __forceinline__ void adjoint_conv(const T* z, const T* p, const T* ab, T* zb) {
    T c[7];
    c[0] = p[1];
    c[1] = p[2]*z[1];
    c[2] = p[2]*z[2];
    c[3] = p[2]*z[3];
    c[4] = jfma(z[4], p[2], p[3]*z[1]*z[1]);
    c[5] = jfma(z[5], p[2], p[3]*z[2]*z[2]);
    c[6] = jfma(z[6], p[2], p[3]*z[3]*z[3]);
    zb[0] = jfma(ab[6], c[6], jfma(ab[5], c[5], jfma(ab[4], c[4], jfma(ab[3], c[3], jfma(ab[2], c[2], jfma(ab[1], c[1], c[0]*ab[0]))))));
    zb[1] = jfma(ab[4], T(2)*c[1], c[0]*ab[1]);
    zb[2] = jfma(ab[5], T(2)*c[2], c[0]*ab[2]);
    zb[3] = jfma(ab[6], T(2)*c[3], c[0]*ab[3]);
    zb[4] = c[0]*ab[4];
    zb[5] = c[0]*ab[5];
    zb[6] = c[0]*ab[6];
  }
};

// ns_psi: d=3, channels 000 100 010 001 200 110 101 020 011 300 210 120 030
struct Cls_ns_psi {
  static constexpr int D = 3;
  static constexpr int C = 13;
  static constexpr int MAXORD = 3;
  static constexpr int NP = 5;  // p[0..MAXORD+1]
  // channel index of the first-order channel e_i (-1 if absent)
  static __host__ __device__ constexpr int first_order(int i) { return i == 0 ? 1 : i == 1 ? 2 : i == 2 ? 3 : -1; }
  // first channel index of the highest derivative order
  static constexpr int TOP_BEGIN = 9;
  template <class T> static __device__ __forceinline__ void compose(const T* z, const T* p, T* a) {
    a[0] = p[0];
    a[1] = p[1]*z[1];
    a[2] = p[1]*z[2];
    a[3] = p[1]*z[3];
    a[4] = jfma(z[4], p[1], p[2]*z[1]*z[1]);
    a[5] = jfma(z[5], p[1], p[2]*z[1]*z[2]);
    a[6] = jfma(z[6], p[1], p[2]*z[1]*z[3]);
    a[7] = jfma(z[7], p[1], p[2]*z[2]*z[2]);
    a[8] = jfma(z[8], p[1], p[2]*z[2]*z[3]);
    a[9] = jfma(z[9], p[1], jfma(z[4], T(3)*p[2]*z[1], p[3]*z[1]*z[1]*z[1]));
    a[10] = jfma(z[10], p[1], jfma(z[5], T(2)*p[2]*z[1], jfma(z[4], p[2]*z[2], p[3]*z[1]*z[1]*z[2])));
    a[11] = jfma(z[11], p[1], jfma(z[7], p[2]*z[1], jfma(z[5], T(2)*p[2]*z[2], p[3]*z[1]*z[2]*z[2])));
    a[12] = jfma(z[12], p[1], jfma(z[7], T(3)*p[2]*z[2], p[3]*z[2]*z[2]*z[2]));
  }
  template <class T> static __device__ __forceinline__ void tangent(const T* z, const T* p, const T* v, T* da) {
    da[0] = p[1]*v[0];
    da[1] = jfma(v[1], p[1], p[2]*z[1]*v[0]);
    da[2] = jfma(v[2], p[1], p[2]*z[2]*v[0]);
    da[3] = jfma(v[3], p[1], p[2]*z[3]*v[0]);
    da[4] = jfma(v[4], p[1], jfma(v[1], T(2)*p[2]*z[1], jfma(z[4], p[2], p[3]*z[1]*z[1])*v[0]));
    da[5] = jfma(v[5], p[1], jfma(v[2], p[2]*z[1], jfma(v[1], p[2]*z[2], jfma(z[5], p[2], p[3]*z[1]*z[2])*v[0])));
    da[6] = jfma(v[6], p[1], jfma(v[3], p[2]*z[1], jfma(v[1], p[2]*z[3], jfma(z[6], p[2], p[3]*z[1]*z[3])*v[0])));
    da[7] = jfma(v[7], p[1], jfma(v[2], T(2)*p[2]*z[2], jfma(z[7], p[2], p[3]*z[2]*z[2])*v[0]));
    da[8] = jfma(v[8], p[1], jfma(v[3], p[2]*z[2], jfma(v[2], p[2]*z[3], jfma(z[8], p[2], p[3]*z[2]*z[3])*v[0])));
    da[9] = jfma(v[9], p[1], jfma(v[4], T(3)*p[2]*z[1], jfma(v[1], jfma(z[4], T(3)*p[2], T(3)*p[3]*z[1]*z[1]), jfma(z[9], p[2], jfma(z[4], T(3)*p[3]*z[1], p[4]*z[1]*z[1]*z[1]))*v[0])));
    da[10] = jfma(v[10], p[1], jfma(v[5], T(2)*p[2]*z[1], jfma(v[4], p[2]*z[2], jfma(v[2], jfma(z[4], p[2], p[3]*z[1]*z[1]), jfma(v[1], jfma(z[5], T(2)*p[2], T(2)*p[3]*z[1]*z[2]), jfma(z[10], p[2], jfma(z[5], T(2)*p[3]*z[1], jfma(z[4], p[3]*z[2], p[4]*z[1]*z[1]*z[2])))*v[0])))));
    da[11] = jfma(v[11], p[1], jfma(v[7], p[2]*z[1], jfma(v[5], T(2)*p[2]*z[2], jfma(v[2], jfma(z[5], T(2)*p[2], T(2)*p[3]*z[1]*z[2]), jfma(v[1], jfma(z[7], p[2], p[3]*z[2]*z[2]), jfma(z[11], p[2], jfma(z[7], p[3]*z[1], jfma(z[5], T(2)*p[3]*z[2], p[4]*z[1]*z[2]*z[2])))*v[0])))));
    da[12] = jfma(v[12], p[1], jfma(v[7], T(3)*p[2]*z[2], jfma(v[2], jfma(z[7], T(3)*p[2], T(3)*p[3]*z[2]*z[2]), jfma(z[12], p[2], jfma(z[7], T(3)*p[3]*z[2], p[4]*z[2]*z[2]*z[2]))*v[0])));
  }
  template <class T> static __device__ __forceinline__ void adjoint(const T* z, const T* p, const T* ab, T* zb) {
    zb[0] = jfma(ab[12], jfma(z[12], p[2], jfma(z[7], T(3)*p[3]*z[2], p[4]*z[2]*z[2]*z[2])), jfma(ab[11], jfma(z[11], p[2], jfma(z[7], p[3]*z[1], jfma(z[5], T(2)*p[3]*z[2], p[4]*z[1]*z[2]*z[2]))), jfma(ab[10], jfma(z[10], p[2], jfma(z[5], T(2)*p[3]*z[1], jfma(z[4], p[3]*z[2], p[4]*z[1]*z[1]*z[2]))), jfma(ab[9], jfma(z[9], p[2], jfma(z[4], T(3)*p[3]*z[1], p[4]*z[1]*z[1]*z[1])), jfma(ab[8], jfma(z[8], p[2], p[3]*z[2]*z[3]), jfma(ab[7], jfma(z[7], p[2], p[3]*z[2]*z[2]), jfma(ab[6], jfma(z[6], p[2], p[3]*z[1]*z[3]), jfma(ab[5], jfma(z[5], p[2], p[3]*z[1]*z[2]), jfma(ab[4], jfma(z[4], p[2], p[3]*z[1]*z[1]), jfma(ab[3], p[2]*z[3], jfma(ab[2], p[2]*z[2], jfma(ab[1], p[2]*z[1], p[1]*ab[0]))))))))))));
    zb[1] = jfma(ab[11], jfma(z[7], p[2], p[3]*z[2]*z[2]), jfma(ab[10], jfma(z[5], T(2)*p[2], T(2)*p[3]*z[1]*z[2]), jfma(ab[9], jfma(z[4], T(3)*p[2], T(3)*p[3]*z[1]*z[1]), jfma(ab[6], p[2]*z[3], jfma(ab[5], p[2]*z[2], jfma(ab[4], T(2)*p[2]*z[1], p[1]*ab[1]))))));
    zb[2] = jfma(ab[12], jfma(z[7], T(3)*p[2], T(3)*p[3]*z[2]*z[2]), jfma(ab[11], jfma(z[5], T(2)*p[2], T(2)*p[3]*z[1]*z[2]), jfma(ab[10], jfma(z[4], p[2], p[3]*z[1]*z[1]), jfma(ab[8], p[2]*z[3], jfma(ab[7], T(2)*p[2]*z[2], jfma(ab[5], p[2]*z[1], p[1]*ab[2]))))));
    zb[3] = jfma(ab[8], p[2]*z[2], jfma(ab[6], p[2]*z[1], p[1]*ab[3]));
    zb[4] = jfma(ab[10], p[2]*z[2], jfma(ab[9], T(3)*p[2]*z[1], p[1]*ab[4]));
    zb[5] = jfma(ab[11], T(2)*p[2]*z[2], jfma(ab[10], T(2)*p[2]*z[1], p[1]*ab[5]));
    zb[6] = p[1]*ab[6];
    zb[7] = jfma(ab[12], T(3)*p[2]*z[2], jfma(ab[11], p[2]*z[1], p[1]*ab[7]));
    zb[8] = p[1]*ab[8];
    zb[9] = p[1]*ab[9];
    zb[10] = p[1]*ab[10];
    zb[11] = p[1]*ab[11];
    zb[12] = p[1]*ab[12];
  }
  template <class T> static __device__ __forceinline__ void adjoint_conv(const T* z, const T* p, const T* ab, T* zb) {
    T c[13];
    c[0] = p[1];
    c[1] = p[2]*z[1];
    c[2] = p[2]*z[2];
    c[3] = p[2]*z[3];
    c[4] = jfma(z[4], p[2], p[3]*z[1]*z[1]);
    c[5] = jfma(z[5], p[2], p[3]*z[1]*z[2]);
    c[6] = jfma(z[6], p[2], p[3]*z[1]*z[3]);
    c[7] = jfma(z[7], p[2], p[3]*z[2]*z[2]);
    c[8] = jfma(z[8], p[2], p[3]*z[2]*z[3]);
    c[9] = jfma(z[9], p[2], jfma(z[4], T(3)*p[3]*z[1], p[4]*z[1]*z[1]*z[1]));
    c[10] = jfma(z[10], p[2], jfma(z[5], T(2)*p[3]*z[1], jfma(z[4], p[3]*z[2], p[4]*z[1]*z[1]*z[2])));
    c[11] = jfma(z[11], p[2], jfma(z[7], p[3]*z[1], jfma(z[5], T(2)*p[3]*z[2], p[4]*z[1]*z[2]*z[2])));
    c[12] = jfma(z[12], p[2], jfma(z[7], T(3)*p[3]*z[2], p[4]*z[2]*z[2]*z[2]));
    zb[0] = jfma(ab[12], c[12], jfma(ab[11], c[11], jfma(ab[10], c[10], jfma(ab[9], c[9], jfma(ab[8], c[8], jfma(ab[7], c[7], jfma(ab[6], c[6], jfma(ab[5], c[5], jfma(ab[4], c[4], jfma(ab[3], c[3], jfma(ab[2], c[2], jfma(ab[1], c[1], c[0]*ab[0]))))))))))));
    zb[1] = jfma(ab[11], c[7], jfma(ab[10], T(2)*c[5], jfma(ab[9], T(3)*c[4], jfma(ab[6], c[3], jfma(ab[5], c[2], jfma(ab[4], T(2)*c[1], c[0]*ab[1]))))));
    zb[2] = jfma(ab[12], T(3)*c[7], jfma(ab[11], T(2)*c[5], jfma(ab[10], c[4], jfma(ab[8], c[3], jfma(ab[7], T(2)*c[2], jfma(ab[5], c[1], c[0]*ab[2]))))));
    zb[3] = jfma(ab[8], c[2], jfma(ab[6], c[1], c[0]*ab[3]));
    zb[4] = jfma(ab[10], c[2], jfma(ab[9], T(3)*c[1], c[0]*ab[4]));
    zb[5] = jfma(ab[11], T(2)*c[2], jfma(ab[10], T(2)*c[1], c[0]*ab[5]));
    zb[6] = c[0]*ab[6];
    zb[7] = jfma(ab[12], T(3)*c[2], jfma(ab[11], c[1], c[0]*ab[7]));
    zb[8] = c[0]*ab[8];
    zb[9] = c[0]*ab[9];
    zb[10] = c[0]*ab[10];
    zb[11] = c[0]*ab[11];
    zb[12] = c[0]*ab[12];
  }
};

// ns_uvp: d=2, channels 00 10 01 20 02
struct Cls_ns_uvp {
  static constexpr int D = 2;
  static constexpr int C = 5;
  static constexpr int MAXORD = 2;
  static constexpr int NP = 4;  // p[0..MAXORD+1]
  // channel index of the first-order channel e_i (-1 if absent)
  static __host__ __device__ constexpr int first_order(int i) { return i == 0 ? 1 : i == 1 ? 2 : -1; }
  // first channel index of the highest derivative order
  static constexpr int TOP_BEGIN = 3;
  template <class T> static __device__ __forceinline__ void compose(const T* z, const T* p, T* a) {
    a[0] = p[0];
    a[1] = p[1]*z[1];
    a[2] = p[1]*z[2];
    a[3] = jfma(z[3], p[1], p[2]*z[1]*z[1]);
    a[4] = jfma(z[4], p[1], p[2]*z[2]*z[2]);
  }
  template <class T> static __device__ __forceinline__ void tangent(const T* z, const T* p, const T* v, T* da) {
    da[0] = p[1]*v[0];
    da[1] = jfma(v[1], p[1], p[2]*z[1]*v[0]);
    da[2] = jfma(v[2], p[1], p[2]*z[2]*v[0]);
    da[3] = jfma(v[3], p[1], jfma(v[1], T(2)*p[2]*z[1], jfma(z[3], p[2], p[3]*z[1]*z[1])*v[0]));
    da[4] = jfma(v[4], p[1], jfma(v[2], T(2)*p[2]*z[2], jfma(z[4], p[2], p[3]*z[2]*z[2])*v[0]));
  }
  template <class T> static __device__ __forceinline__ void adjoint(const T* z, const T* p, const T* ab, T* zb) {
    zb[0] = jfma(ab[4], jfma(z[4], p[2], p[3]*z[2]*z[2]), jfma(ab[3], jfma(z[3], p[2], p[3]*z[1]*z[1]), jfma(ab[2], p[2]*z[2], jfma(ab[1], p[2]*z[1], p[1]*ab[0]))));
    zb[1] = jfma(ab[3], T(2)*p[2]*z[1], p[1]*ab[1]);
    zb[2] = jfma(ab[4], T(2)*p[2]*z[2], p[1]*ab[2]);
    zb[3] = p[1]*ab[3];
    zb[4] = p[1]*ab[4];
  }
  template <class T> static __device__ __forceinline__ void adjoint_conv(const T* z, const T* p, const T* ab, T* zb) {
    T c[5];
    c[0] = p[1];
    c[1] = p[2]*z[1];
    c[2] = p[2]*z[2];
    c[3] = jfma(z[3], p[2], p[3]*z[1]*z[1]);
    c[4] = jfma(z[4], p[2], p[3]*z[2]*z[2]);
    zb[0] = jfma(ab[4], c[4], jfma(ab[3], c[3], jfma(ab[2], c[2], jfma(ab[1], c[1], c[0]*ab[0]))));
    zb[1] = jfma(ab[3], T(2)*c[1], c[0]*ab[1]);
    zb[2] = jfma(ab[4], T(2)*c[2], c[0]*ab[2]);
    zb[3] = c[0]*ab[3];
    zb[4] = c[0]*ab[4];
  }
};

struct ClassInfo { const char* name; int d; int C; int maxord; unsigned char alpha[16][3]; };
static const ClassInfo kClassInfo[] = {
  {"d1o4", 1, 5, 4, {{0, 0, 0}, {1, 0, 0}, {2, 0, 0}, {3, 0, 0}, {4, 0, 0}}},
  {"d2o2", 2, 6, 2, {{0, 0, 0}, {1, 0, 0}, {0, 1, 0}, {2, 0, 0}, {1, 1, 0}, {0, 2, 0}}},
  {"d3o2", 3, 10, 2, {{0, 0, 0}, {1, 0, 0}, {0, 1, 0}, {0, 0, 1}, {2, 0, 0}, {1, 1, 0}, {1, 0, 1}, {0, 2, 0}, {0, 1, 1}, {0, 0, 2}}},
  {"burgers", 2, 4, 2, {{0, 0, 0}, {1, 0, 0}, {0, 1, 0}, {2, 0, 0}}},
  {"ks", 2, 6, 4, {{0, 0, 0}, {1, 0, 0}, {0, 1, 0}, {2, 0, 0}, {3, 0, 0}, {4, 0, 0}}},
  {"helmholtz", 3, 7, 2, {{0, 0, 0}, {1, 0, 0}, {0, 1, 0}, {0, 0, 1}, {2, 0, 0}, {0, 2, 0}, {0, 0, 2}}},
  {"ns_psi", 3, 13, 3, {{0, 0, 0}, {1, 0, 0}, {0, 1, 0}, {0, 0, 1}, {2, 0, 0}, {1, 1, 0}, {1, 0, 1}, {0, 2, 0}, {0, 1, 1}, {3, 0, 0}, {2, 1, 0}, {1, 2, 0}, {0, 3, 0}}},
  {"ns_uvp", 2, 5, 2, {{0, 0, 0}, {1, 0, 0}, {0, 1, 0}, {2, 0, 0}, {0, 2, 0}}},
};
static constexpr int kNumClasses = 8;

template <int ID> struct ClassById;
template <> struct ClassById<0> { using type = Cls_d1o4; };
template <> struct ClassById<1> { using type = Cls_d2o2; };
template <> struct ClassById<2> { using type = Cls_d3o2; };
template <> struct ClassById<3> { using type = Cls_burgers; };
template <> struct ClassById<4> { using type = Cls_ks; };
template <> struct ClassById<5> { using type = Cls_helmholtz; };
template <> struct ClassById<6> { using type = Cls_ns_psi; };
template <> struct ClassById<7> { using type = Cls_ns_uvp; };

// per class id: JET_TC_SHAPES_<id>(M) expands M(PC, G, H, W, NT) for every compiled fixed shape
#define JET_TC_SHAPES_0(M) 
#define JET_TC_SHAPES_1(M) 
#define JET_TC_SHAPES_2(M) 
#define JET_TC_SHAPES_3(M) M(64, 2, 1, 128, 512) M(64, 0, 1, 128, 512) M(48, 0, 1, 128, 512) M(32, 0, 1, 128, 512) M(16, 0, 1, 128, 512)
#define JET_TC_SHAPES_4(M) M(32, 2, 1, 128, 512) M(40, 2, 1, 128, 512) M(16, 2, 1, 128, 256) M(16, 2, 1, 128, 512)
#define JET_TC_SHAPES_5(M) M(16, 1, 2, 256, 512) M(8, 1, 2, 256, 512)
#define JET_TC_SHAPES_6(M) M(16, 1, 1, 128, 512) M(8, 1, 1, 128, 512) M(8, 1, 1, 128, 256)
#define JET_TC_SHAPES_7(M) M(48, 2, 1, 128, 512) M(32, 0, 1, 128, 512) M(16, 0, 1, 128, 512)

// X-macro over the classes: JET_FOR_EACH_CLASS(M) expands M(id, Cls_name)
#define JET_FOR_EACH_CLASS(M) \
  M(0, Cls_d1o4) \
  M(1, Cls_d2o2) \
  M(2, Cls_d3o2) \
  M(3, Cls_burgers) \
  M(4, Cls_ks) \
  M(5, Cls_helmholtz) \
  M(6, Cls_ns_psi) \
  M(7, Cls_ns_uvp)

}  // namespace jet
