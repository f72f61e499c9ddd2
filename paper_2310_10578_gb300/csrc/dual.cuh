// dual.cuh -- dual numbers for the adjoint (reverse) pass.
//
// DualT<S, N> carries a value and its derivatives with respect to N parameters
// of one path: for a path round a body (N = 7) slots 0-3 the centre (x, y, z)
// and radius of that body and 4-6 the transmitter position; for a planar path
// (N = 3) the transmitter position; in FP32 (N = 8) all of them and the
// frequency; N = 2 for the slopes of a function of two
// variables.  Each path's geometry depends on no other parameter once its
// visibility is fixed.  Every operation below applies the first-order chain
// rule to the operation in the value's own precision.
#pragma once
#include "devmath.cuh"

namespace creep {

enum { DS_CX = 0, DS_CY = 1, DS_CZ = 2, DS_A = 3, DS_SX = 4, DS_SY = 5, DS_SZ = 6, DS_F = 7 };

template <typename S, int N>
struct DualT {
    S v;
    S d[N];
    DualT() = default;
    __device__ __forceinline__ DualT(S a) : v(a) {
#pragma unroll
        for (int k = 0; k < N; ++k) d[k] = S(0);
    }
};
typedef DualT<double, 3> D3;         // planar paths: the transmitter
typedef DualT<double, 7> D7;         // paths round a body: its centre and radius, the transmitter
typedef DualT<float, 8> F8;          // FP32: those and the frequency

// the value-precision math of a dual's scalar type
__device__ __forceinline__ void dsincos(double x, double *s, double *c) { sincos(x, s, c); }
__device__ __forceinline__ void dsincos(float x, float *s, float *c) { sincosf(x, s, c); }
__device__ __forceinline__ void dsincospi(double x, double *s, double *c) { sincospi(x, s, c); }
__device__ __forceinline__ void dsincospi(float x, float *s, float *c) { sincospif(x, s, c); }

// a parameter: value a, derivative 1 in slot k
template <typename S, int N>
__device__ __forceinline__ DualT<S, N> dvar_t(S a, int k) {
    DualT<S, N> r(a);
    r.d[k] = S(1);
    return r;
}
// y = f(x) with f'(x) = df: y.d = df x.d
template <typename S, int N>
__device__ __forceinline__ DualT<S, N> dchain(S y, S df, const DualT<S, N> &x) {
    DualT<S, N> r;
    r.v = y;
#pragma unroll
    for (int k = 0; k < N; ++k) r.d[k] = df * x.d[k];
    return r;
}
template <typename S, int N>
__device__ __forceinline__ DualT<S, N> operator+(const DualT<S, N> &a, const DualT<S, N> &b) {
    DualT<S, N> r;
    r.v = a.v + b.v;
#pragma unroll
    for (int k = 0; k < N; ++k) r.d[k] = a.d[k] + b.d[k];
    return r;
}
template <typename S, int N>
__device__ __forceinline__ DualT<S, N> operator-(const DualT<S, N> &a, const DualT<S, N> &b) {
    DualT<S, N> r;
    r.v = a.v - b.v;
#pragma unroll
    for (int k = 0; k < N; ++k) r.d[k] = a.d[k] - b.d[k];
    return r;
}
template <typename S, int N>
__device__ __forceinline__ DualT<S, N> operator-(const DualT<S, N> &a) {
    DualT<S, N> r;
    r.v = -a.v;
#pragma unroll
    for (int k = 0; k < N; ++k) r.d[k] = -a.d[k];
    return r;
}
template <typename S, int N>
__device__ __forceinline__ DualT<S, N> operator*(const DualT<S, N> &a, const DualT<S, N> &b) {
    DualT<S, N> r;
    r.v = a.v * b.v;
#pragma unroll
    for (int k = 0; k < N; ++k) r.d[k] = a.d[k] * b.v + a.v * b.d[k];
    return r;
}
template <typename S, int N>
__device__ __forceinline__ DualT<S, N> operator/(const DualT<S, N> &a, const DualT<S, N> &b) {
    DualT<S, N> r;
    const S ib = S(1) / b.v;
    r.v = a.v * ib;
#pragma unroll
    for (int k = 0; k < N; ++k) r.d[k] = (a.d[k] - r.v * b.d[k]) * ib;
    return r;
}
template <typename S, int N> __device__ __forceinline__ bool operator<(const DualT<S, N> &a, const DualT<S, N> &b) { return a.v < b.v; }
template <typename S, int N> __device__ __forceinline__ bool operator>(const DualT<S, N> &a, const DualT<S, N> &b) { return a.v > b.v; }
template <typename S, int N> __device__ __forceinline__ bool operator<=(const DualT<S, N> &a, const DualT<S, N> &b) { return a.v <= b.v; }
template <typename S, int N> __device__ __forceinline__ bool operator>=(const DualT<S, N> &a, const DualT<S, N> &b) { return a.v >= b.v; }
template <typename S, int N> __device__ __forceinline__ bool operator==(const DualT<S, N> &a, const DualT<S, N> &b) { return a.v == b.v; }
template <typename S, int N> __device__ __forceinline__ bool operator!=(const DualT<S, N> &a, const DualT<S, N> &b) { return a.v != b.v; }

template <typename S, int N>
__device__ __forceinline__ DualT<S, N> Sqrt(const DualT<S, N> &x) {
    const S s = sqrt(x.v);
    return dchain<S, N>(s, s > S(0) ? S(0.5) / s : S(0), x);
}
template <typename S, int N>
__device__ __forceinline__ DualT<S, N> Cbrt(const DualT<S, N> &x) {
    const S c = cbrt(x.v);
    return dchain<S, N>(c, c != S(0) ? S(1) / (S(3) * c * c) : S(0), x);
}
template <typename S, int N>
__device__ __forceinline__ DualT<S, N> Acos(const DualT<S, N> &x) {
    const S s = sqrt(fmax(S(0), S(1) - x.v * x.v));
    return dchain<S, N>(acos(x.v), s > S(0) ? S(-1) / s : S(0), x);
}
template <typename S, int N>
__device__ __forceinline__ DualT<S, N> Atan2(const DualT<S, N> &y, const DualT<S, N> &x) {
    DualT<S, N> r;
    r.v = atan2(y.v, x.v);
    const S q = x.v * x.v + y.v * y.v;
    const S iq = q > S(0) ? S(1) / q : S(0);
#pragma unroll
    for (int k = 0; k < N; ++k) r.d[k] = (x.v * y.d[k] - y.v * x.d[k]) * iq;
    return r;
}
template <typename S, int N>
__device__ __forceinline__ DualT<S, N> Exp(const DualT<S, N> &x) {
    const S e = exp(x.v);
    return dchain<S, N>(e, e, x);
}
template <typename S, int N>
__device__ __forceinline__ DualT<S, N> Fabs(const DualT<S, N> &x) { return dchain<S, N>(fabs(x.v), x.v < S(0) ? S(-1) : S(1), x); }
template <typename S, int N>
__device__ __forceinline__ DualT<S, N> Fmin(const DualT<S, N> &a, const DualT<S, N> &b) { return (b.v < a.v) ? b : a; }
template <typename S, int N>
__device__ __forceinline__ DualT<S, N> Fmax(const DualT<S, N> &a, const DualT<S, N> &b) { return (b.v > a.v) ? b : a; }
template <typename S, int N>
__device__ __forceinline__ void SinCos(const DualT<S, N> &x, DualT<S, N> *s, DualT<S, N> *c) {
    S sv, cv;
    dsincos(x.v, &sv, &cv);
    *s = dchain<S, N>(sv, cv, x);
    *c = dchain<S, N>(cv, -sv, x);
}
template <typename S, int N>
__device__ __forceinline__ void SinCosPi(const DualT<S, N> &x, DualT<S, N> *s, DualT<S, N> *c) {
    S sv, cv;
    dsincospi(x.v, &sv, &cv);
    *s = dchain<S, N>(sv, S(M_PI) * cv, x);
    *c = dchain<S, N>(cv, -S(M_PI) * sv, x);
}
template <typename S, int N>
__device__ __forceinline__ double to_double(const DualT<S, N> &x) { return (double)x.v; }
template <typename S, int N>
__device__ __forceinline__ float to_float(const DualT<S, N> &x) { return (float)x.v; }

}  // namespace creep
