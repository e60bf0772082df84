// lbfd_dual.cuh -- forward-mode (tangent-linear) numbers for the step kernel.
//
// Dual<T, N> carries a value and N directional derivatives.  Every
// arithmetic operation of the step propagates the derivatives by the chain
// rule, so the unchanged step kernel instantiated with this type computes,
// alongside the state, its exact derivative with respect to N parameters
// (the derivative of the discrete scheme, branch decisions such as the
// WENO upwind side or max(Y, 0) taken on the values).
#pragma once
#include <cmath>

#include "lbfd_f2.cuh"

namespace lbfd {

// a constant: c * x, c + x cost one operation per derivative of x, where a
// Dual factor without derivatives would cost two
template <typename T>
struct Cst {
    T v;
    constexpr __host__ __device__ explicit Cst(double x) : v(T(x)) {}
};

// Derivative vectors: r = s x, r = s x + t y, r += x, ... one operation per
// derivative, or per two of them with the packed FP32 instructions.
template <typename T, int N>
struct Vec {
    static __host__ __device__ __forceinline__ void scale(T* r, T s, const T* x)
    {
#pragma unroll
        for (int k = 0; k < N; ++k) r[k] = s * x[k];
    }
    static __host__ __device__ __forceinline__ void comb(T* r, T s, const T* x, T t, const T* y)  // s x + t y
    {
#pragma unroll
        for (int k = 0; k < N; ++k) r[k] = s * x[k] + t * y[k];
    }
    static __host__ __device__ __forceinline__ void axpy(T* r, T s, const T* x)  // r += s x
    {
#pragma unroll
        for (int k = 0; k < N; ++k) r[k] += s * x[k];
    }
    static __host__ __device__ __forceinline__ void add(T* r, const T* x)
    {
#pragma unroll
        for (int k = 0; k < N; ++k) r[k] += x[k];
    }
    static __host__ __device__ __forceinline__ void sub(T* r, const T* x)
    {
#pragma unroll
        for (int k = 0; k < N; ++k) r[k] -= x[k];
    }
};
#ifdef __CUDA_ARCH__
template <>
struct Vec<float, 4> {
    static __device__ __forceinline__ float2 lo(const float* x) { return make_float2(x[0], x[1]); }
    static __device__ __forceinline__ float2 hi(const float* x) { return make_float2(x[2], x[3]); }
    static __device__ __forceinline__ float2 two(float s) { return make_float2(s, s); }
    static __device__ __forceinline__ void put(float* r, float2 a, float2 b)
    {
        r[0] = a.x;
        r[1] = a.y;
        r[2] = b.x;
        r[3] = b.y;
    }
    static __device__ __forceinline__ void scale(float* r, float s, const float* x)
    {
        put(r, __fmul2_rn(two(s), lo(x)), __fmul2_rn(two(s), hi(x)));
    }
    static __device__ __forceinline__ void comb(float* r, float s, const float* x, float t, const float* y)
    {
        put(r, __ffma2_rn(two(s), lo(x), __fmul2_rn(two(t), lo(y))),
            __ffma2_rn(two(s), hi(x), __fmul2_rn(two(t), hi(y))));
    }
    static __device__ __forceinline__ void axpy(float* r, float s, const float* x)
    {
        put(r, __ffma2_rn(two(s), lo(x), lo(r)), __ffma2_rn(two(s), hi(x), hi(r)));
    }
    static __device__ __forceinline__ void add(float* r, const float* x)
    {
        put(r, __fadd2_rn(lo(r), lo(x)), __fadd2_rn(hi(r), hi(x)));
    }
    static __device__ __forceinline__ void sub(float* r, const float* x)
    {
        put(r, f2sub(lo(r), lo(x)), f2sub(hi(r), hi(x)));
    }
};
#endif

template <typename T, int N>
struct Dual {
    T v;
    T d[N];

    __host__ __device__ Dual() {}
    // constants and converted plain values carry no derivative
    __host__ __device__ Dual(double x) : v(T(x))
    {
#pragma unroll
        for (int k = 0; k < N; ++k) d[k] = T(0);
    }
    __host__ __device__ Dual(int x) : Dual(double(x)) {}
    __host__ __device__ Dual(const Cst<T>& x) : Dual(double(x.v)) {}

    __host__ __device__ Dual& operator+=(const Dual& b)
    {
        v += b.v;
        Vec<T, N>::add(d, b.d);
        return *this;
    }
    __host__ __device__ Dual& operator-=(const Dual& b)
    {
        v -= b.v;
        Vec<T, N>::sub(d, b.d);
        return *this;
    }
    __host__ __device__ Dual& operator*=(const Dual& b)
    {
        Vec<T, N>::comb(d, b.v, d, v, b.d);
        v *= b.v;
        return *this;
    }
};

template <typename T, int N>
__host__ __device__ inline Dual<T, N> operator+(Dual<T, N> a, const Dual<T, N>& b) { return a += b; }
template <typename T, int N>
__host__ __device__ inline Dual<T, N> operator-(Dual<T, N> a, const Dual<T, N>& b) { return a -= b; }
template <typename T, int N>
__host__ __device__ inline Dual<T, N> operator*(Dual<T, N> a, const Dual<T, N>& b) { return a *= b; }
template <typename T, int N>
__host__ __device__ inline Dual<T, N> operator-(const Dual<T, N>& a)
{
    Dual<T, N> r;
    r.v = -a.v;
#pragma unroll
    for (int k = 0; k < N; ++k) r.d[k] = -a.d[k];
    return r;
}
template <typename T, int N>
__host__ __device__ inline Dual<T, N> operator/(const Dual<T, N>& a, const Dual<T, N>& b)
{
    Dual<T, N> r;
    const T inv = T(1) / b.v;
    r.v = a.v * inv;
    // (a' - r b') / b: the terms cancel before the last rounding
#pragma unroll
    for (int k = 0; k < N; ++k) r.d[k] = a.d[k];
    Vec<T, N>::axpy(r.d, -r.v, b.d);
    Vec<T, N>::scale(r.d, inv, r.d);
    return r;
}
template <typename T, int N>
__host__ __device__ inline Dual<T, N>& operator/=(Dual<T, N>& a, const Dual<T, N>& b)
{
    a = a / b;
    return a;
}

template <typename T, int N>
struct ConstOf<Dual<T, N>> {
    using type = Cst<T>;
};
template <typename T, int N>
__host__ __device__ inline Dual<T, N> operator*(const Cst<T>& c, Dual<T, N> a)
{
    a.v *= c.v;
    Vec<T, N>::scale(a.d, c.v, a.d);
    return a;
}
template <typename T, int N>
__host__ __device__ inline Dual<T, N> operator*(const Dual<T, N>& a, const Cst<T>& c) { return c * a; }
template <typename T, int N>
__host__ __device__ inline Dual<T, N> operator+(const Cst<T>& c, Dual<T, N> a)
{
    a.v += c.v;
    return a;
}
template <typename T, int N>
__host__ __device__ inline Dual<T, N> operator+(const Dual<T, N>& a, const Cst<T>& c) { return c + a; }
template <typename T, int N>
__host__ __device__ inline Dual<T, N> operator-(Dual<T, N> a, const Cst<T>& c)
{
    a.v -= c.v;
    return a;
}
template <typename T, int N>
__host__ __device__ inline Dual<T, N> operator-(const Cst<T>& c, const Dual<T, N>& a) { return c + (-a); }
template <typename T>
__host__ __device__ inline Cst<T> operator*(const Cst<T>& a, const Cst<T>& b)
{
    return Cst<T>((double)(a.v * b.v));
}

// comparisons act on the values
template <typename T, int N>
__host__ __device__ inline bool operator<(const Dual<T, N>& a, const Dual<T, N>& b) { return a.v < b.v; }
template <typename T, int N>
__host__ __device__ inline bool operator>(const Dual<T, N>& a, const Dual<T, N>& b) { return a.v > b.v; }
template <typename T, int N>
__host__ __device__ inline bool operator<=(const Dual<T, N>& a, const Dual<T, N>& b) { return a.v <= b.v; }
template <typename T, int N>
__host__ __device__ inline bool operator>=(const Dual<T, N>& a, const Dual<T, N>& b) { return a.v >= b.v; }

template <typename T, int N>
__host__ __device__ inline Dual<T, N> exp(const Dual<T, N>& a)
{
    Dual<T, N> r;
    if constexpr (sizeof(T) == 4) r.v = expf(a.v);
    else r.v = ::exp(a.v);
#pragma unroll
    for (int k = 0; k < N; ++k) r.d[k] = r.v * a.d[k];
    return r;
}

template <typename T, int N>
__device__ __forceinline__ Dual<T, N> fdiv(const Dual<T, N>& a, const Dual<T, N>& b) { return a / b; }

// value part of a stored number
__host__ __device__ inline double val(double x) { return x; }
__host__ __device__ inline double val(float x) { return (double)x; }
template <typename T, int N>
__host__ __device__ inline double val(const Dual<T, N>& x) { return (double)x.v; }

// FP64 copy of an FP32 dual number and back (round to nearest)
template <int N>
__host__ __device__ inline Dual<double, N> widen(const Dual<float, N>& a)
{
    Dual<double, N> r;
    r.v = a.v;
#pragma unroll
    for (int k = 0; k < N; ++k) r.d[k] = a.d[k];
    return r;
}
template <int N>
__host__ __device__ inline Dual<float, N> narrow(const Dual<double, N>& a)
{
    Dual<float, N> r;
    r.v = (float)a.v;
#pragma unroll
    for (int k = 0; k < N; ++k) r.d[k] = (float)a.d[k];
    return r;
}

// tangents with respect to (ln A, Ta, T_wall, u_in): FP64, and FP32 (the
// mixed tangent form: FP32 state and arithmetic, FP64 Arrhenius above
// T_fp64 and FP64 accumulation of the objectives)
constexpr int NTAN = 4;
using Tan = Dual<double, NTAN>;
using Tanf = Dual<float, NTAN>;

}  // namespace lbfd
