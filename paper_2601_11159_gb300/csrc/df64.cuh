// Double-float arithmetic for the FP64-class vector mode on the FP32 pipes.
//
// A df64 is the unevaluated sum hi + lo of two FP32 numbers with |lo| <= ulp(hi)/2, about
// 48 significant bits (relative rounding about 2^-48). Sums use Knuth's error-free TwoSum,
// products Dekker's exact product through a fused multiply-add; both renormalise with
// the fast two-sum. Written from the published definitions (Knuth, TAOCP vol. 2, 4.2.2;
// Dekker 1971), not from any library. GB300 runs FP64 at a small fraction of its FP32
// rate, so an element operation in df64 (about 10-20 FP32 operations) costs less than one
// in FP64 when the kernel is arithmetic-bound; storage is 8 bytes, as for FP64.
#pragma once

#include <cuda_runtime.h>

namespace rd {

struct df64 {
    float hi, lo;
    df64() = default;
    __host__ __device__ explicit df64(double x) : hi((float)x), lo((float)(x - (double)(float)x)) {}
    __host__ __device__ explicit df64(float x) : hi(x), lo(0.f) {}
    __host__ __device__ explicit df64(int x) : hi((float)x), lo(0.f) {}
    __host__ __device__ df64(float h, float l, int /*raw*/) : hi(h), lo(l) {}
    __host__ __device__ explicit operator double() const { return (double)hi + (double)lo; }
    __host__ __device__ explicit operator float() const { return hi + lo; }
};

// s + e = a + b exactly (no condition on the magnitudes).
__device__ __forceinline__ df64 df_two_sum(float a, float b)
{
    const float s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return df64(s, e, 0);
}

// s + e = a + b exactly when |a| >= |b| (or a = 0).
__device__ __forceinline__ df64 df_fast_two_sum(float a, float b)
{
    const float s = __fadd_rn(a, b);
    return df64(s, __fsub_rn(b, __fsub_rn(s, a)), 0);
}

// Sum with one error-free transformation of the high parts (Dekker's add): the error is
// at most about 2^-48 (|a| + |b|), the backward-stable bound FP64 arithmetic also has,
// for half the operations of the version that also captures the low parts' rounding.
__device__ __forceinline__ df64 operator+(df64 a, df64 b)
{
    const df64 s = df_two_sum(a.hi, b.hi);
    return df_fast_two_sum(s.hi, __fadd_rn(__fadd_rn(a.lo, b.lo), s.lo));
}

__device__ __forceinline__ df64 operator-(df64 a) { return df64(-a.hi, -a.lo, 0); }
__device__ __forceinline__ df64 operator-(df64 a, df64 b) { return a + (-b); }

__device__ __forceinline__ df64 operator*(df64 a, df64 b)
{
    const float p = __fmul_rn(a.hi, b.hi);
    float e = __fmaf_rn(a.hi, b.hi, -p);  // exact low part of a.hi * b.hi
    e = __fmaf_rn(a.hi, b.lo, e);
    e = __fmaf_rn(a.lo, b.hi, e);
    return df_fast_two_sum(p, e);
}

__device__ __forceinline__ df64& operator+=(df64& a, df64 b)
{
    a = a + b;
    return a;
}

__device__ __forceinline__ df64& operator-=(df64& a, df64 b)
{
    a = a - b;
    return a;
}

// Accumulation of gathered terms into a running sum (the gather loops of the SpMM). For
// float and double a plain multiply-add. For df64 the leading parts go through TwoSum and the
// trailing parts are summed in FP32 without renormalising after every term (about 11 FP32
// operations per weighted term instead of 17); acc_finish renormalises once per row.
template <typename T>
__device__ __forceinline__ void acc_mul_add(T& acc, T w, T x)
{
    acc += w * x;
}
template <typename T>
__device__ __forceinline__ void acc_add(T& acc, T x)
{
    acc += x;
}
template <typename T>
__device__ __forceinline__ void acc_finish(T&)
{
}
template <>
__device__ __forceinline__ void acc_mul_add<df64>(df64& acc, df64 w, df64 x)
{
    const float p = __fmul_rn(w.hi, x.hi);
    float e = __fmaf_rn(w.hi, x.hi, -p);  // exact low part of w.hi * x.hi
    e = __fmaf_rn(w.hi, x.lo, e);
    e = __fmaf_rn(w.lo, x.hi, e);
    const df64 s = df_two_sum(acc.hi, p);
    acc.hi = s.hi;
    acc.lo = __fadd_rn(acc.lo, __fadd_rn(s.lo, e));
}
template <>
__device__ __forceinline__ void acc_add<df64>(df64& acc, df64 x)
{
    const df64 s = df_two_sum(acc.hi, x.hi);
    acc.hi = s.hi;
    acc.lo = __fadd_rn(acc.lo, __fadd_rn(s.lo, x.lo));
}
// An FP32 edge weight (positive and finite) in FP64, exactly, by moving its bits: the conversion
// instruction runs on the FP64 unit, which bounds the FP64 kernels (weighted 500^2 road grid, 16
// columns: 1.95M FP64 warp instructions a step with it and 1.70M without, 135 -> 119 us). Denormals
// are scaled up in FP32 first (exact).
__device__ __forceinline__ double widen(float w)
{
    const bool tiny = w < 1.17549435e-38f;
    const unsigned b = __float_as_uint(tiny ? __fmul_rn(w, 16777216.0f) : w);
    return __hiloint2double((int)((b >> 3) + (tiny ? 0x38000000u - (24u << 20) : 0x38000000u)), (int)(b << 29));
}

// The same with an FP32 edge weight (a df64 with a zero low part): the product's w.lo x.hi
// term, an exact zero, is not formed.
template <typename T>
__device__ __forceinline__ void acc_mul_add_w(T& acc, float w, T x)
{
    acc_mul_add(acc, T(w), x);
}
template <>
__device__ __forceinline__ void acc_mul_add_w<double>(double& acc, float w, double x)
{
    acc = fma(widen(w), x, acc);
}
template <>
__device__ __forceinline__ void acc_mul_add_w<df64>(df64& acc, float w, df64 x)
{
    const float p = __fmul_rn(w, x.hi);
    float e = __fmaf_rn(w, x.hi, -p);  // exact low part of w * x.hi
    e = __fmaf_rn(w, x.lo, e);
    const df64 s = df_two_sum(acc.hi, p);
    acc.hi = s.hi;
    acc.lo = __fadd_rn(acc.lo, __fadd_rn(s.lo, e));
}
template <>
__device__ __forceinline__ void acc_finish<df64>(df64& acc)
{
    acc = df_two_sum(acc.hi, acc.lo);
}

// Two double-float numbers, their leading and their trailing parts each in a register pair, for the
// packed FP32 instructions: the operations above, with the same roundings bit for bit, on two columns
// in one issue slot. A difference is a multiply-add by -1; `na` is -a.
struct df64x2 {
    float2 hi, lo;
};

__device__ __forceinline__ df64x2 df_pack(df64 a, df64 b)
{
    return df64x2{make_float2(a.hi, b.hi), make_float2(a.lo, b.lo)};
}
__device__ __forceinline__ void df_unpack(const df64x2& v, df64& a, df64& b)
{
    a = df64(v.hi.x, v.lo.x, 0);
    b = df64(v.hi.y, v.lo.y, 0);
}

__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }

// s + e = a + b exactly, as df_two_sum.
__device__ __forceinline__ df64x2 df_two_sum(float2 a, float2 b)
{
    const float2 s = __fadd2_rn(a, b);
    const float2 bb = sub2(s, a);
    return df64x2{s, __fadd2_rn(sub2(a, sub2(s, bb)), sub2(b, bb))};
}

__device__ __forceinline__ df64x2 operator+(const df64x2& a, const df64x2& b)
{
    const df64x2 t = df_two_sum(a.hi, b.hi);
    const float2 l = __fadd2_rn(__fadd2_rn(a.lo, b.lo), t.lo);
    const float2 s = __fadd2_rn(t.hi, l);
    return df64x2{s, sub2(l, sub2(s, t.hi))};
}

__device__ __forceinline__ df64x2 df_neg(const df64x2& a)
{
    const float2 m = make_float2(-1.f, -1.f);
    return df64x2{__fmul2_rn(a.hi, m), __fmul2_rn(a.lo, m)};
}

// a b; minus its low part is carried, so that nothing is negated on the way.
__device__ __forceinline__ df64x2 df_mul(const df64x2& a, const df64x2& na, const df64x2& b)
{
    const float2 p = __fmul2_rn(a.hi, b.hi);
    float2 m = __ffma2_rn(na.hi, b.hi, p);  // minus the exact low part of a.hi * b.hi
    m = __ffma2_rn(na.hi, b.lo, m);
    m = __ffma2_rn(na.lo, b.hi, m);
    const float2 s = sub2(p, m);
    return df64x2{s, sub2(sub2(p, s), m)};
}

// A row's W = invd acc - bt qp, and its terms d W q, d W^2 and d W added to the sums: the scalar
// expressions, each product normalised, two columns at a time. Left unnormalised where they go into a
// sum or another product, the products are an eighth of the operations cheaper and their error up to
// twice as large (d W q of 20,000 random rows: 6.0 for 3.1 units of 2^-48 at worst), which no caller
// asks for.
__device__ __forceinline__ df64x2 df_row(df64 invd, const df64x2& acc, const df64x2& bt, const df64x2& qp)
{
    return df_mul(df_pack(invd, invd), df_pack(-invd, -invd), acc) + df_mul(df_neg(bt), bt, qp);
}
__device__ __forceinline__ void df_row_sums(df64 du, const df64x2& w, const df64x2& qc, df64x2& sa, df64x2& sb,
                                            df64x2& sc)
{
    const df64x2 dw = df_mul(df_pack(du, du), df_pack(-du, -du), w), ndw = df_neg(dw);
    sa = sa + df_mul(dw, ndw, qc);
    sb = sb + df_mul(dw, ndw, w);
    sc = sc + dw;
}

// acc_mul_add_w and acc_add on two columns.
__device__ __forceinline__ void acc_mul_add_w(df64 (&acc)[2], float w, const df64x2& x)
{
    const float2 w2 = make_float2(w, w), nw = make_float2(-w, -w);
    df64x2 a = df_pack(acc[0], acc[1]);
    const float2 p = __fmul2_rn(w2, x.hi);
    float2 m = __ffma2_rn(nw, x.hi, p);
    m = __ffma2_rn(nw, x.lo, m);
    const df64x2 s = df_two_sum(a.hi, p);
    a = df64x2{s.hi, __fadd2_rn(a.lo, sub2(s.lo, m))};
    df_unpack(a, acc[0], acc[1]);
}
__device__ __forceinline__ void acc_add(df64 (&acc)[2], const df64x2& x)
{
    df64x2 a = df_pack(acc[0], acc[1]);
    const df64x2 s = df_two_sum(a.hi, x.hi);
    a = df64x2{s.hi, __fadd2_rn(a.lo, __fadd2_rn(s.lo, x.lo))};
    df_unpack(a, acc[0], acc[1]);
}

// Warp shuffles of element values (both halves move together).
__device__ __forceinline__ float shfl_xor_t(unsigned mask, float v, int off, int width = 32)
{
    return __shfl_xor_sync(mask, v, off, width);
}
__device__ __forceinline__ double shfl_xor_t(unsigned mask, double v, int off, int width = 32)
{
    return __shfl_xor_sync(mask, v, off, width);
}
__device__ __forceinline__ df64 shfl_xor_t(unsigned mask, df64 v, int off, int width = 32)
{
    return df64(__shfl_xor_sync(mask, v.hi, off, width), __shfl_xor_sync(mask, v.lo, off, width), 0);
}
__device__ __forceinline__ float shfl_t(unsigned mask, float v, int src, int width = 32)
{
    return __shfl_sync(mask, v, src, width);
}
__device__ __forceinline__ double shfl_t(unsigned mask, double v, int src, int width = 32)
{
    return __shfl_sync(mask, v, src, width);
}
__device__ __forceinline__ df64 shfl_t(unsigned mask, df64 v, int src, int width = 32)
{
    return df64(__shfl_sync(mask, v.hi, src, width), __shfl_sync(mask, v.lo, src, width), 0);
}

// Conversions of element values to double (identity for float and double).
__device__ __forceinline__ double to_double(float v) { return (double)v; }
__device__ __forceinline__ double to_double(double v) { return v; }
__device__ __forceinline__ double to_double(df64 v) { return (double)v; }

}  // namespace rd
