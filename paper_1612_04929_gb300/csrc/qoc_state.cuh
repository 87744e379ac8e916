// Arithmetic helpers of the state-mode kernels (k_state.cu, k_state_cluster.cu).
#pragma once
#include "qoc_device.cuh"
#include "qoc_internal.h"

namespace qoc {

// ---- pair (hi + lo) helpers of the FP32 form ----
__device__ __forceinline__ void st_norm(float& hi, float& lo) {
    const float s = hi + lo;
    lo = lo - (s - hi);
    hi = s;
}
// (hi, lo) += u (b_hi + b_lo), u = (u_hi + u_lo) a pair of the control amplitude
__device__ __forceinline__ void st_pair_fma(float& hi, float& lo, float2 u, float bh, float bl) {
    const float p = u.x * bh;
    float e = fmaf(u.x, bh, -p);
    e = fmaf(u.x, bl, e);
    e = fmaf(u.y, bh, e);
    float s, r;
    two_sum(hi, p, s, r);
    hi = s;
    lo += r + e;
}
// a / i for a pair a
__device__ __forceinline__ void st_div(float& hi, float& lo, float fi) {
    const float q = hi / fi;
    const float r = fmaf(-q, fi, hi);
    lo = (r + lo) / fi;
    hi = q;
    st_norm(hi, lo);
}
__device__ __forceinline__ void st_add(float4& a, const float4 b) {   // pair complex a += b
    float s, r;
    two_sum(a.x, b.x, s, r);
    a.x = s;
    a.z += r + b.z;
    two_sum(a.y, b.y, s, r);
    a.y = s;
    a.w += r + b.w;
    st_norm(a.x, a.z);
    st_norm(a.y, a.w);
}
__device__ __forceinline__ unsigned st_maxbits(const float4 v) { return __float_as_uint(fmaxf(fabsf(v.x), fabsf(v.y))); }
// carried-block helpers: FP32 pairs (float4) and FP64 (double2)
template <typename K> __device__ __forceinline__ K kzero_k();
template <> __device__ __forceinline__ float4 kzero_k<float4>() { return make_float4(0.f, 0.f, 0.f, 0.f); }
template <> __device__ __forceinline__ double2 kzero_k<double2>() { return make_double2(0.0, 0.0); }
__device__ __forceinline__ void st_kadd(float4& a, const float4 b) { st_add(a, b); }
__device__ __forceinline__ void st_kadd(float4& a, const float2 b) { st_add(a, make_float4(b.x, b.y, 0.f, 0.f)); }
__device__ __forceinline__ void st_kadd(double2& a, const double2 b) {
    a.x += b.x;
    a.y += b.y;
}
__device__ __forceinline__ void st_kdiv(float4& a, int i) {
    if (i == 1) return;
    st_div(a.x, a.z, (float)i);
    st_div(a.y, a.w, (float)i);
}
__device__ __forceinline__ void st_kdiv(double2& a, int i) {
    a.x /= i;
    a.y /= i;
}
__device__ __forceinline__ float2 st_round(const float4 a) { return make_float2(a.x + a.z, a.y + a.w); }
__device__ __forceinline__ double2 st_round(const double2 a) { return a; }
// pair times pair: (hi + lo)(bh + bl), the product's rounding error and the cross terms in lo
__device__ __forceinline__ void st_mul(float& hi, float& lo, float bh, float bl) {
    const float pr = hi * bh;
    float e = fmaf(hi, bh, -pr);
    e = fmaf(hi, bl, e);
    e = fmaf(lo, bh, e);
    hi = pr;
    lo = e;
    st_norm(hi, lo);
}
__device__ __forceinline__ void st_kscale(float4& a, double s) {
    const float sh = (float)s, sl = (float)(s - (double)sh);
    st_mul(a.x, a.z, sh, sl);
    st_mul(a.y, a.w, sh, sl);
}
__device__ __forceinline__ void st_kscale(double2& a, double s) {
    a.x *= s;
    a.y *= s;
}
// a <- (i s) a
__device__ __forceinline__ void st_kmul_i(float4& a, double s) {
    st_kscale(a, s);
    a = make_float4(-a.y, a.x, -a.w, a.z);
}
__device__ __forceinline__ void st_kmul_i(double2& a, double s) { a = make_double2(-s * a.y, s * a.x); }
__device__ __forceinline__ void st_ktwice(float4& a) { a = make_float4(2.f * a.x, 2.f * a.y, 2.f * a.z, 2.f * a.w); }
__device__ __forceinline__ void st_ktwice(double2& a) { a = make_double2(2.0 * a.x, 2.0 * a.y); }
__device__ __forceinline__ void st_kneg(float4& a) { a = make_float4(-a.x, -a.y, -a.z, -a.w); }
__device__ __forceinline__ void st_kneg(double2& a) { a = make_double2(-a.x, -a.y); }
// a <- i^r a (r = 0 .. 3)
__device__ __forceinline__ void st_krot(float4& a, int r) {
    if (r == 1) a = make_float4(-a.y, a.x, -a.w, a.z);
    else if (r == 2) a = make_float4(-a.x, -a.y, -a.z, -a.w);
    else if (r == 3) a = make_float4(a.y, -a.x, a.w, -a.z);
}
__device__ __forceinline__ void st_krot(double2& a, int r) {
    if (r == 1) a = make_double2(-a.y, a.x);
    else if (r == 2) a = make_double2(-a.x, -a.y);
    else if (r == 3) a = make_double2(a.y, -a.x);
}

// Matrix element of X as read by the chain: FP32 grid-split pairs (float4: re and im grid parts on
// 2^(ex - 12), then the remainders; written so by k_state_x32); FP64 plain.
template <typename R> struct XElem;
template <> struct XElem<float> { using T = float4; };
template <> struct XElem<double> { using T = double2; };

}  // namespace qoc
