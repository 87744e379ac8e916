// One batched product of a level of the wave's binary tree (k_tree.cu), and what it writes.
#pragma once
#include "qoc_device.cuh"
#include "qoc_internal.h"

namespace qoc {

__device__ __forceinline__ float4 tree_split(const float4 v, float m) {
    float4 o;
    grid_split(v.x, v.z, m, o.x, o.z);
    grid_split(v.y, v.w, m, o.y, o.w);
    return o;
}

// One batched product of a level.  Item (e, i): A = a + e ae + i ai (matrices d x d), B = b + e be + i bi
// (d x cols), out likewise.  A or B may be the slice propagators (float2, rounded; split here).
struct TreeMm {
    int d, cols, E, count, tiles_r, tiles_c;   // tiles: set with the launch's shape
    const void* a;
    size_t ae, ai;
    const void* b;
    size_t be, bi;
    float4* out;              // grid-split with its column's mo
    size_t oe, oi;
    float4* copy;             // optional second carried output (the block handed to the next wave)
    size_t ce;
    float2* round;            // optional rounded output: states, or costates scaled by coef
    size_t re, ri;
    const float4* coef;       // per member and column (re, im hi; re, im lo), or nullptr
    const float* mo;          // grid (magic) of every output column; nullptr: of the propagators' exponent
    const DevParams* prm;     // exponent eu of the propagators (and of out without mo)
};

// element o (column c) of item (e, i): the carried output, its copy and the rounded (scaled) value
__device__ __forceinline__ void tree_store(const TreeMm& t, int e, int i, size_t o, int c, const float4 v, float mo) {
    const float4 g = tree_split(v, mo);
    t.out[e * t.oe + i * t.oi + o] = g;
    if (t.copy) t.copy[e * t.ce + o] = g;
    if (!t.round) return;
    float2 r = make_float2(v.x + v.z, v.y + v.w);
    if (t.coef) {
        const float4 q = t.coef[(size_t)e * t.cols + c];
        float xh = 0.f, xl = 0.f, yh = 0.f, yl = 0.f;
        pair_fma(xh, xl, make_float2(q.x, q.z), v.x, v.z);
        pair_fma(xh, xl, make_float2(-q.y, -q.w), v.y, v.w);
        pair_fma(yh, yl, make_float2(q.x, q.z), v.y, v.w);
        pair_fma(yh, yl, make_float2(q.y, q.w), v.x, v.z);
        r = make_float2(xh + xl, yh + yl);
    }
    t.round[e * t.re + i * t.ri + o] = r;
}

}  // namespace qoc
