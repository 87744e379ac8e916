// Both recursions of a full-unitary evaluation as batched products over a binary tree of the wave.
//
// When every column is propagated (S = d) and the cost acts on the final state alone, the forward
// recursion Psi_j = U_j Psi_{j-1} (Eqs. 2, 4) and the costate G_{j-1} = U_j^dag G_j (Appendix A) are
// d x d products, one a slice each.  The segmented sweeps (k_serial.cu) run them as chains of dependent
// steps, a CTA per column panel and segment, in which every CTA reads every U_j for a few columns: at
// d = 128 a step took 30 us and a pass ran at 12 TFLOP/s executed.  Over the binary tree of a wave's
// slices they become batched products of the same count:
//   up      P(l, i) = P(l-1, 2i+1) P(l-1, 2i), the product of the slices of node i at level l
//   forward state at the start of a right child = P(left child) x the state at its parent's start
//   costate costate at the end of a left child = P(right child)^dag x the costate at its parent's end
// and the root takes the state (costate) across the whole wave: log2(W) launches a pass instead of a
// scan and chains, each over all nodes of a level.  Nodes, states and costates are carried grid-split
// (qoc_device.cuh; the U_j are unitary to the truncation, so products of them share the exponent eu,
// and a block's columns keep the norms of Psi_0 or Psi_T, each with a grid of its own), every product a split product (k_big_mm's
// tiles, qoc_gemm.cuh).  The costate is propagated from Psi_T itself and scaled by the terminal
// coefficient -2 a_fid O_N w_s / (E W) where G_j is written.
// Measured on GB300 (evaluation): d = 128, N = 500 11.7 -> 8.1 ms; d = 64,
// N = 2000 7.05 -> 5.85 ms; d = 256, N = 2000 (BF16_SPLIT) 153 -> 142 ms; where it pays: tree_applies.
//
// BF16_SPLIT with 128 <= d <= 384 runs the same products on the tensor cores (k_oz.cu: both operands cut
// into six seven-bit slices, accurate as the split product; the epilogue writes what k_tree_mm writes):
// 7.6 -> 2.7 us a product of d = 256 with its slicing, the evaluation above 124 -> 94.6 ms, error against
// 64 bits unchanged.  All levels, though a single product is no faster there (62 us either way).
#include <algorithm>
#include <cmath>

#include "qoc_device.cuh"
#include "qoc_gemm.cuh"
#include "qoc_internal.h"
#include "qoc_tree.cuh"

namespace qoc {

namespace {

// acc += conj(A) B for A given transposed (a product with A^dag)
template <int MT>
struct MacSplitConj {
    float acc[MT][MT][4] = {};
    __device__ __forceinline__ void run(const float4 (&a)[MT], const float4 (&b)[MT], int) {
#pragma unroll
        for (int y = 0; y < MT; ++y) {
            const float2 bf = make_float2(b[y].x + b[y].z, b[y].y + b[y].w);
#pragma unroll
            for (int x = 0; x < MT; ++x) {
                float* c = acc[x][y];
                c[0] = fmaf(a[x].x, b[y].x, c[0]);
                c[0] = fmaf(a[x].y, b[y].y, c[0]);
                c[1] = fmaf(a[x].x, b[y].y, c[1]);
                c[1] = fmaf(-a[x].y, b[y].x, c[1]);
                c[2] = fmaf(a[x].x, b[y].z, c[2]);
                c[2] = fmaf(a[x].y, b[y].w, c[2]);
                c[2] = fmaf(a[x].z, bf.x, c[2]);
                c[2] = fmaf(a[x].w, bf.y, c[2]);
                c[3] = fmaf(a[x].x, b[y].w, c[3]);
                c[3] = fmaf(-a[x].y, b[y].z, c[3]);
                c[3] = fmaf(a[x].z, bf.y, c[3]);
                c[3] = fmaf(-a[x].w, bf.x, c[3]);
            }
        }
    }
};

// AK: 0 A carried, 1 A rounded propagators, 2 A carried and taken as A^dag; BL: B rounded propagators
template <int AK, bool BL, class Sh>
__global__ void __launch_bounds__(Sh::NT, Sh::MB) k_tree_mm(TreeMm t) {
    constexpr int MT = Sh::MT, G = Sh::G;
    extern __shared__ __align__(16) unsigned char smraw[];
    const int tiles = t.tiles_r * t.tiles_c;
    const int item = blockIdx.x / tiles, tile = blockIdx.x - item * tiles;
    const int e = item / t.count, i = item - e * t.count;
    const GemmPos<Sh> p(tile, t.tiles_c, t.d);
    const int d = t.d, cols = t.cols;
    const float mu = grid_magic(t.prm->eu);
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    const float4* A4 = static_cast<const float4*>(t.a) + e * t.ae + i * t.ai;
    const float2* A2 = static_cast<const float2*>(t.a) + e * t.ae + i * t.ai;
    const float4* B4 = static_cast<const float4*>(t.b) + e * t.be + i * t.bi;
    const float2* B2 = static_cast<const float2*>(t.b) + e * t.be + i * t.bi;
    auto la = [&](int r, int k, float4* dst) {
        if (r >= d || k >= d) {
            *dst = zero;
        } else if constexpr (AK == 1) {
            const float2 v = A2[(size_t)r * d + k];
            *dst = tree_split(make_float4(v.x, v.y, 0.f, 0.f), mu);
        } else {
            cp_async16(dst, AK == 2 ? &A4[(size_t)k * d + r] : &A4[(size_t)r * d + k]);
        }
    };
    auto lb = [&](int k, int c, float4* dst) {
        if (k >= d || c >= cols) {
            *dst = zero;
        } else if constexpr (BL) {
            const float2 v = B2[(size_t)k * cols + c];
            *dst = tree_split(make_float4(v.x, v.y, 0.f, 0.f), mu);
        } else {
            cp_async16(dst, &B4[(size_t)k * cols + c]);
        }
    };
    std::conditional_t<AK == 2, MacSplitConj<MT>, MacSplit<MT>> mac;
    gemm_loop<float4, Sh, AK == 2>(smraw, p, d, la, lb, mac);
#pragma unroll
    for (int x = 0; x < MT; ++x)
#pragma unroll
        for (int y = 0; y < MT; ++y) {
            const int r = p.r0 + p.ty + G * x, c = p.c0 + p.tx + G * y;
            if (r >= d || c >= cols) continue;
            float4 v;
            two_sum(mac.acc[x][y][0], mac.acc[x][y][2], v.x, v.z);
            two_sum(mac.acc[x][y][1], mac.acc[x][y][3], v.y, v.w);
            const size_t o = (size_t)r * cols + c;
            tree_store(t, e, i, o, c, v, t.mo ? t.mo[c] : mu);
        }
}

// a node without a right child: its left child unchanged (the last node of a level)
__global__ void k_tree_tail(const void* src, size_t se, int leaf, float4* dst, size_t de, size_t dd, const DevParams* prm) {
    const int e = blockIdx.y;
    const float mu = grid_magic(prm->eu);
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < dd; i += (size_t)gridDim.x * blockDim.x) {
        if (leaf) {
            const float2 v = (static_cast<const float2*>(src) + e * se)[i];
            dst[e * de + i] = tree_split(make_float4(v.x, v.y, 0.f, 0.f), mu);
        } else {
            dst[e * de + i] = (static_cast<const float4*>(src) + e * se)[i];
        }
    }
}

// The block a pass starts from (pairs), split on its columns' grids, and its rounded (scaled) value
__global__ void k_tree_init(const float4* src, size_t se, float4* dst, size_t de, float2* rnd, size_t re,
                            const float4* coef, int cols, size_t n, const float* __restrict__ mo) {
    const int e = blockIdx.y;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const float4 v = src[e * se + i];
        dst[e * de + i] = tree_split(v, mo[i % cols]);
        float2 r = make_float2(v.x + v.z, v.y + v.w);
        if (coef) {
            const float4 q = coef[(size_t)e * cols + i % cols];
            float xh = 0.f, xl = 0.f, yh = 0.f, yl = 0.f;
            pair_fma(xh, xl, make_float2(q.x, q.z), v.x, v.z);
            pair_fma(xh, xl, make_float2(-q.y, -q.w), v.y, v.w);
            pair_fma(yh, yl, make_float2(q.x, q.z), v.y, v.w);
            pair_fma(yh, yl, make_float2(q.y, q.w), v.x, v.z);
            r = make_float2(xh + xl, yh + yl);
        }
        rnd[e * re + i] = r;
    }
}

// terminal coefficients -2 a_fid O_N w_s / (E W) per member and column, as pairs
__global__ void k_tree_coef(CostView<float> cv, int E, int cols, const double2* __restrict__ Ofin, float4* __restrict__ coef) {
    const int e = blockIdx.x;
    const double cf = -2.0 * cv.alpha[0] / E / cv.Wsum;
    const double2 o = Ofin[e];
    for (int s = threadIdx.x; s < cols; s += blockDim.x) {
        const double x = cf * cv.w[s] * o.x, y = cf * cv.w[s] * o.y;
        float4 q;
        q.x = (float)x;
        q.y = (float)y;
        q.z = (float)(x - (double)q.x);
        q.w = (float)(y - (double)q.y);
        coef[(size_t)e * cols + s] = q;
    }
}

int tree_ew_blocks(size_t n) { return (int)std::min<size_t>((n + 255) / 256, 64); }

template <int AK, bool BL, class Sh>
cudaError_t mm_tiles(TreeMm t, cudaStream_t st) {
    constexpr size_t smem = Sh::template smem<float4>();
    cudaError_t e = cudaFuncSetAttribute(k_tree_mm<AK, BL, Sh>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    t.tiles_r = Sh::tiles(t.d);
    t.tiles_c = Sh::tiles(t.cols);
    k_tree_mm<AK, BL, Sh><<<t.tiles_r * t.tiles_c * t.E * t.count, Sh::NT, smem, st>>>(t);
    return cudaGetLastError();
}

template <int AK, bool BL>
cudaError_t mm(const TreeArgs& a, const TreeMm& t, cudaStream_t st, int* launches) {
    if (a.oz) return oz_tree_product(*a.oz, t, AK, BL, a.prm, st, launches);
    ++*launches;
    if (gemm_split_small(t.d, (long)t.E * t.count, sm_count())) return mm_tiles<AK, BL, GemmSplitS>(t, st);
    return mm_tiles<AK, BL, GemmSplit>(t, st);
}

TreeMm base(const TreeArgs& a, int cols) {
    TreeMm t{};
    t.d = a.d;
    t.cols = cols;
    t.E = a.E;
    t.prm = a.prm;
    return t;
}

}  // namespace

int tree_levels(int wlen) {
    int l = 0;
    while ((1 << l) < wlen) ++l;
    return l;
}
// first node of level l >= 1 in a member's node array, for waves of at most W slices
static size_t level_offset(int W, int l) {
    size_t o = 0;
    for (int k = 1; k < l; ++k) o += ((size_t)W + (1 << k) - 1) >> k;
    return o;
}
size_t tree_nodes(int W) { return level_offset(W, tree_levels(W) + 1); }

// the matrices of level l from node i0 with a step of two nodes, as the operand of a level's products
static void node_operand(const TreeArgs& a, int l, int i0, bool dag, const void** p, size_t* e, size_t* i) {
    if (l == 0) {
        *p = a.U + (size_t)i0 * a.ustride + (dag ? a.ustride / 2 : 0);
        *e = (size_t)a.W * a.ustride;
        *i = 2 * (size_t)a.ustride;
    } else {
        const size_t dd = (size_t)a.d * a.d;
        *p = a.nodes + (level_offset(a.W, l) + i0) * dd;
        *e = tree_nodes(a.W) * dd;
        *i = 2 * dd;
    }
}

cudaError_t launch_tree_up(const TreeArgs& a, cudaStream_t st, int* launches) {
    const int L = tree_levels(a.wlen);
    const size_t dd = (size_t)a.d * a.d, ne = tree_nodes(a.W) * dd;
    for (int l = 1; l <= L; ++l) {
        const int below = (a.wlen + (1 << (l - 1)) - 1) >> (l - 1), pairs = below / 2;
        float4* lev = a.nodes + level_offset(a.W, l) * dd;
        cudaError_t err;
        if (pairs > 0) {
            TreeMm t = base(a, a.d);
            t.count = pairs;
            node_operand(a, l - 1, 1, false, &t.a, &t.ae, &t.ai);   // the later slices on the left
            node_operand(a, l - 1, 0, false, &t.b, &t.be, &t.bi);
            t.out = lev;
            t.oe = ne;
            t.oi = dd;
            if ((err = l == 1 ? mm<1, true>(a, t, st, launches) : mm<0, false>(a, t, st, launches)) != cudaSuccess) return err;
        }
        if (below & 1) {
            const void* s;
            size_t se, si;
            node_operand(a, l - 1, below - 1, false, &s, &se, &si);
            k_tree_tail<<<dim3(tree_ew_blocks(dd), a.E), 256, 0, st>>>(s, se, l == 1, lev + (size_t)pairs * dd, ne, dd, a.prm);
            ++*launches;
            if ((err = cudaGetLastError()) != cudaSuccess) return err;
        }
    }
    return cudaSuccess;
}

cudaError_t launch_tree_forward(const TreeArgs& a, const float4* start, size_t start_e, float4* next, size_t next_e,
                                float2* states, size_t states_e, const float* mo, cudaStream_t st, int* launches) {
    const int L = tree_levels(a.wlen);
    const size_t n = (size_t)a.d * a.S, ce = (size_t)(a.W + 1) * a.slice;
    cudaError_t err;
    k_tree_init<<<dim3(tree_ew_blocks(n), a.E), 256, 0, st>>>(start, start_e, a.carry, ce, states, states_e, nullptr, a.S, n, mo);
    ++*launches;
    if ((err = cudaGetLastError()) != cudaSuccess) return err;
    {   // across the wave
        TreeMm t = base(a, a.S);
        t.count = 1;
        node_operand(a, L, 0, false, &t.a, &t.ae, &t.ai);
        t.b = a.carry;
        t.be = ce;
        t.out = a.carry + (size_t)a.wlen * a.slice;
        t.oe = ce;
        t.copy = next;
        t.ce = next_e;
        t.round = states + (size_t)a.wlen * a.slice;
        t.re = states_e;
        t.mo = mo;
        if ((err = L == 0 ? mm<1, false>(a, t, st, launches) : mm<0, false>(a, t, st, launches)) != cudaSuccess) return err;
    }
    for (int l = L - 1; l >= 0; --l) {
        const int step = 1 << l;
        TreeMm t = base(a, a.S);
        t.count = (a.wlen - 1 - step) / (2 * step) + 1;   // nodes 2i + 1 of level l that start below wlen
        node_operand(a, l, 0, false, &t.a, &t.ae, &t.ai);
        t.b = a.carry;
        t.be = ce;
        t.bi = 2 * (size_t)step * a.slice;
        t.out = a.carry + (size_t)step * a.slice;
        t.oe = ce;
        t.oi = t.bi;
        t.round = states + (size_t)step * a.slice;
        t.re = states_e;
        t.ri = t.bi;
        t.mo = mo;
        if ((err = l == 0 ? mm<1, false>(a, t, st, launches) : mm<0, false>(a, t, st, launches)) != cudaSuccess) return err;
    }
    return cudaSuccess;
}

cudaError_t launch_tree_coef(const CostView<float>& cv, int E, int S, const double2* Ofin, float4* coef, cudaStream_t st) {
    k_tree_coef<<<E, 256, 0, st>>>(cv, E, S, Ofin, coef);
    return cudaGetLastError();
}

cudaError_t launch_tree_costate(const TreeArgs& a, const float4* start, size_t start_e, float4* next, size_t next_e,
                                float2* G, size_t G_e, const float4* coef, const float* mo, cudaStream_t st, int* launches) {
    const int L = tree_levels(a.wlen);
    const size_t n = (size_t)a.d * a.S, ce = (size_t)(a.W + 1) * a.slice;
    cudaError_t err;
    // costates by position: after slice j at carry + j slice, G_j at G + (j - 1) slice
    k_tree_init<<<dim3(tree_ew_blocks(n), a.E), 256, 0, st>>>(start, start_e, a.carry + (size_t)a.wlen * a.slice, ce,
                                                            G + (size_t)(a.wlen - 1) * a.slice, G_e, coef, a.S, n, mo);
    ++*launches;
    if ((err = cudaGetLastError()) != cudaSuccess) return err;
    if (next) {   // across the wave, for the wave below
        TreeMm t = base(a, a.S);
        t.count = 1;
        node_operand(a, L, 0, true, &t.a, &t.ae, &t.ai);
        t.b = a.carry + (size_t)a.wlen * a.slice;
        t.be = ce;
        t.out = next;
        t.oe = next_e;
        t.mo = mo;
        if ((err = L == 0 ? mm<1, false>(a, t, st, launches) : mm<2, false>(a, t, st, launches)) != cudaSuccess) return err;
    }
    for (int l = L - 1; l >= 0; --l) {
        const int step = 1 << l, cnt = (a.wlen - 1 - step) / (2 * step) + 1;
        // parents whose right child is whole end at (2i + 2) step; the last one may end at wlen
        const int whole = a.wlen >= cnt * 2 * step ? cnt : cnt - 1;
        for (int part = 0; part < 2; ++part) {
            const int i0 = part == 0 ? 0 : whole;
            TreeMm t = base(a, a.S);
            t.count = part == 0 ? whole : cnt - whole;
            if (t.count == 0) continue;
            node_operand(a, l, 2 * i0 + 1, true, &t.a, &t.ae, &t.ai);
            t.b = a.carry + (size_t)(part == 0 ? 2 * step : a.wlen) * a.slice;
            t.be = ce;
            t.bi = 2 * (size_t)step * a.slice;
            t.out = a.carry + (size_t)(2 * i0 + 1) * step * a.slice;
            t.oe = ce;
            t.oi = t.bi;
            t.round = G + ((size_t)(2 * i0 + 1) * step - 1) * a.slice;
            t.re = G_e;
            t.ri = t.bi;
            t.coef = coef;
            t.mo = mo;
            if ((err = l == 0 ? mm<1, false>(a, t, st, launches) : mm<2, false>(a, t, st, launches)) != cudaSuccess) return err;
        }
    }
    return cudaSuccess;
}

}  // namespace qoc
