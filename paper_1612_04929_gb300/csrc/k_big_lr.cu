// Low-rank reverse-mode adjoint of the Paterson-Stockmeyer form on the batched large-d path (FP32
// form): the exact derivative of the same truncated series (Eqs. 9, 10, A3) as the dense reverse
// mode (launch_big_adj_rev_ps), over the same stored operands, with every cotangent kept as factors.
//
// When S columns are propagated, Ubar_j = G_j Psi_{j-1}^dag has rank S, and r = 2^n S after the
// squarings.  With Y = X^3, W_q the chain matrices and c_k = 1/k!:
//   squarings    L <- [L, S_m^dag L], R <- [S_m R, R]                  (Sbar = L R^dag)
//   chain        Wbar_q = L_q R^dag, L_{q+1} = Y^dag L_q, V_q = W_{q+1} R, V_qt = c_3qt+3 R:
//                Ybar = sum_q L_q V_q^dag, Xbar = A1 R^dag, X2bar = A2 R^dag,
//                A1 = sum_q c_3q+1 L_q, A2 = sum_q c_3q+2 L_q
//   powers       X2bar += Ybar X^dag, Xbar += X2^dag Ybar, Xbar += X2bar X^dag + X^dag X2bar
// so Xbar is a sum of 3 (qt + 1) r + 2 r outer products l r^dag whose factors are matrix-vector
// products with the stored operands; it is formed tile by tile in registers and contracted with
// every H_k there.  X is anti-Hermitian (H_0, H_k, H_det are checked to 1e-12 on entry), so X^dag l =
// -X l, Y^dag l = -Y l, (X^2)^dag l = X^2 l to the rounding of the stored operands, and one product
// routine (y = M x from the stored M^dag, a thread per column pair, coalesced rows) serves all but
// the S_m^dag L of the squarings.
//
// Bound: about 25 r columns of d x d by d work against the dense form's 13 d x d by d x d products;
// the operands are read from HBM once ((qt + n + 3) d^2 values a slice) and the kernel is bound by
// FP32 issue and L2 (the chunks of four columns re-read an operand).  d = 154, S = 1, n = 1,
// N = 8000 (r = 2): the adjoint went from 110.6 ms (dense) to 9.5 ms an evaluation,
// and to 7.6 ms where the controls are sparse and Xbar is formed at their elements only.
#include <algorithm>

#include "qoc_device.cuh"
#include "qoc_internal.h"

namespace qoc {

namespace {

constexpr int LT = 256;      // threads
constexpr int LNC = 4;       // columns per pass of a product
constexpr int LKC = 8;       // controls contracted per pass over the tiles

struct LrArgs {
    const DevParams* prm;
    SysView<float> sys;
    StateView<float> sv;
    int j0, wlen, wmax, p, n, qt, r, ldw;
    const float2* states;
    const float2* Gbuf;
    const float2* zst;       // stored operands of item i at zst + i * zs, slot s at + s * ms
    size_t zs, ms;
    int cap;
    double* gpart;
};

// the factor blocks are d x ldw with an even ldw whose half is odd: pairs of columns load as 16
// bytes, and eight rows of one column pair fall in distinct banks
inline int lr_ldw(int w) {
    int l = (w + 1) & ~1;
    if (((l >> 1) & 1) == 0) l += 2;
    return l;
}
// (the last chunk of a product may read up to LNC - 1 columns past a row: slack after each block, so that the
// last row's reads do not touch a block that the same product writes.  After the blocks the warps' partial
// sums of the sparse contraction)
__host__ __device__ inline size_t lr_block(int d, int ldw) { return (size_t)d * ldw + LNC; }
__host__ __device__ inline size_t lr_part_offset(int d, int ldw) { return 6 * lr_block(d, ldw) * sizeof(float2); }
inline size_t lr_smem(int d, int ldw) { return lr_part_offset(d, ldw) + kMaxControls * (LT / 32) * sizeof(double); }

}  // namespace

// acc[v][c] += conj(M[a][b + v]) x[a][c] over the rows a = g, g + G, ..
template <int VW, int NJ>
__device__ __forceinline__ void lr_rows(float2 (&acc)[NJ][VW][LNC], const float2* __restrict__ M,
                                        const float2* const (&x)[NJ], int d, int ldw, int b, int g, int G) {
#pragma unroll 4
    for (int a = g; a < d; a += G) {
        float2 m[VW];
        if constexpr (VW == 2) {
            const float4 q = *reinterpret_cast<const float4*>(M + (size_t)a * d + b);
            m[0] = make_float2(q.x, q.y);
            m[1] = make_float2(q.z, q.w);
        } else {
            m[0] = M[(size_t)a * d + b];
        }
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
            const float4* xr = reinterpret_cast<const float4*>(x[j] + (size_t)a * ldw);
#pragma unroll
            for (int h = 0; h < LNC / 2; ++h) {
                const float4 q = xr[h];
#pragma unroll
                for (int v = 0; v < VW; ++v) {
                    cfma_cj(acc[j][v][2 * h], m[v], make_float2(q.x, q.y));
                    cfma_cj(acc[j][v][2 * h + 1], m[v], make_float2(q.z, q.w));
                }
            }
        }
    }
}

// y_j[:, c] = sgn_j M^dag-stored product of NJ blocks of w columns: the matrix M given as its
// conjugate transpose Md, y = M x = (Md)^dag x.  NJ = 2 with M2 given: two matrices, one block each.
// Row groups add their partial sums in turn (a fixed order).  Reads past w within the last chunk
// touch the padding, the next row or the slack after the block and are not stored.  Ends with a barrier.
template <int VW, int NJ, bool TWO>
__device__ __forceinline__ void lr_mul(const float2* __restrict__ M1, const float2* __restrict__ M2,
                                       const float2* x1, float2* y1, float sg1, const float2* x2, float2* y2, float sg2,
                                       int w, int d, int ldw) {
    const int nb = (d + VW - 1) / VW;
    const int G = nb >= LT ? 1 : LT / nb;
    const int g = nb >= LT ? 0 : threadIdx.x / nb;
    for (int c0 = 0; c0 < w; c0 += LNC) {
        const int nc = min(LNC, w - c0);
        for (int s0 = 0; s0 < nb; s0 += LT) {
            const int slot = s0 + (nb >= LT ? (int)threadIdx.x : (int)threadIdx.x - g * nb);
            const bool on = g < G && slot < nb;
            const int b = slot * VW;
            float2 acc[NJ][VW][LNC];
#pragma unroll
            for (int j = 0; j < NJ; ++j)
#pragma unroll
                for (int v = 0; v < VW; ++v)
#pragma unroll
                    for (int c = 0; c < LNC; ++c) acc[j][v][c] = make_float2(0.f, 0.f);
            if (on) {
                if constexpr (TWO) {
                    float2 (&a1)[1][VW][LNC] = reinterpret_cast<float2 (&)[1][VW][LNC]>(acc[0]);
                    float2 (&a2)[1][VW][LNC] = reinterpret_cast<float2 (&)[1][VW][LNC]>(acc[NJ - 1]);
                    const float2* const xa[1] = {x1 + c0};
                    const float2* const xb[1] = {x2 + c0};
                    lr_rows<VW, 1>(a1, M1, xa, d, ldw, b, g, G);
                    lr_rows<VW, 1>(a2, M2, xb, d, ldw, b, g, G);
                } else if constexpr (NJ == 2) {
                    const float2* const xx[2] = {x1 + c0, x2 + c0};
                    lr_rows<VW, 2>(acc, M1, xx, d, ldw, b, g, G);
                } else {
                    const float2* const xx[1] = {x1 + c0};
                    lr_rows<VW, 1>(acc, M1, xx, d, ldw, b, g, G);
                }
            }
            for (int t = 0; t < G; ++t) {
                if (on && g == t) {
#pragma unroll
                    for (int j = 0; j < NJ; ++j) {
                        float2* y = j == 0 ? y1 : y2;
                        const float sg = j == 0 ? sg1 : sg2;
#pragma unroll
                        for (int v = 0; v < VW; ++v)
#pragma unroll
                            for (int c = 0; c < LNC; ++c)
                                if (c < nc) {
                                    float2& o = y[(size_t)(b + v) * ldw + c0 + c];
                                    const float2 q = make_float2(sg * acc[j][v][c].x, sg * acc[j][v][c].y);
                                    o = t == 0 ? q : make_float2(o.x + q.x, o.y + q.y);
                                }
                    }
                }
                __syncthreads();
            }
        }
    }
}

// y[:, c] = Md x (the stored matrix itself): a warp per row, the lanes along its columns
__device__ __forceinline__ void lr_mul_rows(const float2* __restrict__ Md, const float2* x, float2* y, int w, int d,
                                            int ldw) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int c0 = 0; c0 < w; c0 += 2) {
        const bool two = c0 + 1 < w;
        for (int a = warp; a < d; a += LT / 32) {
            float2 s0 = make_float2(0.f, 0.f), s1 = s0;
#pragma unroll 4
            for (int b = lane; b < d; b += 32) {
                const float2 m = Md[(size_t)a * d + b];
                cfma(s0, m, x[(size_t)b * ldw + c0]);
                if (two) cfma(s1, m, x[(size_t)b * ldw + c0 + 1]);
            }
            for (int o = 16; o > 0; o >>= 1) {
                s0.x += __shfl_xor_sync(0xffffffffu, s0.x, o);
                s0.y += __shfl_xor_sync(0xffffffffu, s0.y, o);
                s1.x += __shfl_xor_sync(0xffffffffu, s1.x, o);
                s1.y += __shfl_xor_sync(0xffffffffu, s1.y, o);
            }
            if (lane == 0) {
                y[(size_t)a * ldw + c0] = s0;
                if (two) y[(size_t)a * ldw + c0 + 1] = s1;
            }
        }
    }
}

// One CTA per (slice, member).  VW: matrix columns per thread (2: 16-byte loads, even d); MT: the
// 16 x 16 threads' outputs a side in the contraction's tiles.
template <int VW, int MT>
__global__ void __launch_bounds__(LT, 2) k_big_adj_lr(LrArgs A) {
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ double red[32];
    const int item = blockIdx.x, jl = item % A.wlen, e = item / A.wlen, j = A.j0 + jl;
    const int tid = threadIdx.x, d = A.sys.d, M = A.sys.M, r = A.r, qt = A.qt, ldw = A.ldw, p = A.p;
    const int S = A.sv.S, w1 = (qt + 1) * r;
    const size_t blk = lr_block(d, ldw);
    float2* Lw = reinterpret_cast<float2*>(smraw);   // L_0 .. L_qt, A2
    float2* Vw = Lw + blk;                           // V_0 .. V_qt, R
    float2* XL = Vw + blk;                           // X^dag L_0 .. X^dag L_qt, X^dag A2
    float2* XV = XL + blk;                           // X V_0 .. X V_qt, X R
    float2* PL = XV + blk;                           // (X^2)^dag L_0 .., then A1 + X^dag A2
    float2* PV = PL + blk;                           // X^2 V_0 .., then X R
    const float2* zi = A.zst + (size_t)item * A.zs;
    auto slot = [&](int s) { return zi + (size_t)s * A.ms; };
    const float2* Xd = slot(A.cap - 1);
    const DevParams* prm = A.prm;
    for (size_t i = tid; i < 6 * blk; i += LT) Lw[i] = make_float2(0.f, 0.f);
    __syncthreads();
    {   // L = G_j, R = Psi_{j-1}
        const size_t slice = A.sv.slice();
        const float2* Gj = A.Gbuf + ((size_t)e * A.wmax + jl) * slice;
        const float2* Pj = A.states + ((size_t)e * (A.wmax + 1) + jl) * slice;
        for (int o = tid; o < d * S; o += LT) {
            const int a = o / S, c = o - a * S;
            const size_t off = (size_t)(c / A.sv.cb) * A.sv.pstride + (size_t)a * A.sv.cb + (c % A.sv.cb);
            Lw[(size_t)a * ldw + c] = Gj[off];
            PL[(size_t)a * ldw + c] = Pj[off];
        }
    }
    __syncthreads();
    float2* Rw = PL;   // R during the squarings; XL holds S_m R
    int rr = S;
    for (int m = A.n - 1; m >= 0; --m) {
        const float2* Sd = slot(qt + 2 + m);
        lr_mul_rows(Sd, Lw, Lw + rr, rr, d, ldw);
        lr_mul<VW, 1, false>(Sd, nullptr, Rw, XL, 1.f, nullptr, nullptr, 0.f, rr, d, ldw);
        for (int o = tid; o < d * rr; o += LT) {
            const int a = o / rr, c = o - a * rr;
            const size_t i = (size_t)a * ldw + c;
            Rw[i + rr] = Rw[i];
            Rw[i] = XL[i];
        }
        __syncthreads();
        rr *= 2;
    }
    for (int o = tid; o < d * r; o += LT) {   // R into its place, V_qt = c_3qt+3 R
        const int a = o / r, c = o - a * r;
        const float2 v = Rw[(size_t)a * ldw + c];
        const float c3 = prm->ch[3 * qt + 3];
        Vw[(size_t)a * ldw + w1 + c] = v;
        Vw[(size_t)a * ldw + qt * r + c] = make_float2(c3 * v.x, c3 * v.y);
    }
    __syncthreads();
    // chain: V_q = W_{q+1} R, L_{q+1} = Y^dag L_q = -Y L_q.  The 16-byte reads of a column chunk want an
    // even first column: R and L_q are staged at column 0 of two blocks that are still free.
    float2* Rs = PV;
    for (int o = tid; o < d * r; o += LT) {
        const int a = o / r, c = o - a * r;
        Rs[(size_t)a * ldw + c] = Vw[(size_t)a * ldw + w1 + c];
    }
    __syncthreads();
    for (int q = 0; q < qt; ++q) {
        for (int o = tid; o < d * r; o += LT) {
            const int a = o / r, c = o - a * r;
            XL[(size_t)a * ldw + c] = Lw[(size_t)a * ldw + q * r + c];
        }
        __syncthreads();
        lr_mul<VW, 2, true>(slot(2 + (qt - 1 - q)), slot(1), Rs, Vw + q * r, 1.f, XL, Lw + (q + 1) * r, -1.f, r, d, ldw);
    }
    for (int o = tid; o < d * r; o += LT) {   // A1 (into PL's last columns), A2
        const int a = o / r, c = o - a * r;
        float2 s1 = make_float2(0.f, 0.f), s2 = s1;
        for (int q = 0; q <= qt; ++q) {
            const float2 l = Lw[(size_t)a * ldw + q * r + c];
            const float c1 = prm->ch[3 * q + 1], c2 = prm->ch[3 * q + 2];
            s1.x = fmaf(c1, l.x, s1.x);
            s1.y = fmaf(c1, l.y, s1.y);
            s2.x = fmaf(c2, l.x, s2.x);
            s2.y = fmaf(c2, l.y, s2.y);
        }
        Lw[(size_t)a * ldw + w1 + c] = s2;
        PL[(size_t)a * ldw + w1 + c] = s1;
    }
    __syncthreads();
    // X^dag [L, A2] = -X [L, A2] and X [V, R]; then X^2 L and X (X V)
    lr_mul<VW, 2, false>(Xd, nullptr, Lw, XL, -1.f, Vw, XV, 1.f, w1 + r, d, ldw);
    if (p >= 3) {
        lr_mul<VW, 1, false>(slot(0), nullptr, Lw, PL, 1.f, nullptr, nullptr, 0.f, w1, d, ldw);
        lr_mul<VW, 1, false>(Xd, nullptr, XV, PV, 1.f, nullptr, nullptr, 0.f, w1, d, ldw);
    } else {   // V = 0: no Y terms
        for (int o = tid; o < d * w1; o += LT) {
            const int a = o / w1, c = o - a * w1;
            PL[(size_t)a * ldw + c] = PV[(size_t)a * ldw + c] = make_float2(0.f, 0.f);
        }
    }
    for (int o = tid; o < d * r; o += LT) {
        const int a = o / r, c = o - a * r;
        const size_t i = (size_t)a * ldw + w1 + c;
        PL[i].x += XL[i].x;
        PL[i].y += XL[i].y;
        PV[i] = XV[i];
        XL[i] = make_float2(0.f, 0.f);   // the pair (X^dag A2, X R) is not one of Xbar's
    }
    // padding columns past w1 + r may hold chunk leftovers of other blocks: none is stored there
    __syncthreads();
    // Xbar = L PV^dag + PL V^dag + XL XV^dag tile by tile, contracted with H_k:
    // dC/du_kj = s sum (Xbar_re Hk_im - Xbar_im Hk_re)
    // its elements one by one at the controls' non-zero elements, all warps on each control
    if (A.sys.hoff) {
        const int warp = tid >> 5, lane = tid & 31, wq = (w1 + r + 1) >> 1;
        double* part = reinterpret_cast<double*>(smraw + lr_part_offset(d, ldw));
        for (int k = 0; k < M; ++k) {
            const int i1 = A.sys.hoff[k + 1];
            float hi = 0.f, lo = 0.f;
            for (int i = A.sys.hoff[k] + tid; i < i1; i += LT) {
                const int ab = A.sys.hidx[i], a = ab >> 16, b = ab & 0xffff;
                const float2 h = A.sys.hval[i];
                float2 x = make_float2(0.f, 0.f);
#pragma unroll
                for (int f = 0; f < 3; ++f) {
                    const float4* l = reinterpret_cast<const float4*>((f == 0 ? Lw : (f == 1 ? PL : XL)) + (size_t)a * ldw);
                    const float4* v = reinterpret_cast<const float4*>((f == 0 ? PV : (f == 1 ? Vw : XV)) + (size_t)b * ldw);
                    for (int t = 0; t < wq; ++t) {
                        const float4 lq = l[t], vq = v[t];
                        cfma_bcj(x, make_float2(lq.x, lq.y), make_float2(vq.x, vq.y));
                        cfma_bcj(x, make_float2(lq.z, lq.w), make_float2(vq.z, vq.w));
                    }
                }
                pair_acc(hi, lo, x.x, h.y);
                pair_acc(hi, lo, -x.y, h.x);
            }
            double v = (double)hi + (double)lo;
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (lane == 0) part[k * (LT / 32) + warp] = v;
        }
        __syncthreads();
        for (int k = tid; k < M; k += LT) {
            double v = 0.0;
            for (int w = 0; w < LT / 32; ++w) v += part[k * (LT / 32) + w];
            A.gpart[((size_t)e * M + k) * A.sys.N + j] = prm->s * v;
        }
        return;
    }
    constexpr int T = 16 * MT;
    const int tx = tid & 15, ty = tid >> 4, nt = (d + T - 1) / T;
    const int wp = (w1 + r + 1) >> 1;   // column pairs
    const size_t dd = (size_t)d * d;
    for (int k0 = 0; k0 < M; k0 += LKC) {
        float sh[LKC], sl[LKC];
#pragma unroll
        for (int k = 0; k < LKC; ++k) sh[k] = sl[k] = 0.f;
        for (int tile = 0; tile < nt * nt; ++tile) {
            const int r0 = (tile / nt) * T, c0 = (tile % nt) * T;
            float2 acc[MT][MT];
#pragma unroll
            for (int a = 0; a < MT; ++a)
#pragma unroll
                for (int b = 0; b < MT; ++b) acc[a][b] = make_float2(0.f, 0.f);
            for (int f = 0; f < 3; ++f) {
                const float4* l = reinterpret_cast<const float4*>(f == 0 ? Lw : (f == 1 ? PL : XL));
                const float4* v = reinterpret_cast<const float4*>(f == 0 ? PV : (f == 1 ? Vw : XV));
                for (int t = 0; t < wp; ++t) {
                    float4 lq[MT], vq[MT];
#pragma unroll
                    for (int a = 0; a < MT; ++a) {
                        const int row = min(r0 + ty + 16 * a, d - 1), col = min(c0 + tx + 16 * a, d - 1);
                        lq[a] = l[(size_t)row * (ldw >> 1) + t];
                        vq[a] = v[(size_t)col * (ldw >> 1) + t];
                    }
#pragma unroll
                    for (int a = 0; a < MT; ++a)
#pragma unroll
                        for (int b = 0; b < MT; ++b) {
                            cfma_bcj(acc[a][b], make_float2(lq[a].x, lq[a].y), make_float2(vq[b].x, vq[b].y));
                            cfma_bcj(acc[a][b], make_float2(lq[a].z, lq[a].w), make_float2(vq[b].z, vq[b].w));
                        }
                }
            }
#pragma unroll
            for (int k = 0; k < LKC; ++k) {
                if (k0 + k >= M) break;
                const float2* hk = A.sys.Hk + (size_t)(k0 + k) * dd;
#pragma unroll
                for (int a = 0; a < MT; ++a)
#pragma unroll
                    for (int b = 0; b < MT; ++b) {
                        const int row = r0 + ty + 16 * a, col = c0 + tx + 16 * b;
                        if (row < d && col < d) {
                            const float2 h = hk[(size_t)row * d + col];
                            pair_acc(sh[k], sl[k], acc[a][b].x, h.y);
                            pair_acc(sh[k], sl[k], -acc[a][b].y, h.x);
                        }
                    }
            }
        }
#pragma unroll
        for (int k = 0; k < LKC; ++k) {
            if (k0 + k >= M) break;
            const double v = block_sum((double)sh[k] + (double)sl[k], red);
            if (tid == 0) A.gpart[((size_t)e * M + k0 + k) * A.sys.N + j] = prm->s * v;
        }
    }
}

// the low-rank form applies to an evaluation's (p, n): small enough a rank, and the factors fit
bool big_lr_applies(int d, int S, int p, int n) {
    if (p < 1 || !adj_lowrank_applies(S, n, d)) return false;
    return lr_smem(d, lr_ldw((ps_top(p) + 2) * (S << n))) <= kMaxDynSmem;
}

template <int VW, int MT>
static cudaError_t lr_launch(const LrArgs& a, int items, cudaStream_t st) {
    const size_t smem = lr_smem(a.sys.d, a.ldw);
    cudaError_t e = cudaFuncSetAttribute(k_big_adj_lr<VW, MT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_big_adj_lr<VW, MT><<<items, LT, smem, st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_big_adj_lr(const BigArgs<float>& a, const SysView<float>& sys, const StateView<float>& sv,
                              const float2* states, const float2* Gbuf, double* gpart, const DevParams& hp,
                              const float2* zst, cudaStream_t st) {
    if (sys.M == 0) return cudaSuccess;
    if (!zst || !big_lr_applies(a.d, sv.S, hp.p, hp.n)) return cudaErrorInvalidValue;
    LrArgs x{};
    x.prm = a.prm;
    x.sys = sys;
    x.sv = sv;
    x.j0 = a.j0;
    x.wlen = a.wlen;
    x.wmax = a.wmax;
    x.p = hp.p;
    x.n = hp.n;
    x.qt = ps_top(hp.p);
    x.r = sv.S << hp.n;
    x.ldw = lr_ldw((x.qt + 2) * x.r);
    x.states = states;
    x.Gbuf = Gbuf;
    x.zst = zst;
    x.cap = ps_big_slots(hp.p, hp.n);
    x.ms = a.mstride;
    x.zs = (size_t)x.cap * a.mstride;
    x.gpart = gpart;
    const int items = a.wlen * a.E;
    const bool v2 = (a.d & 1) == 0;   // 16-byte rows
    // contraction tiles of 64 or 80 rows, whichever pads less
    const int d = a.d;
    const bool t5 = (d + 79) / 80 * 80 < (d + 63) / 64 * 64;
    if (v2) return t5 ? lr_launch<2, 5>(x, items, st) : lr_launch<2, 4>(x, items, st);
    return t5 ? lr_launch<1, 5>(x, items, st) : lr_launch<1, 4>(x, items, st);
}

}  // namespace qoc
