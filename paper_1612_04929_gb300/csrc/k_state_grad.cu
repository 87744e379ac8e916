// Per-slice exact gradient of the state-mode map for sparse controls (FP32 form): the derivative that
// k_state_grad (k_state.cu) takes, with Xbar kept as its rank-one terms.
//
// Both series are chains y -> X y (Chebyshev: phi_k = 2 A phi_{k-1} - phi_{k-2}, A = (i / theta) X; Taylor:
// Z_i = v + X Z_{i+1} / i), and their reverse modes are chains with the same X that start from the
// slice's costate and do not depend on the forward values (b_k = conj(c_k) wbar + f A b_{k+1} - b_{k+2};
// zbar_{i+1} = -X zbar_i / i), so the two chains advance together: one pass over X a step for both.
// Xbar = sum_t w_t left_t right_t^dag over the steps t is formed only at the controls' non-zero elements.
//
// k_state_grad read X (16 bytes an element) from L2 twice a step, one column at a time, and added every
// step's rank-one term to a d x d block in shared memory.  Here the CTA's warps hold X, rounded to FP32,
// in registers (NR rows of QB 32-column chunks a warp): a step is NR x QB complex multiply-adds for two
// vectors, a reduce-scatter that leaves lane (row, chain) with its element, and one barrier.  Bound:
// FP32 issue.  d = 154, K = 14, 16 members x 1000 slices: 84.8 -> 5.2 ms.
#include <algorithm>

#include "qoc_device.cuh"
#include "qoc_internal.h"
#include "qoc_slice.cuh"
#include "qoc_state.cuh"

namespace qoc {

namespace {
constexpr int SGW = 16;                       // warps
constexpr int SGT = SGW * 32;
constexpr int kSgMaxChunks = 5;               // 32-column chunks: d <= 160 (registers)

// steps (rank-one terms) per column, the factor blocks' leading dimension (odd: rows in distinct banks)
__host__ __device__ inline int sg_terms(int p, int n, int K) { return K > 0 ? K : (p << n); }
inline size_t sg_smem(int d, int S, int p, int n, int K) {
    const int ldt = (sg_terms(p, n, K) * S) | 1;
    return (size_t)2 * d * ldt * sizeof(float2);
}
}  // namespace

template <int QB>
__global__ void __launch_bounds__(SGT, 1) k_state_grad_lr(StateGradArgs<float> A, SysView<float> sys, int terms, int ldt) {
    constexpr int NR = 2 * QB;                // rows of X a warp holds: 16 warps cover 32 QB >= d rows
    extern __shared__ __align__(16) unsigned char sm[];
    __shared__ float wt[kChebMax + 1];        // weights of a column's terms (Taylor: 1 / i, by index mod p)
    const int item = blockIdx.x, jl = item % A.wlen, e = item / A.wlen, j = A.j0 + jl;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, d = A.d, S = A.sv.S;
    const int p = A.prm->p, n = A.prm->n;
    const bool cheb = A.cheb != nullptr;
    float2* Lf = reinterpret_cast<float2*>(sm);   // left factors (cotangents), term t of row a at a * ldt + t
    float2* Rf = Lf + (size_t)d * ldt;            // right factors (forward terms)
    const size_t slice = A.sv.slice();
    const float4* X = reinterpret_cast<const float4*>(A.X) + (size_t)item * A.xs;
    const float2* Psi = A.states + ((size_t)e * (A.wmax + 1) + jl) * slice;
    const float2* Gj = A.G + ((size_t)e * A.wmax + jl) * slice;
    float2 x[NR][QB];
#pragma unroll
    for (int r = 0; r < NR; ++r)
#pragma unroll
        for (int q = 0; q < QB; ++q) {
            const int a = warp * NR + r, b = q * 32 + lane;
            x[r][q] = make_float2(0.f, 0.f);
            if (a < d && b < d) {
                const float4 v = X[(size_t)a * d + b];
                x[r][q] = make_float2(v.x + v.z, v.y + v.w);
            }
        }
    const float th = cheb ? (float)A.cheb->inv_theta : 0.f;
    if (cheb) {
        for (int t = tid; t < terms; t += SGT) wt[t] = t == 0 ? 1.f : 2.f;
    } else {
        for (int t = tid; t < p; t += SGT) wt[t] = 1.f / (float)(t + 1);
    }
    // after the reduce-scatter lane l holds row (l >> 1) of the warp's (16 slots, NR used), the forward
    // chain in even lanes and the cotangent chain in odd ones
    const int lr = lane >> 1, my = warp * NR + lr;
    const bool own = lr < NR && my < d, back = lane & 1;
    for (int s = 0; s < S; ++s) {
        const int t0 = s * terms;
        // this lane's chain: its start (Psi or G), the running and previous elements
        float2 v0 = make_float2(0.f, 0.f);
        if (own) {
            const size_t o = (size_t)(s / A.sv.cb) * A.sv.pstride + (size_t)my * A.sv.cb + (s % A.sv.cb);
            v0 = back ? Gj[o] : Psi[o];
        }
        float2 cur = v0, prev = make_float2(0.f, 0.f);
        if (cheb && back) {                   // b_K = conj(c_K) wbar = i^K a_K wbar
            float2 t = v0;
            const int rot = A.K & 3;
            t = rot == 1 ? make_float2(-v0.y, v0.x) : rot == 2 ? make_float2(-v0.x, -v0.y) : rot == 3 ? make_float2(v0.y, -v0.x) : v0;
            const float aK = (float)A.cheb->a[A.K];
            cur = make_float2(t.x * aK, t.y * aK);
        }
        // Chebyshev: right t = phi_t, left t = b_{t+1}.  Taylor, application m and Horner step i: term
        // m p + i - 1 with right Z_{i+1} and left zbar_i.
        float2 acc_v = make_float2(0.f, 0.f); // Taylor: forward, the application's input; backward, sum of zbar_i
        if (!cheb && !back) acc_v = v0;
        int slot = back ? (cheb ? terms - 1 : (terms - p)) : (cheb ? 0 : p - 1);
        if (own) (back ? Lf : Rf)[(size_t)my * ldt + t0 + slot] = cur;
        int ri = t0 + (cheb ? 0 : p - 1), li = t0 + (cheb ? terms - 1 : terms - p);   // the step's inputs
        for (int t = 0; t + 1 < terms; ++t) {
            __syncthreads();
            float2 z[2][QB];
#pragma unroll
            for (int q = 0; q < QB; ++q) {
                const int b = q * 32 + lane;
                z[0][q] = b < d ? Rf[(size_t)b * ldt + ri] : make_float2(0.f, 0.f);
                z[1][q] = b < d ? Lf[(size_t)b * ldt + li] : make_float2(0.f, 0.f);
            }
            // reduce-scatter: lane bit 4 takes rows 8 .. of the warp's 16 slots (NR used), bit 3 rows 4 .. 7
            // of its half, then bit 2, bit 1, and bit 0 the chain; each pair of rows folds as it is done
            float s4[8][4];
            const bool up4 = lane & 16;
#pragma unroll
            for (int r = 0; r < (NR < 8 ? NR : 8); ++r) {
                float2 lo[2], hi[2];
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    lo[c] = hi[c] = make_float2(0.f, 0.f);
#pragma unroll
                    for (int q = 0; q < QB; ++q) {
                        cfma(lo[c], x[r][q], z[c][q]);
                        if (r + 8 < NR) cfma(hi[c], x[r + 8 < NR ? r + 8 : 0][q], z[c][q]);
                    }
                }
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    s4[r][2 * c] = (up4 ? hi[c].x : lo[c].x) + __shfl_xor_sync(0xffffffffu, up4 ? lo[c].x : hi[c].x, 16);
                    s4[r][2 * c + 1] = (up4 ? hi[c].y : lo[c].y) + __shfl_xor_sync(0xffffffffu, up4 ? lo[c].y : hi[c].y, 16);
                }
            }
#pragma unroll
            for (int r = NR < 8 ? NR : 8; r < 8; ++r)
#pragma unroll
                for (int i = 0; i < 4; ++i) s4[r][i] = 0.f;
#pragma unroll
            for (int h = 4, o = 8; h >= 1; h >>= 1, o >>= 1) {
                const bool up = lane & o;
#pragma unroll
                for (int r = 0; r < h; ++r)
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float keep = up ? s4[r + h][i] : s4[r][i], give = up ? s4[r][i] : s4[r + h][i];
                        s4[r][i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
                    }
            }
            float2 y;
            {
                const float gx = back ? s4[0][0] : s4[0][2], gy = back ? s4[0][1] : s4[0][3];
                const float kx = back ? s4[0][2] : s4[0][0], ky = back ? s4[0][3] : s4[0][1];
                y.x = kx + __shfl_xor_sync(0xffffffffu, gx, 1);
                y.y = ky + __shfl_xor_sync(0xffffffffu, gy, 1);
            }
            if (cheb) {
                const float2 ay = make_float2(-th * y.y, th * y.x);      // A y
                float2 nx;
                if (!back) {
                    const float f = t == 0 ? 1.f : 2.f;                  // phi_1 = A phi_0
                    nx = make_float2(f * ay.x - prev.x, f * ay.y - prev.y);
                } else {                                                 // b_k, k = K - 1 - t >= 1
                    const int k = A.K - 1 - t, rot = k & 3;
                    const float ak = (float)A.cheb->a[k];
                    const float2 w = rot == 1 ? make_float2(-v0.y, v0.x)
                                              : rot == 2 ? make_float2(-v0.x, -v0.y) : rot == 3 ? make_float2(v0.y, -v0.x) : v0;
                    nx = make_float2(w.x * ak + (2.f * ay.x - prev.x), w.y * ak + (2.f * ay.y - prev.y));
                }
                prev = cur;
                cur = nx;
                ++ri;
                --li;
                slot = (back ? li : ri) - t0;
            } else {
                const int st = t % p;
                if (!back) {                                             // Z_i, i = p - st
                    const float wi = 1.f / (float)(p - st);
                    cur = make_float2(fmaf(y.x, wi, acc_v.x), fmaf(y.y, wi, acc_v.y));
                    if (st == p - 1) acc_v = cur;                        // the next application's input
                } else {                                                 // zbar_{i+1}, i = st + 1
                    const float wi = -1.f / (float)(st + 1);
                    acc_v.x += cur.x;
                    acc_v.y += cur.y;
                    cur = make_float2(y.x * wi, y.y * wi);
                    if (st == p - 1) {                                   // zbar_{p+1} and the application's sum
                        cur.x += acc_v.x;
                        cur.y += acc_v.y;
                        acc_v = make_float2(0.f, 0.f);
                    }
                }
                // forward term indices run p - 1 .. 0 within an application, applications upwards;
                // backward ones 0 .. p - 1, applications downwards
                ri = st == p - 1 ? ri + 2 * p - 1 : ri - 1;
                li = st == p - 1 ? li - 2 * p + 1 : li + 1;
                slot = (back ? li : ri) - t0;
            }
            if (own) (back ? Lf : Rf)[(size_t)my * ldt + t0 + slot] = cur;
        }
        __syncthreads();
    }
    // Xbar at the controls' elements; Chebyshev: Xbar = (-i / theta) sum_t w_t left right^dag
    const int nt = terms * S;
    for (int k = warp; k < A.M; k += SGW) {           // a warp per control (and its elements over the lanes)
        double v = 0.0;   // in FP64 as in k_state_grad: two products an element, beside its sum over the terms
        for (int i = sys.hoff[k] + lane; i < sys.hoff[k + 1]; i += 32) {
            const int ab = sys.hidx[i];
            const float2 h = sys.hval[i];
            const float2* l = Lf + (size_t)(ab >> 16) * ldt;
            const float2* r = Rf + (size_t)(ab & 0xffff) * ldt;
            float2 xb = make_float2(0.f, 0.f);
            int w = 0;
            for (int t = 0; t < nt; ++t) {
                const float ww = wt[w];
                if (++w == (cheb ? terms : p)) w = 0;
                const float2 q = l[t];
                cfma_bcj(xb, make_float2(ww * q.x, ww * q.y), r[t]);
            }
            if (cheb) xb = make_float2(th * xb.y, -th * xb.x);
            v = fma((double)xb.x, (double)h.y, v);
            v = fma(-(double)xb.y, (double)h.x, v);
        }
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) A.gpart[((size_t)e * A.M + k) * A.N + j] = A.prm->s * v;
    }
}

// applies: FP32 form, sparse controls, few enough columns chunks for the registers, and a term to have
bool state_grad_lr_applies(const SysView<float>& sys, int d, int S, int p, int n, int K, bool cheb) {
    const int terms = sg_terms(p, n, cheb ? K : 0);
    // small d with several columns: the columns go one after another here, and a CTA of k_state_grad takes little
    // more than one (d = 16, 900 slices, Chebyshev: S = 2 133 us against 193 there, S = 4 246 against 213, S = 8
    // 324 against 217; d = 24, S = 8 334 against 387)
    if (d < 24 && S > 2) return false;
    if (!sys.hoff || d > 32 * kSgMaxChunks || (cheb && K < 1) || (!cheb && n > 16)) return false;
    if (!cheb && p > kChebMax) return false;
    return (long long)terms * S < 4096 && sg_smem(d, S, p, n, cheb ? K : 0) <= kMaxDynSmem;
}

template <int QB>
static cudaError_t sg_launch(const StateGradArgs<float>& a, const SysView<float>& sys, int terms, int ldt, size_t smem,
                             cudaStream_t st) {
    cudaError_t e = cudaFuncSetAttribute(k_state_grad_lr<QB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_state_grad_lr<QB><<<a.wlen * a.E, SGT, smem, st>>>(a, sys, terms, ldt);
    return cudaGetLastError();
}

cudaError_t launch_state_grad_lr(const StateGradArgs<float>& a, const SysView<float>& sys, int p, int n, cudaStream_t st) {
    if (a.M == 0) return cudaSuccess;
    const int K = a.cheb ? a.K : 0, terms = sg_terms(p, n, K), ldt = (terms * a.sv.S) | 1;
    const size_t smem = sg_smem(a.d, a.sv.S, p, n, K);
    switch ((a.d + 31) / 32) {
        case 1: return sg_launch<1>(a, sys, terms, ldt, smem, st);
        case 2: return sg_launch<2>(a, sys, terms, ldt, smem, st);
        case 3: return sg_launch<3>(a, sys, terms, ldt, smem, st);
        case 4: return sg_launch<4>(a, sys, terms, ldt, smem, st);
        case 5: return sg_launch<5>(a, sys, terms, ldt, smem, st);
    }
    return cudaErrorInvalidValue;
}

}  // namespace qoc
