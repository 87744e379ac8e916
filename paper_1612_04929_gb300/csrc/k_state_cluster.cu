// The serial recursions of state mode across a thread-block cluster (single-column panels).
//
// One trajectory is a chain of matrix-vector products with X_j (p 2^n of them a slice for Taylor, K
// for Chebyshev; see k_state.cu for the map, its adjoint and its arithmetic, which are the same
// here but for the grids of Chebyshev's vectors).  On one CTA a product of a d = 154 system took 8.5 us, bound by that SM's issue rate and by
// the barriers and shared-memory passes between products, while the other SMs had no work.  Here a
// cluster of CS CTAs owns the trajectory, each CTA d / CS rows of X_j and a warp RW rows:
//   * a warp keeps its rows of X_j in registers for all the products of the slice (RW x QB elements
//     a lane, the next slice's rows loaded meanwhile when they fit too);
//   * the vector lives in every CTA's shared memory.  A row's new element is computed redundantly by
//     the lanes of its warp, and lane (target, row) sends it to the target CTA with st.async, whose
//     bytes complete a transaction on that CTA's mbarrier: one message a product, no other barrier.
//     Two buffers alternate: a CTA sends message m + 2 only after it has all of message m + 1, which
//     every warp of the cluster sends after it has read message m;
//   * the FP32 form splits a vector before a product on the grid of its largest component: it arrives as
//     pairs, and every warp takes that component and splits the vector in registers.  Chebyshev's later
//     vectors keep the grid of the one that starts the application (|phi_k| <= |v|, which that grid
//     bounds), so their owners send them already split.  Taylor's Z_i may be e^(ts) |v|, whose grid
//     would take up to 2 bits of the exact leading part at a norm of 1 a slice and all of it at 8, so each takes
//     a grid of its own.
//     Cost error against 64 bits, d = 154, N = 1000, E = 2, Chebyshev: 5.96e-9 and 3.72e-9 (two problems)
//     with the sender's split, 5.91e-9 and 3.70e-9 with a grid per product, 5.90e-9 and 3.74e-9 in
//     k_state_chain; d = 88, N = 600, E = 4: 1.70e-7 and 1.72e-7 in all three.
// Bound: the latency of one message and of the dependent arithmetic of one product: at d = 154 0.76 us
// on 16 CTAs, 0.97 on 8, 1.31 on 4 (with a grid per product, as Taylor has it, 0.83, 1.02, 1.41; with plain
// remote stores and a cluster barrier per product instead of st.async 1.2 on 8).  d = 154, N = 1000,
// K = 14, 16 members: a recursion went from 119 to 14 ms; one member: from 119 to 10.5 ms.
// Every mbarrier wait is bounded; one that runs out sets kErrTimeout and its warp leaves the loop, the
// others' waits run out in turn, and all meet at the final cluster barrier before any CTA leaves (no
// message can reach a CTA that has gone).
#include <algorithm>

#include "qoc_device.cuh"
#include "qoc_internal.h"
#include "qoc_state.cuh"

namespace qoc {

namespace {

constexpr uint32_t kScWaitLimit = 1u << 22;
// warps a CTA may have by rows a warp: registers for the rows (and, at two, the next slice's)
constexpr int sc_max_warps(int rw) { return rw == 2 ? 12 : 10; }

__device__ __forceinline__ uint32_t sc_su32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t sc_mapa(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ uint32_t sc_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// (the .aligned forms ask every thread of a warp to be there together: lanes may have parted before)
__device__ __forceinline__ void sc_cluster_sync() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void sc_expect(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool sc_wait(uint32_t bar, uint32_t parity) {
    for (uint32_t it = 0; it < kScWaitLimit; ++it) {
        uint32_t done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
            " selp.u32 %0, 1, 0, p;\n}"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}
// 16 bytes to a CTA of the cluster, completing a transaction on its mbarrier
__device__ __forceinline__ void sc_send(uint32_t addr, uint32_t bar, const float4 v) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(addr),
                 "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void sc_send(uint32_t addr, uint32_t bar, const double2 v) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f64 [%0], {%1, %2}, [%3];" ::"r"(addr),
                 "d"(v.x), "d"(v.y), "r"(bar)
                 : "memory");
}

// a scalar coefficient in the recursion's arithmetic
template <typename R> struct ScCoef;
template <> struct ScCoef<float> {
    float2 v;
    __device__ __forceinline__ static ScCoef make(double s) {
        const float h = (float)s;
        return {make_float2(h, (float)(s - (double)h))};
    }
};
template <> struct ScCoef<double> {
    double v;
    __device__ __forceinline__ static ScCoef make(double s) { return {s}; }
};
__device__ __forceinline__ void sc_scale(float4& a, const ScCoef<float> s) {
    st_mul(a.x, a.z, s.v.x, s.v.y);
    st_mul(a.y, a.w, s.v.x, s.v.y);
}
__device__ __forceinline__ void sc_scale(double2& a, const ScCoef<double> s) {
    a.x *= s.v;
    a.y *= s.v;
}

// the running sums of one row: FP32 grid sums and cross terms (re, im); FP64 re, im
template <typename R> struct ScAcc;
template <> struct ScAcc<float> {
    static constexpr int NV = 4;
    float s[4] = {0.f, 0.f, 0.f, 0.f};
    __device__ __forceinline__ void mac(const float4 u, const float2 uf, const float4 x) {
        s[0] = fmaf(u.x, x.x, s[0]);
        s[0] = fmaf(-u.y, x.y, s[0]);
        s[1] = fmaf(u.x, x.y, s[1]);
        s[1] = fmaf(u.y, x.x, s[1]);
        s[2] = fmaf(u.z, x.x, s[2]);
        s[2] = fmaf(-u.w, x.y, s[2]);
        s[2] = fmaf(uf.x, x.z, s[2]);
        s[2] = fmaf(-uf.y, x.w, s[2]);
        s[3] = fmaf(u.z, x.y, s[3]);
        s[3] = fmaf(u.w, x.x, s[3]);
        s[3] = fmaf(uf.x, x.w, s[3]);
        s[3] = fmaf(uf.y, x.z, s[3]);
    }
};
template <> struct ScAcc<double> {
    static constexpr int NV = 2;
    double s[2] = {0.0, 0.0};
};

// exponent of the vector's grid as st_block_magic takes it: 2^e bounds c m
__device__ __forceinline__ int sc_exp(unsigned mbits, float c) {
    const float b = c * __uint_as_float(mbits);
    const int e = b < 1e30f ? (int)(__float_as_uint(b) >> 23) - 126 : 100;
    return e < -100 ? -100 : e;
}
__device__ __forceinline__ float sc_magic(int e) {   // grid_magic for -100 <= e <= 100
    return __uint_as_float(((unsigned)(e + 11 + 127) << 23) | 0x400000u);
}
__device__ __forceinline__ float4 sc_split(const float4 v, float m) {
    float4 g;
    grid_split(v.x, v.z, m, g.x, g.z);
    grid_split(v.y, v.w, m, g.y, g.w);
    return g;
}
__device__ __forceinline__ double2 sc_split(const double2 v, float) { return v; }

}  // namespace

template <typename R, int RW, int QB>
__global__ void __launch_bounds__(sc_max_warps(RW) * 32) k_state_cluster(StateChainArgs<R> A, int rows, int CS) {
    using C = C_t<R>;
    using K = K_t<R>;
    using XE = typename XElem<R>::T;
    constexpr bool kPre = RW == 2;                     // the next slice's rows fit in registers too
    __shared__ __align__(16) K zbuf[2][QB * 32];
    __shared__ __align__(8) uint64_t bars[2];
    __shared__ ScCoef<R> ca[kChebMax + 1];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rank = (int)sc_rank(), kb = blockIdx.x / CS, e = blockIdx.y, d = A.d;
    const int a0 = rank * rows + warp * RW;            // the warp's rows a0 .. a0 + RW - 1
    const int aend = min(d, rank * rows + rows);
    const int mya = a0 + (lane & (RW - 1)), target = lane / RW;
    const bool own = mya < aend;                       // this lane's row exists
    const bool writer = own && target == 0;
    const bool live = a0 < aend;                       // the warp has rows (uniform in the warp)
    const size_t slice = A.sv.slice(), poff = (size_t)kb * A.sv.pstride + mya;
    const int p = A.prm->p, n = A.prm->n;
    const bool fwd = A.dir == 0, cheb = A.cheb != nullptr;
    const int Kc = cheb ? A.cheb->K : 0;
    const int nmv = cheb ? Kc : p << n;                // products (messages) per slice
    const float cmag = sqrtf(2.0f * d) * 1.0625f;
    if (tid == 0) {
        for (int b = 0; b < 2; ++b)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(sc_su32(&bars[b])) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int i = tid; i < 2 * QB * 32; i += blockDim.x) (&zbuf[0][0])[i] = kzero_k<K>();
    for (int k = tid; k <= Kc; k += blockDim.x) ca[k] = ScCoef<R>::make(cheb ? A.cheb->a[k] : 0.0);
    const ScCoef<R> ith = ScCoef<R>::make(cheb ? A.cheb->inv_theta : 0.0);
    __syncthreads();
    const uint32_t bytes = (uint32_t)d * sizeof(K);
    if (tid == 0) {
        sc_expect(sc_su32(&bars[0]), bytes);
        sc_expect(sc_su32(&bars[1]), bytes);
    }
    sc_cluster_sync();                                 // every CTA's barriers and buffers are ready
    bool ok = true;
    const bool sender = own && target < CS;
    uint32_t raddr = 0, rbar = 0;                      // the second buffer and barrier follow the first
    if (sender) {
        raddr = sc_mapa(sc_su32(&zbuf[0][mya]), (uint32_t)target);
        rbar = sc_mapa(sc_su32(&bars[0]), (uint32_t)target);
    }
    unsigned msg = 0, got = 0;                         // messages sent / received so far
    auto send = [&](const K& v) {
        if (sender) sc_send(raddr + (msg & 1) * (uint32_t)sizeof(zbuf[0]), rbar + (msg & 1) * 8u, v);
        ++msg;
    };
    const size_t eoff = (size_t)e;
    K v = kzero_k<K>();
    if (own) {   // starting block (see k_state_chain)
        if (A.cin) v = A.cin[eoff * A.cin_es + poff];
        if (!fwd) st_kadd(v, A.src[eoff * A.src_es + (size_t)(A.wlen - 1) * slice + poff]);
        if (writer) A.out[eoff * A.out_es + (fwd ? 0 : (size_t)(A.wlen - 1) * slice) + poff] = st_round(v);
    }
    const XE* Xe = reinterpret_cast<const XE*>(A.X) + (size_t)e * A.wlen * A.xs;
    XE xc[RW][QB], xn[kPre ? RW : 1][kPre ? QB : 1];
    auto load = [&](auto& x, int t) {
        const XE* Xg = Xe + (size_t)(fwd ? t : A.wlen - 1 - t) * A.xs;
#pragma unroll
        for (int r = 0; r < RW; ++r)
#pragma unroll
            for (int q = 0; q < QB; ++q) {
                const int a = a0 + r, b = q * 32 + lane;
                if (a < aend && b < d) x[r][q] = Xg[(size_t)a * d + b];
                else x[r][q] = XE{};
            }
    };
    if (live) {
        load(xc, 0);
        if (nmv > 0) send(v);
    }
    // y = X b for the message that arrives next: this lane's row.  pairs: the message is a vector of pairs,
    // split here on the grid of its largest component, which becomes mgrid
    float mgrid = 0.f;
    auto product = [&](bool pairs) -> K {
        const uint32_t b = got & 1;
        if (ok) ok = __all_sync(0xffffffffu, sc_wait(sc_su32(&bars[b]), (got >> 1) & 1));
        if (tid == 0) sc_expect(sc_su32(&bars[b]), bytes);   // message got + 2
        ++got;
        K zq[QB];
#pragma unroll
        for (int q = 0; q < QB; ++q) zq[q] = zbuf[b][q * 32 + lane];
        ScAcc<R> acc[RW];
        if constexpr (sizeof(R) == 4) {
            if (pairs) {
                unsigned mb = 0u;
#pragma unroll
                for (int q = 0; q < QB; ++q) mb = max(mb, st_maxbits(zq[q]));
                mb = __reduce_max_sync(0xffffffffu, mb);
                mgrid = sc_magic(sc_exp(mb, cmag));
#pragma unroll
                for (int q = 0; q < QB; ++q) zq[q] = sc_split(zq[q], mgrid);
            }
#pragma unroll
            for (int q = 0; q < QB; ++q)
#pragma unroll
                for (int r = 0; r < RW; ++r) {
                    const float4 u = xc[r][q];
                    acc[r].mac(u, make_float2(u.x + u.z, u.y + u.w), zq[q]);
                }
        } else {
#pragma unroll
            for (int q = 0; q < QB; ++q)
#pragma unroll
                for (int r = 0; r < RW; ++r) {
                    double2 t = make_double2(acc[r].s[0], acc[r].s[1]);
                    cfma(t, xc[r][q], zq[q]);
                    acc[r].s[0] = t.x;
                    acc[r].s[1] = t.y;
                }
        }
        // reduce-scatter: lane l ends with row l % RW
#pragma unroll
        for (int h = RW / 2, o = 1; h >= 1; h >>= 1, o <<= 1) {
            const bool up = lane & o;
#pragma unroll
            for (int r = 0; r < h; ++r)
#pragma unroll
                for (int i = 0; i < ScAcc<R>::NV; ++i) {
                    // rows r (bit clear) and r + h (bit set) of what is left; see the row order below
                    const auto keep = up ? acc[2 * r + 1].s[i] : acc[2 * r].s[i];
                    const auto give = up ? acc[2 * r].s[i] : acc[2 * r + 1].s[i];
                    acc[r].s[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
                }
        }
#pragma unroll
        for (int o = RW; o < 32; o <<= 1)
#pragma unroll
            for (int i = 0; i < ScAcc<R>::NV; ++i) acc[0].s[i] += __shfl_xor_sync(0xffffffffu, acc[0].s[i], o);
        if constexpr (sizeof(R) == 4) {
            float4 y;
            two_sum(acc[0].s[0], acc[0].s[2], y.x, y.z);
            two_sum(acc[0].s[1], acc[0].s[3], y.y, y.w);
            return y;
        } else {
            return make_double2(acc[0].s[0], acc[0].s[1]);
        }
    };
    if (live) {
#pragma unroll 1
        for (int t = 0; t < A.wlen && ok; ++t) {
            const int jl = fwd ? t : A.wlen - 1 - t;
            const bool last = t + 1 == A.wlen;
            if constexpr (kPre) {
                if (!last) load(xn, t + 1);
            }
            K add = kzero_k<K>();                      // costate: the source below
            if (!fwd && jl >= 1 && own) st_kadd(add, A.src[eoff * A.src_es + (size_t)(jl - 1) * slice + poff]);
            if (!cheb) {
#pragma unroll 1
                for (int m = 0; m < (1 << n); ++m) {
                    const bool final_app = m + 1 == (1 << n);
#pragma unroll 1
                    for (int i = p; i >= 1; --i) {
                        K w = product(true);
                        if (!fwd) st_kneg(w);          // T(X^dag) = T(-X)
                        st_kdiv(w, i);
                        st_kadd(w, v);                 // z = v + y / i
                        if (i == 1) v = w;
                        if (i > 1 || !final_app) send(w);
                    }
                }
            } else {
                // w = sum_k a_k rot_k(phi_k), phi_{k+1} = 2 A phi_k - phi_{k-1}, A = (i / theta) X
                K z = v, zprev = v, wacc = v;
                sc_scale(wacc, ca[0]);
#pragma unroll 1
                for (int k = 1; k <= Kc; ++k) {
                    K nx = product(k == 1);
                    sc_scale(nx, ith);
                    st_krot(nx, 1);
                    if (k > 1) {
                        st_ktwice(nx);
                        st_kneg(zprev);
                        st_kadd(nx, zprev);
                    }
                    zprev = z;
                    z = nx;
                    if (k < Kc) send(sc_split(z, mgrid));
                    K q = nx;                          // off the critical path
                    st_krot(q, fwd ? ((4 - (k & 3)) & 3) : (k & 3));
                    sc_scale(q, ca[k]);
                    st_kadd(wacc, q);
                }
                v = wacc;
            }
            // the slice's result: forward Psi_{jl+1}; costate U_jl^dag G_jl, then + src_{jl-1}
            if (!fwd && jl >= 1) st_kadd(v, add);
            if (!last && nmv > 0) send(v);
            if (writer) {
                if (fwd) {
                    A.out[eoff * A.out_es + (size_t)(jl + 1) * slice + poff] = st_round(v);
                    if (last && A.cout) A.cout[eoff * A.cout_es + poff] = v;
                } else if (jl >= 1) {
                    A.out[eoff * A.out_es + (size_t)(jl - 1) * slice + poff] = st_round(v);
                } else if (A.cout) {
                    A.cout[eoff * A.cout_es + poff] = v;
                }
            }
            if (!last) {
                if constexpr (kPre) {
#pragma unroll
                    for (int r = 0; r < RW; ++r)
#pragma unroll
                        for (int q = 0; q < QB; ++q) xc[r][q] = xn[r][q];
                } else {
                    load(xc, t + 1);
                }
            }
        }
    }
    if (!ok && lane == 0) atomicOr(&const_cast<DevParams*>(A.prm)->err, kErrTimeout);
    sc_cluster_sync();
}

// Launches with cs CTAs a cluster, or (resident given) only counts the clusters of that size that the
// device holds at once.
template <typename R, int RW, int QB>
static cudaError_t cluster_launch(const StateChainArgs<R>& a, int cs, int rows, cudaStream_t st, int* resident) {
    cudaError_t e = cudaFuncSetAttribute(k_state_cluster<R, RW, QB>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(a.sv.ncb * cs, a.E);
    cfg.blockDim = dim3((rows + RW - 1) / RW * 32);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cs;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (resident) return cudaOccupancyMaxActiveClusters(resident, k_state_cluster<R, RW, QB>, &cfg);
    return cudaLaunchKernelEx(&cfg, k_state_cluster<R, RW, QB>, a, rows, cs);
}

template <typename R, int RW>
static cudaError_t cluster_qb(const StateChainArgs<R>& a, int cs, int rows, cudaStream_t st, int* resident) {
    switch ((a.d + 31) / 32) {
        case 1: return cluster_launch<R, RW, 1>(a, cs, rows, st, resident);
        case 2: return cluster_launch<R, RW, 2>(a, cs, rows, st, resident);
        case 3: return cluster_launch<R, RW, 3>(a, cs, rows, st, resident);
        case 4: return cluster_launch<R, RW, 4>(a, cs, rows, st, resident);
        case 5: return cluster_launch<R, RW, 5>(a, cs, rows, st, resident);
        case 6: return cluster_launch<R, RW, 6>(a, cs, rows, st, resident);
    }
    return cudaErrorInvalidValue;
}

// two rows a warp while its warps hold the CTA's rows, else four (and at most eight targets)
template <typename R>
static cudaError_t cluster_rows(const StateChainArgs<R>& a, int cs, cudaStream_t st, int* resident) {
    const int rows = (a.d + cs - 1) / cs;
    if (rows <= 2 * sc_max_warps(2)) return cluster_qb<R, 2>(a, cs, rows, st, resident);
    if (rows <= 4 * sc_max_warps(4) && cs <= 8) return cluster_qb<R, 4>(a, cs, rows, st, resident);
    return cudaErrorInvalidValue;
}

// CTAs per cluster for a state-mode plan, the one with the least rounds of resident clusters x time of
// a product, about 0.55 + 0.004 rows x QB us a product (measured at d = 154: 0.77 us on 16 CTAs, 0.97 on
// 8, 1.31 on 4).  What the device holds at once is asked, not counted: a second round doubles a
// recursion (16 members on clusters of 8 took 2.07 us a product, on the size chosen here 1.03), and how
// many clusters of a size fit depends on each GPC's free SMs.  0: k_state_chain's one CTA per panel,
// for panels of several columns, which the plan makes above two chains an SM (S E > 304 here); at d = 154
// that one takes 8.5 us a product, so rounds of small clusters would be faster there too: not built.
// (State mode ends near d = 167, where its gradient's block fills a CTA's shared memory.)
template <typename R>
int state_cluster_size(int d, const StateView<R>& sv, int E) {
    if (sv.cb != 1 || d > 192) return 0;
    StateChainArgs<R> a{};
    a.d = d;
    a.E = E;
    a.sv = sv;
    const long chains = (long)sv.ncb * E;
    double best = 0.0;
    int size = 0;
    for (int cs = 16; cs >= 1; --cs) {
        const int rows = (d + cs - 1) / cs;
        if (cs > 1 && (d < 8 * cs || (cs - 1) * rows >= d)) continue;   // at least eight rows, no CTA without any
        int resident = 0;
        if (cluster_rows(a, cs, nullptr, &resident) != cudaSuccess || resident < 1) {
            cudaGetLastError();
            continue;
        }
        const double cost = (double)((chains + resident - 1) / resident) * (0.55 + 0.004 * rows * ((d + 31) / 32));
        if (size == 0 || cost < best) {
            best = cost;
            size = cs;
        }
    }
    return size;
}

template <typename R>
cudaError_t launch_state_cluster(const StateChainArgs<R>& a, cudaStream_t st) {
    return cluster_rows(a, a.cs, st, nullptr);
}

template int state_cluster_size<float>(int, const StateView<float>&, int);
template int state_cluster_size<double>(int, const StateView<double>&, int);
template cudaError_t launch_state_cluster<float>(const StateChainArgs<float>&, cudaStream_t);
template cudaError_t launch_state_cluster<double>(const StateChainArgs<double>&, cudaStream_t);

}  // namespace qoc
