// Tile engine of the batched SIMT products: one CTA computes a T x T tile (T = G MT) of C = A B for one
// item, a G x G grid of threads owning MT x MT outputs each (rows ty + G x, columns tx + G y), the
// operands streamed through a ring of ST K-chunks of 16 in shared memory, filled by cp.async (one
// barrier a chunk).
//
// These products are bound by FP32 issue: per k a thread loads 2 MT operands and issues 12 MT^2 (split)
// or 4 MT^2 (plain) FMAs, so what counts is the outputs a thread, the registers that keep the next loads
// in flight, and the padding of the tiles.  Measured on GB300 (TFLOP/s executed, padding included; the
// FMA peak is 78.5, and the packed FMA form takes two issue slots, so it gains nothing):
//   split  8 x 8 threads, MT = 4: 55 (168 registers, 6 CTAs an SM), 52 at 128 registers;
//          16 x 16, MT = 4: 53; MT = 2 (the former tile up to d = 96): 41; grids that are no multiple of
//          four warps, 20 x 20 or 21 x 21: 38 (the schedulers' loads differ)
//   plain  16 x 16 threads, MT = 4: 44, MT = 5: 47, MT = 6: 46; 8 x 8, MT = 4: 39
// so split products take 32 x 32 tiles of 64 threads (d = 154 as 160 rows, not 192), or 16 x 16 tiles where
// there are few products or 32 pads much, and plain products the 16 x 16 grid with an MT that depends on d and
// on their number (gemm_time).  Rows of an edge tile past d are left out
// in the plain products, whose tiles are large; in the split ones the branches (591 against 548 us) or
// loops of their own for the edges (instruction cache) cost more than the padding.  Against the former
// tiles a split product went, per 300 items of d = 154, 700 -> 548 us (the plain-operand chain products
// 366 -> 277); per 500 of d = 81 161 -> 113 (chain), 195 -> 194
// (others); d = 128 is as before (264 us per 250).
#pragma once
#include <algorithm>
#include <type_traits>

#include "qoc_device.cuh"
#include "qoc_internal.h"

namespace qoc {

constexpr int kGemmK = 16;   // K-chunk

// tile shapes: thread grid G x G, MT outputs a side, ring stages, resident CTAs asked of the compiler, and
// whether rows past d are left out (plain products; a branch a row)
template <int MT_, int G_, int ST_, int MB_, bool SKIP_>
struct GemmShape {
    static constexpr bool SKIP = SKIP_;
    static constexpr int MT = MT_, G = G_, ST = ST_, MB = MB_, T = MT * G, NT = G * G;
    static int tiles(int d) { return (d + T - 1) / T; }
    template <typename E> static constexpr size_t smem() { return ST * sizeof(E) * ((size_t)T * (kGemmK + 1) + (size_t)kGemmK * (T + 1)); }
};
using GemmSplit = GemmShape<4, 8, 2, 6, false>;
using GemmSplitS = GemmShape<2, 8, 2, 12, false>;    // small tiles: few items, or d that 32 pads
using GemmPlain1 = GemmShape<1, 16, 3, 6, true>;     // 1 to 3: few items
using GemmPlain2 = GemmShape<2, 16, 3, 4, true>;
using GemmPlain3 = GemmShape<3, 16, 3, 3, true>;
using GemmPlain4 = GemmShape<4, 16, 3, 2, true>;
using GemmPlain4F = GemmShape<4, 16, 3, 2, false>;   // d a multiple of 64: nothing to leave out (203 -> 194 us)
using GemmPlain5 = GemmShape<5, 16, 3, 2, true>;
using GemmPlain6 = GemmShape<6, 16, 3, 2, true>;
using GemmWide = GemmShape<2, 16, 2, 2, true>;       // FP64 operands (bound by the FP64 pipe)
inline int sm_count() {   // of the current device
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return 1;
    return std::max(n, 1);
}
// Time of a launch of `items` products in tiles of one shape, in units that scale with d: a CTA alone on an SM
// takes `alone`, a full SM gives one every `each`, and the SMs' CTAs come in whole numbers.
inline double gemm_time(int d, long items, int T, double alone, double each, int sms) {
    const long n = (d + T - 1) / T, ctas = n * n * items;
    return std::max(alone, (double)((ctas + sms - 1) / sms) * each);
}
// Shapes by that model; alone and each as measured at d = 128 (us; launches of 1 and of 400 products):
// split   32 x 32 tiles 24.8 and 9.2, 16 x 16 10.6 and 2.8
// plain   T = 16 .. 96 11, 23, 33, 45, 63, 88 and 4.2, 9.9, 17.6, 33, 46.5, 75
// It picks the fastest shape, or one within 15 % of it, of 1 to 400 products of d = 48 .. 256.  From a product
// an SM on, plain tiles of at least 64: the smaller ones are no faster then (400 of d = 81 133 us as 48 x 48,
// 135 as 96 x 96) and take more of the chip from kernels beside them (a batch of sixteen problems 172.7 against
// 175.2 ms).  By padding alone, few products ran on few SMs: 50 of d = 81 as one 96 x 96 tile each took 62 us a reverse step, now 27;
// an evaluation of d = 81, N = 100 with the Horner series went from 2.02 (32 x 32 tiles) to 2.63 ms.
inline bool gemm_split_small(int d, long items, int sms) {
    return gemm_time(d, items, 16, 10.6, 2.8, sms) < gemm_time(d, items, 32, 24.8, 9.2, sms);
}
inline int gemm_plain_mt(int d, long items, int sms) {
    const double alone[6] = {11, 23, 33, 45, 63, 88}, each[6] = {4.2, 9.9, 17.6, 33, 46.5, 75};
    int best = 4;
    double cost = 1e300;
    for (int mt = items < sms ? 1 : 4; mt <= 6; ++mt) {
        // the smaller tiles only where they are clearly ahead (their CTAs' last rounds cost more than the model says)
        const double c = gemm_time(d, items, 16 * mt, alone[mt - 1], each[mt - 1], sms) * (mt < 4 ? 1.35 : 1.0);
        if (c < cost) {
            cost = c;
            best = mt;
        }
    }
    return best;
}
// position of this thread in its tile
template <class Sh>
struct GemmPos {
    int tx, ty, r0, c0;
    int xw;   // rows x < xw of this warp's threads reach below d in some lane (edge tiles skip the rest)
    __device__ __forceinline__ GemmPos(int tile, int n, int d) {
        ty = threadIdx.x / Sh::G;
        tx = threadIdx.x - ty * Sh::G;
        const int tm = tile / n;
        r0 = tm * Sh::T;
        c0 = (tile - tm * n) * Sh::T;
        const int ty0 = (int)(threadIdx.x & ~31u) / Sh::G;   // the warp's first row
        xw = min(Sh::MT, max(0, (d - r0 - ty0 + Sh::G - 1) / Sh::G));
    }
};

// `mac.run(a, b, xw)` for every k, with the MT operands of each side.  la(row, k, dst) and lb(k, column,
// dst) bring one element of an operand into shared memory (zero past its edge).  The caller has passed
// a barrier since the ring was last read; ends with a barrier.
// AT: A's elements are brought row-fastest (the caller reads A transposed).
template <typename E, class Sh, bool AT = false, typename LA, typename LB, typename Mac>
__device__ __forceinline__ void gemm_loop(unsigned char* smraw, const GemmPos<Sh>& p, int kd, LA la, LB lb, Mac& mac) {
    constexpr int MT = Sh::MT, G = Sh::G, T = Sh::T, ST = Sh::ST, NT = Sh::NT;
    constexpr int asz = T * (kGemmK + 1), bsz = kGemmK * (T + 1), per = T * kGemmK / NT;
    static_assert(T * kGemmK % NT == 0 && NT % kGemmK == 0, "whole passes");
    E* A0 = reinterpret_cast<E*>(smraw);
    E* B0 = A0 + ST * asz;
    auto issue = [&](int st, int k0) {
        E* as = A0 + st * asz;
        E* bs = B0 + st * bsz;
        const int k = threadIdx.x % kGemmK;
#pragma unroll
        for (int q = 0; q < per; ++q) {
            if constexpr (AT) {
                const int idx = threadIdx.x + q * NT, kt = idx / T, r = idx - kt * T;
                la(p.r0 + r, k0 + kt, as + r * (kGemmK + 1) + kt);
            } else {
                const int r = threadIdx.x / kGemmK + q * (NT / kGemmK);
                la(p.r0 + r, k0 + k, as + r * (kGemmK + 1) + k);
            }
        }
#pragma unroll
        for (int q = 0; q < per; ++q) {
            const int idx = threadIdx.x + q * NT, kb = idx / T, c = idx - kb * T;
            lb(k0 + kb, p.c0 + c, bs + kb * (T + 1) + c);
        }
    };
    const int nch = (kd + kGemmK - 1) / kGemmK;
#pragma unroll
    for (int s = 0; s < ST - 1; ++s) {
        if (s < nch) issue(s, s * kGemmK);
        cp_async_commit();
    }
    int st = 0;
    for (int ch = 0; ch < nch; ++ch) {
        cp_async_wait<ST - 2>();
        __syncthreads();   // chunk ch is there for every thread, and every thread is done with chunk ch - 1
        {
            int sn = st + ST - 1;
            if (sn >= ST) sn -= ST;
            if (ch + ST - 1 < nch) issue(sn, (ch + ST - 1) * kGemmK);
            cp_async_commit();
        }
        const E* As = A0 + st * asz + p.ty * (kGemmK + 1);
        const E* Bs = B0 + st * bsz + p.tx;
        if (++st == ST) st = 0;
        const int kmax = min(kGemmK, kd - ch * kGemmK);
#pragma unroll 4
        for (int k = 0; k < kmax; ++k) {
            E a[MT], b[MT];
#pragma unroll
            for (int x = 0; x < MT; ++x) a[x] = As[G * x * (kGemmK + 1) + k];
#pragma unroll
            for (int y = 0; y < MT; ++y) b[y] = Bs[k * (T + 1) + G * y];
            mac.run(a, b, Sh::SKIP ? p.xw : MT);
        }
    }
    __syncthreads();
}
// one k of a split product: grid parts' sums (exact) and cross terms
template <int MT>
__device__ __forceinline__ void split_mac(float (&acc)[MT][MT][4], const float4 (&a)[MT], const float4 (&b)[MT]) {
#pragma unroll
    for (int y = 0; y < MT; ++y) {
        const float2 bf = make_float2(b[y].x + b[y].z, b[y].y + b[y].w);
#pragma unroll
        for (int x = 0; x < MT; ++x) {
            float* c = acc[x][y];
            c[0] = fmaf(a[x].x, b[y].x, c[0]);
            c[0] = fmaf(-a[x].y, b[y].y, c[0]);
            c[1] = fmaf(a[x].x, b[y].y, c[1]);
            c[1] = fmaf(a[x].y, b[y].x, c[1]);
            c[2] = fmaf(a[x].x, b[y].z, c[2]);
            c[2] = fmaf(-a[x].y, b[y].w, c[2]);
            c[2] = fmaf(a[x].z, bf.x, c[2]);
            c[2] = fmaf(-a[x].w, bf.y, c[2]);
            c[3] = fmaf(a[x].x, b[y].w, c[3]);
            c[3] = fmaf(a[x].y, b[y].z, c[3]);
            c[3] = fmaf(a[x].z, bf.y, c[3]);
            c[3] = fmaf(a[x].w, bf.x, c[3]);
        }
    }
}

// accumulators: a split product, the same operands multiplied plainly (A's full value, B in full form), or
// a plain product
template <int MT>
struct MacSplit {
    float acc[MT][MT][4] = {};
    __device__ __forceinline__ void run(const float4 (&a)[MT], const float4 (&b)[MT], int) { split_mac(acc, a, b); }
};
template <int MT>
struct MacFull {
    float acc[MT][MT][4] = {};
    __device__ __forceinline__ void run(const float4 (&a)[MT], const float4 (&b)[MT], int) {
#pragma unroll
        for (int x = 0; x < MT; ++x) {
            const float2 af = make_float2(a[x].x + a[x].z, a[x].y + a[x].w);
#pragma unroll
            for (int y = 0; y < MT; ++y) {
                float* c = acc[x][y];
                c[0] = fmaf(af.x, b[y].x, c[0]);
                c[0] = fmaf(-af.y, b[y].y, c[0]);
                c[1] = fmaf(af.x, b[y].y, c[1]);
                c[1] = fmaf(af.y, b[y].x, c[1]);
            }
        }
    }
};
template <typename C, int MT>
struct MacPlain {
    C acc[MT][MT] = {};
    __device__ __forceinline__ void run(const C (&a)[MT], const C (&b)[MT], int xw) {
#pragma unroll
        for (int x = 0; x < MT; ++x) {
            if (x >= xw) break;
#pragma unroll
            for (int y = 0; y < MT; ++y) cfma(acc[x][y], a[x], b[y]);
        }
    }
};

}  // namespace qoc
