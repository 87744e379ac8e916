// Tensor-core products of the large-d adjoint with exact leading-level accumulation (BF16_SPLIT).
//
// The reverse-mode adjoint of the truncated series (the exact derivative of Eqs. 9-10 applied to
// Ubar, Appendix A) needs FP32-accurate complex products.  The tensor core's FP32 accumulator
// truncates, and a truncation bias in the leading part of a product adds up over the Horner and
// squaring recursion, so the leading part is made exact instead (an integer-slice splitting in
// the manner of Ozaki's error-free matrix product):
//   * every row of an A operand (every column of a B operand) is scaled by a power of two 2^e
//     with max |entry| < 2^e; the scaled value y = x 2^-e (|y| < 1) is cut into four slices of
//     seven bits, y = sum_s a_s 2^(-7 (s + 1)) + r, |r| <= 2^-29, with integers |a_0| <= 128 and
//     |a_s| <= 64 after it;
//   * the A planes hold a_s 2^(7 - 7 s) and the B planes b_t 2^(-7 t) (BF16, exact), so the MMA
//     of slices s and t contributes a_s b_t 2^(7 - 7 (s + t)): the pair (0, 0) is 2^7 times an
//     integer product of at most 2^14, and over k < 512 (two products per k for each complex
//     part) its accumulator stays an exact multiple of 2^7 below 2^31, whatever the rounding of
//     the FP32 accumulation;
//   * the nine pairs with 1 <= s + t <= 3 accumulate, already weighted, into a second FP32
//     accumulator whose size is about 2^-7 of the leading one, so its truncation errors stay far
//     below the FP32 rounding of the result; the pairs with s + t >= 4 (below 2^-28) are dropped;
//   * the epilogue scales the sum of the two accumulators by 2^(eA + eB - 21) (exact).
// Measured in emulation on identity-dominant Horner matrices this is as accurate as an FP32 SIMT
// product (and several times more accurate on dense ones); four six-bit slices scaled the same
// way lose the small off-diagonal entries of I + X / i.
//
// The forward products of the Paterson-Stockmeyer form (X^2, X^3, the chain products, the
// squarings; Eqs. 9-10) need the accuracy of the split SIMT products (about 2^-36 of the scale),
// so there the operands are value pairs cut into six seven-bit slices (42 bits), and the slice
// levels s + t = 0, 1 and 2 accumulate exactly in accumulators of their own (pre-weighted by
// 2^(7 - 7 (s + t)), level L is a multiple of 2^(7 - 7L); per k and complex part at most two
// products of 2^21, 2^14 and 2^14.3 for L = 0, 1, 2, so the sums stay below 2^24 units of their
// granularity for d <= 384), the levels 3 to 5 into a fourth.  That last accumulator is the only
// inexact one: the tensor core's accumulation truncates, and in emulation of a truncating FP32
// accumulator per MMA the product of two identity-dominant matrices keeps a relative error of
// 1.5e-11 (with levels 2 to 5 in one accumulator: 7.9e-9).  128 x 64 tiles keep the eight FP32
// accumulators within the tensor memory, and the epilogue adds the Paterson-Stockmeyer block in
// pair arithmetic and writes grid-split value pairs.
//
// k_oz_mm computes 128 x 128 tiles of C = alpha A B (+ C) (+ I), a persistent CTA per SM:
// warp 0 issues the TMA loads of a three-stage ring (one stage: the eight slice planes of A and
// of B for a 16-wide K chunk, four to a SWIZZLE_128B tile, 64 KB), warp 1 issues the tcgen05.mma (kind::f16,
// BF16 in, FP32 accumulators in tensor memory: leading re, leading im, rest re, rest im, 128
// columns each) and commits each stage back to the producer, warps 2-9 read tensor memory with
// tcgen05.ld into registers, hand it back to the MMA warp and then add and write the tile while the next
// one's products run.  Every mbarrier wait is bounded; a wait that runs out sets
// kErrTimeout in DevParams.err and the CTA stops issuing, waits (bounded) for its copies in
// flight, frees its tensor memory and returns.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <type_traits>

#include "qoc_device.cuh"
#include "qoc_internal.h"
#include "qoc_tree.cuh"

namespace qoc {

namespace {

constexpr int BM = 128, BK = 16;                   // BK in BF16 elements
constexpr int GRP = 4;                             // planes side by side in a 128-byte row (per K chunk)
constexpr int SBITS = 7;
constexpr int EPI_WARPS = 8;                       // two per tensor-memory lane quarter
constexpr int NTHREADS = 64 + 32 * EPI_WARPS;      // producer warp, MMA warp, epilogue warps

// One product configuration: NS slices per value, BN-wide tiles, NLEV accumulator levels (every
// level below NLEV - 1 exact, the last one taking the remaining slice pairs), NST stages.
template <int NS_, int BN_, int NLEV_, int NST_>
struct OzCfg {
    static constexpr int NS = NS_, BN = BN_, NLEV = NLEV_, NST = NST_;
    static constexpr int NPART = 2 * NS;                      // re slices, then im slices
    static constexpr int NG = NPART / GRP;                    // groups of planes
    static constexpr int TILE_A = BM * BK * 2 * GRP;          // one group's A tile, 16 KB
    static constexpr int TILE_B = BN * BK * 2 * GRP;          // one group's B tile
    static constexpr int STAGE = NG * (TILE_A + TILE_B);
    static_assert(NPART % GRP == 0, "whole groups");
    static constexpr int SMEM = NST * STAGE + 1024;           // + alignment slack
    static constexpr uint32_t TMEM_COLS = 512;
};
using AdjCfg = OzCfg<kOzSlices, 128, 2, 3>;     // 64 KB stages, four 128-column accumulators
using FwdCfg = OzCfg<kOzFwdSlices, 64, 4, 3>;   // 72 KB stages, eight 64-column accumulators
static_assert(2 * AdjCfg::NLEV * AdjCfg::BN <= 512 && 2 * FwdCfg::NLEV * FwdCfg::BN <= 512, "tensor memory");
static_assert(AdjCfg::SMEM <= (int)kMaxDynSmem && FwdCfg::SMEM <= (int)kMaxDynSmem, "shared memory");
constexpr uint32_t WAIT_LIMIT = 1u << 24;
constexpr uint32_t WAIT_LIMIT_TEST = 1u << 12;     // fault-injection runs

__device__ __forceinline__ uint32_t su32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint64_t* b, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(su32(b)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* b, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(su32(b)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_wait(uint64_t* b, uint32_t parity, uint32_t limit) {
    for (uint32_t it = 0; it < limit; ++it) {
        uint32_t done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
            : "=r"(done)
            : "r"(su32(b)), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}
__device__ __forceinline__ void tma_3d(void* smem, const CUtensorMap* map, int x, int y, int z, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(
            su32(smem)),
        "l"((uint64_t)map), "r"(x), "r"(y), "r"(z), "r"(su32(bar))
        : "memory");
}
// UMMA shared-memory descriptor: K-major, SWIZZLE_128B (one 128-byte row per M / N index holding the
// K chunk of four planes, 8-row groups 1024 bytes apart), descriptor version 1.  lo: sdesc_lo of the
// group's tile (1024-byte aligned) plus 2 per plane (its 32 bytes), in units of 16 bytes.
__device__ __forceinline__ uint32_t sdesc_lo(uint32_t smem) { return ((smem >> 4) & 0x3FFFu) | (1u << 16); }
__device__ __forceinline__ uint64_t sdesc(uint32_t lo) {
    return ((uint64_t)((1024u >> 4) | (1u << 14) | (2u << 29)) << 32) | lo;
}
// one lane of a converged warp: the MMA operands are in uniform registers, which the compiler finds by
// itself only where the choice of the lane is this instruction and all around it is uniform.  (Under
// `lane == 0` an MMA took 72 cycles to issue whatever its size: 1200 us a forward product of 450 items
// at d = 256, 939 with the choice alone by elect.)
__device__ __forceinline__ bool elect() {
    uint32_t p;
    asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}" : "=r"(p));
    return p != 0;
}
// One MMA of a run that shares its A operand (and its descriptor): the first of the run fills the A
// collector from shared memory, the others read A from it
enum { A_FILL, A_USE, A_LAST, A_NONE };
#define QOC_MMA(OP)                                                                                                   \
    asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"                                                        \
                 " tcgen05.mma.cta_group::1.kind::f16.collector::a::" OP " [%0], %1, %2, %3, p;\n}" ::"r"(tmem),       \
                 "l"(a), "l"(b), "r"(idesc), "r"(acc)                                                                 \
                 : "memory")
__device__ __forceinline__ void mma_bf16(uint32_t tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc, int use) {
    if (use == A_FILL) QOC_MMA("fill");
    else if (use == A_USE) QOC_MMA("use");
    else if (use == A_LAST) QOC_MMA("lastuse");
    else QOC_MMA("discard");
}
#undef QOC_MMA
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(su32(bar))
                 : "memory");
}
// 16 columns of this lane's row; the values may be read after tmem_wait
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, "
        "[%16];"
        : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]), "=f"(r[4]), "=f"(r[5]), "=f"(r[6]), "=f"(r[7]), "=f"(r[8]),
          "=f"(r[9]), "=f"(r[10]), "=f"(r[11]), "=f"(r[12]), "=f"(r[13]), "=f"(r[14]), "=f"(r[15])
        : "r"(taddr));
}
// the loads before it have landed; their values pass through an empty asm after the wait, so no use of
// them can move above it
__device__ __forceinline__ void tmem_pass(float (&r)[16]) {
    asm volatile("" : "+f"(r[0]), "+f"(r[1]), "+f"(r[2]), "+f"(r[3]), "+f"(r[4]), "+f"(r[5]), "+f"(r[6]), "+f"(r[7]),
                 "+f"(r[8]), "+f"(r[9]), "+f"(r[10]), "+f"(r[11]), "+f"(r[12]), "+f"(r[13]), "+f"(r[14]), "+f"(r[15]));
}
__device__ __forceinline__ void tmem_wait(float (&a)[16], float (&b)[16], float (&c)[16], float (&d)[16]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
    tmem_pass(a);
    tmem_pass(b);
    tmem_pass(c);
    tmem_pass(d);
}

// exponent e with |x| < 2^e for the largest |x| of a row or column (0 for an all-zero one)
__device__ __forceinline__ int scale_exp(float m) {
    int e = 0;
    if (m > 0.f) frexpf(m, &e);
    return e;
}
// NS seven-bit slices of y = (hi + lo) 2^-e (|y| < 1), weighted for their operand role: A planes
// hold a_s 2^(7 - 7 s), B planes b_s 2^(-7 s).  The pair is normalised first (a grid-split pair
// on a grid much coarser than the row's largest value has a low part far above the high part's
// last bit, which would push the slices past the eight bits BF16 holds exactly); the residual is
// then carried as an error-free pair: a_s = rint(H), (H, L) <- TwoSum(H - a_s, L) 2^7, exact at
// every step.  FP32 values (PAIR false) need no second part: H - a_s is exact.
__device__ __forceinline__ float rint_small(float h) {   // |h| < 2^22, by two additions: FRND has a quarter of their rate
    const float m = 12582912.0f;                         // 1.5 * 2^23
    return __fadd_rn(__fadd_rn(h, m), -m);
}
template <int NS, bool PAIR>
__device__ __forceinline__ void slices(float hi, float lo, int e, bool role_a, float (&q)[NS]) {
    float h0 = hi, l0 = 0.f;
    if constexpr (PAIR) two_sum(hi, lo, h0, l0);
    float h = ldexpf(h0, SBITS - e), l = PAIR ? ldexpf(l0, SBITS - e) : 0.f;
    float w = role_a ? (float)(1 << SBITS) : 1.0f;
#pragma unroll
    for (int s = 0; s < NS; ++s) {
        const float a = rint_small(h);
        q[s] = a * w;
        if constexpr (PAIR) {
            float t, u;
            two_sum(h - a, l, t, u);
            h = t * (float)(1 << SBITS);
            l = u * (float)(1 << SBITS);
        } else {
            h = (h - a) * (float)(1 << SBITS);
        }
        w *= 1.0f / (float)(1 << SBITS);
    }
}
// a complex element as value pairs (re_hi, re_lo, im_hi, im_lo)
__device__ __forceinline__ float4 as_pairs(float2 v) { return make_float4(v.x, 0.f, v.y, 0.f); }
__device__ __forceinline__ float4 as_pairs(float4 v) { return make_float4(v.x, v.z, v.y, v.w); }

}  // namespace

// Planes are stored in groups of four: a row of a group holds, for each 16-wide K chunk, the chunk of the
// group's four planes side by side (128 bytes), so one SWIZZLE_128B tile brings four planes of a chunk.
// (With a plane per tile and 32-byte rows a forward product of 150 items at d = 256 took 477 us instead of
// 458 and an adjoint one 269 instead of 250; the slicer pays 5 % for it.)  Group (item, matrix, g):
template <int NPART>
__host__ __device__ inline size_t oz_group(int item, int mats, int mat, int g) {
    return ((size_t)item * mats + mat) * (NPART / GRP) + g;
}
__host__ __device__ inline int oz_row(int d) { return (d + BK - 1) / BK * BK * GRP; }   // elements of a group's row
// element k of plane `part` within a row of its group
__device__ __forceinline__ size_t oz_at(int part, int k) { return (size_t)(k / BK) * (BK * GRP) + (part % GRP) * BK + k % BK; }

// ------------------------------------------------------------------------------------------
// slicing: FP32 complex d x d matrices (row-major, item-strided) -> exponents and BF16 planes
// ------------------------------------------------------------------------------------------
// Row layout (A operand): plane row r = row r of M, exponent per row.  Column layout (B operand,
// K-major): plane row c = column c of M, exponent per column (no conjugation is applied).  Conjugated
// column layout: M^dag as an A operand, plane row c = conjugated column c of M.  Conjugated row layout:
// M^dag as a B operand.
// Eight consecutive elements of one plane row (half a K chunk), as one 16-byte store
__device__ __forceinline__ void store8(__nv_bfloat16* dst, const float (&v)[8]) {
    uint4 w;
    __nv_bfloat162 h;
    h = __floats2bfloat162_rn(v[0], v[1]);
    w.x = *reinterpret_cast<uint32_t*>(&h);
    h = __floats2bfloat162_rn(v[2], v[3]);
    w.y = *reinterpret_cast<uint32_t*>(&h);
    h = __floats2bfloat162_rn(v[4], v[5]);
    w.z = *reinterpret_cast<uint32_t*>(&h);
    h = __floats2bfloat162_rn(v[6], v[7]);
    w.w = *reinterpret_cast<uint32_t*>(&h);
    *reinterpret_cast<uint4*>(dst) = w;
}

// the slices of eight consecutive elements k0 .. k0 + 7 of plane row `row` (zero past d), written as
// 16-byte stores into the row's 2 NS planes; gsz: elements of a group (d rows)
template <int NS, bool PAIR>
__device__ __forceinline__ void put8(__nv_bfloat16* __restrict__ planes, size_t pbase, size_t gsz, int row, int rowlen,
                                     int k0, const float4 (&q)[8], int e, bool role_a) {
    float sr[8][NS], si[8][NS];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        slices<NS, PAIR>(q[i].x, q[i].y, e, role_a, sr[i]);
        slices<NS, PAIR>(q[i].z, q[i].w, e, role_a, si[i]);
    }
#pragma unroll
    for (int s = 0; s < NS; ++s) {
        float vr[8], vi[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            vr[i] = sr[i][s];
            vi[i] = si[i][s];
        }
        __nv_bfloat16* pr = planes + (size_t)row * rowlen;
        store8(pr + (pbase + s / GRP) * gsz + oz_at(s, k0), vr);
        store8(pr + (pbase + (NS + s) / GRP) * gsz + oz_at(NS + s, k0), vi);
    }
}

template <int NS, typename In>
__global__ void __launch_bounds__(256)
k_oz_slice(OzSliceJobs jobs, __nv_bfloat16* __restrict__ planes, int* __restrict__ exps, int d) {
    constexpr int NPART = 2 * NS;
    constexpr bool PAIR = std::is_same_v<In, float4>;
    constexpr int KT = 64;                       // rows of M per staged tile (column layout)
    __shared__ In tile[KT][33];
    __shared__ float cmax[8][32];
    __shared__ int cexp[32];
    const OzSliceJob jb = jobs.job[blockIdx.z];
    const int item = blockIdx.y, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int it = jobs.item0 + item, se = jobs.count ? it / jobs.count : 0;   // member, and its item
    const In* M = static_cast<const In*>(jb.src) + se * jb.estride + (size_t)(it - se * jobs.count) * jb.stride;
    const int rowlen = oz_row(d), dk = rowlen / GRP;   // dk: d rounded up to whole K chunks
    const size_t gsz = (size_t)d * rowlen;
    const size_t pbase = oz_group<NPART>(item, jobs.mats, jb.mat, 0);
    const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
    // the exponent comes from the rounded values |re|, |im| (a pair's sum rounded up to 2^e only
    // raises e: conservative)
    auto mag = [](float4 q) { return fmaxf(fabsf(q.x + q.y), fabsf(q.z + q.w)); };
    if (jb.col == 0 || jb.col == 3) {
        // row layout: one warp per row, each lane eight consecutive columns per 256-column chunk
        // (d <= 512: at most two chunks, held in registers between the maximum and the slicing)
        const int r = blockIdx.x * 8 + warp;
        if (r >= d) return;
        float4 v[2][8];
        float m = 0.f;
#pragma unroll
        for (int ch = 0; ch < 2; ++ch)
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int b = ch * 256 + lane * 8 + i;
                v[ch][i] = b < d ? as_pairs(M[(size_t)r * d + b]) : zero4;
                m = fmaxf(m, mag(v[ch][i]));
            }
        for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        const int e = scale_exp(m);
        if (lane == 0) exps[((size_t)item * jobs.mats + jb.mat) * d + r] = e;
#pragma unroll
        for (int ch = 0; ch < 2; ++ch) {
            const int b0 = ch * 256 + lane * 8;
            if (b0 >= dk) continue;
            if (jb.col == 3) {
#pragma unroll
                for (int i = 0; i < 8; ++i) v[ch][i].z = -v[ch][i].z, v[ch][i].w = -v[ch][i].w;
            }
            put8<NS, PAIR>(planes, pbase, gsz, r, rowlen, b0, v[ch], e, jb.col != 3);
        }
        return;
    }
    // column layout: 32 columns c0 .. c0 + 31 per CTA; plane row c (a column of M) with k along it
    const int c0 = blockIdx.x * 32;
    if (c0 >= d) return;
    const int c = c0 + lane;
    float m = 0.f;
    if (c < d)
        for (int k = warp; k < d; k += 8) m = fmaxf(m, mag(as_pairs(M[(size_t)k * d + c])));
    cmax[warp][lane] = m;
    __syncthreads();
    if (warp == 0) {
        float mm = cmax[0][lane];
        for (int w = 1; w < 8; ++w) mm = fmaxf(mm, cmax[w][lane]);
        const int e = scale_exp(mm);
        cexp[lane] = e;
        if (c < d) exps[((size_t)item * jobs.mats + jb.mat) * d + c] = e;
    }
    __syncthreads();
    // tiles of KT rows: staged with the lanes along the columns (coalesced reads), then thread t slices
    // column (t / 2) % 32 over eight rows of the tile: two neighbours write one 32-byte sector of a plane
    // (with the lanes along the columns each wrote half a sector: d = 256, 450 items, four matrices 577 us
    // instead of 453)
    const int tc = (tid >> 1) & 31, tk = (tid >> 6) * 16 + (tid & 1) * 8;
    for (int k0 = 0; k0 < d; k0 += KT) {
        for (int q = warp; q < KT; q += 8) {
            const int k = k0 + q;
            tile[q][lane] = (k < d && c < d) ? M[(size_t)k * d + c] : In{};
        }
        __syncthreads();
        const int cc = c0 + tc, kk = k0 + tk;
        if (cc < d && kk < dk) {
            float4 q8[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                q8[i] = as_pairs(tile[tk + i][tc]);
                if (jb.col == 2) q8[i].z = -q8[i].z, q8[i].w = -q8[i].w;
            }
            put8<NS, PAIR>(planes, pbase, gsz, cc, rowlen, kk, q8, cexp[tc], jb.col == 2);
        }
        __syncthreads();
    }
}

// The forward epilogue's job: out = A B (kind 1) or A B + c0 I + c1 X + c2 X^2 (kind 2), written as
// value pairs grid-split with `magic` (item stride ostride)
struct OzFwdEpi {
    float4* out;
    long long ostride;
    int kind;
    float magic;
    const float4* X;
    const float4* X2;
    float2 c0, c1, c2;
    float2* ct;             // optional: the output's rounded conjugate transpose (item stride cts)
    size_t cts;
};

struct OzAdjEpi {};
// The tree's epilogue: out = A B grid-split with its columns' magics mo (none: of the propagators' exponent), the
// optional second output and the optional rounded (scaled) value of TreeMm
struct OzTreeEpi {
    TreeMm t;
    int item0;
};

// ------------------------------------------------------------------------------------------
// 128 x BN output tiles of the jobs' items: adjoint products (OzAdjEpi) C = alpha A B (+ beta C) (+ I)
// in FP32; forward products (OzFwdEpi) and the tree's (OzTreeEpi) as value pairs.  A persistent CTA per SM takes tiles
// blockIdx.x, + gridDim.x, ..: while the epilogue warps add and write one tile, the products of the next
// run, and only the read-out of tensor memory stands between the products of two tiles.
// A forward product at d = 256 (450 items, us): 1375 with a CTA per tile (from 150 items); 1204 persistent; 929 with the
// MMAs' operands in uniform registers (elect); 742 with A read once per run by the collector, 1.71 PFLOP/s
// of executed MMAs, 0.90 of the measured cuBLAS burst rate.  What is left: the copies alone (4.2 GB of plane tiles through L2 a launch, 2.8 GB of HBM traffic) take 599,
// the MMAs 530.  An adjoint product (mean of single and double launches): 750, 622, 608, 583, the copies
// alone 490.
// ------------------------------------------------------------------------------------------
template <class Cfg, class Epi>
__global__ void __launch_bounds__(NTHREADS, 1)
k_oz_mm(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB, OzJobs jobs, int njobs,
        int items, Epi fe, const int* __restrict__ exps, int d, DevParams* __restrict__ prm) {
    constexpr bool FWD = !std::is_same_v<Epi, OzAdjEpi>;
    constexpr int NS = Cfg::NS, BN = Cfg::BN, NLEV = Cfg::NLEV, NST = Cfg::NST, NPART = Cfg::NPART;
    constexpr int TILE_A = Cfg::TILE_A, TILE_B = Cfg::TILE_B, STAGE = Cfg::STAGE, NG = Cfg::NG;
    extern __shared__ __align__(1024) unsigned char smraw[];
    unsigned char* base = reinterpret_cast<unsigned char*>(((uintptr_t)smraw + 1023) & ~(uintptr_t)1023);
    __shared__ __align__(8) uint64_t full[NST], empty[NST], acc_full, acc_empty;
    __shared__ uint32_t tmem_holder;
    __shared__ int skip;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // once a wait has run out in this evaluation, later launches skip their work (the result is
    // reported as QOC_ERR_TIMEOUT); thread 0 decides for the whole CTA
    if (tid == 0) skip = (*(volatile int*)&prm->err & kErrTimeout) != 0;
    __syncthreads();
    if (skip) return;
    const uint32_t limit = jobs.fault ? WAIT_LIMIT_TEST : WAIT_LIMIT;
    const int ntn = (d + BN - 1) / BN, per_item = ((d + BM - 1) / BM) * ntn;
    const int per_job = per_item * items, total = per_job * njobs;
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(&tmem_holder)),
                     "r"(Cfg::TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int b = 0; b < NST; ++b) {
            mbar_init(&full[b], 1);
            mbar_init(&empty[b], 1);
        }
        mbar_init(&acc_full, 1);
        mbar_init(&acc_empty, EPI_WARPS);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_holder;
    const int nk = (d + BK - 1) / BK;
    auto job_of = [&](int t) { return jobs.j[t / per_job]; };

    if (warp == 0 && lane == 0) {
        // ---- producer: the plane groups of A and of B for one K chunk per stage ----
        bool ok = true;
        int last_issued[NST];
#pragma unroll
        for (int b = 0; b < NST; ++b) last_issued[b] = -1;
        int g = 0;   // stages so far, over all tiles
        for (int t = blockIdx.x; t < total && ok; t += gridDim.x) {
            const OzJob jb = job_of(t);
            const int rest = t % per_job, item = rest / per_item, tile = rest - item * per_item;
            const int r0 = (tile / ntn) * BM, c0 = (tile % ntn) * BN;
            for (int s = 0; s < nk; ++s, ++g) {
                const int b = g % NST;
                if (g >= NST && !mbar_wait(&empty[b], (uint32_t)((g / NST - 1) & 1), limit)) {
                    ok = false;
                    break;
                }
                if (jobs.fault && g == 0) continue;   // fault injection: the first copy is withheld
                unsigned char* st = base + b * STAGE;
                mbar_expect_tx(&full[b], STAGE);
                for (int q = 0; q < NG; ++q) {
                    tma_3d(st + q * TILE_A, &mapA, s * BK * GRP, r0, (int)oz_group<NPART>(item, jobs.mats, jb.a_mat, q), &full[b]);
                    tma_3d(st + NG * TILE_A + q * TILE_B, &mapB, s * BK * GRP, c0,
                           (int)oz_group<NPART>(item, jobs.mats, jb.b_mat, q), &full[b]);
                }
                last_issued[b] = g;
            }
        }
        if (!ok) atomicOr(&prm->err, kErrTimeout);
        // every copy issued into this CTA's shared memory lands before the CTA can leave (bounded)
        for (int b = 0; b < NST; ++b)
            if (last_issued[b] >= 0) mbar_wait(&full[b], (uint32_t)((last_issued[b] / NST) & 1), limit);
    } else if (warp == 1) {
        // ---- MMA issuer: the whole warp goes through the waits, one lane issues ----
        // instruction descriptor: D f32, A/B bf16, both K-major, N = BN, M = 128
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
        const uint32_t idesc_nA = idesc | (1u << 13);   // negate A
        const uint32_t acc0 = __shfl_sync(0xffffffffu, tmem, 0);
        const uint32_t lo0 = sdesc_lo((su32(smraw) + 1023) & ~1023u);
        bool ok = true;
        int b = 0, n = 0;        // stage, tiles so far
        uint32_t par = 0;        // the stage's phase
        for (int t = blockIdx.x; t < total && ok; t += gridDim.x, ++n) {
            if (n > 0) ok = __all_sync(0xffffffffu, mbar_wait(&acc_empty, (uint32_t)((n - 1) & 1), limit));   // read out
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            for (int s = 0; s < nk && ok; ++s) {
                ok = __all_sync(0xffffffffu, mbar_wait(&full[b], par, limit));
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                if (elect()) {
                    const uint32_t lo = lo0 + (uint32_t)b * (STAGE >> 4);
                    // plane p: group p / 4, 32 bytes per plane within its rows
                    auto dA = [&](int p) { return sdesc(lo + (uint32_t)((p / GRP) * TILE_A + (p % GRP) * (BK * 2)) / 16); };
                    auto dB = [&](int p) {
                        return sdesc(lo + (uint32_t)(NG * TILE_A + (p / GRP) * TILE_B + (p % GRP) * (BK * 2)) / 16);
                    };
#pragma unroll
                    for (int sa = 0; sa < NS; ++sa) {
                        // slice level sa + sb goes to its own accumulators below NLEV - 1, the rest to the last
                        const int nb = NS - sa;
                        auto acc = [&](int sb) { return acc0 + (uint32_t)(2 * min(sa + sb, NLEV - 1) * BN); };
                        // re += Ar Br, im += Ar Bi: one run of A operand Ar.  The first MMA into each accumulator
                        // (sa = 0, sb = its level) overwrites it
#pragma unroll
                        for (int sb = 0; sb < nb; ++sb) {
                            const uint32_t en = (s > 0 || sa > 0 || sb > NLEV - 1) ? 1u : 0u;
                            mma_bf16(acc(sb), dA(sa), dB(sb), idesc, en, sb == 0 ? A_FILL : A_USE);
                            mma_bf16(acc(sb) + BN, dA(sa), dB(NS + sb), idesc, en, sb == nb - 1 ? A_LAST : A_USE);
                        }
                        // re -= Ai Bi, then im += Ai Br: the negation goes with A, so a run each
#pragma unroll
                        for (int neg = 1; neg >= 0; --neg)
#pragma unroll
                            for (int sb = 0; sb < nb; ++sb) {
                                const int use = nb == 1 ? A_NONE : sb == 0 ? A_FILL : sb == nb - 1 ? A_LAST : A_USE;
                                mma_bf16(acc(sb) + (neg ? 0 : BN), dA(NS + sa), dB(neg ? NS + sb : sb),
                                         neg ? idesc_nA : idesc, 1, use);
                            }
                    }
                    mma_commit(&empty[b]);   // the stage is free once these MMAs have read it
                    if (s == nk - 1) mma_commit(&acc_full);
                }
                __syncwarp();
                if (++b == NST) {
                    b = 0;
                    par ^= 1;
                }
            }
        }
        if (!ok && lane == 0) atomicOr(&prm->err, kErrTimeout);
    } else if (warp >= 2) {
        // ---- epilogue warp: 32 tile rows (the lane quarter of tensor memory it may read, a row a lane)
        // and half the columns, in registers from the read-out on; a lane's columns are consecutive in
        // memory, so its 16-byte (8-byte) accesses fill the sectors of its row one after another, under
        // the next tile's products ----
        constexpr int HC = BN / 2;
        const int q4 = warp & 3, half = (warp - 2) >> 2;
        int n = 0;
        for (int t = blockIdx.x; t < total; t += gridDim.x, ++n) {
            const OzJob jb = job_of(t);
            const int rest = t % per_job, item = rest / per_item, tile = rest - item * per_item;
            const int row = (tile / ntn) * BM + q4 * 32 + lane, ch0 = (tile % ntn) * BN + half * HC;
            const int ncols = min(HC, d - ch0);
            const int* eBp = exps + ((size_t)item * jobs.mats + jb.b_mat) * d;
            const int eA = row < d ? exps[((size_t)item * jobs.mats + jb.a_mat) * d + row] : 0;
            int eB[HC / 32];   // this lane's columns' exponents, broadcast by shuffle
#pragma unroll
            for (int j = 0; j < HC / 32; ++j) eB[j] = ch0 + 32 * j + lane < d ? eBp[ch0 + 32 * j + lane] : 0;
            float mB = 0.f;   // the tree's: its column's grid, likewise
            if constexpr (std::is_same_v<Epi, OzTreeEpi>) {
                static_assert(HC == 32, "a column a lane");
                mB = !fe.t.mo ? grid_magic(prm->eu) : (ch0 + lane < d ? fe.t.mo[ch0 + lane] : 0.f);
            }
            if (!__all_sync(0xffffffffu, mbar_wait(&acc_full, (uint32_t)(n & 1), limit))) {
                if (lane == 0) atomicOr(&prm->err, kErrTimeout);
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t lane_base = tmem + ((uint32_t)(q4 * 32) << 16) + (uint32_t)(half * HC);
            std::conditional_t<FWD, float4, float2> res[HC];   // FWD: (re_hi, im_hi, re_lo, im_lo)
#pragma unroll
            for (int cc = 0; cc < HC; cc += 16) {
                if constexpr (!FWD) {
                    float lr[16], li[16], rr[16], ri[16];
                    tmem_ld16(lane_base + (uint32_t)cc, lr);
                    tmem_ld16(lane_base + (uint32_t)(BN + cc), li);
                    tmem_ld16(lane_base + (uint32_t)(2 * BN + cc), rr);
                    tmem_ld16(lane_base + (uint32_t)(3 * BN + cc), ri);
                    tmem_wait(lr, li, rr, ri);
#pragma unroll
                    for (int q = 0; q < 16; ++q) {
                        const int e = __shfl_sync(0xffffffffu, eB[(cc + q) / 32], (cc + q) % 32);
                        const float sc = ldexpf(jb.alpha, eA + e - 3 * SBITS);
                        res[cc + q] = make_float2((lr[q] + rr[q]) * sc, (li[q] + ri[q]) * sc);
                    }
                } else {
                    // the three exact levels summed without error, the remainder level added to the low
                    // part; every scaling is by a power of two
                    static_assert(!FWD || NLEV == 4, "three exact levels and a remainder");
#pragma unroll
                    for (int part = 0; part < 2; ++part) {   // re, then im
                        float a0[16], a1[16], a2[16], a3[16];
                        tmem_ld16(lane_base + (uint32_t)(part * BN + cc), a0);
                        tmem_ld16(lane_base + (uint32_t)((2 + part) * BN + cc), a1);
                        tmem_ld16(lane_base + (uint32_t)((4 + part) * BN + cc), a2);
                        tmem_ld16(lane_base + (uint32_t)((6 + part) * BN + cc), a3);
                        tmem_wait(a0, a1, a2, a3);
#pragma unroll
                        for (int q = 0; q < 16; ++q) {
                            float h, l, h2, l2;
                            two_sum(a0[q], a1[q], h, l);
                            two_sum(h, a2[q], h2, l2);
                            l = l + l2 + a3[q];
                            if (part == 0) {
                                res[cc + q].x = h2;
                                res[cc + q].z = l;
                            } else {
                                res[cc + q].y = h2;
                                res[cc + q].w = l;
                            }
                        }
                    }
                }
            }
            // tensor memory is read: the next tile's products may start
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(su32(&acc_empty)) : "memory");
            if constexpr (!FWD) {
                float2* out = jb.out + (size_t)item * jb.ostride + (size_t)row * d + ch0;
#pragma unroll
                for (int c8 = 0; c8 < HC; c8 += 8) {
                    float2 old[8];
                    if (jb.beta) {
#pragma unroll
                        for (int q = 0; q < 8; ++q)
                            old[q] = (row < d && c8 + q < ncols) ? out[c8 + q] : make_float2(0.f, 0.f);
                    }
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        if (row >= d || c8 + q >= ncols) continue;
                        float2 v = res[c8 + q];
                        if (jb.beta) {
                            v.x += old[q].x;
                            v.y += old[q].y;
                        }
                        if (jb.ident && row == ch0 + c8 + q) v.x += 1.0f;
                        out[c8 + q] = v;
                    }
                }
            } else if constexpr (std::is_same_v<Epi, OzTreeEpi>) {
                const TreeMm& tm = fe.t;
                const int it = fe.item0 + item, te = it / tm.count, ti = it - te * tm.count;
                const size_t o0 = (size_t)row * d + ch0;
#pragma unroll
                for (int q = 0; q < HC; ++q) {
                    const int e = __shfl_sync(0xffffffffu, eB[0], q);
                    const float mo = __shfl_sync(0xffffffffu, mB, q);
                    if (row >= d || q >= ncols) continue;
                    const float sc = ldexpf(1.0f, eA + e - 3 * SBITS);
                    tree_store(tm, te, ti, o0 + q, ch0 + q, make_float4(res[q].x * sc, res[q].y * sc, res[q].z * sc, res[q].w * sc), mo);
                }
            } else {
                const size_t o0 = (size_t)item * fe.ostride + (size_t)row * d + ch0;
#pragma unroll
                for (int c4 = 0; c4 < HC; c4 += 4) {
                    float4 xv[4], yv[4];
                    if (fe.kind == 2) {
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const bool in = row < d && c4 + q < ncols;
                            xv[q] = in ? fe.X[o0 + c4 + q] : make_float4(0.f, 0.f, 0.f, 0.f);
                            yv[q] = in ? fe.X2[o0 + c4 + q] : make_float4(0.f, 0.f, 0.f, 0.f);
                        }
                    }
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int e = __shfl_sync(0xffffffffu, eB[0], c4 + q);
                        if (row >= d || c4 + q >= ncols) continue;
                        const float sc = ldexpf(1.0f, eA + e - 3 * SBITS);
                        const float4 v = res[c4 + q];
                        float rh = v.x * sc, rl = v.z * sc, ih = v.y * sc, il = v.w * sc;
                        if (fe.kind == 2) {
                            pair_fma(rh, rl, fe.c1, xv[q].x, xv[q].z);
                            pair_fma(ih, il, fe.c1, xv[q].y, xv[q].w);
                            pair_fma(rh, rl, fe.c2, yv[q].x, yv[q].z);
                            pair_fma(ih, il, fe.c2, yv[q].y, yv[q].w);
                            if (row == ch0 + c4 + q) df_addc(rh, rl, fe.c0);
                        }
                        float4 o;
                        grid_split(rh, rl, fe.magic, o.x, o.z);
                        grid_split(ih, il, fe.magic, o.y, o.w);
                        fe.out[o0 + c4 + q] = o;
                        if (fe.ct)   // the lanes' rows are consecutive there
                            fe.ct[(size_t)item * fe.cts + (size_t)(ch0 + c4 + q) * d + row] =
                                make_float2(o.x + o.z, -(o.y + o.w));
                    }
                }
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(Cfg::TMEM_COLS) : "memory");
}

// ------------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn oz_encode_fn() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    }
    return fn;
}

template <class Cfg>
static size_t plane_bytes(int d, int items, int mats = kOzMats) {
    return (size_t)items * mats * Cfg::NG * (size_t)d * oz_row(d) * 2;
}
template <class Cfg>
static size_t scratch_bytes(int d, int items, int mats = kOzMats) {
    return (plane_bytes<Cfg>(d, items, mats) + 255) / 256 * 256 + (size_t)items * mats * d * 4;
}
template <class Cfg>
static int* exps_of(unsigned char* scratch, int d, int cap, int mats) {
    return reinterpret_cast<int*>(scratch + (plane_bytes<Cfg>(d, cap, mats) + 255) / 256 * 256);
}

template <class Cfg>
static cudaError_t make_maps(void* planes, int d, int items, TcMaps* maps, int mats = kOzMats) {
    EncodeTiledFn enc = oz_encode_fn();
    if (!enc) return cudaErrorNotSupported;
    const int row = oz_row(d);
    // x: the row of a group, y: plane rows (d), z: groups; rows beyond d fill zeros
    cuuint64_t dims[3] = {(cuuint64_t)row, (cuuint64_t)d, (cuuint64_t)items * mats * Cfg::NG};
    cuuint64_t strides[2] = {(cuuint64_t)row * 2, (cuuint64_t)row * d * 2};
    cuuint32_t estr[3] = {1, 1, 1};
    cuuint32_t boxA[3] = {BK * GRP, BM, 1}, boxB[3] = {BK * GRP, (cuuint32_t)Cfg::BN, 1};
    CUresult r1 = enc(reinterpret_cast<CUtensorMap*>(maps->a), CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, planes, dims,
                      strides, boxA, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                      CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    CUresult r2 = enc(reinterpret_cast<CUtensorMap*>(maps->b), CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, planes, dims,
                      strides, boxB, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                      CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return (r1 == CUDA_SUCCESS && r2 == CUDA_SUCCESS) ? cudaSuccess : cudaErrorInvalidValue;
}

template <class Cfg, typename In>
static cudaError_t slice_launch(const OzSliceJobs& jobs, int njobs, int d, int items, int cap, unsigned char* scratch,
                                cudaStream_t st) {
    if (njobs < 1 || njobs > 4 || items > cap) return cudaErrorInvalidValue;
    __nv_bfloat16* planes = reinterpret_cast<__nv_bfloat16*>(scratch);
    const int gx = std::max((d + 7) / 8, (d + 31) / 32);
    k_oz_slice<Cfg::NS, In><<<dim3(gx, items, njobs), 256, 0, st>>>(jobs, planes, exps_of<Cfg>(scratch, d, cap, jobs.mats), d);
    return cudaGetLastError();
}

template <class Cfg, class Epi>
static cudaError_t mm_launch(const OzJobs& jobs, int njobs, const Epi& fe, int d, int items, int cap,
                             unsigned char* scratch, const TcMaps& maps, DevParams* prm, cudaStream_t st) {
    cudaError_t e = cudaFuncSetAttribute(k_oz_mm<Cfg, Epi>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg::SMEM);   // of each device
    if (e != cudaSuccess) return e;
    if (njobs < 1 || njobs > 2 || d > kMaxD || items > cap) return cudaErrorInvalidValue;
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return cudaErrorInvalidDevice;
    const long long ntiles = (long long)((d + BM - 1) / BM) * ((d + Cfg::BN - 1) / Cfg::BN) * items * njobs;
    if (ntiles > 0x7fffffffll - sms) return cudaErrorInvalidValue;
    k_oz_mm<Cfg, Epi><<<(int)std::min<long long>(ntiles, sms), NTHREADS, Cfg::SMEM, st>>>(
        *reinterpret_cast<const CUtensorMap*>(maps.a), *reinterpret_cast<const CUtensorMap*>(maps.b), jobs, njobs, items,
        fe, exps_of<Cfg>(scratch, d, cap, jobs.mats), d, prm);
    return cudaGetLastError();
}

size_t oz_plane_bytes(int d, int items) { return plane_bytes<AdjCfg>(d, items); }
size_t oz_scratch_bytes(int d, int items) { return scratch_bytes<AdjCfg>(d, items); }
cudaError_t oz_make_maps(void* planes, int d, int items, TcMaps* maps) { return make_maps<AdjCfg>(planes, d, items, maps); }

// items: the wave's items; cap: the items the plane array was sized for (oz_scratch_bytes)
cudaError_t launch_oz_slice(const OzSliceJobs& jobs, int njobs, int d, int items, int cap, unsigned char* scratch,
                            cudaStream_t st) {
    return slice_launch<AdjCfg, float2>(jobs, njobs, d, items, cap, scratch, st);
}

cudaError_t launch_oz_mm(const OzJobs& jobs, int njobs, int d, int items, int cap, unsigned char* scratch,
                         const TcMaps& maps, DevParams* prm, cudaStream_t st) {
    return mm_launch<AdjCfg>(jobs, njobs, OzAdjEpi{}, d, items, cap, scratch, maps, prm, st);
}

size_t oz_fwd_scratch_bytes(int d, int items) { return scratch_bytes<FwdCfg>(d, items); }
cudaError_t oz_fwd_make_maps(void* planes, int d, int items, TcMaps* maps) {
    return make_maps<FwdCfg>(planes, d, items, maps);
}

cudaError_t oz_fwd_product(const OzFwd& z, const float4* a_src, int a_mat, const float4* b_src, int b_mat,
                           float4* out, size_t ms, int kind, float magic, const float4* X, const float4* X2, float2 c0,
                           float2 c1, float2 c2, float2* ct, size_t cts, cudaStream_t st, int* launches) {
    auto count = [&]() { if (launches) ++*launches; };
    if (magic == 0.f || (kind == 2 && (!X || !X2))) return cudaErrorInvalidValue;
    OzSliceJobs sj{};
    int n = 0;
    if (a_src) sj.job[n++] = {a_src, ms, a_mat, 0};
    if (b_src) sj.job[n++] = {b_src, ms, b_mat, 1};
    cudaError_t e;
    if (n) {
        if ((e = slice_launch<FwdCfg, float4>(sj, n, z.d, z.items, z.cap, z.scratch, st)) != cudaSuccess) return e;
        count();
    }
    OzJobs jobs{};
    jobs.fault = z.fault;
    jobs.j[0] = {a_mat, b_mat, nullptr, 0, 1.0f, 0, 0};
    OzFwdEpi fe{out, (long long)ms, kind, magic, X, X2, c0, c1, c2, ct, cts};
    e = mm_launch<FwdCfg>(jobs, 1, fe, z.d, z.items, z.cap, z.scratch, z.maps, z.prm, st);
    count();
    return e;
}

size_t oz_tree_scratch_bytes(int d, int items) { return scratch_bytes<FwdCfg>(d, items, 2); }
cudaError_t oz_tree_make_maps(void* planes, int d, int items, TcMaps* maps) {
    return make_maps<FwdCfg>(planes, d, items, maps, 2);
}

cudaError_t oz_tree_product(const OzTree& z, const TreeMm& t, int ak, bool bl, DevParams* prm, cudaStream_t st, int* launches) {
    const int total = t.E * t.count;
    for (int i0 = 0; i0 < total; i0 += z.cap) {   // the planes hold cap items at a time
        const int items = std::min(z.cap, total - i0);
        OzSliceJobs sa{}, sb{};
        sa.mats = sb.mats = 2;
        sa.count = sb.count = t.count;
        sa.item0 = sb.item0 = i0;
        sa.job[0] = {t.a, t.ai, 0, ak == 2 ? 2 : 0, t.ae};
        sb.job[0] = {t.b, t.bi, 1, 1, t.be};
        cudaError_t e;
        if ((ak == 1) == bl) {   // operands of one type: one launch
            sa.job[1] = sb.job[0];
            e = bl ? slice_launch<FwdCfg, float2>(sa, 2, t.d, items, z.cap, z.scratch, st)
                   : slice_launch<FwdCfg, float4>(sa, 2, t.d, items, z.cap, z.scratch, st);
        } else {
            e = ak == 1 ? slice_launch<FwdCfg, float2>(sa, 1, t.d, items, z.cap, z.scratch, st)
                        : slice_launch<FwdCfg, float4>(sa, 1, t.d, items, z.cap, z.scratch, st);
            if (e != cudaSuccess) return e;
            ++*launches;
            e = bl ? slice_launch<FwdCfg, float2>(sb, 1, t.d, items, z.cap, z.scratch, st)
                   : slice_launch<FwdCfg, float4>(sb, 1, t.d, items, z.cap, z.scratch, st);
        }
        if (e != cudaSuccess) return e;
        ++*launches;
        OzJobs jobs{};
        jobs.mats = 2;
        jobs.fault = z.fault;
        jobs.j[0] = {0, 1, nullptr, 0, 1.0f, 0, 0};
        e = mm_launch<FwdCfg>(jobs, 1, OzTreeEpi{t, i0}, t.d, items, z.cap, z.scratch, z.maps, prm, st);
        if (e != cudaSuccess) return e;
        ++*launches;
    }
    return cudaSuccess;
}

cudaError_t oz_ubar(const OzRev& z, const OzSliceJob& G, const OzSliceJob& P, int count, float2* out, size_t ms,
                    cudaStream_t st, int* launches) {
    OzSliceJobs sj{};
    sj.count = count;
    sj.job[0] = G;
    sj.job[1] = P;
    cudaError_t e = launch_oz_slice(sj, 2, z.d, z.items, z.cap, z.scratch, st);
    if (launches) ++*launches;
    if (e != cudaSuccess) return e;
    OzJobs jobs{};
    jobs.fault = z.fault;
    jobs.j[0] = {G.mat, P.mat, out, (long long)ms, 1.0f, 0, 0};
    e = launch_oz_mm(jobs, 1, z.d, z.items, z.cap, z.scratch, z.maps, z.prm, st);
    if (launches) ++*launches;
    return e;
}

cudaError_t oz_rev_step(const OzRev& z, const float2* const ops[4], const size_t strides[4], float2* O1, float2* O2,
                        size_t ms, int mode, int i, cudaStream_t st, int* launches) {
    auto count = [&]() { if (launches) ++*launches; };
    // slices: A1 row (mat 0), B1 column (mat 1), A2 row (mat 2), B2 column (mat 3); in Horner
    // steps A1 is X^dag, sliced once per wave into mat 4
    const bool horner = mode == 0;
    OzSliceJobs sj{};
    int n = 0;
    if (!horner || ops[0] != z.xh || !*z.xh_sliced) {
        const int mat = (horner && ops[0] == z.xh) ? 4 : 0;
        sj.job[n++] = {ops[0], strides[0], mat, 0};
        if (mat == 4) *z.xh_sliced = 1;
    }
    sj.job[n++] = {ops[1], strides[1], 1, 1};
    sj.job[n++] = {ops[2], strides[2], 2, 0};
    sj.job[n++] = {ops[3], strides[3], 3, 1};
    cudaError_t e = launch_oz_slice(sj, n, z.d, z.items, z.cap, z.scratch, st);
    count();
    if (e != cudaSuccess) return e;
    const int a1 = (horner && ops[0] == z.xh) ? 4 : 0;
    if (horner) {   // O1 = A1 B1 / i, O2 += A2 B2 / i
        const float ri = 1.0f / (float)i;
        OzJobs jobs{};
        jobs.fault = z.fault;
        jobs.j[0] = {a1, 1, O1, (long long)ms, ri, 0, 0};
        jobs.j[1] = {2, 3, O2, (long long)ms, ri, 1, 0};
        e = launch_oz_mm(jobs, 2, z.d, z.items, z.cap, z.scratch, z.maps, z.prm, st);
        count();
        return e;
    }
    // squaring: O1 = A1 B1, then O1 += A2 B2
    OzJobs jobs{};
    jobs.fault = z.fault;
    jobs.j[0] = {0, 1, O1, (long long)ms, 1.0f, 0, 0};
    if ((e = launch_oz_mm(jobs, 1, z.d, z.items, z.cap, z.scratch, z.maps, z.prm, st)) != cudaSuccess) return e;
    count();
    jobs.j[0] = {2, 3, O1, (long long)ms, 1.0f, 1, 0};
    e = launch_oz_mm(jobs, 1, z.d, z.items, z.cap, z.scratch, z.maps, z.prm, st);
    count();
    return e;
}

}  // namespace qoc
