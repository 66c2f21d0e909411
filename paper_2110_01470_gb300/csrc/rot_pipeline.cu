// rot_pipeline.cu -- one SSO generation of a rotated-function swarm with
// FP32 fitness and FP64 recheck, as a short sequence of kernels around the
// tensor-core rotation (z = M (x - o) for the whole swarm is one N x D x D
// GEMM, which the per-particle persistent kernel cannot share across
// particles).
//
// Generation g (the number g is read from device memory, so the sequence can
// be replayed by a CUDA graph):
//   1. rot_update    Eq. 2.1 for every variable (the same draws as the
//                    persistent kernel), X written in place, d = x - o (exactly, a
//                    float pair) as four BF16 planes of integer slices, the slice
//                    scale and sum |d_k| per row, "x equals pBest" flag per row.
//   2. rot_gemm_fit  the tcgen05 GEMM; its epilogue turns each z into the
//                    function's FP32 terms and per-term error bounds and
//                    writes per-(particle, 64-column group) partial sums.
//   3. rot_decide    FP32 fitness and bound per particle; pBest update when
//                    the interval decides it (Alg. 3, <=); else the particle
//                    goes on list 1.
//   4. rot_z32       refinement of list-1 rows: z by a compensated FP32 dot
//                    product (Ogita, Rump, Oishi, "Accurate sum and dot
//                    product", SISC 2005, Algorithm Dot2), error below
//                    u |z| + 2 gamma_n^2 sum |M||d| -- some thousand times
//                    tighter than the tensor-core bound.
//   5. rot_fix32     fitness intervals from the refined z; decides the pBest
//                    update, or the particle goes on list 3.
//   6. rot_z64       FP64 z = M (x - o) of list-3 rows in the oracle's order
//                    (k ascending, fma from +0) and their fitness terms, one
//                    thread per output.
//   7. rot_fix       the FP64 sums of those rows (the oracle's summation) and
//                    the exact pBest decision.
//   8. rot_argmin(0) gBest candidates (Alg. 4, lowest index): unique from the
//                    intervals, or the pBests that can still be the minimum
//                    go on list 2.
//   9-10.            steps 6-7 for list 2 (pBest rows only).
//  11. rot_argmin(1) the exact arg-min if needed, gBest record, log, gBest
//                    row, generation counter + 1.
// Steps 4-7 and 9-10 exit at once when their list is empty.  The refinement
// exists because FP64 on this GPU runs at a small fraction of the FP32 rate:
// one FP64 row costs D^2 FP64 fmas, the refinement about 14 D^2 FP32 ops.
#include <algorithm>
#include <cfloat>
#include <climits>
#include <cuda_bf16.h>

#include "psso.h"
#include "psso_internal.h"
#include "rot_pipeline.h"
#include "sso_kernel.cuh"
#include "tc_gemm.cuh"
#include "tc_pair.cuh"

namespace psso {
namespace rot {

// Appends v to a list of capacity cap (the counter may live in shared memory).
__device__ __forceinline__ void list_push(int32_t* list, unsigned* count, long long cap, int32_t v)
{
    const unsigned slot = atomicAdd(count, 1u);
    if (PSSO_CHK((long long)slot < cap, CHK_LIST, slot)) list[slot] = v;
}

using tc::BM;
using tc::BN;

__global__ void set_gen(RotCtl* ctl, long long g)
{
    ctl->gen = g;
    if (g == 0) ctl->refined = 0;    // counters restart with the swarm, like the gBest record's
    ctl->n1 = 0;
    ctl->n2 = 0;
    ctl->n3 = 0;
    ctl->amb = 0;
    ctl->acc = 0;
    ctl->rck = 0;
}

// ---- 1. update --------------------------------------------------------------
// A warp per row, in grid-stride order, the row staged in the warp's shared
// memory: the interval draws; the fresh-value blocks of the chunks that need
// one (about a third), 32 a round; X and the row's scale and norm; the slices.
// Bound: instruction issue (Philox 56 of about 130 lane-operations a variable)
// close to HBM (28 bytes a variable: X, P read, X and four BF16 planes written;
// 34 us at N = 8192, D = 1000).  With the row held in registers (64 of them at D =
// 1000) an SM ran 8 to 16 warps, both Philox blocks of every chunk, and the
// slices one rounding after the other: 54 -> 47 us per launch; N = 4096,
// D = 256: 13 -> 13 us.
constexpr int UPDATE_WARPS = 8;
__global__ void __launch_bounds__(32 * UPDATE_WARPS, 4) rot_update(const RotDev r)
{
    __shared__ __align__(16) float stage[UPDATE_WARPS][1024];
    __shared__ uint32_t reqs[UPDATE_WARPS][256];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float* const row = stage[warp];
    uint32_t* const req = reqs[warp];
    const unsigned lt_mask = (1u << lane) - 1u;
    const InstDev& d = *r.inst;
    const long long g = r.ctl->gen;
    const uint32_t gg = (uint32_t)g;
    const int nch = d.nchunks, D = d.D, Dp = d.Dp, nq = (nch + 31) >> 5;
    if (!PSSO_CHK(Dp <= 1024, CHK_ROT_ROW, Dp)) return;
    const uint32_t k0 = d.k0, k1 = d.k1;
    const float* const o32 = as_global(d.o32);
    const size_t plane = (size_t)r.Np * r.Kp;
    const int nwarps = (int)gridDim.x * UPDATE_WARPS, N = (int)d.N;
    for (int i = (int)blockIdx.x * UPDATE_WARPS + warp; i < N; i += nwarps) {
        float* const xr = as_global(static_cast<float*>(d.X)) + (int64_t)i * Dp;
        const float* const pr = as_global(static_cast<const float*>(d.P)) + (int64_t)i * Dp;
        const uint32_t ii = (uint32_t)i + d.i_base;
        __syncwarp();                    // the previous row's stage is consumed
        bool eqp = true;
        int nreq = 0;
        {
            const uint32_t Tg = d.Tg > 0xffffffffull ? 0xffffffffu : (uint32_t)d.Tg;
            const uint32_t Tp = d.Tp > 0xffffffffull ? 0xffffffffu : (uint32_t)d.Tp;
            const uint32_t Tw = d.Tw > 0xffffffffull ? 0xffffffffu : (uint32_t)d.Tw;
            const bool fg = d.Tg > 0xffffffffull, fp = d.Tp > 0xffffffffull, fw = d.Tw > 0xffffffffull;
            const uint32_t ctr3 = TAG_RHO | (d.sid << 8);
            const float* const gs = as_global(static_cast<const float*>(d.gbrow));
            // sources of the first and third interval (Eq. 2.1 as printed keeps x first
            // and takes gBest third)
            const float* const src1 = d.order ? xr : gs;
            const float* const src3 = d.order ? gs : xr;
#pragma unroll 2
            for (int q = 0; q < nq; ++q) {
                const int c = lane + 32 * q;
                uint32_t nf = 0;
                if (c < nch) {
                    const uint32_t valid = 4 * c + 4 <= D ? 15u : (1u << (D - 4 * c)) - 1u;
                    float x[4] = {0.f, 0.f, 0.f, 0.f};
                    if (g == 0) {
                        nf = valid;
                    } else {
                        float v1[4], v2[4], v3[4];
                        ld4_cg(src1 + 4 * c, v1);
                        ld4_cg(pr + 4 * c, v2);
                        ld4_cg(src3 + 4 * c, v3);
                        const uint4 rb = philox10(make_uint4((uint32_t)c, ii, gg, ctr3), k0, k1);
#pragma unroll
                        for (int m = 0; m < 4; ++m) {
                            const uint32_t w = word_of(rb, m);
                            const bool lg = w < Tg || fg, lp = w < Tp || fp, lw = w < Tw || fw;
                            // a variable of the last interval holds its pBest value until it is
                            // drawn (beyond D every source is 0)
                            x[m] = lg ? v1[m] : (lp || !lw) ? v2[m] : v3[m];
                            if (!lw) nf |= 1u << m;
                            eqp = eqp && same_bits(x[m], v2[m]);
                        }
                        nf &= valid;
                    }
                    st4(row + 4 * c, x);
                }
                const unsigned want = __ballot_sync(0xffffffffu, nf != 0u);
                if (nf) req[nreq + __popc(want & lt_mask)] = (uint32_t)c | (nf << 8);
                nreq += __popc(want);
            }
        }
        __syncwarp();
        {
            Hot fh;                      // the fields fresh_chunk reads
            fh.sid = d.sid;
            fh.k0 = k0;
            fh.k1 = k1;
            fh.S32 = d.S32;
            fh.L32 = d.L32;
            fh.lbf = d.lbf;
            fh.ubf = d.ubf;
            for (int base = 0; base < nreq; base += 32) {
                const int e = base + lane;
                if (e < nreq) {
                    const uint32_t rq = req[e], c = rq & 0xffu, nf = rq >> 8;
                    float fv[4], pv[4];
                    ld4(row + 4 * c, pv);
                    fresh_chunk(fv, nf, c, ii, gg, g == 0 ? TAG_INIT : TAG_FRESH, fh);
#pragma unroll
                    for (int m = 0; m < 4; ++m)
                        if (nf & (1u << m)) {
                            eqp = eqp && same_bits(fv[m], pv[m]);
                            pv[m] = fv[m];
                        }
                    st4(row + 4 * c, pv);
                }
            }
        }
        __syncwarp();
        eqp = __all_sync(0xffffffffu, eqp);
        // X, the row maximum and the L1 norm of d = x - o (exactly a float pair, TwoSum)
        float dmax = 0.f, l1 = 0.f;
        for (int q = 0; q < nq; ++q) {
            const int c = lane + 32 * q;
            if (c >= nch) continue;
            float x[4], o[4];
            ld4(row + 4 * c, x);
            ld4_nc(o32 + 4 * c, o);
            st4(xr + 4 * c, x);
#pragma unroll
            for (int m = 0; m < 4; ++m) {            // beyond D: x = o = 0
                const float ad = fabsf(__fsub_rn(x[m], o[m]));
                dmax = fmaxf(dmax, ad);
                l1 = __fadd_ru(l1, ad);
            }
        }
        for (int off = 16; off > 0; off >>= 1) {
            dmax = fmaxf(dmax, __shfl_xor_sync(0xffffffffu, dmax, off));
            l1 = __fadd_ru(l1, __shfl_xor_sync(0xffffffffu, l1, off));
        }
        // |d| <= |fl(d)| (1 + 2^-24): the scale and the L1 norm cover the exact d
        l1 = __fmul_ru(l1, 1.f + 0x1p-22f);
        // the 7-bit integer slices of d / s_d (tc_gemm.cuh), four planes
        const float sd = tc::slice_scale(dmax), inv = 1.f / sd;   // powers of two: exact
        // differences whose scale leaves the range of a float: no bound holds
        if (!(dmax < 0x1p120f) || sd < 0x1p-120f) l1 = INFINITY;
        __nv_bfloat16* const arow = r.A + (size_t)i * r.Kp;
        for (int q = 0; q < nq; ++q) {
            const int c = lane + 32 * q;
            if (c >= nch) continue;
            float x[4], o[4];
            ld4(row + 4 * c, x);
            ld4_nc(o32 + 4 * c, o);
            uint32_t u[4];
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                const float v = x[m], w = -o[m];
                const float sum = __fadd_rn(v, w), bb = __fsub_rn(sum, v);   // TwoSum
                const float lo = __fadd_rn(__fsub_rn(v, __fsub_rn(sum, bb)), __fsub_rn(w, bb));
                u[m] = tc::slice_fields(__fmul_rn(sum, inv), __fmul_rn(lo, inv));
            }
#pragma unroll
            for (int p = 0; p < tc::SLICES; ++p)     // 4 consecutive bf16 (8 bytes) per plane
                *reinterpret_cast<uint2*>(arow + p * plane + 4 * c) =
                    make_uint2(tc::slice_pack(u[0], u[1], p), tc::slice_pack(u[2], u[3], p));
        }
        if (lane == 0) {
            r.dscale[i] = sd;
            r.dl1[i] = l1;
            r.same[i] = (g > 0 && eqp) ? 1u : 0u;
        }
    }
}

// ---- 2. GEMM with the fitness epilogue ------------------------------------------
// Per element z~ with error ez (the integer-slice GEMM of tc_gemm.cuh of the
// exact d = x - o and the FP64 M: dropped slice products and remainders, the
// FP32 join, against the FP64 rotation M (x - o)),
// the terms and bounds of the rotated functions (as in the FP32 path of the
// persistent kernel): ellipsoid w z^2; Rastrigin z^2 + 20 sin^2(pi z);
// Ackley z^2 and sin^2(pi z) (two sums).  Sums: 32 terms per column block,
// then 4 blocks per tile, then the tiles (in rot_decide).
__device__ __forceinline__ void term32(int fn, float zt, float ez, const float* w32, int j, float& s,
                                       float& s2, float& e, float& eq)
{
    const float az = fabsf(zt);
    const float xi = az + ez;
    if (fn == FN_ELLIPSOID) {
        const float w = __ldg(w32 + j);
        const float tv = __fmul_rn(w, __fmul_rn(zt, zt));
        s = __fadd_rn(s, tv);
        e = __fadd_rn(e, 4.2f * 0x1p-24f * tv + 1.01f * w * (2.f * az + ez) * ez);
    } else if (fn == FN_RASTRIGIN) {
        const float sn = sinpi_reduced_f32(__fsub_rn(zt, rint_f32(zt)));
        const float tv = __fmaf_rn(zt, zt, __fmul_rn(20.f, __fmul_rn(sn, sn)));
        s = __fadd_rn(s, tv);
        e = __fadd_rn(e, (2.f * SINPI32_ERR_U + 4.f) * 0x1p-24f * tv +
                             1.01f * (2.f * xi + 62.8318558f * fminf(1.f, 6.28318548f * xi)) * ez);
    } else {   // Ackley
        s = __fadd_rn(s, __fmul_rn(zt, zt));
        const float sn = sinpi_reduced_f32(__fsub_rn(zt, rint_f32(zt)));
        s2 = __fadd_rn(s2, __fmul_rn(sn, sn));
        e = __fadd_rn(e, 1.01f * (2.f * az + ez) * ez);
        eq = __fadd_rn(eq, 1.01f * 3.14159275f * fminf(1.f, 6.28318548f * xi) * ez);
    }
}

template <bool ONE>
struct FitEpi {
    const RotDev* r;
    int fn, D;
    float drop;                   // SLICE_DROP * D
    // the current row and 64-column group: particle i, group nt, s_d, sum |d_k|
    int64_t i;
    int nt;
    float ds, dl1;
    // ONE: no pair has a second item, so the accumulators need not make way and are
    // read eight columns at a time where they are used
    float t[ONE ? 8 : 64], em[ONE ? 8 : 64];   // joined accumulators, sums of the partial sums' magnitudes
    uint32_t at;                  // ONE: the accumulators' address
    __device__ __forceinline__ void tile(int tm, int g, int row)
    {
        i = (int64_t)tm * tc::PBM + row;
        nt = g;
        ds = i < r->N ? r->dscale[i] : 1.f;
        dl1 = i < r->N ? r->dl1[i] : 0.f;
        // the scales (and weights) of the group's columns: two lines each
        const int lane = threadIdx.x & 31, j = nt * 64 + 32 * (lane & 1);
        const float* const at = lane < 2 ? r->mscale : lane < 4 ? r->ml1 : r->inst_w32;
        if (lane < 6 && at && j < D) asm volatile("prefetch.global.L1 [%0];" ::"l"(at + j));
    }
    // joins the accumulators of column q (v: by weight) from the smallest weight up;
    // each step one rounding (the scaled accumulator is exact)
    __device__ __forceinline__ void join_low(int q, float v2, float v3)
    {
        t[q] = __fmaf_rn(v2, 0x1p-14f, __fmul_rn(v3, 0x1p-21f));   // the product is exact
        em[q] = fabsf(t[q]);
    }
    __device__ __forceinline__ void join_high(int q, float v0, float v1)
    {
        const float t1 = __fmaf_rn(v1, 0x1p-7f, t[q]);
        const float t2 = __fadd_rn(v0, t1);
        em[q] = __fadd_ru(__fadd_ru(em[q], fabsf(t1)), fabsf(t2));
        t[q] = t2;
    }
    template <int C>
    __device__ __forceinline__ void load32(uint32_t taddr)
    {
        float v[32], w[32];
        tc::tmem_ld32(taddr + (uint32_t)(3 * 128), v);
        tc::tmem_ld32(taddr + (uint32_t)(2 * 128), w);
#pragma unroll
        for (int q = 0; q < 32; ++q) join_low(32 * C + q, w[q], v[q]);
        tc::tmem_ld32(taddr + (uint32_t)128, v);
        tc::tmem_ld32(taddr, w);
#pragma unroll
        for (int q = 0; q < 32; ++q) join_high(32 * C + q, w[q], v[q]);
    }
    __device__ __forceinline__ void load(uint32_t taddr, int n)
    {
        if constexpr (ONE) {
            at = taddr;
        } else {
            load32<0>(taddr);
            if (n == 2) load32<1>(taddr + 32);
        }
    }
    // The terms of the 32-column blocks c0 .. c0 + n - 1 of the group, eight columns a
    // step (without ONE the rest of the registers move up): unrolled over 64 columns,
    // the code of a tile takes longer to fetch than to run where a CTA has one tile.
    __device__ __forceinline__ void compute(int c0, int n, float4* xch)
    {
        float acc = 0.f, acc2 = 0.f, accE = 0.f, rQ = 0.f;
        float s = 0.f, s2 = 0.f, e = 0.f, eq = 0.f;
#pragma unroll 1
        for (int h = 0; h < 4 * n; ++h) {
            const int j0 = nt * 64 + 32 * c0 + 8 * h;
            if constexpr (ONE) {
                float v[4][8];
                tc::tmem_ld8x4(at + (uint32_t)(8 * h), 128u, v);
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    join_low(q, v[2][q], v[3][q]);
                    join_high(q, v[0][q], v[1][q]);
                }
            }
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int j = j0 + q;
                if (j >= D) break;
                const float sm = __ldg(r->mscale + j), l1m = __ldg(r->ml1 + j);
                const float sc = __fmul_rn(ds, sm);                 // a power of two
                const float zt = __fmul_rn(t[q], __fmul_rn(sc, 0x1p-14f));
                const float rd = __fmul_rn(sm, dl1), rm = __fmul_rn(ds, l1m);
                // dropped slice products, slice remainders, the FP64 reference's
                // own rounding (D <= 2^13 terms: 2^-40 sum |M||d|), the FP32 join
                const float ez = 1.01f * (drop * sc + tc::SLICE_REM * (rd + rm) + 0x1p-40f * fminf(rd, rm) +
                                          0x1p-38f * em[q] * sc) + 0x1p-126f;
                term32(fn, zt, ez, r->inst_w32, j, s, s2, e, eq);
            }
 if constexpr (!ONE) {
#pragma unroll
                for (int q = 0; q < 56; ++q) {
                    t[q] = t[q + 8];
                    em[q] = em[q + 8];
                }
            }
            if ((h & 3) == 3) {                 // a block of 32 terms ends
                acc = __fadd_rn(acc, s);
                acc2 = __fadd_rn(acc2, s2);
                accE = __fadd_rn(accE, e);
                rQ = __fadd_rn(rQ, eq);
                s = s2 = e = eq = 0.f;
            }
        }
        if (n == 1) {                           // the group's other 32 columns are the other warp's
            const float4 o = tc::pair_exchange(make_float4(acc, acc2, accE, rQ), c0, xch);
            if (c0 == 1) return;
            acc = __fadd_rn(acc, o.x);
            acc2 = __fadd_rn(acc2, o.y);
            accE = __fadd_rn(accE, o.z);
            rQ = __fadd_rn(rQ, o.w);
        }
        if (i < r->N && PSSO_CHK(nt < r->nJt, CHK_TILE, nt))
            r->part[i * r->nJt + nt] = make_float4(acc, acc2, accE, rQ);
    }
};

// The ten slice products of weight <= 3 (tc_gemm.cuh), one accumulator per weight.
struct SliceCfg {
    static constexpr int PLANES = tc::SLICES, STG = 2, PRODUCTS = 10;
    __device__ static constexpr int pa(int q) { constexpr int T[10] = {0, 0, 1, 0, 1, 2, 0, 1, 2, 3}; return T[q]; }
    __device__ static constexpr int pb(int q) { constexpr int T[10] = {0, 1, 0, 2, 1, 0, 3, 2, 1, 0}; return T[q]; }
    __device__ static constexpr int acc(int q, int) { constexpr int T[10] = {0, 1, 1, 2, 2, 2, 3, 3, 3, 3}; return T[q]; }
    __device__ static constexpr bool first(int q, int kb, int ks)
    {
        return (q == 0 || q == 1 || q == 3 || q == 6) && kb == 0 && ks == 0;
    }
};

// Persistent, one CTA pair per two SMs (tc_pair.cuh).  N = 8192, D = 1000: 160 ->
// 138 us per launch.  A launch of at most one item a pair is latency: the loads of
// the row's and the columns' scales start before the wait for the accumulators, and
// ONE moves no registers (N = 169, D = 33: 17.6 -> 14.6 us between events, 5 of them
// the events'; N = 4096, D = 256 has 64 items for 76 pairs).  The kernel of one CTA per
// 128 x 64 tile took 14.1 us there, but 19.2 against 16.8 at N = 256, D = 128.
template <bool ONE>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(tc::P_THREADS, 1)
    rot_gemm_fit(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                 const __grid_constant__ RotDev r)
{
    FitEpi<ONE> epi;
    epi.r = &r;
    epi.fn = base_fn(r.fn);
    epi.D = r.D;
    epi.drop = tc::SLICE_DROP * (float)r.D;
    tc::GemmArgs a{r.Np, r.Jp, r.Kp, &r.ctl->status};
    tc::gemm_pair<SliceCfg>(&tmA, &tmB, a, epi);
}

// ---- 3. FP32 decisions ------------------------------------------------------------
// FP32 fitness and its bound from the sums of the terms (the rotated branches
// of the FP32 path); csum = summation depth + 2 (GEMM epilogue: 32 + 4 +
// tiles + 2).
__device__ inline Fit32 rot_final(int fn, int D, float acc, float acc2, float accE, float rQ, float csum)
{
    const float U = 0x1p-24f;
    Fit32 f;
    if (fn != FN_ACKLEY) {
        f.f = acc;
        f.E = 1.1f * (accE + csum * U * acc);
        f.E = __fadd_ru(f.E, 0x1p-40f * (acc + accE));
        return f;
    }
    const float Df = (float)D;
    const float A = __fsqrt_rn(__fdiv_rn(acc, Df));
    const float B = expm1_f32(__fmul_rn(-0.2f, A));
    const float C = expm1_f32(__fmul_rn(-2.f, __fdiv_rn(acc2, Df)));
    const float f1 = __fmul_rn(-20.f, B), f2 = __fmul_rn(-0x1.5bf0a8p+1f, C);
    f.f = __fadd_rn(f1, f2);
    const float ES = accE + (3.1f + csum) * U * acc;
    const float EQ = rQ + (2.f * SINPI32_ERR_U + 1.f + csum) * U * acc2;
    const float d1 = (ES <= 0.5f * acc) ? 1.5f * f1 * ES / acc : 4.f * __fsqrt_ru(ES / Df);
    f.E = 1.1f * (d1 + (EXPM1F_ERR_U + 6.f) * U * f1 + (2.f * 2.7182818f / Df) * EQ +
                  (EXPM1F_ERR_U + 8.f) * U * f2 + U * f.f);
    f.E = __fadd_ru(f.E, 0x1p-40f * (f.f + accE));
    return f;
}

__global__ void rot_decide(const RotDev r)
{
    __shared__ unsigned long long blk_acc;
    if (threadIdx.x == 0) blk_acc = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int64_t i = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const InstDev& d = *r.inst;
    const int64_t g = r.ctl->gen;
    if (i < d.N) {
        // tile sums in tile order by lane 0 (a fixed order)
        float4 p = make_float4(0.f, 0.f, 0.f, 0.f);
        if (lane < r.nJt) p = r.part[i * r.nJt + lane];
        float a = 0.f, a2 = 0.f, ae = 0.f, aq = 0.f;
        for (int t = 0; t < r.nJt; ++t) {
            a = __fadd_rn(a, __shfl_sync(0xffffffffu, p.x, t));
            a2 = __fadd_rn(a2, __shfl_sync(0xffffffffu, p.y, t));
            ae = __fadd_rn(ae, __shfl_sync(0xffffffffu, p.z, t));
            aq = __fadd_rn(aq, __shfl_sync(0xffffffffu, p.w, t));
        }
        const Fit32 f = rot_final(base_fn(r.fn), r.D, a, a2, ae, aq, 38.f + (float)r.nJt);
        // (beyond the floats' range f - E is a NaN: nothing is known of the value)
        const float lo = fmaxf(__fsub_rd(f.f, f.E), -INFINITY), hi = fminf(__fadd_ru(f.f, f.E), INFINITY);
        int accept = 0, write = 0, undecided = 0;
        if (g == 0) {
            accept = write = 1;
        } else if (r.same[i]) {
            accept = 1;              // identical row: identical fitness, state unchanged
        } else if (hi < d.plo[i]) {
            accept = write = 1;
        } else if (!(lo > d.phi[i])) {
            undecided = 1;
        }
        if (write) {
            const float* xr = static_cast<const float*>(d.X) + i * d.Dp;
            float* prow = static_cast<float*>(d.P) + i * d.Dp;
            for (int c = lane; c < d.nchunks; c += 32) {
                float v[4];
                ld4(xr + 4 * c, v);
                st4(prow + 4 * c, v);
            }
            if (lane == 0) {
                d.plo[i] = lo;
                d.phi[i] = hi;
                d.pflag[i] = 0u;
                d.pf64[i] = 0.0;
                d.pver[i] = (uint32_t)g;
            }
        }
        if (lane == 0) {
            if (undecided) list_push(r.list1, &r.ctl->n1, r.N, (int32_t)i);
            if (accept) atomicAdd(&blk_acc, 1ull);
        }
    }
    __syncthreads();
    if (threadIdx.x == 0 && blk_acc) atomicAdd(&r.ctl->acc, blk_acc);
}

// ---- 4. refinement: compensated FP32 rotation of list-1 rows ---------------------------
// d = x - o exactly as a float pair (TwoSum), M = Mh + Ml.  Per output j the
// 32 lanes of a warp take k = l, l + 32, ... (coalesced rows of M): the Dot2
// recurrence per lane (TwoProduct of Mh d_h, TwoSum into p, the rounding
// errors and the cross terms Mh d_l + Ml d_h into s), then the 32 lane sums
// merged by a TwoSum butterfly, z = p + s.  With n = ceil(D / 32) + 8 and
// g = gamma_n: |z~ - z| <= 1.01 u |z~| + (2 g^2 + 4 u g + 2^-42) S, where
// S = sum |M||d| <= S~ (1 + 2 gamma_D)(1 + 2^-22) from the FP32 sum S~ of
// |Mh||d_h|; 2^-42 S also covers the oracle's own FP64 rounding of z.
// A block takes Z32_OUT outputs of one listed row, each warp Z32_NJ of them
// (independent chains sharing the loads of d).  The lists are short (about ten
// rows), so a launch is one block's chain of loads, and M has left L2 since the
// last generation: Z32_AHEAD steps' loads of M travel together, and a warp has
// one group of outputs (one step's loads at a time and two groups a warp: 52 ->
// 36 us per launch, rotated Rastrigin, N = 8192, D = 1000; ellipsoid 31 -> 12).
constexpr int Z32_NJ = 4;                       // outputs per warp
constexpr int Z32_OUT = 4 * Z32_NJ;             // outputs per block
constexpr int Z32_AHEAD = 4;                    // steps of 32 k
__global__ void __launch_bounds__(128) rot_z32(const RotDev r)
{
    __shared__ float dh[1024], dl[1024];
    const InstDev& d = *r.inst;
    const unsigned n = r.ctl->n1;
    const int D = r.D;
    if (!PSSO_CHK(n <= r.N && D <= 1024, CHK_LIST, n)) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nJb = (D + Z32_OUT - 1) / Z32_OUT;
    const float U = 0x1p-24f;
    const float nl = (float)((D + 31) / 32 + 8);
    const float gam = nl * U / (1.f - nl * U);
    const float gD = (float)D * U / (1.f - (float)D * U);
    const float cS = 1.01f * (2.f * gam * gam + 4.f * U * gam + 0x1p-42f) * (1.f + 2.f * gD) * (1.f + 0x1p-22f);
    const long long items = (long long)n * 2 * nJb;
    for (long long it = blockIdx.x; it < items; it += gridDim.x) {
        const int jb = (int)(it % nJb);
        const int row = (int)((it / nJb) & 1);
        const long long e = it / nJb / 2;
        const int32_t i = r.list1[e];
        if (!PSSO_CHK(i >= 0 && i < r.N, CHK_ROT_ROW, i)) continue;
        if (row == 1 && (d.pflag[i] & 1u)) continue;     // uniform over the block
        const float* src = static_cast<const float*>(row == 0 ? d.X : d.P) + (int64_t)i * d.Dp;
        __syncthreads();
        for (int k = threadIdx.x; k < D; k += blockDim.x) {
            const float a = src[k], b = -__ldg(d.o32 + k);
            const float sum = __fadd_rn(a, b);
            const float bb = __fsub_rn(sum, a);
            dh[k] = sum;
            dl[k] = __fadd_rn(__fsub_rn(a, __fsub_rn(sum, bb)), __fsub_rn(b, bb));
        }
        __syncthreads();
        const size_t o = (size_t)(2 * e + row) * d.Dp;
        const int j0 = jb * Z32_OUT + warp * Z32_NJ;   // warp-uniform
        int nv = D - j0;                               // outputs of this group inside the row
        nv = nv < 0 ? 0 : nv > Z32_NJ ? Z32_NJ : nv;
        if (lane == 0)
            for (int t = nv; t < Z32_NJ; ++t)
                if (j0 + t < d.Dp) {
                    r.z32[o + j0 + t] = 0.f;
                    r.ez32[o + j0 + t] = 0.f;
                }
        if (nv == 0) continue;
        const float* mh[Z32_NJ];
        const float* ml[Z32_NJ];
        float p[Z32_NJ], sc[Z32_NJ], S[Z32_NJ];
#pragma unroll
        for (int t = 0; t < Z32_NJ; ++t) {
            const int j = t < nv ? j0 + t : j0;        // rows past the end repeat a valid one, unused
            mh[t] = r.Mh + (size_t)j * D;
            ml[t] = r.Ml + (size_t)j * D;
            p[t] = sc[t] = S[t] = 0.f;
        }
#pragma unroll 1
        for (int k0 = lane; k0 < D; k0 += 32 * Z32_AHEAD) {
            float ah[Z32_AHEAD][Z32_NJ], al[Z32_AHEAD][Z32_NJ];
#pragma unroll
            for (int s = 0; s < Z32_AHEAD; ++s)
#pragma unroll
                for (int t = 0; t < Z32_NJ; ++t) {
                    const int k = k0 + 32 * s;
                    ah[s][t] = k < D ? __ldg(mh[t] + k) : 0.f;
                    al[s][t] = k < D ? __ldg(ml[t] + k) : 0.f;
                }
#pragma unroll
            for (int s = 0; s < Z32_AHEAD; ++s) {
                const int k = k0 + 32 * s;
                const float b = k < D ? dh[k] : 0.f, bl = k < D ? dl[k] : 0.f;   // beyond D: adds nothing
#pragma unroll
                for (int t = 0; t < Z32_NJ; ++t) {
                    const float a = ah[s][t];
                    const float h = __fmul_rn(a, b);
                    const float rr = __fmaf_rn(a, b, -h);                 // a b = h + rr exactly
                    const float tt = __fadd_rn(p[t], h);
                    const float bb = __fsub_rn(tt, p[t]);
                    const float q = __fadd_rn(__fsub_rn(p[t], __fsub_rn(tt, bb)), __fsub_rn(h, bb));   // p + h = tt + q
                    p[t] = tt;
                    const float cross = __fmaf_rn(a, bl, __fmul_rn(al[s][t], b));
                    sc[t] = __fadd_rn(sc[t], __fadd_rn(__fadd_rn(q, rr), cross));
                    S[t] = __fmaf_rn(fabsf(a), fabsf(b), S[t]);
                }
            }
        }
#pragma unroll
        for (int t = 0; t < Z32_NJ; ++t) {
            for (int off = 16; off > 0; off >>= 1) {           // every lane ends with the same values
                const float po = __shfl_xor_sync(0xffffffffu, p[t], off);
                const float so = __shfl_xor_sync(0xffffffffu, sc[t], off);
                const float Sq = __shfl_xor_sync(0xffffffffu, S[t], off);
                const float tt = __fadd_rn(p[t], po);
                const float bb = __fsub_rn(tt, p[t]);
                const float q = __fadd_rn(__fsub_rn(p[t], __fsub_rn(tt, bb)), __fsub_rn(po, bb));
                p[t] = tt;
                sc[t] = __fadd_rn(__fadd_rn(sc[t], so), q);
                S[t] = __fadd_rn(S[t], Sq);
            }
            if (lane == 0 && t < nv) {
                const float z = __fadd_rn(p[t], sc[t]);
                r.z32[o + j0 + t] = z;
                r.ez32[o + j0 + t] = __fmaf_ru(cS, S[t], 1.01f * U * fabsf(z));
            }
        }
    }
}

// ---- 5. decisions from the refined intervals ---------------------------------------------
// One warp per refined row, two per list entry.  The kernel runs once over a
// handful of entries, so its time is instruction fetch and the chains of one
// warp: the loops stay rolled (unrolled over the widest row, the straight-line
// code took longer to fetch than to run) and the entry's two rows run side by
// side (33 -> 14 us per launch at D = 1000).
__device__ Fit32 fit_refined(const RotDev& r, const InstDev& d, const float* z, const float* ez, int lane)
{
    const int fn = base_fn(r.fn);
    float s = 0.f, s2 = 0.f, e = 0.f, eq = 0.f;
#pragma unroll 1
    for (int c = lane; c < d.nchunks; c += 32) {
        float zv[4], ev[4];
        ld4(z + 4 * c, zv);
        ld4(ez + 4 * c, ev);
#pragma unroll 1
        for (int m = 0; m < 4; ++m)
            if (4 * c + m < d.D)
                term32(fn, m == 0 ? zv[0] : m == 1 ? zv[1] : m == 2 ? zv[2] : zv[3],
                       m == 0 ? ev[0] : m == 1 ? ev[1] : m == 2 ? ev[2] : ev[3], r.inst_w32, 4 * c + m, s, s2, e, eq);
    }
#pragma unroll 1
    for (int off = 16; off > 0; off >>= 1) {
        s = __fadd_rn(s, __shfl_xor_sync(0xffffffffu, s, off));
        s2 = __fadd_rn(s2, __shfl_xor_sync(0xffffffffu, s2, off));
        e = __fadd_rn(e, __shfl_xor_sync(0xffffffffu, e, off));
        eq = __fadd_rn(eq, __shfl_xor_sync(0xffffffffu, eq, off));
    }
    return rot_final(fn, d.D, s, s2, e, eq, (float)(4 * d.maxc + 5 + 2));
}

// Copies particle i's position to its pBest row (n threads, this one t).
__device__ __forceinline__ void accept_row(const InstDev& d, int64_t i, int t, int n)
{
    const float* xr = static_cast<const float*>(d.X) + i * d.Dp;
    float* prow = static_cast<float*>(d.P) + i * d.Dp;
    for (int c = t; c < d.nchunks; c += n) {
        float v[4];
        ld4(xr + 4 * c, v);
        st4(prow + 4 * c, v);
    }
}

__global__ void __launch_bounds__(64) rot_fix32(const RotDev r)
{
    __shared__ Fit32 sh[2];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const InstDev& d = *r.inst;
    const unsigned n = r.ctl->n1;
    if (!PSSO_CHK(n <= r.N, CHK_LIST, n)) return;
    const int64_t g = r.ctl->gen;
    for (long long e = blockIdx.x; e < (long long)n; e += gridDim.x) {
        const int32_t i = r.list1[e];
        if (!PSSO_CHK(i >= 0 && i < r.N, CHK_ROT_ROW, i)) continue;
        const bool have_p = (d.pflag[i] & 1u) != 0;
        float plo = d.plo[i], phi = d.phi[i];
        __syncthreads();                      // the previous entry's results are consumed
        if (warp == 0 || !have_p) {
            const size_t at = (size_t)(2 * e + warp) * d.Dp;
            const Fit32 f = fit_refined(r, d, r.z32 + at, r.ez32 + at, lane);
            if (lane == 0) sh[warp] = f;
        }
        __syncthreads();
        const Fit32 fx = sh[0];
        const float lox = __fsub_rd(fx.f, fx.E), hix = __fadd_ru(fx.f, fx.E);
        if (!have_p) {       // the pBest's interval, tightened the same way (intersection of two bounds)
            const Fit32 fp = sh[1];
            plo = fmaxf(plo, __fsub_rd(fp.f, fp.E));
            phi = fminf(phi, __fadd_ru(fp.f, fp.E));
        }
        const bool accept = hix < plo;
        const bool reject = lox > phi;
        if (accept) accept_row(d, i, threadIdx.x, 64);
        if (threadIdx.x == 0) {
            if (accept) {
                d.plo[i] = lox;
                d.phi[i] = hix;
                d.pflag[i] = 0u;
                d.pf64[i] = 0.0;
                d.pver[i] = (uint32_t)g;
                atomicAdd(&r.ctl->acc, 1ull);
            } else {
                d.plo[i] = plo;
                d.phi[i] = phi;
                if (!reject) list_push(r.list3, &r.ctl->n3, r.N, i);
            }
            atomicAdd(&r.ctl->refined, have_p ? 1ull : 2ull);
        }
    }
}

// The float pair of M for the refinement (setup).
__global__ void split_m64(const double* M64, long long DD, float* Mh, float* Ml)
{
    for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < DD; q += (long long)gridDim.x * blockDim.x) {
        const double m = M64[q];
        const float h = __double2float_rn(m);
        Mh[q] = h;
        Ml[q] = __double2float_rn(m - (double)h);
    }
}

// M^T for the FP64 rotation (setup): tiles of 32 x 32 through shared memory.
__global__ void transpose_m64(const double* __restrict__ M, int D, double* __restrict__ Mt)
{
    __shared__ double tile[32][33];
    const int x = blockIdx.x * 32, y = blockIdx.y * 32;
    for (int r = threadIdx.y; r < 32; r += blockDim.y)
        if (y + r < D && x + (int)threadIdx.x < D) tile[r][threadIdx.x] = M[(size_t)(y + r) * D + x + threadIdx.x];
    __syncthreads();
    for (int r = threadIdx.y; r < 32; r += blockDim.y)
        if (x + r < D && y + (int)threadIdx.x < D) Mt[(size_t)(x + r) * D + y + threadIdx.x] = tile[threadIdx.x][r];
}

// ---- 4/7. FP64 rotation of listed rows and their terms -----------------------------------
// which = 1: entries of list3, row 2e = X_i and row 2e+1 = P_i when its FP64
// value is not known; which = 2 or 4: entries of list2, row 2e+1 = P_i.
//
// One thread per output: z_j is a chain of D dependent FP64 fmas (the oracle's
// order, k ascending from +0).  An FP64 instruction takes 64 clocks and a warp
// has one in flight, so a chain of 1000 is 31 us however few rows there are;
// M^T (outputs of neighbouring threads side by side, 16 loads in flight) keeps
// the loads off that chain.  The thread then makes its variable's FP64 term
// too, where every output has a thread, and leaves the sums to rot_fix:
//   ellipsoid z^2;  Rastrigin z^2 + 20 sin^2(pi z);  Ackley z and sin(pi r).
constexpr int Z64_AHEAD = 16;
__global__ void __launch_bounds__(128) rot_z64(const RotDev r, int which)
{
    __shared__ double dsh[1024];
    const InstDev& d = *r.inst;
    const unsigned n = which == 1 ? r.ctl->n3 : r.ctl->n2;   // which 2 or 4: list 2
    const int D = r.D;
    if (!PSSO_CHK(n <= r.N && D <= 1024, CHK_LIST, n)) return;
    const int fn = base_fn(r.fn);
    const int nJb = (D + 127) / 128;
    const long long items = (long long)n * 2 * nJb;
    for (long long it = blockIdx.x; it < items; it += gridDim.x) {
        const int jb = (int)(it % nJb);
        const int row = (int)((it / nJb) & 1);
        const long long e = it / nJb / 2;
        const int32_t i = which == 1 ? r.list3[e] : r.list2[e];
        if (!PSSO_CHK(i >= 0 && i < r.N, CHK_ROT_ROW, i)) continue;
        const bool needed = which == 1 ? (row == 0 || !(d.pflag[i] & 1u)) : row == 1;
        if (!needed) continue;          // uniform over the block
        const float* src = static_cast<const float*>(row == 0 ? d.X : d.P) + (int64_t)i * d.Dp;
        __syncthreads();
        for (int k = threadIdx.x; k < D; k += blockDim.x) dsh[k] = __dsub_rn((double)src[k], d.o64[k]);
        __syncthreads();
        const int j = jb * 128 + threadIdx.x;
        const double* mt = r.Mt + (j < D ? j : D - 1);
        double a[Z64_AHEAD], z = 0.0;
#pragma unroll
        for (int q = 0; q < Z64_AHEAD; ++q) a[q] = q < D ? __ldg(mt + (size_t)q * D) : 0.0;
        int k = 0;
        for (; k + 2 * Z64_AHEAD <= D; k += Z64_AHEAD) {
            double b[Z64_AHEAD];
#pragma unroll
            for (int q = 0; q < Z64_AHEAD; ++q) b[q] = __ldg(mt + (size_t)(k + Z64_AHEAD + q) * D);
#pragma unroll
            for (int q = 0; q < Z64_AHEAD; ++q) z = __fma_rn(a[q], dsh[k + q], z);
#pragma unroll
            for (int q = 0; q < Z64_AHEAD; ++q) a[q] = b[q];
        }
#pragma unroll
        for (int q = 0; q < Z64_AHEAD; ++q)
            if (k + q < D) z = __fma_rn(a[q], dsh[k + q], z);
        for (k += Z64_AHEAD; k < D; ++k) z = __fma_rn(__ldg(mt + (size_t)k * D), dsh[k], z);
        if (j < D) {
            const size_t at = (size_t)(2 * e + row) * d.Dp + j;
            if (fn == FN_ELLIPSOID) {
                r.zbuf[at] = __dmul_rn(z, z);
            } else if (fn == FN_RASTRIGIN) {
                r.zbuf[at] = __fma_rn(z, z, __dmul_rn(20.0, sinpi_sq_f64(z)));
            } else {
                r.zbuf[at] = z;
                r.sbuf[at] = sinpi_reduced_f64(__dsub_rn(z, rint(z)));
            }
        }
    }
}

// ---- 5/8. FP64 fitness of the rotated rows and the exact decisions --------------------
// One warp's sum over a row's stored values in the oracle's order: lane
// partials in ascending variable order from +0, then the xor butterfly.
//   kind 0: sum t_j (Rastrigin's terms); 1: sum w_j t_j (ellipsoid);
//   2: sum t_j^2 (Ackley's z and sines).
__device__ double sum_row(const InstDev& d, const double* t, int kind, int lane)
{
    double acc = 0.0, nx[4];
    int c = lane;
    if (c < d.nchunks) ld4(t + 4 * c, nx);
#pragma unroll 1
    while (c < d.nchunks) {
        double v[4];
#pragma unroll
        for (int m = 0; m < 4; ++m) v[m] = nx[m];
        const int c0 = c;
        c += 32;
        if (c < d.nchunks) ld4(t + 4 * c, nx);       // the next chunk travels while this one is added
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            if (4 * c0 + m >= d.D) break;
            if (kind == 0) acc = __dadd_rn(acc, v[m]);
            else if (kind == 1) acc = __fma_rn(__ldg(d.w64 + 4 * c0 + m), v[m], acc);
            else acc = __fma_rn(v[m], v[m], acc);
        }
    }
#pragma unroll 1
    for (int off = 16; off > 0; off >>= 1) acc = __dadd_rn(acc, __shfl_xor_sync(0xffffffffu, acc, off));
    return acc;
}

// One block of four warps per entry: warp 2 s + row sums row `row` (X_i, P_i),
// Ackley's second sum on s = 1.  The terms are rot_z64's, so a sum is 32
// dependent additions per lane (76 -> 8 us per launch, rotated Rastrigin,
// D = 1000, against evaluating the row's terms in one warp).
__global__ void __launch_bounds__(128) rot_fix(const RotDev r, int which)
{
    __shared__ double sums[2][2], fit[2];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const InstDev& d = *r.inst;
    const int fn = base_fn(r.fn);
    const unsigned n = which == 1 ? r.ctl->n3 : r.ctl->n2;
    if (!PSSO_CHK(n <= r.N, CHK_LIST, n)) return;
    const int64_t g = r.ctl->gen;
    const int row = warp & 1, second = warp >> 1;
    for (long long e = blockIdx.x; e < (long long)n; e += gridDim.x) {
        const int32_t i = which == 1 ? r.list3[e] : r.list2[e];
        if (!PSSO_CHK(i >= 0 && i < r.N, CHK_ROT_ROW, i)) continue;
        const bool have_p = which == 1 && (d.pflag[i] & 1u) != 0;
        const double known = have_p ? d.pf64[i] : 0.0;
        const bool mine = row == 0 ? which == 1 : !have_p;
        __syncthreads();                     // the previous entry's results are consumed
        if (mine && (second == 0 || fn == FN_ACKLEY)) {
            const size_t at = (size_t)(2 * e + row) * d.Dp;
            const double s = sum_row(d, (second ? r.sbuf : r.zbuf) + at,
                                     fn == FN_RASTRIGIN ? 0 : fn == FN_ELLIPSOID ? 1 : 2, lane);
            if (lane == 0) sums[row][second] = s;
        }
        __syncthreads();
        if (mine && second == 0 && lane == 0) {
            double f = sums[row][0];
            if (fn == FN_ACKLEY) {
                const double Dd = (double)d.D;
                const double A = __dsqrt_rn(__ddiv_rn(f, Dd));
                const double B = expm1_f64(__dmul_rn(-0.2, A));
                const double C = expm1_f64(__dmul_rn(-2.0, __ddiv_rn(sums[row][1], Dd)));
                f = -__dadd_rn(__dmul_rn(20.0, B), __dmul_rn(0x1.5bf0a8b145769p+1, C));   // e
            }
            fit[row] = f;
        }
        __syncthreads();
        if (which == 1) {
            const double fx = fit[0], fp = have_p ? known : fit[1];
            const bool accept = fx <= fp;
            if (accept) accept_row(d, i, threadIdx.x, 128);
            if (threadIdx.x == 0) {
                const double v = accept ? fx : fp;
                d.pf64[i] = v;
                d.pflag[i] = 1u;
                d.plo[i] = f64_to_f32_rd(v);
                d.phi[i] = f64_to_f32_ru(v);
                if (accept) d.pver[i] = (uint32_t)g;
                atomicAdd(&r.ctl->rck, have_p ? 1ull : 2ull);
                if (accept) atomicAdd(&r.ctl->acc, 1ull);
            }
        } else if (threadIdx.x == 0) {   // list 2 (which 2: in a generation; 4: on demand, outside the counters)
            const double fp = fit[1];
            d.pf64[i] = fp;
            d.pflag[i] = 1u;
            d.plo[i] = f64_to_f32_rd(fp);
            d.phi[i] = f64_to_f32_ru(fp);
            if (which == 2) atomicAdd(&r.ctl->rck, 1ull);
        }
    }
}


// ---- 6/9. gBest --------------------------------------------------------------------------
// Lowest-index arg-min of the pBest bounds by one block: only the keys are
// read and reduced (the smallest and second-smallest lower bound, the first's
// index, the smallest upper bound), four particles per thread and load; the
// winner's other fields are read afterwards, together (12.3 -> 10.1 us at N = 8192).
struct Key {
    float l1, l2, mh;
    int i;
};
__device__ __forceinline__ Key key_merge(const Key& a, const Key& b)
{
    const bool bf = b.l1 < a.l1 || (b.l1 == a.l1 && b.i < a.i);
    Key r;
    r.l1 = bf ? b.l1 : a.l1;
    r.i = bf ? b.i : a.i;
    r.l2 = fminf(fminf(a.l2, b.l2), bf ? a.l1 : b.l1);
    r.mh = fminf(a.mh, b.mh);
    return r;
}
__device__ __forceinline__ Key key_warp(Key k)
{
#pragma unroll 1
    for (int off = 16; off > 0; off >>= 1) {
        Key o;
        o.l1 = __shfl_xor_sync(0xffffffffu, k.l1, off);
        o.l2 = __shfl_xor_sync(0xffffffffu, k.l2, off);
        o.mh = __shfl_xor_sync(0xffffffffu, k.mh, off);
        o.i = __shfl_xor_sync(0xffffffffu, k.i, off);
        k = key_merge(k, o);
    }
    return k;
}

// FP64 value and index, compared as integers (order_key): a compare of doubles
// takes the FP64 unit's 64 clocks.
struct Exact {
    long long v;
    int i;
};
__device__ __forceinline__ Exact exact_merge(const Exact& a, const Exact& b)
{
    return (b.v < a.v || (b.v == a.v && b.i < a.i)) ? b : a;
}
__device__ __forceinline__ Exact exact_warp(Exact k)
{
#pragma unroll 1
    for (int off = 16; off > 0; off >>= 1) {
        Exact o;
        o.v = __shfl_xor_sync(0xffffffffu, k.v, off);
        o.i = __shfl_xor_sync(0xffffffffu, k.i, off);
        k = exact_merge(k, o);
    }
    return k;
}

__global__ void __launch_bounds__(1024) rot_argmin(const RotDev r, int phase)
{
    __shared__ Key shk[32];
    __shared__ Exact she[32];
    __shared__ unsigned n2;
    __shared__ long long winner;
    const InstDev& d = *r.inst;
    RotCtl* ctl = r.ctl;
    const int64_t g = ctl->gen;
    const int N = (int)d.N, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if (phase == 0) {
        const Key none = {FLT_MAX, FLT_MAX, FLT_MAX, INT_MAX};
        Key k = none;
        for (int i = 4 * (int)threadIdx.x; i < N; i += 4 * (int)blockDim.x) {
            if (i + 4 <= N) {
                float lo[4], hi[4];
                ld4(d.plo + i, lo);
                ld4(d.phi + i, hi);
#pragma unroll
                for (int m = 0; m < 4; ++m) k = key_merge(k, Key{lo[m], FLT_MAX, hi[m], i + m});
            } else {
                for (int m = i; m < N; ++m) k = key_merge(k, Key{d.plo[m], FLT_MAX, d.phi[m], m});
            }
        }
        k = key_warp(k);
        if (lane == 0) shk[warp] = k;
        __syncthreads();
        k = key_warp(lane < nw ? shk[lane] : none);     // every warp has the block's result
        if (k.i >= N) k.i = 0;             // no finite bound at all
        if (k.l2 > k.mh) {                 // one interval lies below every other: the arg-min
            if (threadIdx.x == 0) {
                // the gBest value the generation reports must lie within 1e-6 of
                // FP64: an interval too wide for that gets the winner's FP64 value
                // (list 2; the exact pass of phase 1 then keeps the same winner)
                const int has = (int)(d.pflag[k.i] & 1u);      // (the four loads travel together)
                const float hi = d.phi[k.i];
                const double v = d.pf64[k.i];
                const uint32_t ver = d.pver[k.i];
                const bool wide = !has && too_wide(r.fn, k.l1, hi);
                ctl->amb = wide ? 1 : 0;
                if (wide) {
                    r.list2[0] = k.i;
                    ctl->n2 = 1;
                }
                ctl->win_i = k.i;
                ctl->win_v = has ? v : DBL_MAX;
                ctl->win_lo = k.l1;
                ctl->win_hi = hi;
                ctl->win_has = has;
                ctl->win_ver = ver;
            }
            return;
        }
        // several pBests may be the minimum: those without an FP64 value go on list2
        if (threadIdx.x == 0) n2 = 0;
        __syncthreads();
        for (int i = threadIdx.x; i < N; i += blockDim.x)
            if (d.plo[i] <= k.mh && !(d.pflag[i] & 1u)) list_push(r.list2, &n2, r.N, i);
        __syncthreads();
        if (threadIdx.x == 0) {
            ctl->amb = 1;
            ctl->n2 = n2;
        }
        return;
    }
    // phase 1
    if (ctl->amb) {
        // every pBest that can be the minimum now has its FP64 value; the others
        // have a lower bound above the smallest upper bound
        Exact k = {LLONG_MAX, INT_MAX};
        for (int i = threadIdx.x; i < N; i += blockDim.x)
            if (d.pflag[i] & 1u) k = exact_merge(k, Exact{order_key(d.pf64[i]), i});
        k = exact_warp(k);
        if (lane == 0) she[warp] = k;
        __syncthreads();
        k = exact_warp(lane < nw ? she[lane] : Exact{LLONG_MAX, INT_MAX});
        if (k.i >= N) k.i = 0;
        if (threadIdx.x == 0) {
            const double v = d.pf64[k.i];
            ctl->win_i = k.i;
            ctl->win_v = v;
            ctl->win_lo = f64_to_f32_rd(v);
            ctl->win_hi = f64_to_f32_ru(v);
            ctl->win_has = 1;
            ctl->win_ver = d.pver[k.i];
            winner = k.i;
        }
    } else if (threadIdx.x == 0) {
        winner = ctl->win_i;
    }
    __syncthreads();
    const long long wi = winner;
    const float* src = static_cast<const float*>(d.P) + wi * d.Dp;
    float* dst = static_cast<float*>(d.gbrow);
    for (int j = threadIdx.x; j < d.Dp; j += blockDim.x) dst[j] = src[j];
    __syncthreads();
    if (threadIdx.x == 0) {
        Winner w;
        w.idx = wi;
        w.has64 = ctl->win_has;
        w.f64 = w.has64 ? ctl->win_v : 0.0;
        w.lo = ctl->win_lo;
        w.hi = ctl->win_hi;
        w.ver = ctl->win_ver;
        w.acc = ctl->acc;
        w.rck = ctl->rck;
        write_gbest(d, w, g);
        ctl->gen = g + 1;
        ctl->n1 = 0;
        ctl->n2 = 0;
        ctl->n3 = 0;
        ctl->amb = 0;
        ctl->acc = 0;
        ctl->rck = 0;
    }
}

// ---- values on demand --------------------------------------------------------------------
// Every pBest whose value is known only by an interval too wide for 1e-6
// relative goes on list 2; its FP64 value is then computed (rot_z64 and
// rot_fix with which = 4) -- once, when the state is read.  The trajectory
// does not change: only the stored intervals become exact.
__global__ void list_wide(const RotDev r)
{
    const InstDev& d = *r.inst;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < d.N; i += (int64_t)gridDim.x * blockDim.x)
        if (!(d.pflag[i] & 1u) && too_wide(r.fn, d.plo[i], d.phi[i]))
            list_push(r.list2, &r.ctl->n2, r.N, (int32_t)i);
}

__global__ void clear_n2(RotCtl* ctl) { ctl->n2 = 0; }

// ---- host --------------------------------------------------------------------------------
cudaError_t exact_values_for_read(const RotHost& h, cudaStream_t s)
{
    const RotDev& r = h.dev;
    clear_n2<<<1, 1, 0, s>>>(r.ctl);
    list_wide<<<(unsigned)std::min<long long>((h.N + 255) / 256, 1024), 256, 0, s>>>(r);
    rot_z64<<<h.z64_grid, 128, 0, s>>>(r, 4);
    rot_fix<<<h.fix_grid, 128, 0, s>>>(r, 4);
    clear_n2<<<1, 1, 0, s>>>(r.ctl);
    return cudaGetLastError();
}

cudaError_t enqueue_generation_timed(const RotHost& h, cudaStream_t s, cudaEvent_t* ev);

cudaError_t enqueue_generation(const RotHost& h, cudaStream_t s)
{
    return enqueue_generation_timed(h, s, nullptr);
}

// With ev (KERNELS_PER_GENERATION + 1 events), an event is recorded before
// the first kernel and after each kernel.
cudaError_t enqueue_generation_timed(const RotHost& h, cudaStream_t s, cudaEvent_t* ev)
{
    int q = 0;
    auto mark = [&] {
        if (ev) cudaEventRecord(ev[q++], s);
    };
    mark();
    const RotDev& r = h.dev;
    const int N = (int)h.N;
    const int wpb = 8;
    rot_update<<<std::min(4 * h.fix_grid, (N + UPDATE_WARPS - 1) / UPDATE_WARPS), 32 * UPDATE_WARPS, 0, s>>>(r);
    mark();
    if (h.gemm_one)
        rot_gemm_fit<true><<<h.gemm_grid, tc::P_THREADS, tc::pair_smem<SliceCfg::PLANES, SliceCfg::STG>(), s>>>(h.tmA, h.tmB, r);
    else
        rot_gemm_fit<false><<<h.gemm_grid, tc::P_THREADS, tc::pair_smem<SliceCfg::PLANES, SliceCfg::STG>(), s>>>(h.tmA, h.tmB, r);
    mark();
    rot_decide<<<(N + wpb - 1) / wpb, 32 * wpb, 0, s>>>(r);
    mark();
    rot_z32<<<h.z32_grid, 128, 0, s>>>(r);
    mark();
    rot_fix32<<<h.fix_grid, 64, 0, s>>>(r);
    mark();
    rot_z64<<<h.z64_grid, 128, 0, s>>>(r, 1);
    mark();
    rot_fix<<<h.fix_grid, 128, 0, s>>>(r, 1);
    mark();
    rot_argmin<<<1, h.argmin_threads, 0, s>>>(r, 0);
    mark();
    rot_z64<<<h.z64_grid, 128, 0, s>>>(r, 2);
    mark();
    rot_fix<<<h.fix_grid, 128, 0, s>>>(r, 2);
    mark();
    rot_argmin<<<1, h.argmin_threads, 0, s>>>(r, 1);
    mark();
    return cudaGetLastError();
}

// The generation number lives in device memory, so one captured generation
// replays unchanged; graphs are captured on a private stream and launched on
// the caller's.
cudaError_t make_graphs(RotHost& h)
{
    cudaStream_t cs;
    cudaError_t e = cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking);
    if (e != cudaSuccess) return e;
    for (int which = 0; which < 2 && e == cudaSuccess; ++which) {
        const int gens = which == 0 ? 1 : GRAPH_GENS;
        cudaGraph_t g = nullptr;
        e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
        for (int q = 0; q < gens && e == cudaSuccess; ++q) e = enqueue_generation(h, cs);
        const cudaError_t e2 = cudaStreamEndCapture(cs, &g);
        if (e == cudaSuccess) e = e2;
        if (e == cudaSuccess) e = cudaGraphInstantiate(which == 0 ? &h.graph1 : &h.graphG, g, 0);
        if (g) cudaGraphDestroy(g);
    }
    cudaStreamDestroy(cs);
    return e;
}

void destroy_graphs(RotHost& h)
{
    if (h.graph1) cudaGraphExecDestroy(h.graph1);
    if (h.graphG) cudaGraphExecDestroy(h.graphG);
    h.graph1 = h.graphG = nullptr;
}

cudaError_t run_generations(const RotHost& h, long long count, cudaStream_t s)
{
    for (; count >= GRAPH_GENS; count -= GRAPH_GENS) {
        const cudaError_t e = cudaGraphLaunch(h.graphG, s);
        if (e != cudaSuccess) return e;
    }
    for (; count > 0; --count) {
        const cudaError_t e = cudaGraphLaunch(h.graph1, s);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// B planes of the integer-slice GEMM from the FP64 rotation: one block per
// row j of the padded [Jp][Kp] planes (rows >= D and columns >= D are zero),
// its scale s_M and sum_k |M_jk| (rounded up).
__global__ void slice_matrix(const double* __restrict__ M64, int D, int Jp, int Kp, __nv_bfloat16* B,
                             float* mscale, float* ml1)
{
    const int j = blockIdx.x;
    double mx = 0.0, l1 = 0.0;
    for (int k = threadIdx.x; k < D; k += blockDim.x) {
        const double v = j < D ? M64[(size_t)j * D + k] : 0.0;
        mx = fmax(mx, fabs(v));
        l1 = __dadd_ru(l1, fabs(v));
    }
    __shared__ double rmx[32], rl1[32];
    __shared__ float sm;
    for (int off = 16; off > 0; off >>= 1) {
        mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, off));
        l1 = __dadd_ru(l1, __shfl_xor_sync(0xffffffffu, l1, off));
    }
    if ((threadIdx.x & 31) == 0) {
        rmx[threadIdx.x >> 5] = mx;
        rl1[threadIdx.x >> 5] = l1;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double m = 0.0, t = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
            m = fmax(m, rmx[w]);
            t = __dadd_ru(t, rl1[w]);
        }
        sm = tc::slice_scale(__double2float_ru(m));
        mscale[j] = sm;
        ml1[j] = __double2float_ru(t);
    }
    __syncthreads();
    const double inv = 1.0 / (double)sm;
    const size_t plane = (size_t)Jp * Kp;
    for (int k = threadIdx.x; k < Kp; k += blockDim.x) {
        const double v = (j < D && k < D) ? M64[(size_t)j * D + k] : 0.0;
        __nv_bfloat16 sl[tc::SLICES];
        tc::slice4_f64(__dmul_rn(v, inv), sl);
        for (int p = 0; p < tc::SLICES; ++p) B[p * plane + (size_t)j * Kp + k] = sl[p];
    }
}

cudaError_t build_constants(const RotHost& h, cudaStream_t s)
{
    const RotDev& r = h.dev;
    const long long DD = (long long)r.D * r.D;
    split_m64<<<(unsigned)std::min<long long>((DD + 255) / 256, 4096), 256, 0, s>>>(h.M64, DD, h.Mh, h.Ml);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const unsigned tiles = (unsigned)((r.D + 31) / 32);
    transpose_m64<<<dim3(tiles, tiles), dim3(32, 8), 0, s>>>(h.M64, r.D, h.Mt);
    slice_matrix<<<r.Jp, 256, 0, s>>>(h.M64, r.D, r.Jp, r.Kp, h.B, r.mscale, r.ml1);
    return cudaGetLastError();
}

cudaError_t set_generation(const RotHost& h, long long g, cudaStream_t s)
{
    set_gen<<<1, 1, 0, s>>>(h.dev.ctl, g);
    return cudaGetLastError();
}

cudaError_t configure()
{
    constexpr int smem = tc::pair_smem<SliceCfg::PLANES, SliceCfg::STG>();
    const cudaError_t e = cudaFuncSetAttribute(rot_gemm_fit<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(rot_gemm_fit<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
}

}  // namespace rot
}  // namespace psso
