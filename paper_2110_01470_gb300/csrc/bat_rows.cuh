// bat_rows.cuh -- step kernel of the batched throughput pipeline for the five
// plain functions (sphere, ellipsoid, Rastrigin, Rosenbrock, Ackley) at every
// row width: the Eq. 2.1 update, the fitness and the pBest commit of every
// particle of a class (one function, rows up to or over 128 variables).
//
// A warp takes a task: consecutive particles of one swarm that fill up to 8
// slices (32 chunks of 4 variables; a slice holds one slice of a wide row, or
// 32 / G narrow rows of G lanes each).  The slices are staged in the warp's
// shared memory and processed in three passes:
//   1. Eq. 2.1's interval draw of every chunk (the same draws as the persistent
//      kernel), the selected source values into the stage; a chunk with
//      variables in the last interval (about a third of them) queues a request
//      for its fresh-value block, and its staged values there hold the pBest
//      value;
//   2. the queued fresh-value blocks, 32 per round, one per lane: the Philox
//      work of the last branch is paid only for the chunks that need it, and
//      over 8 slices the rounds are nearly full;
//   3. the staged rows stored to X and their fitness terms; the pBest decision
//      of each particle; accepted rows copied to P from the stage.
// A lane meets its variables in ascending order, so the FP64 value keeps the
// oracle's summation order bit for bit.
//
// FP64 fitness.  The FP64 unit retires 1.66 lanes per clock and SM, so a
// Rastrigin or Ackley term (about 16 FP64 instructions) costs as much as some
// thousand FP32 lanes.  Most particles do not beat their pBest, and for those
// no FP64 value is needed: pass 3 first takes the FP32 fitness of z =
// fl32(fl64(x - o)) with its rigorous bound E, and only the particles that
// f32 - E does not place above their pBest are evaluated in FP64 (queued, so
// that narrow rows fill the warp again).  Decisions and stored values are
// those of the FP64 fitness.  Sphere and ellipsoid terms are two or three FP64
// instructions, no more than the filter's own; they are evaluated directly.
//
// Bound: instruction issue (Philox 40 multiplies and xors per 4 variables, the
// FP32 terms), and for FP64 fitness the FP64 unit.  Against the former pair of
// kernels (one warp per wide row with the function dispatched per chunk, and
// the whole-row code for narrow rows), whole runs with their arg-mins and
// read-backs: 512 swarms, 1.19e8 variables, 150 generations, FP32 223 -> 167
// ms; 40 swarms, 7.6e6 variables, 50 generations, FP64 21.9 -> 13.6 ms.
// The interval's three sources chosen as pointers by the order, and FP32 terms
// without a range check (a variable beyond D, where x = o = w = 0, adds zero; FP64 terms keep theirs,
// the FP64 unit would work for the padding): 118.8 -> 111.2 ms of the FP32 run's
// generations.  Loads of the next task's rows to L2 ahead, a slice loop unrolled
// by 2 or 4, and 3 or 5 blocks an SM instead of 4 gained nothing.
#pragma once
#include <type_traits>

#include "sso_kernel.cuh"

namespace psso {

constexpr int ROWS_SLICES = 8;

// Running sums of one lane in FP64 (the oracle's forms).
template <int FN>
struct RowSum64 {
    double acc = 0.0, acc2 = 0.0;
    // term of variable j < D (d1: the next variable's z)
    __device__ __forceinline__ void term(const double* w64, int D, int j, double z, double d1)
    {
        if constexpr (FN == FN_SPHERE) {
            acc = __fma_rn(z, z, acc);
        } else if constexpr (FN == FN_ELLIPSOID) {
            acc = __fma_rn(__ldg(w64 + j), __dmul_rn(z, z), acc);
        } else if constexpr (FN == FN_RASTRIGIN) {
            acc = __dadd_rn(acc, __fma_rn(z, z, __dmul_rn(20.0, sinpi_sq_f64(z))));
        } else if constexpr (FN == FN_ROSENBROCK) {
            if (j < D - 1) {
                const double a0 = __dadd_rn(z, 1.0), a1 = __dadd_rn(d1, 1.0);
                const double u = __fma_rn(-a0, a0, a1);
                acc = __dadd_rn(acc, __fma_rn(__dmul_rn(100.0, u), u, __dmul_rn(z, z)));
            }
        } else {   // Ackley
            acc = __fma_rn(z, z, acc);
            const double s = sinpi_reduced_f64(__dsub_rn(z, rint(z)));
            acc2 = __fma_rn(s, s, acc2);
        }
    }
    __device__ __forceinline__ double finish(int G, int D)
    {
        for (int off = G >> 1; off > 0; off >>= 1) acc = __dadd_rn(acc, __shfl_xor_sync(0xffffffffu, acc, off));
        if constexpr (FN == FN_ACKLEY) {
            for (int off = G >> 1; off > 0; off >>= 1)
                acc2 = __dadd_rn(acc2, __shfl_xor_sync(0xffffffffu, acc2, off));
            const double Dd = (double)D;
            const double A = __dsqrt_rn(__ddiv_rn(acc, Dd));
            const double B = expm1_f64(__dmul_rn(-0.2, A));
            const double C = expm1_f64(__dmul_rn(-2.0, __ddiv_rn(acc2, Dd)));
            return -__dadd_rn(__dmul_rn(20.0, B), __dmul_rn(0x1.5bf0a8b145769p+1, C));   // e
        } else {
            return acc;
        }
    }
};

// Running sums in FP32 with the terms' error bounds (fit32's forms).  UE: the
// relative error the bounds allow z and every operation, 2^-24 for z = fl(x - o)
// of float positions, 2^-23 where z is a truncated conversion (to_f32_trunc).
template <int FN, bool EXACT_Z>
struct RowSum32 {
    static constexpr float UE = EXACT_Z ? U32 : 2.f * U32;
    float acc = 0.f, acc2 = 0.f, accE = 0.f, accZ = 0.f;
    __device__ __forceinline__ void term(const float* w32, int D, int j, float z, float d1)
    {
        if constexpr (FN == FN_SPHERE) {
            acc = __fadd_rn(acc, __fmul_rn(z, z));
        } else if constexpr (FN == FN_ELLIPSOID) {
            acc = __fadd_rn(acc, __fmul_rn(__ldg(w32 + j), __fmul_rn(z, z)));
        } else if constexpr (FN == FN_RASTRIGIN) {
            const float s = sinpi_reduced_f32(__fsub_rn(z, rint_f32(z)));
            acc = __fadd_rn(acc, __fmaf_rn(z, z, __fmul_rn(20.f, __fmul_rn(s, s))));
        } else if constexpr (FN == FN_ROSENBROCK) {
            if (j < D - 1) {
                const float s0 = __fadd_rn(z, 2.f);
                const float u = __fmaf_rn(-z, s0, d1);
                const float d2 = __fmul_rn(z, z);
                const float t = __fmaf_rn(__fmul_rn(100.f, u), u, d2);
                acc = __fadd_rn(acc, t);
                const float e0 = 1.01f * UE * fabsf(z), e1 = 1.01f * UE * fabsf(d1);
                const float as0 = fabsf(s0);
                const float eu = 1.01f * (UE * fabsf(u) + e1 + fabsf(z) * (UE * as0 + e0) + (1.01f * as0 + e0) * e0);
                float et = 100.f * eu * (2.f * fabsf(u) + eu) + 3.f * UE * 100.f * u * u + 3.1f * UE * d2 + UE * t;
                const float a0 = fabsf(z) + 1.f, a1 = fabsf(d1) + 1.f;
                const float eu64 = 0x1p-51f * (a1 + 2.f * a0 * a0 + fabsf(u) + 2.f);
                et += 200.f * fabsf(u) * eu64 + 100.f * eu64 * eu64 + 0x1p-50f * t;
                accE = __fadd_rn(accE, et);
            }
        } else {   // Ackley
            acc = __fadd_rn(acc, __fmul_rn(z, z));
            const float s = sinpi_reduced_f32(__fsub_rn(z, rint_f32(z)));
            acc2 = __fadd_rn(acc2, __fmul_rn(s, s));
            accZ = __fadd_rn(accZ, fabsf(z));
        }
    }
    // Value and bound; nq = chunks per lane (summation depth 4 nq, then log2 G
    // butterfly levels).
    __device__ __forceinline__ Fit32 finish(int G, int D, int nq)
    {
        for (int off = G >> 1; off > 0; off >>= 1) acc = __fadd_rn(acc, __shfl_xor_sync(0xffffffffu, acc, off));
        const float csum = (float)(4 * nq) + (float)(__ffs(G) - 1) + 2.f;
        Fit32 r;
        if constexpr (FN == FN_SPHERE) {
            r.f = acc;
            r.E = 1.1f * (3.1f + csum) * UE * acc;
        } else if constexpr (FN == FN_ELLIPSOID) {
            r.f = acc;
            r.E = 1.1f * (5.2f + csum) * UE * acc;
        } else if constexpr (FN == FN_RASTRIGIN) {
            r.f = acc;
            r.E = 1.1f * (2.f * SINPI32_ERR_U + 3.f + 16.1f + 1.f + csum) * UE * acc;
        } else if constexpr (FN == FN_ROSENBROCK) {
            for (int off = G >> 1; off > 0; off >>= 1)
                accE = __fadd_rn(accE, __shfl_xor_sync(0xffffffffu, accE, off));
            r.f = acc;
            r.E = 1.1f * (accE + csum * UE * acc);
        } else {   // Ackley
            for (int off = G >> 1; off > 0; off >>= 1) {
                acc2 = __fadd_rn(acc2, __shfl_xor_sync(0xffffffffu, acc2, off));
                accZ = __fadd_rn(accZ, __shfl_xor_sync(0xffffffffu, accZ, off));
            }
            const float Df = (float)D;
            const float A = __fsqrt_rn(__fdiv_rn(acc, Df));
            const float B = expm1_f32(__fmul_rn(-0.2f, A));
            const float C = expm1_f32(__fmul_rn(-2.f, __fdiv_rn(acc2, Df)));
            const float f1 = __fmul_rn(-20.f, B), f2 = __fmul_rn(-0x1.5bf0a8p+1f, C);
            r.f = __fadd_rn(f1, f2);
            const float relS = (3.1f + csum) * UE;
            const float EQ = 1.01f * 3.14159275f * UE * accZ + (2.f * SINPI32_ERR_U + 1.f + csum) * UE * acc2;
            r.E = 1.1f * (0.5f * relS * f1 + (EXPM1F_ERR_U + 6.f) * UE * f1 + (2.f * 2.7182818f / Df) * EQ +
                          (EXPM1F_ERR_U + 8.f) * UE * f2 + UE * r.f);
            acc = r.f;
        }
        r.E = __fadd_ru(r.E, 0x1p-40f * (acc + accE));
        return r;
    }
};

// z truncated to a float by its bit pattern (relative error below 2^-23; a
// conversion instruction would take the FP64 unit).  Below the normal floats'
// range: below 2^-126 in magnitude; above it: infinite or NaN.
__device__ __forceinline__ float to_f32_trunc(double z)
{
    const int hi = __double2hiint(z), lo = __double2loint(z);
    int m = (hi & 0x7fffffff) - (896 << 20);
    m = min(max(m, 0), 255 << 20);
    return __uint_as_float(((uint32_t)hi & 0x80000000u) | __funnelshift_l((uint32_t)lo, (uint32_t)m, 3));
}

// FP64 fitness of the row whose chunk lane_g + 32 q lies at src + 128 q (a
// staged row, or a pBest row from its lane_g-th chunk on), one row per group
// of G lanes; every lane of the warp takes part (valid: the group has a row).
template <int FN, class Pos>
__device__ __forceinline__ double row_f64(const Pos* src, bool valid, int lane_g, int G, int nch, int nq, int D,
                                          const double* o64, const double* w64)
{
    RowSum64<FN> rs;
    for (int q = 0; q < nq; ++q) {
        const int c = lane_g + 32 * q;
        if (c >= nch || !valid) continue;
        Pos x[4];
        ld4(src + 128 * q, x);
        double ov[4], z[4];
        ld4(o64 + 4 * c, ov);
#pragma unroll
        for (int m = 0; m < 4; ++m) z[m] = __dsub_rn((double)x[m], ov[m]);
        double next = 0.0;
        if (FN == FN_ROSENBROCK && 4 * c + 4 < D)
            next = __dsub_rn((double)src[128 * q + 4], __ldg(o64 + 4 * c + 4));
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            if (4 * c + m >= D) break;
            rs.term(w64, D, 4 * c + m, z[m], m < 3 ? z[(m + 1) & 3] : next);
        }
    }
    return rs.finish(G, D);
}

// x is a NaN (by its bits: a compare would take the FP64 unit).
__device__ __forceinline__ bool is_nan_bits(double x)
{
    return ((unsigned long long)__double_as_longlong(x) << 1) > 0xffe0000000000000ull;
}

template <class Pos>
__host__ __device__ constexpr size_t rows_smem_per_warp()
{
    return (size_t)ROWS_SLICES * 128 * sizeof(Pos) + ROWS_SLICES * 32 * sizeof(uint32_t);
}

// The FP32 filter decides only above this lower bound.  E is relative to the
// sums, so each sum must stand clear of the denormal floats, where a square or a
// partial sum errs by up to 2^-149 absolutely.  Rastrigin and Rosenbrock: the
// value is the sum itself; 1024 such errors are below 2^-39 of 1e-30.  Ackley's
// value is at most 4 sqrt(s / D) + 54 s / D in s = sum z^2, so above 1e-16 s / D
// exceeds 6e-34: an error of 2^-149 a term is below 2^-38 of it.  (With 1e-30 for
// Ackley too, s of 1e-40 passed, whose squares had lost most of their bits.)
template <int FN> constexpr float FILTER_MIN = FN == FN_ACKLEY ? 1e-16f : 1e-30f;

// Blocks of 8 warps per SM the kernel is compiled for.
template <class Pos, bool F32R> struct RowsBound { static constexpr int min_blocks = F32R ? 4 : 3; };

template <class Pos, bool F32R, int FN, bool WIDE>
__global__ void __launch_bounds__(256, RowsBound<Pos, F32R>::min_blocks) bat_rows(const BatRowsParams p)
{
    constexpr bool FILTER = !F32R && FN != FN_SPHERE && FN != FN_ELLIPSOID;
    extern __shared__ __align__(16) unsigned char rows_smem[];
    const int lane = threadIdx.x & 31;
    const unsigned lt_mask = (1u << lane) - 1u;
    Pos* const stage = reinterpret_cast<Pos*>(rows_smem + (threadIdx.x >> 5) * rows_smem_per_warp<Pos>());
    uint32_t* const req = reinterpret_cast<uint32_t*>(stage + ROWS_SLICES * 128);
    const long long g = *p.gen;
    const uint32_t gg = (uint32_t)g;
    const int nwarps = (int)(gridDim.x * (blockDim.x >> 5));
    for (int t = (int)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)); t < p.n_tasks; t += nwarps) {
        const RowTask task = p.tasks[t];
        const InstDev& d = p.inst[task.inst];
        const int G = WIDE ? 32 : d.G;
        const int gpw = WIDE ? 1 : 32 / G;
        const int lane_g = lane & (G - 1), sub = WIDE ? 0 : lane / G;
        const unsigned gmask = WIDE || G == 32 ? 0xffffffffu : (((1u << G) - 1u) << (lane & ~(G - 1)));
        const int nch = d.nchunks, D = d.D, Dp = d.Dp;
        const int nq = WIDE ? (nch + 31) >> 5 : 1;
        const int np = task.n;
        const int rounds = (np + gpw - 1) / gpw;
        if (!PSSO_CHK(task.i0 >= 0 && task.i0 + np <= d.N && rounds * nq <= ROWS_SLICES && nch <= 32 * nq,
                      CHK_BAT_ROW, task.i0))
            continue;
        const uint32_t k0 = d.k0, k1 = d.k1;
        const uint32_t ibase = d.i_base + (uint32_t)task.i0;
        Pos* const X = static_cast<Pos*>(d.X) + (int64_t)task.i0 * Dp;
        Pos* const P = static_cast<Pos*>(d.P) + (int64_t)task.i0 * Dp;
        uint32_t neq = 0;       // bit r: this lane's chunks of round r differ from the pBest row
        int nreq = 0;           // warp-uniform
        __syncwarp();           // the previous task's stage is consumed

        // ---- pass 1: the interval draws; fresh-value requests ------------------------------
        {
            const uint32_t Tg = d.Tg > 0xffffffffull ? 0xffffffffu : (uint32_t)d.Tg;
            const uint32_t Tp = d.Tp > 0xffffffffull ? 0xffffffffu : (uint32_t)d.Tp;
            const uint32_t Tw = d.Tw > 0xffffffffull ? 0xffffffffu : (uint32_t)d.Tw;
            const bool fg = d.Tg > 0xffffffffull, fp = d.Tp > 0xffffffffull, fw = d.Tw > 0xffffffffull;
            const uint32_t ctr3 = TAG_RHO | (d.sid << 8);
            const bool paper = d.order != 0;
            const Pos* const gs = static_cast<const Pos*>(d.gbrow) + 4 * lane_g;
            int s = 0;
            for (int r = 0; r < rounds; ++r) {
                const int pi = r * gpw + sub;
                // sources of the first, second and third interval (Eq. 2.1 as printed
                // keeps x first and takes gBest third)
                const Pos* const own = X + (int64_t)pi * Dp + 4 * lane_g;
                const Pos* const src1 = paper ? own : gs;
                const Pos* const src2 = P + (int64_t)pi * Dp + 4 * lane_g;
                const Pos* const src3 = paper ? gs : own;
                for (int q = 0; q < nq; ++q, ++s) {
                    const int c = lane_g + 32 * q;
                    uint32_t nf = 0;
                    if (c < nch && pi < np) {
                        const uint32_t valid = 4 * c + 4 <= D ? 15u : (1u << (D - 4 * c)) - 1u;
                        Pos x[4] = {Pos(0), Pos(0), Pos(0), Pos(0)};
                        if (g == 0) {
                            nf = valid;
                        } else {
                            Pos v1[4], v2[4], v3[4];
                            ld4(src1 + 128 * q, v1);
                            ld4(src2 + 128 * q, v2);
                            ld4(src3 + 128 * q, v3);
                            const uint4 rb = philox10(make_uint4((uint32_t)c, ibase + (uint32_t)pi, gg, ctr3), k0, k1);
                            bool ne = false;
#pragma unroll
                            for (int m = 0; m < 4; ++m) {
                                const uint32_t w = word_of(rb, m);
                                const bool lg = w < Tg || fg, lp = w < Tp || fp, lw = w < Tw || fw;
                                // a variable of the last interval holds its pBest value (beyond
                                // D every source is 0)
                                x[m] = lg ? v1[m] : (lp || !lw) ? v2[m] : v3[m];
                                if (!lw) nf |= 1u << m;
                                ne = ne || !same_bits(x[m], v2[m]);
                            }
                            nf &= valid;
                            if (ne || nf) neq |= 1u << r;
                        }
                        st4(stage + 4 * (32 * s + lane), x);
                    }
                    const unsigned want = __ballot_sync(0xffffffffu, nf != 0u);
                    if (nf)   // slot | mask << 8 | chunk << 12 | particle << 20
                        req[nreq + __popc(want & lt_mask)] =
                            (uint32_t)(32 * s + lane) | (nf << 8) | ((uint32_t)c << 12) | ((uint32_t)pi << 20);
                    nreq += __popc(want);
                }
            }
        }
        __syncwarp();

        // ---- pass 2: the queued fresh-value blocks, one per lane and round --------------------
        bool equal_chunk = false;      // a request whose fresh values all equal the pBest's
        {
            Hot fh;                    // the fields fresh_chunk reads
            fh.sid = d.sid;
            fh.k0 = k0;
            fh.k1 = k1;
            fh.S32 = d.S32;
            fh.L32 = d.L32;
            fh.lbf = d.lbf;
            fh.ubf = d.ubf;
            fh.lb = d.lb;
            fh.ub = d.ub;
            fh.span = d.span;
            const uint32_t tag = g == 0 ? TAG_INIT : TAG_FRESH;
            for (int base = 0; base < nreq; base += 32) {
                const int e = base + lane;
                if (e < nreq) {
                    const uint32_t rq = req[e];
                    const uint32_t nf = (rq >> 8) & 15u;
                    Pos* const at = stage + 4 * (rq & 0xffu);
                    Pos fv[4], pv[4];
                    ld4(at, pv);
                    fresh_chunk(fv, nf, (rq >> 12) & 0xffu, ibase + (rq >> 20), gg, tag, fh);
                    bool ne = false;
#pragma unroll
                    for (int m = 0; m < 4; ++m)
                        if (nf & (1u << m)) {
                            ne = ne || !same_bits(fv[m], pv[m]);
                            pv[m] = fv[m];
                        }
                    st4(at, pv);
                    equal_chunk = equal_chunk || !ne;
                }
            }
        }
        // (in about one of 2^24 requests: the rows are then compared again)
        equal_chunk = __any_sync(0xffffffffu, equal_chunk) && g > 0;
        __syncwarp();

        // ---- pass 3: X, the fitness and the pBest decisions -----------------------------------
        // whether particle pi's staged row equals its pBest row (uniform over its group)
        auto same_row = [&](int r, int pi, bool valid) {
            bool ne = (neq >> r) & 1u;
            if (equal_chunk && ne) {
                ne = false;
                for (int q = 0; q < nq; ++q) {
                    const int c = lane_g + 32 * q;
                    if (!valid || c >= nch) continue;
                    Pos a[4], b[4];
                    ld4(stage + 4 * (32 * (r * nq + q) + lane), a);
                    ld4(P + (int64_t)pi * Dp + 4 * c, b);
#pragma unroll
                    for (int m = 0; m < 4; ++m) ne = ne || !same_bits(a[m], b[m]);
                }
            }
            return g > 0 && (__ballot_sync(0xffffffffu, ne) & gmask) == 0u;
        };
        // copies the staged row of particle pi (first slot s0) to its pBest row
        auto keep_row = [&](int pi, int s0) {
            for (int q = 0; q < nq; ++q) {
                const int c = lane_g + 32 * q;
                if (c >= nch) break;
                Pos v[4];
                ld4(stage + 4 * (s0 + 32 * q), v);
                st4(P + (int64_t)pi * Dp + 4 * c, v);
            }
        };
        int n_acc = 0;          // warp-uniform
        const float* const o32 = d.o32;
        const float* const w32 = d.w32;
        const double* const o64 = d.o64;
        double* const pf64 = d.pf64 + task.i0;
        uint32_t* const pver = d.pver + task.i0;
        float* const plo = F32R ? d.plo + task.i0 : nullptr;
        float* const phi = F32R ? d.phi + task.i0 : nullptr;
        uint32_t* const pflag = F32R ? d.pflag + task.i0 : nullptr;
        int nque = 0;           // particles left to FP64 (warp-uniform)
        if constexpr (F32R || FILTER) {
            for (int r = 0; r < rounds; ++r) {
                const int pi = r * gpw + sub;
                const bool valid = pi < np;
                float bl = 0.f, bh = 0.f;
                double pf = 0.0;
                if (valid && g > 0) {
                    if constexpr (F32R) {
                        bl = plo[pi];
                        bh = phi[pi];
                    } else {
                        pf = pf64[pi];
                    }
                }
                RowSum32<FN, F32R> rs;
                for (int q = 0; q < nq; ++q) {
                    const int c = lane_g + 32 * q;
                    if (c >= nch || !valid) continue;
                    const int slot = 32 * (r * nq + q) + lane;
                    Pos x[4];
                    ld4(stage + 4 * slot, x);
                    st4(X + (int64_t)pi * Dp + 4 * c, x);
                    float z[4], next = 0.f;
                    if constexpr (F32R) {
                        float ov[4];
                        ld4(o32 + 4 * c, ov);
#pragma unroll
                        for (int m = 0; m < 4; ++m) z[m] = __fsub_rn((float)x[m], ov[m]);
                        if (FN == FN_ROSENBROCK && 4 * c + 4 < D)
                            next = __fsub_rn((float)stage[4 * slot + 4], __ldg(o32 + 4 * c + 4));
                    } else {
                        double ov[4];
                        ld4(o64 + 4 * c, ov);
#pragma unroll
                        for (int m = 0; m < 4; ++m) z[m] = to_f32_trunc(__dsub_rn((double)x[m], ov[m]));
                        if (FN == FN_ROSENBROCK && 4 * c + 4 < D)
                            next = to_f32_trunc(__dsub_rn((double)stage[4 * slot + 4], __ldg(o64 + 4 * c + 4)));
                    }
#pragma unroll
                    for (int m = 0; m < 4; ++m) rs.term(w32, D, 4 * c + m, z[m], m < 3 ? z[(m + 1) & 3] : next);
                }
                const Fit32 fr = rs.finish(G, D, nq);
                const bool same = same_row(r, pi, valid);
                // (beyond the floats' range f - E is a NaN: nothing is known of the value)
                const float lo0 = fmaxf(__fsub_rd(fr.f, fr.E), -INFINITY);
                if constexpr (F32R) {
                    const float hi = fminf(__fadd_ru(fr.f, fr.E), INFINITY);
                    // an identical row: identical fitness, its state is kept
                    const bool keep = valid && same;
                    const bool take = valid && !same && (g == 0 || hi < bl);
                    const bool undecided = valid && !same && !take && !(lo0 > bh);
                    if (take) {
                        keep_row(pi, 32 * r * nq + lane);
                        if (lane_g == 0) {
                            pver[pi] = gg;
                            pf64[pi] = 0.0;
                            pflag[pi] = 0u;
                            plo[pi] = lo0;
                            phi[pi] = hi;
                        }
                    }
                    n_acc += __popc(__ballot_sync(0xffffffffu, (keep || take) && lane_g == 0));
                    const unsigned want = __ballot_sync(0xffffffffu, undecided && lane_g == 0);
                    if (undecided && lane_g == 0) req[nque + __popc(want & lt_mask)] = (uint32_t)pi;
                    nque += __popc(want);
                } else {
                    // an identical row has its pBest's value: accepted (<=) as it is;
                    // f32 - E above the pBest's value: rejected.  A NaN bound, and
                    // sums so small that the floats' range ends, go to FP64.
                    const bool keep = valid && same && !is_nan_bits(pf);
                    const bool reject = g > 0 && lo0 > FILTER_MIN<FN> && (double)lo0 > pf;
                    const bool need = valid && !keep && !reject;
                    if (keep && lane_g == 0) pver[pi] = gg;
                    n_acc += __popc(__ballot_sync(0xffffffffu, keep && lane_g == 0));
                    const unsigned want = __ballot_sync(0xffffffffu, need && lane_g == 0);
                    if (need && lane_g == 0) req[nque + __popc(want & lt_mask)] = (uint32_t)pi;
                    nque += __popc(want);
                }
            }
        }
        // FP64: the particles the bounds left undecided (all of them without a filter)
        __syncwarp();
        const int todo = (F32R || FILTER) ? nque : np;
        for (int base = 0; base < todo; base += gpw) {
            const int e = base + sub;
            const bool valid = e < todo;
            const int pi = !valid ? 0 : (F32R || FILTER) ? (int)req[e] : e;
            const int s0 = WIDE ? 32 * pi * nq + lane : 32 * (pi / gpw) + (pi & (gpw - 1)) * G + lane_g;
            if constexpr (!F32R && !FILTER) {
                for (int q = 0; q < nq; ++q) {
                    const int c = lane_g + 32 * q;
                    if (c >= nch || !valid) continue;
                    Pos x[4];
                    ld4(stage + 4 * (s0 + 32 * q), x);
                    st4(X + (int64_t)pi * Dp + 4 * c, x);
                }
            }
            const double f = row_f64<FN>(stage + 4 * s0, valid, lane_g, G, nch, nq, D, o64, d.w64);
            double pf = valid && g > 0 ? pf64[pi] : 0.0;
            bool accept;
            if constexpr (F32R) {
                const bool have_p = !valid || (pflag[pi] & 1u) != 0;
                if (__any_sync(0xffffffffu, !have_p)) {
                    const double fp = row_f64<FN>(P + (int64_t)pi * Dp + 4 * lane_g, !have_p, lane_g, G, nch, nq, D,
                                                  o64, d.w64);
                    if (!have_p) pf = fp;
                }
                accept = valid && f <= pf;
                __syncwarp();            // the group's reads of pf64 / pflag come first
                if (valid && lane_g == 0) {
                    const double v = accept ? f : pf;
                    pf64[pi] = v;
                    pflag[pi] = 1u;
                    plo[pi] = f64_to_f32_rd(v);
                    phi[pi] = f64_to_f32_ru(v);
                    if (accept) pver[pi] = gg;
                    atomicAdd(&p.cnt[task.inst].rck, have_p ? 1ull : 2ull);
                }
            } else {
                accept = valid && (g == 0 || f <= pf);
                __syncwarp();
                if (accept && lane_g == 0) {
                    pver[pi] = gg;
                    pf64[pi] = f;
                }
            }
            if (accept) keep_row(pi, s0);
            n_acc += __popc(__ballot_sync(0xffffffffu, accept && lane_g == 0));
        }
        if (lane == 0 && n_acc) atomicAdd(&p.cnt[task.inst].acc, (unsigned long long)n_acc);
    }
}

template <class Pos, bool F32R, int FN, bool WIDE>
inline cudaError_t rows_entry(int op, const BatRowsParams* p, int grid, cudaStream_t s, int* out)
{
    const size_t smem = 8 * rows_smem_per_warp<Pos>();
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(bat_rows<Pos, F32R, FN, WIDE>,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    if (op == 1) return cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, bat_rows<Pos, F32R, FN, WIDE>, 256, smem);
    bat_rows<Pos, F32R, FN, WIDE><<<grid, 256, smem, s>>>(*p);
    return cudaGetLastError();
}

template <class Pos, bool F32R>
inline cudaError_t rows_dispatch(int fn, bool wide, int op, const BatRowsParams* p, int grid, cudaStream_t s, int* out)
{
    switch (fn) {
#define PSSO_ROWS_FN(F) \
    case F: return wide ? rows_entry<Pos, F32R, F, true>(op, p, grid, s, out) : rows_entry<Pos, F32R, F, false>(op, p, grid, s, out)
    PSSO_ROWS_FN(FN_SPHERE);
    PSSO_ROWS_FN(FN_ELLIPSOID);
    PSSO_ROWS_FN(FN_RASTRIGIN);
    PSSO_ROWS_FN(FN_ROSENBROCK);
    PSSO_ROWS_FN(FN_ACKLEY);
#undef PSSO_ROWS_FN
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace psso
