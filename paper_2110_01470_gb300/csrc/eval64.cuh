// eval64.cuh -- FP64 fitness of many rows (psso_evaluate, psso_evaluate_noalloc)
// for the unrotated functions whose lane partials are independent (all but
// Schwefel 1.2, whose prefix sums cross the lanes).
//
// Bound: the FP64 unit.  On sm_103a an SM retires 1.66 FP64 lanes per clock
// and every FP64 instruction -- also compares, conversions and roundings --
// holds it for a whole warp, whatever the number of useful lanes, so what
// counts is the number of FP64 warp instructions per row.  One warp per row
// spent as many on the row's tail (Ackley: two expm1, two divisions, a square
// root, ten butterfly additions, all 32 lanes computing the same value) as on
// its terms, and ran the terms on 25 of 32 lanes at D = 100.  Here a warp
// takes up to 32 rows:
//   1. terms  the (row, summation lane) pairs of its rows are dealt to the
//             warp's lanes without gaps; a pair is a chain of its own (the
//             oracle's lane partial), stored to shared memory;
//   2. sums   the xor-butterfly tree of each row as a tree reduction over the
//             stored partials, at most 31 additions per row, dealt to all lanes
//             (a + b = b + a, so the tree gives lane 0's bits; a lane without
//             variables holds +0, or 1 in a product, and changes no bit: a
//             partial is never -0, since it starts from +0);
//   3. tail   one row per lane.
// The operations on each value and their order are the oracle's; only the
// lane that performs them changed.
// Ackley, N = 65536, D = 100: 650 -> 228 us per call (213 us of FP64 work).
#pragma once
#include "sso_common.cuh"

namespace psso {
namespace ev64 {

constexpr int WARPS = 4;          // per block: four warps saturate an SM's FP64 unit
constexpr int MAX_ROWS = 32;      // rows per warp
template <int FN> constexpr bool two_sums = FN == FN_ACKLEY || FN == FN_GRIEWANK;

// Summation lanes of a row that hold variables; its partials in shared memory
// are an odd number of doubles apart (no bank conflicts down a column).
__host__ __device__ inline int row_lanes(int nchunks) { return nchunks < 32 ? nchunks : 32; }
__host__ __device__ inline int row_pitch(int nchunks) { return row_lanes(nchunks) | 1; }

// The four terms of a chunk, in ascending variable order (z = 0 beyond D);
// dn is the next chunk's first z (Rosenbrock).  Griewank: w64 holds sqrt(j + 1).
template <int FN>
__device__ __forceinline__ void chunk_terms(const Hot& in, int c, const double (&z)[4], double dn, double& acc,
                                            double& acc2)
{
    if constexpr (FN == FN_POWELL) {
        const double a = __fma_rn(10.0, z[1], z[0]), b = __dsub_rn(z[2], z[3]);
        const double cc = __fma_rn(-2.0, z[2], z[1]), dd = __dsub_rn(z[0], z[3]);
        const double c2 = __dmul_rn(cc, cc), d2 = __dmul_rn(dd, dd);
        acc = __dadd_rn(acc, __fma_rn(a, a, __fma_rn(__dmul_rn(5.0, b), b,
                                                     __fma_rn(c2, c2, __dmul_rn(10.0, __dmul_rn(d2, d2))))));
    } else {
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const int j = 4 * c + m;
            if (j >= in.D) break;
            const double zj = z[m];
            if constexpr (FN == FN_SPHERE) {
                acc = __fma_rn(zj, zj, acc);
            } else if constexpr (FN == FN_ELLIPSOID) {
                acc = __fma_rn(__ldg(in.w64 + j), __dmul_rn(zj, zj), acc);
            } else if constexpr (FN == FN_RASTRIGIN) {
                acc = __dadd_rn(acc, __fma_rn(zj, zj, __dmul_rn(20.0, sinpi_sq_f64(zj))));
            } else if constexpr (FN == FN_ROSENBROCK) {
                if (j < in.D - 1) {
                    const double d1 = m < 3 ? z[(m + 1) & 3] : dn;
                    const double a0 = __dadd_rn(zj, 1.0), a1 = __dadd_rn(d1, 1.0);
                    const double u = __fma_rn(-a0, a0, a1);
                    acc = __dadd_rn(acc, __fma_rn(__dmul_rn(100.0, u), u, __dmul_rn(zj, zj)));
                }
            } else if constexpr (FN == FN_ACKLEY) {
                acc = __fma_rn(zj, zj, acc);
                const double s = sinpi_reduced_f64(__dsub_rn(zj, rint(zj)));
                acc2 = __fma_rn(s, s, acc2);
            } else if constexpr (FN == FN_GRIEWANK) {
                acc = __fma_rn(zj, zj, acc);
                acc2 = __dmul_rn(acc2, cos_rad_f64(__ddiv_rn(zj, __ldg(in.w64 + j))));
            } else {   // Schwefel
                acc = __fma_rn(zj, sin_rad_f64(__dsqrt_rn(fabs(zj))), acc);
            }
        }
    }
}

template <int FN>
__device__ __forceinline__ double tail(const Hot& in, double s, double s2)
{
    if constexpr (FN == FN_ACKLEY) {
        const double Dd = (double)in.D;
        const double A = __dsqrt_rn(__ddiv_rn(s, Dd));
        const double B = expm1_f64(__dmul_rn(-0.2, A));
        const double C = expm1_f64(__dmul_rn(-2.0, __ddiv_rn(s2, Dd)));
        return -__dadd_rn(__dmul_rn(20.0, B), __dmul_rn(0x1.5bf0a8b145769p+1, C));   // e
    } else if constexpr (FN == FN_GRIEWANK) {
        return __dadd_rn(__dsub_rn(1.0, s2), __ddiv_rn(s, 4000.0));
    } else if constexpr (FN == FN_SCHWEFEL) {
        return __dsub_rn(__dmul_rn(418.9829, (double)in.D), s);
    } else {
        return s;
    }
}

// Rows of X (pitch doubles apart) by warps of `rows` rows each.
template <int FN>
__global__ void __launch_bounds__(32 * WARPS) eval64(const Hot in, const double* __restrict__ X, int64_t pitch,
                                                     int64_t N, int rows, double* f, double* err)
{
    extern __shared__ double ev_smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t r0 = ((int64_t)blockIdx.x * WARPS + warp) * rows;
    if (r0 >= N) return;
    if (!PSSO_CHK(rows >= 1 && rows <= MAX_ROWS && in.nchunks * 4 >= in.D, CHK_EVAL_ROW, r0)) return;
    const int n = (int)(N - r0 < rows ? N - r0 : rows);
    const int L = row_lanes(in.nchunks), pitch_s = row_pitch(in.nchunks);
    constexpr int SUMS = two_sums<FN> ? 2 : 1;
    double* part = ev_smem + (size_t)warp * SUMS * rows * pitch_s;
    double* part2 = part + (SUMS - 1) * rows * pitch_s;
    constexpr double ONE2 = FN == FN_GRIEWANK ? 1.0 : 0.0;

    // 1. lane partials
    int row = lane / L, l = lane - row * L;
    const int step_r = 32 / L, step_l = 32 - step_r * L;
    for (; row < n;) {
        const double* xr = X + (r0 + row) * pitch;
        double acc = 0.0, acc2 = ONE2;
        for (int c = l; c < in.nchunks; c += 32) {
            double z[4];
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                const int j = 4 * c + m;
                z[m] = j < in.D ? __dsub_rn(xr[j], __ldg(in.o64 + j)) : 0.0;
            }
            double dn = 0.0;
            if constexpr (FN == FN_ROSENBROCK)
                if (4 * c + 4 < in.D) dn = __dsub_rn(xr[4 * c + 4], __ldg(in.o64 + 4 * c + 4));
            chunk_terms<FN>(in, c, z, dn, acc, acc2);
        }
        part[row * pitch_s + l] = acc;
        if constexpr (SUMS == 2) part2[row * pitch_s + l] = acc2;
        l += step_l;
        row += step_r;
        if (l >= L) { l -= L; ++row; }
    }
    __syncwarp();

    // 2. each row's butterfly, offsets 16, 8, 4, 2, 1: `off` pairs per row
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        for (int k = lane; k < n * off; k += 32) {
            const int at = (k / off) * pitch_s + (k & (off - 1));
            if ((k & (off - 1)) + off >= L) continue;
            double* p = part + at;
            p[0] = __dadd_rn(p[0], p[off]);
            if constexpr (SUMS == 2) {
                double* p2 = part2 + at;
                p2[0] = FN == FN_GRIEWANK ? __dmul_rn(p2[0], p2[off]) : __dadd_rn(p2[0], p2[off]);
            }
        }
        __syncwarp();
    }

    // 3. one row per lane
    if (lane < n) {
        f[r0 + lane] = tail<FN>(in, part[lane * pitch_s], SUMS == 2 ? part2[lane * pitch_s] : 0.0);
        if (err) err[r0 + lane] = 0.0;
    }
}

// Whether eval64 covers function fn (else the warp-per-row kernels).
inline bool covers(int fn)
{
    return fn >= FN_SPHERE && fn <= FN_SCHWEFEL && !(fn >= FN_ROT_ELLIPSOID && fn <= FN_ROT_ACKLEY) &&
           fn != FN_SCHWEFEL12 && fn != FN_HYPER_ELLIPSOID;
}

template <int FN>
inline cudaError_t launch_fn(const Hot& in, const double* X, int64_t pitch, int64_t N, int rows, double* f,
                             double* err, cudaStream_t s)
{
    const size_t smem = (size_t)WARPS * rows * row_pitch(in.nchunks) * sizeof(double) * (two_sums<FN> ? 2 : 1);
    if (smem > 48 * 1024) {
        // an SM's whole 227 KB, whatever this call uses: calls on other threads share the kernel
        const cudaError_t e = cudaFuncSetAttribute(eval64<FN>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        if (e != cudaSuccess) return e;
    }
    const int64_t per_block = (int64_t)WARPS * rows;
    eval64<FN><<<(unsigned)((N + per_block - 1) / per_block), 32 * WARPS, smem, s>>>(in, X, pitch, N, rows, f, err);
    return cudaGetLastError();
}

// Rows per warp: the blocks (four warps) come out as a whole number per SM, so
// no SM works through a second wave alone; at least two per SM (one's tail
// hides under the other's terms) and as many as 32 rows per warp need.  Few
// rows spread over as many warps, down to one row each.
inline int rows_per_warp(int64_t N, int sms)
{
    const int64_t slots = (int64_t)sms * WARPS;
    const int64_t k = std::max<int64_t>(2, (N + slots * MAX_ROWS - 1) / (slots * MAX_ROWS));
    return (int)((N + slots * k - 1) / (slots * k));
}

inline cudaError_t launch(const Hot& in, const double* X, int64_t pitch, int64_t N, int sms, double* f, double* err,
                          cudaStream_t s)
{
    const int rows = rows_per_warp(N, sms);
    switch (in.fn) {
    case FN_SPHERE: return launch_fn<FN_SPHERE>(in, X, pitch, N, rows, f, err, s);
    case FN_ELLIPSOID: return launch_fn<FN_ELLIPSOID>(in, X, pitch, N, rows, f, err, s);
    case FN_RASTRIGIN: return launch_fn<FN_RASTRIGIN>(in, X, pitch, N, rows, f, err, s);
    case FN_ROSENBROCK: return launch_fn<FN_ROSENBROCK>(in, X, pitch, N, rows, f, err, s);
    case FN_ACKLEY: return launch_fn<FN_ACKLEY>(in, X, pitch, N, rows, f, err, s);
    case FN_GRIEWANK: return launch_fn<FN_GRIEWANK>(in, X, pitch, N, rows, f, err, s);
    case FN_POWELL: return launch_fn<FN_POWELL>(in, X, pitch, N, rows, f, err, s);
    case FN_SCHWEFEL: return launch_fn<FN_SCHWEFEL>(in, X, pitch, N, rows, f, err, s);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace ev64
}  // namespace psso
