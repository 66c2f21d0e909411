// gradient.cu -- differentiable batched fitness: FP32 forward and backward
// kernels for every test function (psso_fitness_forward / _backward), and the
// gBest gradient polish of a swarm (the kernel behind psso_polish).
//
// Gradients with z the function's coordinates (z = x - o, or z = M (x - o)):
//   sphere      2 z_j                        ellipsoid   2 w_j z_j
//   Rastrigin   2 z_j + 20 pi sin(2 pi z_j)
//   Rosenbrock  [j<D-1] (2 d_j - 400 a_j u_j) + [j>0] 200 u_{j-1},
//               a = d + 1, u_j = a_{j+1} - a_j^2 = d_{j+1} - d_j (d_j + 2)
//   Ackley      4 e^{-0.2 A} z_j / (A D) + 2 pi e^{C} sin(2 pi z_j) / D,
//               A = sqrt(sum z^2 / D), C = sum cos(2 pi z) / D = 1 - 2 Q / D
// and for rotated functions df/dx = M^T df/dz.
#include "psso.h"
#include "rot_pipeline.h"
#include "sso_kernel.cuh"
#include "tc_pair.cuh"

namespace psso {

// sin(2 pi z) in FP32: 2z = n + r, sin(pi (n + r)) = (-1)^n sin(pi r).
__device__ __forceinline__ float sin2pi_f32(float z)
{
    const float y = __fmul_rn(2.f, z);
    const float n = rintf(y);
    const float s = sinpi_reduced_f32(__fsub_rn(y, n));
    return (((int)n) & 1) ? -s : s;
}

// Fitness (FP32) and its gradient with respect to x for one row held by a full
// warp in the 32-lane chunk layout (x: lane chunks lane + 32 q).
template <int MAXC, bool WANT_GRAD = true>
__device__ float grad32(const Hot& in, const float (&x)[MAXC][4], float (&gx)[MAXC][4])
{
    const int lane = threadIdx.x & 31;
    const int D = in.D;
    const bool rot = is_rotated(in.fn);
    const int fn = base_fn(in.fn);
    float z[MAXC][4], gz[MAXC][4];
    if (rot) {
        float ez[MAXC][4];
        rot_matvec32<MAXC>(in, x, lane, 0xffffffffu, 32, z, ez);
    } else {
#pragma unroll
        for (int q = 0; q < MAXC; ++q)
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                const int j = 4 * (lane + 32 * q) + m;
                z[q][m] = (j < D) ? __fsub_rn(x[q][m], __ldg(in.o32 + j)) : 0.f;
            }
    }
    // Sums each function needs (all lanes end with the totals).
    float s1 = 0.f, s2 = 0.f;
#pragma unroll
    for (int q = 0; q < MAXC; ++q)
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const int j = 4 * (lane + 32 * q) + m;
            if (j >= D) continue;
            const float zj = z[q][m];
            if (fn == FN_ACKLEY) {
                s1 = __fmaf_rn(zj, zj, s1);
                const float s = sinpi_reduced_f32(__fsub_rn(zj, rintf(zj)));
                s2 = __fmaf_rn(s, s, s2);
            }
        }
    float Ae = 0.f, Ce = 0.f, A = 0.f;
    if (fn == FN_ACKLEY) {
        for (int off = 16; off > 0; off >>= 1) {
            s1 += __shfl_xor_sync(0xffffffffu, s1, off);
            s2 += __shfl_xor_sync(0xffffffffu, s2, off);
        }
        A = sqrtf(s1 / (float)D);
        Ae = expf(-0.2f * A);                        // e^{-0.2 A}
        Ce = 2.7182818f * expf(-2.f * s2 / (float)D);  // e^{C}
    }
    // Rosenbrock terms u_j = d_{j+1} - d_j (d_j + 2): d_{j+1} is the same lane's
    // next variable, or the first variable of the next chunk (lane + 1, or lane 0
    // of the next q for lane 31).
    float u[MAXC][4];
#pragma unroll
    for (int q = 0; q < MAXC; ++q) {
        const float first_next = __shfl_down_sync(0xffffffffu, z[q][0], 1);
        const float wrap = __shfl_sync(0xffffffffu, z[(q + 1) % MAXC][0], 0);
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const int j = 4 * (lane + 32 * q) + m;
            float nx = (m < 3) ? z[q][m < 3 ? m + 1 : 0] : (lane == 31 ? (q + 1 < MAXC ? wrap : 0.f) : first_next);
            if (j + 1 >= D) nx = 0.f;
            u[q][m] = __fmaf_rn(-z[q][m], __fadd_rn(z[q][m], 2.f), nx);
        }
    }
    float f = 0.f;
#pragma unroll
    for (int q = 0; q < MAXC; ++q) {
        // u_{j-1}: same lane (m > 0), lane - 1's last term, or lane 31's last term of q - 1
        const float last_prev = __shfl_up_sync(0xffffffffu, u[q][3], 1);
        const float wrap = __shfl_sync(0xffffffffu, u[(q + MAXC - 1) % MAXC][3], 31);
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const int j = 4 * (lane + 32 * q) + m;
            const float up = (m > 0) ? u[q][m > 0 ? m - 1 : 0] : (lane == 0 ? (q > 0 ? wrap : 0.f) : last_prev);
            float g = 0.f;
            const float zj = z[q][m];
            if (j < D) {
                switch (fn) {
                case FN_SPHERE:
                    g = 2.f * zj;
                    f = __fmaf_rn(zj, zj, f);
                    break;
                case FN_ELLIPSOID: {
                    const float w = __ldg(in.w32 + j);
                    g = 2.f * w * zj;
                    f = __fmaf_rn(w * zj, zj, f);
                    break;
                }
                case FN_RASTRIGIN: {
                    const float s = sinpi_reduced_f32(__fsub_rn(zj, rintf(zj)));
                    g = __fmaf_rn(62.8318548f, sin2pi_f32(zj), 2.f * zj);
                    f = __fadd_rn(f, __fmaf_rn(zj, zj, 20.f * s * s));
                    break;
                }
                case FN_ROSENBROCK: {
                    const float a = __fadd_rn(zj, 1.f);
                    if (j < D - 1) {
                        g = __fmaf_rn(-400.f * a, u[q][m], 2.f * zj);
                        f = __fadd_rn(f, __fmaf_rn(100.f * u[q][m], u[q][m], zj * zj));
                    }
                    if (j > 0) g = __fmaf_rn(200.f, up, g);
                    break;
                }
                default: {   // Ackley
                    const float lin = (A > 0.f) ? 4.f * Ae * zj / (A * (float)D) : 0.f;
                    g = __fmaf_rn(6.28318548f * Ce / (float)D, sin2pi_f32(zj), lin);
                    break;
                }
                }
            }
            gz[q][m] = g;
        }
    }
    if (fn == FN_ACKLEY) {
        f = -20.f * expm1f(-0.2f * A) - 2.7182818f * expm1f(-2.f * s2 / (float)D);
    } else {
        for (int off = 16; off > 0; off >>= 1) f += __shfl_xor_sync(0xffffffffu, f, off);
    }
    if (!rot || !WANT_GRAD) {
#pragma unroll
        for (int q = 0; q < MAXC; ++q)
#pragma unroll
            for (int m = 0; m < 4; ++m) gx[q][m] = gz[q][m];
        return f;
    }
    // df/dx_k = sum_j M_jk df/dz_j: each df/dz_j broadcast from its lane.
#pragma unroll
    for (int q = 0; q < MAXC; ++q)
#pragma unroll
        for (int m = 0; m < 4; ++m) gx[q][m] = 0.f;
#pragma unroll
    for (int qj = 0; qj < MAXC; ++qj) {
        for (int l = 0; l < 32; ++l) {
            if (128 * qj + 4 * l >= D) break;
#pragma unroll
            for (int mj = 0; mj < 4; ++mj) {
                const int j = 128 * qj + 4 * l + mj;
                const float gj = __shfl_sync(0xffffffffu, gz[qj][mj], l);
                if (j < D) {
#pragma unroll
                    for (int q = 0; q < MAXC; ++q)
#pragma unroll
                        for (int m = 0; m < 4; ++m) {
                            const int k = 4 * (lane + 32 * q) + m;
                            if (k < D) gx[q][m] = __fmaf_rn(__ldg(in.M32 + (size_t)j * D + k), gj, gx[q][m]);
                        }
                }
            }
        }
    }
    return f;
}

// One warp per row of X (N x D floats, unpadded): f (forward) or grad_X =
// grad_f[row] * df/dx (backward).
template <bool BWD, int MAXC>
__device__ void fb_row(const Hot& in, const float* xr, float gfr, float* f, float* gxr)
{
    const int lane = threadIdx.x & 31;
    float x[MAXC][4], g[MAXC][4];
#pragma unroll
    for (int q = 0; q < MAXC; ++q)
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const int j = 4 * (lane + 32 * q) + m;
            x[q][m] = j < in.D ? xr[j] : 0.f;
        }
    const float v = grad32<MAXC, BWD>(in, x, g);
    if constexpr (!BWD) {
        if (lane == 0) *f = v;
    } else {
#pragma unroll
        for (int q = 0; q < MAXC; ++q)
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                const int j = 4 * (lane + 32 * q) + m;
                if (j < in.D) gxr[j] = gfr * g[q][m];
            }
    }
}

template <bool BWD>
__global__ void fitness_fb(const Hot in, const float* X, int64_t N, const float* gf, float* f, float* gx)
{
    const int64_t row = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (row >= N) return;
    if (!PSSO_CHK(in.maxc * 128 >= in.D, CHK_EVAL_ROW, in.D)) return;
    const float* xr = X + row * in.D;
    const float gfr = BWD ? gf[row] : 0.f;
    float* fo = BWD ? nullptr : f + row;
    float* gxr = BWD ? gx + row * in.D : nullptr;
    switch (in.maxc) {
    case 1: fb_row<BWD, 1>(in, xr, gfr, fo, gxr); break;
    case 2: fb_row<BWD, 2>(in, xr, gfr, fo, gxr); break;
    case 4: fb_row<BWD, 4>(in, xr, gfr, fo, gxr); break;
    default: fb_row<BWD, 8>(in, xr, gfr, fo, gxr); break;
    }
}

// gBest polish of instance k: `steps` gradient steps x <- clamp(x - lr df/dx)
// from the gBest row, then the polished row's FP64 fitness in the oracle's
// order; it replaces the gBest particle's pBest (and the gBest) only if that
// value is lower.  Multi-block instances also get the owner block's record
// and row of generation g rewritten, so the next launch sees the new gBest.
template <class Pos, int MAXC>
__device__ void polish_row(const InstDev& in, int owner_rank, int64_t g, int steps, float lr)
{
    const int lane = threadIdx.x & 31;
    const Hot hin = hot_of(in);
    const Pos lo_b = sizeof(Pos) == 4 ? (Pos)in.lbf : (Pos)in.lb;
    const Pos hi_b = sizeof(Pos) == 4 ? (Pos)in.ubf : (Pos)in.ub;
    Pos xp[MAXC][4];
#pragma unroll
    for (int q = 0; q < MAXC; ++q) {
        const int c = lane + 32 * q;
        if (c < in.nchunks) ld4(static_cast<const Pos*>(in.gbrow) + 4 * c, xp[q]);
        else xp[q][0] = xp[q][1] = xp[q][2] = xp[q][3] = Pos(0);
    }
    const double fold = in.gb->has64 ? in.gb->f64 : fit64<Pos, MAXC>(hin, xp, lane, 0xffffffffu, 32);
    // The gradient is taken in FP32 at the row rounded to floats; the step is
    // applied to the row in its own precision and clamped to the box.
    for (int s = 0; s < steps; ++s) {
        float x[MAXC][4], gr[MAXC][4];
#pragma unroll
        for (int q = 0; q < MAXC; ++q)
#pragma unroll
            for (int m = 0; m < 4; ++m) x[q][m] = (float)xp[q][m];
        grad32<MAXC, true>(hin, x, gr);
#pragma unroll
        for (int q = 0; q < MAXC; ++q)
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                const int j = 4 * (lane + 32 * q) + m;
                if (j < in.D) {
                    const Pos v = xp[q][m] - (Pos)(lr * gr[q][m]);
                    xp[q][m] = v < lo_b ? lo_b : (v > hi_b ? hi_b : v);
                }
            }
    }
    const double fnew = fit64<Pos, MAXC>(hin, xp, lane, 0xffffffffu, 32);
    if (!(fnew < fold)) return;
    const int64_t b = in.gb->idx;
    if (!PSSO_CHK(b >= 0 && b < in.N && owner_rank < in.R, CHK_GBEST_SRC, b)) return;
    Pos* prow = static_cast<Pos*>(in.P) + b * in.Dp;
    Pos* gw = static_cast<Pos*>(in.gbrow);
#pragma unroll
    for (int q = 0; q < MAXC; ++q) {
        const int c = lane + 32 * q;
        if (c < in.nchunks) {
            st4(prow + 4 * c, xp[q]);
            st4(gw + 4 * c, xp[q]);
        }
    }
    const float lo = f64_to_f32_rd(fnew), hi = f64_to_f32_ru(fnew);
    if (in.R > 1 && owner_rank >= 0) {
        constexpr int WPE = WordsPer<Pos>::value;
        const uint32_t tag = (uint32_t)g;
        uint64_t* rw = static_cast<uint64_t*>(in.grow) +
                       ((size_t)slot_of(g) * in.R + owner_rank) * (size_t)in.Dp * WPE;
#pragma unroll
        for (int q = 0; q < MAXC; ++q) {
            const int c = lane + 32 * q;
            if (c < in.nchunks) put_chunk(rw + (size_t)4 * c * WPE, tag, xp[q]);
        }
    }
    __syncwarp();
    if (lane == 0) {
        in.pf64[b] = fnew;
        in.pver[b] = (uint32_t)g;
        if (in.plo) {
            in.plo[b] = lo;
            in.phi[b] = hi;
            in.pflag[b] = 1u;
        }
        in.gb->f64 = fnew;
        in.gb->has64 = 1;
        in.gb->lo = lo;
        in.gb->hi = hi;
        in.gb->ver = (uint32_t)g;
        if (in.R > 1 && owner_rank >= 0) {
            uint64_t* rec = in.rec + ((size_t)slot_of(g) * in.R + owner_rank) * REC_WORDS;
            Winner w;
            w.idx = b;
            w.ver = (uint32_t)g;
            w.has64 = 1;
            w.f64 = fnew;
            w.lo = lo;
            w.hi = hi;
            w.acc = rec[RW_ACC] & 0xffffffffffffULL;
            w.rck = rec[RW_RCK] & 0xffffffffffffULL;
            publish_record(rec, (uint32_t)g, w);
        }
    }
}

template <class Pos>
__global__ void polish_kernel(const InstDev* inst, int k, int owner_rank, int64_t g, int steps, float lr)
{
    const InstDev& in = inst[k];
    switch (in.maxc) {
    case 1: polish_row<Pos, 1>(in, owner_rank, g, steps, lr); break;
    case 2: polish_row<Pos, 2>(in, owner_rank, g, steps, lr); break;
    case 4: polish_row<Pos, 4>(in, owner_rank, g, steps, lr); break;
    default: polish_row<Pos, 8>(in, owner_rank, g, steps, lr); break;
    }
}

cudaError_t launch_polish(const InstDev* inst, int k, int lattice, int owner_rank, int64_t g, int steps,
                          float lr, cudaStream_t s)
{
    if (lattice == 1) polish_kernel<float><<<1, 32, 0, s>>>(inst, k, owner_rank, g, steps, lr);
    else polish_kernel<double><<<1, 32, 0, s>>>(inst, k, owner_rank, g, steps, lr);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Rotated functions on the tensor cores (the *_ws entry points):
//   forward   planes of d = x - o and of M          prep_planes
//             Z = (X - O) M^T, its epilogue the     pair GEMM, SumEpi
//             terms of f summed per row and 64 columns
//             f_i from the sums                     finish_rows
//   backward  planes of d, M and M^T                prep_planes
//             Z = (X - O) M^T                       pair GEMM, StoreEpi
//             planes of G_i = grad_f_i df/dz        gz_rows
//             grad_X = G M                          pair GEMM, StoreEpi
// The GEMMs (tc_pair.cuh) run the six split products of tc_gemm.cuh with FP32
// accumulation: each output carries an error below 2^-20 per MMA of
// sum |A_ik| |B_jk| (tc_gemm.cuh), typically far less.
//
// Bound: the tensor pipe for large N D^2 (six products each), HBM for the
// planes, launches for small ones.  Against one CTA per 128 x 128 tile with Z
// stored a word at a time, a warp per row for f and for the planes of G, and
// the outputs pre-filled with NaN (forward + backward): rotated Ackley, N =
// 4096, D = 256: 123 -> 63 us; rotated Rastrigin, N = 8192, D = 1000: 568
// -> 303 us; with the sequence's launches overlapped (pdl.cuh) 51 and 288 us.
namespace gtc {

using tc::BM;
using tc::BN;
using tc::BK;

// Four consecutive values as the three planes' BF16 (8 bytes each at offset o).
__device__ __forceinline__ void put_planes(const float (&v)[4], __nv_bfloat16* A, size_t plane, size_t o)
{
    uint32_t w[3][2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        __nv_bfloat16 a[3], b[3];
        tc::split3(v[2 * h], a[0], a[1], a[2]);
        tc::split3(v[2 * h + 1], b[0], b[1], b[2]);
#pragma unroll
        for (int p = 0; p < 3; ++p)
            w[p][h] = (uint32_t)__bfloat16_as_ushort(a[p]) | ((uint32_t)__bfloat16_as_ushort(b[p]) << 16);
    }
#pragma unroll
    for (int p = 0; p < 3; ++p) *reinterpret_cast<uint2*>(A + p * plane + o) = make_uint2(w[p][0], w[p][1]);
}

// Values 4 c .. 4 c + 3 of a row of D floats (zero beyond); vec: 16-byte loads.
__device__ __forceinline__ void row4(const float* row, int c, int D, bool vec, float (&v)[4])
{
    if (vec && 4 * c + 4 <= D) {
        ld4(row + 4 * c, v);
        return;
    }
#pragma unroll
    for (int m = 0; m < 4; ++m) v[m] = 4 * c + m < D ? __ldg(row + 4 * c + m) : 0.f;
}

// Operand planes of one call in one launch: a warp per row of X (d = x - o) and
// per row of M, then 32 x 32 tiles of M^T.  Columns D .. Kp - 1 are zero; rows
// beyond N and D are left as they are (an output element depends on its own
// row and column only, and theirs are not stored).
struct PrepArgs {
    const float* X;
    const float* o;
    const float* M;
    __nv_bfloat16 *A, *B, *Bt;      // Bt may be null
    int* status;
    int N, D, Np, Jp, Kp;
    int row_blocks;                 // blocks of 8 rows of X and M together
    bool vec_x, vec_m;
};
__global__ void __launch_bounds__(256) prep_planes(const PrepArgs a)
{
    pdl_trigger();
    __shared__ float tile[32][33];
    if (blockIdx.x == 0 && threadIdx.x == 0) *a.status = 0;
    if ((int)blockIdx.x < a.row_blocks) {
        const int lane = threadIdx.x & 31;
        const int r = (int)blockIdx.x * 8 + (threadIdx.x >> 5);
        if (r >= a.N + a.D) return;
        const bool is_x = r < a.N;
        const int i = is_x ? r : r - a.N;
        const float* src = (is_x ? a.X : a.M) + (size_t)i * a.D;
        __nv_bfloat16* dst = is_x ? a.A : a.B;
        const size_t plane = (size_t)(is_x ? a.Np : a.Jp) * a.Kp;
        const bool vec = is_x ? a.vec_x : a.vec_m;
        for (int c = lane; c < a.Kp / 4; c += 32) {
            float v[4];
            row4(src, c, a.D, vec, v);
            if (is_x) {
#pragma unroll
                for (int m = 0; m < 4; ++m)
                    if (4 * c + m < a.D) v[m] = __fsub_rn(v[m], __ldg(a.o + 4 * c + m));
            }
            put_planes(v, dst, plane, (size_t)i * a.Kp + 4 * c);
        }
        return;
    }
    // Bt[k][j] = M[j][k]: tile (k0, j0)
    const int t = (int)blockIdx.x - a.row_blocks, nt = a.Kp / 32;
    const int k0 = (t / nt) * 32, j0 = (t % nt) * 32;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    for (int y = ty; y < 32; y += 8)
        tile[y][tx] = (j0 + y < a.D && k0 + tx < a.D) ? __ldg(a.M + (size_t)(j0 + y) * a.D + k0 + tx) : 0.f;
    __syncthreads();
    const int k = k0 + (threadIdx.x >> 3), c = threadIdx.x & 7;
    if (k < a.D) {
        const float v[4] = {tile[4 * c][k - k0], tile[4 * c + 1][k - k0], tile[4 * c + 2][k - k0],
                            tile[4 * c + 3][k - k0]};
        put_planes(v, a.Bt, (size_t)a.Jp * a.Kp, (size_t)k * a.Kp + j0 + 4 * c);
    }
}

// The terms of f summed over the 64 columns: part[i][g] = (s1, s2) (ellipsoid
// sum w z^2, Rastrigin sum z^2 + 20 sin^2, Ackley sum z^2 and sum sin^2).
// Blocks of 32 terms, then the two blocks: with the tree of finish_rows the longest
// chain is 32 + 1 + 4 additions (D = 1024).
struct SumEpi : tc::JoinEpi {
    float2* part;
    const float* w;
    int fn, groups;
    __device__ __forceinline__ void compute(int c0, int n, float4* xch)
    {
        float s1 = 0.f, s2 = 0.f, a1 = 0.f, a2 = 0.f;
#pragma unroll 1
        for (int h = 0; h < 4 * n; ++h) {            // eight columns a step (short code)
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int j = 64 * g + 32 * c0 + 8 * h + q;
                if (j >= D) break;
                const float zj = z[0][q];
                if (fn == FN_ELLIPSOID) {
                    a1 = __fmaf_rn(__fmul_rn(__ldg(w + j), zj), zj, a1);
                } else {
                    const float sn = sinpi_reduced_f32(__fsub_rn(zj, rint_f32(zj)));
                    if (fn == FN_RASTRIGIN) {
                        a1 = __fadd_rn(a1, __fmaf_rn(zj, zj, __fmul_rn(__fmul_rn(20.f, sn), sn)));
                    } else {
                        a1 = __fmaf_rn(zj, zj, a1);
                        a2 = __fmaf_rn(sn, sn, a2);
                    }
                }
            }
#pragma unroll
            for (int q = 0; q < 56; ++q) z[q >> 5][q & 31] = z[(q + 8) >> 5][(q + 8) & 31];
            if ((h & 3) == 3) {                      // a block of 32 terms ends
                s1 = __fadd_rn(s1, a1);
                s2 = __fadd_rn(s2, a2);
                a1 = a2 = 0.f;
            }
        }
        if (n == 1) {
            const float4 o = tc::pair_exchange(make_float4(s1, s2, 0.f, 0.f), c0, xch);
            if (c0 == 1) return;
            s1 = __fadd_rn(s1, o.x);
            s2 = __fadd_rn(s2, o.y);
        }
        if (i < N && g < groups) part[(size_t)i * groups + g] = make_float2(s1, s2);
    }
};

template <class Epi>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(tc::P_THREADS, 1)
    pair_gemm(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const tc::GemmArgs a,
              const __grid_constant__ Epi epi0)
{
    Epi epi = epi0;
    epi.chains = a.Kp / BK < 3 ? a.Kp / BK : 3;
    tc::gemm_pair<tc::SplitCfg>(&tmA, &tmB, a, epi);
}

// f from the sums of its terms (a thread per row); NaN if a GEMM wait ran out.
__global__ void finish_rows(const float2* part, int groups, int fn, int N, int D, const int* status, float* f)
{
    pdl_entry();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    float p1[16], p2[16];                    // at most 1024 / 64 groups, added as a tree
#pragma unroll
    for (int t = 0; t < 16; ++t) {
        const float2 p = t < groups ? part[(size_t)i * groups + t] : make_float2(0.f, 0.f);
        p1[t] = p.x;
        p2[t] = p.y;
    }
#pragma unroll
    for (int w = 8; w > 0; w >>= 1)
#pragma unroll
        for (int t = 0; t < 8; ++t)
            if (t < w) {
                p1[t] = __fadd_rn(p1[t], p1[t + w]);
                p2[t] = __fadd_rn(p2[t], p2[t + w]);
            }
    const float s1 = p1[0], s2 = p2[0];
    float v = s1;
    if (fn == FN_ACKLEY)
        v = -20.f * expm1f(-0.2f * sqrtf(s1 / (float)D)) - 2.7182818f * expm1f(-2.f * s2 / (float)D);
    f[i] = *status ? __int_as_float(0x7fffffff) : v;
}

// Outputs of a backward pass whose GEMM wait ran out: NaN, never stale values.
__global__ void poison(float* out, size_t n, const int* status)
{
    pdl_entry();
    if (!*status) return;
    for (size_t q = (size_t)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += (size_t)gridDim.x * blockDim.x)
        out[q] = __int_as_float(0x7fffffff);
}

// A planes of G = grad_f_i df/dz for the rows of Z, a warp per row (the
// functions' gradients as in grad32; Ackley's row sums first, the row kept in
// registers).
template <int FN, int MAXC>
__global__ void __launch_bounds__(256) gz_rows(const float* __restrict__ Z, const float* __restrict__ w,
                                               const float* __restrict__ gf, int N, int D, int Np, int Kp,
                                               __nv_bfloat16* A)
{
    pdl_entry();
    const int i = (int)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (i >= N) return;
    const int lane = threadIdx.x & 31, nc = Kp / 4;
    const float* row = Z + (size_t)i * D;
    const bool vec = (D & 3) == 0;
    float z[MAXC][4];
#pragma unroll
    for (int q = 0; q < MAXC; ++q) row4(row, lane + 32 * q, D, vec, z[q]);
    float c_lin = 0.f, c_sin = 0.f;
    if constexpr (FN == FN_ACKLEY) {
        float s1 = 0.f, s2 = 0.f;
#pragma unroll
        for (int q = 0; q < MAXC; ++q)
#pragma unroll
            for (int m = 0; m < 4; ++m) {       // zero beyond D
                s1 = __fmaf_rn(z[q][m], z[q][m], s1);
                const float s = sinpi_reduced_f32(__fsub_rn(z[q][m], rint_f32(z[q][m])));
                s2 = __fmaf_rn(s, s, s2);
            }
        for (int off = 16; off > 0; off >>= 1) {
            s1 += __shfl_xor_sync(0xffffffffu, s1, off);
            s2 += __shfl_xor_sync(0xffffffffu, s2, off);
        }
        const float Av = sqrtf(s1 / (float)D);
        c_lin = Av > 0.f ? 4.f * expf(-0.2f * Av) / (Av * (float)D) : 0.f;
        c_sin = 6.28318548f * (2.7182818f * expf(-2.f * s2 / (float)D)) / (float)D;
    }
    const float scale = gf[i];
    const size_t plane = (size_t)Np * Kp;
#pragma unroll
    for (int q = 0; q < MAXC; ++q) {
        const int c = lane + 32 * q;
        if (c >= nc) break;
        float g[4];
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const float zj = z[q][m];
            float v;
            if constexpr (FN == FN_ELLIPSOID) v = 4 * c + m < D ? 2.f * __ldg(w + 4 * c + m) * zj : 0.f;
            else if constexpr (FN == FN_RASTRIGIN) v = __fmaf_rn(62.8318548f, sin2pi_f32(zj), 2.f * zj);
            else v = __fmaf_rn(c_sin, sin2pi_f32(zj), c_lin * zj);
            g[m] = __fmul_rn(scale, v);
            if (4 * c + m >= D) g[m] = 0.f;      // (an infinite scale would make a NaN of 0)
        }
        put_planes(g, A, plane, (size_t)i * Kp + 4 * c);
    }
}

template <int FN>
inline void launch_gz(int maxc, const float* Z, const float* w, const float* gf, int N, int D, int Np, int Kp,
                      __nv_bfloat16* A, cudaStream_t s)
{
    const unsigned grid = (unsigned)((N + 7) / 8);
    switch (maxc) {
    case 1: launch_pdl(gz_rows<FN, 1>, dim3(grid), dim3(256), 0, s, Z, w, gf, N, D, Np, Kp, A); break;
    case 2: launch_pdl(gz_rows<FN, 2>, dim3(grid), dim3(256), 0, s, Z, w, gf, N, D, Np, Kp, A); break;
    case 4: launch_pdl(gz_rows<FN, 4>, dim3(grid), dim3(256), 0, s, Z, w, gf, N, D, Np, Kp, A); break;
    default: launch_pdl(gz_rows<FN, 8>, dim3(grid), dim3(256), 0, s, Z, w, gf, N, D, Np, Kp, A); break;
    }
}

// Workspace layout of the tensor-core path (byte offsets, 256-aligned).
struct WsLayout {
    int Np, Jp, Kp;
    size_t a, b, bt, z, status, total;
};
inline size_t al256(size_t v) { return (v + 255) & ~(size_t)255; }
inline WsLayout ws_layout(int64_t N, int64_t D)
{
    WsLayout w{};
    w.Np = (int)((N + BM - 1) / BM * BM);
    w.Jp = (int)((D + BN - 1) / BN * BN);
    w.Kp = (int)((D + BK - 1) / BK * BK);
    size_t off = 0;
    auto take = [&](size_t n) { const size_t at = off; off = al256(off + n); return at; };
    w.a = take((size_t)3 * w.Np * w.Kp * 2);
    w.b = take((size_t)3 * w.Jp * w.Kp * 2);
    w.bt = take((size_t)3 * w.Jp * w.Kp * 2);
    w.z = take((size_t)N * D * 4);     // Z; a forward pass: the row sums (8 bytes per 64 columns)
    w.status = take(4);
    w.total = off;
    return w;
}

}  // namespace gtc
}  // namespace psso

namespace {

psso_status fb_check(psso_fn fn, int64_t N, int64_t D, const float* X, const float* shift,
                     const float* weights, const float* rotation)
{
    using namespace psso;
    if (fn > PSSO_ROT_ACKLEY && fn <= PSSO_SCHWEFEL) {
        set_last_error("psso_fitness_forward/backward: no FP32 gradient for this function "
                       "(the hyper-ellipsoid is ELLIPSOID with weights j + 1)");
        return PSSO_ERR_UNSUPPORTED;
    }
    if (!X || !shift || N < 1 || D < 1 || D > 1024 || fn < PSSO_SPHERE || fn > PSSO_ROT_ACKLEY) {
        set_last_error("psso_fitness_forward/backward: need X, shift, N >= 1, 1 <= D <= 1024, a known function");
        return PSSO_ERR_ARG;
    }
    if ((fn == PSSO_ELLIPSOID || fn == PSSO_ROT_ELLIPSOID) && !weights) {
        set_last_error("psso_fitness_forward/backward: the ellipsoid needs weights");
        return PSSO_ERR_ARG;
    }
    if (fn >= PSSO_ROT_ELLIPSOID && !rotation) {
        set_last_error("psso_fitness_forward/backward: rotated functions need a rotation matrix");
        return PSSO_ERR_ARG;
    }
    return PSSO_OK;
}

psso::Hot fb_hot(psso_fn fn, int64_t D, const float* shift, const float* weights, const float* rotation)
{
    psso::Hot in{};
    const int nchunks = (int)((D + 3) / 4);
    int maxc = 1;
    while (maxc < (nchunks + 31) / 32) maxc <<= 1;
    in.fn = fn;
    in.D = (int)D;
    in.Dp = 4 * nchunks;
    in.nchunks = nchunks;
    in.G = 32;
    in.maxc = maxc;
    in.o32 = shift;
    in.w32 = weights;
    in.M32 = rotation;
    return in;
}

}  // namespace

extern "C" psso_status psso_fitness_forward(psso_fn fn, int64_t N, int64_t D, const float* X,
                                            const float* shift, const float* weights,
                                            const float* rotation, float* f, void* stream)
{
    using namespace psso;
    psso_status st = fb_check(fn, N, D, X, shift, weights, rotation);
    if (st != PSSO_OK) return st;
    if (!f) {
        set_last_error("psso_fitness_forward: f is NULL");
        return PSSO_ERR_ARG;
    }
    const Hot in = fb_hot(fn, D, shift, weights, rotation);
    const int wpb = 8;
    fitness_fb<false><<<(unsigned)((N + wpb - 1) / wpb), 32 * wpb, 0, static_cast<cudaStream_t>(stream)>>>(
        in, X, N, nullptr, f, nullptr);
    if (cudaGetLastError() != cudaSuccess) {
        set_last_error("psso_fitness_forward: launch failed");
        return PSSO_ERR_CUDA;
    }
    return PSSO_OK;
}

extern "C" psso_status psso_fitness_backward(psso_fn fn, int64_t N, int64_t D, const float* X,
                                             const float* shift, const float* weights,
                                             const float* rotation, const float* grad_f,
                                             float* grad_X, void* stream)
{
    using namespace psso;
    psso_status st = fb_check(fn, N, D, X, shift, weights, rotation);
    if (st != PSSO_OK) return st;
    if (!grad_f || !grad_X) {
        set_last_error("psso_fitness_backward: grad_f / grad_X is NULL");
        return PSSO_ERR_ARG;
    }
    const Hot in = fb_hot(fn, D, shift, weights, rotation);
    const int wpb = 8;
    fitness_fb<true><<<(unsigned)((N + wpb - 1) / wpb), 32 * wpb, 0, static_cast<cudaStream_t>(stream)>>>(
        in, X, N, grad_f, nullptr, grad_X);
    if (cudaGetLastError() != cudaSuccess) {
        set_last_error("psso_fitness_backward: launch failed");
        return PSSO_ERR_CUDA;
    }
    return PSSO_OK;
}

// ---------------------------------------------------------------------------
// Tensor-core entry points (rotated functions; the others run the warp kernels
// above and need no workspace).
namespace {

bool uses_tc(psso_fn fn, int64_t D) { return fn >= PSSO_ROT_ELLIPSOID && fn <= PSSO_ROT_ACKLEY && D >= 16; }

int plain_fn(psso_fn fn)
{
    return fn == PSSO_ROT_ELLIPSOID ? psso::FN_ELLIPSOID : fn == PSSO_ROT_RASTRIGIN ? psso::FN_RASTRIGIN : psso::FN_ACKLEY;
}

// Number of SMs of the current device; sets the GEMM kernels' shared-memory
// limit on the first call a thread makes on a device (the attribute is per device).
int device_sms()
{
    using namespace psso;
    static thread_local int dev_of = -1, sms = 0;
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (dev != dev_of) {
        const int smem = tc::pair_smem<tc::SplitCfg::PLANES, tc::SplitCfg::STG>();
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
            cudaFuncSetAttribute(gtc::pair_gemm<tc::StoreEpi>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) !=
                cudaSuccess ||
            cudaFuncSetAttribute(gtc::pair_gemm<gtc::SumEpi>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) !=
                cudaSuccess)
            return 0;
        sms = n;
        dev_of = dev;
    }
    return sms;
}

template <class Epi>
void launch_gemm(const CUtensorMap& ta, const CUtensorMap& tb, const psso::gtc::WsLayout& L, int* status, Epi epi,
                 int64_t N, int64_t D, int sms, cudaStream_t s)
{
    using namespace psso;
    epi.N = (int)N;
    epi.D = (int)D;
    const tc::GemmArgs ga{L.Np, L.Jp, L.Kp, status};
    launch_pdl(gtc::pair_gemm<Epi>, dim3(tc::pair_grid(L.Np, L.Jp, sms)), dim3(tc::P_THREADS),
               tc::pair_smem<tc::SplitCfg::PLANES, tc::SplitCfg::STG>(), s, ta, tb, ga, epi);
}

// Operand planes of d = x - o and M (and M^T), and the tensor maps of A and M.
psso_status tc_prepare(int64_t N, int64_t D, const float* X, const float* shift, const float* rotation, char* ws,
                       const psso::gtc::WsLayout& L, bool transposed, cudaStream_t s, CUtensorMap* ta, CUtensorMap* tb,
                       CUtensorMap* tbt)
{
    using namespace psso;
    gtc::PrepArgs a{};
    a.X = X;
    a.o = shift;
    a.M = rotation;
    a.A = reinterpret_cast<__nv_bfloat16*>(ws + L.a);
    a.B = reinterpret_cast<__nv_bfloat16*>(ws + L.b);
    a.Bt = transposed ? reinterpret_cast<__nv_bfloat16*>(ws + L.bt) : nullptr;
    a.status = reinterpret_cast<int*>(ws + L.status);
    a.N = (int)N;
    a.D = (int)D;
    a.Np = L.Np;
    a.Jp = L.Jp;
    a.Kp = L.Kp;
    a.vec_x = D % 4 == 0 && tc::aligned(X, 16);
    a.vec_m = D % 4 == 0 && tc::aligned(rotation, 16);
    const int64_t rb = (N + D + 7) / 8;
    const int64_t tiles = transposed ? (int64_t)((D + 31) / 32) * (L.Kp / 32) : 0;
    a.row_blocks = (int)rb;
    if (!tc::make_tmap_bf16(ta, a.A, L.Kp, 3 * L.Np) || !tc::make_tmap_bf16(tb, a.B, L.Kp, 3 * L.Jp, 64) ||
        (transposed && !tc::make_tmap_bf16(tbt, a.Bt, L.Kp, 3 * L.Jp, 64))) {
        set_last_error("psso_fitness_*_ws: cuTensorMapEncodeTiled failed");
        return PSSO_ERR_CUDA;
    }
    gtc::prep_planes<<<(unsigned)(rb + tiles), 256, 0, s>>>(a);
    if (cudaGetLastError() != cudaSuccess) {
        set_last_error("psso_fitness_*_ws: operand preparation failed");
        return PSSO_ERR_CUDA;
    }
    return PSSO_OK;
}

}  // namespace

extern "C" psso_status psso_fitness_workspace_size(psso_fn fn, int64_t N, int64_t D, size_t* bytes)
{
    using namespace psso;
    if (!bytes || N < 1 || D < 1 || D > 1024) {
        set_last_error("psso_fitness_workspace_size: need bytes, N >= 1, 1 <= D <= 1024");
        return PSSO_ERR_ARG;
    }
    *bytes = uses_tc(fn, D) ? gtc::ws_layout(N, D).total : 0;
    return PSSO_OK;
}

extern "C" psso_status psso_fitness_forward_ws(psso_fn fn, int64_t N, int64_t D, const float* X,
                                               const float* shift, const float* weights, const float* rotation,
                                               float* f, void* workspace, size_t ws_bytes, void* stream)
{
    using namespace psso;
    if (!uses_tc(fn, D)) return psso_fitness_forward(fn, N, D, X, shift, weights, rotation, f, stream);
    psso_status st = fb_check(fn, N, D, X, shift, weights, rotation);
    if (st != PSSO_OK) return st;
    const gtc::WsLayout L = gtc::ws_layout(N, D);
    if (!f || !workspace || ws_bytes < L.total || (reinterpret_cast<uintptr_t>(workspace) & 255)) {
        set_last_error("psso_fitness_forward_ws: need f and a 256-byte aligned workspace of "
                       "psso_fitness_workspace_size bytes");
        return PSSO_ERR_ARG;
    }
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    char* ws = static_cast<char*>(workspace);
    const int sms = device_sms();
    CUtensorMap ta, tb;
    st = tc_prepare(N, D, X, shift, rotation, ws, L, false, s, &ta, &tb, nullptr);
    if (st != PSSO_OK) return st;
    if (sms < 2) {
        set_last_error("psso_fitness_forward_ws: cannot configure the GEMM kernel");
        return PSSO_ERR_CUDA;
    }
    int* status = reinterpret_cast<int*>(ws + L.status);
    gtc::SumEpi epi{};
    epi.part = reinterpret_cast<float2*>(ws + L.z);
    epi.w = weights;
    epi.fn = plain_fn(fn);
    epi.groups = (int)((D + 63) / 64);
    launch_gemm(ta, tb, L, status, epi, N, D, sms, s);
    launch_pdl(gtc::finish_rows, dim3((unsigned)((N + 127) / 128)), dim3(128), 0, s, (const float2*)epi.part, epi.groups,
               epi.fn, (int)N, (int)D, (const int*)status, f);
    if (cudaGetLastError() != cudaSuccess) {
        set_last_error("psso_fitness_forward_ws: launch failed");
        return PSSO_ERR_CUDA;
    }
    return PSSO_OK;
}

extern "C" psso_status psso_fitness_backward_ws(psso_fn fn, int64_t N, int64_t D, const float* X,
                                                const float* shift, const float* weights,
                                                const float* rotation, const float* grad_f, float* grad_X,
                                                void* workspace, size_t ws_bytes, void* stream)
{
    using namespace psso;
    if (!uses_tc(fn, D))
        return psso_fitness_backward(fn, N, D, X, shift, weights, rotation, grad_f, grad_X, stream);
    psso_status st = fb_check(fn, N, D, X, shift, weights, rotation);
    if (st != PSSO_OK) return st;
    const gtc::WsLayout L = gtc::ws_layout(N, D);
    if (!grad_f || !grad_X || !workspace || ws_bytes < L.total || (reinterpret_cast<uintptr_t>(workspace) & 255)) {
        set_last_error("psso_fitness_backward_ws: need grad_f, grad_X and a 256-byte aligned workspace of "
                       "psso_fitness_workspace_size bytes");
        return PSSO_ERR_ARG;
    }
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    char* ws = static_cast<char*>(workspace);
    const int sms = device_sms();
    CUtensorMap ta, tb, tbt;
    st = tc_prepare(N, D, X, shift, rotation, ws, L, true, s, &ta, &tb, &tbt);
    if (st != PSSO_OK) return st;
    if (sms < 2) {
        set_last_error("psso_fitness_backward_ws: cannot configure the GEMM kernel");
        return PSSO_ERR_CUDA;
    }
    int* status = reinterpret_cast<int*>(ws + L.status);
    float* Z = reinterpret_cast<float*>(ws + L.z);
    tc::StoreEpi epi{};
    epi.out = Z;
    epi.vec = tc::store_width(Z, D);
    launch_gemm(ta, tb, L, status, epi, N, D, sms, s);
    auto* A = reinterpret_cast<__nv_bfloat16*>(ws + L.a);   // reused: the planes of G
    int maxc = 1;                                            // chunks of 4 columns per lane, padding included
    while (128 * maxc < L.Kp) maxc <<= 1;
    switch (plain_fn(fn)) {
    case FN_ELLIPSOID: gtc::launch_gz<FN_ELLIPSOID>(maxc, Z, weights, grad_f, (int)N, (int)D, L.Np, L.Kp, A, s); break;
    case FN_RASTRIGIN: gtc::launch_gz<FN_RASTRIGIN>(maxc, Z, weights, grad_f, (int)N, (int)D, L.Np, L.Kp, A, s); break;
    default: gtc::launch_gz<FN_ACKLEY>(maxc, Z, weights, grad_f, (int)N, (int)D, L.Np, L.Kp, A, s); break;
    }
    epi.out = grad_X;
    epi.vec = tc::store_width(grad_X, D);
    launch_gemm(ta, tbt, L, status, epi, N, D, sms, s);
    launch_pdl(gtc::poison, dim3((unsigned)sms), dim3(256), 0, s, grad_X, (size_t)N * D, (const int*)status);
    if (cudaGetLastError() != cudaSuccess) {
        set_last_error("psso_fitness_backward_ws: launch failed");
        return PSSO_ERR_CUDA;
    }
    return PSSO_OK;
}
