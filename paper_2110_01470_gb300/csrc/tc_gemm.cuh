// tc_gemm.cuh -- what the tensor-core GEMMs over operand planes (tc_pair.cuh)
// share: mbarrier and tensor-memory access, descriptors, and the two ways of
// writing FP32 and FP64 operands as BF16 planes -- the exact split into three parts
// (this comment) and the exact integer slices (below).
//
// Split BF16 (z = M (x - o) of psso_rotate and the differentiable fitness): d =
// fl32(x - o) and the FP32 copy of M are each written exactly as three BF16 parts,
// v = v_h + v_m + v_l (RN splits: |v_m| <= 2^-8 |v| (1.01), |v_l| <= 2^-16 |v|
// (1.01); the third remainder is exactly representable, so the split loses
// nothing).  Of the nine products of the parts, the six above 2^-24 are formed:
//     acc0[kb % 3] += d_h M_h               (main part; three accumulators, K
//                                            blocks dealt round robin, so each
//                                            chain is a third as long)
//     acc1 += d_h M_m + d_m M_h + d_h M_l + d_l M_h + d_m M_m   (corrections)
// and z = fl(fl(fl(acc0[0] + acc0[1]) + acc0[2]) + acc1).  BF16 x BF16
// products are exact in FP32.
//
// Operand layout in global memory (bf16, row-major, K contiguous):
//     A: [planes][Np][Kp]   plane p of d for particle i at (p, i, k)
//     B: [planes][Jp][Kp]   plane p of M_jk at (p, j, k)
// Np a multiple of 128, Jp of 64 (slices) or 128, Kp of 64.  Columns k >= D are zero.
// Rows beyond N and D may hold anything: an output depends on its own row of A and
// of B only, and theirs are not stored.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <cstdint>

namespace psso {
namespace tc {

constexpr int BM = 128, BN = 128, BK = 64;                 // what Np, Jp and Kp are padded to
constexpr long long WAIT_CYCLES = 4000000000LL;            // ~2 s at 2 GHz

__device__ __forceinline__ uint32_t smem_u32(const void* p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

// ---- mbarrier ---------------------------------------------------------------
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// Waits for the phase with the given parity to complete; false after
// WAIT_CYCLES (the caller then reports PSSO_ERR_TIMEOUT instead of hanging).
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity)
{
    const long long t0 = clock64();
    for (int it = 0;; ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((it & 63) == 63 && clock64() - t0 > WAIT_CYCLES) return false;
    }
}

// ---- tcgen05 ------------------------------------------------------------------
__device__ __forceinline__ void tc_fence_before()
{
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after()
{
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
// Instruction descriptor, kind::f16: FP32 accumulator (bits 4-5 = 1), A and
// B BF16 (bits 7-9, 10-12 = 1), both K-major (bits 15, 16 = 0), N >> 3 in
// bits 17-22, M >> 4 in bits 24-28.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) |
           ((uint32_t)(M >> 4) << 24);
}

// Shared-memory matrix descriptor of a K-major tile with the 128-byte swizzle:
// start address >> 4 (bits 0-13), leading offset 16 B (unused with this
// swizzle, bits 16-29), stride between 8-row groups 1024 B (bits 32-45),
// descriptor version 1 (bits 46-47), base offset 0 (the tile is 1024-byte
// aligned), swizzle mode 2 = 128 B (bits 61-63).
__device__ __forceinline__ uint64_t sdesc_sw128(uint32_t saddr)
{
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

// 32 consecutive FP32 columns of this warp's 32 lanes (one row per lane).
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32])
{
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
          "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]),
          "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]),
          "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
    // The wait names the registers so that no use of them moves above it.
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]),
                   "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]),
                   "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]), "+r"(r[16]), "+r"(r[17]),
                   "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]),
                   "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]),
                   "+r"(r[30]), "+r"(r[31])
                 :
                 : "memory");
#pragma unroll
    for (int t = 0; t < 32; ++t) v[t] = __uint_as_float(r[t]);
}

// Eight consecutive columns of each of four accumulators (`step` columns apart).
__device__ __forceinline__ void tmem_ld8x4(uint32_t taddr, uint32_t step, float (&v)[4][8])
{
    uint32_t r[4][8];
#pragma unroll
    for (int a = 0; a < 4; ++a)
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
            : "=r"(r[a][0]), "=r"(r[a][1]), "=r"(r[a][2]), "=r"(r[a][3]), "=r"(r[a][4]), "=r"(r[a][5]), "=r"(r[a][6]),
              "=r"(r[a][7])
            : "r"(taddr + (uint32_t)a * step));
    // The wait names the registers so that no use of them moves above it.
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0][0]), "+r"(r[0][1]), "+r"(r[0][2]), "+r"(r[0][3]), "+r"(r[0][4]), "+r"(r[0][5]),
                   "+r"(r[0][6]), "+r"(r[0][7]), "+r"(r[1][0]), "+r"(r[1][1]), "+r"(r[1][2]), "+r"(r[1][3]),
                   "+r"(r[1][4]), "+r"(r[1][5]), "+r"(r[1][6]), "+r"(r[1][7]), "+r"(r[2][0]), "+r"(r[2][1]),
                   "+r"(r[2][2]), "+r"(r[2][3]), "+r"(r[2][4]), "+r"(r[2][5]), "+r"(r[2][6]), "+r"(r[2][7]),
                   "+r"(r[3][0]), "+r"(r[3][1]), "+r"(r[3][2]), "+r"(r[3][3]), "+r"(r[3][4]), "+r"(r[3][5]),
                   "+r"(r[3][6]), "+r"(r[3][7])
                 :
                 : "memory");
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int q = 0; q < 8; ++q) v[a][q] = __uint_as_float(r[a][q]);
}

// Exact three-part BF16 split of a float (see the header comment).
__device__ __forceinline__ void split3(float v, __nv_bfloat16& h, __nv_bfloat16& m, __nv_bfloat16& l)
{
    h = __float2bfloat16_rn(v);
    const float r1 = __fsub_rn(v, __bfloat162float(h));
    m = __float2bfloat16_rn(r1);
    const float r2 = __fsub_rn(r1, __bfloat162float(m));
    l = __float2bfloat16_rn(r2);
}

// Bound model of the accumulation.  Adversarial probes of kind::f16 MMAs with
// FP32 accumulation on sm_103a (tests/test_gpu_mma_model.py) show an adder
// that aligns its 17 addends (accumulator + 16 exact products) to the largest
// one, truncating each to a multiple of 2^-25 of that addend's leading power
// of two, and truncates the sum to 24 bits: addends below a quarter ulp of
// the largest vanish (an accumulator of 1 absorbs any number of products of
// magnitude 0.99 * 2^-25 unchanged).  One MMA then errs by less than
// 16 * 2^-25 * max|addend| + 2^-23 |sum| <= 0.625 * 2^-20 (|accumulator| +
// sum |products|); MMA_EPS takes 2^-20, a margin of 1.6 over that (the figure that
// psso.h states for the differentiable fitness and psso_rotate).
constexpr float MMA_EPS = 0x1p-20f;

struct GemmArgs {
    int Np, Jp, Kp;   // padded extents (multiples of 128, of 64 or 128, of 64)
    int* status;      // set to 1 when a wait ran out (device memory)
};

// Host: tensor map of a [rows][Kp] bf16 matrix, boxes of 64 x box_rows,
// 128-byte swizzle.
bool make_tmap_bf16(CUtensorMap* map, const void* base, int Kp, int rows, int box_rows = BM);

// ---------------------------------------------------------------------------
// Exact integer-slice GEMM (the tensor pipeline's rotation).
//
// Each operand row is scaled by a power of two s (s_d per particle, s_M per
// output j) such that every entry satisfies |v| < s / 2, and the exact value
// (d = x - o as a float pair, M from its FP64 copy) is written as four 7-bit
// integer slices,
//     v = s (V0 2^-7 + V1 2^-14 + V2 2^-21 + V3 2^-28 + r),
// |V0..V3| <= 64, |r| <= 1.01 2^-29 (successive round-to-nearest with exact
// steps, slicers below).  The slice products of weight w = s + t <= 3 are
// accumulated in four accumulators, one per weight:
//     acc0: D0 M0                        acc1: D0 M1 + D1 M0
//     acc2: D0 M2 + D1 M1 + D2 M0        acc3: D0 M3 + D1 M2 + D2 M1 + D3 M0
// (ten MMAs per K step).  Every product is an integer of magnitude at most
// 64^2 = 4096, so per k an accumulator gains at most 4 * 4096 = 16384; for
// D <= 1023 nonzero k every partial sum stays below 2^24 in magnitude, an FP32
// accumulator represents all of them exactly, and the accumulation is exact
// whatever the MMA datapath's alignment and rounding (24 bits suffice).  The
// products of weight 4 .. 6 and the remainders r are dropped and bounded: per k,
//     s_d s_M SLICE_DROP + SLICE_REM (s_M |d_k| + s_d |M_jk|).
// The epilogue joins the accumulators in FP32 from the smallest weight up,
// t = acc0 + 2^-7 acc1 + 2^-14 acc2 + 2^-21 acc3 (three rounded operations),
// and z = 2^-14 s_d s_M t exactly.
//
// The GEMM runs on CTA pairs (tc_pair.cuh).
constexpr int SBN = 64;                                     // output columns per group of the epilogue
constexpr int SLICES = 4;
constexpr int S_MAX_K = 1024;                               // padded K extent (D <= 1023 for exactness)
constexpr int S_MAX_D = 1023;
// weight 4..6: 3 * 64^2 * 2^-42 + 2 * 64^2 * 2^-49 + 64^2 * 2^-56, and 3 r^2
constexpr float SLICE_DROP = 3.04f * 0x1p-30f;              // per k, units of s_d s_M
constexpr float SLICE_REM = 1.01f * 0x1p-29f;               // per k, of s_M |d_k| + s_d |M_jk|

// Power-of-two scale s of a row with max |v| <= vmax (1 + 2^-22): every entry
// satisfies |v| < s / 2 (s = 1 if vmax is 0).
__host__ __device__ inline float slice_scale(float vmax)
{
    if (!(vmax > 0.f)) return 1.f;
    int e = 0;
    const float m = vmax * 2.f * (1.f + 0x1p-20f);                 // rounded up
    (void)frexpf(m, &e);                                            // m < 2^e
    return ldexpf(1.f, e);
}

// The four slices of u = u_hi + u_lo (an exact float pair, |u| <= 1/2), as 7-bit
// fields of T + 64 (1 + 2^7 + 2^14 + 2^21), T the integer nearest to 2^28 u: field
// k less 64 is the balanced base-128 digit of weight 128^k, the top one within
// [-64, 64].  Two additions of 1.5 2^n round u to multiples of 2^-14 and the rest
// to multiples of 2^-28, leaving the integers in the mantissas; |2^28 u - T| <=
// 1/2 + 2^-10 (u_lo joins the rest in one rounding), so the rest after four
// slices is within 1.01 2^-29.  Rounding off one slice after the other, the rest
// kept as a float pair, took 44 instead of 19 instructions a value.
__device__ __forceinline__ uint32_t slice_fields(float u_hi, float u_lo)
{
    const float a = __fadd_rn(u_hi, 0x1.8p9f);
    const float rest = __fsub_rn(u_hi, __fsub_rn(a, 0x1.8p9f));              // exact
    const float b = __fadd_rn(__fadd_rn(rest, u_lo), 0x1.8p-5f);
    constexpr uint32_t BIAS = 64u * (1u + (1u << 7) + (1u << 14) + (1u << 21));
    // 0x44400000 = 1.5 2^9, 0x3d400000 = 1.5 2^-5
    return ((uint32_t)__float_as_int(a) << 14) + (uint32_t)__float_as_int(b) + (BIAS - (0x44400000u << 14) - 0x3d400000u);
}

// Slice p (0: the largest) of two values as two BF16 integers: 0x4300 | f is
// 128 + f, exactly, and so is the difference.
__device__ __forceinline__ uint32_t slice_pack(uint32_t u0, uint32_t u1, int p)
{
    const int sh = 7 * (SLICES - 1 - p);
    const uint32_t f = __byte_perm(u0 >> sh, u1 >> sh, 0x5410);
    const uint32_t w = (f & (p == 0 ? 0x00ff00ffu : 0x007f007fu)) | 0x43004300u;
    __nv_bfloat162 v = __hsub2(reinterpret_cast<const __nv_bfloat162&>(w), __float2bfloat162_rn(192.f));
    return reinterpret_cast<const uint32_t&>(v);
}

// The same for an FP64 value u (|u| < 1/2): the steps are exact in FP64.
__device__ __forceinline__ void slice4_f64(double u, __nv_bfloat16 (&o)[SLICES])
{
    double w = __dmul_rn(u, 128.0);
#pragma unroll
    for (int q = 0; q < SLICES; ++q) {
        const double iq = rint(w);
        o[q] = __float2bfloat16_rn((float)iq);
        w = __dmul_rn(__dsub_rn(w, iq), 128.0);
    }
}

__device__ __forceinline__ int vload(const int& v) { return *(volatile const int*)&v; }

}  // namespace tc
}  // namespace psso
