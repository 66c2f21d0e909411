// rotate.cu -- the tensor maps of the operand planes, and psso_rotate: z = M (x - o)
// for N rows on the tensor cores (split BF16 planes).
#include <cmath>
#include <cstdio>
#include <cudaTypedefs.h>
#include <mutex>

#include "psso.h"
#include "psso_internal.h"
#include "sso_common.cuh"
#include "rot_pipeline.h"
#include "tc_pair.cuh"

namespace psso {
namespace tc {

bool make_tmap_bf16(CUtensorMap* map, const void* base, int Kp, int rows, int box_rows)
{
    static PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    });
    if (!encode) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)Kp, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)Kp * 2};
    const cuuint32_t box[2] = {(cuuint32_t)BK, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// B planes of the FP32 rotation: one block per row j of the padded [Jp][Kp]
// planes (rows >= D and columns >= D are zero).
__global__ void split_matrix(const float* __restrict__ M32, int D, int Jp, int Kp, __nv_bfloat16* B)
{
    const int j = blockIdx.x;
    for (int k = threadIdx.x; k < Kp; k += blockDim.x) {
        const float v = (j < D && k < D) ? M32[(size_t)j * D + k] : 0.f;
        __nv_bfloat16 h, m, l;
        split3(v, h, m, l);
        const size_t o = (size_t)j * Kp + k, plane = (size_t)Jp * Kp;
        B[o] = h;
        B[plane + o] = m;
        B[2 * plane + o] = l;
    }
}

// A planes of z = M (x - o) for plain rows (psso_rotate): warp per row.
__global__ void split_rows(const float* __restrict__ X, const float* __restrict__ o, int N, int D, int Np,
                           int Kp, __nv_bfloat16* A)
{
    const int i = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (i >= Np) return;
    const int lane = threadIdx.x & 31;
    const size_t plane = (size_t)Np * Kp;
    for (int k = lane; k < Kp; k += 32) {
        const float d = (i < N && k < D) ? __fsub_rn(X[(size_t)i * D + k], o[k]) : 0.f;
        __nv_bfloat16 h, m, l;
        split3(d, h, m, l);
        const size_t p = (size_t)i * Kp + k;
        A[p] = h;
        A[plane + p] = m;
        A[2 * plane + p] = l;
    }
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(P_THREADS, 1)
    rotate_gemm(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const GemmArgs a,
                const __grid_constant__ StoreEpi epi0)
{
    StoreEpi epi = epi0;
    epi.chains = a.Kp / BK < 3 ? a.Kp / BK : 3;
    gemm_pair<SplitCfg>(&tmA, &tmB, a, epi);
}

}  // namespace tc
}  // namespace psso

extern "C" psso_status psso_rotate(int64_t N, int64_t D, const float* X, const float* shift,
                                   const float* rotation, float* Z, void* stream)
{
    using namespace psso;
    using namespace psso::tc;
    if (!X || !shift || !rotation || !Z || N < 1 || D < 1 || D > 8192 || N > (1 << 24)) {
        set_last_error("psso_rotate: need X, shift, rotation, Z, 1 <= N <= 2^24, 1 <= D <= 8192");
        return PSSO_ERR_ARG;
    }
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int Np = (int)((N + BM - 1) / BM * BM), Jp = (int)((D + BN - 1) / BN * BN),
              Kp = (int)((D + BK - 1) / BK * BK);
    __nv_bfloat16 *A = nullptr, *B = nullptr;
    int* status = nullptr;
    auto cleanup = [&] {
        cudaFree(A);
        cudaFree(B);
        cudaFree(status);
    };
    if (cudaMalloc(&A, (size_t)3 * Np * Kp * 2) != cudaSuccess || cudaMalloc(&B, (size_t)3 * Jp * Kp * 2) != cudaSuccess ||
        cudaMalloc(&status, 4) != cudaSuccess) {
        cleanup();
        set_last_error("psso_rotate: device allocation failed");
        return PSSO_ERR_OOM;
    }
    CUtensorMap ta, tb;
    if (!make_tmap_bf16(&ta, A, Kp, 3 * Np) || !make_tmap_bf16(&tb, B, Kp, 3 * Jp, 64)) {
        cleanup();
        set_last_error("psso_rotate: cuTensorMapEncodeTiled failed");
        return PSSO_ERR_CUDA;
    }
    cudaMemsetAsync(status, 0, 4, s);
    split_matrix<<<Jp, 256, 0, s>>>(rotation, (int)D, Jp, Kp, B);
    split_rows<<<(Np + 7) / 8, 256, 0, s>>>(X, shift, (int)N, (int)D, Np, Kp, A);
    constexpr int smem = pair_smem<SplitCfg::PLANES, SplitCfg::STG>();
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaFuncSetAttribute(rotate_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    GemmArgs ga{Np, Jp, Kp, status};
    StoreEpi epi{};
    epi.N = (int)N;
    epi.D = (int)D;
    epi.out = Z;
    epi.vec = store_width(Z, D);
    if (sms >= 2) rotate_gemm<<<pair_grid(Np, Jp, sms), P_THREADS, smem, s>>>(ta, tb, ga, epi);
    cudaError_t e = cudaGetLastError();
    int st = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&st, status, 4, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cleanup();
    if (e != cudaSuccess) {
        char msg[256];
        snprintf(msg, sizeof msg, "psso_rotate: %s", cudaGetErrorString(e));
        set_last_error(msg);
        return PSSO_ERR_CUDA;
    }
    if (st) {
        set_last_error("psso_rotate: a tensor-core pipeline wait ran out");
        return PSSO_ERR_TIMEOUT;
    }
    return PSSO_OK;
}
