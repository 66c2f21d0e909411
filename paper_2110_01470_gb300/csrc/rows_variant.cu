// rows_variant.cu -- one precision variant of the batched row kernel
// (bat_rows.cuh), compiled once per variant with -DPSSO_VARIANT=v (0: positions
// in double, FP64 fitness; 1: positions in float, FP64 fitness; 2: positions
// in float, FP32 fitness with FP64 recheck).
#include "bat_rows.cuh"

#if !defined(PSSO_VARIANT)
#error "rows_variant.cu is compiled with -DPSSO_VARIANT=v"
#endif

#define PSSO_CAT2(a, b) a##b
#define PSSO_NAME(v) PSSO_CAT2(rows_variant_, v)

namespace psso {

cudaError_t PSSO_NAME(PSSO_VARIANT)(int fn, bool wide, int op, const BatRowsParams* p, int grid, cudaStream_t s,
                                    int* out)
{
#if PSSO_VARIANT == 0
    return rows_dispatch<double, false>(fn, wide, op, p, grid, s, out);
#elif PSSO_VARIANT == 1
    return rows_dispatch<float, false>(fn, wide, op, p, grid, s, out);
#else
    return rows_dispatch<float, true>(fn, wide, op, p, grid, s, out);
#endif
}

}  // namespace psso
