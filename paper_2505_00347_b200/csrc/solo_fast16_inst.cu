// The sixteen-elements-per-thread kernels for one block size (SOLO_G = 4, 8, 16, 128 lanes per
// block: blocks of 64, 128, 256, 2048 elements) and one set of modes (SOLO_MODES = 0: the paper's plain step, 3 with
// Eq. 5, 4 with a baseline codebook, fixed at compile time; 1, 2: read from the arguments, see solo_fast16.cuh): fp32 or bf16 parameters, 2/3/4-bit states
// (SOLO_W8 = 0) or an 8-bit state and any other (SOLO_W8 = 1).
#include "solo_dispatch.h"
#include "solo_fast16.cuh"

#ifndef SOLO_G
#error "compile with -DSOLO_G=4|8|16|128"
#endif
#ifndef SOLO_MODES
#error "compile with -DSOLO_MODES=0|1|2|3|4"
#endif

#ifndef SOLO_W8
#error "compile with -DSOLO_W8=0|1"
#endif

#define SOLO_CAT_(a, b) a##b
#define SOLO_CAT(a, b) SOLO_CAT_(a, b)
#define SOLO_CAT4(a, b, c, d) SOLO_CAT(SOLO_CAT(a, b), SOLO_CAT(c, d))

namespace solo {

#define SOLO_K16(BM, BV)                                                                                             \
    (!param_bf16 ? solo_step_fast16_kernel<BM, BV, false, SOLO_G, SOLO_MODES, false>                                 \
     : param_sr  ? solo_step_fast16_kernel<BM, BV, true, SOLO_G, SOLO_MODES, ROUNDING_INSTANCES<SOLO_G, SOLO_MODES>> \
                 : solo_step_fast16_kernel<BM, BV, true, SOLO_G, SOLO_MODES, false>)
#define SOLO_S16(BM, BV) \
    (param_bf16 ? sizeof(Fast16Shared<BM, BV, true, SOLO_G>) : sizeof(Fast16Shared<BM, BV, false, SOLO_G>))

#if SOLO_W8
#define SOLO_WIDTHS(X) X(2, 8) X(3, 8) X(4, 8) X(8, 2) X(8, 3) X(8, 4) X(8, 8)
#define SOLO_NAME(stem) SOLO_CAT(stem, _w8)
#else
#define SOLO_WIDTHS(X) X(2, 2) X(2, 3) X(2, 4) X(3, 2) X(3, 3) X(3, 4) X(4, 2) X(4, 3) X(4, 4)
#define SOLO_NAME(stem) stem
#endif

StepKernel SOLO_NAME(SOLO_CAT4(fast16_kernel_g, SOLO_G, _m, SOLO_MODES))(int bits_m, int bits_v, bool param_bf16, bool param_sr) {
    switch (bits_m * 10 + bits_v) {
#define SOLO_CASE(BM, BV) case BM * 10 + BV: return SOLO_K16(BM, BV);
        SOLO_WIDTHS(SOLO_CASE)
#undef SOLO_CASE
        default: return nullptr;
    }
}

#if SOLO_MODES == 0
size_t SOLO_NAME(SOLO_CAT(fast16_smem_g, SOLO_G))(int bits_m, int bits_v, bool param_bf16) {
    switch (bits_m * 10 + bits_v) {
#define SOLO_CASE(BM, BV) case BM * 10 + BV: return SOLO_S16(BM, BV);
        SOLO_WIDTHS(SOLO_CASE)
#undef SOLO_CASE
        default: return 0;
    }
}
#endif

}  // namespace solo
