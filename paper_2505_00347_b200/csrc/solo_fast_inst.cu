// Instantiations of the streamlined step kernel for one first-moment width (SOLO_BM = 2, 3, 4, 8): for all tiles
// (SOLO_TAILS = 0) or for those the sixteen-per-thread kernel leaves (SOLO_TAILS = 1: a few tiles, modes read at run time).
#include "solo_dispatch.h"
#include "solo_fast.cuh"

#ifndef SOLO_BM
#error "compile with -DSOLO_BM=2|3|4|8"
#endif
#ifndef SOLO_TAILS
#error "compile with -DSOLO_TAILS=0|1"
#endif

#define SOLO_CAT_(a, b) a##b
#define SOLO_CAT(a, b) SOLO_CAT_(a, b)

namespace solo {

#define SOLO_ROW(BV, PBF, PLAIN)                                                                                          \
    {solo_step_fast_kernel<SOLO_BM, BV, 8, PBF, PLAIN, SOLO_TAILS>, solo_step_fast_kernel<SOLO_BM, BV, 16, PBF, PLAIN, SOLO_TAILS>, \
     solo_step_fast_kernel<SOLO_BM, BV, 32, PBF, PLAIN, SOLO_TAILS>, solo_step_fast_kernel<SOLO_BM, BV, 256, PBF, PLAIN, SOLO_TAILS>}
#define SOLO_PLANE(PBF, PLAIN) \
    {SOLO_ROW(2, PBF, PLAIN), SOLO_ROW(3, PBF, PLAIN), SOLO_ROW(4, PBF, PLAIN), SOLO_ROW(8, PBF, PLAIN)}

static int block_index(int block) {
    return block == 64 ? 0 : block == 128 ? 1 : block == 256 ? 2 : block == 2048 ? 3 : -1;
}

#if SOLO_TAILS
StepKernel SOLO_CAT(fast_tails_kernel_bm, SOLO_BM)(int bv_index, int block, bool param_bf16) {
    static const StepKernel table[2][4][4] = {SOLO_PLANE(false, false), SOLO_PLANE(true, false)};
    const int g = block_index(block);
    if (bv_index < 0 || bv_index > 3 || g < 0) return nullptr;
    return table[param_bf16 ? 1 : 0][bv_index][g];
}
#else
StepKernel SOLO_CAT(fast_kernel_bm, SOLO_BM)(int bv_index, int block, bool param_bf16, bool plain) {
    static const StepKernel table[2][2][4][4] = {
        {SOLO_PLANE(false, false), SOLO_PLANE(true, false)},
        {SOLO_PLANE(false, true), SOLO_PLANE(true, true)},
    };
    const int g = block_index(block);
    if (bv_index < 0 || bv_index > 3 || g < 0) return nullptr;
    return table[plain ? 1 : 0][param_bf16 ? 1 : 0][bv_index][g];
}
#endif

#if SOLO_BM == 2 && !SOLO_TAILS
// Exhaustive check of the error model used above: for every binary32 x with bit pattern
// in [lo, hi] (positive, finite) the largest value of
//   |lg2.approx(x) - log2_sp(x)| - (LG2_REL / 2) |log2_sp(x)|
// is written (as a maximum over the launch) to *out_max_excess, which starts at -1.
__global__ void fast_log_check_kernel(uint32_t lo, uint32_t hi, float* out_max_excess) {
    float worst = -1.0f;
    for (uint64_t b = (uint64_t)lo + blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; b <= hi;
         b += (uint64_t)gridDim.x * blockDim.x) {
        const float x = __uint_as_float((uint32_t)b);
        const float exact = log2_sp(x);
        const float ex = fabsf(lg2_approx(x) - exact) - (0.5f * LG2_REL) * fabsf(exact);
        worst = fmaxf(worst, ex);
    }
    worst = fmaxf(worst, __shfl_xor_sync(0xffffffffu, worst, 16));
    worst = fmaxf(worst, __shfl_xor_sync(0xffffffffu, worst, 8));
    worst = fmaxf(worst, __shfl_xor_sync(0xffffffffu, worst, 4));
    worst = fmaxf(worst, __shfl_xor_sync(0xffffffffu, worst, 2));
    worst = fmaxf(worst, __shfl_xor_sync(0xffffffffu, worst, 1));
    if ((threadIdx.x & 31) == 0 && worst > 0.0f)
        atomicMax(reinterpret_cast<int*>(out_max_excess), __float_as_int(worst));
}

// Comparison of neg_sqrt2 and neg_div2 with the IEEE operations: for every binary32 with pattern in [lo, hi] its square
// root, and as a denominator (brought to exponents from -40 to 43) its quotients with eight numerators: one close to the
// denominator, the others below 2^20 down to the smallest subnormal number, where the quotient is a normal number.
__global__ void update_math_check_kernel(uint32_t lo, uint32_t hi, unsigned long long* mismatches) {
    unsigned long long bad = 0;
    for (uint64_t b = (uint64_t)lo + 2 * (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x); b <= hi;
         b += 2 * (uint64_t)gridDim.x * blockDim.x) {
        const float x[2] = {__uint_as_float((uint32_t)b), __uint_as_float((uint32_t)min(b + 1, (uint64_t)hi))};
        if (x[0] < 0x1p27f && x[1] < 0x1p27f) {
            const F2 s = neg_sqrt2(mul2(F2::pack(x[0], x[1]), F2::dup(-0x1p100f)));
            bad += (-s.lo() * 0x1p-50f != __fsqrt_rn(x[0])) + (-s.hi() * 0x1p-50f != __fsqrt_rn(x[1]));
        }
        uint32_t w[4], w2[4];
        philox4x32_10((uint32_t)b, 1u, 2u, 3u, 4u, 5u, w);
        philox4x32_10((uint32_t)b, 7u, 2u, 3u, 4u, 5u, w2);
        for (int i = 0; i < 4; ++i) {
            float d[2], m[2];
            for (int k = 0; k < 2; ++k) {
                const uint32_t r = k ? w2[i] : w[i];
                d[k] = __uint_as_float((__float_as_uint(x[k]) & 0x007FFFFFu) | ((127u - 40u + r % 84u) << 23));
                // exponents from 2^-126 on, a fifth of the numerators subnormal with 1 to 23 bits
                const uint32_t e = (r >> 7) % 183u;
                m[k] = __uint_as_float((r & 0x80000000u) | (e < 146u ? (r & 0x007FFFFFu) | ((e + 1u) << 23)
                                                                     : (0x00400000u | (r & 0x003FFFFFu)) >> ((r >> 15) % 23u)));
                if (i == 0) m[k] = __uint_as_float(__float_as_uint(min(d[k], 0x1p19f)) + (r & 3u) - 1u);   // quotients around 1
            }
            const F2 q = neg_div2(mul2(F2::pack(m[0], m[1]), F2::dup(0x1p64f)), F2::pack(d[0], d[1]));
            auto differs = [](float a, float b) { return fabsf(b) > 0x1p-126f && a != b; };
            bad += differs(-q.lo() * 0x1p-64f, __fdiv_rn(m[0], d[0])) + differs(-q.hi() * 0x1p-64f, __fdiv_rn(m[1], d[1]));
        }
    }
    if (bad) atomicAdd(mismatches, bad);
}

cudaError_t launch_update_math_check(uint32_t lo, uint32_t hi, unsigned long long* mismatches, cudaStream_t stream) {
    update_math_check_kernel<<<148 * 8, 256, 0, stream>>>(lo, hi, mismatches);
    return cudaGetLastError();
}

cudaError_t launch_fast_log_check(uint32_t lo, uint32_t hi, float* out_max_excess, cudaStream_t stream) {
    fast_log_check_kernel<<<148 * 8, 256, 0, stream>>>(lo, hi, out_max_excess);
    return cudaGetLastError();
}
float fast_log_abs_bound() { return LG2_ABS; }
size_t fast_kernel_smem(int bits_m, int bits_v) {
    const bool m8 = bits_m == 8, v8 = bits_v == 8;
    return m8 ? (v8 ? sizeof(FastSharedT<2, 2>) : sizeof(FastSharedT<2, 1>))
              : (v8 ? sizeof(FastSharedT<1, 2>) : sizeof(FastSharedT<1, 1>));
}
#endif

}  // namespace solo
