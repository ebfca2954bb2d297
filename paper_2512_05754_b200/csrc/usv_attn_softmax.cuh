// Softmax weights of a piece of a row, as the tcgen05 attention kernels take them.
#pragma once
#include "usv_tcgen05.cuh"

namespace usv {
namespace t5 {

// exp2 of 32 scaled logits -> 16 packed bf16 pairs; adds to the two lanes of `acc` nothing, the weights as rounded to
// bf16 (what the P.V product multiplies by, so that numerator and denominator of a row carry the same
// rounding), or the weights before the rounding (for the log-sum-exp).  Two logits at a time on the packed-fp32 pipe.
enum { SUM_NONE = 0, SUM_ROUNDED = 1, SUM_EXACT = 2 };
template <bool MASKED, int SUM, int POLY>
__device__ __forceinline__ void weights32(const uint32_t* sr, uint32_t* pk, uint64_t c2, uint64_t nref2, int col0,
                                          int nvalid, uint64_t& acc) {
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        const uint64_t x2 = fma_f32x2(pack_f32x2(__uint_as_float(sr[2 * j]), __uint_as_float(sr[2 * j + 1])), c2, nref2);
        float p0, p1;
        if (POLY && j % (POLY ? POLY : 1) == POLY - 1) {
            exp2_fma(x2, p0, p1);
        } else {
            float x0, x1;
            unpack_f32x2(x2, x0, x1);
            p0 = ex2(x0);
            p1 = ex2(x1);
        }
        if (MASKED) {
            if (col0 + 2 * j >= nvalid) p0 = 0.f;
            if (col0 + 2 * j + 1 >= nvalid) p1 = 0.f;
        }
        pk[j] = pack_bf16x2(p0, p1);
        if (SUM == SUM_ROUNDED) acc = add_f32x2(acc, pack_f32x2(__uint_as_float(pk[j] << 16), __uint_as_float(pk[j] & 0xffff0000u)));
        if (SUM == SUM_EXACT) acc = add_f32x2(acc, pack_f32x2(p0, p1));
    }
}

}  // namespace t5
}  // namespace usv
