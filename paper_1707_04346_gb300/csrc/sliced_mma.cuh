// Device helpers shared by the dense contractions on the bf16 tensor cores (the
// 2-RDM's Gram matrices and the same-spin sigma terms): operand staging by bulk
// copies.
//
// Digit scheme: an operand value x is written in fixed point relative to a
// power of two 2^e that bounds it, X = round(x 2^(46 - e)) (|X| < 2^46), cut
// into six balanced 8-bit digits d_s (X = sum_s d_s 2^(40 - 8 s), top digit in
// [-64, 64], the others in [-128, 128]) held exactly by bf16 as d_s 2^(-8 s).
// The product of two values is the sum of the 36 digit products of weight
// s + t; the 21 of weight <= 5 are accumulated, one FP32 accumulator per
// weight 0..3 (exact integers in units 2^(-8 (s + t)): at most 3 2^22 units
// for 256 products, and FP32 holds integers up to 2^24) and one for weights
// 4 and 5 (plain FP32: terms 2^-32 below the leading ones).  The products of
// weight >= 6 are left out (below 2^-46 of the leading product, zero mean).
#pragma once
#include "sigma_wide_kernel.cuh"

namespace fci {
namespace sm {

__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void *src, uint32_t bytes, uint32_t mbar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(mbar)
                 : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t mbar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mbar), "r"(bytes) : "memory");
}

}  // namespace sm
}  // namespace fci
