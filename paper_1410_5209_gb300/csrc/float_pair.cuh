// Sums and products carried as unevaluated pairs of floats (h + l, about 48 significant
// bits): the error-free transformations of Knuth (two-sum) and of the fused multiply-add
// (two-product), as collected in Ogita, Rump and Oishi, "Accurate sum and dot product"
// (SIAM J. Sci. Comput. 26, 2005).  FP64 arithmetic and float <-> double conversions run at
// 1/64 of the FP32 rate on this GPU, so where a float result only needs sums that are much
// more accurate than FP32, a pair (6 FP32 operations an addition, 2 a product) is an order
// of magnitude cheaper than a double.  The rounded intrinsics keep the compiler from
// contracting or reassociating the error terms.
#pragma once

namespace tfs {

struct FloatPair {
    float h, l;
};

// a + b exactly as s + err
__device__ __forceinline__ float two_sum(float a, float b, float &err) {
    const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
    err = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return s;
}

// a * b exactly as p + err (barring underflow of err)
__device__ __forceinline__ float two_prod(float a, float b, float &err) {
    const float p = __fmul_rn(a, b);
    err = __fmaf_rn(a, b, -p);
    return p;
}

// acc += t + e, e a correction much smaller than t; acc.h takes the rounded sum, acc.l the
// errors (not renormalised: a chain of additions needs no more)
__device__ __forceinline__ void pair_add(FloatPair &acc, float t, float e) {
    float err;
    acc.h = two_sum(acc.h, t, err);
    acc.l = __fadd_rn(acc.l, __fadd_rn(err, e));
}

// p * x, p a pair
__device__ __forceinline__ FloatPair pair_mul(const FloatPair &p, float x) {
    FloatPair r;
    r.h = two_prod(p.h, x, r.l);
    r.l = __fmaf_rn(p.l, x, r.l);
    return r;
}

// Sum of a over groups of `width` neighbouring lanes (a power of two), in every lane of the
// group; both partners of an exchange form the same sum.  All lanes of `mask` call it.
__device__ __forceinline__ FloatPair pair_group_sum(FloatPair a, int width, unsigned mask) {
    for (int o = width >> 1; o > 0; o >>= 1) {
        const float h = __shfl_xor_sync(mask, a.h, o), l = __shfl_xor_sync(mask, a.l, o);
        float err;
        a.h = two_sum(a.h, h, err);
        a.l = __fadd_rn(__fadd_rn(a.l, l), err);
    }
    return a;
}

}  // namespace tfs
