// Double-float arithmetic on the FP32 pipe.
//
// A value is the unevaluated sum hi + lo of two floats (|lo| <= ulp(hi) / 2),
// about 48 significant bits, computed on the FP32 pipe: on this GPU the FP64
// pipe runs at 1/64 of the FP32 rate, so for the ill-conditioned parts of the
// dual step and for the pixel step two-float arithmetic is several times
// cheaper than FP64.  The
// error-free transformations are Knuth's TwoSum and Dekker's exact product in
// its FMA form (Dekker 1971); additions are the accurate ("IEEE-style")
// double-word sum of Hida, Li and Bailey (2001), which keeps its accuracy under
// cancellation; the reciprocal is one Newton step from the FP32 reciprocal.
// Every operation is spelled with _rn intrinsics so that the compiler cannot
// contract or reassociate them.
#pragma once
#include <cuda_runtime.h>

namespace osscir {

struct dfl {
    float hi, lo;
};

__device__ __forceinline__ dfl df_fast2sum(float a, float b) {   // |a| >= |b| (or a = 0)
    const float s = __fadd_rn(a, b);
    return {s, __fsub_rn(b, __fsub_rn(s, a))};
}

__device__ __forceinline__ dfl df_2sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}

__device__ __forceinline__ dfl df_2prod(float a, float b) {
    const float p = __fmul_rn(a, b);
    return {p, __fmaf_rn(a, b, -p)};
}

__device__ __forceinline__ dfl df_add(dfl x, dfl y) {
    const dfl s = df_2sum(x.hi, y.hi), t = df_2sum(x.lo, y.lo);
    const dfl u = df_fast2sum(s.hi, __fadd_rn(s.lo, t.hi));
    return df_fast2sum(u.hi, __fadd_rn(u.lo, t.lo));
}

__device__ __forceinline__ dfl df_sub(dfl x, dfl y) { return df_add(x, dfl{-y.hi, -y.lo}); }

__device__ __forceinline__ dfl df_mul(dfl x, dfl y) {
    const dfl p = df_2prod(x.hi, y.hi);
    return df_fast2sum(p.hi, __fmaf_rn(x.hi, y.lo, __fmaf_rn(x.lo, y.hi, p.lo)));
}

__device__ __forceinline__ dfl df_mulf(dfl x, float y) {
    const dfl p = df_2prod(x.hi, y);
    return df_fast2sum(p.hi, __fmaf_rn(x.lo, y, p.lo));
}

__device__ __forceinline__ float df_f(dfl x) { return __fadd_rn(x.hi, x.lo); }

// 1 / x: r + r (1 - x r) with r the FP32 reciprocal of x.hi.
__device__ __forceinline__ dfl df_rcp(dfl x) {
    const float r = __frcp_rn(x.hi);
    const dfl e = df_sub(dfl{1.0f, 0.0f}, df_mulf(x, r));
    return df_add(dfl{r, 0.0f}, df_mulf(e, r));
}

// The same in a sixth of the instructions: the residual is one exact FMA plus x.lo's
// share (|residual| <= 2^-23, so FP32 holds it to 2^-47).  Not for the dual step, whose
// most attenuated rays carry a last bit of it into y' (1e-3 of its size at 512 x 512).
__device__ __forceinline__ dfl df_rcp_fma(dfl x) {
    const float r = __frcp_rn(x.hi);
    const float e = __fmaf_rn(-x.lo, r, __fmaf_rn(-x.hi, r, 1.0f));
    return df_fast2sum(r, __fmul_rn(r, e));
}

// sqrt of a positive double-float: s = sqrt(hi) corrected by one Newton step,
// s + (x - s^2) / (2 s) (Karp and Markstein 1997), the correction in FP32.
__device__ __forceinline__ dfl df_sqrt(dfl x) {
    const float s = __fsqrt_rn(x.hi);
    const float e = df_f(df_sub(x, df_2prod(s, s)));
    return df_fast2sum(s, __fmul_rn(e, __fdiv_rn(0.5f, s)));
}

__device__ __forceinline__ dfl df_neg(dfl x) { return dfl{-x.hi, -x.lo}; }

}  // namespace osscir
