// Wide sums of FP32 values in three FP32 words (far.cu's split-coordinate kernels). No CUDA needed:
// the host tests compile it on its own.
#pragma once

namespace pb {

#ifdef __CUDACC__
#define PB_WIDE_FN __device__ __forceinline__
#else
#define PB_WIDE_FN inline
#endif

// hi + mid + lo += b: b is added to hi and the exact rounding error (Knuth's two-sum) to mid, whose
// own exact error goes into lo; only lo's additions round. lo is about 2^-48 of the sum, so the sum is
// good to 2^-72 a term, where FP64's rounds at 2^-53. Ops: add and sub of the word type F.
template <typename Ops, typename F>
PB_WIDE_FN void wide_add(F& hi, F& mid, F& lo, F b) {
    F s = Ops::add(hi, b), bb = Ops::sub(s, hi);
    const F e = Ops::add(Ops::sub(hi, Ops::sub(s, bb)), Ops::sub(b, bb));
    hi = s;
    s = Ops::add(mid, e);
    bb = Ops::sub(s, mid);
    lo = Ops::add(lo, Ops::add(Ops::sub(mid, Ops::sub(s, bb)), Ops::sub(e, bb)));
    mid = s;
}

// the sum in FP64 (past FP32's range hi alone: the other words are then no numbers)
PB_WIDE_FN double wide_value(float hi, float mid, float lo) {
    return hi - hi == 0.0f ? (double)hi + ((double)mid + (double)lo) : (double)hi;
}

}  // namespace pb
