// Sums of FP32 values kept to FP64-like accuracy on the FP32 pipe.
//
// GB300 adds doubles at 1.6 per clock and SM (measured; FP32: 118), and a
// float -> double conversion goes through the same pipe, so a kernel that adds
// every stored FP32 value in FP64 is bound by that pipe: k_balances spent 108
// of these per node, 1.30 ms at 384x128x128 where its bytes take 0.21 ms.
#pragma once

namespace lbmd {

// Running sum of R values.  float: Knuth's two-sum keeps the rounding error of
// every addition (exactly representable) and adds it up beside the sum.  The sum
// of those errors is an FP32 sum itself: after n additions it is off by at most
// n^2 2^-49 of the largest partial sum (about n 2^-48 for values of either
// sign), so a pair serves the few dozen values of a node or a warp, and what
// lasts longer is kept in FP64.  Six FP32 additions per value.  An infinity or
// NaN among the values shows in `hi`, as does a partial sum beyond the float
// range.  double: one FP64 addition.
template <typename R> struct WideSum {
    R hi = R(0);
    __device__ __forceinline__ void add(R x) { hi += x; }
    __device__ __forceinline__ void merge(const WideSum& v) { hi += v.hi; }
    // adds the sum of the lane o lanes up
    __device__ __forceinline__ void merge_down(int o) { hi += __shfl_down_sync(0xffffffffu, hi, o); }
    __device__ __forceinline__ double value() const { return (double)hi; }
};
template <> struct WideSum<float> {
    float hi = 0.0f, lo = 0.0f;
    __device__ __forceinline__ void add(float x) {
        const float s = __fadd_rn(hi, x);
        const float b = __fadd_rn(s, -hi);  // the part of x that s holds
        lo = __fadd_rn(lo, __fadd_rn(__fadd_rn(hi, -__fadd_rn(s, -b)), __fadd_rn(x, -b)));
        hi = s;
    }
    __device__ __forceinline__ void merge(const WideSum& v) {
        add(v.hi);
        lo = __fadd_rn(lo, v.lo);
    }
    __device__ __forceinline__ void merge_down(int o) {
        WideSum v;
        v.hi = __shfl_down_sync(0xffffffffu, hi, o);
        v.lo = __shfl_down_sync(0xffffffffu, lo, o);
        merge(v);
    }
    __device__ __forceinline__ double value() const {
        return isfinite(hi) ? (double)hi + (double)lo : (double)hi;
    }
};

}  // namespace lbmd
