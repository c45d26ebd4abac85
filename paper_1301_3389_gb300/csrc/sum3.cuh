// A sum held as three float32 values, for sums that must not be coarser than float64 ones in
// kernels that a float64 add per term would bound (64 cycles per warp instruction on this GPU,
// against 4 for a float32 add).
#pragma once

#include <cuda_runtime.h>

namespace dna {

// s + e + f: s is the float32 sum, e the sum of its rounding errors, f the sum of e's.  The
// errors come from the two-sum of Knuth and are exact, so only f rounds: after n terms the
// error is at most n^3 2^-72 of the largest partial sum (typically n^1.5 2^-72), which lies
// below the n 2^-53 of float64 adds up to n = 700.  The range is float32's: a caller whose
// sums can leave it goes on (large), or starts again, in float64.
struct Sum3 {
    float s = 0.f, e = 0.f, f = 0.f;

    // x += t, returning the rounding error
    static __device__ __forceinline__ float two_sum(float& x, float t) {
        const float n = __fadd_rn(x, t), b = __fsub_rn(n, x);
        const float err = __fadd_rn(__fsub_rn(x, __fsub_rn(n, b)), __fsub_rn(t, b));
        x = n;
        return err;
    }
    // a term that is itself an error term, far below s
    __device__ __forceinline__ void add_low(float t) { f = __fadd_rn(f, two_sum(e, t)); }
    __device__ __forceinline__ void add(float t) { add_low(two_sum(s, t)); }
    __device__ __forceinline__ void add(float ts, float te, float tf) {
        add(ts);
        add_low(te);
        f = __fadd_rn(f, tf);
    }
    // s alone once a term was infinite or NaN (the errors are then inf - inf): an infinite
    // sum stays infinite
    __device__ __forceinline__ double value() const {
        return isfinite(s) ? (double)s + ((double)e + (double)f) : (double)s;
    }
    // near the end of float32's range (or infinite)
    static __device__ __forceinline__ bool large(float t) { return fabsf(t) > 1e36f; }
};

// The same interface on float64 alone.
struct Sum64 {
    double s = 0.0;
    __device__ __forceinline__ void add(float t) { s += (double)t; }
    __device__ __forceinline__ double value() const { return s; }
};

}  // namespace dna
