// A sum of FP32 terms beside the rounding errors made in it (Knuth's two-sum): some 48 bits,
// without the narrow FP64 pipe.
#pragma once

namespace cva {
namespace {

struct SumPair {
    float hi, lo;
    __device__ void add(float p, float e = 0.f)   // p + e, e the error of p
    {
        const float s = hi + p, b = s - hi;
        lo += ((hi - (s - b)) + (p - b)) + e;
        hi = s;
    }
};

}  // namespace
}  // namespace cva
