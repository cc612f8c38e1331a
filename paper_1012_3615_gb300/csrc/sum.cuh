// Accumulator of the FP32 solver's dot products.
#pragma once
#include "common.cuh"

namespace bri {

// sum of FP32 numbers with its rounding errors (Knuth's two-sum), exact to about
// 2^-47 of the terms for any few of them
struct SumF32 {
    float s = 0.f, e = 0.f;
    BRI_HD void add(float v) {
        const float t = s + v, z = t - s;
        e += (s - (t - z)) + (v - z);
        s = t;
    }
    BRI_HD double get() const { return (double)s + (double)e; }
};

}  // namespace bri
