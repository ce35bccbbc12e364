// Sample records of the flat-sky maps (flat.cu, flattree.cu).
#pragma once

#include "isw_internal.cuh"

namespace isw {

struct __align__(16) Flat32 {
    float4 a;   // xi_s hi, eta_s hi, xi_s lo, eta_s lo
    float4 b;   // w1, w2, 0, 0
};
struct __align__(16) Flat64 {
    double xs, ys, w1, w2;
};

}  // namespace isw
