#pragma once
#include "cuda_runtime.h"
struct __half {
    unsigned short bits;
};
float __half2float(__half);
__half __float2half_rn(float);
__half __ushort_as_half(unsigned short);
