#pragma once
#include "cuda_runtime.h"
struct __nv_bfloat16 {
    unsigned short bits;
};
float __bfloat162float(__nv_bfloat16);
__nv_bfloat16 __float2bfloat16_rn(float);
__nv_bfloat16 __ushort_as_bfloat16(unsigned short);
