// What lbm_device.cuh needs of the CUDA headers to compile as plain C++: the
// collision functions then run on the host in any arithmetic type.
#pragma once
#include <math.h>
#include <stdint.h>
#define __device__
#define __host__
#define __global__
#define __forceinline__ inline
template <typename T> inline T __ldg(const T* p) { return *p; }
