// The power-of-two scale of one column of the fp16 projection.  Plain C++ apart
// from the qualifiers, so that it can be compiled and checked without a GPU.
#pragma once

#include <math.h>

#ifdef __CUDACC__
#define ZM_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define ZM_HOST_DEVICE inline
#endif

namespace zm {

// Puts a column whose largest |F| is mx just below 2^14, so the fp16 halves
// neither overflow nor lose the low part to subnormals; a_scale (a power of two,
// 1 or more) is the scale of the other operand, and the product leaves the
// kernel divided by both.  Their product is kept at 2^126 or less: it, the scale
// alone and the reciprocal are then finite and normal for every mx (the smallest
// denormal, 2^-149, would ask for 2^162, and inf * 0 in the halves is a NaN).
// Slices below 2^-86 with weights scaled by 2^26 come out smaller than 2^14
// instead and lose low bits, never more than 2^-137 a node in absolute terms;
// smooth images do have such slices, where they fall off to zero.
ZM_HOST_DEVICE float column_scale(float mx, float a_scale) {
    if (!(mx > 0.f) || !(mx <= 3.402823466e38f)) return 1.f;
    int e, ea;
    frexpf(mx, &e);
    frexpf(a_scale, &ea);                    // a_scale = 2^(ea - 1)
    const int up = 14 - e, most = 126 - (ea - 1);
    return ldexpf(1.f, up < most ? up : most);
}

}  // namespace zm
