// The power-of-two scale of one column of the fp16 projection.  Plain C++ apart
// from the qualifiers, so that it can be compiled and checked without a GPU.
#pragma once

#include <string.h>

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
    // On the exponent fields: mx lies in [2^(f-127), 2^(f-126)); a denormal has
    // f = 0 and asks for 2^140, so it takes the limit like its true exponent would.
    // (The scales come before anything else of the kernel can start:
    // with frexpf and ldexpf order 57 on 21 nodes, 4 images, took 12.65 us for 12.43.)
    unsigned f, fa;
    memcpy(&f, &mx, 4);
    memcpy(&fa, &a_scale, 4);
    const int up = 140 - (int)(f >> 23), most = 126 - ((int)(fa >> 23) - 127);
    const unsigned s = (unsigned)((up < most ? up : most) + 127) << 23;
    float scale;
    memcpy(&scale, &s, 4);
    return scale;
}

}  // namespace zm
