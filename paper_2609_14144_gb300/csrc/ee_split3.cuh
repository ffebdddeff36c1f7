// Two floats as three packed bf16 parts each, the first in the low halves:
// high = bf16(x), middle = bf16(x - high), low = bf16(x - high - middle).  The
// differences are exact in fp32 and the low part holds what is left, so high +
// middle + low = x.
#ifndef EE_SPLIT3_CUH_
#define EE_SPLIT3_CUH_

#include <cuda_bf16.h>
#include <stdint.h>

namespace ee {

__device__ __forceinline__ void split3(float a, float b, uint32_t (&p)[3]) {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);  // a in the low half
        p[k] = *reinterpret_cast<const uint32_t*>(&v);
        a -= __uint_as_float(p[k] << 16);
        b -= __uint_as_float(p[k] & 0xffff0000u);
    }
}

}  // namespace ee

#endif  // EE_SPLIT3_CUH_
