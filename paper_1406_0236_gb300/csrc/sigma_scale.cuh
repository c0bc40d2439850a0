// Scales of the densities of a call, one power of two per right-hand side, for the kernels that
// hold them in formats of limited range: key[r] is the largest high word of |Re|, |Im| of the
// (weighted) densities of column r over its finite entries (sigma_keys, nbody_dfl.cu), 0 for
// none, so that every such value is below 2^sigma_exponent(key[r]).
#pragma once

#include <cuda_runtime.h>

namespace hzb {

__device__ __forceinline__ int sigma_exponent(int key)
{
    return key ? min(960, max(-960, (key >> 20) - 1022)) : 0;
}
__device__ __forceinline__ double sigma_pow2(int e) { return __hiloint2double((1023 + e) << 20, 0); }

}  // namespace hzb
