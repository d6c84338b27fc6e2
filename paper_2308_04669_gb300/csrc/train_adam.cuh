// Adam (Kingma & Ba 2015; beta 0.9 / 0.999, eps 1e-8, bias-corrected) on one packed master weight of
// the regression NeDF, and the place of that weight in the renderer's transposed copy.
#pragma once

#include "nedf_device.cuh"

namespace nedf {

// theta after one step with gradient g; m and v are the weight's moments, c1 and c2 the corrections
// 1 - beta^step
__device__ __forceinline__ float adam_step(float th, float g, float &m, float &v, float lr, float c1, float c2)
{
    m = 0.9f * m + 0.1f * g;
    v = 0.999f * v + 0.001f * g * g;
    return th - lr * (m / c1) / (sqrtf(v / c2) + 1e-8f);
}

// packed index (W[out][in] then b per layer) -> kernel layout index (Wt[in][out] then b)
__device__ __forceinline__ long long kernel_index(long long i, int L, int W)
{
    long long off = 0, j = i;
    int fi = kNedfIn;
    for (int l = 0; l <= L; ++l) {
        const int fo = l < L ? W : 2;
        const long long sz = (long long)fi * fo + fo;
        if (j < sz) return j < (long long)fi * fo ? off + (j % fi) * fo + j / fi : off + j;
        j -= sz;
        off += sz;
        fi = W;
    }
    return off;
}

}  // namespace nedf
