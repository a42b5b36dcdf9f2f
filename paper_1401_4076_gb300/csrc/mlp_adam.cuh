// The Adam step of one parameter of the seeding network, shared by the
// training paths.
#pragma once

#include <cuda_bf16.h>

#include "mucal_internal.h"

namespace mucal {

constexpr float kAdamBeta1 = 0.9f, kAdamBeta2 = 0.999f, kAdamEps = 1e-8f;

// Adam (Kingma and Ba) on the fp32 master parameter, then its bf16 copies.
__device__ __forceinline__ void adam_step(const AdamState &st, int i, float gr, float lr, float c1, float c2)
{
    const float a = kAdamBeta1 * st.m1[i] + (1.f - kAdamBeta1) * gr;
    const float b = kAdamBeta2 * st.m2[i] + (1.f - kAdamBeta2) * gr * gr;
    st.m1[i] = a;
    st.m2[i] = b;
    const float v = st.w[i] - lr * (a / c1) / (sqrtf(b / c2) + kAdamEps);
    st.w[i] = v;
    const __nv_bfloat16 q = __float2bfloat16_rn(v);
    st.wq[i] = q;
    const int k = i - kMlpOffW2;
    if (k >= 0 && k < kMlpH * kMlpH) st.w2t[(k % kMlpH) * kMlpH + k / kMlpH] = q;
}

}  // namespace mucal
