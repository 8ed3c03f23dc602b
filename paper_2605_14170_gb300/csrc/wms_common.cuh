// Device code shared by the weighted min-sum (WMS) kernels.
#pragma once

namespace mbbp {

// Binary cross-entropy of sigmoid(-post) against the error bit e.
__device__ __forceinline__ float bce_neg_sigmoid(float post, int e) {
    const float x = e ? post : -post;
    return fmaxf(x, 0.f) + log1pf(expf(-fabsf(x)));
}

}  // namespace mbbp
