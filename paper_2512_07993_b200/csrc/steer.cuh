// Device body of the steering add, shared by skipkv_steer and the decode-attention epilogue.
#pragma once
#include "common.cuh"

namespace skipkv {

// Element group i of 8 bf16: hidden[b][8k..8k+7] = bf16_rne(fmaf(alpha[b], v, hidden)) if flag[b], in two halves so that a
// caller can put work between the loads (independent of one another: row b is read whatever its flag) and the store.
struct SteerVec { uint4 h, s; float alpha; bool on; };

__device__ __forceinline__ SteerVec steer_load(int i, int vec_per_row, const __nv_bfloat16* hidden, const __nv_bfloat16* v,
                                               const float* alpha, const uint8_t* flag) {
    const int b = i / vec_per_row, k = i % vec_per_row;
    SteerVec x;
    x.on = flag[b] != 0;
    x.alpha = alpha[b];
    x.h = reinterpret_cast<const uint4*>(hidden)[size_t(b) * vec_per_row + k];
    x.s = reinterpret_cast<const uint4*>(v)[k];
    return x;
}
__device__ __forceinline__ void steer_store(int i, int vec_per_row, __nv_bfloat16* hidden, const SteerVec& x) {
    if (!x.on) return;
    uint32_t hw[4] = {x.h.x, x.h.y, x.h.z, x.h.w};
    const uint32_t sw[4] = {x.s.x, x.s.y, x.s.z, x.s.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float lo = __fmaf_rn(x.alpha, bf16lo(sw[j]), bf16lo(hw[j]));
        const float hi = __fmaf_rn(x.alpha, bf16hi(sw[j]), bf16hi(hw[j]));
        const __nv_bfloat162 r = __floats2bfloat162_rn(lo, hi);
        hw[j] = *reinterpret_cast<const uint32_t*>(&r);
    }
    reinterpret_cast<uint4*>(hidden)[i] = make_uint4(hw[0], hw[1], hw[2], hw[3]);
}

}  // namespace skipkv
