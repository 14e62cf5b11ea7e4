// qint8 arithmetic shared by the kernel translation units: quantisation,
// requantisation with one rounding per written operation, vector types.
#pragma once

#include <cmath>
#include <type_traits>

#include "kern_common.cuh"

namespace sn {
namespace k {

// N consecutive elements moved as one aligned access
template <typename T, int N> struct alignas(sizeof(T) * N) Vec { T v[N]; };

constexpr int QMAX = 127;

__device__ __forceinline__ int8_t q8_code(float y, float inv) {
    const int q = __float2int_rn(__fmul_rn(y, inv));
    return (int8_t)max(-QMAX, min(QMAX, q));
}

// the fused activations with one rounding per operation (DIV: the same values by
// the division, see act_apply_div)
template <bool DIV = false>
__device__ __forceinline__ float q8_act(float v, int act) {
    if (act == SN_ACT_RELU) return fmaxf(v, 0.0f);
    if (act == SN_ACT_NONE) return v;
    if (act == SN_ACT_RELU6) return fminf(fmaxf(v, 0.0f), 6.0f);
    const float r = fminf(fmaxf(__fadd_rn(v, 3.0f), 0.0f), 6.0f);
    const float t = DIV ? __fdiv_rn(r, 6.0f) : sixth(r);  // hard sigmoid: r / 6 to the bit
    return act == SN_ACT_HSWISH ? __fmul_rn(v, t) : t;
}

// act(float(acc) * (s_x * s_w) + bias [+ residual value]) in fp32
template <bool DIV = false>
__device__ __forceinline__ float q8_value(int acc, float s_x, float s_w, float bias, float resid, int act) {
    float y = __fadd_rn(__fmul_rn(__int2float_rn(acc), __fmul_rn(s_x, s_w)), bias);
    y = __fadd_rn(y, resid);
    return q8_act<DIV>(y, act);
}

// the output element: a code of the output blob's scale, or, when the routine
// writes a float schema (dequantisation fused into the epilogue), the fp32
// value rounded to that type
template <typename TO>
__device__ __forceinline__ TO q8_out(float y, float inv) {
    if constexpr (std::is_same<TO, int8_t>::value) return q8_code(y, inv);
    else return cvt<TO>(y);
}

// code of a weight of scale s
__device__ __forceinline__ int q8_weight_code(float v, float s) {
    return max(-QMAX, min(QMAX, __float2int_rn(__fdiv_rn(v, s))));
}

// the scales that a launch reads and writes codes with
struct Q8Scales {
    float s_x, s_r, inv_out;
};
inline int out_dtype(const LaunchArgs &a) { return a.out_schema.dtype < 0 ? a.schema.dtype : a.out_schema.dtype; }
inline Q8Scales scales_of(const LaunchArgs &a) {
    return Q8Scales{a.qs_in[0], a.qs_in[1], a.qs_out > 0.0f ? 1.0f / a.qs_out : 0.0f};
}
// the input scales, and the output scale when the output is qint8
inline bool scales_ok(const LaunchArgs &a, int n_in) {
    for (int i = 0; i < n_in; ++i)
        if (!(a.qs_in[i] > 0.0f) || !std::isfinite(a.qs_in[i])) return false;
    return out_dtype(a) != SN_QI8 || (a.qs_out > 0.0f && std::isfinite(a.qs_out));
}

// per-output-channel scales max |w[k, .]| / 127 (1 for an all-zero channel) of fp32 weights [K][per_k]
cudaError_t q8_weight_scales(const float *w, float *scale, int64_t K, int64_t per_k, cudaStream_t st);

}  // namespace k
}  // namespace sn
