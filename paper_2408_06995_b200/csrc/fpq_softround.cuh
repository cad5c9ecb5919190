// Device functions that the kernels of the rounding-learning step share (Sec. V-B).
#pragma once

#include "fpq_common.cuh"

namespace fpq {

namespace {

// sigma(alpha), sigma (1 - sigma) and u = 2 |sigma - 0.5| = tanh(|alpha| / 2), each from expressions without
// cancellation (1 - sigma and sigma - 0.5 formed by subtraction lose most of their bits once sigma saturates,
// and the regulariser raises u to the 19th power).
struct SoftTerms {
    float sig, sp, u;
};
__device__ __forceinline__ SoftTerms soft_terms(float al)
{
    float t = expf(-fabsf(al));
    float inv = 1.0f / (1.0f + t);
    SoftTerms o;
    o.sig = al >= 0.f ? inv : t * inv;
    o.sp = t * inv * inv;
    o.u = tanhf(0.5f * fabsf(al));
    return o;
}

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Adds one value per thread over the block and then into *dst (one atomic per block).
__device__ __forceinline__ void block_atomic_add(double v, double* dst)
{
    __shared__ double warp_part[32];
    v = warp_sum(v);
    int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0)
        warp_part[wid] = v;
    __syncthreads();
    if (wid == 0) {
        int nw = (blockDim.x + 31) >> 5;
        double s = lane < nw ? warp_part[lane] : 0.0;
        s = warp_sum(s);
        if (lane == 0)
            atomicAdd(dst, s);
    }
}

// Learned-rounding equation of Sec. V-B with the sigmoid kept soft, for one weight.
struct SoftWeight {
    float e, dq;               // Wq(alpha) - w, dWq/dalpha
};
__device__ __forceinline__ SoftWeight soft_weight(float wv, float al, float g, float r, float c, const QFormat& f, bool& nan)
{
    const float t = __fmul_rn(wv, r);
    if (t != t) {
        nan = true;
        return {0.f, 0.f};
    }
    const SoftTerms st = soft_terms(al);
    const float a = fminf(fmaxf(t, -c), c);
    const int Eb = (int)((__float_as_uint(a) >> 23) & 0xffu);
    const int e_eff = max(Eb - 127, 1 - f.B);                                 // binade whose step applies
    const float s = __uint_as_float((uint32_t)(e_eff - f.m + 127) << 23);     // step, a power of two
    const float s_inv = __uint_as_float((uint32_t)(f.m - e_eff + 127) << 23);
    const float fl = floorf(a * s_inv);                                       // exact: power-of-two scaling
    const float pre = s * (fl + st.sig);
    const float q = fminf(fmaxf(pre, -c), c);
    return {fmaf(g, q, -wv), (pre >= -c && pre <= c) ? g * s * st.sp : 0.f};
}

// reg * dlambda/dalpha; lam += lambda(alpha)
__device__ __forceinline__ float regulariser_gradient(const SoftTerms& st, float al, float reg, float& lam)
{
    const float u = st.u;
    const float u2 = u * u, u4 = u2 * u2, u8 = u4 * u4, u16 = u8 * u8;
    lam += 1.0f - u16 * u4;
    const float u19 = u16 * u2 * u;
    const float dlam = -40.0f * u19 * (al > 0.f ? 1.f : (al < 0.f ? -1.f : 0.f)) * st.sp;
    return reg * dlam;
}

// gradient of one weight's alpha: g * dWq/dalpha + reg * dlambda/dalpha; lam += lambda(alpha)
__device__ __forceinline__ float weight_gradient(float g, float dq, float al, float reg, float& lam)
{
    return fmaf(g, dq, regulariser_gradient(soft_terms(al), al, reg, lam));
}

}  // namespace

}  // namespace fpq
