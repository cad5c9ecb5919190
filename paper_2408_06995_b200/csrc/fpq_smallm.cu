// Quantized linear layer with a handful of rows (the time-embedding projections of a
// U-Net: M = batch): y = (x_scale * w_scale[n]) * sum_k value(q(x[i][k])) * value(wq[n][k]) + bias[n]
// (Sec. V-B, Y = W A; Sec. VI-A).  With M <= 8 and few weights the tensor-core path spends its time on launches
// and pipeline set-up, while the whole layer is one pass over the weights: a warp, or a few, per
// output column reads that column's codes once, decodes them on the CUDA cores and keeps one FP32
// sum per row (the few activation rows come from the caches, quantized again by every warp).  Every product of an E4M3 value and an E4M3 / E2M1 value is exact in FP32, so
// this path differs from the tensor-core path only in the order of the FP32 additions.
#include <cuda_fp16.h>

#include "fpq_common.cuh"
#include "fpq_kernels.h"

namespace fpq {

constexpr int SMALLM_THREADS = 128;
constexpr int SMALLM_MAX_ROWS = 8;

// two E4M3 codes (low byte first) -> their values
__device__ __forceinline__ float2 e4m3x2_values(uint16_t codes)
{
    uint32_t h2;
    asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(h2) : "h"(codes));
    return __half22float2(*reinterpret_cast<__half2*>(&h2));
}

// one E2M1 code (bias 1): 0, 0.5, 1, 1.5, 2, 3, 4, 6 with a sign bit, built as FP32 bits
__device__ __forceinline__ float e2m1_value(uint32_t code)
{
    const uint32_t mag = code & 7u;
    const uint32_t normal = ((126u + (mag >> 1)) << 23) | ((mag & 1u) << 22);     // (1 + d/2) 2^(p-1)
    const uint32_t sub = (mag & 1u) ? 0x3f000000u : 0u;                            // d * 0.5
    return __uint_as_float((mag >= 2u ? normal : sub) | ((code & 8u) << 28));
}

// MR = rows held per thread (M rounded up to 1, 2, 4 or 8).  A warp owns an output column, or every KS-th step of one; per
// step a lane takes 4 bytes of that column's codes (4 or 8 reduction elements) and the matching 16 or 32 bytes of every
// activation row, quantizes the activations to E4M3 values on the fly (Sec. IV-B; hardware convert there and back) and adds
// the products.  Weights and activations of several steps are requested before the first is used.  What bounds it:
// instructions (the conversions are done again for every column) where there are many columns, the chain of steps where
// there are few, hence KS.  Steps past the end of the rows are left out as a whole: they took as long as the others (64
// -> 10240, 4-bit weights, one row: 16.7 us with them, 4.5 without).
template <bool W4, int MR, int KS>
__global__ void __launch_bounds__(SMALLM_THREADS) small_m_linear_kernel(const float* __restrict__ x, int M, int K, int Kp,
                                                                        const uint8_t* __restrict__ w, int N,
                                                                        const float* __restrict__ w_scale, float x_scale,
                                                                        float rinv, const float* __restrict__ bias,
                                                                        float* __restrict__ y, int* status)
{
    constexpr int PER = W4 ? 8 : 4;                   // reduction elements per lane and step
    constexpr int STEP = 32 * PER;
    constexpr int U = (MR * PER >= 32) ? 2 : (MR * PER >= 16 ? 4 : 8);     // steps in flight
    asm volatile("griddepcontrol.wait;" ::: "memory");
    bool nan = false;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int row_bytes = W4 ? Kp / 2 : Kp;
    constexpr int COLUMNS = SMALLM_THREADS / 32 / KS;  // per block; KS neighbouring warps share one, every KS-th step each
    const int part = warp % KS, steps = (K + STEP - 1) / STEP;
    __shared__ float parts[KS > 1 ? SMALLM_THREADS / 32 : 1][MR];
    for (int n0 = blockIdx.x * COLUMNS; n0 < N; n0 += gridDim.x * COLUMNS) {
        const int n = min(n0 + warp / KS, N - 1);
        float acc[MR];
#pragma unroll
        for (int m = 0; m < MR; ++m)
            acc[m] = 0.f;
        const uint8_t* wr = w + (int64_t)n * row_bytes;
        for (int first = part; first < steps; first += U * KS) {
            uint32_t cw[U];
            float4 xv[U][MR][PER / 4];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (first + u * KS >= steps)
                    break;
                const int k0 = (first + u * KS) * STEP + lane * PER;
                const bool in = k0 < K;               // K is a multiple of 4: a group of four never straddles the end
                cw[u] = in ? __ldg(reinterpret_cast<const uint32_t*>(wr + (W4 ? k0 / 2 : k0))) : 0u;
#pragma unroll
                for (int m = 0; m < MR; ++m)
#pragma unroll
                    for (int e = 0; e < PER / 4; ++e)
                        xv[u][m][e] = (in && m < M && k0 + 4 * e < K)
                                          ? __ldg(reinterpret_cast<const float4*>(x + (int64_t)m * K + k0) + e)
                                          : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (first + u * KS >= steps)
                    break;
                float wv[PER];
                if (W4) {
#pragma unroll
                    for (int e = 0; e < 8; ++e)
                        wv[e] = e2m1_value(cw[u] >> (4 * e));               // even index in the low nibble
                } else {
                    const float2 a = e4m3x2_values((uint16_t)(cw[u] & 0xffffu)), b = e4m3x2_values((uint16_t)(cw[u] >> 16));
                    wv[0] = a.x; wv[1] = a.y; wv[2] = b.x; wv[3] = b.y;
                }
#pragma unroll
                for (int m = 0; m < MR; ++m) {
#pragma unroll
                    for (int e = 0; e < PER / 4; ++e) {
                        const float4 t = xv[u][m][e];
                        const uint32_t c4 = e4m3x4_from_scaled(__fmul_rn(t.x, rinv), __fmul_rn(t.y, rinv),
                                                               __fmul_rn(t.z, rinv), __fmul_rn(t.w, rinv), nan);
                        const float2 lo = e4m3x2_values((uint16_t)(c4 & 0xffffu)), hi = e4m3x2_values((uint16_t)(c4 >> 16));
                        acc[m] = fmaf(lo.x, wv[4 * e], acc[m]);
                        acc[m] = fmaf(lo.y, wv[4 * e + 1], acc[m]);
                        acc[m] = fmaf(hi.x, wv[4 * e + 2], acc[m]);
                        acc[m] = fmaf(hi.y, wv[4 * e + 3], acc[m]);
                    }
                }
            }
        }
        const float sv = x_scale * __ldg(w_scale + n), bv = bias ? __ldg(bias + n) : 0.f;
#pragma unroll
        for (int m = 0; m < MR; ++m) {
            float a = acc[m];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
                a += __shfl_xor_sync(0xffffffffu, a, o);
            acc[m] = a;
            if (KS > 1 && lane == 0)
                parts[warp][m] = a;
        }
        if (KS > 1)
            __syncthreads();
        if (lane == 0 && part == 0 && n0 + warp / KS < N) {
#pragma unroll
            for (int m = 0; m < MR; ++m) {
                float a = acc[m];
#pragma unroll
                for (int k = 1; k < KS; ++k)
                    a += parts[warp + k][m];
                if (m < M)
                    y[(int64_t)m * N + n] = fmaf(a, sv, bv);
            }
        }
        if (KS > 1)
            __syncthreads();
    }
    if (nan)
        flag_status(status, FPQ_ERR_NAN_INPUT);
}

namespace {

struct SmallPlan {
    int mr, steps, ks;
    double ns;                 // estimate
};
// A column is shared by several warps while there are few columns and several steps (1280 -> 1280, 4-bit weights, two rows: one
// warp 4.5 us, two 3.9, four 4.2; 5120 -> 320: 6.7, 5.4, 4.5; 1280 -> 5120: 9.7, 9.8, 11.8).
SmallPlan plan_small(int64_t M, int64_t K, int64_t N, int w4)
{
    SmallPlan p;
    const int i = M <= 1 ? 0 : (M <= 2 ? 1 : (M <= 4 ? 2 : 3));
    p.mr = 1 << i;
    p.steps = (int)((K + (w4 ? 255 : 127)) / (w4 ? 256 : 128));
    p.ks = 1;
    if (N <= 2560 && p.steps >= (N <= 640 ? 2 : 4))
        p.ks = p.steps >= (N <= 640 ? 3 : 16) ? 4 : 2;
    // measured: ns per column and step, per column, and per step of a warp's chain
    static const double step[2][4] = {{0.061, 0.10, 0.17, 0.32}, {0.185, 0.266, 0.41, 0.754}};
    static const double column[2][4] = {{0.085, 0.17, 0.19, 0.29}, {0.115, 0.124, 0.16, 0.36}};
    static const double chain[2][4] = {{107, 127, 190, 330}, {150, 255, 430, 690}};
    p.ns = 1400.0 + (double)N * (p.steps * step[w4][i] + column[w4][i]) + ((p.steps + p.ks - 1) / p.ks) * chain[w4][i];
    return p;
}

}  // namespace

static bool in_range(int64_t M, int64_t K, int64_t N)
{
    // (rows are read as 16-byte pieces: K a multiple of 4)
    return M >= 1 && M <= SMALLM_MAX_ROWS && K % 4 == 0 && K <= (1 << 20) && N >= 1 && N <= 0x7fffffff;
}

double small_m_linear_ns(int64_t M, int64_t K, int64_t N, int w4) { return in_range(M, K, N) ? plan_small(M, K, N, w4).ns : 1e30; }

double two_kernels_ns(int64_t M, int64_t K, int64_t N)
{
    const double head = (double)(K < 320 ? K : 320), tail = (double)(K > 320 ? K - 320 : 0), weights = (double)N * (double)K;
    const double few = 4200.0 + 2.8 * head + 0.3 * tail + 3.3e-4 * weights + 0.05 * (double)N;
    if (M <= SMALLM_MAX_ROWS)
        return few;
    // (fitted to 9894 shapes of 9 to 127 rows and up to 13 us, 7 % rms; up to 24 rows large weights take longer: 9 x 5120 -> 10240 23.7 us,
    // 32 x 5120 -> 10240 15.5; 24 x 1920 -> 5120 9.9, 32 x 1920 -> 5120 7.4)
    const double more = 4350.0 + 2.44 * head + 0.385 * tail + 2.2e-4 * weights + 0.018 * (double)N + 3.6 * (double)M;
    return M <= 24 && few > more ? few : more;
}

// Whether one pass on the CUDA cores is expected to be faster than the quantize kernel and the contraction (where the route may be one
// kernel, few_rows_preferred is asked first and leaves this one layers of few columns and single rows of short reductions), whose
// time in chains of its kind is fitted by two_kernels_ns (us, here / there: 1280 -> 1280, 4-bit weights, 2 rows 3.9 / 6.3,
// 8 rows 9.4 / 6.5; 1280 -> 10240, one row 11.7 / 8.9; 5120 -> 10240, 8 rows 156 / 23; 8-bit weights: 1280 -> 10240, one row
// 8.2 / 9.8, 8 rows 37 / 9.8; 5120 -> 320, 4 rows 5.2 / 7.2, 8 rows 8.5 / 7.3).
bool small_m_linear_preferred(int64_t M, int64_t K, int64_t N, int w4)
{
    return in_range(M, K, N) && plan_small(M, K, N, w4).ns <= two_kernels_ns(M, K, N);
}

template <bool W4, int MR, int KS>
static void launch_small(int blocks, const float* x, int M, int K, int Kp, const uint8_t* w, int N, const float* w_scale,
                         float x_scale, const float* bias, float* y, cudaStream_t st)
{
    (void)launch_overlapped(small_m_linear_kernel<W4, MR, KS>, dim3(blocks), SMALLM_THREADS, 0, st, x, M, K, Kp, w, N, w_scale,
                            x_scale, 1.0f / x_scale, bias, y, status_word());
}

fpq_status launch_small_m_linear(const float* x, int M, int K, const void* w_prepared, int w4, int N, const float* w_scale,
                                 float x_scale, const float* bias, float* y, cudaStream_t st)
{
    const int Kp = (int)round_up(K, 128);
    const uint8_t* w = (const uint8_t*)w_prepared;
    const SmallPlan p = plan_small(M, K, N, w4);
    const int mr = p.mr, ks = p.ks;
    const int64_t blocks64 = ((int64_t)N * ks + SMALLM_THREADS / 32 - 1) / (SMALLM_THREADS / 32);
    const int blocks = (int)(blocks64 > 148 * 16 ? 148 * 16 : blocks64);
#define FPQ_SMALL_KS(W4, MR, KS) launch_small<W4, MR, KS>(blocks, x, M, K, Kp, w, N, w_scale, x_scale, bias, y, st)
#define FPQ_SMALL(W4, MR) (ks == 1 ? FPQ_SMALL_KS(W4, MR, 1) : ks == 2 ? FPQ_SMALL_KS(W4, MR, 2) : FPQ_SMALL_KS(W4, MR, 4))
    if (w4) {
        if (mr == 1) FPQ_SMALL(true, 1); else if (mr == 2) FPQ_SMALL(true, 2); else if (mr == 4) FPQ_SMALL(true, 4); else FPQ_SMALL(true, 8);
    } else {
        if (mr == 1) FPQ_SMALL(false, 1); else if (mr == 2) FPQ_SMALL(false, 2); else if (mr == 4) FPQ_SMALL(false, 4); else FPQ_SMALL(false, 8);
    }
#undef FPQ_SMALL
#undef FPQ_SMALL_KS
    return cudaGetLastError() == cudaSuccess ? FPQ_OK : FPQ_ERR_CUDA;
}

}  // namespace fpq
