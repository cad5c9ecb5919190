// Quantized linear layer with few rows in one kernel: y = (x_scale * w_scale[n]) * sum_k value(q(x[i][k])) * value(wq[n][k]) +
// bias[n] (Sec. V-B, Y = W A; Sec. VI-A).
//
// With few rows the layer is a chain of latencies: two launches, a round trip to memory in each, the set-up of tensor memory
// and of the rings.  Here a block of eight warps has 8 or 16 rows and 16 to 64 columns, every warp takes each eighth 64 elements of
// the reduction from global memory straight into registers, turns the activations into codes and both operands into FP16
// numbers (every E4M3, E5M2 and E2M1 value is one) and multiplies them with mma.sync: no shared memory, no barrier until the
// warps' sums are added up.  A 128-row tcgen05 tile would be mostly empty, and its operands would have to go through shared
// memory first.  Products are exact and sums FP32, as on the other routes (error against 64 bits 3.5e-8 to 6e-8, theirs 3.5e-8 to 9e-8).
// What bounds it: with one block per SM the chain of loads, converts and MMAs, some 0.4 to 0.9 us per 64 elements of a warp; with
// several the conversions, which every block does for itself.  Whole layer, us here / two kernels, E2M1 weights: 16 x 320 -> 320 1.7 /
// 5.3, 64 x 320 -> 1280 3.2 / 5.4, 8 x 1280 -> 1280 2.8 / 6.3, 32 x 1280 -> 1280 3.6 / 6.6; against a warp per column on the CUDA cores
// (fpq_smallm.cu): 2 x 1280 -> 1280 2.4 / 3.8, 8 x 320 -> 1280 1.8 / 4.7.
#include <cuda_fp16.h>

#include "fpq_common.cuh"
#include "fpq_kernels.h"

namespace fpq {

namespace {

constexpr int WARPS = 8, THREADS = 32 * WARPS, KG = 64;
enum { W_E4M3 = 0, W_E2M1 = 1, W_E5M2 = 2 };

// values of two 8-bit codes (low byte first) as FP16
template <bool E5>
__device__ __forceinline__ uint32_t two_values(uint16_t codes)
{
    uint32_t h2;
    if (E5)
        asm("cvt.rn.f16x2.e5m2x2 %0, %1;" : "=r"(h2) : "h"(codes));
    else
        asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(h2) : "h"(codes));
    return h2;
}
// The values that two activations are quantized to (Sec. IV-B; hardware converts there and back); NaN stays one here, and minus
// zero: neither sign of a zero reaches a sum that starts with +0.
template <bool E5>
__device__ __forceinline__ uint32_t quantized(float lo, float hi, unsigned long long rinv2)
{
    unsigned long long t;
    asm("mov.b64 %0, {%1, %2};" : "=l"(t) : "f"(lo), "f"(hi));
    asm("mul.rn.f32x2 %0, %0, %1;" : "+l"(t) : "l"(rinv2));
    float a, b;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(t));
    uint16_t c;
    if (E5)
        asm("cvt.rn.satfinite.e5m2x2.f32 %0, %1, %2;" : "=h"(c) : "f"(b), "f"(a));
    else
        asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(c) : "f"(b), "f"(a));
    return two_values<E5>(c);
}
// NaN counts as zero
__device__ __forceinline__ void nan_to_zero(uint32_t& v)
{
    if ((v & 0x7fffu) > 0x7c00u) v &= 0xffff0000u;
    if ((v & 0x7fff0000u) > 0x7c000000u) v &= 0xffffu;
}
__device__ __forceinline__ __half2 as_half2(uint32_t v) { return *reinterpret_cast<__half2*>(&v); }

// values of eight E2M1 codes (low nibble first)
__device__ __forceinline__ void eight_values(uint32_t codes, uint32_t (&v)[4])
{
    asm("{\n\t.reg .b8 a, b, c, d;\n\t"
        "mov.b32 {a, b, c, d}, %4;\n\t"
        "cvt.rn.f16x2.e2m1x2 %0, a;\n\t"
        "cvt.rn.f16x2.e2m1x2 %1, b;\n\t"
        "cvt.rn.f16x2.e2m1x2 %2, c;\n\t"
        "cvt.rn.f16x2.e2m1x2 %3, d;\n\t}"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
        : "r"(codes));
}

__device__ __forceinline__ void mma_f16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

struct FewArgs {
    const float* x;
    const uint8_t* w;          // [N][terms][Kp] codes, 4-bit ones packed
    const float *w_scale, *bias;
    float* y;
    int M, N, K, Kp;
    float rinv, x_scale;       // of the codes; of the result
    int* status;
};

// A block has 8 R rows (R = 1, 2) and 8 NT columns.  The lanes of a quad have 16 neighbouring elements of the reduction each;
// the MMA's step s takes the fourth s of them (its own order of the reduction is the same for both operands, so any will do).
template <int WF, bool E5, int R, int NT, bool SHORT>
__global__ void __launch_bounds__(THREADS, NT < 8 ? 2 : 1) few_rows_kernel(const FewArgs g)
{
    constexpr int COLS = 8 * NT;
    __shared__ float sums[WARPS][8 * R][COLS + 4];
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, q = lane & 3, r = lane >> 2;
    const int n0 = blockIdx.x * COLS, m0 = blockIdx.y * (8 * R);
    const int row_bytes = WF == W_E2M1 ? g.Kp / 2 : g.Kp;
    unsigned long long rinv2;
    asm("mov.b64 %0, {%1, %1};" : "=l"(rinv2) : "f"(g.rinv));
    float acc[NT][4] = {};
    bool nan = false;
    const uint8_t* wp[NT];
#pragma unroll
    for (int j = 0; j < NT; ++j)
        wp[j] = g.w + (int64_t)min(n0 + 8 * j + r, g.N - 1) * row_bytes + (WF == W_E2M1 ? 8 : 16) * q;
    const float* xp[R];
    bool there[R];
#pragma unroll
    for (int i = 0; i < R; ++i) {
        there[i] = m0 + 8 * i + r < g.M;
        xp[i] = g.x + (int64_t)(there[i] ? m0 + 8 * i + r : 0) * g.K + 16 * q;
    }
    if constexpr (SHORT) {
        // Four warps share a group of 64, a step of the MMA each; no sum is longer than 16 products, to which the MMA adds zero
        // (it cuts off what it adds to an accumulator).
        for (int k0 = (warp >> 2) * KG; k0 < g.K; k0 += 2 * KG) {
            const int s = warp & 3, k = k0 + 16 * q + 4 * s;
            uint32_t codes[NT], a[R][2];
#pragma unroll
            for (int j = 0; j < NT; ++j)
                codes[j] = __ldg(reinterpret_cast<const uint32_t*>(wp[j] + (WF == W_E2M1 ? k0 / 2 + (s & 2) * 2 : k0 + 4 * s)));
#pragma unroll
            for (int i = 0; i < R; ++i) {
                const float4 v = there[i] && k < g.K ? __ldg(reinterpret_cast<const float4*>(xp[i] + k0 + 4 * s)) : make_float4(0.f, 0.f, 0.f, 0.f);
                a[i][0] = quantized<E5>(v.x, v.y, rinv2);
                a[i][1] = quantized<E5>(v.z, v.w, rinv2);
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    if (__hisnan(__low2half(as_half2(a[i][h]))) || __hisnan(__high2half(as_half2(a[i][h])))) {
                        nan = true;
                        nan_to_zero(a[i][h]);
                    }
            }
            const uint32_t av[4] = {a[0][0], R == 1 ? 0u : a[R - 1][0], a[0][1], R == 1 ? 0u : a[R - 1][1]};
#pragma unroll
            for (int j = 0; j < NT; ++j) {
                uint32_t b[4];
                if (WF == W_E2M1) {
                    eight_values(codes[j], b);
                    if (s & 1) b[0] = b[2], b[1] = b[3];
                } else {
                    b[0] = two_values<WF == W_E5M2>((uint16_t)(codes[j] & 0xffffu));
                    b[1] = two_values<WF == W_E5M2>((uint16_t)(codes[j] >> 16));
                }
                float part[4] = {};
                mma_f16(part, av, b[0], b[1]);
#pragma unroll
                for (int h = 0; h < 4; ++h)
                    acc[j][h] += part[h];
            }
        }
    } else {
        uint4 wv[NT];
        float4 xv[R][4];
        auto load = [&](int k0) {
#pragma unroll
            for (int j = 0; j < NT; ++j) {
                if (WF == W_E2M1) {
                    const uint2 v = __ldg(reinterpret_cast<const uint2*>(wp[j] + k0 / 2));
                    wv[j] = make_uint4(v.x, v.y, 0u, 0u);
                } else {
                    wv[j] = __ldg(reinterpret_cast<const uint4*>(wp[j] + k0));
                }
            }
#pragma unroll
            for (int i = 0; i < R; ++i)
#pragma unroll
                for (int s = 0; s < 4; ++s)
                    xv[i][s] = there[i] && k0 + 16 * q + 4 * s < g.K ? __ldg(reinterpret_cast<const float4*>(xp[i] + k0 + 4 * s))
                                                                      : make_float4(0.f, 0.f, 0.f, 0.f);
        };
        int k0 = warp * KG;
        if (k0 < g.K)
            load(k0);
        for (; k0 < g.K; k0 += WARPS * KG) {
            uint32_t a[R][4][2];
            __half2 most = __float2half2_rn(0.f);
#pragma unroll
            for (int i = 0; i < R; ++i)
#pragma unroll
                for (int s = 0; s < 4; ++s) {
                    a[i][s][0] = quantized<E5>(xv[i][s].x, xv[i][s].y, rinv2);
                    a[i][s][1] = quantized<E5>(xv[i][s].z, xv[i][s].w, rinv2);
                    most = __hmax2_nan(most, __hmax2_nan(__habs2(as_half2(a[i][s][0])), __habs2(as_half2(a[i][s][1]))));
                }
            if (__hisnan(__low2half(most)) || __hisnan(__high2half(most))) {
                nan = true;
#pragma unroll
                for (int i = 0; i < R; ++i)
#pragma unroll
                    for (int s = 0; s < 4; ++s)
#pragma unroll
                        for (int h = 0; h < 2; ++h)
                            nan_to_zero(a[i][s][h]);
            }
            uint32_t b[NT][4][2];
#pragma unroll
            for (int j = 0; j < NT; ++j) {
                if (WF == W_E2M1) {
                    uint32_t lo[4], hi[4];
                    eight_values(wv[j].x, lo);
                    eight_values(wv[j].y, hi);
                    b[j][0][0] = lo[0], b[j][0][1] = lo[1], b[j][1][0] = lo[2], b[j][1][1] = lo[3];
                    b[j][2][0] = hi[0], b[j][2][1] = hi[1], b[j][3][0] = hi[2], b[j][3][1] = hi[3];
                } else {
                    const uint32_t c[4] = {wv[j].x, wv[j].y, wv[j].z, wv[j].w};
#pragma unroll
                    for (int s = 0; s < 4; ++s) {
                        b[j][s][0] = two_values<WF == W_E5M2>((uint16_t)(c[s] & 0xffffu));
                        b[j][s][1] = two_values<WF == W_E5M2>((uint16_t)(c[s] >> 16));
                    }
                }
            }
            if (k0 + WARPS * KG < g.K)
                load(k0 + WARPS * KG);
            // (the MMA cuts off what it adds to an accumulator, so a sum of 64 products starts from zero and is added by an FP32 addition)
            float part[NT][4] = {};
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                const uint32_t av[4] = {a[0][s][0], R == 1 ? 0u : a[R - 1][s][0], a[0][s][1], R == 1 ? 0u : a[R - 1][s][1]};
#pragma unroll
                for (int j = 0; j < NT; ++j)
                    mma_f16(part[j], av, b[j][s][0], b[j][s][1]);
            }
#pragma unroll
            for (int j = 0; j < NT; ++j)
#pragma unroll
                for (int h = 0; h < 4; ++h)
                    acc[j][h] += part[j][h];
        }
    }
#pragma unroll
    for (int j = 0; j < NT; ++j) {
        *reinterpret_cast<float2*>(&sums[warp][r][8 * j + 2 * q]) = make_float2(acc[j][0], acc[j][1]);
        if (R > 1)
            *reinterpret_cast<float2*>(&sums[warp][8 * (R - 1) + r][8 * j + 2 * q]) = make_float2(acc[j][2], acc[j][3]);
    }
    __syncthreads();
    for (int id = threadIdx.x; id < 8 * R * COLS; id += THREADS) {
        const int i = id / COLS, c = id % COLS, n = n0 + c;
        // In pairs; what the last two levels, whose sums are the largest, round away is kept (Knuth's two-sum) and added last: the error
        // of the layer against 64 bits is 9 % below that of a warp per column (1 to 8 rows of 64 to 5120) and 25 % below
        // that of the two kernels, where the warps' sums one after the other were 1 % above the former; 0.3 % of the time.
        float v[WARPS], lost = 0.f;
#pragma unroll
        for (int k = 0; k < WARPS; ++k)
            v[k] = sums[k][i][c];
#pragma unroll
        for (int s = 1; s < WARPS; s *= 2)
#pragma unroll
            for (int k = 0; k < WARPS; k += 2 * s) {
                const float t = __fadd_rn(v[k], v[k + s]);
                if (s > 1) {
                    const float z = __fsub_rn(t, v[k]);
                    lost += __fadd_rn(__fsub_rn(v[k], __fsub_rn(t, z)), __fsub_rn(v[k + s], z));
                }
                v[k] = t;
            }
        if (m0 + i < g.M && n < g.N) {
            const float scale = g.x_scale * __ldg(g.w_scale + n), low = lost * scale;
            // (nothing where that is not finite: with an infinite scale the result is infinite, not 0 * infinity)
            g.y[(int64_t)(m0 + i) * g.N + n] = fmaf(v[0], scale, (g.bias ? __ldg(g.bias + n) : 0.f) + (fabsf(low) < INFINITY ? low : 0.f));
        }
    }
    if (nan)
        flag_status(g.status, FPQ_ERR_NAN_INPUT);
}

// Whether sums of a group of 64 are formed in four warps instead of one: where otherwise the error against 64 bits is above that of the
// route that such a layer takes without this kernel (8 rows of 64 / 128 / 136 0.8 / 1.4 / 0.3 % above a warp per column, so 0.4 / 1.8 / 2 %
// below it, and below it in any case from 144 on; 16 and 64 rows of 64 0.3 % above two kernels, so 1.3 % below), and nowhere else: where all
// warps are busy anyway it takes longer (127 x 128 -> 1280 3.2 us, so 3.6; 8 x 256 -> 7680 2.1 and 2.8).  By the rows of the whole call:
// results do not depend on how it is cut.
bool short_sums(int64_t whole, int64_t K) { return K <= KG || (whole <= 8 && K < 2 * KG + 16); }

// Rows and columns of a block.  us: a launch with its first round trip and one block per SM; more per 512 elements of the reduction;
// and what every further block of an SM adds, and adds per 512 elements.  Fitted to the choices at 1896 shapes of 1 to 127 rows, 64 to
// 5120 elements and 64 to 10240 columns with either size of weights: what is chosen takes 0.5 % more than the fastest of the forms and the two
// kernels.  (Of 4700 others 8 take more than 1.1 times as long as without this kernel, at most 1.19; with whole steps of 512 and a
// time of the two kernels that did not know the rows 48, at most 1.47: 24 x 1024 -> 10240 11.2 us, two kernels 7.9.)
struct Form {
    int R, NT;
    double first, first_step, more, more_step;
};
constexpr Form FORMS[] = {{1, 2, 1.39, 0.29, 0.29, 0.33}, {1, 4, 1.45, 0.34, 0.44, 0.54}, {1, 8, 1.82, 0.71, 1.28, 0.75},
                          {2, 4, 1.77, 0.76, 0.47, 0.78}, {2, 8, 2.57, 0.87, 1.58, 1.03}};
const Form& best_form(int64_t M, int64_t N, int64_t K, int64_t whole, double* us)
{
    const Form* best = nullptr;
    for (const Form& f : FORMS) {
        if (f.R == 2 && f.NT == 8 && short_sums(whole, K))
            continue;                                  // (never the fastest; not built)
        const int64_t blocks = (N + 8 * f.NT - 1) / (8 * f.NT) * ((M + 8 * f.R - 1) / (8 * f.R));
        const double steps = (double)K / (WARPS * KG), per_sm = (double)((blocks + 147) / 148);
        const double t = f.first + steps * f.first_step + (per_sm - 1.0) * (f.more + steps * f.more_step);
        if (!best || t < *us) {
            best = &f;
            *us = t;
        }
    }
    return *best;
}

template <int WF, bool E5, bool SHORT>
auto kernel_of(const Form& f)
{
    return f.R == 1 ? (f.NT == 2   ? few_rows_kernel<WF, E5, 1, 2, SHORT>
                       : f.NT == 4 ? few_rows_kernel<WF, E5, 1, 4, SHORT>
                                   : few_rows_kernel<WF, E5, 1, 8, SHORT>)
           : SHORT || f.NT == 4 ? few_rows_kernel<WF, E5, 2, 4, SHORT>
                                : few_rows_kernel<WF, E5, 2, 8, false>;
}

template <int WF, bool E5>
cudaError_t launch(const FewArgs& g, int64_t whole, cudaStream_t st)
{
    double us;
    const Form& f = best_form(g.M, g.N, g.K, whole, &us);
    const dim3 grid((unsigned)((g.N + 8 * f.NT - 1) / (8 * f.NT)), (unsigned)((g.M + 8 * f.R - 1) / (8 * f.R)));
    const auto kernel = short_sums(whole, g.K) ? kernel_of<WF, E5, true>(f) : kernel_of<WF, E5, false>(f);
    return launch_overlapped(kernel, grid, THREADS, 0, st, g);
}

bool few_rows_applies(const GemmProblem& p)
{
    // Rows are read as 16-byte pieces: K a multiple of 4.  Less than the 128 rows of a tcgen05 tile: from there on a layer gives,
    // bit for bit, what the 1 x 1 convolution of the same numbers gives, whose MMAs add in the same order (128 x 96 -> 160
    // would be faster here too, 1.8 us against 5.0; 128 x 1280 -> 1280 would not, 8.5 against 7.0).
    return !p.conv && p.c_seg == 0 && p.C % 4 == 0 && p.C >= 4 && p.C <= (1 << 20) && p.M >= 1 && p.M < 128 && p.N <= (1 << 24) &&
           (uintptr_t)p.x % 16 == 0;
}

}  // namespace

bool few_rows_preferred(const GemmProblem& p)
{
    if (!few_rows_applies(p))
        return false;
    double us;
    best_form(p.M, p.N, p.C, p.M, &us);
    if (1000.0 * us > two_kernels_ns(p.M, p.C, p.N))
        return false;
    // (0.88: the form on the CUDA cores is up to 15 % below its estimate at the smallest sizes; 1 x 64 -> 320 1.33 us there, 1.53 here)
    return p.w_e5m2 || p.a_e5m2 || 1000.0 * us < 0.88 * small_m_linear_ns(p.M, p.C, p.N, p.w4);
}

fpq_status launch_few_rows(const GemmProblem& p, int64_t whole, cudaStream_t st)
{
    if (!few_rows_applies(p))
        return FPQ_ERR_UNSUPPORTED;
    FewArgs g;
    g.x = p.x, g.w = (const uint8_t*)p.w_prepared, g.w_scale = p.w_scale, g.bias = p.bias, g.y = p.y;
    g.M = (int)p.M, g.N = p.N, g.K = p.C, g.Kp = p.Cp;
    g.rinv = 1.0f / p.x_scale, g.x_scale = p.x_scale;
    g.status = status_word();
    if (!g.status)
        return FPQ_ERR_CUDA;
    cudaError_t e;
    if (p.a_e5m2)
        e = p.w4 ? launch<W_E2M1, true>(g, whole, st) : p.w_e5m2 ? launch<W_E5M2, true>(g, whole, st) : launch<W_E4M3, true>(g, whole, st);
    else
        e = p.w4 ? launch<W_E2M1, false>(g, whole, st) : p.w_e5m2 ? launch<W_E5M2, false>(g, whole, st) : launch<W_E4M3, false>(g, whole, st);
    return e == cudaSuccess ? FPQ_OK : FPQ_ERR_CUDA;
}

}  // namespace fpq
