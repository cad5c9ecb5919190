// Rounding learning (Sec. V-B): one evaluation of the objective
//     mean((A Wq(alpha)^T - A W^T)^2) + reg * sum_i lambda(alpha_i)
// and of its gradient with respect to alpha, for a bias-free linear layer with FP32 calibration
// activations A [M][K].  The paper runs this step in FP32, and the contractions keep at least that: the
// direct form as three TF32 tensor-core products per FP32 product (fpq_tf32.cu), or FP32 multiply-adds on the CUDA cores
// where rows are no multiple of 4 floats; the form with A^T A in double.
//
//   prepare_kernel          E = Wq(alpha) - W and dWq/dalpha per weight; A^T for the TF32 contractions
// direct form
//   tf32x3_gemm_kernel, or  D = A E^T            (= Yq - Y by linearity), sum of D^2; with few output tiles the
//   sgemm128<true>          reduction is cut into slices that reduce_d_kernel adds
//   the same, <false>       partial sums of D^T A over slices of the M rows
//   grad_finalize_kernel    slices added in a fixed order, chain rule, sum of lambda, optional descent update
// with many calibration rows (make_plan), where D^T A = E (A^T A) and sum D^2 = <E (A^T A), E> are less work
//   gram_kernel             A^T A in double, slices of rows; gram_reduce_kernel adds them
//   gram_grad_kernel        E (A^T A) in double, both losses, chain rule, optional descent update
//
//   harden_kernel           the inference rule: decision bit = (sigma(alpha) >= 0.5)
//   unfold_kernel           a convolution's input rows, so that the same step serves convolution weights
#include <math.h>

#include <mutex>

#include "fpq_kernels.h"

namespace fpq {

namespace {

constexpr int TILE = 128;      // output tile edge
constexpr int BK = 16;         // reduction elements per shared-memory stage
constexpr int LDS = TILE + 4;  // padded row length of a stage (floats)

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

// Two FP32 values in one 64-bit register, and the packed multiply-add on such pairs (each half an IEEE fused
// multiply-add, round to nearest): half the issue slots of two scalar instructions.
__device__ __forceinline__ unsigned long long pack2(float lo, float hi)
{
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(unsigned long long v, float& lo, float& hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ void fma2(unsigned long long& d, unsigned long long a, unsigned long long b)
{
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
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

// The first blocks: E and dWq/dalpha, four weights per thread (VEC, rows of a multiple of four) or one; block 0 empties
// the losses.  The others, where A is transposed: one 32 x 32 tile of A^T each.  One launch: both are short.
template <bool VEC>
__global__ void __launch_bounds__(256) prepare_kernel(const float* __restrict__ w, const float* __restrict__ scale, QFormat f,
                                                      const float* __restrict__ alpha, float* __restrict__ E,
                                                      float* __restrict__ DQ, double* __restrict__ loss, int64_t N, int64_t K,
                                                      int weight_blocks, const float* __restrict__ A, int64_t M,
                                                      float* __restrict__ AT, int64_t Mp, unsigned* __restrict__ ticket,
                                                      int* __restrict__ status)
{
    __shared__ float tile[32][33];
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if ((int)blockIdx.x >= weight_blocks) {
        const int64_t tiles_k = (K + 31) / 32, id = (int64_t)blockIdx.x - weight_blocks;
        const int64_t m0 = id / tiles_k * 32, k0 = (id - id / tiles_k * tiles_k) * 32;
        const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
#pragma unroll
        for (int r = ty; r < 32; r += 8)
            tile[r][tx] = (m0 + r < M && k0 + tx < K) ? A[(m0 + r) * K + k0 + tx] : 0.f;
        __syncthreads();
#pragma unroll
        for (int r = ty; r < 32; r += 8)
            if (k0 + r < K && m0 + tx < M)
                AT[(k0 + r) * Mp + m0 + tx] = tile[tx][r];
        return;
    }
    if (blockIdx.x == 0 && threadIdx.x < 2)
        loss[threadIdx.x] = 0.0;
    if (blockIdx.x == 0 && threadIdx.x == 2)
        *ticket = 0;
    constexpr int V = VEC ? 4 : 1;
    const float c = __uint_as_float(f.cmax_bits);
    const int64_t per_row = K / V, total = N * per_row;
    bool nan = false;
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < total; i += (int64_t)weight_blocks * 256) {
        const int64_t n = total < 0x80000000ll ? (int64_t)((uint32_t)i / (uint32_t)per_row) : i / per_row;
        const float g = __ldg(scale + n), r = __fdiv_rn(1.0f, g);
        if (VEC) {
            const float4 wv = __ldg(reinterpret_cast<const float4*>(w) + i), al = __ldg(reinterpret_cast<const float4*>(alpha) + i);
            const SoftWeight o0 = soft_weight(wv.x, al.x, g, r, c, f, nan), o1 = soft_weight(wv.y, al.y, g, r, c, f, nan),
                             o2 = soft_weight(wv.z, al.z, g, r, c, f, nan), o3 = soft_weight(wv.w, al.w, g, r, c, f, nan);
            reinterpret_cast<float4*>(E)[i] = make_float4(o0.e, o1.e, o2.e, o3.e);
            reinterpret_cast<float4*>(DQ)[i] = make_float4(o0.dq, o1.dq, o2.dq, o3.dq);
        } else {
            const SoftWeight o = soft_weight(__ldg(w + i), __ldg(alpha + i), g, r, c, f, nan);
            E[i] = o.e;
            DQ[i] = o.dq;
        }
    }
    if (nan)
        flag_status(status, FPQ_ERR_NAN_INPUT);
}

// C[i][j] = sum_r P(i, r) Q(j, r) over r in [z * r_per_split, min(R, (z + 1) * r_per_split)), z = blockIdx.z,
// written to C + z * I * ldc.  RED_CONTIG: P(i, r) = P[i * ldp + r] (reduction index contiguous); otherwise
// P(i, r) = P[r * ldp + i] (output index contiguous); the same for Q.  256 threads, 8 x 8 outputs per thread,
// next stage fetched into registers while the current one is multiplied.  sq_sum (optional) receives the sum
// of the squared outputs.
template <bool RED_CONTIG>
__global__ void __launch_bounds__(256, 2) sgemm128(const float* __restrict__ P, int64_t ldp, const float* __restrict__ Q,
                                                   int64_t ldq, float* __restrict__ C, int64_t ldc, int I, int J,
                                                   int64_t R, int64_t r_per_split, double* __restrict__ sq_sum)
{
    __shared__ __align__(16) float Ps[2][BK][LDS];
    __shared__ __align__(16) float Qs[2][BK][LDS];
    asm volatile("griddepcontrol.wait;" ::: "memory");

    const int t = threadIdx.x;
    const int i0 = blockIdx.x * TILE, j0 = blockIdx.y * TILE;
    const int64_t r_begin = (int64_t)blockIdx.z * r_per_split;
    const int64_t r_end = min(R, r_begin + r_per_split);
    C += (int64_t)blockIdx.z * I * ldc;
    const bool vec_p = (ldp % 4 == 0) && (((uintptr_t)P) % 16 == 0);
    const bool vec_q = (ldq % 4 == 0) && (((uintptr_t)Q) % 16 == 0);

    float4 pf[2], qf[2];

    // fetch one stage (16 reduction elements x 128 outputs of each operand) into registers
    auto fetch = [&](const float* __restrict__ X, int64_t ld, int x0, int X_extent, bool vec, int64_t r0, float4* out) {
#pragma unroll
        for (int pass = 0; pass < 2; ++pass) {
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (RED_CONTIG) {
                int row = (t >> 2) + 64 * pass;
                int64_t r = r0 + (t & 3) * 4;
                int xi = x0 + row;
                if (xi < X_extent) {
                    const float* src = X + (int64_t)xi * ld + r;
                    if (vec && r + 3 < r_end) {
                        v = __ldg(reinterpret_cast<const float4*>(src));
                    } else {
                        if (r + 0 < r_end) v.x = __ldg(src + 0);
                        if (r + 1 < r_end) v.y = __ldg(src + 1);
                        if (r + 2 < r_end) v.z = __ldg(src + 2);
                        if (r + 3 < r_end) v.w = __ldg(src + 3);
                    }
                }
            } else {
                int64_t r = r0 + (t >> 5) + 8 * pass;
                int xi = x0 + (t & 31) * 4;
                if (r < r_end) {
                    const float* src = X + r * ld + xi;
                    if (vec && xi + 3 < X_extent) {
                        v = __ldg(reinterpret_cast<const float4*>(src));
                    } else {
                        if (xi + 0 < X_extent) v.x = __ldg(src + 0);
                        if (xi + 1 < X_extent) v.y = __ldg(src + 1);
                        if (xi + 2 < X_extent) v.z = __ldg(src + 2);
                        if (xi + 3 < X_extent) v.w = __ldg(src + 3);
                    }
                }
            }
            out[pass] = v;
        }
    };
    // registers -> shared memory, reduction index outermost
    auto stash = [&](float (*S)[LDS], const float4* in) {
#pragma unroll
        for (int pass = 0; pass < 2; ++pass) {
            if (RED_CONTIG) {
                int row = (t >> 2) + 64 * pass;
                int r4 = (t & 3) * 4;
                S[r4 + 0][row] = in[pass].x;
                S[r4 + 1][row] = in[pass].y;
                S[r4 + 2][row] = in[pass].z;
                S[r4 + 3][row] = in[pass].w;
            } else {
                int r = (t >> 5) + 8 * pass;
                *reinterpret_cast<float4*>(&S[r][(t & 31) * 4]) = in[pass];
            }
        }
    };

    unsigned long long acc2[8][4];   // acc2[a][b] = outputs (a, 2 b) and (a, 2 b + 1) of the thread's 8 x 8
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b)
            acc2[a][b] = 0ull;

    const int ty = t >> 4, tx = t & 15;
    int buf = 0;
    if (r_begin < r_end) {
        fetch(P, ldp, i0, I, vec_p, r_begin, pf);
        fetch(Q, ldq, j0, J, vec_q, r_begin, qf);
        stash(Ps[0], pf);
        stash(Qs[0], qf);
    }
    __syncthreads();
    for (int64_t r0 = r_begin; r0 < r_end; r0 += BK) {
        const bool more = r0 + BK < r_end;
        if (more) {
            fetch(P, ldp, i0, I, vec_p, r0 + BK, pf);
            fetch(Q, ldq, j0, J, vec_q, r0 + BK, qf);
        }
#pragma unroll
        for (int r = 0; r < BK; ++r) {
            float4 p0 = *reinterpret_cast<const float4*>(&Ps[buf][r][ty * 4]);
            float4 p1 = *reinterpret_cast<const float4*>(&Ps[buf][r][64 + ty * 4]);
            float4 q0 = *reinterpret_cast<const float4*>(&Qs[buf][r][tx * 4]);
            float4 q1 = *reinterpret_cast<const float4*>(&Qs[buf][r][64 + tx * 4]);
            float pv[8] = {p0.x, p0.y, p0.z, p0.w, p1.x, p1.y, p1.z, p1.w};
            unsigned long long qq[4] = {pack2(q0.x, q0.y), pack2(q0.z, q0.w), pack2(q1.x, q1.y), pack2(q1.z, q1.w)};
#pragma unroll
            for (int a = 0; a < 8; ++a) {
                unsigned long long pp = pack2(pv[a], pv[a]);
#pragma unroll
                for (int b = 0; b < 4; ++b)
                    fma2(acc2[a][b], pp, qq[b]);
            }
        }
        if (more) {
            stash(Ps[buf ^ 1], pf);
            stash(Qs[buf ^ 1], qf);
        }
        __syncthreads();
        buf ^= 1;
    }

    float acc[8][8];
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b)
            unpack2(acc2[a][b], acc[a][2 * b], acc[a][2 * b + 1]);

    float sq = 0.f;
    const bool vec_c = (ldc % 4 == 0) && (((uintptr_t)C) % 16 == 0);
#pragma unroll
    for (int a = 0; a < 8; ++a) {
        int i = i0 + (a < 4 ? ty * 4 + a : 64 + ty * 4 + (a - 4));
        if (i >= I)
            continue;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            int j = j0 + h * 64 + tx * 4;
            float* dst = C + (int64_t)i * ldc + j;
            const float* v = &acc[a][h * 4];
            if (vec_c && j + 3 < J) {
                *reinterpret_cast<float4*>(dst) = make_float4(v[0], v[1], v[2], v[3]);
                sq += v[0] * v[0] + v[1] * v[1] + v[2] * v[2] + v[3] * v[3];
            } else {
#pragma unroll
                for (int b = 0; b < 4; ++b)
                    if (j + b < J) {
                        dst[b] = v[b];
                        sq += v[b] * v[b];
                    }
            }
        }
    }
    if (sq_sum)
        block_atomic_add((double)sq, sq_sum);
}

// gradient of one weight's alpha: g * dWq/dalpha + reg * dlambda/dalpha; lam += lambda(alpha)
__device__ __forceinline__ float weight_gradient(float g, float dq, float al, float reg, float& lam)
{
    const SoftTerms st = soft_terms(al);
    const float u = st.u;
    const float u2 = u * u, u4 = u2 * u2, u8 = u4 * u4, u16 = u8 * u8;
    lam += 1.0f - u16 * u4;
    const float u19 = u16 * u2 * u;
    const float dlam = -40.0f * u19 * (al > 0.f ? 1.f : (al < 0.f ? -1.f : 0.f)) * st.sp;
    return fmaf(g, dq, reg * dlam);
}

// grad = (2 / (M N)) (sum of the slices of D^T A) * dWq/dalpha + reg * dlambda/dalpha; alpha -= lr * grad when
// lr != 0; sum of lambda.  Thread 0 of block 0 turns the sum of squares into the mean.
// VEC: four weights per thread.  Few blocks, each ending in two atomics: those of a thousand blocks took longer than the
// rest (7.7 us for 960 x 320 weights).
template <bool VEC>
__global__ void __launch_bounds__(256) grad_finalize_kernel(const float* __restrict__ GP, int splits,
                                                            const float* __restrict__ DQ, float* __restrict__ alpha,
                                                            float* __restrict__ grad, double* __restrict__ loss,
                                                            int64_t total, float coef, double inv_mn, float reg, float lr)
{
    constexpr int V = VEC ? 4 : 1;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (blockIdx.x == 0 && threadIdx.x == 0)
        loss[0] *= inv_mn;
    float lam = 0.f;
    auto load = [](const float* p, float (&v)[V]) {
        if (VEC) {
            const float4 t = *reinterpret_cast<const float4*>(p);
            v[0] = t.x, v[V > 1 ? 1 : 0] = t.y, v[V > 2 ? 2 : 0] = t.z, v[V > 3 ? 3 : 0] = t.w;
        } else {
            v[0] = *p;
        }
    };
    auto store = [](float* p, const float (&v)[V]) {
        if (VEC)
            *reinterpret_cast<float4*>(p) = make_float4(v[0], v[V > 1 ? 1 : 0], v[V > 2 ? 2 : 0], v[V > 3 ? 3 : 0]);
        else
            *p = v[0];
    };
    for (int64_t i = V * ((int64_t)blockIdx.x * blockDim.x + threadIdx.x); i < total; i += V * ((int64_t)gridDim.x * blockDim.x)) {
        float g[V] = {}, dq[V], al[V], gr[V];
        load(DQ + i, dq);
        load(alpha + i, al);
#pragma unroll 4
        for (int z = 0; z < splits; ++z) {
            float t[V];
            load(GP + (int64_t)z * total + i, t);
#pragma unroll
            for (int v = 0; v < V; ++v)
                g[v] += t[v];
        }
#pragma unroll
        for (int v = 0; v < V; ++v) {
            gr[v] = weight_gradient(coef * g[v], dq[v], al[v], reg, lam);
            al[v] = al[v] - lr * gr[v];
        }
        store(grad + i, gr);
        if (lr != 0.f)
            store(alpha + i, al);
    }
    block_atomic_add((double)lam, loss + 1);
}

// ---- the gradient from S = A^T A, in double ----------------------------------------------------------------------
// sum D^2 = <E S, E> squares what cancels in D = A E^T, and descent makes E small along the rows' leading directions, where
// all of it cancels.  With S and E S in FP32 the loss of 4096 rows of rank 32 was up to 93 % off and negative at times; in
// double (products of FP32 numbers are exact) it is closer than the FP32 sum of squares.  The FP64 matrix instructions give
// 37 TFLOP/s and bound both kernels (70 % busy in gram_kernel, 42 % in gram_grad_kernel, whose blocks are short): 4096 x 320
// rows and 960 x 320 weights 43.8 us for the whole step; with S in TF32 products 29.5, the direct form 59.6.

// d += a b: 8 x 8 += (8 x 4) (4 x 8); lane l holds a[l / 4][l % 4], b[l % 4][l / 4], d[l / 4][2 (l % 4) + 0, 1]
__device__ __forceinline__ void mma_f64(double (&d)[2], double a, double b)
{
    asm("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};" : "+d"(d[0]), "+d"(d[1]) : "d"(a), "d"(b));
}
// 16 bytes to shared memory, zeros where there is nothing
__device__ __forceinline__ void copy16(uint32_t to, const void* from, bool there)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(to), "l"(from), "r"(there ? 16 : 0) : "memory");
}

// S: 64 x 64 tiles on and above the diagonal, each over slices of the rows (blockIdx.y); slice z of tile t goes to SP + (z *
// tiles + t) * 4096.  Stages of 32 rows; four warps have 32 x 32 outputs each, twice, for half of a stage's rows.
// Rows of shared memory are 72 floats: the 4 x 8 elements of a fragment lie in 32 banks.
constexpr int ST = 64, S_ROWS = 32, S_STAGES = 4, S_LD = ST + 8, S_STAGE = 2 * S_ROWS * S_LD;
constexpr int S_SMEM = S_STAGES * S_STAGE * 4;
static_assert(S_SMEM >= ST * ST * 8, "the second half's sums");
__global__ void __launch_bounds__(256, 2) gram_kernel(const float* __restrict__ A, int64_t M, int64_t K, int tiles, int64_t per,
                                                      double* __restrict__ SP)
{
    extern __shared__ __align__(16) float gsm[];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, half = warp >> 2;
    int ti = 0, left = (int)blockIdx.x;
    for (; left >= tiles - ti; ++ti)
        left -= tiles - ti;
    const int64_t i0 = (int64_t)ti * ST, j0 = (int64_t)(ti + left) * ST;
    const int64_t m_lo = (int64_t)blockIdx.y * per, m_hi = min(m_lo + per, M);
    const int wi = (warp & 1) * 32, wj = (warp >> 1 & 1) * 32;
    auto fetch = [&](int stage, int64_t m) {
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(gsm + stage * S_STAGE);
        const int row = t / 16, c = t % 16 * 4;
#pragma unroll
        for (int q = 0; q < S_ROWS; q += 16) {
            const int64_t at = m + row + q;
            const uint32_t to = dst + ((row + q) * S_LD + c) * 4;
            const bool in_i = at < m_hi && i0 + c < K, in_j = at < m_hi && j0 + c < K;
            copy16(to, in_i ? A + at * K + i0 + c : A, in_i);
            copy16(to + S_ROWS * S_LD * 4, in_j ? A + at * K + j0 + c : A, in_j);
        }
    };
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int stages = (int)((m_hi - m_lo + S_ROWS - 1) / S_ROWS);
#pragma unroll
    for (int s = 0; s < S_STAGES - 1; ++s) {
        if (s < stages)
            fetch(s, m_lo + s * S_ROWS);
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    double acc[4][4][2] = {};
    for (int s = 0; s < stages; ++s) {
        asm volatile("cp.async.wait_group %0;" ::"n"(S_STAGES - 2) : "memory");
        __syncthreads();                               // (and everybody is done with the stage that is filled next)
        if (s + S_STAGES - 1 < stages)
            fetch((s + S_STAGES - 1) % S_STAGES, m_lo + (int64_t)(s + S_STAGES - 1) * S_ROWS);
        asm volatile("cp.async.commit_group;" ::: "memory");
        const float* p = gsm + s % S_STAGES * S_STAGE + (half * (S_ROWS / 2) + (lane & 3)) * S_LD + (lane >> 2);
#pragma unroll
        for (int k = 0; k < S_ROWS / 2; k += 4) {
            double a[4], b[4];
#pragma unroll
            for (int f = 0; f < 4; ++f) {
                a[f] = (double)p[k * S_LD + wi + 8 * f];
                b[f] = (double)p[(S_ROWS + k) * S_LD + wj + 8 * f];
            }
#pragma unroll
            for (int x = 0; x < 4; ++x)
#pragma unroll
                for (int y = 0; y < 4; ++y)
                    mma_f64(acc[x][y], a[x], b[y]);
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    double* other = reinterpret_cast<double*>(gsm);
    double* out = SP + ((int64_t)blockIdx.y * gridDim.x + blockIdx.x) * (ST * ST);
    const int at = (wi + (lane >> 2)) * ST + wj + 2 * (lane & 3);
    if (half) {
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
            for (int y = 0; y < 4; ++y)
                *reinterpret_cast<double2*>(other + at + 8 * x * ST + 8 * y) = make_double2(acc[x][y][0], acc[x][y][1]);
    }
    __syncthreads();
    if (!half) {
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
            for (int y = 0; y < 4; ++y) {
                const double2 o = *reinterpret_cast<const double2*>(other + at + 8 * x * ST + 8 * y);
                *reinterpret_cast<double2*>(out + at + 8 * x * ST + 8 * y) = make_double2(acc[x][y][0] + o.x, acc[x][y][1] + o.y);
            }
    }
}

// S [K][K] = the slices added in their order, both triangles.  A block has 8 rows of a tile (blockIdx.y), a thread two columns.
__global__ void __launch_bounds__(256) gram_reduce_kernel(const double* __restrict__ SP, int slices, int tiles, double* __restrict__ S,
                                                          int64_t K)
{
    __shared__ double turn[8][ST + 1];
    asm volatile("griddepcontrol.wait;" ::: "memory");
    int ti = 0, left = (int)blockIdx.x;
    for (; left >= tiles - ti; ++ti)
        left -= tiles - ti;
    const int64_t i0 = (int64_t)ti * ST + blockIdx.y * 8, j0 = (int64_t)(ti + left) * ST;
    const int row = threadIdx.x / 32, c = threadIdx.x % 32 * 2;
    const double* p = SP + (int64_t)blockIdx.x * (ST * ST) + (blockIdx.y * 8 + row) * ST + c;
    double2 sum = make_double2(0.0, 0.0);
#pragma unroll 8
    for (int z = 0; z < slices; ++z) {
        const double2 v = *reinterpret_cast<const double2*>(p + (int64_t)z * gridDim.x * (ST * ST));
        sum.x += v.x, sum.y += v.y;
    }
    if (i0 + row < K && j0 + c < K)                    // (K is even)
        *reinterpret_cast<double2*>(S + (i0 + row) * K + j0 + c) = sum;
    turn[row][c] = sum.x, turn[row][c + 1] = sum.y;
    __syncthreads();
    const int col = threadIdx.x / 4, r = threadIdx.x % 4 * 2;
    if (left && j0 + col < K && i0 + r < K)
        *reinterpret_cast<double2*>(S + (j0 + col) * K + i0 + r) = make_double2(turn[r][col], turn[r + 1][col]);
}

// The rest of the step from S in one kernel: a ROWS x 64 tile of E S per block, reduced over all of K, then what
// grad_finalize_kernel does.  S is symmetric, so both operands are read as they lie.  64 reduction elements per stage, three
// stages of asynchronous copies; each of the eight warps has half of the columns and a quarter of a stage's elements, and
// the quarters' sums are added through shared memory.  Rows are padded so that a fragment's elements lie in different banks.
constexpr int GK = 64, GR = 64, G_STAGES = 3;
constexpr int GE_LD = GR + 4, GS_LD = GK + 4, GO_LD = GK + 2;      // floats of E, doubles of S, doubles of a sum
__host__ __device__ constexpr int gram_stage(int rows) { return rows * GE_LD * 4 + GR * GS_LD * 8; }      // bytes
constexpr int gram_smem(int rows)
{
    return G_STAGES * gram_stage(rows) > 4 * rows * GO_LD * 8 ? G_STAGES * gram_stage(rows) : 4 * rows * GO_LD * 8;
}
template <int ROWS>
__global__ void __launch_bounds__(256, 1) gram_grad_kernel(const float* __restrict__ E, const double* __restrict__ S,
                                                           const float* __restrict__ DQ, float* __restrict__ alpha,
                                                           float* __restrict__ grad, double* __restrict__ loss,
                                                           unsigned* __restrict__ ticket, int64_t N, int64_t K, double coef,
                                                           double inv_mn, float reg, float lr, int vec)
{
    constexpr int F = ROWS / 8;
    extern __shared__ __align__(16) uint8_t gsm8[];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, col0 = (warp & 1) * 32, part = warp >> 1;
    const int64_t n0 = (int64_t)blockIdx.x * ROWS, k0 = (int64_t)blockIdx.y * GK;
    auto fetch = [&](int stage, int64_t r0) {
        const uint32_t e = (uint32_t)__cvta_generic_to_shared(gsm8 + stage * gram_stage(ROWS)), s = e + ROWS * GE_LD * 4;
#pragma unroll
        for (int id = t; id < ROWS * (GR / 4); id += 256) {
            const int row = id / (GR / 4), c = id % (GR / 4) * 4;
            const bool there = n0 + row < N && r0 + c < K;
            copy16(e + (row * GE_LD + c) * 4, there ? E + (n0 + row) * K + r0 + c : E, there);
        }
#pragma unroll
        for (int id = t; id < GR * (GK / 2); id += 256) {
            const int row = id / (GK / 2), c = id % (GK / 2) * 2;
            const bool there = r0 + row < K && k0 + c < K;
            copy16(s + (row * GS_LD + c) * 8, there ? S + (r0 + row) * K + k0 + c : S, there);
        }
    };
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int stages = (int)((K + GR - 1) / GR);
#pragma unroll
    for (int i = 0; i < G_STAGES - 1; ++i) {
        if (i < stages)
            fetch(i, (int64_t)i * GR);
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    double acc[F][4][2] = {};
    for (int i = 0; i < stages; ++i) {
        asm volatile("cp.async.wait_group %0;" ::"n"(G_STAGES - 2) : "memory");
        __syncthreads();                               // (and everybody is done with the stage that is filled next)
        if (i + G_STAGES - 1 < stages)
            fetch((i + G_STAGES - 1) % G_STAGES, (int64_t)(i + G_STAGES - 1) * GR);
        asm volatile("cp.async.commit_group;" ::: "memory");
        const uint8_t* stage = gsm8 + i % G_STAGES * gram_stage(ROWS);
        const float* es = reinterpret_cast<const float*>(stage) + (lane >> 2) * GE_LD + part * (GR / 4) + (lane & 3);
        const double* ss = reinterpret_cast<const double*>(stage + ROWS * GE_LD * 4) + (part * (GR / 4) + (lane & 3)) * GS_LD +
                           col0 + (lane >> 2);
#pragma unroll
        for (int r = 0; r < GR / 4; r += 4) {
            double b[4];
#pragma unroll
            for (int y = 0; y < 4; ++y)
                b[y] = ss[r * GS_LD + 8 * y];
#pragma unroll
            for (int x = 0; x < F; ++x) {
                const double a = (double)es[8 * x * GE_LD + r];
#pragma unroll
                for (int y = 0; y < 4; ++y)
                    mma_f64(acc[x][y], a, b[y]);
            }
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    double* sums = reinterpret_cast<double*>(gsm8);
#pragma unroll
    for (int x = 0; x < F; ++x)
#pragma unroll
        for (int y = 0; y < 4; ++y)
            *reinterpret_cast<double2*>(sums + (part * ROWS + 8 * x + (lane >> 2)) * GO_LD + col0 + 8 * y + 2 * (lane & 3)) =
                make_double2(acc[x][y][0], acc[x][y][1]);
    __syncthreads();
    float lam = 0.f;
    double sq = 0.0;
    for (int id = t; id < ROWS * GK / 4; id += 256) {
        const int row = id / (GK / 4), c = id % (GK / 4) * 4;
        if (n0 + row >= N || k0 + c >= K)
            continue;
        const int64_t at = (n0 + row) * K + k0 + c;
        const float4 dq = *reinterpret_cast<const float4*>(DQ + at), e = *reinterpret_cast<const float4*>(E + at);
        float al[4], gr[4];
        if (vec) {
            const float4 v = *reinterpret_cast<const float4*>(alpha + at);
            al[0] = v.x, al[1] = v.y, al[2] = v.z, al[3] = v.w;
        } else {
#pragma unroll
            for (int v = 0; v < 4; ++v)
                al[v] = alpha[at + v];
        }
        const float d[4] = {dq.x, dq.y, dq.z, dq.w}, ev[4] = {e.x, e.y, e.z, e.w};
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            double g = 0.0;
#pragma unroll
            for (int q = 0; q < 4; ++q)
                g += sums[(q * ROWS + row) * GO_LD + c + v];
            sq = fma(g, (double)ev[v], sq);
            gr[v] = weight_gradient((float)(coef * g), d[v], al[v], reg, lam);
            al[v] = al[v] - lr * gr[v];
        }
        if (vec) {
            *reinterpret_cast<float4*>(grad + at) = make_float4(gr[0], gr[1], gr[2], gr[3]);
            if (lr != 0.f)
                *reinterpret_cast<float4*>(alpha + at) = make_float4(al[0], al[1], al[2], al[3]);
        } else {
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                grad[at + v] = gr[v];
                if (lr != 0.f)
                    alpha[at + v] = al[v];
            }
        }
    }
    block_atomic_add((double)lam, loss + 1);
    __syncthreads();                                   // (the helper's shared memory is used again)
    block_atomic_add(sq * inv_mn, loss);
    // a sum of squares: rounding must not leave it below zero (the block that comes last looks)
    if (t == 0) {
        __threadfence();
        if (atomicAdd(ticket, 1u) == gridDim.x * gridDim.y - 1) {
            __threadfence();
            if (__ldcg(loss) < 0.0)
                *loss = 0.0;
        }
    }
}

// D = sum over the reduction slices of the first contraction (fixed order), and the sum of its squares.
__global__ void __launch_bounds__(256) reduce_d_kernel(const float* __restrict__ DP, int splits, float* __restrict__ D,
                                                       int64_t total, int64_t N, int64_t N4, double* __restrict__ sq_sum)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    float sq = 0.f;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        if (i % N4 >= N)
            continue;                                   // padding columns are never written or read
        float v = 0.f;
        for (int z = 0; z < splits; ++z)
            v += DP[(int64_t)z * total + i];
        D[i] = v;
        sq += v * v;
    }
    block_atomic_add((double)sq, sq_sum);
}

// One thread per output byte: bit k of a row = (alpha >= 0), i.e. sigma(alpha) >= 0.5 rounds up.
__global__ void __launch_bounds__(256) harden_kernel(const float* __restrict__ alpha, int64_t N, int64_t K,
                                                     int64_t row_bytes, uint8_t* __restrict__ bits)
{
    int64_t total = N * row_bytes;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        int64_t n = i / row_bytes, b = i - n * row_bytes;
        uint32_t v = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            int64_t k = b * 8 + j;
            if (k < K && alpha[n * K + k] >= 0.f)
                v |= 1u << j;
        }
        bits[i] = (uint8_t)v;
    }
}

// Input rows of a convolution written out: row (b, oy, ox), column (c, r, s) in the weight's own [C][R][S]
// order, zero where the tap falls into the padding.  One thread per output element (writes coalesced).
__global__ void __launch_bounds__(256) unfold_kernel(const float* __restrict__ x, int C, int H, int W, int R, int S,
                                                     int pad, int stride, int Ho, int Wo, int64_t total,
                                                     float* __restrict__ rows)
{
    const int64_t K = (int64_t)C * R * S;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        int64_t m = i / K;
        int k = (int)(i - m * K);
        int s = k % S, r = (k / S) % R, c = k / (S * R);
        int ox = (int)(m % Wo), oy = (int)((m / Wo) % Ho);
        int64_t b = m / ((int64_t)Wo * Ho);
        int iy = oy * stride - pad + r, ix = ox * stride - pad + s;
        float v = 0.f;
        if (iy >= 0 && iy < H && ix >= 0 && ix < W)
            v = __ldg(x + ((b * C + c) * H + iy) * W + ix);
        rows[i] = v;
    }
}

int grid_for(int64_t total)
{
    int64_t blocks = (total + 255) / 256;
    return (int)(blocks < 1 ? 1 : (blocks > 148 * 16 ? 148 * 16 : blocks));
}

struct Plan {
    int64_t N4;
    int splits1;            // slices of K in the first contraction (1 = written straight to D)
    int64_t k_per_split;
    int splits;             // slices of M in the second contraction
    int64_t r_per_split;
    size_t off_E, off_DQ, off_D, off_DP, off_GP, bytes;
    // tensor-core route (K a multiple of 4): A^T and D^T with rows of Mp floats, slices of 32-wide blocks of M
    int64_t Mp;
    int kb_per_split_tc, splits_tc;
    int kb_per_split1_tc, splits1_tc;       // first contraction: sliced too when it has few output tiles
    size_t off_AT, off_DT;
    // with A^T A: 64-wide tiles per side, slices of M
    int gram, tiles_s, slices_s;
    int64_t rows_s;
    size_t off_SP, off_S, off_ticket;
};

// Rows of gram_grad_kernel's tiles: the fewest whose blocks all run at once, one per SM; with several rounds of them, 64.
int gram_tile_rows(int64_t N, int64_t K)
{
    for (int rows : {32, 40, 48})
        if ((N + rows - 1) / rows * ((K + 63) / 64) <= 148)
            return rows;
    return 64;
}

// As many slices of a reduction of length R as still fit into one wave of two resident blocks per SM (one more
// would add a second, nearly empty wave), each at least 128 long.
void slice(int64_t tiles, int64_t R, int* splits, int64_t* per)
{
    int64_t want = (2 * 148) / tiles;
    int64_t cap = (R + 127) / 128;
    int64_t s = want < cap ? want : cap;
    s = s < 1 ? 1 : (s > 64 ? 64 : s);
    *per = round_up((R + s - 1) / s, BK);
    *splits = (int)((R + *per - 1) / *per);
}

Plan make_plan(int64_t M, int64_t N, int64_t K)
{
    Plan p;
    p.N4 = round_up(N, 4);
    slice(((N + TILE - 1) / TILE) * ((K + TILE - 1) / TILE), M, &p.splits, &p.r_per_split);
    int64_t tiles1 = ((M + TILE - 1) / TILE) * ((N + TILE - 1) / TILE);
    p.splits1 = 1;
    p.k_per_split = K;
    if (tiles1 < 148)
        slice(tiles1, K, &p.splits1, &p.k_per_split);
    size_t o = 0;
    p.off_E = o;
    o += (size_t)round_up(N * K * 4, 256);
    p.off_DQ = o;
    o += (size_t)round_up(N * K * 4, 256);
    p.off_D = o;
    o += (size_t)round_up(M * p.N4 * 4, 256);
    {
        const int64_t tiles1 = ((M + 127) / 128) * ((N + tf32x3_columns(N) - 1) / tf32x3_columns(N));
        const int64_t kblocks = (K + 31) / 32;
        p.kb_per_split1_tc = (int)kblocks;
        p.splits1_tc = 1;
        if (tiles1 * 2 <= 148 && kblocks >= 16) {
            int64_t per = (kblocks + 148 / tiles1 - 1) / (148 / tiles1);
            per = per < 8 ? 8 : per;
            p.kb_per_split1_tc = (int)per;
            p.splits1_tc = (int)((kblocks + per - 1) / per);
        }
    }
    p.off_DP = o;
    {
        const int slices = p.splits1 > p.splits1_tc ? p.splits1 : p.splits1_tc;
        if (slices > 1)
            o += (size_t)round_up((int64_t)slices * M * p.N4 * 4, 256);
    }
    // second contraction on the tensor cores: one CTA per SM, so about 148 / tiles slices of at least 4 blocks
    p.Mp = round_up(M, 4);
    {
        const int64_t tiles2 = ((N + 127) / 128) * ((K + tf32x3_columns(K) - 1) / tf32x3_columns(K));
        const int64_t kblocks = (M + 31) / 32;
        int64_t want = 148 / tiles2;
        want = want < 1 ? 1 : (want > 64 ? 64 : want);
        int64_t per = (kblocks + want - 1) / want;
        per = per < 4 ? 4 : per;
        p.kb_per_split_tc = (int)per;
        p.splits_tc = (int)((kblocks + per - 1) / per);
    }
    p.off_GP = o;
    o += (size_t)round_up((int64_t)(p.splits > p.splits_tc ? p.splits : p.splits_tc) * N * K * 4, 256);
    p.off_AT = o;
    o += (size_t)round_up(K * p.Mp * 4, 256);
    p.off_DT = o;
    o += (size_t)round_up(N * p.Mp * 4, 256);
    {
        // E (A^T A) in place of (A E^T)^T A: half of M K^2 and N K^2 products in double instead of 2 M N K on the TF32 tensor
        // cores.  The slices of M with the shortest rounds of blocks (a stage of 32 rows 1.25 us, the sums' way out two of
        // them), the rounds of gram_grad_kernel's blocks over K (42 ns per row of a tile and 64 of K), against the direct
        // form's products (us so / direct, M x N x K: 4096 x 960 x 320 43.8 / 59.6, 8192 x 2560 x 320 88.4 / 195.5, 1024 x 512 x 256 22.9 /
        // 38.0, 139 x 1394 x 192 19.2 / 32.4, 2048 x 320 x 320 30.9 / 33.0, 8192 x 320 x 320 59.5 / 43.8, 2048 x 640 x 640 68.5 / 50.8,
        // 1024 x 2560 x 640 132 / 72.8, 94 x 19 x 1164, whose 19 blocks reduce 19 times 64 elements each, 50.3 / 35.0).
        p.tiles_s = (int)((K + ST - 1) / ST);
        const int64_t tiles = (int64_t)p.tiles_s * (p.tiles_s + 1) / 2, stages = (M + S_ROWS - 1) / S_ROWS;
        int64_t best = 0;
        for (int64_t want = 1; want <= 64 && want <= stages; ++want) {
            const int64_t each = (stages + want - 1) / want, slices = (stages + each - 1) / each;
            const int64_t cost = (tiles * slices + 147) / 148 * (each + 2);
            if (best == 0 || cost < best) {
                best = cost;
                p.slices_s = (int)slices;
                p.rows_s = each * S_ROWS;
            }
        }
        const int rows = gram_tile_rows(N, K);
        const int64_t rounds = ((N + rows - 1) / rows * p.tiles_s + 147) / 148;
        const double gram = 8.0 + 1.25 * (double)best + (double)rounds * (6.0 + 0.042 * rows * p.tiles_s);
        p.gram = K % 4 == 0 && gram <= 28.0 + 2.0 * (double)M * (double)N * (double)K / 83e6;
    }
    if (p.gram) {
        const int64_t tiles = (int64_t)p.tiles_s * (p.tiles_s + 1) / 2;
        p.off_SP = o;
        o += (size_t)round_up((int64_t)p.slices_s * tiles * ST * ST * 8, 256);
        p.off_S = o;
        o += (size_t)round_up(K * K * 8, 256);
    }
    p.off_ticket = o;
    o += 256;
    p.bytes = o;
    return p;
}

// most dynamic shared memory of a kernel, set once per device
template <typename Kernel>
bool allow_smem(Kernel kernel, int bytes, bool (&set)[64])
{
    static std::mutex mu;
    std::lock_guard<std::mutex> lock(mu);
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64)
        return false;
    if (!set[dev])
        set[dev] = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) == cudaSuccess;
    return set[dev];
}

template <int ROWS>
cudaError_t launch_gram_grad(const float* E, const double* S, const float* DQ, float* alpha, float* grad, double* loss, unsigned* ticket,
                             int64_t N, int64_t K, double coef, double inv_mn, float reg, float lr, cudaStream_t st)
{
    static bool set[64] = {};
    if (!allow_smem(gram_grad_kernel<ROWS>, gram_smem(ROWS), set))
        return cudaErrorUnknown;
    const int vec = (uintptr_t)alpha % 16 == 0 && (uintptr_t)grad % 16 == 0;
    return launch_overlapped(gram_grad_kernel<ROWS>, dim3((unsigned)((N + ROWS - 1) / ROWS), (unsigned)((K + GK - 1) / GK)), 256,
                             gram_smem(ROWS), st, E, S, DQ, alpha, grad, loss, ticket, N, K, coef, inv_mn, reg, lr, vec);
}

}  // namespace

size_t round_learn_workspace_bytes(int64_t M, int64_t N, int64_t K) { return make_plan(M, N, K).bytes; }

fpq_status launch_round_learn(const float* w, const float* scale, const QFormat& f, float* alpha, const float* a,
                              int64_t M, int64_t N, int64_t K, float reg, float lr, float* grad, double* loss,
                              void* workspace, cudaStream_t st)
{
    Plan p = make_plan(M, N, K);
    char* ws = (char*)workspace;
    float* E = (float*)(ws + p.off_E);
    float* DQ = (float*)(ws + p.off_DQ);
    float* D = (float*)(ws + p.off_D);
    float* DP = (float*)(ws + p.off_DP);
    float* GP = (float*)(ws + p.off_GP);
    int* status = status_word();
    if (!status)
        return FPQ_ERR_CUDA;
    const double inv_mn = 1.0 / ((double)M * (double)N);
    const float coef = (float)(2.0 * inv_mn);
    const bool tc = tf32x3_applies(a, K, E, K, M, N, K) && M <= (1 << 21) && N <= (1 << 21) && K <= (1 << 21);
    float* AT = (float*)(ws + p.off_AT);
    unsigned* ticket = (unsigned*)(ws + p.off_ticket);
    {
        const bool vec = K % 4 == 0 && (uintptr_t)w % 16 == 0 && (uintptr_t)alpha % 16 == 0;
        const int weight_blocks = grid_for(vec ? N * K / 4 : N * K);
        const int64_t blocks = weight_blocks + (tc && !p.gram ? ((M + 31) / 32) * ((K + 31) / 32) : 0);
        if (blocks > 0x7fffffff)
            return FPQ_ERR_SHAPE;
        if (launch_overlapped(vec ? prepare_kernel<true> : prepare_kernel<false>, dim3((unsigned)blocks), 256, 0, st, w, scale, f,
                              alpha, E, DQ, loss, N, K, weight_blocks, a, M, AT, p.Mp, ticket, status) != cudaSuccess)
            return FPQ_ERR_CUDA;
    }
    auto finalize = [&](int splits) {
        const bool vec = N * K % 4 == 0 && (uintptr_t)alpha % 16 == 0 && (uintptr_t)grad % 16 == 0;
        int blocks = grid_for(vec ? N * K / 4 : N * K);
        blocks = blocks > 2 * 148 ? 2 * 148 : blocks;
        return launch_overlapped(vec ? grad_finalize_kernel<true> : grad_finalize_kernel<false>, dim3(blocks), 256, 0, st, GP,
                                 splits, DQ, alpha, grad, loss, N * K, coef, inv_mn, reg, lr) == cudaSuccess
                   ? FPQ_OK
                   : FPQ_ERR_CUDA;
    };
    if (tc && p.gram) {
        double* SP = (double*)(ws + p.off_SP);
        double* S = (double*)(ws + p.off_S);
        const unsigned tiles = (unsigned)(p.tiles_s * (p.tiles_s + 1) / 2);
        static bool set[64] = {};
        if (!allow_smem(gram_kernel, S_SMEM, set) ||
            launch_overlapped(gram_kernel, dim3(tiles, (unsigned)p.slices_s), 256, S_SMEM, st, a, M, K, p.tiles_s, p.rows_s, SP) !=
                cudaSuccess ||
            launch_overlapped(gram_reduce_kernel, dim3(tiles, ST / 8), 256, 0, st, SP, p.slices_s, p.tiles_s, S, K) != cudaSuccess)
            return FPQ_ERR_CUDA;
        const int rows = gram_tile_rows(N, K);
        const auto launch = rows == 32 ? launch_gram_grad<32> : rows == 40 ? launch_gram_grad<40>
                            : rows == 48 ? launch_gram_grad<48> : launch_gram_grad<64>;
        return launch(E, S, DQ, alpha, grad, loss, ticket, N, K, 2.0 * inv_mn, inv_mn, reg, lr, st) == cudaSuccess ? FPQ_OK
                                                                                                                  : FPQ_ERR_CUDA;
    }
    if (tc) {
        // Both contractions on the tensor cores (three TF32 products per FP32 product): D^T = (A E^T)^T is written
        // transposed by the first one's epilogue, so that the second one, D^T A, again reduces over the contiguous
        // index of both operands (it reads A^T).
        float* DT = (float*)(ws + p.off_DT);
        fpq_status s1;
        if (p.splits1_tc == 1) {
            s1 = launch_tf32x3(a, K, E, K, M, N, K, p.kb_per_split1_tc, 1, DT, p.Mp, 0, loss, st);
        } else {
            // few output tiles and a long reduction: slices of it, added up in a fixed order, then transposed
            s1 = launch_tf32x3(a, K, E, K, M, N, K, p.kb_per_split1_tc, 0, DP, p.N4, M * p.N4, nullptr, st);
            if (s1 == FPQ_OK && (launch_overlapped(reduce_d_kernel, dim3(grid_for(M * p.N4)), 256, 0, st, DP, p.splits1_tc, D,
                                                   M * p.N4, N, p.N4, loss) != cudaSuccess ||
                                 launch_transpose(D, p.N4, M, N, DT, p.Mp, st) != cudaSuccess))
                return FPQ_ERR_CUDA;
        }
        if (s1 != FPQ_OK)
            return s1;
        s1 = launch_tf32x3(DT, p.Mp, AT, p.Mp, N, K, M, p.kb_per_split_tc, 0, GP, K, N * K, nullptr, st);
        if (s1 != FPQ_OK)
            return s1;
        return finalize(p.splits_tc);
    }
    dim3 g1((unsigned)((M + TILE - 1) / TILE), (unsigned)((N + TILE - 1) / TILE), (unsigned)p.splits1);
    if (p.splits1 == 1) {
        sgemm128<true><<<g1, 256, 0, st>>>(a, K, E, K, D, p.N4, (int)M, (int)N, K, K, loss);
    } else {
        sgemm128<true><<<g1, 256, 0, st>>>(a, K, E, K, DP, p.N4, (int)M, (int)N, K, p.k_per_split, nullptr);
        reduce_d_kernel<<<grid_for(M * p.N4), 256, 0, st>>>(DP, p.splits1, D, M * p.N4, N, p.N4, loss);
    }
    dim3 g2((unsigned)((N + TILE - 1) / TILE), (unsigned)((K + TILE - 1) / TILE), (unsigned)p.splits);
    sgemm128<false><<<g2, 256, 0, st>>>(D, p.N4, a, K, GP, K, (int)N, (int)K, M, p.r_per_split, nullptr);
    return cudaGetLastError() == cudaSuccess ? finalize(p.splits) : FPQ_ERR_CUDA;
}

fpq_status launch_round_harden(const float* alpha, int64_t N, int64_t K, uint8_t* bits, cudaStream_t st)
{
    int64_t row_bytes = (K + 7) / 8;
    if (N * row_bytes == 0)
        return FPQ_OK;
    harden_kernel<<<grid_for(N * row_bytes), 256, 0, st>>>(alpha, N, K, row_bytes, bits);
    return cudaGetLastError() == cudaSuccess ? FPQ_OK : FPQ_ERR_CUDA;
}

// C[i][j] = sum_r P[i][r] Q[j][r] (both operands with the reduction index contiguous), FP32 multiply-adds.
fpq_status launch_sgemm_nt(const float* P, int64_t ldp, const float* Q, int64_t ldq, float* C, int64_t ldc, int64_t I,
                           int64_t J, int64_t R, cudaStream_t st)
{
    if (I == 0 || J == 0)
        return FPQ_OK;
    dim3 g((unsigned)((I + TILE - 1) / TILE), (unsigned)((J + TILE - 1) / TILE), 1);
    sgemm128<true><<<g, 256, 0, st>>>(P, ldp, Q, ldq, C, ldc, (int)I, (int)J, R, R, nullptr);
    return cudaGetLastError() == cudaSuccess ? FPQ_OK : FPQ_ERR_CUDA;
}

fpq_status launch_unfold(const float* x, int B, int C, int H, int W, int R, int S, int pad, int stride, int Ho, int Wo,
                         float* rows, cudaStream_t st)
{
    int64_t total = (int64_t)B * Ho * Wo * C * R * S;
    if (total == 0)
        return FPQ_OK;
    unfold_kernel<<<grid_for(total), 256, 0, st>>>(x, C, H, W, R, S, pad, stride, Ho, Wo, total, rows);
    return cudaGetLastError() == cudaSuccess ? FPQ_OK : FPQ_ERR_CUDA;
}

}  // namespace fpq
