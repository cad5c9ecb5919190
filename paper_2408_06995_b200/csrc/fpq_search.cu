// Encoding and bias search of one tensor (Sec. V-A, Algorithm 1): the mean squared
// error of quantizing the tensor with every (encoding, clipping value) candidate, then
// the selection rule of Algorithm 1.
//
// Two forms, 444 candidates on 3.7 M elements: 658 us with every candidate applied to every element, 61 us sorted.  Small
// tensors: every candidate is applied to every element (search_mse_kernel), which is bound by instruction issue.  Large tensors: a
// candidate's quantizer is a staircase of at most 127 steps, so between two of its
// thresholds all elements round to the same grid value and only counts and sums of the
// elements matter.  The elements are sorted into bins a fraction of a step wide; a bin
// without a threshold contributes through its count and its sum, and only the bins that
// a threshold cuts (some 1 % of the elements per candidate) are looked at element by
// element.  What is left is bound by latency: a fixed 30 us (look-ups of 444 x 127 thresholds, tables, four launches)
// and some 10 us per million elements (shared-memory atomics of the sort, the walk over the cut bins).
// Counts and sums are integers, so they do not depend on the order in which
// the elements arrive, and everything derived from them is in double.
#include <mutex>

#include "fpq_common.cuh"
#include "fpq_kernels.h"

namespace fpq {

constexpr int SEARCH_THREADS = 256;
constexpr int SEARCH_PER_THREAD = 16;
constexpr int SEARCH_MAX_ENC = 8;
constexpr int SEARCH_MAX_CLIP = 256;
constexpr int SEARCH_MAX_CAND = 1024;
constexpr int SEARCH_CHUNK = SEARCH_THREADS * SEARCH_PER_THREAD;
constexpr int SEARCH_DIRECT_BLOCKS = 1184;     // most blocks of the direct form
// Sorted form: bins of |x| by exponent and the leading 10 mantissa bits, over the 16 binades below (and with) the
// one of the largest clipping value.  Steps are at least 2^-6 of the value, so a threshold cuts one bin in 16 or fewer.
constexpr int LOW_BITS = 13;                   // mantissa bits inside a bin
constexpr int BINS = 16 << (23 - LOW_BITS);
constexpr int SORT_THREADS = 1024;
constexpr int SORT_ROUND = 4 * SORT_THREADS;   // elements: four a thread
constexpr int SORT_FLIGHT = 4;                 // rounds whose loads are in flight together
constexpr int SORT_PIECE = 15 * SORT_ROUND;    // most elements sorted at a time
constexpr int SORT_LIST = 4096;                // elements outside the bins, handled one by one
constexpr int SORT_BLOCKS = 148;
constexpr int MAX_THRESHOLDS = 128;            // per candidate, padded
constexpr int SORT_SLOTS = SORT_PIECE + BINS;       // every bin padded to an even number
constexpr size_t SORT_SMEM = (size_t)BINS * 4 + SORT_SLOTS * 2 + SEARCH_MAX_CAND * sizeof(double);
constexpr int PACK_SHIFT = 37;                 // a bin's count above its sum of low bits
constexpr int64_t PACK_MAX = 1 << 24;          // ... which holds up to this many elements

struct SearchEnc {
    uint32_t cmax_bits;      // FP32 bit pattern of the format's own clipping value
    uint32_t ebmin_bits;     // exponent field (in place, << 23) of the smallest normal value
    uint32_t cbase;          // added to an exponent field: the rounding constant 1.5 * 2^(23 - m) of that binade
    float cmax;
    float spread;            // 2^(23 - m)
    float floor_c;           // 1.5 * 2^23 * (step of the smallest normal binade)
    int m, bias_bits;        // mantissa bits; (127 - B) << 23
    int thresholds;          // between neighbouring magnitudes: the number of positive codes
    float sub_step;          // step below the smallest normal value
};

struct SearchArgs {
    SearchEnc enc[SEARCH_MAX_ENC];
    int n_enc, n_clip;
    int64_t n;
    const float* x;
    const float* clip;
    int* status;
    double* partial;                 // [blocks][n_enc * n_clip]
    double* spread_sq;               // [blocks]: sum of squared distances from the bins' centres
    unsigned long long* bin_sum;     // [BINS]: sum of low bits, with the count above it
    uint32_t* threshold;             // [candidates][MAX_THRESHOLDS]: smallest |x| (bit pattern) above each threshold
    char4* nudge;                    // [candidates][32]: threshold k = 32 q + lane less midpoint * scale, component q
    ulonglong2* below;               // [BINS + MAX_THRESHOLDS]: what Prefix holds (search_prefix_kernel)
    ulonglong2* below_sq;            // [BINS + MAX_THRESHOLDS]
    unsigned* ticket;
    int blocks;
    int add_to;                      // tensors of more than PACK_MAX elements go in parts: not the first one
    double divide_by;                // the whole tensor's size in its last part, else 0
    double* mse;
    int32_t* best;
};

__device__ __forceinline__ uint64_t pack2(float lo, float hi)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ float2 unpack2(uint64_t v)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b)
{
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b)
{
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// Selection rule of Algorithm 1 (Sec. V-A), by one block: the candidate with the smallest error; among equal errors
// the one that comes first in encoding-major, candidate-minor order (the flat index).  The listing's start value for
// the best error is read as +infinity; a NaN error never wins.  Every thread takes the flat indices t, t + THREADS,
// ..., then the (error, index) pairs are reduced with the smaller index breaking ties.
template <int THREADS>
__device__ __forceinline__ void select_best(const double* mse, int ncand, int n_clip, int32_t* best)
{
    __shared__ double s_err[THREADS / 32];
    __shared__ int s_arg[THREADS / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double err = INFINITY;
    int arg = 0x7fffffff;                        // "nothing yet": loses every tie
#pragma unroll
    for (int u = 0; u < (SEARCH_MAX_CAND + THREADS - 1) / THREADS; ++u) {
        const int c = u * THREADS + threadIdx.x;
        const double e = c < ncand ? __ldcg(mse + c) : INFINITY;
        if (e < err) {                           // false for NaN; indices grow, so the first of equal errors stays
            err = e;
            arg = c;
        }
    }
    auto reduce = [&]() {
#pragma unroll
        for (int d = 16; d >= 1; d >>= 1) {
            const double oe = __shfl_xor_sync(0xffffffffu, err, d);
            const int oa = __shfl_xor_sync(0xffffffffu, arg, d);
            if (oe < err || (oe == err && oa < arg)) {
                err = oe;
                arg = oa;
            }
        }
    };
    reduce();
    if (lane == 0) {
        s_err[warp] = err;
        s_arg[warp] = arg;
    }
    __syncthreads();
    if (warp == 0) {
        err = lane < THREADS / 32 ? s_err[lane] : INFINITY;
        arg = lane < THREADS / 32 ? s_arg[lane] : 0x7fffffff;
        reduce();
        if (lane == 0) {
            const bool none = arg == 0x7fffffff;
            best[0] = none ? -1 : arg / n_clip;
            best[1] = none ? -1 : arg % n_clip;
        }
    }
}

// ---- direct form ---------------------------------------------------------------------------------
//
// Per candidate (i, j): scale = clip[j] / c(F_i) and 1 / scale, both FP32 divisions.
// Per element: t = |x| / scale, clipped at c.  With p = 2^(23 - m) * t, or 1.5 * 2^23 steps of the smallest normal
// binade where that is more, u = t + p has t's step as its last place, and u + (t - u) is t rounded to a multiple of
// that step (splitting a number at m + 1 bits by multiplication, after Dekker; the fixed p does the same where steps no
// longer shrink, and lies in the middle of its binade so that u - t has the same last place).  A tie may go either way,
// which leaves the error as it is.
// error = |x| - scale * q with one rounding (FMA).  The quantizer is odd, so signs drop out.
// Two elements per instruction but for the two comparisons: 5.5 issue slots per element and candidate where exponent
// arithmetic on the integer pipe took 9.
// blockIdx.y: the share of the candidates, so that a few thousand elements still fill the GPU.
__global__ void __launch_bounds__(SEARCH_THREADS) search_mse_kernel(const SearchArgs a)
{
    extern __shared__ double s_dyn[];
    const int ncand = a.n_enc * a.n_clip;
    const int c_lo = (int)((int64_t)blockIdx.y * ncand / gridDim.y), c_hi = (int)((int64_t)(blockIdx.y + 1) * ncand / gridDim.y);
    const int nc = c_hi - c_lo;
    double* wsum = s_dyn;                                                   // [8 warps][nc]
    float* s_rinv = reinterpret_cast<float*>(wsum + (SEARCH_THREADS / 32) * nc);   // [nc]
    float* s_scale = s_rinv + nc;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int c = threadIdx.x; c < nc; c += SEARCH_THREADS) {
        const int i = (c_lo + c) / a.n_clip, j = c_lo + c - i * a.n_clip;
        const float scale = __fdiv_rn(__ldg(a.clip + j), a.enc[i].cmax);
        s_scale[c] = scale;
        s_rinv[c] = __fdiv_rn(1.0f, scale);
    }
    for (int c = threadIdx.x; c < (SEARCH_THREADS / 32) * nc; c += SEARCH_THREADS)
        wsum[c] = 0.0;
    __syncthreads();

    bool nan = false;
    const int64_t nchunks = (a.n + SEARCH_CHUNK - 1) / SEARCH_CHUNK;
    for (int64_t ch = blockIdx.x; ch < nchunks; ch += gridDim.x) {
        float ax[SEARCH_PER_THREAD];
        const int64_t base = ch * SEARCH_CHUNK;
        if (base + SEARCH_CHUNK <= a.n && ((uintptr_t)a.x % 16) == 0) {
#pragma unroll
            for (int v = 0; v < SEARCH_PER_THREAD / 4; ++v) {
                const float4 f = __ldg(reinterpret_cast<const float4*>(a.x + base) + v * SEARCH_THREADS + threadIdx.x);
                ax[4 * v] = fabsf(f.x);
                ax[4 * v + 1] = fabsf(f.y);
                ax[4 * v + 2] = fabsf(f.z);
                ax[4 * v + 3] = fabsf(f.w);
            }
        } else {
#pragma unroll
            for (int v = 0; v < SEARCH_PER_THREAD; ++v) {
                const int64_t k = base + (int64_t)v * SEARCH_THREADS + threadIdx.x;
                ax[v] = k < a.n ? fabsf(__ldg(a.x + k)) : 0.f;      // a zero adds no error to any candidate
            }
        }
        uint64_t ax2[SEARCH_PER_THREAD / 2];
#pragma unroll
        for (int v = 0; v < SEARCH_PER_THREAD; ++v)
            nan |= __float_as_uint(ax[v]) > 0x7f800000u;
#pragma unroll
        for (int v = 0; v < SEARCH_PER_THREAD / 2; ++v)
            ax2[v] = pack2(ax[2 * v], ax[2 * v + 1]);

        const uint64_t minus1 = pack2(-1.f, -1.f);
        int c = 0;
        for (int i = c_lo / a.n_clip; c < nc; ++i) {
            const float cmax = a.enc[i].cmax, floor_c = a.enc[i].floor_c;
            const uint64_t spread = pack2(a.enc[i].spread, a.enc[i].spread);
            const int last = min(nc, (i + 1) * a.n_clip - c_lo);
            for (; c < last; ++c) {
                const uint64_t rinv = pack2(s_rinv[c], s_rinv[c]), nscale = pack2(-s_scale[c], -s_scale[c]);
                uint64_t acc2 = 0;
#pragma unroll
                for (int v = 0; v < SEARCH_PER_THREAD / 2; ++v) {
                    float2 t = unpack2(mul2(ax2[v], rinv));
                    const uint64_t t2 = pack2(fminf(t.x, cmax), fminf(t.y, cmax));
                    const float2 p = unpack2(mul2(t2, spread));
                    const uint64_t u = add2(t2, pack2(fmaxf(p.x, floor_c), fmaxf(p.y, floor_c)));
                    const uint64_t q = add2(u, fma2(u, minus1, t2));
                    const uint64_t err = fma2(nscale, q, ax2[v]);
                    acc2 = fma2(err, err, acc2);
                }
                const float2 s = unpack2(acc2);
                float acc = s.x + s.y;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1)
                    acc += __shfl_xor_sync(0xffffffffu, acc, o);
                if (lane == 0)
                    wsum[warp * nc + c] += (double)acc;
            }
        }
    }
    __syncthreads();
    for (int c = threadIdx.x; c < nc; c += SEARCH_THREADS) {
        double s = 0.0;
#pragma unroll
        for (int w = 0; w < SEARCH_THREADS / 32; ++w)
            s += wsum[w * nc + c];
        a.partial[(int64_t)blockIdx.x * ncand + c_lo + c] = s;
    }
    if (nan)
        flag_status(a.status, FPQ_ERR_NAN_INPUT);
}

// Block partial sums -> mse (in a fixed order: the same whatever the timing), then the selection.  One block, whose threads
// share a candidate's blocks as far as there are fewer candidates than threads, and add up their shares pairwise: a thread
// that adds all 1184 blocks waits for one load after the other (3.3 M elements, 4 candidates: 64.9 us, 12.4 so).
__global__ void __launch_bounds__(1024) search_finish_kernel(const SearchArgs a)
{
    __shared__ double part[1024];
    const int t = threadIdx.x, ncand = a.n_enc * a.n_clip;
    int shares = min(1024 / ncand, (a.blocks + 7) / 8);
    const int share = t / ncand, c = t - share * ncand;
    double s = 0.0;
    if (share < shares) {
        // (eight loads in flight, whatever the count)
        for (int b = share; b < a.blocks; b += 8 * shares) {
            double v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u)
                v[u] = b + u * shares < a.blocks ? a.partial[(int64_t)(b + u * shares) * ncand + c] : 0.0;
#pragma unroll
            for (int u = 0; u < 8; ++u)
                s += v[u];
        }
    }
    part[t] = s;
    while (shares > 1) {
        const int half = (shares + 1) / 2;
        __syncthreads();
        if (share < shares - half)
            part[t] += part[t + half * ncand];
        shares = half;
    }
    __syncthreads();
    if (t < ncand)
        a.mse[t] = a.n > 0 ? part[t] / (double)a.n : 0.0;
    __syncthreads();
    select_best<1024>(a.mse, ncand, a.n_clip, a.best);
}

// ---- sorted form ---------------------------------------------------------------------------------

// First key of the binned range: the bins end with the binade of the largest clipping value (above it no candidate
// has a threshold).  Every warp works it out for itself.
__device__ __forceinline__ int first_key(const SearchArgs& a, int lane)
{
    uint32_t top = 0;
    for (int j = lane; j < a.n_clip; j += 32)
        top = max(top, __float_as_uint(__ldg(a.clip + j)));
    top = __reduce_max_sync(0xffffffffu, top);
    return (int)(((top >> 23) + 1) << (23 - LOW_BITS)) - BINS;
}

// magnitude of code k of an encoding and the midpoint between codes k and k + 1 (both FP32 numbers)
__device__ __forceinline__ float code_magnitude(const SearchEnc& e, int k)
{
    return k >= (1 << e.m) ? __uint_as_float(((uint32_t)k << (23 - e.m)) + e.bias_bits) : (float)k * e.sub_step;
}
__device__ __forceinline__ float code_midpoint(const SearchEnc& e, int k)
{
    return k >= (1 << e.m) ? __uint_as_float(((uint32_t)k << (23 - e.m)) + (1u << (22 - e.m)) + e.bias_bits)
                           : ((float)k + 0.5f) * e.sub_step;
}

__device__ __forceinline__ void candidate_scale(const SearchArgs& a, int c, int& i, float& scale)
{
    i = c / a.n_clip;
    scale = __fdiv_rn(__ldg(a.clip + (c - i * a.n_clip)), a.enc[i].cmax);
}

// Thresholds of all candidates in the domain of |x|, and empty bins.  x * (1 / scale) rounded to FP32 grows with x, so
// "x rounds to code k + 1 or above" is x >= threshold; it is found from midpoint * scale by stepping single floats.
__global__ void __launch_bounds__(256) search_tables_kernel(const SearchArgs a)
{
    const int id = blockIdx.x * 256 + threadIdx.x;
    asm volatile("griddepcontrol.launch_dependents;");
    if (id == 0)
        *a.ticket = 0;
    for (int b = id; b < BINS; b += gridDim.x * 256) {
        a.bin_sum[b] = 0;
    }
    const int c = id / MAX_THRESHOLDS, k = id % MAX_THRESHOLDS;
    if (c >= a.n_enc * a.n_clip)
        return;
    int i;
    float scale;
    candidate_scale(a, c, i, scale);
    uint32_t at = 0xffffffffu;                                     // no such threshold
    if (k < a.enc[i].thresholds) {
        const float rinv = __fdiv_rn(1.0f, scale), mid = code_midpoint(a.enc[i], k);
        const bool tie_up = k & 1;                                 // ties go to the even code
        auto above = [&](uint32_t bits) {
            const float t = __fmul_rn(__uint_as_float(bits), rinv);
            return t > mid || (tie_up && t == mid);
        };
        at = __float_as_uint(__fmul_rn(mid, scale));
        for (int s = 0; s < 8 && at > 1 && above(at - 1); ++s)
            --at;
        for (int s = 0; s < 8 && at < 0x7f800000u && !above(at); ++s)
            ++at;
    }
    a.threshold[id] = at;
    reinterpret_cast<signed char*>(a.nudge + c * 32 + k % 32)[k / 32] =
        k < a.enc[i].thresholds ? (signed char)(at - __float_as_uint(__fmul_rn(code_midpoint(a.enc[i], k), scale))) : 0;
}

// Sums over a range of bins, in units of the last place of the lowest binade (so that all elements are whole numbers
// below 2^40): n elements, their sum x, and sq = sum over the bins of (2 c * (sum of x - c) + n * c^2), c a bin's centre,
// which is the sum of the squares less the sum of the squared distances from the centres.  Exact.
struct Prefix {
    unsigned long long n;
    unsigned long long x;            // n <= PACK_MAX elements below 2^39 each: below 2^63
    unsigned __int128 sq;
};
__device__ __forceinline__ Prefix operator+(const Prefix& a, const Prefix& b) { return {a.n + b.n, a.x + b.x, a.sq + b.sq}; }
__device__ __forceinline__ unsigned __int128 wide(unsigned long long lo, unsigned long long hi)
{
    return ((unsigned __int128)hi << 64) | lo;
}
__device__ __forceinline__ double to_double(__int128 v)
{
    const bool neg = v < 0;
    const unsigned __int128 u = neg ? -(unsigned __int128)v : (unsigned __int128)v;
    const double d = fma((double)(unsigned long long)(u >> 64), 18446744073709551616.0, (double)(unsigned long long)u);
    return neg ? -d : d;
}
__device__ __forceinline__ int lowest_exponent(int base) { return max(base >> (23 - LOW_BITS), 1); }
__device__ __forceinline__ Prefix bin_sums(const SearchArgs& a, int b, int base, int e0)
{
    const unsigned long long v = __ldcg(a.bin_sum + b);
    const unsigned long long cnt = v >> PACK_SHIFT, low = v & ((1ull << PACK_SHIFT) - 1);
    if (cnt == 0)
        return {0, 0, 0};
    const uint32_t key = (uint32_t)(b + base);
    const int e = (int)(key >> (23 - LOW_BITS));
    const int up = max(e, 1) - e0;
    const unsigned long long edge =
        (unsigned long long)((key & ((1u << (23 - LOW_BITS)) - 1)) << LOW_BITS | (e ? 1u << 23 : 0u)) << up;
    const unsigned long long centre = edge + ((1ull << (LOW_BITS - 1)) << up);
    Prefix r;
    r.n = cnt;
    r.x = cnt * edge + (low << up);
    // 2 c (x - n c) + n c^2 = c (2 x - n c)
    r.sq = (unsigned __int128)centre * r.x * 2 - (unsigned __int128)centre * centre * cnt;
    return r;
}

// Exclusive prefix sum over the block's threads; s_warp: 32 words of shared memory.  (Every thread has to have left an
// earlier scan before the next one: there is a barrier between them.)
__device__ __forceinline__ uint32_t block_scan(uint32_t mine, uint32_t* s_warp, uint32_t& total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
        incl += lane >= o ? t : 0u;
    }
    if (lane == 31)
        s_warp[warp] = incl;
    __syncthreads();
    uint32_t w = s_warp[lane], wsum = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, wsum, o);
        wsum += lane >= o ? t : 0u;
    }
    total = __shfl_sync(0xffffffffu, wsum, 31);
    return __shfl_sync(0xffffffffu, wsum - w, warp) + incl - mine;
}

// Sorts the block's elements by bin in shared memory, adds the bins' counts and sums to the global table and works
// out, per candidate, what its thresholds change: in a bin that a threshold cuts, the elements above it take the next
// grid value instead of the one of the bin's lower edge (which is what search_eval_kernel gives to the whole bin).
// The change is -2 D * sum(x - mu) over those elements, D the step and mu the midpoint, both times the scale.
// blockIdx.y: the share of the candidates (every share sorts for itself).
// What bounds it: instructions (0.7 issued per cycle and scheduler), more than half of them in the candidates' walk below.
// So a bin's slots start at an even place and are padded with zeros, and a threshold walks its bin two elements to a
// register and two registers a step; the thresholds themselves are worked out again (a multiplication and a stored offset
// in ulps) rather than read, 57 instead of 227 KB per block; a warp's candidates are neighbours, so that it seldom changes
// the encoding; and a piece may have 61440 elements, because half of the walk does not depend on them.  3.7 M elements,
// 444 candidates, whole search: 69.8 -> 60.4 us (walk 73 K -> 56 K of the block's 105 K cycles); 1 M: 47.5 -> 41.2 us;
// 262144: 35.3 -> 33.6 us.  (Four elements a step from slots in fours: 59.2 us there, but more pieces above 4.2 M.)
static_assert(BINS == 16 * SORT_THREADS, "four 16-byte words of a thread");
static_assert(4 * SORT_PIECE / SORT_ROUND <= 64, "one bit per element of a thread");
static_assert(SORT_PIECE < 65536 && SORT_SLOTS / 2 < 65536, "a bin's word");
static_assert(SORT_SLOTS * 2 >= SORT_LIST * 4 + SORT_THREADS * 8, "the list lies where the elements will");
static_assert(SEARCH_MAX_CAND <= 32 * (SORT_THREADS / 32), "a lane per candidate of its warp");
__global__ void __launch_bounds__(SORT_THREADS, 1) search_sort_kernel(const SearchArgs a)
{
    extern __shared__ __align__(16) uint8_t s_raw[];
    uint32_t* words = reinterpret_cast<uint32_t*>(s_raw);                            // start / 2 << 16 | count
    uint16_t* sorted = reinterpret_cast<uint16_t*>(s_raw + BINS * 4);                // low bits, bin after bin
    double* acc = reinterpret_cast<double*>(s_raw + BINS * 4 + SORT_SLOTS * 2);      // [candidates]
    float* list = reinterpret_cast<float*>(sorted);                                  // (before there are sorted elements)
    double* s_part = reinterpret_cast<double*>(list + SORT_LIST);
    __shared__ uint32_t s_warp[32];
    __shared__ double s_red[32];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int ncand = a.n_enc * a.n_clip;
    const int c_lo = (int)((int64_t)blockIdx.y * ncand / gridDim.y), c_hi = (int)((int64_t)(blockIdx.y + 1) * ncand / gridDim.y);

    // four consecutive elements' magnitudes; 0 (which no candidate changes) past the end
    const bool vec = ((uintptr_t)a.x % 16) == 0;
    auto load4 = [&](int64_t k, int64_t end, uint32_t (&v)[4]) {
        if (vec && k + 4 <= end) {
            const uint4 f = __ldg(reinterpret_cast<const uint4*>(a.x + k));
            v[0] = f.x, v[1] = f.y, v[2] = f.z, v[3] = f.w;
        } else {
#pragma unroll
            for (int q = 0; q < 4; ++q)
                v[q] = k + q < end ? __float_as_uint(__ldg(a.x + k + q)) : 0u;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
            v[q] &= 0x7fffffffu;
    };

    const int64_t share = round_up((a.n + gridDim.x - 1) / gridDim.x, 4);
    const int64_t lo = min((int64_t)blockIdx.x * share, a.n), hi = min(lo + share, a.n);
    const int pieces = (int)((hi - lo + SORT_PIECE - 1) / SORT_PIECE);
    const int base = first_key(a, lane);
    for (int c = tid; c < c_hi - c_lo; c += SORT_THREADS)
        acc[c] = 0.0;
    double spread_sq = 0.0;
    bool nan = false;
    for (int piece = 0; piece < pieces; ++piece) {
        const int64_t p_lo = lo + round_up((hi - lo) * piece / pieces, 4);
        const int64_t p_hi = piece + 1 == pieces ? hi : lo + round_up((hi - lo) * (piece + 1) / pieces, 4);
        uint32_t v[SORT_FLIGHT][4];
        auto load = [&](int64_t k) {
#pragma unroll
            for (int f = 0; f < SORT_FLIGHT; ++f)
                load4(k + f * SORT_ROUND + 4 * tid, p_hi, v[f]);
        };
        load(p_lo);
#pragma unroll
        for (int w = 0; w < BINS / 4; w += SORT_THREADS)
            reinterpret_cast<uint4*>(words)[w + tid] = make_uint4(0, 0, 0, 0);
        __syncthreads();

        // counts per bin; one bit of `outside` per element of this thread that has none
        uint64_t outside = 0;
        for (int64_t k = p_lo; k < p_hi; k += SORT_FLIGHT * SORT_ROUND) {
            if (k > p_lo)
                load(k);
            const int first = (int)(k - p_lo) / SORT_ROUND * 4;
#pragma unroll
            for (int f = 0; f < SORT_FLIGHT; ++f)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const uint32_t bits = v[f][q];
                    const int key = (int)(bits >> LOW_BITS) - base;
                    if ((unsigned)key < (unsigned)BINS && bits != 0) {
                        atomicAdd(words + key, 1u);
                        const float centre = __uint_as_float((bits & ~((1u << LOW_BITS) - 1)) | (1u << (LOW_BITS - 1)));
                        const double d = (double)(__uint_as_float(bits) - centre);
                        spread_sq = fma(d, d, spread_sq);
                    } else if (bits != 0) {
                        outside |= 1ull << (first + 4 * f + q);
                    }
                }
        }
        if (__syncthreads_or(outside != 0)) {
            // elements below or above the bins (and infinities and NaNs): every thread puts its own into the list, in
            // thread order, then applies its candidates to the whole list; more than the list holds: in several turns
            uint32_t total, at = block_scan((uint32_t)__popcll(outside), s_warp, total);
            for (uint32_t first = 0; first < total; first += SORT_LIST) {
                while (outside && at < first + SORT_LIST) {
                    const int e = __ffsll((long long)outside) - 1;
                    outside &= outside - 1;
                    const uint32_t bits = __float_as_uint(__ldg(a.x + p_lo + (int64_t)(e >> 2) * SORT_ROUND + 4 * tid + (e & 3)));
                    nan |= (bits & 0x7fffffffu) > 0x7f800000u;
                    list[at++ - first] = __uint_as_float(bits & 0x7fffffffu);
                }
                __syncthreads();
                const uint32_t cnt = min(total - first, (uint32_t)SORT_LIST);
                // (a tensor with one huge entry has most of its elements here: all threads take part, in slices of the
                // list, and a candidate that rounds all of it to zero takes the sum of the squares)
                uint32_t most = 0;
                double squares = 0.0;
                for (uint32_t e = tid; e < cnt; e += SORT_THREADS) {
                    const double ax = (double)list[e];
                    most = max(most, __float_as_uint(list[e]));
                    squares = fma(ax, ax, squares);
                }
                most = __reduce_max_sync(0xffffffffu, most);
#pragma unroll
                for (int o = 16; o > 0; o >>= 1)
                    squares += __shfl_xor_sync(0xffffffffu, squares, o);
                if (lane == 0) {
                    s_warp[warp] = most;
                    s_red[warp] = squares;
                }
                __syncthreads();
                most = __reduce_max_sync(0xffffffffu, s_warp[lane]);
                squares = s_red[lane];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1)
                    squares += __shfl_xor_sync(0xffffffffu, squares, o);
                asm volatile("griddepcontrol.wait;" ::: "memory");     // (the thresholds)
                const int width = min((int)round_up(c_hi - c_lo, 32), SORT_THREADS), slices = SORT_THREADS / width;
                const int slice = tid / width, lane_c = tid - slice * width;
                for (int c0 = c_lo; c0 < c_hi; c0 += width) {
                    const int c = c0 + lane_c;
                    double s = 0.0;
                    if (slice < slices && c < c_hi && most < __ldcg(a.threshold + c * MAX_THRESHOLDS)) {
                        s = slice == 0 ? squares : 0.0;
                    } else if (slice < slices && c < c_hi) {
                        int i;
                        float scale;
                        candidate_scale(a, c, i, scale);
                        const float rinv = __fdiv_rn(1.0f, scale);
                        // (a slice is a run of the list; sixteen squares at a time are added up in FP32, as above)
                        const uint32_t e1 = cnt * (slice + 1) / slices;
                        for (uint32_t e0 = cnt * slice / slices; e0 < e1; e0 += 16) {
                            float part = 0.f;
#pragma unroll
                            for (uint32_t q = 0; q < 16; ++q) {
                                const float ax = e0 + q < e1 ? list[e0 + q] : 0.f;
                                const float t = __fmul_rn(ax, rinv);
                                const uint32_t tb = min(__float_as_uint(t), a.enc[i].cmax_bits);
                                const float big = __uint_as_float(max(tb & 0x7f800000u, a.enc[i].ebmin_bits) + a.enc[i].cbase);
                                const float g = __fsub_rn(__fadd_rn(__uint_as_float(tb), big), big);
                                const float err = __fmaf_rn(-scale, g, ax);
                                part = __fmaf_rn(err, err, part);
                            }
                            s += (double)part;
                        }
                    }
                    s_part[tid] = s;
                    __syncthreads();
                    if (slice == 0 && c < c_hi) {
                        for (int k = 1; k < slices; ++k)
                            s += s_part[k * width + lane_c];
                        acc[c - c_lo] += s;
                    }
                    __syncthreads();
                }
            }
        }

        // starts, in place of the counts, which the elements' placing counts up again; zeros in all slots
        {
            uint4* mine = reinterpret_cast<uint4*>(words) + warp * 128 + lane;
            auto padded = [](uint32_t count) { return (count + 1) & ~1u; };
            uint32_t below[4], run = 0;
            uint4 t[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                t[q] = mine[32 * q];
                const uint32_t sum = padded(t[q].x) + padded(t[q].y) + padded(t[q].z) + padded(t[q].w);
                uint32_t incl = sum;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t u = __shfl_up_sync(0xffffffffu, incl, o);
                    incl += lane >= o ? u : 0u;
                }
                below[q] = run + incl - sum;
                run += __shfl_sync(0xffffffffu, incl, 31);
            }
            if (lane == 0)
                s_warp[warp] = run;
            __syncthreads();
            const uint32_t of_warp = s_warp[lane], total = __reduce_add_sync(0xffffffffu, of_warp);
            const uint32_t before = __reduce_add_sync(0xffffffffu, lane < warp ? of_warp : 0u);
            uint32_t at = 0;
            auto place = [&](uint32_t& word) {
                const uint32_t count = word;
                word = at << 15;
                at += padded(count);
            };
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                at = before + below[q];
                place(t[q].x), place(t[q].y), place(t[q].z), place(t[q].w);
                mine[32 * q] = t[q];
            }
            for (uint32_t w = tid; w * 8 < total; w += SORT_THREADS)
                reinterpret_cast<uint4*>(sorted)[w] = make_uint4(0, 0, 0, 0);
        }
        __syncthreads();

        // low bits to their places
        for (int64_t k = p_lo; k < p_hi; k += SORT_FLIGHT * SORT_ROUND) {
            load(k);
#pragma unroll
            for (int f = 0; f < SORT_FLIGHT; ++f)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const uint32_t bits = v[f][q];
                    const int key = (int)(bits >> LOW_BITS) - base;
                    if ((unsigned)key < (unsigned)BINS && bits != 0) {
                        const uint32_t word = atomicAdd(words + key, 1u);
                        sorted[(word >> 16) * 2 + (word & 0xffffu)] = (uint16_t)(bits & ((1u << LOW_BITS) - 1));
                    }
                }
        }
        __syncthreads();

        // the block's share of the global table (which the kernel in front empties)
        asm volatile("griddepcontrol.wait;" ::: "memory");
        // (every block starts elsewhere: atomics of many blocks on one bin wait for each other)
        for (int turn = blockIdx.y == 0 ? 0 : BINS / SORT_THREADS; turn < BINS / SORT_THREADS; ++turn) {
            const int b = (turn + (int)blockIdx.x) % (BINS / SORT_THREADS) * SORT_THREADS + tid;
            const uint32_t word = words[b], count = word & 0xffffu;
            if (count) {
                const uint32_t* at = reinterpret_cast<const uint32_t*>(sorted) + (word >> 16);
                uint32_t sum = 0;                               // (below 2^29)
#pragma unroll 1
                for (uint32_t e = 0; e < count; e += 2) {
                    const uint32_t l = *at++;
                    sum += (l & 0xffffu) + (l >> 16);
                }
                atomicAdd(a.bin_sum + b, sum | ((unsigned long long)count << PACK_SHIFT));
            }
        }

        // What the thresholds change: a warp per candidate, four thresholds per lane (their look-ups in flight
        // together).  x - mu = (low bits of x - low bits of the threshold) * ulp - (mu - threshold), the last difference
        // with a single rounding, so FP32 is enough.
        // Lane j has the encoding, the scale and the result of the warp's j-th candidate.  (Neighbouring candidates: most
        // warps stay with one encoding.)
        const int per_warp = (c_hi - c_lo + SORT_THREADS / 32 - 1) / (SORT_THREADS / 32);
        const int c_first = c_lo + warp * per_warp, count_c = min(per_warp, c_hi - c_first);
        int known = -1, its_enc = 0;
        float its_scale = 0.f, its_sum = 0.f, mid[4], step[4];
        if (lane < count_c)
            candidate_scale(a, c_first + lane, its_enc, its_scale);
        const char4* nudges = a.nudge + c_first * 32 + lane;
        char4 next = count_c > 0 ? __ldcg(nudges) : char4{};
        for (int turn = 0; turn < count_c; ++turn) {
            const char4 nudge = next;
            nudges += 32;
            if (turn + 1 < count_c)
                next = __ldcg(nudges);
            const int i = __shfl_sync(0xffffffffu, its_enc, turn);
            const float scale = __shfl_sync(0xffffffffu, its_scale, turn);
            if (i != known) {
                known = i;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int k = 32 * q + lane;
                    mid[q] = k >= a.enc[i].thresholds ? INFINITY : code_midpoint(a.enc[i], k);
                    step[q] = k >= a.enc[i].thresholds ? 0.f
                              : __uint_as_float((uint32_t)((max(k >> a.enc[i].m, 1) - a.enc[i].m) << 23) + a.enc[i].bias_bits);
                }
            }
            uint32_t at[4], span[4];
            const int off[4] = {nudge.x, nudge.y, nudge.z, nudge.w};
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                at[q] = __float_as_uint(__fmul_rn(mid[q], scale)) + (uint32_t)off[q];
                const int key = (int)(at[q] >> LOW_BITS) - base;
                // (a threshold on a bin's edge has the whole bin above it; one that is not there, at infinity, has no bin)
                const bool cuts = (unsigned)key < (unsigned)BINS && (at[q] & ((1u << LOW_BITS) - 1)) != 0;
                span[q] = cuts ? words[key] : 0u;
            }
            float s = 0.f;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint32_t count = span[q] & 0xffffu;
                if (count) {
                    const uint32_t less = ((1u - (at[q] & ((1u << LOW_BITS) - 1))) & 0xffffu) * 0x10001u;
                    const uint32_t* p = reinterpret_cast<const uint32_t*>(sorted) + (span[q] >> 16);
                    const uint32_t* const end = p + (count + 1) / 2;
                    uint32_t hits = 0, over = 0;                // (hits: two halves)
#pragma unroll 1
                    do {
                        // per half: 0 below the threshold, else 1 + by how much above
                        const uint32_t l = p + 1 < end ? p[1] : 0u;
                        const uint32_t d0 = __viaddmax_s16x2_relu(p[0], less, 0u), d1 = __viaddmax_s16x2_relu(l, less, 0u);
                        hits += __vminu2(d0, 0x00010001u) + __vminu2(d1, 0x00010001u);
                        over = __dp2a_lo(d0 + d1, 0x0101u, over);
                        p += 2;
                    } while (p < end);
                    const uint32_t cnt = (hits & 0xffffu) + (hits >> 16);
                    const float ulp_up = __uint_as_float(max(at[q] & 0x7f800000u, 1u << 23));       // 2^23 ulps
                    const float past = __fmaf_rn(scale, mid[q], -__uint_as_float(at[q]));           // mu - threshold
                    s = __fmaf_rn(step[q] * scale, __fmaf_rn((float)(over - cnt) * 0x1p-23f, ulp_up, -(float)cnt * past), s);
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
                s += __shfl_xor_sync(0xffffffffu, s, o);
            its_sum = lane == turn ? s : its_sum;
        }
        if (lane < count_c)
            acc[c_first - c_lo + lane] -= 2.0 * (double)its_sum;
        __syncthreads();
    }

    asm volatile("griddepcontrol.launch_dependents;");
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        spread_sq += __shfl_xor_sync(0xffffffffu, spread_sq, o);
    if (lane == 0)
        s_red[warp] = spread_sq;
    __syncthreads();
    for (int c = c_lo + tid; c < c_hi; c += SORT_THREADS)
        a.partial[(int64_t)blockIdx.x * ncand + c] = acc[c - c_lo];
    if (tid == 0 && blockIdx.y == 0) {
        double s = 0.0;
        for (int w = 0; w < 32; ++w)
            s += s_red[w];
        a.spread_sq[blockIdx.x] = s;
    }
    if (nan)
        flag_status(a.status, FPQ_ERR_NAN_INPUT);
}

__device__ __forceinline__ Prefix shuffle_up(const Prefix& p, int o)
{
    Prefix r;
    r.n = __shfl_up_sync(0xffffffffu, p.n, o);
    r.x = __shfl_up_sync(0xffffffffu, p.x, o);
    r.sq = wide(__shfl_up_sync(0xffffffffu, (unsigned long long)p.sq, o),
                __shfl_up_sync(0xffffffffu, (unsigned long long)(p.sq >> 64), o));
    return r;
}
// Sum of `mine` over the block's threads below this one; `warps`: one Prefix per warp in shared memory.
__device__ __forceinline__ Prefix prefix_scan(const Prefix& mine, Prefix* warps)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    Prefix incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const Prefix t = shuffle_up(incl, o);
        if (lane >= o)
            incl = incl + t;
    }
    if (lane == 31)
        warps[warp] = incl;
    __syncthreads();
    Prefix run = shuffle_up(incl, 1);
    if (lane == 0)
        run = {0, 0, 0};
    for (int w = 0; w < warp; ++w)
        run = run + warps[w];
    return run;
}

// Sums from the bottom of each run of BINS / MAX_THRESHOLDS bins, and the runs' totals behind them.
constexpr int RUN = BINS / MAX_THRESHOLDS;
__global__ void __launch_bounds__(RUN) search_prefix_kernel(const SearchArgs a)
{
    __shared__ Prefix s_warps[RUN / 32];
    const int base = first_key(a, threadIdx.x & 31), e0 = lowest_exponent(base);
    asm volatile("griddepcontrol.launch_dependents;");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int b = blockIdx.x * RUN + threadIdx.x;
    const Prefix mine = bin_sums(a, b, base, e0);
    const Prefix below = prefix_scan(mine, s_warps);
    auto store = [&](int at, const Prefix& p) {
        a.below[at] = make_ulonglong2(p.n, p.x);
        a.below_sq[at] = make_ulonglong2((unsigned long long)p.sq, (unsigned long long)(p.sq >> 64));
    };
    store(b, below);
    if (threadIdx.x == RUN - 1)
        store(BINS + blockIdx.x, below + mine);
}

// Error of every candidate, a block each, a thread per grid value g: the bins whose lower edges round to g lie between
// two thresholds, so the sums over them are differences of the sums from the bottom.  With c the whole number next to
// g, the sum of (x - c)^2 is exact and the rest of the distance (c - g) a small correction: nothing cancels, and data
// that lies on a candidate's grid keeps its error's relative accuracy.  The sum of squared distances from the bins'
// centres is the same for all candidates and was added up while sorting, as was what the thresholds change.
// The last block to finish applies the selection rule.
__global__ void __launch_bounds__(MAX_THRESHOLDS) search_eval_kernel(const SearchArgs a)
{
    __shared__ double s_red[2][MAX_THRESHOLDS / 32];
    __shared__ Prefix s_warps[MAX_THRESHOLDS / 32], s_runs[MAX_THRESHOLDS + 1], s_at[MAX_THRESHOLDS];
    __shared__ bool s_last;
    const int k = threadIdx.x, warp = k >> 5, lane = k & 31;
    const int ncand = a.n_enc * a.n_clip, c = blockIdx.x;
    const int base = first_key(a, lane), e0 = lowest_exponent(base);
    int i;
    float scale;
    candidate_scale(a, c, i, scale);
    const SearchEnc& enc = a.enc[i];
    asm volatile("griddepcontrol.wait;" ::: "memory");
    auto load = [&](int at) {
        const ulonglong2 p = __ldcg(a.below + at), q = __ldcg(a.below_sq + at);
        return Prefix{p.x, p.y, wide(q.x, q.y)};
    };
    {
        const Prefix mine = load(BINS + k), run = prefix_scan(mine, s_warps);
        s_runs[k] = run;
        if (k == MAX_THRESHOLDS - 1)
            s_runs[MAX_THRESHOLDS] = run + mine;
    }
    __syncthreads();
    // everything below the first bin whose lower edge is at or above threshold k
    Prefix top = s_runs[MAX_THRESHOLDS];
    if (k < enc.thresholds) {
        const uint32_t at = __ldcg(a.threshold + c * MAX_THRESHOLDS + k);
        const int64_t key = (int64_t)(((uint64_t)at + ((1u << LOW_BITS) - 1)) >> LOW_BITS) - base;
        const int b = (int)min(max(key, (int64_t)0), (int64_t)BINS);
        if (b < BINS)
            top = s_runs[b / RUN] + load(b);
    }
    s_at[k] = top;
    __syncthreads();
    double err = 0.0, rest = 0.0;
    if (k <= enc.thresholds) {
        const Prefix bottom = k ? s_at[k - 1] : Prefix{0, 0, 0};
        const unsigned long long n = top.n - bottom.n, x = top.x - bottom.x;
        if (n) {
            const unsigned __int128 sq = top.sq - bottom.sq;
            const double unit = __longlong_as_double((long long)(e0 - 150 + 1023) << 52);
            const double per = __longlong_as_double((long long)(150 - e0 + 1023) << 52);
            const double g = (double)scale * (double)code_magnitude(enc, k) * per;
            // (never beyond the bins: a grid value so far above all elements cannot be theirs)
            const unsigned long long centre = (unsigned long long)llrint(fmin(g, 1099511627776.0));
            const double d = (double)centre - g;
            const __int128 e2 = (__int128)(sq - (unsigned __int128)centre * x * 2 + (unsigned __int128)centre * centre * n);
            const __int128 e1 = (__int128)((unsigned __int128)x - (unsigned __int128)centre * n);
            err = (to_double(e2) + fma(2.0 * d, to_double(e1), d * d * (double)n)) * unit * unit;
        }
    }
    static_assert(SORT_BLOCKS <= 2 * MAX_THRESHOLDS, "two partial sums per thread");
#pragma unroll
    for (int u = 0; u < 2; ++u)
        if (const int b = k + u * MAX_THRESHOLDS; b < a.blocks)
            rest += __ldcg(a.partial + (int64_t)b * ncand + c) + __ldcg(a.spread_sq + b);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        err += __shfl_xor_sync(0xffffffffu, err, o);
        rest += __shfl_xor_sync(0xffffffffu, rest, o);
    }
    if (lane == 0) {
        s_red[0][warp] = err;
        s_red[1][warp] = rest;
    }
    __syncthreads();
    if (k == 0) {
        double s = 0.0, r = 0.0;
#pragma unroll
        for (int w = 0; w < MAX_THRESHOLDS / 32; ++w) {
            s += s_red[0][w];
            r += s_red[1][w];
        }
        s += r;
        // (a sum of squares: rounding must not leave it below zero)
        s = (s < 0.0 ? 0.0 : s) + (a.add_to ? a.mse[c] : 0.0);
        a.mse[c] = a.divide_by > 0.0 ? s / a.divide_by : s;
        __threadfence();
        s_last = a.divide_by > 0.0 && atomicAdd(a.ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (s_last) {
        __threadfence();
        select_best<MAX_THRESHOLDS>(a.mse, ncand, a.n_clip, a.best);
    }
}

// ---- host side -----------------------------------------------------------------------------------

size_t search_workspace_bytes(int n_enc, int n_clip)
{
    return (size_t)SEARCH_DIRECT_BLOCKS * (size_t)n_enc * (size_t)n_clip * sizeof(double);
}

// Scratch of the sorted form inside the workspace (which is 8-byte aligned): offsets from its first 16-byte boundary.
struct SortScratch {
    size_t below, below_sq, bin_sum, threshold, nudge, spread_sq, partial, ticket, bytes;
};
static SortScratch sort_scratch(int ncand)
{
    SortScratch s = {};
    s.below = 0;
    s.below_sq = s.below + sizeof(ulonglong2) * (BINS + MAX_THRESHOLDS);
    s.bin_sum = s.below_sq + sizeof(ulonglong2) * (BINS + MAX_THRESHOLDS);
    s.threshold = s.bin_sum + sizeof(unsigned long long) * BINS;
    s.nudge = s.threshold + sizeof(uint32_t) * MAX_THRESHOLDS * (size_t)ncand;
    s.spread_sq = s.nudge + sizeof(char4) * 32 * (size_t)ncand;
    s.partial = s.spread_sq + sizeof(double) * SORT_BLOCKS;
    s.ticket = s.partial + sizeof(double) * SORT_BLOCKS * (size_t)ncand;
    s.bytes = s.ticket + sizeof(unsigned) + 8;
    return s;
}

// In how many shares the candidates are walked: every share sorts all elements again, and walks fewer candidates.  Pays
// while a block's elements are few beside the candidates (444 candidates in 1, 2, 4, 8 shares: 262144 elements 45.5, 37.9,
// 33.6, 32.3 us, 1 M elements 48.6, 42.0, 41.2, 48.5, 1.6 M elements 50.5, 47.1, 47.7, 72.1; 222 candidates: 400000 elements
// 31.2, 28.5, 27.9, 31.7, 1 M elements 32.2, 30.2, 33.2, 42.3).
static int sort_shares(int64_t n, int ncand)
{
    int shares = 4;
    while (shares > 1 && n * shares > (int64_t)7000 * ncand)
        shares /= 2;
    return shares;
}

// The sorted form has a fixed cost that grows less with the candidates than the direct form's time (444 candidates: 29.7 us
// direct and 31.9 us sorted at 131072 elements, 41.7 and 33.5 at 200000; 222 candidates: 26.6 and 26.9 us at 200000, 32.5
// and 26.9 at 262144), and its tables have to fit the workspace (90 candidates or more).
static bool sorted_form(int64_t n, int n_enc, int n_clip)
{
    const int64_t ncand = n_enc * n_clip;
    return n * ncand >= 26000000 + 86000 * ncand && sort_scratch((int)ncand).bytes <= search_workspace_bytes(n_enc, n_clip);
}

static fpq_status launch_sorted(SearchArgs a, void* workspace, cudaStream_t st)
{
    const int ncand = a.n_enc * a.n_clip;
    const SortScratch s = sort_scratch(ncand);
    uint8_t* ws = (uint8_t*)(((uintptr_t)workspace + 15) & ~(uintptr_t)15);
    a.below = (ulonglong2*)(ws + s.below);
    a.below_sq = (ulonglong2*)(ws + s.below_sq);
    a.bin_sum = (unsigned long long*)(ws + s.bin_sum);
    a.threshold = (uint32_t*)(ws + s.threshold);
    a.nudge = (char4*)(ws + s.nudge);
    a.spread_sq = (double*)(ws + s.spread_sq);
    a.partial = (double*)(ws + s.partial);
    a.ticket = (unsigned*)(ws + s.ticket);
    const float* x = a.x;
    const int64_t total = a.n, parts = (total + PACK_MAX - 1) / PACK_MAX;
    cudaLaunchAttribute behind[1];
    behind[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    behind[0].val.programmaticStreamSerializationAllowed = 1;
    for (int64_t part = 0, done = 0; part < parts; ++part) {
        a.x = x + done;
        a.n = part + 1 == parts ? total - done : round_up((total - done) / (parts - part), 4);
        done += a.n;
        a.add_to = part > 0;
        a.divide_by = part + 1 == parts ? (double)total : 0.0;
        const int shares = sort_shares(a.n, ncand);
        a.blocks = SORT_BLOCKS / shares;
        search_tables_kernel<<<(ncand * MAX_THRESHOLDS + 255) / 256, 256, 0, st>>>(a);
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)a.blocks, (unsigned)shares);
        cfg.blockDim = dim3(SORT_THREADS);
        cfg.dynamicSmemBytes = SORT_SMEM;
        cfg.stream = st;
        cfg.attrs = behind;
        cfg.numAttrs = 1;
        if (cudaLaunchKernelEx(&cfg, search_sort_kernel, (const SearchArgs)a) != cudaSuccess)
            return FPQ_ERR_CUDA;
        cfg.gridDim = dim3(MAX_THRESHOLDS);
        cfg.blockDim = dim3(RUN);
        cfg.dynamicSmemBytes = 0;
        if (cudaLaunchKernelEx(&cfg, search_prefix_kernel, (const SearchArgs)a) != cudaSuccess)
            return FPQ_ERR_CUDA;
        cfg.gridDim = dim3((unsigned)ncand);
        cfg.blockDim = dim3(MAX_THRESHOLDS);
        if (cudaLaunchKernelEx(&cfg, search_eval_kernel, (const SearchArgs)a) != cudaSuccess)
            return FPQ_ERR_CUDA;
    }
    return cudaGetLastError() == cudaSuccess ? FPQ_OK : FPQ_ERR_CUDA;
}

fpq_status launch_search(const float* x, int64_t n, const fpq_format* enc, int n_enc, const float* clip, int n_clip,
                         double* mse, int32_t* best, void* workspace, cudaStream_t st)
{
    SearchArgs a{};
    for (int i = 0; i < n_enc; ++i) {
        QFormat q;
        if (!resolve_format(enc[i], &q))
            return FPQ_ERR_FORMAT;
        SearchEnc& e = a.enc[i];
        e.cmax_bits = q.cmax_bits;
        e.ebmin_bits = (uint32_t)(128 - q.B) << 23;
        e.cbase = ((uint32_t)(23 - q.m) << 23) | 0x400000u;
        e.cmax = format_cmax(enc[i]);
        e.spread = ldexpf(1.0f, 23 - q.m);
        e.floor_c = ldexpf(1.5f, 23 + 1 - q.B - q.m);
        e.m = q.m;
        e.bias_bits = (127 - q.B) * (1 << 23);
        e.thresholds = q.code_max;
        e.sub_step = ldexpf(1.0f, 1 - q.B - q.m);
    }
    a.n_enc = n_enc;
    a.n_clip = n_clip;
    a.n = n;
    a.x = x;
    a.clip = clip;
    a.mse = mse;
    a.best = best;
    a.status = status_word();
    if (!a.status)
        return FPQ_ERR_CUDA;
    const int ncand = n_enc * n_clip;
    a.partial = (double*)workspace;
    constexpr size_t kDirectSmem = (size_t)(SEARCH_THREADS / 32) * SEARCH_MAX_CAND * sizeof(double) +
                                   (size_t)SEARCH_MAX_CAND * 2 * sizeof(float);
    {
        static std::mutex attr_mutex;
        std::lock_guard<std::mutex> lock(attr_mutex);
        static bool smem_set[64] = {};
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64)
            return FPQ_ERR_CUDA;
        if (!smem_set[dev]) {
            if (cudaFuncSetAttribute(search_mse_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDirectSmem) !=
                    cudaSuccess ||
                cudaFuncSetAttribute(search_sort_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SORT_SMEM) !=
                    cudaSuccess)
                return FPQ_ERR_CUDA;
            smem_set[dev] = true;
        }
    }
    if (sorted_form(n, n_enc, n_clip))
        return launch_sorted(a, workspace, st);
    int64_t blocks = (n + SEARCH_CHUNK - 1) / SEARCH_CHUNK;
    if (blocks > SEARCH_DIRECT_BLOCKS)
        blocks = SEARCH_DIRECT_BLOCKS;
    if (blocks < 1)
        blocks = 1;
    a.blocks = (int)blocks;
    // about four blocks per SM, but at least four candidates each
    int64_t shares = (592 + blocks - 1) / blocks;
    if (shares > (ncand + 3) / 4)
        shares = (ncand + 3) / 4;
    const int nc = (ncand + (int)shares - 1) / (int)shares;
    const size_t smem = (size_t)(SEARCH_THREADS / 32) * nc * sizeof(double) + (size_t)nc * 2 * sizeof(float);
    search_mse_kernel<<<dim3((unsigned)blocks, (unsigned)shares), SEARCH_THREADS, smem, st>>>(a);
    search_finish_kernel<<<1, 1024, 0, st>>>(a);
    return cudaGetLastError() == cudaSuccess ? FPQ_OK : FPQ_ERR_CUDA;
}

int search_max_enc() { return SEARCH_MAX_ENC; }
int search_max_clip() { return SEARCH_MAX_CLIP; }
int search_max_cand() { return SEARCH_MAX_CAND; }

}  // namespace fpq
