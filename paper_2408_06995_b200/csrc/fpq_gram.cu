// The rounding-learning step (Sec. V-B) from S = A^T A: the data gradient D^T A = E S and the squared error <E S, E>, with
// E = Wq(alpha) - W, for A [M][K] and E [N][K] in FP32: half of M K^2 and N K^2 products instead of 2 M N K.
//
// <E S, E> squares what cancels in D = A E^T, and descent makes E small along the rows' leading directions, where all of it
// cancels: FP32 sums are not enough (4096 rows of rank 32: the loss up to 93 % off and negative at times).  Both contractions
// are therefore exact sums of whole numbers on the INT8 tensor cores.  A column of A (in a slice of rows), a row of E and a
// row of S are written as whole numbers of 32 bits times a power of two, the largest magnitude just below 2^31, and these as
// four signed bytes, digits of base 256 from -128 to 127, one plane of bytes per digit.  The product of two such numbers is
// the sum of 16 products of digits; the 10 whose digit numbers add up to 3 or less are formed, each order 0 ... 3 into an
// accumulator of its own (whole numbers of 32 bits, exact), and put together in 64 bits; for S also the product of the third
// digits, which on the diagonal is a sum of squares (without it the loss was 7e-9 off, with it 2e-10, the rounding of E to FP32
// to begin with 4e-9).  What is left out has no sign of its own and is below 2^-30 of the product of the two largest magnitudes
// per term; an FP32 number down to 2^-7 of the largest is represented exactly.
// (FP64 matrix instructions, 37 TFLOP/s, took 20 and 13 us for the two contractions of 4096 x 320 rows and 960 x 320 weights.)
//
//   column_max_kernel    largest magnitudes of 256 rows, where a slice has more rows than a block sees
//   sliced_prepare_kernel  E, dWq/dalpha, the regulariser's gradient and E's planes; A's planes, transposed
//   sliced_mma_kernel<false>  S: tiles on and above the diagonal, slices of the rows, in double
//   sliced_sum_kernel    the slices added in their order, both triangles; S and its planes
//   sliced_mma_kernel<true>   E S, squared error, chain rule, optional descent update
//
// What is not finite stays out of the planes and is worked out in double directly (E S for such a row of E or column of S, an
// entry of S for such a column of A), so that infinities and NaN end where they did.
#include <cuda.h>

#include <mutex>

#include "fpq_common.cuh"
#include "fpq_kernels.h"
#include "fpq_softround.cuh"
#include "fpq_tensormap.h"

namespace fpq {

namespace {

constexpr int P = 4;                           // digits
__host__ __device__ constexpr int orders(bool grad) { return grad ? P : P + 1; }
constexpr int BM = 128, BK = 128;              // rows of a tile; bytes (reduction elements) of a chunk
constexpr int MMA_W = 1, EPI_W0 = 2, NUM_EPI = 16, EPI_T = 32 * NUM_EPI;
constexpr int NTHREADS = 32 * (EPI_W0 + NUM_EPI);
constexpr int SMEM_BUDGET = 227 * 1024;
constexpr int MAX_SLOTS = 10, CTL = 2048;
constexpr int BATCH = 2;                       // items of four columns of the finished gradient in registers at once
constexpr int SUM_ROW = 1024;                  // columns of S that sliced_sum_kernel keeps in shared memory
constexpr int NOT_FINITE = 0x7fffffff;         // in the place of an exponent

// e with |v| < 127 / 128 2^e for magnitudes of these bits (the largest of several), and 2^(3 - e); below 2^-124 they share an
// exponent, of which 32 bits reach the last place of the smallest FP32 numbers
__device__ __forceinline__ int exponent_of(uint32_t max_bits)
{
    return max_bits >= 0x7f800000u ? NOT_FINITE : max((int)((max_bits + 0x20000u) >> 23) - 126, -124);
}
__device__ __forceinline__ float scale_of(int e) { return e == NOT_FINITE ? 0.f : __uint_as_float((uint32_t)(130 - e) << 23); }

// The signed bytes d0 ... d3 (from the top) of x = 2^24 d0 + 2^16 d1 + 2^8 d2 + d3, |x| < 127 2^24.
__device__ __forceinline__ int whole(float v, float scale) { return __float2int_rn(__fmul_rn(__fmul_rn(v, scale), 268435456.f)); }
__device__ __forceinline__ uint32_t digits_of(int x) { return ((uint32_t)x + 0x00808080u) ^ 0x00808080u; }
// byte p from the top of four numbers, for all p
__device__ __forceinline__ void four_digits(const uint32_t (&x)[4], uint32_t (&o)[P])
{
    const uint32_t a = __byte_perm(x[0], x[1], 0x7362), b = __byte_perm(x[2], x[3], 0x7362);      // bytes 3 3 2 2
    const uint32_t c = __byte_perm(x[0], x[1], 0x5140), d = __byte_perm(x[2], x[3], 0x5140);      // bytes 1 1 0 0
    o[0] = __byte_perm(a, b, 0x7632);
    o[1] = __byte_perm(a, b, 0x5410);
    o[2] = __byte_perm(c, d, 0x7632);
    o[3] = __byte_perm(c, d, 0x5410);
}

__device__ __forceinline__ double power_of_two(int k) { return __hiloint2double((1023 + k) << 20, 0); }   // -1022 <= k <= 1023

// four neighbouring numbers, of which `there` exist; vec: they are 16-byte aligned and all there or none
__device__ __forceinline__ void load4(const float* p, int64_t at, int64_t there, int vec, float (&v)[4])
{
    if (vec) {
        const float4 x = there > 0 ? *reinterpret_cast<const float4*>(p + at) : make_float4(0.f, 0.f, 0.f, 0.f);
        v[0] = x.x, v[1] = x.y, v[2] = x.z, v[3] = x.w;
        return;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
        v[q] = q < there ? p[at + q] : 0.f;
}
__device__ __forceinline__ void store4(float* p, int64_t at, int64_t there, int vec, const float (&v)[4])
{
    if (vec) {
        *reinterpret_cast<float4*>(p + at) = make_float4(v[0], v[1], v[2], v[3]);
        return;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
        if (q < there)
            p[at + q] = v[q];
}

// largest magnitude (as bits) of 256 rows of each column: PM[piece][K]
__global__ void __launch_bounds__(256) column_max_kernel(const float* __restrict__ A, int64_t M, int64_t K, uint32_t* __restrict__ PM)
{
    __shared__ uint32_t part[8][32];
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t col = (int64_t)blockIdx.x * 32 + lane, m0 = (int64_t)blockIdx.y * 256 + 32 * warp;
    uint32_t big = 0;
    if (col < K) {
#pragma unroll 16
        for (int r = 0; r < 32; ++r)
            if (m0 + r < M)
                big = max(big, __float_as_uint(__ldg(A + (m0 + r) * K + col)) & 0x7fffffffu);
    }
    part[warp][lane] = big;
    __syncthreads();
    if (warp == 0 && col < K) {
#pragma unroll
        for (int w = 1; w < 8; ++w)
            big = max(big, part[w][lane]);
        PM[(int64_t)blockIdx.y * K + col] = big;
    }
}

struct SlicedPrepare {
    const float *w, *scale, *alpha, *A;
    float *E, *DQ, *RG;        // errors, dWq/dalpha, the regulariser's part of the gradient
    uint8_t *PE, *PA;          // planes of E [P][N][K16] and of A^T [P][K][Mp]
    int *eE, *eA;              // exponents: of E's rows [N], of A's columns in a slice [slices][K]
    const uint32_t* PM;        // largest magnitudes of 256 rows, where a slice has more (else NULL)
    double* lam;               // sum of lambda of each block
    unsigned* ticket;
    int64_t M, N, K, K16, Mp;
    int warps_per_row;         // a block has 8 / warps_per_row rows of E
    int row_blocks, col_blocks, rows;   // blocks of A: 32 columns and up to 256 of a slice's `rows` each
    float reg;
    QFormat f;
    int* status;
};
// Blocks of A come first: a thread has 32 rows of one column in registers, so that it writes whole 32-byte sectors of the
// transposed planes.  Blocks of weights: a row's largest error is known when all of it has been worked out; the regulariser is
// done here too, where all SMs are busy, not in the last kernel's few blocks.  Bound by instructions (0.65 issued per cycle and
// scheduler); five blocks per SM, so that 960 x 320 weights and 4096 rows are one round of blocks (four: 9.3 us, five: 8.0).
template <bool VEC>
__global__ void __launch_bounds__(256, 5) sliced_prepare_kernel(const SlicedPrepare g)
{
    __shared__ uint32_t part[8][32];
    __shared__ double lam_part[8];
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    if ((int)blockIdx.x < g.row_blocks) {
        const int64_t id = blockIdx.x, piece = id / g.col_blocks;
        const int64_t col = (id - piece * g.col_blocks) * 32 + lane;
        const int64_t block_rows = min(g.rows, 256), m0 = piece * block_rows + 32 * warp;
        const bool mine = 32 * warp < block_rows && m0 < g.Mp && col < g.K;
        float v[32];
        uint32_t big = 0;
        if (mine) {
            const float* src = g.A + m0 * g.K + col;
            const int rows = (int)max((int64_t)0, min((int64_t)32, g.M - m0));
#pragma unroll
            for (int r = 0; r < 32; ++r, src += g.K)
                v[r] = r < rows ? __ldg(src) : 0.f;
#pragma unroll
            for (int r = 0; r < 32; ++r)
                big = max(big, __float_as_uint(v[r]) & 0x7fffffffu);
        }
        const int64_t slice = piece * block_rows / g.rows;
        if (g.PM) {
            big = 0;
            const int64_t pieces = (g.M + 255) / 256, each = g.rows / 256;
            for (int64_t q = slice * each; q < min((slice + 1) * each, pieces) && col < g.K; ++q)
                big = max(big, __ldg(g.PM + q * g.K + col));
        } else {
            part[warp][lane] = big;
            __syncthreads();
#pragma unroll
            for (int w = 0; w < 8; ++w)
                big = max(big, part[w][lane]);
        }
        if (!mine)
            return;
        const int e = exponent_of(big);
        if (m0 == slice * g.rows)
            g.eA[slice * g.K + col] = e;
        const float f = scale_of(e);
        uint32_t o[8][P];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            uint32_t x[4];
#pragma unroll
            for (int h = 0; h < 4; ++h)
                x[h] = e == NOT_FINITE ? 0u : digits_of(whole(v[4 * q + h], f));
            four_digits(x, o[q]);
        }
        uint8_t* dst = g.PA + col * g.Mp + m0;
#pragma unroll
        for (int p = 0; p < P; ++p, dst += g.K * g.Mp) {
            reinterpret_cast<uint4*>(dst)[0] = make_uint4(o[0][p], o[1][p], o[2][p], o[3][p]);
            reinterpret_cast<uint4*>(dst)[1] = make_uint4(o[4][p], o[5][p], o[6][p], o[7][p]);
        }
        return;
    }
    const int block = (int)blockIdx.x - g.row_blocks;
    if (block == 0 && t == 0)
        *g.ticket = 0;
    const float c = __uint_as_float(g.f.cmax_bits);
    const int per_block = 8 / g.warps_per_row, share = warp % g.warps_per_row;
    const int64_t n = (int64_t)block * per_block + warp / g.warps_per_row;
    bool nan = false;
    float lam = 0.f;
    uint32_t big = 0;
    // (up to 128 columns per warp and row: the errors stay in registers until their exponent is known)
    float v[4] = {};
    const int64_t k0 = 128 * share + 4 * lane, k_step = 128 * g.warps_per_row;
    if (n < g.N) {
        const float gs = __ldg(g.scale + n);
        for (int64_t k = k0; k < g.K; k += k_step) {
            const int64_t i = n * g.K + k;
            float wv[4], al[4], dq[4], rg[4];
            load4(g.w, i, g.K - k, VEC, wv);
            load4(g.alpha, i, g.K - k, VEC, al);
            const float r = __fdiv_rn(1.0f, gs);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const bool there = VEC || k + q < g.K;
                const SoftWeight o = soft_weight(wv[q], al[q], gs, r, c, g.f, nan);
                v[q] = there ? o.e : 0.f;
                dq[q] = o.dq;
                float l = 0.f;
                rg[q] = regulariser_gradient(soft_terms(al[q]), al[q], g.reg, l);
                lam += there ? l : 0.f;
                big = max(big, __float_as_uint(v[q]) & 0x7fffffffu);
            }
            store4(g.E, i, g.K - k, VEC, v);
            store4(g.DQ, i, g.K - k, VEC, dq);
            store4(g.RG, i, g.K - k, VEC, rg);
        }
    }
    if (nan)
        flag_status(g.status, FPQ_ERR_NAN_INPUT);
    big = __reduce_max_sync(0xffffffffu, big);
    const double lam_sum = warp_sum((double)lam);
    if (lane == 0) {
        part[0][warp] = big;
        lam_part[warp] = lam_sum;
    }
    __syncthreads();
    if (t == 0) {
        double sum = 0.0;
        for (int q = 0; q < 8; ++q)
            sum += lam_part[q];
        g.lam[block] = sum;
    }
    if (n >= g.N)
        return;
    for (int q = warp - share; q < warp - share + g.warps_per_row; ++q)
        big = max(big, part[0][q]);
    const int e = exponent_of(big);
    if (share == 0 && lane == 0)
        g.eE[n] = e;
    const float f = scale_of(e);
    for (int64_t k = k0; k < g.K16; k += k_step) {
        if (g.K > k_step) {
            // (each thread reads the errors that it has written)
            load4(g.E, n * g.K + k, g.K - k, VEC, v);
        }
        uint32_t x[4], o[P];
#pragma unroll
        for (int q = 0; q < 4; ++q)
            x[q] = e == NOT_FINITE ? 0u : digits_of(whole(v[q], f));
        four_digits(x, o);
        uint8_t* dst = g.PE + n * g.K16 + k;
#pragma unroll
        for (int p = 0; p < P; ++p, dst += g.N * g.K16)
            *reinterpret_cast<uint32_t*>(dst) = o[p];
    }
}

// D[tmem] (+)= A * B on signed bytes, 32-bit whole numbers; acc == 0 overwrites D
__device__ __forceinline__ void mma_i8(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t idesc, uint32_t acc)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
        "setp.ne.u32 p, %5, 0;\n\t"
        "mov.b64 da, {%1, %3};\n\t"
        "mov.b64 db, {%2, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::i8 [%0], da, db, %4, p;\n\t}"
        ::"r"(d_tmem), "r"(a_lo), "r"(b_lo), "r"(SMEM_DESC_HI_K_SW128), "r"(idesc), "r"(acc)
        : "memory");
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, int (&r)[8])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr)
                 : "memory");
}

struct SlicedArgs {
    int rows_x, rows_y;        // rows of the two operands: K and K, or N and K
    int BN;                    // columns of a tile, a multiple of 16, up to 128 (S: 96)
    int tiles_j;               // column tiles
    int tiles;                 // S: tiles on and above the diagonal
    int length, per;           // the reduction, and of it a block's slice (blockIdx.y)
    int slots, slot_bytes;
    uint32_t idesc, tmem_cols;
    const int *eX, *eY;        // exponents of the operands' rows (S: + slice * K)
    double* SP;                // S: tile t of slice z at (z * tiles + t) * 128 * BN
    // E S
    const double* S;
    const float *E, *DQ, *RG;
    float *alpha, *grad;
    double* loss;
    unsigned* ticket;
    double coef, inv_mn;
    float lr;
    FastDiv div_quads;         // by BN / 4
    int vec, vec_own;          // alpha and grad, E and dWq/dalpha: rows of whole 16-byte pieces
    int* status;
};

// Column tile of BN that the first row of row tile ti (of 128) lies in: tiles (ti, tj) with tj from there on reach the diagonal or
// lie above it; they are numbered row by row.
__device__ __forceinline__ int first_tile(int ti, int BN) { return ti * BM / BN; }
// A tile of sums lies in blocks of 4 x 4, 128 bytes each, 32 of them one below the other: rows and columns of S are both read
// in whole lines.
__device__ __forceinline__ int in_tile(int row, int col) { return ((col >> 2) * (BM / 4) + (row >> 2)) * 16 + (col & 3) * 4 + (row & 3); }

// The product of two operands of digit planes, 128 x BN outputs per block.  Warp 0 loads (one plane of a chunk of both
// operands per slot, so that MMAs start with the first plane), warp 1 issues the MMAs, warps 2-17 put the orders together.
// Bound by the arrival of the operands, some 37 bytes per clock and SM, by the MMAs, some 52 clocks each (10 or 11 per 32
// elements), and by the chains at both ends (first load 1500 clocks, the last sums 1200 to 5000): of 4096 x 320 rows, 64-wide tiles in
// 16 slices, 9.2 us (ncu), FP64 matrix instructions 20; with 960 x 320 weights in 32-wide tiles 10.8 us, FP64 13.
template <bool GRAD>
__global__ void __launch_bounds__(NTHREADS, 1) sliced_mma_kernel(const __grid_constant__ CUtensorMap tmX,
                                                                 const __grid_constant__ CUtensorMap tmY, const SlicedArgs g)
{
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* smem = smem_raw + (smem_base - smem_u32(smem_raw));
    // layout: [ring][barriers, tensor-memory slot][512: sums of the warps][1024: exponents of the columns]
    const uint32_t ctl = (uint32_t)(g.slots * g.slot_bytes);
    const uint32_t full = smem_base + ctl, empty = full + 8 * MAX_SLOTS, acc_full = empty + 8 * MAX_SLOTS;
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem + ctl + 16 * MAX_SLOTS + 8);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int ti, tj;
    if (GRAD) {
        ti = (int)blockIdx.x / g.tiles_j, tj = (int)blockIdx.x - ti * g.tiles_j;
    } else {
        int left = (int)blockIdx.x;
        for (ti = 0; left >= g.tiles_j - first_tile(ti, g.BN); ++ti)
            left -= g.tiles_j - first_tile(ti, g.BN);
        tj = first_tile(ti, g.BN) + left;
    }
    const int x0 = ti * BM, y0 = tj * g.BN;
    const int r_lo = (int)blockIdx.y * g.per, r_hi = min(r_lo + g.per, g.length);
    const int steps = (r_hi - r_lo + 31) / 32, chunks = (steps + 3) / 4;

    if (warp == 0) {
        if (lane < MAX_SLOTS) {
            mbar_init(full + 8 * lane, 1);
            mbar_init(empty + 8 * lane, 1);
        }
        if (lane == 0) {
            mbar_init(acc_full, 1);
            tma_prefetch_desc(&tmX);
            tma_prefetch_desc(&tmY);
        }
        fence_barrier_init();
    }
    if (warp == MMA_W) {
        tmem_alloc(smem_u32((const void*)tmem_slot), g.tmem_cols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");

    bool failed = false;
    if (warp == 0) {
        if (elect_one()) {
            uint32_t s = 0, ph = 1;
            bool dead = false;
            const uint32_t bytes = (uint32_t)(BM + g.BN) * BK;
            for (int c = 0; c < chunks && !dead; ++c)
                for (int p = 0; p < P; ++p) {
                    if (!mbar_wait(empty + 8 * s, ph)) { dead = true; break; }
                    mbar_expect_tx(full + 8 * s, bytes);
                    // (what lies past the rows or the reduction reads as zeros; past a slice, its neighbour's is not multiplied)
                    tma_load_3d(smem_base + s * g.slot_bytes, &tmX, full + 8 * s, r_lo + c * BK, x0, p);
                    tma_load_3d(smem_base + s * g.slot_bytes + BM * BK, &tmY, full + 8 * s, r_lo + c * BK, y0, p);
                    if (++s == (uint32_t)g.slots) { s = 0; ph ^= 1; }
                }
            settle_ring(full, empty, s, ph, g.slots, true, dead);
            failed = dead;
        }
    } else if (warp == MMA_W) {
        if (elect_one()) {
            uint32_t s = 0, ph = 0;
            bool dead = false;
            for (int c = 0; c < chunks && !dead; ++c) {
                const int n = min(4, steps - 4 * c);
                uint32_t x[P], y[P], slot[P];
#pragma unroll
                for (int p = 0; p < P; ++p) {
                    if (dead || !mbar_wait(full + 8 * s, ph)) { dead = true; continue; }
                    tc_fence_after();
                    slot[p] = s;
                    x[p] = smem_desc_lo(smem_base + s * g.slot_bytes);
                    y[p] = smem_desc_lo(smem_base + s * g.slot_bytes + BM * BK);
                    if (++s == (uint32_t)g.slots) { s = 0; ph ^= 1; }
                    // all products of the planes that are there with this one
#pragma unroll
                    for (int q = 0; q <= p; ++q)
#pragma unroll
                        for (int side = 0; side < 2; ++side) {
                            const int i = side ? q : p, j = side ? p : q;
                            if ((i + j >= P && (GRAD || i != 2 || j != 2)) || (side && p == q))
                                continue;
                            // (the first products of the orders 0 ... 4: 0 0, 1 0, 1 1, 2 1, 2 2)
                            const bool first = side == 0 && (p < 2 || (p == 2 && q > 0));
                            const uint32_t d = tmem_base + (uint32_t)((i + j) * g.BN);
                            for (int k = 0; k < n; ++k)
                                mma_i8(d, x[i] + 2 * k, y[j] + 2 * k, g.idesc, !first || c > 0 || k > 0);
                        }
                }
                if (dead)
                    break;
#pragma unroll
                for (int p = 0; p < P; ++p)
                    mma_commit(empty + 8 * slot[p]);
            }
            if (!dead)
                mma_commit(acc_full);
            failed = dead;
        }
    } else {
        const int et = (int)threadIdx.x - 32 * EPI_W0, quarter = warp & 3, group = (warp - EPI_W0) >> 2;
        const int row = quarter * 32 + lane;
        const int* eX = GRAD ? g.eX : g.eX + (int64_t)blockIdx.y * g.rows_x;
        const int* eY = GRAD ? g.eY : g.eY + (int64_t)blockIdx.y * g.rows_y;
        const int ex = x0 + row < g.rows_x ? __ldg(eX + x0 + row) : 0;
        double* tile = GRAD ? reinterpret_cast<double*>(smem) : g.SP + ((int64_t)blockIdx.y * g.tiles + blockIdx.x) * (BM * g.BN);
        const int ld = g.BN + 1;
        int* col_e = reinterpret_cast<int*>(smem + ctl + 1024);
        if (et < g.BN)
            col_e[et] = y0 + et < g.rows_y ? __ldg(eY + y0 + et) : 0;
        // what the gradient is finished with, four columns of a row per item, the first items' while the MMAs run
        const int64_t K = g.rows_y;
        const int quads = g.BN / 4;
        float al[BATCH][4], dq[BATCH][4], e[BATCH][4], rg[BATCH][4];
        auto fetch = [&](int id) {
#pragma unroll
            for (int u = 0; u < BATCH; ++u) {
                const int r = (int)fdiv((uint32_t)(id + u * EPI_T), g.div_quads), c = 4 * (id + u * EPI_T - r * quads);
                const int64_t n = x0 + r, k = y0 + c, at = n * K + k, there = r < BM && n < g.rows_x ? K - k : 0;
                load4(g.alpha, at, g.lr != 0.f ? there : 0, g.vec, al[u]);
                load4(g.RG, at, there, g.vec_own, rg[u]);
                load4(g.DQ, at, there, g.vec_own, dq[u]);
                load4(g.E, at, there, g.vec_own, e[u]);
            }
        };
        if (GRAD)
            fetch(et);
        asm volatile("bar.sync 1, %0;" ::"n"(EPI_T) : "memory");
        if (mbar_wait(acc_full, 0)) {
            tc_fence_after();
            const uint32_t t_addr = tmem_base + ((uint32_t)(quarter * 32) << 16);
            constexpr int O = orders(GRAD);
            for (int c = 8 * group; c < g.BN; c += 2 * NUM_EPI) {
                int r[O][8];
#pragma unroll
                for (int p = 0; p < O; ++p)
                    tmem_ld8(t_addr + (uint32_t)(p * g.BN + c), r[p]);
                tmem_ld_wait();
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    int64_t v = r[0][q];
#pragma unroll
                    for (int p = 1; p < O; ++p)
                        v = v * 256 + r[p][q];
                    const int ey = col_e[c + q];
                    // (the numbers are 2^(31 - e) times as large; the last orders of seven are missing)
                    const double o = ex != NOT_FINITE && ey != NOT_FINITE ? (double)v * power_of_two(ex + ey - 62 + 8 * (7 - O))
                                                                          : __longlong_as_double(0x7ff8000000000000ll);
                    if (GRAD)
                        tile[row * ld + c + q] = o;
                    else
                        tile[in_tile(row, c + q)] = o;
                }
            }
        } else {
            failed = true;
        }
        if (GRAD) {
            asm volatile("bar.sync 1, %0;" ::"n"(EPI_T) : "memory");
            double sq = 0.0;
            for (int id = et; id < BM * quads && !failed; id += BATCH * EPI_T) {
                if (id != et)
                    fetch(id);
#pragma unroll
                for (int u = 0; u < BATCH; ++u) {
                    const int r = (int)fdiv((uint32_t)(id + u * EPI_T), g.div_quads), c = 4 * (id + u * EPI_T - r * quads);
                    const int64_t n = x0 + r, k = y0 + c, at = n * K + k;
                    if (r >= BM || n >= g.rows_x || k >= K)
                        continue;
                    float gr[4];
                    double v[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        v[q] = k + q < K ? tile[r * ld + c + q] : 0.0;
                    if (!(v[0] == v[0] && v[1] == v[1] && v[2] == v[2] && v[3] == v[3])) {
                        // a row of E or a column of S that is not finite
                        for (int q = 0; q < 4 && k + q < K; ++q) {
                            v[q] = 0.0;
                            for (int64_t i = 0; i < K; ++i)
                                v[q] += (double)g.E[n * K + i] * g.S[i * K + k + q];
                        }
                    }
                    sq += fma(v[0], (double)e[u][0], v[1] * (double)e[u][1]) + fma(v[2], (double)e[u][2], v[3] * (double)e[u][3]);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        gr[q] = fmaf((float)(g.coef * v[q]), dq[u][q], rg[u][q]);
                        al[u][q] = al[u][q] - g.lr * gr[q];
                    }
                    store4(g.grad, at, K - k, g.vec, gr);
                    if (g.lr != 0.f)
                        store4(g.alpha, at, K - k, g.vec, al[u]);
                }
            }
            sq = warp_sum(sq);
            double* part = reinterpret_cast<double*>(smem + ctl + 512);
            if (lane == 0)
                part[warp - EPI_W0] = sq;
            asm volatile("bar.sync 1, %0;" ::"n"(EPI_T) : "memory");
            if (warp == EPI_W0) {
                sq = warp_sum(lane < NUM_EPI ? part[lane] : 0.0);
                if (lane == 0) {
                    atomicAdd(g.loss, sq * g.inv_mn);
                    // a sum of squares: rounding must not leave it below zero (the block that comes last looks)
                    uint32_t before;
                    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(before) : "l"(g.ticket) : "memory");
                    if (before == gridDim.x - 1 && __ldcg(g.loss) < 0.0)
                        *g.loss = 0.0;
                }
            }
        }
    }
    tc_fence_before();
    if (failed)
        flag_status(g.status, FPQ_ERR_TIMEOUT);
    __syncthreads();
    if (warp == MMA_W) {
        tc_fence_after();
        tmem_dealloc(tmem_base, g.tmem_cols);
    }
}

// Four rows of S = the slices added in their order, and their digits, for which a whole row has to be seen.  Block 0 also starts
// the losses: the regulariser's is the sum of the prepare kernel's blocks.  Bound by the latency of reading 9.4 MB of sums (320 x
// 320 in 16 slices) and of the second pass: 7 us (ncu); with a column's 128 rows together instead of 4 x 4 blocks 8.6.
__global__ void __launch_bounds__(1024) sliced_sum_kernel(const double* __restrict__ SP, int slices, int tiles, int tiles_j, int BN,
                                                          FastDiv div_bn, const float* __restrict__ A, int64_t M, int K, int K16,
                                                          double* __restrict__ S, uint8_t* __restrict__ PG, int* __restrict__ eG,
                                                          const double* __restrict__ lam, int lams, double* __restrict__ loss)
{
    __shared__ int before[SLICED_MAX_K / BM + 1];      // tiles in front of a row of tiles
    __shared__ uint32_t part[32][4];
    __shared__ double rows[4][SUM_ROW];                // (longer rows are read again)
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    if (t < (K + BM - 1) / BM) {
        int n = 0;
        for (int u = 0; u < t; ++u)
            n += tiles_j - first_tile(u, BN);
        before[t] = n;
    }
    __syncthreads();
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");
    const int jg = (int)blockIdx.x, j0 = 4 * jg;
    const int64_t slice = (int64_t)tiles * (BM * BN);
    uint32_t across = 0, down = 0;                     // upper halves of the largest magnitudes, by lane % 4 and (lane / 4) % 4
    for (int ig = t >> 4; 4 * ig < K; ig += 64) {
        // block (lo, hi) of S, as it lies: for ig below jg its rows are i, its columns j
        const int lo = min(ig, jg), hi = max(ig, jg), ti = 4 * lo / BM, tj = (int)fdiv(4u * (uint32_t)hi, div_bn);
        const double* p = SP + (int64_t)(before[ti] + tj - first_tile(ti, BN)) * (BM * BN) + in_tile(4 * lo - ti * BM, 4 * hi - tj * BN) +
                          (t & 15);
        const int i = 4 * ig + (ig < jg ? t & 3 : (t >> 2) & 3), j = j0 + (ig < jg ? (t >> 2) & 3 : t & 3);
        double sum = 0.0;
        int z = slices;
        for (; z >= 16; z -= 16) {
            double v[16];
#pragma unroll
            for (int q = 0; q < 16; ++q, p += slice)
                v[q] = __ldcg(p);
#pragma unroll
            for (int q = 0; q < 16; ++q)
                sum += v[q];
        }
        for (; z >= 4; z -= 4) {
            double v[4];
#pragma unroll
            for (int q = 0; q < 4; ++q, p += slice)
                v[q] = __ldcg(p);
#pragma unroll
            for (int q = 0; q < 4; ++q)
                sum += v[q];
        }
        for (; z > 0; --z, p += slice)
            sum += __ldcg(p);
        if (i >= K || j >= K)
            continue;
        if (((uint32_t)__double2hiint(sum) & 0x7ff00000u) == 0x7ff00000u) {
            // a column of A that is not finite
            sum = 0.0;
            for (int64_t m = 0; m < M; ++m)
                sum += (double)__ldg(A + m * K + i) * (double)__ldg(A + m * K + j);
        }
        S[(int64_t)j * K + i] = sum;
        if (K <= SUM_ROW)
            rows[j & 3][i] = sum;
        const uint32_t big = (uint32_t)__double2hiint(sum) & 0x7fffffffu;
        if (ig < jg)
            down = max(down, big);
        else
            across = max(across, big);
    }
    for (int o = 4; o < 32; o <<= 1)
        across = max(across, __shfl_xor_sync(0xffffffffu, across, o));
    for (int o = 1; o < 32; o <<= 1)
        if (o == 16 || o < 4)
            down = max(down, __shfl_xor_sync(0xffffffffu, down, o));
    // (lane l has row l of those across, lane 4 l of those down)
    uint32_t big = max(across, __shfl_sync(0xffffffffu, down, 4 * (lane & 3)));
    if (lane < 4)
        part[warp][lane] = big;
    __syncthreads();
    const int r = t >> 8, row = j0 + r;
    if (row < K && warp % 8 * 128 < K16) {
        big = __reduce_max_sync(0xffffffffu, part[lane][r]);
        // (nothing but zeros: any exponent; the products of FP32 numbers stay far above the smallest double)
        const int e = big >= 0x7ff00000u ? NOT_FINITE : max((int)((big + 0x4000u) >> 20) - 1022, -600);
        if ((t & 255) == 0)
            eG[row] = e;
        const double f = e == NOT_FINITE ? 0.0 : power_of_two(31 - e);
        for (int i = 4 * (t & 255); i < K16; i += 1024) {
            uint32_t x[4], o[P];
#pragma unroll
            for (int q = 0; q < 4; ++q)
                x[q] = i + q < K && e != NOT_FINITE
                           ? digits_of(__double2int_rn((K <= SUM_ROW ? rows[r][i + q] : S[(int64_t)row * K + i + q]) * f)) : 0u;
            four_digits(x, o);
#pragma unroll
            for (int p = 0; p < P; ++p)
                *reinterpret_cast<uint32_t*>(PG + ((int64_t)p * K + row) * K16 + i) = o[p];
        }
    }
    if (blockIdx.x == 0 && warp == 31) {
        double sum = 0.0;
        for (int q = lane; q < lams; q += 32)
            sum += lam[q];
        sum = warp_sum(sum);
        if (lane < 2)
            loss[lane] = lane ? sum : 0.0;
    }
}

int ring(int BN)
{
    const int slots = (SMEM_BUDGET - 1024 - CTL) / ((BM + BN) * BK);
    return slots > MAX_SLOTS ? MAX_SLOTS : slots;
}

int64_t upper_tiles(int64_t K, int BN)
{
    const int64_t tj = (K + BN - 1) / BN;
    int64_t n = 0;
    for (int64_t ti = 0; ti * BM < K; ++ti)
        n += tj - ti * BM / BN;
    return n;
}

bool planes_map(EncodeTiledFn enc, CUtensorMap* map, const uint8_t* planes, int64_t length, int64_t rows, int box_rows)
{
    cuuint64_t dims[3] = {(cuuint64_t)length, (cuuint64_t)rows, (cuuint64_t)P};
    cuuint64_t strides[2] = {(cuuint64_t)length, (cuuint64_t)(length * rows)};
    cuuint32_t box[3] = {BK, (cuuint32_t)box_rows, 1}, estr[3] = {1, 1, 1};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, (void*)planes, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <bool GRAD>
cudaError_t launch_mma(const CUtensorMap& x, const CUtensorMap& y, SlicedArgs g, dim3 grid, cudaStream_t st)
{
    static std::mutex mu;
    static bool set[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64)
        return cudaErrorUnknown;
    {
        std::lock_guard<std::mutex> lock(mu);
        if (!set[dev] && cudaFuncSetAttribute(sliced_mma_kernel<GRAD>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BUDGET) != cudaSuccess)
            return cudaErrorUnknown;
        set[dev] = true;
    }
    g.slot_bytes = (BM + g.BN) * BK;
    g.slots = ring(g.BN);
    g.div_quads = make_fastdiv((uint32_t)g.BN / 4);
    // both operands signed bytes, K-major; 32-bit accumulators
    g.idesc = (2u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(g.BN >> 3) << 17) | ((128u >> 4) << 24);
    g.tmem_cols = 32;
    while ((int)g.tmem_cols < orders(GRAD) * g.BN)
        g.tmem_cols *= 2;
    return launch_overlapped(sliced_mma_kernel<GRAD>, grid, NTHREADS, (size_t)(1024 + CTL + g.slots * g.slot_bytes), st, x, y, g);
}

}  // namespace

SlicedPlan sliced_plan(int64_t M, int64_t N, int64_t K)
{
    SlicedPlan p = {};
    if (K > SLICED_MAX_K || M > (1 << 21) || N > (1 << 21))
        return p;
    p.K16 = round_up(K, 16);
    // S: column tile and slices of the rows with the fewest clocks, the rounds of its blocks and the slices' sums together
    const int64_t steps = (M + 31) / 32;
    double best = 0.0, blocks = 0.0, sums = 0.0;
    for (int bn : {48, 64, 80, 96}) {
        const int64_t tiles = upper_tiles(K, bn);
        for (int64_t want = 1; want <= 64 && want <= steps; ++want) {
            int64_t each = (steps + want - 1) / want;
            if (each > 8)
                each = round_up(each, 8);              // (slices of more than 256 rows: whole blocks of the prepare kernel)
            if (each > 512)
                continue;                              // (an order's sum of 16384 rows stays below 2^30)
            const int64_t slices = (steps + each - 1) / each;
            const double fetch = (128.0 + bn) * 128 / 37.0, step = fetch > 11 * 52.0 ? fetch : 11 * 52.0, bytes = 128.0 * bn * 8;
            const double run = (double)((tiles * slices + 147) / 148) * (2500.0 + each * step + bytes / 20.0);
            const double add = (double)(slices * tiles) * bytes / 2500.0, cost = run + add + (each > 8 ? 4000.0 : 0.0);
            if (best == 0.0 || cost < best) {
                best = cost, blocks = run, sums = add;
                p.BN = bn, p.tiles = (int)tiles, p.slices = (int)slices, p.rows = (int)(32 * each);
            }
        }
    }
    if (best == 0.0)
        return p;
    double grad = 0.0;
    for (int bn : {32, 48, 64, 80, 96, 128}) {
        const int64_t tiles = (N + 127) / 128 * ((K + bn - 1) / bn);
        const double mma = bn * 0.55 > 48.0 ? bn * 0.55 : 48.0, fetch = (128.0 + bn) * 128 / 37.0 / 10.0;
        const double cost = (double)((tiles + 147) / 148) * (7000.0 + 20.0 * bn + (double)((K + 31) / 32) * 10.0 * (mma > fetch ? mma : fetch));
        if (grad == 0.0 || cost < grad) {
            grad = cost;
            p.grad_BN = bn;
        }
    }
    // (fitted to 35 shapes from 64 x 128 x 128 to 8192 x 2560 x 320 and 8192 x 1000 x 1000, within 10 %)
    p.us = 8.5 + (1.06 * blocks + 1.73 * sums + 0.82 * grad) / 1900.0 + (p.rows > 256 ? 4.0 : 0.0) +
           (10.9 * (double)(N * K) + 2.6 * (double)(M * K) + 8.3 * (double)(K * K)) / 1e6;
    p.Mp = (int64_t)p.slices * p.rows;
    size_t o = 0;
    auto take = [&](int64_t bytes) {
        const size_t at = o;
        o += (size_t)round_up(bytes, 256);
        return at;
    };
    p.off_E = take(N * K * 4);
    p.off_DQ = take(N * K * 4);
    p.off_RG = take(N * K * 4);
    p.off_PE = take(P * N * p.K16);
    p.off_PA = take(P * K * p.Mp);
    p.off_PG = take(P * K * p.K16);
    p.off_SP = take((int64_t)p.slices * p.tiles * BM * p.BN * 8);
    p.off_S = take(K * K * 8);
    p.off_PM = take(p.rows > 256 ? (M + 255) / 256 * K * 4 : 0);
    p.off_eE = take(N * 4);
    p.off_eA = take((int64_t)p.slices * K * 4);
    p.off_eG = take(K * 4);
    p.off_lam = take(N * 8);
    p.off_ticket = take(4);
    p.bytes = o;
    p.applies = true;
    return p;
}

fpq_status launch_sliced_step(const SlicedPlan& p, const float* w, const float* scale, const QFormat& f, float* alpha, const float* a,
                              int64_t M, int64_t N, int64_t K, float reg, float lr, float* grad, double* loss, void* workspace,
                              cudaStream_t st)
{
    char* ws = (char*)workspace;
    EncodeTiledFn enc = tensor_map_encoder();
    int* status = status_word();
    if (!enc || !status)
        return FPQ_ERR_CUDA;
    SlicedPrepare q = {};
    q.w = w, q.scale = scale, q.alpha = alpha, q.A = a;
    q.E = (float*)(ws + p.off_E), q.DQ = (float*)(ws + p.off_DQ), q.RG = (float*)(ws + p.off_RG);
    q.PE = (uint8_t*)(ws + p.off_PE), q.PA = (uint8_t*)(ws + p.off_PA);
    q.eE = (int*)(ws + p.off_eE), q.eA = (int*)(ws + p.off_eA);
    q.PM = p.rows > 256 ? (const uint32_t*)(ws + p.off_PM) : nullptr;
    q.lam = (double*)(ws + p.off_lam), q.reg = reg, q.ticket = (unsigned*)(ws + p.off_ticket);
    q.M = M, q.N = N, q.K = K, q.K16 = p.K16, q.Mp = p.Mp;
    q.warps_per_row = K <= 128 ? 1 : (K <= 256 ? 2 : (K <= 512 ? 4 : 8));
    const int weight_blocks = (int)((N + 8 / q.warps_per_row - 1) / (8 / q.warps_per_row));
    q.col_blocks = (int)((K + 31) / 32);
    q.row_blocks = (int)(p.Mp / (p.rows < 256 ? p.rows : 256)) * q.col_blocks;
    q.rows = p.rows;
    q.f = f;
    q.status = status;
    if (q.PM && launch_overlapped(column_max_kernel, dim3((unsigned)q.col_blocks, (unsigned)((M + 255) / 256)), 256, 0, st, a, M, K,
                                  (uint32_t*)(ws + p.off_PM)) != cudaSuccess)
        return FPQ_ERR_CUDA;
    const bool vec = K % 4 == 0 && (uintptr_t)w % 16 == 0 && (uintptr_t)alpha % 16 == 0;
    if (launch_overlapped(vec ? sliced_prepare_kernel<true> : sliced_prepare_kernel<false>,
                          dim3((unsigned)(q.row_blocks + weight_blocks)), 256, 0, st, q) != cudaSuccess)
        return FPQ_ERR_CUDA;

    CUtensorMap x, y;
    SlicedArgs g = {};
    g.status = status;
    if (!planes_map(enc, &x, q.PA, p.Mp, K, BM) || !planes_map(enc, &y, q.PA, p.Mp, K, p.BN))
        return FPQ_ERR_CUDA;
    g.rows_x = g.rows_y = (int)K;
    g.BN = p.BN;
    g.tiles_j = (int)((K + p.BN - 1) / p.BN);
    g.tiles = p.tiles;
    g.length = (int)p.Mp, g.per = p.rows;
    g.eX = g.eY = q.eA;
    g.SP = (double*)(ws + p.off_SP);
    if (launch_mma<false>(x, y, g, dim3((unsigned)p.tiles, (unsigned)p.slices), st) != cudaSuccess)
        return FPQ_ERR_CUDA;
    double* S = (double*)(ws + p.off_S);
    uint8_t* PG = (uint8_t*)(ws + p.off_PG);
    int* eG = (int*)(ws + p.off_eG);
    if (launch_overlapped(sliced_sum_kernel, dim3((unsigned)((K + 3) / 4)), 1024, 0, st, g.SP, p.slices, p.tiles, g.tiles_j, p.BN,
                          make_fastdiv((uint32_t)p.BN), a, M, (int)K, (int)p.K16, S, PG, eG, q.lam, weight_blocks, loss) != cudaSuccess)
        return FPQ_ERR_CUDA;

    if (!planes_map(enc, &x, q.PE, p.K16, N, BM) || !planes_map(enc, &y, PG, p.K16, K, p.grad_BN))
        return FPQ_ERR_CUDA;
    g.rows_x = (int)N;
    g.BN = p.grad_BN;
    g.tiles_j = (int)((K + p.grad_BN - 1) / p.grad_BN);
    g.length = g.per = (int)K;
    g.eX = q.eE, g.eY = eG;
    g.S = S, g.E = q.E, g.DQ = q.DQ, g.RG = q.RG, g.alpha = alpha, g.grad = grad, g.loss = loss, g.ticket = q.ticket;
    g.inv_mn = 1.0 / ((double)M * (double)N);
    g.coef = 2.0 * g.inv_mn;
    g.lr = lr;
    g.vec_own = K % 4 == 0;
    g.vec = g.vec_own && (uintptr_t)alpha % 16 == 0 && (uintptr_t)grad % 16 == 0;
    return launch_mma<true>(x, y, g, dim3((unsigned)((N + BM - 1) / BM * g.tiles_j)), st) == cudaSuccess ? FPQ_OK : FPQ_ERR_CUDA;
}

}  // namespace fpq
