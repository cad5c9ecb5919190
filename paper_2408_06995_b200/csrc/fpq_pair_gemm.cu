// The low-bit contraction of a convolution on CTA pairs (tcgen05 cta_group::2, M = 256): the
// wide-MMA form for layers whose time is the tensor cores' (long reductions, many output channels).
// Activation codes come from the quantize kernel (zero-framed channels-last E4M3, as for the general
// contraction), weights from the prepared copy; both are streamed by TMA.
//
// One MMA spans two CTAs: each CTA holds its own 128 output pixels (rows of A and of the accumulator in
// its tensor memory) and HALF of the weight rows of the column tile, so per MMA an SM reads 4 KB of
// activations and 2 KB (BN = 128) or 4 KB (BN = 256) of weights from shared memory instead of 4 + 4 KB
// for half the work, and every weight byte is fetched once per 256 pixels.  Per CTA: warp 0 TMA producer
// (its own activation chunk, its half of the weight blocks, three taps per box: a TMA load costs about
// one memory latency whatever its size), warp 1 tensor-memory owner (and, in the pair's first CTA, the
// MMA issuer for both), warps 2-9 epilogue (tcgen05.ld -> acc * (x_scale * w_scale[n]) + bias[n] -> NCHW).
// Two accumulators: a unit's epilogue overlaps the next unit's MMAs.  Every wait is bounded; no TMA multicast.
//
// A layer whose input is two concatenated tensors with their own scales keeps one accumulator per tensor, joined in the
// epilogue.
//
// 3 x 3 windows at stride 2 (PHASED): the framed image falls into four sub-images by the parities of row and column, and
// within one of them the taps are rows of one loaded operand again.  Per chunk four boxes of every second pixel are
// fetched instead of nine, into operands that all taps of a phase share: the general contraction, which loads every tap
// apart, is bound by that fetch (some 43 bytes per clock and SM: 32 KB per block of 4 MMAs).  A tile is a box of
// output pixels whose rows and columns in the operand are one longer than its own.  The many small loads need a thread
// per operand.  320 -> 320 channels, batch 3 at 45 x 77, whole layer: 16.2 -> 12.5 us; batch 2 at 64 x 64: 17.0 -> 11.6;
// 512 -> 1280, batch 7 at 48 x 48: 41.7 -> 28.0.
#include <cuda.h>

#include <mutex>

#include "fpq_common.cuh"
#include "fpq_kernels.h"
#include "fpq_tensormap.h"

namespace fpq {

namespace {

constexpr int BM = 128;
constexpr int BK = 128;
constexpr int EPI_W0 = 2, NUM_EPI = 8;
constexpr int B_WARP = EPI_W0 + NUM_EPI;       // stride 2 only
constexpr int num_threads(bool phased) { return 32 * (B_WARP + (phased ? 1 : 0)); }
constexpr int SMEM_BUDGET = 227 * 1024;

struct PGArgs {
    int64_t M;                 // framed pixels B * Hp * Wp
    int N, BN;                 // outputs; column tile (a multiple of 32), BN / 2 weight rows per CTA
    int seg_chunk;             // two input tensors: chunks from here on belong to the second one (0: one tensor)
    float x_scale2;
    double estimate;           // host side only: cycles of the launch
    int acc_cols, acc_bufs;    // TMEM columns of a unit's accumulator(s); units whose accumulators fit at once (1 or 2)
    int cchunks, taps, S;
    int tgroup, ngroups;       // taps per weight stage, weight stages per chunk
    int Wp, HpWp;
    FastDiv div_Wp, div_HpWp, div_nt;
    int B, Ho, Wo;
    int m_tiles, n_tiles, units;   // a unit = (pair of row tiles, column tile), column tile fastest
    int a_boxes, a_box_rows, a_stage_bytes, a_stages;
    int b_tap_bytes, b_stage_bytes, b_stages;
    uint32_t a_tx, b_tx;       // bytes one CTA's loads of a stage report
    uint32_t idesc, tmem_cols;
    // stride 2: a tile of w x h x nb output pixels, row (ib * h2 + iy) * w2 + ix of its operand (w2 = w + 1, h2 = h + 1)
    int w, h, nb, w2, h2, tiles_x, tiles_y;
    FastDiv div_tx, div_ty, div_w2, div_h2;
    int n_pad;                 // N rounded up to the column tile: x_scale * w_scale[n] and bias[n] of all columns sit in shared memory
    const float* w_scale;
    float x_scale;
    const float* bias;
    float* y;
    int* status;
};

// The nine taps of a 3 x 3 window at stride 2, those of one phase (parity of the framed row and column) together: the
// phases' sub-images are loaded one after the other, and a tap reads its phase's operand whole rows further down.
__device__ constexpr int TAP_ORDER[9] = {0, 2, 6, 8, 1, 7, 3, 5, 4};
__device__ constexpr int TAP_DOWN[9] = {0, 0, 1, 1, 0, 1, 0, 0, 0}, TAP_RIGHT[9] = {0, 1, 0, 1, 0, 0, 0, 1, 0};
__device__ constexpr bool phase_first(int i) { return i == 0 || i == 4 || i == 6 || i == 8; }
__device__ constexpr bool phase_last(int i) { return i == 3 || i == 5 || i == 7 || i == 8; }

template <bool PHASED>
__global__ void __launch_bounds__(num_threads(PHASED), 1) fpq_pair_gemm_kernel(const __grid_constant__ CUtensorMap tmA,
                                                                    const __grid_constant__ CUtensorMap tmB,
                                                                    const PGArgs g)
{
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* smem = smem_raw + (smem_base - smem_u32(smem_raw));

    // layout: [A ring][B ring][barriers][x_scale * w_scale | bias of the CTA's current column tile, two copies]
    const uint32_t a_ring = smem_base;
    const uint32_t b_ring = a_ring + g.a_stages * g.a_stage_bytes;
    const uint32_t bars = b_ring + g.b_stages * g.b_stage_bytes;
    const uint32_t a_full = bars, a_empty = bars + 64, b_full = bars + 128, b_empty = bars + 192;
    const uint32_t acc_full = bars + 256, acc_empty = bars + 272;
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem + (bars - smem_base) + 288);
    float* s_scale = reinterpret_cast<float*>(smem + (bars - smem_base) + 512);   // [n_pad] x_scale * w_scale, then [n_pad] bias
    float* s_bias = s_scale + g.n_pad;
    float* s_scale2 = s_bias + g.n_pad;            // two input tensors: x_scale2 * w_scale[n]

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank();
    const int cluster = (int)blockIdx.x >> 1, nclusters = (int)gridDim.x >> 1;
    const int BNh = g.BN >> 1;
    // every cluster walks a contiguous range of units: consecutive units share the pair of row tiles
    const int u_lo = (int)((int64_t)cluster * g.units / nclusters), u_hi = (int)((int64_t)(cluster + 1) * g.units / nclusters);

    if (threadIdx.x == 0) {
        for (int s = 0; s < 8; ++s) {
            mbar_init(a_full + 8 * s, 1);
            mbar_init(a_empty + 8 * s, 1);
            mbar_init(b_full + 8 * s, 1);
            mbar_init(b_empty + 8 * s, 1);
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(acc_full + 8 * s, 1);
            mbar_init(acc_empty + 8 * s, 2 * NUM_EPI);   // the epilogue warps of both CTAs
        }
        fence_barrier_init();
        tma_prefetch_desc(&tmA);
        tma_prefetch_desc(&tmB);
    }
    if (warp == 1) {
        tmem_alloc_pair(smem_u32((const void*)tmem_slot), g.tmem_cols);
        tmem_relinquish_pair();
    }
    tc_fence_before();
    __syncwarp();
    cluster_sync_all();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    // the activation codes are written by the kernel in front (and the output may alias something it reads)
    asm volatile("griddepcontrol.wait;" ::: "memory");

    bool failed = false;                               // a wait of this thread's role ran out
    auto leader = [&](uint32_t bar) { return peer_smem_addr(bar, 0u); };
    auto decode = [&](int u, int& mu, int& nt) {
        mu = (int)fdiv((uint32_t)u, g.div_nt);
        nt = u - mu * g.n_tiles;
    };
    auto tile_origin = [&](int mt, int& x0, int& y0, int& b0) {
        const uint32_t r1 = fdiv((uint32_t)mt, g.div_tx), r2 = fdiv(r1, g.div_ty);
        x0 = (mt - (int)r1 * g.tiles_x) * g.w;
        y0 = ((int)r1 - (int)r2 * g.tiles_y) * g.h;
        b0 = (int)r2 * g.nb;
    };

    if (PHASED && warp == 0) {
        // ---------------- stride 2: activation producer, four phases per chunk ----------------
        if (elect_one()) {
            uint32_t sa = 0, pa = 1;
            bool dead = false;
            const uint32_t full = leader(a_full);
            for (int u = u_lo; u < u_hi && !dead; ++u) {
                int mu, nt, x0, y0, b0;
                decode(u, mu, nt);
                tile_origin(2 * mu + (int)rank, x0, y0, b0);
                for (int cc = 0; cc < g.cchunks && !dead; ++cc)
                    for (int ph = 0; ph < 4; ++ph) {
                        if (!mbar_wait(a_empty + 8 * sa, pa)) { dead = true; break; }
                        if (rank == 0)
                            mbar_expect_tx(a_full + 8 * sa, 2u * g.a_tx);
                        tma_load_4d_pair(a_ring + sa * g.a_stage_bytes, &tmA, full + 8 * sa, cc * BK, 2 * x0 + (ph & 1),
                                         2 * y0 + (ph >> 1), b0);
                        if (++sa == (uint32_t)g.a_stages) { sa = 0; pa ^= 1; }
                    }
            }
            settle_ring(a_full, a_empty, sa, pa, g.a_stages, rank == 0, dead);
            failed = dead;
        }
    } else if (PHASED && warp == B_WARP) {
        // ---------------- stride 2: weight producer ----------------
        if (elect_one()) {
            uint32_t sb = 0, pb = 1;
            bool dead = false;
            const uint32_t full = leader(b_full);
            for (int u = u_lo; u < u_hi && !dead; ++u) {
                int mu, nt;
                decode(u, mu, nt);
                const int n0 = nt * g.BN + (int)rank * BNh;
                for (int cc = 0; cc < g.cchunks && !dead; ++cc) {
#pragma unroll
                    for (int i = 0; i < 9; i += 3) {
                        if (!mbar_wait(b_empty + 8 * sb, pb)) { dead = true; break; }
                        if (rank == 0)
                            mbar_expect_tx(b_full + 8 * sb, 2u * g.b_tx);
                        const uint32_t dst = b_ring + sb * g.b_stage_bytes;
#pragma unroll
                        for (int t = 0; t < 3; ++t)
                            tma_load_3d_pair(dst + t * g.b_tap_bytes, &tmB, full + 8 * sb, cc * BK, n0, TAP_ORDER[i + t]);
                        if (++sb == (uint32_t)g.b_stages) { sb = 0; pb ^= 1; }
                    }
                }
            }
            settle_ring(b_full, b_empty, sb, pb, g.b_stages, rank == 0, dead);
            failed = dead;
        }
    } else if (!PHASED && warp == 0) {
        // ---------------- TMA producer: loads in the order the MMAs consume them ----------------
        if (elect_one()) {
            uint32_t sa = 0, pa = 0, sb = 0, pb = 0;
            bool dead = false;
            const uint32_t ra_full = leader(a_full), rb_full = leader(b_full);
            for (int u = u_lo; u < u_hi && !dead; ++u) {
                int mu, nt;
                decode(u, mu, nt);
                const int mt = 2 * mu + (int)rank;
                const int n0 = nt * g.BN + (int)rank * BNh;
                for (int cc = 0; cc < g.cchunks && !dead; ++cc) {
                    if (!mbar_wait(a_empty + 8 * sa, pa ^ 1)) { dead = true; break; }
                    if (rank == 0)
                        mbar_expect_tx(a_full + 8 * sa, 2u * g.a_tx);
                    for (int bx = 0; bx < g.a_boxes; ++bx)
                        tma_load_4d_pair(a_ring + sa * g.a_stage_bytes + bx * g.a_box_rows * 128, &tmA, ra_full + 8 * sa,
                                         cc * BK, mt * BM + bx * g.a_box_rows, 0, 0);
                    if (++sa == (uint32_t)g.a_stages) { sa = 0; pa ^= 1; }
                    for (int tg = 0; tg < g.ngroups; ++tg) {
                        if (!mbar_wait(b_empty + 8 * sb, pb ^ 1)) { dead = true; break; }
                        if (rank == 0)
                            mbar_expect_tx(b_full + 8 * sb, 2u * g.b_tx);
                        tma_load_3d_pair(b_ring + sb * g.b_stage_bytes, &tmB, rb_full + 8 * sb, cc * BK, n0, tg * g.tgroup);
                        if (++sb == (uint32_t)g.b_stages) { sb = 0; pb ^= 1; }
                    }
                }
            }
            settle_ring(b_full, b_empty, sb, pb ^ 1, g.b_stages, rank == 0, dead);
            settle_ring(a_full, a_empty, sa, pa ^ 1, g.a_stages, rank == 0, dead);
            failed = dead;
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer: one thread of the pair's first CTA ----------------
        if (rank == 0 && elect_one()) {
            uint32_t sa = 0, pa = 0, sb = 0, pb = 0;
            bool dead = false;
            const uint32_t HI = SMEM_DESC_HI_K_SW128;
            const uint32_t TSTEP = (uint32_t)g.b_tap_bytes >> 4;
            const uint32_t row_wrap8 = (uint32_t)(g.Wp - g.S) * 8u;
            uint32_t buf = 0, aph = 0;
            for (int u = u_lo; u < u_hi && !dead; ++u) {
                if (!mbar_wait_cluster(acc_empty + 8 * buf, aph ^ 1)) { dead = true; break; }
                tc_fence_after();
                uint32_t d = tmem_base + buf * (uint32_t)g.acc_cols;
                bool first = true;
                if (PHASED) {
                    const uint32_t down8 = (uint32_t)g.w2 * 8u;
                    for (int cc = 0; cc < g.cchunks && !dead; ++cc) {
                        uint32_t abase = 0, bbase = 0;
#pragma unroll
                        for (int i = 0; i < 9; ++i) {
                            if (phase_first(i)) {
                                if (!mbar_wait_cluster(a_full + 8 * sa, pa)) { dead = true; break; }
                                abase = smem_desc_lo(a_ring + sa * g.a_stage_bytes);
                            }
                            if (i % 3 == 0) {
                                if (!mbar_wait_cluster(b_full + 8 * sb, pb)) { dead = true; break; }
                                bbase = smem_desc_lo(b_ring + sb * g.b_stage_bytes);
                            }
                            if (phase_first(i) || i % 3 == 0)
                                tc_fence_after();
                            const uint32_t al = abase + TAP_DOWN[i] * down8 + TAP_RIGHT[i] * 8u, bl = bbase + (i % 3) * TSTEP;
                            if (i == 0 && cc == 0)
                                mma_f8f6f4_pair<false>(d, al, bl, HI, g.idesc);
                            else
                                mma_f8f6f4_pair<true>(d, al, bl, HI, g.idesc);
                            mma_f8f6f4_pair<true>(d, al + 2, bl + 2, HI, g.idesc);
                            mma_f8f6f4_pair<true>(d, al + 4, bl + 4, HI, g.idesc);
                            mma_f8f6f4_pair<true>(d, al + 6, bl + 6, HI, g.idesc);
                            if (i % 3 == 2) {
                                mma_commit_pair(b_empty + 8 * sb, 3);
                                if (++sb == (uint32_t)g.b_stages) { sb = 0; pb ^= 1; }
                            }
                            if (phase_last(i)) {
                                mma_commit_pair(a_empty + 8 * sa, 3);
                                if (++sa == (uint32_t)g.a_stages) { sa = 0; pa ^= 1; }
                            }
                        }
                    }
                }
                for (int cc = 0; !PHASED && cc < g.cchunks && !dead; ++cc) {
                    if (cc == g.seg_chunk && cc != 0) {
                        d += (uint32_t)g.BN;                       // the second tensor's accumulator
                        first = true;
                    }
                    if (!mbar_wait_cluster(a_full + 8 * sa, pa)) { dead = true; break; }
                    tc_fence_after();
                    const uint32_t abase = smem_desc_lo(a_ring + sa * g.a_stage_bytes);
                    uint32_t off8 = 0;
                    int sxx = 0;
                    for (int tg = 0; tg < g.ngroups && !dead; ++tg) {
                        if (!mbar_wait_cluster(b_full + 8 * sb, pb)) { dead = true; break; }
                        tc_fence_after();
                        const uint32_t bbase = smem_desc_lo(b_ring + sb * g.b_stage_bytes);
                        for (int t = 0; t < g.tgroup; ++t) {
                            const uint32_t al = abase + off8, bl = bbase + (uint32_t)t * TSTEP;
                            if (first)
                                mma_f8f6f4_pair<false>(d, al, bl, HI, g.idesc);
                            else
                                mma_f8f6f4_pair<true>(d, al, bl, HI, g.idesc);
                            first = false;
                            mma_f8f6f4_pair<true>(d, al + 2, bl + 2, HI, g.idesc);
                            mma_f8f6f4_pair<true>(d, al + 4, bl + 4, HI, g.idesc);
                            mma_f8f6f4_pair<true>(d, al + 6, bl + 6, HI, g.idesc);
                            off8 += 8;
                            if (++sxx == g.S) { sxx = 0; off8 += row_wrap8; }
                        }
                        mma_commit_pair(b_empty + 8 * sb, 3);
                        if (++sb == (uint32_t)g.b_stages) { sb = 0; pb ^= 1; }
                    }
                    if (dead)
                        break;
                    mma_commit_pair(a_empty + 8 * sa, 3);
                    if (++sa == (uint32_t)g.a_stages) { sa = 0; pa ^= 1; }
                }
                if (dead)
                    break;
                mma_commit_pair(acc_full + 8 * buf, 3);
                if (++buf == (uint32_t)g.acc_bufs) { buf = 0; aph ^= 1; }
            }
            failed = dead;
        }
    } else {
        // ---------------- epilogue: y = acc * (x_scale * w_scale[n]) + bias[n], NCHW ----------------
        const int quarter = warp & 3, half = (warp - EPI_W0) >> 2;
        const int row = quarter * 32 + lane;
        const uint32_t racc_empty = leader(acc_empty);
        const int64_t nstride = (int64_t)g.Ho * g.Wo;
        for (int i = threadIdx.x - 32 * EPI_W0; i < g.n_pad; i += 32 * NUM_EPI) {
            s_scale[i] = (i < g.N) ? g.x_scale * __ldg(g.w_scale + i) : 0.f;
            s_bias[i] = (g.bias && i < g.N) ? __ldg(g.bias + i) : 0.f;
            if (g.seg_chunk)
                s_scale2[i] = (i < g.N) ? g.x_scale2 * __ldg(g.w_scale + i) : 0.f;
        }
        asm volatile("bar.sync 1, %0;" ::"n"(32 * NUM_EPI) : "memory");
        uint32_t buf = 0, aph = 0;
        bool dead = false;
        for (int u = u_lo; u < u_hi && !dead; ++u) {
            int mu, nt;
            decode(u, mu, nt);
            const int mt = 2 * mu + (int)rank;
            uint32_t b;
            int oy, ox;
            bool row_valid = true;
            if (PHASED) {
                const uint32_t q1 = fdiv((uint32_t)row, g.div_w2), q2 = fdiv(q1, g.div_h2);
                const int ix = row - (int)q1 * g.w2, iy = (int)q1 - (int)q2 * g.h2;
                int b0;
                tile_origin(mt, ox, oy, b0);
                ox += ix, oy += iy, b = (uint32_t)b0 + q2;
                row_valid = ix < g.w && iy < g.h && (int)q2 < g.nb;
            } else {
                const uint32_t q = (uint32_t)mt * BM + row;
                b = fdiv(q, g.div_HpWp);
                const uint32_t rem = q - b * (uint32_t)g.HpWp;
                oy = (int)fdiv(rem, g.div_Wp);
                ox = (int)rem - oy * g.Wp;
                row_valid = (int64_t)q < g.M;
            }
            row_valid = row_valid && ox < g.Wo && oy < g.Ho && (int)b < g.B;
            float* yrow = g.y + ((int64_t)b * g.N * g.Ho + oy) * g.Wo + ox;
            if (!mbar_wait(acc_full + 8 * buf, aph)) { dead = true; break; }
            tc_fence_after();
            const uint32_t t_addr = tmem_base + buf * (uint32_t)g.acc_cols + ((uint32_t)(quarter * 32) << 16);
            for (int c = 32 * half; c < g.BN; c += 64) {           // (every second 32 columns of the tile)
                const int nb = nt * g.BN + c;                      // output channel of the chunk's first column
                if (nb >= g.N)
                    break;
                uint32_t r[32];
                tmem_ld32(t_addr + c, r);
                tmem_ld_wait();
                const float4* s4 = reinterpret_cast<const float4*>(s_scale + nb);
                const float4* b4 = reinterpret_cast<const float4*>(s_bias + nb);
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const float4 sv = s4[k], bv = b4[k];
                    r[4 * k + 0] = __float_as_uint(fmaf(__uint_as_float(r[4 * k + 0]), sv.x, bv.x));
                    r[4 * k + 1] = __float_as_uint(fmaf(__uint_as_float(r[4 * k + 1]), sv.y, bv.y));
                    r[4 * k + 2] = __float_as_uint(fmaf(__uint_as_float(r[4 * k + 2]), sv.z, bv.z));
                    r[4 * k + 3] = __float_as_uint(fmaf(__uint_as_float(r[4 * k + 3]), sv.w, bv.w));
                }
                if (g.seg_chunk) {
                    uint32_t r2[32];
                    tmem_ld32(t_addr + g.BN + c, r2);
                    tmem_ld_wait();
                    const float4* t4 = reinterpret_cast<const float4*>(s_scale2 + nb);
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const float4 tv = t4[k];
                        r[4 * k + 0] = __float_as_uint(fmaf(__uint_as_float(r2[4 * k + 0]), tv.x, __uint_as_float(r[4 * k + 0])));
                        r[4 * k + 1] = __float_as_uint(fmaf(__uint_as_float(r2[4 * k + 1]), tv.y, __uint_as_float(r[4 * k + 1])));
                        r[4 * k + 2] = __float_as_uint(fmaf(__uint_as_float(r2[4 * k + 2]), tv.z, __uint_as_float(r[4 * k + 2])));
                        r[4 * k + 3] = __float_as_uint(fmaf(__uint_as_float(r2[4 * k + 3]), tv.w, __uint_as_float(r[4 * k + 3])));
                    }
                }
                if (row_valid) {
                    float* dst = yrow + (int64_t)nb * nstride;
                    if (nb + 32 <= g.N) {
#pragma unroll
                        for (int k = 0; k < 32; ++k)
                            dst[(int64_t)k * nstride] = __uint_as_float(r[k]);
                    } else {
#pragma unroll
                        for (int k = 0; k < 32; ++k)
                            if (nb + k < g.N)
                                dst[(int64_t)k * nstride] = __uint_as_float(r[k]);
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0 && u + g.acc_bufs < u_hi)                // (somebody waits for it)
                mbar_arrive_cluster(racc_empty + 8 * buf);
            if (++buf == (uint32_t)g.acc_bufs) { buf = 0; aph ^= 1; }
        }
        failed = dead;
    }

    // Nobody leaves while the other CTA may still arrive on its barriers.  Every arrival but a failed role's has been waited
    // for (the MMAs' last ones by the producers), so the barrier need not wait for the stores of the output: the next kernel's blocks move in that much earlier
    // (320 -> 320 channels at 64 x 64, batch 1, whole layer: 11.2 -> 10.5 us).
    tc_fence_before();
    if (failed)
        flag_status(g.status, FPQ_ERR_TIMEOUT);
    if (__any_sync(0xffffffffu, failed))
        cluster_arrive();
    else
        cluster_arrive_relaxed();
    cluster_wait();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc_pair(tmem_base, g.tmem_cols);
    }
}

// Column tile of a layer: the one with the shortest estimate, in SM cycles.  A chunk of the reduction takes its MMAs
// (0.53 cycles per column and 32 reduction elements, 52 at least) or the arrival of its operands (some 43 bytes per clock
// and SM); an epilogue stores some 15 bytes per clock and SM and is hidden behind the next unit's MMAs, except the last
// one's.  (32 columns, whose MMAs take as long as 64's, only where there are no more.)  A width that just fits the columns and
// the SM pairs beats the widest one: 640 -> 320 channels at 64 x 64, batch
// 2, whole layer: 35 units x 3 tiles of 128 in two rounds 24.1 us, x 2 of 160 in one 19.3 us; 256 -> 256 at 32 x 32,
// batch 16: 15.5 us with 128, 18.6 us with 64 or 192.
// loads: those of a chunk where every tap's weights are one, which takes their thread some 400 cycles each (4 x 348 -> 98
// channels at 7 x 7, 25 taps: 22.5 us for 3 x 26 of them, the general kernel 15.7).
int choose_tile(int N, int m_units, int nclusters, int cchunks, int taps, int a_bytes, int accs, int loads, double* cycles)
{
    int pick = 128;
    double best = 0.0;
    for (int bn = N <= 32 ? 32 : 64; bn <= 256; bn += 32) {
        if (bn - 32 >= N)
            break;
        const int64_t units = (int64_t)m_units * ((N + bn - 1) / bn);
        const double waves = (double)((units + nclusters - 1) / nclusters);
        double mmas = taps * 4 * (bn * 0.53 > 52.0 ? bn * 0.53 : 52.0);
        if (mmas < 400.0 * loads)
            mmas = 400.0 * loads;
        const double fill = (taps * bn * 64.0 + a_bytes) / 43.0;
        const double unit = 800.0 + cchunks * (mmas > fill ? mmas : fill), epi = 128.0 * bn * 4 / 15;
        const bool hidden = 2 * bn * accs <= 512;
        const double cost = hidden ? waves * (waves > 1 && epi > unit ? epi : unit) + epi : waves * (unit + epi);
        if (best == 0.0 || cost < best) {
            best = cost;
            pick = bn;
        }
    }
    *cycles = best;
    return pick;
}

// Stride 2: image rows cut into equal parts, then as many image rows and images as the 128 operand rows hold, one column
// and row of each sub-image more than the tile's (the second and third taps' reach); the cut with the fewest tiles.
void choose_phase_tile(PGArgs& g)
{
    int64_t best = 0;
    for (int cut = (g.Wo + 126) / 127; cut <= g.Wo; ++cut) {
        const int w = (g.Wo + cut - 1) / cut, w2 = w + 1;
        const int hmax = (BM - w) / w2 + 1, tiles_x = (g.Wo + w - 1) / w, tiles_y = (g.Ho + hmax - 1) / hmax;
        const int h = (g.Ho + tiles_y - 1) / tiles_y, h2 = h + 1;
        int nb = (BM - w - (h - 1) * w2) / (h2 * w2) + 1;
        if (nb > g.B)
            nb = g.B;
        const int64_t tiles = (int64_t)tiles_x * tiles_y * ((g.B + nb - 1) / nb);
        if (h2 <= 128 && (best == 0 || tiles < best)) {
            best = tiles;
            g.w = w, g.h = h, g.nb = nb, g.w2 = w2, g.h2 = h2, g.tiles_x = tiles_x, g.tiles_y = tiles_y;
        }
        if (w <= 8)
            break;
    }
    g.m_tiles = (int)best;
    g.div_tx = make_fastdiv((uint32_t)g.tiles_x);
    g.div_ty = make_fastdiv((uint32_t)g.tiles_y);
    g.div_w2 = make_fastdiv((uint32_t)g.w2);
    g.div_h2 = make_fastdiv((uint32_t)g.h2);
}

// geometry and shared-memory plan; FPQ_ERR_UNSUPPORTED outside the kernel's range
fpq_status plan_pg(const GemmProblem& p, int nsm, PGArgs& g, int* dyn_bytes)
{
    const bool phased = p.stride == 2;
    if (!p.conv || p.x != nullptr || p.N < 1 || p.R * p.S > 64 ||
        !(p.stride == 1 || (phased && p.R == 3 && p.S == 3 && p.c_seg == 0)))
        return FPQ_ERR_UNSUPPORTED;
    const int Hp = p.H + 2 * p.pad, Wp = p.W + 2 * p.pad;
    const int64_t framed = (int64_t)p.B * Hp * Wp;
    if (framed >= 0x7fffff00ll)
        return FPQ_ERR_UNSUPPORTED;
    g = PGArgs{};
    g.M = framed;
    g.N = p.N;
    g.cchunks = p.Cp / BK;
    g.taps = p.R * p.S;
    g.S = p.S;
    g.tgroup = (g.taps % 3 == 0) ? 3 : 1;
    g.ngroups = g.taps / g.tgroup;
    g.Wp = Wp;
    g.HpWp = Hp * Wp;
    g.div_Wp = make_fastdiv((uint32_t)Wp);
    g.div_HpWp = make_fastdiv((uint32_t)g.HpWp);
    g.B = p.B; g.Ho = p.Ho; g.Wo = p.Wo;
    int halo_rows;
    if (phased) {
        choose_phase_tile(g);
        halo_rows = BM + g.w2 + 1;                     // (the last tap's reach; the box itself may be shorter)
        if (g.nb * g.h2 * g.w2 > halo_rows)
            halo_rows = g.nb * g.h2 * g.w2;
        g.a_tx = (uint32_t)(g.nb * g.h2 * g.w2 * 128);
    } else {
        halo_rows = BM + (p.R - 1) * Wp + (p.S - 1);
        g.m_tiles = (int)((framed + BM - 1) / BM);
    }
    if (halo_rows > 2 * 256 - 16)
        return FPQ_ERR_UNSUPPORTED;
    const int m_units = (g.m_tiles + 1) / 2;
    const int nclusters = nsm / 2;
    g.seg_chunk = p.c_seg;
    g.x_scale2 = p.x_scale2;
    const int accs = p.c_seg ? 2 : 1;
    const int a_bytes = phased ? 4 * (int)g.a_tx : (int)round_up(halo_rows, 8) * 128;
    g.a_boxes = halo_rows > 256 && !phased ? 2 : 1;
    const int loads = g.taps >= 4 && g.tgroup == 1 ? g.ngroups + g.a_boxes : 0;
    g.BN = choose_tile(p.N, m_units, nclusters, g.cchunks, g.taps, a_bytes, accs, loads, &g.estimate);
    g.acc_cols = g.BN * accs;
    g.acc_bufs = 2 * g.acc_cols <= 512 ? 2 : 1;
    g.n_tiles = (p.N + g.BN - 1) / g.BN;
    g.div_nt = make_fastdiv((uint32_t)g.n_tiles);
    g.units = m_units * g.n_tiles;
    g.a_box_rows = (int)round_up((halo_rows + g.a_boxes - 1) / g.a_boxes, 8);
    g.a_stage_bytes = g.a_boxes * g.a_box_rows * 128;
    if (!phased)
        g.a_tx = (uint32_t)g.a_stage_bytes;
    g.b_tap_bytes = (g.BN / 2) * BK;
    g.b_stage_bytes = g.tgroup * g.b_tap_bytes;
    g.b_tx = (uint32_t)g.b_stage_bytes / (p.w4 ? 2 : 1);
    g.n_pad = g.n_tiles * g.BN;
    if (g.n_pad * 8 > 32 * 1024)
        return FPQ_ERR_UNSUPPORTED;
    const int ctl = 512 + 1024 + g.n_pad * 4 * (1 + accs);
    g.a_stages = 2;
    g.b_stages = (SMEM_BUDGET - ctl - g.a_stages * g.a_stage_bytes) / g.b_stage_bytes;
    if (g.b_stages > 8)
        g.b_stages = 8;
    if (g.b_stages < 2)
        return FPQ_ERR_UNSUPPORTED;
    // a third activation stage if the weights still keep three (stride 2: one per phase)
    if (phased && SMEM_BUDGET - ctl - 4 * g.a_stage_bytes - 3 * g.b_stage_bytes >= 0) {
        g.a_stages = 4;
        g.b_stages = (SMEM_BUDGET - ctl - g.a_stages * g.a_stage_bytes) / g.b_stage_bytes;
        if (g.b_stages > 8)
            g.b_stages = 8;
    } else if (g.b_stages >= 4 && SMEM_BUDGET - ctl - 3 * g.a_stage_bytes - 3 * g.b_stage_bytes >= 0) {
        g.a_stages = 3;
        g.b_stages = (SMEM_BUDGET - ctl - g.a_stages * g.a_stage_bytes) / g.b_stage_bytes;
        if (g.b_stages > 8)
            g.b_stages = 8;
    }
    g.idesc = idesc_f8f6f4_pair(p.a_e5m2 ? 1u : 0u, p.w4 ? 5u : (p.w_e5m2 ? 1u : 0u), (uint32_t)g.BN);
    g.tmem_cols = 32;
    while ((int)g.tmem_cols < g.acc_bufs * g.acc_cols)
        g.tmem_cols *= 2;
    *dyn_bytes = ctl + g.a_stages * g.a_stage_bytes + g.b_stages * g.b_stage_bytes;
    return FPQ_OK;
}

}  // namespace

// Whether this kernel is expected to be faster than the general contraction.
bool pair_gemm_preferred(const GemmProblem& p)
{
    PGArgs g;
    int dyn = 0;
    constexpr int SMS = 148;
    if (plan_pg(p, SMS, g, &dyn) != FPQ_OK)
        return false;
    const int blocks = g.cchunks * g.taps;
    // one tap: both kernels are bound by their epilogues and the fetch of the activations; the pairs win where they get
    // through in one round (320 channels at 64 x 64, batch 2: 10.0 against 11.0 us; 960 -> 320: 15.1 against 17.1) and
    // lose in several (1024 -> 1024 at 32 x 32, batch 16: 48.6 against 43.9) or to a split reduction (2560 -> 1280 at
    // 16 x 16: 14.5 against 12.4)
    if (g.taps < 4)
        return p.N > 64 && g.units >= 40 && g.units <= SMS / 2 && blocks >= 3 && blocks <= 12;
    // otherwise against an estimate of the general one: 128 x 128 tiles whose blocks of 128 reduction elements take some
    // 520 cycles each, the reduction split over clusters when the tiles leave SMs idle.  (1280 channels at 16 x 16, batch
    // 2: 17.1 against 20.3 us; batch 1: 16.6 against 15.0; 256 channels at 16 x 16: 8.0 against 11.1; 1280 -> 128 at
    // 32 x 32: 17.7 against 14.2.)
    // (at stride 2, and where the frame is much of the image, it tiles the image itself and loads every tap apart: 416 -> 608 channels at
    // 11 x 11, batch 50: 49.8 us so, 24.3 us on pairs with the framed pixels)
    int64_t m_tiles = g.m_tiles;
    double block = 520.0;
    if (p.stride > 1 || m_tiles * 4 > ((int64_t)p.B * p.Ho * p.Wo + BM - 1) / BM * 5 + 4) {
        m_tiles = choose_taps_tile(p.B, p.Ho, p.Wo, p.stride).tiles;
        block = 700.0;
    }
    if (p.N <= 64)
        block *= 0.65;         // (its column tile is 64 wide there)
    const int64_t tiles = m_tiles * ((p.N + 127) / 128);
    double general;
    const bool split = 2 * tiles <= SMS && g.cchunks >= 2;
    if (split) {
        int64_t sp = SMS / tiles < 8 ? SMS / tiles : 8;
        if (sp > g.cchunks) sp = g.cchunks;
        general = block * (double)((g.cchunks + sp - 1) / sp) * g.taps + 2000.0;
    } else {
        general = block * (double)((tiles + SMS - 1) / SMS) * blocks;
    }
    // up to 64 outputs the general kernel has little besides its blocks (batch x channels, us here / there: 8 x 320 -> 32 at
    // 64 x 64, stride 2 17.1 / 19.6; 16 x 256 -> 32 at 32 x 32 10.8 / 11.8; 8 x 640 -> 32 at 32 x 32 15.1 / 13.9; 15 x 992 -> 24 at 21 x 21
    // 19.8 / 16.6; 25 x 320 -> 48 at 15 x 15 11.6 / 13.0; 2 x 320 -> 64 at 30 x 30 9.7 / 8.6; 2 x 352 -> 40 at 28 x 28 9.8 / 8.0; and where it
    // cannot split the reduction 4 x 128 -> 8 at 59 x 59 7.8 / 8.4).  Of 144 drawn 3 x 3 layers with so few outputs seven take the
    // slower one by more than 3 %, at stride 1 by 8 % at most; with the margin of wider layers 16 do.
    if (p.N <= 64)
        return g.estimate <= general + (split && p.N <= 32 ? 0.0 : 1000.0);
    // (stride 2 in several rounds: 256 -> 1280 channels at 16 x 16, batch 57: 20.4 us there, 22.8 here)
    return g.estimate <= general + (p.stride > 1 && g.units > SMS / 2 ? 2000.0 : 4300.0);
}

fpq_status launch_pair_gemm(const GemmProblem& p, cudaStream_t st)
{
    static std::mutex mu;
    static EncodeTiledFn enc = nullptr;
    static bool attr_set[64] = {};
    static int sms[64] = {};
    int dev = 0, nsm = 0;
    {
        std::lock_guard<std::mutex> lock(mu);
        if (!enc) {
            enc = tensor_map_encoder();
            if (!enc)
                return FPQ_ERR_CUDA;
        }
        if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64)
            return FPQ_ERR_CUDA;
        if (!attr_set[dev]) {
            if (cudaFuncSetAttribute(fpq_pair_gemm_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BUDGET) !=
                    cudaSuccess ||
                cudaFuncSetAttribute(fpq_pair_gemm_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BUDGET) !=
                    cudaSuccess)
                return FPQ_ERR_CUDA;
            int v = 0;
            if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v < 2)
                v = 148;
            sms[dev] = v;
            attr_set[dev] = true;
        }
        nsm = sms[dev];
    }
    PGArgs g;
    int dyn = 0;
    const fpq_status planned = plan_pg(p, nsm, g, &dyn);
    if (planned != FPQ_OK)
        return planned;
    g.w_scale = p.w_scale;
    g.x_scale = p.x_scale;
    g.bias = p.bias;
    g.y = p.y;
    g.status = status_word();
    if (!g.status)
        return FPQ_ERR_CUDA;

    const bool phased = p.stride == 2;
    CUtensorMap tmA, tmB;
    if (phased) {
        // every second pixel of every second row of the zero-framed images
        const int Hp = p.H + 2 * p.pad;
        cuuint64_t dims[4] = {(cuuint64_t)p.Ca, (cuuint64_t)g.Wp, (cuuint64_t)Hp, (cuuint64_t)p.B};
        cuuint64_t strides[3] = {(cuuint64_t)p.Ca, (cuuint64_t)p.Ca * g.Wp, (cuuint64_t)p.Ca * g.Wp * Hp};
        cuuint32_t box[4] = {BK, (cuuint32_t)(2 * g.w2), (cuuint32_t)(2 * g.h2), (cuuint32_t)g.nb};
        cuuint32_t estr[4] = {1, 2, 2, 1};
        if (enc(&tmA, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, (void*)p.a_codes, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return FPQ_ERR_CUDA;
    } else {
        // activation codes: the zero-framed channels-last pixel list [B Hp Wp][Ca]
        cuuint64_t dims[4] = {(cuuint64_t)p.Ca, (cuuint64_t)g.M, 1, 1};
        cuuint64_t strides[3] = {(cuuint64_t)p.Ca, (cuuint64_t)p.Ca * (cuuint64_t)g.M, (cuuint64_t)p.Ca * (cuuint64_t)g.M};
        cuuint32_t box[4] = {BK, (cuuint32_t)g.a_box_rows, 1, 1};
        cuuint32_t estr[4] = {1, 1, 1, 1};
        if (enc(&tmA, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, (void*)p.a_codes, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return FPQ_ERR_CUDA;
    }
    {
        // prepared weights [N][taps][Cp]; a box = this CTA's half of a column tile for `tgroup` taps of one chunk
        cuuint64_t dims[3] = {(cuuint64_t)p.Cp, (cuuint64_t)p.N, (cuuint64_t)g.taps};
        const cuuint64_t rowB = p.w4 ? (cuuint64_t)p.Cp / 2 : (cuuint64_t)p.Cp;
        cuuint64_t strides[2] = {rowB * g.taps, rowB};
        cuuint32_t box[3] = {BK, (cuuint32_t)(g.BN / 2), phased ? 1u : (cuuint32_t)g.tgroup};
        cuuint32_t estr[3] = {1, 1, 1};
        if (enc(&tmB, p.w4 ? CU_TENSOR_MAP_DATA_TYPE_16U4_ALIGN16B : CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, (void*)p.w_prepared,
                dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return FPQ_ERR_CUDA;
    }
    int nclusters = nsm / 2;
    if (nclusters > g.units)
        nclusters = g.units;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(2 * nclusters));
    cfg.blockDim = dim3((unsigned)num_threads(phased));
    cfg.dynamicSmemBytes = (size_t)dyn;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, phased ? fpq_pair_gemm_kernel<true> : fpq_pair_gemm_kernel<false>, tmA, tmB,
                              (const PGArgs)g) == cudaSuccess ? FPQ_OK : FPQ_ERR_CUDA;
}

}  // namespace fpq
