// The low-bit contraction of a linear layer on CTA pairs (tcgen05 cta_group::2, M = 256), for long reductions: their time
// is the arrival of operands, some 45 bytes per clock and SM, and a pair fetches every weight byte once per 256 rows.
// Activation codes [M][Ca] come from the quantize kernel, weights from the prepared copy; both are streamed by TMA.
//
// Weights that are the sum of two terms share the activations: a stage of activation chunks serves the MMAs of both
// terms' weight chunks, so that the codes are written, and fetched, once.
//
// Per CTA: warp 0 activation producer (its own 128 rows), warp 10 weight producer (its half of the column tile), warp 1
// tensor-memory owner (and, in the pair's first CTA, the MMA issuer for both), warps 2-9 epilogue (tcgen05.ld ->
// acc * (x_scale * w_scale[n]) + bias[n] -> 32 x 32 blocks through swizzled staging and TMA stores).  Two accumulators.
// Every wait is bounded; no TMA multicast.
#include <cuda.h>

#include <mutex>

#include "fpq_common.cuh"
#include "fpq_kernels.h"
#include "fpq_tensormap.h"

namespace fpq {

namespace {

constexpr int BM = 128, BK = 128;
constexpr int EPI_W0 = 2, NUM_EPI = 8, B_WARP = EPI_W0 + NUM_EPI;
constexpr int NTHREADS = 32 * (B_WARP + 1);
constexpr int SMEM_BUDGET = 227 * 1024;
constexpr int EPI_STAGE = 8192;                // per epilogue warp: two 32 x 32 blocks
constexpr int EPI_SCALES = 2 * 128 * 4;        // per epilogue warp: scale and bias of its (up to 128) columns of a tile
constexpr int CTL = 512 + NUM_EPI * EPI_SCALES;

struct PRArgs {
    int64_t M;
    int N, BN;                 // outputs; column tile (a multiple of 32), BN / 2 weight rows per CTA
    int kc, terms, span;       // chunks of the reduction; weight terms; chunks per stage
    int n_tiles, units;        // a unit = (256 rows, column tile), column tile fastest
    FastDiv div_nt;
    int a_wide;                // a stage's activation chunks in one box
    int a_stage_bytes, a_stages, b_stage_bytes, b_stages;
    uint32_t b_tx;             // bytes one CTA's load of a weight stage reports
    uint32_t idesc, tmem_cols;
    int acc_bufs;
    int early_weights;
    bool narrowed;             // host side only: a wider tile would be faster, but two stages of it do not fit
    const float* w_scale;
    float x_scale;
    const float* bias;
    float* y;
    int* status;
};

__global__ void __launch_bounds__(NTHREADS, 1) fpq_pair_rows_kernel(const __grid_constant__ CUtensorMap tmA,
                                                                    const __grid_constant__ CUtensorMap tmB,
                                                                    const __grid_constant__ CUtensorMap tmY, const PRArgs g)
{
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* smem = smem_raw + (smem_base - smem_u32(smem_raw));
    // layout: [A ring][B ring][epilogue staging][barriers][scales]
    const uint32_t a_ring = smem_base;
    const uint32_t b_ring = a_ring + g.a_stages * g.a_stage_bytes;
    const uint32_t stage_off = g.a_stages * g.a_stage_bytes + g.b_stages * g.b_stage_bytes;
    const uint32_t ctl_off = stage_off + NUM_EPI * EPI_STAGE;
    const uint32_t bars = smem_base + ctl_off;
    const uint32_t a_full = bars, a_empty = bars + 64, b_full = bars + 128, b_empty = bars + 192;
    const uint32_t acc_full = bars + 256, acc_empty = bars + 272;
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem + ctl_off + 288);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank();
    const int cluster = (int)blockIdx.x >> 1, nclusters = (int)gridDim.x >> 1;
    // every cluster walks a contiguous range of units: consecutive units share their rows
    const int u_lo = (int)((int64_t)cluster * g.units / nclusters), u_hi = (int)((int64_t)(cluster + 1) * g.units / nclusters);

    if (warp == 0 && lane < 8) {
        mbar_init(a_full + 8 * lane, 1);
        mbar_init(a_empty + 8 * lane, 1);
        mbar_init(b_full + 8 * lane, 1);
        mbar_init(b_empty + 8 * lane, 1);
        if (lane < 2) {
            mbar_init(acc_full + 8 * lane, 1);
            mbar_init(acc_empty + 8 * lane, 2 * NUM_EPI);      // the epilogue warps of both CTAs
        }
        fence_barrier_init();
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
    // Nothing of global memory before the kernel in front is complete - but weights, when that one is the layer's own
    // quantize kernel (what wrote them was complete before it let this kernel start).
    if (!(g.early_weights && warp == B_WARP))
        asm volatile("griddepcontrol.wait;" ::: "memory");

    bool failed = false;                               // a wait of this thread's role ran out
    auto leader = [&](uint32_t bar) { return peer_smem_addr(bar, 0u); };

    if (warp == 0) {
        // ---------------- activation producer ----------------
        if (elect_one()) {
            uint32_t s = 0, ph = 1;
            bool dead = false;
            const uint32_t full = leader(a_full);
            for (int u = u_lo; u < u_hi && !dead; ++u) {
                const int row = (2 * (int)fdiv((uint32_t)u, g.div_nt) + (int)rank) * BM;
                for (int c = 0; c < g.kc; c += g.span) {
                    if (!mbar_wait(a_empty + 8 * s, ph)) { dead = true; break; }
                    const int loads = g.a_wide ? g.span : min(g.span, g.kc - c);
                    if (rank == 0)
                        mbar_expect_tx(a_full + 8 * s, 2u * (uint32_t)(loads * BM * BK));
                    const uint32_t dst = a_ring + s * g.a_stage_bytes;
                    if (g.a_wide) {
                        // (chunks past the last one read as zeros)
                        tma_load_4d_pair(dst, &tmA, full + 8 * s, 0, row, c, 0);
                    } else {
                        for (int l = 0; l < loads; ++l)
                            tma_load_4d_pair(dst + l * BM * BK, &tmA, full + 8 * s, (c + l) * BK, row, 0, 0);
                    }
                    if (++s == (uint32_t)g.a_stages) { s = 0; ph ^= 1; }
                }
            }
            settle_ring(a_full, a_empty, s, ph, g.a_stages, rank == 0, dead);
            failed = dead;
        }
    } else if (warp == B_WARP) {
        // ---------------- weight producer ----------------
        if (elect_one()) {
            uint32_t s = 0, ph = 1, issued = 0;
            bool dead = false;
            const uint32_t full = leader(b_full);
            for (int u = u_lo; u < u_hi && !dead; ++u) {
                const int mu = (int)fdiv((uint32_t)u, g.div_nt);
                const int n0 = (u - mu * g.n_tiles) * g.BN + (int)rank * (g.BN >> 1);
                for (int c = 0; c < g.kc && !dead; c += g.span)
                    for (int t = 0; t < g.terms; ++t) {
                        // (the limits of its waits start counting once the kernel in front has finished)
                        if (issued++ == (uint32_t)g.b_stages)
                            asm volatile("griddepcontrol.wait;" ::: "memory");
                        if (!mbar_wait(b_empty + 8 * s, ph)) { dead = true; break; }
                        if (rank == 0)
                            mbar_expect_tx(b_full + 8 * s, 2u * g.b_tx);
                        tma_load_4d_pair(b_ring + s * g.b_stage_bytes, &tmB, full + 8 * s, 0, n0, 0, t * g.kc + c);
                        if (++s == (uint32_t)g.b_stages) { s = 0; ph ^= 1; }
                    }
            }
            asm volatile("griddepcontrol.wait;" ::: "memory");
            settle_ring(b_full, b_empty, s, ph, g.b_stages, rank == 0, dead);
            failed = dead;
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer: one thread of the pair's first CTA ----------------
        if (rank == 0 && elect_one()) {
            uint32_t sa = 0, pa = 0, sb = 0, pb = 0, buf = 0, aph = 1;
            bool dead = false;
            const uint32_t HI = SMEM_DESC_HI_K_SW128;
            const uint32_t b_step = (uint32_t)g.BN * 4u;               // BN / 2 rows of 128 bytes, in 16-byte units
            for (int u = u_lo; u < u_hi && !dead; ++u) {
                if (!mbar_wait_cluster(acc_empty + 8 * buf, aph)) { dead = true; break; }
                tc_fence_after();
                const uint32_t d = tmem_base + buf * (uint32_t)g.BN;
                bool fresh = true;
                for (int c = 0; c < g.kc && !dead; c += g.span) {
                    const int count = min(g.span, g.kc - c);
                    if (!mbar_wait_cluster(a_full + 8 * sa, pa)) { dead = true; break; }
                    const uint32_t a0 = smem_desc_lo(a_ring + sa * g.a_stage_bytes);
                    for (int t = 0; t < g.terms; ++t) {
                        if (!mbar_wait_cluster(b_full + 8 * sb, pb)) { dead = true; break; }
                        tc_fence_after();
                        uint32_t al = a0, bl = smem_desc_lo(b_ring + sb * g.b_stage_bytes);
                        for (int j = 0; j < count; ++j, al += BM * BK / 16, bl += b_step) {
                            if (fresh)
                                mma_f8f6f4_pair<false>(d, al, bl, HI, g.idesc);
                            else
                                mma_f8f6f4_pair<true>(d, al, bl, HI, g.idesc);
                            fresh = false;
                            mma_f8f6f4_pair<true>(d, al + 2, bl + 2, HI, g.idesc);
                            mma_f8f6f4_pair<true>(d, al + 4, bl + 4, HI, g.idesc);
                            mma_f8f6f4_pair<true>(d, al + 6, bl + 6, HI, g.idesc);
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
        // ---------------- epilogue ----------------
        const int quarter = warp & 3, half = (warp - EPI_W0) >> 2;
        const uint32_t racc_empty = leader(acc_empty);
        uint8_t* stage0 = smem + stage_off + (warp - EPI_W0) * EPI_STAGE;
        float* w_sc = reinterpret_cast<float*>(smem + ctl_off + 512 + (warp - EPI_W0) * EPI_SCALES);
        uint32_t buf = 0, aph = 0, nstore = 0;
        bool dead = false;
        for (int u = u_lo; u < u_hi && !dead; ++u) {
            const int mu = (int)fdiv((uint32_t)u, g.div_nt);
            const int n0 = (u - mu * g.n_tiles) * g.BN;
            const int64_t row0 = (int64_t)(2 * mu + (int)rank) * BM + quarter * 32;
            // scales and biases of the warp's columns (every second 32 of the tile), fetched while the MMAs run
            __syncwarp();
            for (int c = 32 * half, k = 0; c < g.BN; c += 64, ++k) {
                const int col = n0 + c + lane;
                const bool in = col < g.N;
                w_sc[32 * k + lane] = in ? g.x_scale * __ldg(g.w_scale + col) : 0.f;
                w_sc[128 + 32 * k + lane] = in && g.bias ? __ldg(g.bias + col) : 0.f;
            }
            __syncwarp();
            if (!mbar_wait(acc_full + 8 * buf, aph)) { dead = true; break; }
            tc_fence_after();
            const uint32_t t_addr = tmem_base + buf * (uint32_t)g.BN + ((uint32_t)(quarter * 32) << 16);
            if (row0 < g.M) {
                for (int c = 32 * half, k = 0; c < g.BN && n0 + c < g.N; c += 64, ++k) {
                    uint32_t r[32];
                    tmem_ld32(t_addr + c, r);
                    tmem_ld_wait();
                    const float4* s4 = reinterpret_cast<const float4*>(w_sc + 32 * k);
                    const float4* b4 = reinterpret_cast<const float4*>(w_sc + 128 + 32 * k);
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        const float4 sv = s4[q], bv = b4[q];
                        r[4 * q + 0] = __float_as_uint(fmaf(__uint_as_float(r[4 * q + 0]), sv.x, bv.x));
                        r[4 * q + 1] = __float_as_uint(fmaf(__uint_as_float(r[4 * q + 1]), sv.y, bv.y));
                        r[4 * q + 2] = __float_as_uint(fmaf(__uint_as_float(r[4 * q + 2]), sv.z, bv.z));
                        r[4 * q + 3] = __float_as_uint(fmaf(__uint_as_float(r[4 * q + 3]), sv.w, bv.w));
                    }
                    uint8_t* stage = stage0 + (nstore & 1u) * 4096;
                    ++nstore;
                    if (lane == 0)
                        asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
                    __syncwarp();
#pragma unroll
                    for (int q = 0; q < 8; ++q)
                        *reinterpret_cast<uint4*>(stage + lane * 128 + ((q ^ (lane & 7)) << 4)) =
                            make_uint4(r[4 * q], r[4 * q + 1], r[4 * q + 2], r[4 * q + 3]);
                    if (g.N % 4) {
                        // rows start anywhere: 32 neighbouring floats of one per instruction (12263 x 1536 -> 2570, whole
                        // layer: 85.0 us with the general contraction, 71.9 here; 2048 x 2560 -> 638 14.0 and 12.6)
                        __syncwarp();
                        const int rows = (int)min((int64_t)32, g.M - row0);
                        float* dst = g.y + row0 * g.N + n0 + c + lane;
                        if (n0 + c + lane < g.N) {
#pragma unroll 8
                            for (int q = 0; q < rows; ++q, dst += g.N)
                                *dst = *reinterpret_cast<const float*>(stage + q * 128 + (((lane >> 2) ^ (q & 7)) << 4) + (lane & 3) * 4);
                        }
                        continue;
                    }
                    fence_proxy_async();
                    __syncwarp();
                    if (lane == 0) {
                        // (rows past M and columns past N are clipped by the tensor map)
                        asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];"
                                     ::"l"(&tmY), "r"(smem_u32(stage)), "r"(n0 + c), "r"((int)row0)
                                     : "memory");
                        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0 && u + g.acc_bufs < u_hi)                // (somebody waits for it)
                mbar_arrive_cluster(racc_empty + 8 * buf);
            if (++buf == (uint32_t)g.acc_bufs) { buf = 0; aph ^= 1; }
        }
        if (lane == 0)
            asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); // the staging must outlive its stores
        failed = dead;
    }

    // Nobody leaves while the other CTA may still arrive on its barriers.  Every arrival but a failed role's has been waited
    // for (the MMAs' last ones by the producers), so the barrier need not wait for the stores of the output: the next kernel's blocks move in that much earlier
    // (2048 x 2560 -> 640, whole layer: 13.5 -> 12.6 us).
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

// Column tile and rings; *cycles = the estimate of the launch.  False if out of range.
bool plan_rows(const GemmProblem& p, int terms, int nsm, PRArgs& g, double* cycles)
{
    if (p.conv || p.x != nullptr || p.c_seg != 0 || p.N < 4 || p.M < 1 || p.M > 0x7fffffff - 512 ||
        (uintptr_t)p.y % 16 != 0)
        return false;
    g = PRArgs{};
    g.M = p.M;
    g.N = p.N;
    g.terms = terms;
    g.kc = p.Cp / BK / terms;
    g.span = g.kc >= 2 ? 2 : 1;
    g.a_wide = p.Ca % BK == 0 ? 1 : 0;
    const int nclusters = nsm / 2;
    const int64_t m_units = (p.M + 2 * BM - 1) / (2 * BM);
    // A chunk takes its MMAs or the arrival of its operands; an epilogue stores some 21 bytes per clock and SM and is hidden
    // behind the next unit, except the last one's.  The tile that just fits columns and SM pairs wins, of those with two
    // stages of a chunk pair and all terms' weights (two terms: up to 160 columns).
    const int room = SMEM_BUDGET - 1024 - CTL - NUM_EPI * EPI_STAGE;
    double best = 0.0, best_any = 0.0;
    for (int bn = 32; bn <= 256; bn += 32) {
        if (bn - 32 >= p.N)
            break;
        const int64_t units = m_units * ((p.N + bn - 1) / bn);
        const double waves = (double)((units + nclusters - 1) / nclusters);
        const double mmas = g.terms * 4 * (bn * 0.53 > 52.0 ? bn * 0.53 : 52.0);
        const double fill = (BM * BK + g.terms * bn * 64.0) / 45.0;
        const double unit = 800.0 + g.kc * (mmas > fill ? mmas : fill), epi = 400.0 + BM * bn * 4 / 21.0;
        const double cost = waves * (waves > 1 && epi > unit ? epi : unit) + epi;
        if (best_any == 0.0 || cost < best_any)
            best_any = cost;
        if (2 * g.span * (BM * BK + terms * (bn / 2) * BK) <= room && (best == 0.0 || cost < best)) {
            best = cost;
            g.BN = bn;
        }
    }
    g.narrowed = best_any < best;
    *cycles = best;
    g.n_tiles = (p.N + g.BN - 1) / g.BN;
    g.div_nt = make_fastdiv((uint32_t)g.n_tiles);
    if (m_units * g.n_tiles > 0x7fffff00ll)
        return false;
    g.units = (int)(m_units * g.n_tiles);
    g.a_stage_bytes = g.span * BM * BK;
    g.b_stage_bytes = g.span * (g.BN / 2) * BK;
    g.b_tx = (uint32_t)g.b_stage_bytes / (p.w4 ? 2 : 1);
    // as many weight stages per activation stage as there are terms
    int n = room / (g.a_stage_bytes + terms * g.b_stage_bytes);
    if (n > 8 / terms) n = 8 / terms;
    if (n < 2)
        return false;
    g.a_stages = n;
    g.b_stages = n * terms;
    g.idesc = idesc_f8f6f4_pair(p.a_e5m2 ? 1u : 0u, p.w4 ? 5u : (p.w_e5m2 ? 1u : 0u), (uint32_t)g.BN);
    g.acc_bufs = 2;
    g.tmem_cols = 32;
    while ((int)g.tmem_cols < 2 * g.BN)
        g.tmem_cols *= 2;
    return true;
}

}  // namespace

// Measured against the general contraction (whole layers on B200).  One term: where 64-wide column tiles would already
// fill the GPU and the weights of a column tile do not stay resident there beside whole rows of stores: 640 -> 5120 at
// M = 16384 121.6 -> 85.6 us, 1344 -> 2944 at 33076 250 -> 200, 1280 -> 320 at 65536 116 -> 108; it loses with few tiles
// (1280 -> 1280 at 512: 7.6 -> 8.6) and to resident weights (640 -> 640 at 32768: 45.6 -> 46.6).  Two terms: from a few
// hundred rows on (320 -> 320 at 8192 13.0 -> 9.6, 2560 -> 640 at 2048 20.7 -> 16.1, 5120 -> 1280 at 128 12.6 -> 19.4).
// Where a wider tile than fits would be faster, only large layers of several rounds (codes written twice and one term's
// kernel / once and both terms': 320 -> 2560 at 65536 192 / 170, 2560 -> 2560 at 8192 136 / 99, 2560 -> 640 at 16384 109 / 83,
// 640 -> 5120 at 2048 23.3 / 21.6, 1152 -> 512 at 6985 20.7 / 17.6; in one round 2560 -> 2560 at 1024 18.6 / 19.5, 4928 -> 4192 at
// 425 23.6 / 24.7; small 320 -> 224 at 12215 10.5 / 11.2).
bool pair_rows_preferred(const GemmProblem& p, int terms)
{
    PRArgs g;
    double cycles;
    constexpr int SMS = 148;
    if (!plan_rows(p, terms, SMS, g, &cycles))
        return false;
    if (p.M <= 256)
        return false;
    if (terms > 1)
        return g.kc >= 3 && p.M * g.kc >= 2500 && (!g.narrowed || (g.units > SMS / 2 && p.M * p.N * g.kc >= 20000000));
    const int64_t m_tiles = (p.M + 127) / 128, n_tiles = (p.N + 127) / 128;
    const int64_t col_grid = SMS / n_tiles * n_tiles;
    const bool resident = n_tiles > 1 && col_grid * 10 >= SMS * 9 && g.kc <= 5;
    return g.kc >= 4 && !resident && m_tiles * ((p.N + 63) / 64) > SMS && (m_tiles * n_tiles > SMS || g.kc >= 12);
}

fpq_status launch_pair_rows(const GemmProblem& p, int terms, cudaStream_t st)
{
    static std::mutex mu;
    static int sms[64] = {};
    EncodeTiledFn enc = tensor_map_encoder();
    int dev = 0, nsm = 0;
    if (!enc || cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64)
        return FPQ_ERR_CUDA;
    {
        std::lock_guard<std::mutex> lock(mu);
        if (!sms[dev]) {
            int v = 0;
            if (cudaFuncSetAttribute(fpq_pair_rows_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BUDGET) != cudaSuccess)
                return FPQ_ERR_CUDA;
            if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v < 2)
                v = 148;
            sms[dev] = v;
        }
        nsm = sms[dev];
    }
    PRArgs g;
    double cycles;
    if (!plan_rows(p, terms, nsm, g, &cycles))
        return FPQ_ERR_UNSUPPORTED;
    g.w_scale = p.w_scale;
    g.x_scale = p.x_scale;
    g.bias = p.bias;
    g.y = p.y;
    g.early_weights = p.after_stage1;
    g.status = status_word();
    if (!g.status)
        return FPQ_ERR_CUDA;
    CUtensorMap tmA, tmB, tmY;
    cuuint32_t estr[4] = {1, 1, 1, 1};
    {
        // rows of whole chunks: (position in chunk, row, chunk), a stage's chunks in one box; else one box per chunk
        const cuuint64_t ca = (cuuint64_t)p.Ca, m = (cuuint64_t)p.M;
        cuuint64_t wide[4] = {(cuuint64_t)BK, m, ca / BK, 1}, wide_s[3] = {ca, (cuuint64_t)BK, ca * m};
        cuuint64_t flat[4] = {ca, m, 1, 1}, flat_s[3] = {ca, ca * m, ca * m};
        cuuint32_t box[4] = {BK, BM, g.a_wide ? (cuuint32_t)g.span : 1u, 1};
        if (enc(&tmA, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, (void*)p.a_codes, g.a_wide ? wide : flat, g.a_wide ? wide_s : flat_s, box,
                estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return FPQ_ERR_CUDA;
    }
    {
        const cuuint64_t row = p.w4 ? (cuuint64_t)p.Cp / 2 : (cuuint64_t)p.Cp;
        cuuint64_t dims[4] = {(cuuint64_t)BK, (cuuint64_t)p.N, 1, (cuuint64_t)(p.Cp / BK)};
        cuuint64_t strides[3] = {row, row, p.w4 ? (cuuint64_t)BK / 2 : (cuuint64_t)BK};
        cuuint32_t box[4] = {BK, (cuuint32_t)(g.BN / 2), 1, (cuuint32_t)g.span};
        if (enc(&tmB, p.w4 ? CU_TENSOR_MAP_DATA_TYPE_16U4_ALIGN16B : CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, (void*)p.w_prepared, dims,
                strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return FPQ_ERR_CUDA;
    }
    tmY = tmA;
    if (p.N % 4 == 0) {
        cuuint64_t dims[2] = {(cuuint64_t)p.N, (cuuint64_t)p.M};
        cuuint64_t strides[1] = {(cuuint64_t)p.N * 4};
        cuuint32_t box[2] = {32, 32};
        if (enc(&tmY, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, (void*)p.y, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return FPQ_ERR_CUDA;
    }
    int nclusters = nsm / 2;
    if (nclusters > g.units)
        nclusters = g.units;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(2 * nclusters));
    cfg.blockDim = dim3(NTHREADS);
    cfg.dynamicSmemBytes = (size_t)(1024 + CTL + NUM_EPI * EPI_STAGE + g.a_stages * g.a_stage_bytes + g.b_stages * g.b_stage_bytes);
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
    return cudaLaunchKernelEx(&cfg, fpq_pair_rows_kernel, tmA, tmB, tmY, (const PRArgs)g) == cudaSuccess ? FPQ_OK : FPQ_ERR_CUDA;
}

}  // namespace fpq
