// Dense bf16 projections of the block (Q', K/V over all latents, output
// projections, FFN on the active latents; Sec. 3.3) on the 5th-generation
// tensor cores:  out = act(A W^T + bias) + resid.
//
// Persistent CTA pairs: a cluster of two CTAs on two SMs walks 256 x BN output
// tiles (BN 256, or 128 for small outputs) in a banded order and computes each
// with tcgen05.mma.cta_group::2 (M 256, N BN, K 16): the even CTA holds rows
// 0..127 of the tile, the odd CTA rows 128..255, and each holds one half of the W
// tile, so each SM loads 32 KB per 64-deep k-block (BN 256) instead of the 48 KB
// of a one-SM 128 x 256 tile.  12 warps per CTA:
//   warp 0      TMA producer: the CTA's A [128 x 64] and W-half [BN/2 x 64] bf16
//               tiles, 128-byte swizzle, into a ring of 6 (BN 256) or 8 stages;
//               both CTAs' copies complete their bytes on the even CTA's barrier;
//   warp 1      (even CTA) one elected lane issues the pair MMAs into one of two
//               BN-column fp32 accumulators (the same columns in both CTAs) and
//               commits each stage back to both producers, so the epilogue of one
//               tile overlaps the main loop of the next;
//   warp 2      allocates / frees the tensor-memory columns of the pair;
//   warps 4..11 epilogue, in each CTA (warp w reads TMEM lanes 32 (w mod 4) .. and
//               one half of the columns): 32 x 32 blocks through shared memory, so
//               that bias, GELU, residual and the stores run on whole row segments
//               (8 lanes a row).  A row per lane instead, with four warps, took as
//               long as the main loop of a 1024-deep tile: 1560 x 1024 x 1024 with
//               an fp32 residual 19.1 -> 10.6 us, 20000 x 768 x 768 94 -> 43 us,
//               6552 x 5120 x 5120 221 -> 196 us.
// Every mbarrier wait is bounded (ECHO_ERR_TIMEOUT); a CTA that gives up lets its
// copies land and drains its MMAs before it frees tensor memory, and a cluster
// barrier keeps either CTA from leaving while the other may still reach it.
#include "common.cuh"
#include "internal.h"

namespace {

constexpr int BM = 128, BK = 64;             // BM: rows per CTA of a pair tile
constexpr int A_BYTES = BM * BK * 2;         // 16 KB
constexpr int EPI_WARPS = 8;
constexpr int STG_BYTES = 32 * 32 * 4;       // one 32 x 32 fp32 block per epilogue warp
constexpr int THREADS = 128 + 32 * EPI_WARPS;
constexpr int BAND_COLS = 4096;              // output columns per raster band

template <int BN>
struct Cfg {
    static constexpr int HB_BYTES = (BN / 2) * BK * 2;   // half of a W tile
    static constexpr int STAGE_BYTES = A_BYTES + HB_BYTES;
    static constexpr int STAGES = BN == 256 ? 6 : 8;
    static constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + EPI_WARPS * STG_BYTES + 1024;
    static constexpr uint32_t TMEM_COLS = 2 * BN;        // two accumulators
    static constexpr int GROUP_N = BAND_COLS / BN;       // N tiles per raster band
    static constexpr uint32_t IDESC = idesc_bf16_f32(2 * BM, BN);
};

// EPI_ROWAMAX: also fold max |v| of each bf16 output row into row_amax (fp32
// bits, atomic max over the row's column tiles; a NaN beats every number)
enum : int { EPI_GELU = 1, EPI_RES_BF16 = 2, EPI_RES_F32 = 4, EPI_OUT_F32 = 8, EPI_ROWAMAX = 16 };

struct GemmParams {
    int M, N, Kd;
    const __nv_bfloat16 *bias;
    const void *resid;
    const int32_t *resid_rows;
    void *out;
    int64_t ldo;
    const int32_t *out_rows;   // output row m goes to row out_rows[m] (NULL: m)
    uint32_t *row_amax;
    int *err;
};

ECHO_DEV float gelu_tanh(float x) {
    const float k0 = 0.7978845608028654f;  // sqrt(2 / pi)
    const float u = k0 * (x + 0.044715f * x * x * x);
    return 0.5f * x * (1.f + tanhf(u));
}

// Tile order: bands of BAND_COLS columns; inside a band M is swept with the
// band's N-tiles adjacent, so the CTAs in flight share a few A row blocks and one
// band of W, which stay in L2 while the band is processed.
template <int BN>
ECHO_DEV void tile_coords(int t, int num_m, int num_n, int &mt, int &nt) {
    constexpr int GROUP_N = Cfg<BN>::GROUP_N;
    const int band = t / (GROUP_N * num_m);
    const int first_n = band * GROUP_N;
    const int gn = min(GROUP_N, num_n - first_n);
    const int r = t - band * GROUP_N * num_m;
    mt = r / gn;
    nt = first_n + r % gn;
}

// GELU of a value that is rounded to bf16: x (1 + tanh u) / 2 = x / (1 + 2^w),
// w = -2 u log2(e).  About 8 instructions where tanhf takes about 30, with which an
// epilogue outlasted a 1024-deep main loop (7800 x 4096 x 1024: 56.6 us).  Before the
// rounding its error against 64 bits is 5e-8 of the norm, tanhf's 4e-8; after it, of
// 200000 normal values of deviation 1 (3), 1 (43) are not the bf16 next to the exact
// one, where tanhf leaves 10 (15278, from the cancellation in 1 + tanh u of negative
// x).  fp32 outputs keep tanhf.  Infinities and NaN come out alike.
ECHO_DEV float gelu_tanh_bf16(float x) {
    const float c1 = -2.3022081986f;   // -2 sqrt(2 / pi) log2(e)
    const float c2 = -0.1029432397f;   // 0.044715 c1
    return __fdividef(x, 1.f + ex2_approx(x * fmaf(c2, x * x, c1)));
}

// One warp's 32 rows x COLS columns of a tile, 32 columns at a time: tcgen05.ld
// (a row per lane), through the warp's staging block (16-byte chunks XOR-swizzled
// by the row, so that both sides spread over the banks), then 8 lanes per row
// with 4 columns each: bias, GELU, residual and store run on whole row segments.
// What can be read early is: the bias and the first block's residual before the
// accumulator is waited for (`wait`), the next block's residual a block ahead;
// the staged block comes back in one batch of loads.  `release` is called once,
// as soon as the last of the accumulator has been read; it must not wait for the
// stores (a releasing arrive did, 1200 to 2000 cycles a tile).  A 256-column
// tile's epilogue takes about 7000 cycles (10000 before), less than the main loop
// of a 1024-deep tile: 7800 x 2048 x 1024 30.3 -> 25.5 us.  False: `wait` gave up.
template <int EPI, int COLS, typename Wait, typename Release>
ECHO_DEV bool epilogue_rows(const GemmParams &p, uint32_t tacc, uint8_t *stage, int row0, int n0,
                            Wait wait, Release release) {
    const int lane = threadIdx.x & 31, sub = lane >> 3, cc = lane & 7;
    const bool lane_ok = row0 + lane < p.M;
    int orow = row0 + lane, rrow = row0 + lane;   // of the warp's row `lane`
    if (p.out_rows && lane_ok) orow = p.out_rows[row0 + lane];
    if ((EPI & EPI_RES_BF16) && p.resid_rows && lane_ok) rrow = p.resid_rows[row0 + lane];
    // the bias of the COLS (<= 128) columns, 4 per lane; lane (c / 4 + cc) holds a
    // block's columns c + 4 cc ..
    uint2 bias_all = make_uint2(0, 0);
    if (p.bias && 4 * lane < min(COLS, p.N - n0))
        bias_all = __ldg(reinterpret_cast<const uint2 *>(p.bias + n0 + 4 * lane));
    int out_row[8], res_row[8];                   // rows 4 i + sub
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        out_row[i] = __shfl_sync(0xffffffffu, orow, 4 * i + sub);
        if (EPI & EPI_RES_BF16) res_row[i] = __shfl_sync(0xffffffffu, rrow, 4 * i + sub);
        else res_row[i] = row0 + 4 * i + sub;
    }
    const int rows_left = p.M - row0 - sub;       // row 4 i + sub exists: 4 i < rows_left
    float4 rf[8];
    uint2 rb[8];
    auto fetch = [&](int c, float4 *f, uint2 *h) {   // residual of the block at column c
        const int64_t col = n0 + c + 4 * cc;
        if (EPI & EPI_RES_F32) {
#pragma unroll
            for (int i = 0; i < 8; ++i)
                f[i] = 4 * i < rows_left ? __ldg(reinterpret_cast<const float4 *>(
                                               static_cast<const float *>(p.resid) +
                                               (int64_t)res_row[i] * p.N + col))
                                         : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        if (EPI & EPI_RES_BF16) {
#pragma unroll
            for (int i = 0; i < 8; ++i)
                h[i] = 4 * i < rows_left
                           ? __ldg(reinterpret_cast<const uint2 *>(
                                 static_cast<const __nv_bfloat16 *>(p.resid) +
                                 (int64_t)res_row[i] * p.N + col))
                           : make_uint2(0, 0);
        }
    };
    const int cols = min(COLS, p.N - n0);         // a multiple of 32, or <= 0
    if (cols > 0) fetch(0, rf, rb);
    if (!wait()) return false;
    if (cols <= 0) release();
    uint32_t rmax[8] = {0, 0, 0, 0, 0, 0, 0, 0};  // EPI_ROWAMAX: max |v| of rows 4 i + sub, as bits
#pragma unroll 1
    for (int c = 0; c < cols; c += 32) {
        float4 rf_next[8];
        uint2 rb_next[8];
        if (c + 32 < cols) fetch(c + 32, rf_next, rb_next);
        {
            uint32_t r[32];
            tmem_ld32(tacc + (uint32_t)c, r);
            tmem_ld_wait();
            if (c + 32 >= cols) release();
            __syncwarp();                         // the previous block has been read
#pragma unroll
            for (int k = 0; k < 8; ++k)
                *reinterpret_cast<uint4 *>(stage + lane * 128 + ((k ^ (lane & 7)) * 16)) =
                    make_uint4(r[4 * k], r[4 * k + 1], r[4 * k + 2], r[4 * k + 3]);
        }
        __syncwarp();
        float v[8][4];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int lr = 4 * i + sub;
            const float4 a = *reinterpret_cast<const float4 *>(stage + lr * 128 + ((cc ^ (lr & 7)) * 16));
            v[i][0] = a.x; v[i][1] = a.y; v[i][2] = a.z; v[i][3] = a.w;
        }
        const uint32_t b01 = __shfl_sync(0xffffffffu, bias_all.x, (c >> 2) + cc);
        const uint32_t b23 = __shfl_sync(0xffffffffu, bias_all.y, (c >> 2) + cc);
        const float bias[4] = {bf16lo(b01), bf16hi(b01), bf16lo(b23), bf16hi(b23)};
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            if (p.bias) {
#pragma unroll
                for (int e = 0; e < 4; ++e) v[i][e] += bias[e];
            }
            if (EPI & EPI_GELU) {
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    v[i][e] = (EPI & EPI_OUT_F32) ? gelu_tanh(v[i][e]) : gelu_tanh_bf16(v[i][e]);
            }
            if (EPI & EPI_RES_BF16) {
                v[i][0] += bf16lo(rb[i].x); v[i][1] += bf16hi(rb[i].x);
                v[i][2] += bf16lo(rb[i].y); v[i][3] += bf16hi(rb[i].y);
            }
            if (EPI & EPI_RES_F32) {
                v[i][0] += rf[i].x; v[i][1] += rf[i].y; v[i][2] += rf[i].z; v[i][3] += rf[i].w;
            }
        }
        const int64_t col = n0 + c + 4 * cc;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            if (EPI & EPI_OUT_F32) {
                if (4 * i < rows_left)
                    *reinterpret_cast<float4 *>(static_cast<float *>(p.out) + (int64_t)out_row[i] * p.ldo + col) =
                        make_float4(v[i][0], v[i][1], v[i][2], v[i][3]);
            } else {
                const uint2 w = make_uint2(pack_bf16(v[i][0], v[i][1]), pack_bf16(v[i][2], v[i][3]));
                if (4 * i < rows_left)
                    *reinterpret_cast<uint2 *>(static_cast<__nv_bfloat16 *>(p.out) +
                                               (int64_t)out_row[i] * p.ldo + col) = w;
                if (EPI & EPI_ROWAMAX)
                    rmax[i] = max(rmax[i], max(max((w.x & 0x7FFFu) << 16, w.x & 0x7FFF0000u),
                                               max((w.y & 0x7FFFu) << 16, w.y & 0x7FFF0000u)));
            }
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            if (EPI & EPI_RES_F32) rf[i] = rf_next[i];
            if (EPI & EPI_RES_BF16) rb[i] = rb_next[i];
        }
    }
    if (EPI & EPI_ROWAMAX) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
#pragma unroll
            for (int s = 1; s < 8; s *= 2)
                rmax[i] = max(rmax[i], __shfl_xor_sync(0xffffffffu, rmax[i], s));
            if (cc == 0 && 4 * i < rows_left) atomicMax(&p.row_amax[row0 + 4 * i + sub], rmax[i]);
        }
    }
    return true;
}

// DUAL: a second projection of the same depth (A2 W2^T, p2) continues the tile
// list; its tiles fill the wave that the first one's leave part empty.
template <int EPI, int BN, bool DUAL>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(THREADS, 1)
gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
            const __grid_constant__ CUtensorMap tmA2, const __grid_constant__ CUtensorMap tmB2,
            const __grid_constant__ GemmParams p, const __grid_constant__ GemmParams p2) {
    using C = Cfg<BN>;
    constexpr int STAGES = C::STAGES, STAGE_BYTES = C::STAGE_BYTES;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                ~static_cast<uintptr_t>(1023));
    __shared__ __align__(8) uint64_t full_bar[STAGES], empty_bar[STAGES];
    __shared__ __align__(8) uint64_t acc_full[2], acc_empty[2], drain_bar;
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();
    const int pair = blockIdx.x >> 1, num_pairs = gridDim.x >> 1;
    const int num_kb = p.Kd / BK;
    const int num_m = (p.M + 2 * BM - 1) / (2 * BM), num_n = (p.N + BN - 1) / BN;
    const int tiles1 = num_m * num_n;
    const int num_m2 = DUAL ? (p2.M + 2 * BM - 1) / (2 * BM) : 0;
    const int num_n2 = DUAL ? (p2.N + BN - 1) / BN : 0;
    const int num_tiles = tiles1 + num_m2 * num_n2;
    auto coords = [&](int t, int &mt, int &nt) {
        if (DUAL && t >= tiles1) tile_coords<BN>(t - tiles1, num_m2, num_n2, mt, nt);
        else tile_coords<BN>(t, num_m, num_n, mt, nt);
    };
    // Arrivals that nothing waits for are left out (the ring slots of the last
    // STAGES k-blocks, the accumulators of the last two tiles): they may land after
    // this CTA has left, on the barriers that the next kernel has set up there.
    const int my_tiles = (num_tiles - pair + num_pairs - 1) / num_pairs;
    const int my_kbs = my_tiles * num_kb;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&full_bar[s], 1);    // used in the even CTA
            mbar_init(&empty_bar[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], 2 * EPI_WARPS);   // lane 0 of both CTAs' epilogue warps
        }
        mbar_init(&drain_bar, 1);
        abort_flag = 0;
        fence_barrier_init();
        tma_prefetch_desc(&tmA);
        tma_prefetch_desc(&tmB);
        if (DUAL) {
            tma_prefetch_desc(&tmA2);
            tma_prefetch_desc(&tmB2);
        }
    }
    cluster_sync_all();   // both CTAs' barriers exist before any arrival from the other CTA
    if (warp == 2) tmem_alloc_pair(&tmem_slot, C::TMEM_COLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;
    volatile int *abort_v = &abort_flag;
    pdl_enter();   // set up: from here on global memory is read and written

    if (warp == 0 && lane == 0) {
        // ---------------- TMA producer (both CTAs) ----------------
        // A stage is refilled only after the pair's MMAs of its previous use are
        // done (both producers see the same commit), so the bytes of one use
        // never mix with the next on the even CTA's barrier.
        const uint32_t full0 = mapa_shared(smem_u32(&full_bar[0]), 0);
        int it = 0;
        bool ok = true;
        for (int t = pair; ok && t < num_tiles; t += num_pairs) {
            int mt, nt;
            coords(t, mt, nt);
            const CUtensorMap *ma = DUAL && t >= tiles1 ? &tmA2 : &tmA;
            const CUtensorMap *mb = DUAL && t >= tiles1 ? &tmB2 : &tmB;
            for (int kb = 0; kb < num_kb; ++kb, ++it) {
                const int s = it % STAGES;
                if (!mbar_wait_cluster(&empty_bar[s], ((it / STAGES) & 1) ^ 1, abort_v, p.err)) {
                    ok = false;
                    break;
                }
                uint8_t *a = smem + s * STAGE_BYTES;
                const uint32_t bar = full0 + (uint32_t)(s * sizeof(uint64_t));
                if (rank == 0) mbar_arrive_expect_tx(&full_bar[s], 2 * STAGE_BYTES);
                tma_load_2d_pair(a, ma, bar, kb * BK, mt * 2 * BM + (int)rank * BM);
                tma_load_2d_pair(a + A_BYTES, mb, bar, kb * BK, nt * BN + (int)rank * (BN / 2));
            }
        }
        if (*abort_v) {  // let this CTA's copies land before it exits
            if (rank == 0) {
                for (int k = it - STAGES < 0 ? 0 : it - STAGES; k < it; ++k)
                    mbar_wait(&full_bar[k % STAGES], (k / STAGES) & 1, abort_v, nullptr, 100000000ull);
            } else {   // its copies complete on the other CTA's barrier: give them time
                const uint64_t t0 = globaltimer_ns();
                while (globaltimer_ns() - t0 < 200000ull) {
                }
            }
        }
    } else if (warp == 1 && rank == 0) {
        // ---------------- MMA issuer (even CTA) ----------------
        // The whole warp runs the loop (stage arithmetic and descriptors stay
        // warp-uniform) and one elected lane issues the MMAs and commits.
        // Descriptor words: the low word holds the start address in 16-byte
        // units (leading byte offset unused for K-major), the high word the
        // 1024-byte stride of eight 128-byte rows, the version and the 128-byte
        // swizzle; a K step of 16 adds 32 bytes to the start address.  The same
        // offsets address the odd CTA's halves.
        const bool leader = elect_one_sync();
        constexpr uint32_t DESC_HI = (1024u >> 4) | (1u << 14) | (2u << 29);
        const uint32_t smem_lo = ((smem_u32(smem) & 0x3FFFFu) >> 4) | (1u << 16);
        auto desc = [](uint32_t lo) -> uint64_t { return ((uint64_t)DESC_HI << 32) | lo; };
        bool ok = true;
        int it = 0, local = 0;
        for (int t = pair; ok && t < num_tiles; t += num_pairs, ++local) {
            const int buf = local & 1;
            if (!__all_sync(0xffffffffu, mbar_wait_cluster(&acc_empty[buf], ((local >> 1) & 1) ^ 1,
                                                           abort_v, p.err))) {
                ok = false;
                break;
            }
            tc_fence_after();
            const uint32_t d_tmem = tmem + (uint32_t)(buf * BN);
            for (int kb = 0; kb < num_kb; ++kb, ++it) {
                const int s = it % STAGES;
                if (!__all_sync(0xffffffffu,
                                mbar_wait_cluster(&full_bar[s], (it / STAGES) & 1, abort_v, p.err))) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t a_lo = smem_lo + (uint32_t)(s * (STAGE_BYTES >> 4));
                const uint32_t b_lo = a_lo + (uint32_t)(A_BYTES >> 4);
                if (leader) {
#pragma unroll
                    for (int k = 0; k < BK / 16; ++k)
                        tc_mma_pair_f16(d_tmem, desc(a_lo + 2 * k), desc(b_lo + 2 * k), C::IDESC,
                                        (kb | k) != 0);
                    if (it + STAGES < my_kbs)
                        tc_commit_pair(&empty_bar[s], 0x3);   // the stage is free in both CTAs
                }
                __syncwarp();
            }
            if (ok && leader) tc_commit_pair(&acc_full[buf], 0x3);
            __syncwarp();
        }
        if (!ok && leader) {  // wait for the MMAs already issued before tensor memory is freed
            tc_commit_pair(&drain_bar, 0x1);
            mbar_wait(&drain_bar, 0, abort_v, nullptr, 100000000ull);
        }
    } else if (warp >= 4) {
        // ---------------- epilogue (both CTAs) ----------------
        // two warps per TMEM lane quarter, each with half of the columns
        const int q = warp & 3, half = (warp - 4) >> 2;
        const uint32_t lane_base = (uint32_t)(q * 32) << 16;
        uint8_t *stage = smem + STAGES * STAGE_BYTES + (warp - 4) * STG_BYTES;
        const uint32_t empty_even[2] = {mapa_shared(smem_u32(&acc_empty[0]), 0),
                                        mapa_shared(smem_u32(&acc_empty[1]), 0)};
        int local = 0;
        for (int t = pair; t < num_tiles; t += num_pairs, ++local) {
            const int buf = local & 1;
            int mt, nt;
            coords(t, mt, nt);
            const bool ok = epilogue_rows<EPI, BN / 2>(
                DUAL && t >= tiles1 ? p2 : p, tmem + lane_base + (uint32_t)(buf * BN + half * (BN / 2)), stage,
                mt * 2 * BM + (int)rank * BM + q * 32, nt * BN + half * (BN / 2),
                [&]() {
                    const bool w = __all_sync(0xffffffffu,
                                              mbar_wait_cluster(&acc_full[buf], (local >> 1) & 1,
                                                                abort_v, p.err, 4000000000ull));
                    tc_fence_after();
                    return w;
                },
                [&]() {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0 && local + 2 < my_tiles) mbar_arrive_remote_relaxed(empty_even[buf]);
                });
            if (!ok) break;
        }
    }
    tc_fence_before();
    __syncwarp();
    cluster_sync_all();   // neither CTA leaves while the other may still reach its memory
    if (warp == 2) {
        tc_fence_after();
        tmem_dealloc_pair(tmem, C::TMEM_COLS);
    }
}

int num_sms() {
    static int cached[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 1;
    if (!cached[dev]) {
        int n = 0;
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        cached[dev] = n > 0 ? n : 1;
    }
    return cached[dev];
}

// tensor maps and parameters of one projection
struct Problem {
    CUtensorMap a, b;
    GemmParams p;
};

template <int EPI, int BN, bool DUAL>
echo_status run_bn(const Problem &x, const Problem &y, cudaStream_t st) {
    static int pairs_max[64] = {};   // per device: co-resident CTA pairs (0: not set up yet)
    constexpr int SMEM_BYTES = Cfg<BN>::SMEM_BYTES;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return ECHO_ERR_CUDA;
    if (!pairs_max[dev]) {   // a benign race computes the same value twice
        if (cudaFuncSetAttribute(gemm_kernel<EPI, BN, DUAL>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 SMEM_BYTES) != cudaSuccess)
            return ECHO_ERR_CUDA;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(2 * num_sms(), 1, 1);
        cfg.blockDim = dim3(THREADS, 1, 1);
        cfg.dynamicSmemBytes = SMEM_BYTES;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, gemm_kernel<EPI, BN, DUAL>, &cfg) != cudaSuccess || n < 1)
            return ECHO_ERR_CUDA;
        pairs_max[dev] = n;
    }
    auto tiles_of = [](const GemmParams &p) {
        return ((p.M + 2 * BM - 1) / (2 * BM)) * ((p.N + BN - 1) / BN);
    };
    const int tiles = tiles_of(x.p) + (DUAL ? tiles_of(y.p) : 0);
    const int pairs = tiles < pairs_max[dev] ? tiles : pairs_max[dev];
    // two projections count as one with the rows that give the same operations
    const int64_t m = x.p.M + (DUAL ? (int64_t)y.p.M * y.p.N / x.p.N : 0);
    echo::LaunchScope ls(ECHO_K_GEMM, m, x.p.N, x.p.Kd, st);
    echo::launch_chained(gemm_kernel<EPI, BN, DUAL>, dim3(2 * pairs), dim3(THREADS), SMEM_BYTES, st, x.a,
                         x.b, y.a, y.b, x.p, y.p);
    return echo::last_launch_status();
}

// Tile width, by the cycles of the waves with every SM pair at work: a 64-deep k-block
// of 256 columns takes 512 (0.262 us), of 128 columns 440 (0.225 us: the copies into
// shared memory, which the pairs share the L2 for), plus a tile's own part and the
// last tile's epilogue, which nothing overlaps.  So 128 columns gain where they spread
// a small output over pairs that would be idle, or save most of a wave.  Of 3901
// measured calls (M 16 .. 20000, N 128 .. 13824, depth 128 .. 5120; plain, GELU, fp32
// residual) the choice is 0.1% from the better width on average; by more than 8% it
// is 12 times (16 rows at depth 3072; GELU or a residual at depth 512, 3 waves for 2).
// 256 against 128 columns: 1560 x 1024 x 1024 9.8 and 8.6 us, 1560 x 1024 x 4096 22.5
// and 19.7, 400 x 640 x 2048 13.8 and 11.3; 1560 x 4096 x 1024 14.9 and 17.3, 2560 x
// 2048 x 5120 48.6 and 60.3, 600 x 5120 x 5120 28.1 and 41.8.
bool narrow_tiles(int M, int N, int Kd, int M2 = 0, int N2 = 0) {
    const int64_t pairs = num_sms() / 2, kb = Kd / BK;
    const int64_t nm = (M + 2 * BM - 1) / (2 * BM), nm2 = (M2 + 2 * BM - 1) / (2 * BM);
    const int64_t w256 = (nm * ((N + 255) / 256) + nm2 * ((N2 + 255) / 256) + pairs - 1) / pairs;
    const int64_t w128 = (nm * ((N + 127) / 128) + nm2 * ((N2 + 127) / 128) + pairs - 1) / pairs;
    return w128 * (kb * 440 + 900) < w256 * (kb * 512 + 1800) + 500;
}

bool make_problem(const echo::LinearArgs &a, bool narrow, Problem &x) {
    GemmParams &p = x.p;
    p.M = a.M; p.N = a.N; p.Kd = a.Kd;
    p.bias = static_cast<const __nv_bfloat16 *>(a.bias);
    p.resid = a.resid;
    p.resid_rows = a.resid_rows;
    p.out = a.out;
    p.ldo = a.ldo;
    p.out_rows = a.out_rows;
    p.row_amax = a.row_amax;
    p.err = echo::device_error_ptr();
    return echo::make_tmap_bf16(&x.a, a.A, (uint64_t)a.M, (uint64_t)a.Kd, (uint64_t)a.lda, BM) &&
           echo::make_tmap_bf16(&x.b, a.W, (uint64_t)a.N, (uint64_t)a.Kd, (uint64_t)a.Kd,
                                narrow ? 64 : 128);
}

template <int EPI>
echo_status run(const echo::LinearArgs &a, cudaStream_t st) {
    const bool narrow = narrow_tiles(a.M, a.N, a.Kd);
    Problem x;
    if (!make_problem(a, narrow, x)) return ECHO_ERR_CUDA;
    return narrow ? run_bn<EPI, 128, false>(x, x, st) : run_bn<EPI, 256, false>(x, x, st);
}

}  // namespace

namespace echo {

echo_status launch_linear(const LinearArgs &a, cudaStream_t st) {
    if (a.M <= 0) return ECHO_OK;
    int epi = 0;
    if (a.act == 1) epi |= EPI_GELU;
    if (a.resid) epi |= (a.resid_t == ECHO_BF16) ? EPI_RES_BF16 : EPI_RES_F32;
    if (a.out_t == ECHO_F32) epi |= EPI_OUT_F32;
    if (a.row_amax) {
        if (epi != EPI_RES_F32) return ECHO_ERR_INVALID_ARG;   // bf16 out, fp32 residual only
        return run<EPI_RES_F32 | EPI_ROWAMAX>(a, st);
    }
    switch (epi) {
        case 0: return run<0>(a, st);
        case EPI_GELU: return run<EPI_GELU>(a, st);
        case EPI_RES_BF16: return run<EPI_RES_BF16>(a, st);
        case EPI_RES_F32: return run<EPI_RES_F32>(a, st);
        case EPI_GELU | EPI_RES_BF16: return run<EPI_GELU | EPI_RES_BF16>(a, st);
        case EPI_GELU | EPI_RES_F32: return run<EPI_GELU | EPI_RES_F32>(a, st);
        case EPI_OUT_F32: return run<EPI_OUT_F32>(a, st);
        case EPI_GELU | EPI_OUT_F32: return run<EPI_GELU | EPI_OUT_F32>(a, st);
        case EPI_RES_BF16 | EPI_OUT_F32: return run<EPI_RES_BF16 | EPI_OUT_F32>(a, st);
        case EPI_RES_F32 | EPI_OUT_F32: return run<EPI_RES_F32 | EPI_OUT_F32>(a, st);
        case EPI_GELU | EPI_RES_BF16 | EPI_OUT_F32:
            return run<EPI_GELU | EPI_RES_BF16 | EPI_OUT_F32>(a, st);
        case EPI_GELU | EPI_RES_F32 | EPI_OUT_F32:
            return run<EPI_GELU | EPI_RES_F32 | EPI_OUT_F32>(a, st);
    }
    return ECHO_ERR_INVALID_ARG;
}

echo_status launch_linear_pair(const LinearArgs &a, const LinearArgs &b, cudaStream_t st) {
    if (a.M <= 0) return launch_linear(b, st);
    if (b.M <= 0) return launch_linear(a, st);
    if (a.Kd != b.Kd || a.act || b.act || a.resid || b.resid || a.row_amax || b.row_amax ||
        a.out_t != ECHO_BF16 || b.out_t != ECHO_BF16)
        return ECHO_ERR_INVALID_ARG;
    const bool narrow = narrow_tiles(a.M, a.N, a.Kd, b.M, b.N);
    Problem x, y;
    if (!make_problem(a, narrow, x) || !make_problem(b, narrow, y)) return ECHO_ERR_CUDA;
    return narrow ? run_bn<0, 128, true>(x, y, st) : run_bn<0, 256, true>(x, y, st);
}

}  // namespace echo

extern "C" echo_status echo_linear(const void *A, int64_t lda, int32_t M, int32_t Kd, const void *W,
                                   const void *bias, int32_t N, int32_t act, const void *resid,
                                   echo_dtype resid_t, const int32_t *resid_rows, void *out,
                                   int64_t ldo, echo_dtype out_t, echo_stream_t stream) {
    using namespace echo;
    if (M < 0 || Kd < 64 || Kd % 64 || N < 64 || N % 64) return ECHO_ERR_SHAPE;
    if (lda < Kd || lda % 8 || ldo < N || ldo % 8) return ECHO_ERR_SHAPE;
    if (M == 0) return ECHO_OK;
    if (!A || !W || !out) return ECHO_ERR_INVALID_ARG;
    if (act != 0 && act != 1) return ECHO_ERR_INVALID_ARG;
    if ((resid && resid_t != ECHO_BF16 && resid_t != ECHO_F32) ||
        (out_t != ECHO_BF16 && out_t != ECHO_F32))
        return ECHO_ERR_INVALID_ARG;
    if (resid_rows && (!resid || resid_t != ECHO_BF16)) return ECHO_ERR_INVALID_ARG;
    if (!aligned16(A) || !aligned16(W) || !aligned16(out) || (bias && !aligned16(bias)) ||
        (resid && !aligned16(resid)) || (resid_rows && !aligned16(resid_rows)))
        return ECHO_ERR_INVALID_ARG;
    if (!device_supported()) return ECHO_ERR_UNSUPPORTED;
    LinearArgs a{A, lda, M, Kd, W, bias, N, act, resid, resid_t, resid_rows, out, ldo, out_t};
    return launch_linear(a, reinterpret_cast<cudaStream_t>(stream));
}
