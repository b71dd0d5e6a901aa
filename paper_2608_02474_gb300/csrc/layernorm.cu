// Layer norm without affine, eps 1e-6, biased variance (the block's LN), with
// an optional row gather: out[j] = LN(in[rows[j]]), or, for every row of a bf16
// input, a second copy of the rows a map selects (the "select active latents"
// step of Sec. 3.3 fused with the LN over all latents that the K/V path needs).
//
// A row lives in registers: for bf16 input one warp per row holds it packed (up
// to 32 16-byte chunks per lane); for fp32 input up to 8 chunks of 8 values per
// thread, one warp per row for D <= 1024, four warps per row up to D = 8192.
// Mean first, then the centred variance, both fp32 tree reductions; one HBM
// read, one write.
#include "common.cuh"
#include "internal.h"

namespace {

constexpr int kThreads = 256;
constexpr int kMaxChunks = 8;
// Up to this width a warp holds a row in its registers and every row gets a warp of
// its own: short rows are bound by latency, and streaming them two at a time per
// warp, or one per CTA, kept too few loads in flight.  7800 rows of 1024: bf16 13.0
// -> 4.4 us, fp32 16.7 -> 4.9 us; 63960 rows of 2048: 97 -> 80, 154 -> 112 us.  At
// 3072 the streaming forms are as fast (7800 rows: 15.5 us against 17.8).
constexpr int kWarpRowMax = 2048;

template <typename T>
ECHO_DEV void ld8(const T *p, float *f);
template <>
ECHO_DEV void ld8<__nv_bfloat16>(const __nv_bfloat16 *p, float *f) {
    unpack8_bf16(__ldg(reinterpret_cast<const uint4 *>(p)), f);
}
template <>
ECHO_DEV void ld8<float>(const float *p, float *f) {
    const float4 a = __ldg(reinterpret_cast<const float4 *>(p));
    const float4 b = __ldg(reinterpret_cast<const float4 *>(p) + 1);
    f[0] = a.x; f[1] = a.y; f[2] = a.z; f[3] = a.w;
    f[4] = b.x; f[5] = b.y; f[6] = b.z; f[7] = b.w;
}

template <int TPR>
ECHO_DEV float row_sum(float v, float *red) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (TPR == 32) return v;
    constexpr int W = TPR / 32;
    const int warp = threadIdx.x >> 5;
    const int row_in_block = threadIdx.x / TPR;
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[warp] = v;
    __syncthreads();
    float s = 0.f;
#pragma unroll
    for (int w = 0; w < W; ++w) s += red[row_in_block * W + w];
    return s;
}

template <typename T, int TPR>
__global__ void __launch_bounds__(kThreads)
layernorm_kernel(const T *__restrict__ in, const int32_t *__restrict__ rows, int n_rows, int D,
                 __nv_bfloat16 *__restrict__ out) {
    pdl_enter();
    __shared__ float red[kThreads / 32];
    constexpr int RPB = kThreads / TPR;
    const int t = threadIdx.x % TPR;
    const int C = D >> 3;
    const float invD = 1.f / (float)D;
    for (int base = blockIdx.x * RPB; base < n_rows; base += gridDim.x * RPB) {
        const int j = base + threadIdx.x / TPR;
        const bool live = j < n_rows;
        const int r = live ? (rows ? rows[j] : j) : 0;
        const T *src = in + (int64_t)r * D;
        float v[kMaxChunks][8];
        float s = 0.f;
#pragma unroll
        for (int k = 0; k < kMaxChunks; ++k) {
            const int c = t + k * TPR;
            if (live && c < C) {
                ld8<T>(src + 8 * c, v[k]);
#pragma unroll
                for (int e = 0; e < 8; ++e) s += v[k][e];
            } else {
#pragma unroll
                for (int e = 0; e < 8; ++e) v[k][e] = 0.f;
            }
        }
        const float mean = row_sum<TPR>(s, red) * invD;
        float ss = 0.f;
#pragma unroll
        for (int k = 0; k < kMaxChunks; ++k) {
            const int c = t + k * TPR;
            if (live && c < C) {
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const float dlt = v[k][e] - mean;
                    ss += dlt * dlt;
                }
            }
        }
        const float var = row_sum<TPR>(ss, red) * invD;
        const float rstd = rsqrtf(var + 1e-6f);
        if (live) {
            __nv_bfloat16 *dst = out + (int64_t)j * D;
#pragma unroll
            for (int k = 0; k < kMaxChunks; ++k) {
                const int c = t + k * TPR;
                if (c < C) {
                    float o[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) o[e] = (v[k][e] - mean) * rstd;
                    *reinterpret_cast<uint4 *>(dst + 8 * c) = pack8_bf16(o);
                }
            }
        }
    }
}

// position of v in idx[0 .. n) (ascending, distinct), or -1: 32 probes at a time
ECHO_DEV int warp_find(const int32_t *__restrict__ idx, int n, int v) {
    const int lane = threadIdx.x & 31;
    int lo = 0;
    while (n > 0) {
        const int step = (n + 31) >> 5;   // each lane looks at the first of `step` entries
        const int x = lane * step < n ? idx[lo + lane * step] : INT32_MAX;
        const uint32_t le = __ballot_sync(0xffffffffu, x <= v);
        if (!le) return -1;
        const int b = 31 - __clz((int)le);
        lo += b * step;
        n = min(step, n - b * step);
        if (n == 1) return __shfl_sync(0xffffffffu, x, b) == v ? lo : -1;
    }
    return -1;
}

// bf16 input: one warp per row, the row held packed in registers (CPL 16-byte
// chunks per lane), so each row is read from HBM once and no block barrier is
// needed.  With idx (ascending, distinct), row j is also looked up there: its
// position p (-1: not in it) goes to rowmap[j], zero[p] is cleared, and the result
// is written to out2[p] as well.
template <int CPL>
__global__ void __launch_bounds__(kThreads)
layernorm_warp_bf16(const __nv_bfloat16 *__restrict__ in, const int32_t *__restrict__ rows,
                    int n_rows, int D, __nv_bfloat16 *__restrict__ out, __nv_bfloat16 *__restrict__ out2,
                    const int32_t *__restrict__ idx, int n_idx, int32_t *__restrict__ rowmap,
                    uint32_t *__restrict__ zero) {
    pdl_enter();
    const int lane = threadIdx.x & 31;
    const int warps = kThreads / 32;
    const int C = D >> 3;
    const float invD = 1.f / (float)D;
    for (RowWalk walk = grid_rows(warps); walk.below(n_rows); walk.next()) {
        const int j = (int)walk.row;
        const int r = rows ? rows[j] : j;
        const uint4 *src = reinterpret_cast<const uint4 *>(in + (int64_t)r * D);
        uint4 v[CPL];
#pragma unroll
        for (int k = 0; k < CPL; ++k) {
            const int c = lane + 32 * k;
            v[k] = c < C ? __ldcs(src + c) : make_uint4(0, 0, 0, 0);
        }
        int j2 = -1;
        if (idx) {   // while the row is on its way
            j2 = warp_find(idx, n_idx, j);
            if (lane == 0) {
                rowmap[j] = j2;
                if (j2 >= 0) zero[j2] = 0u;
            }
        }
        float s = 0.f;
#pragma unroll
        for (int k = 0; k < CPL; ++k) {
            float f[8];
            unpack8_bf16(v[k], f);
#pragma unroll
            for (int e = 0; e < 8; ++e) s += f[e];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        const float mean = s * invD;
        float ss = 0.f;
#pragma unroll
        for (int k = 0; k < CPL; ++k) {
            if (lane + 32 * k < C) {
                float f[8];
                unpack8_bf16(v[k], f);
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const float dlt = f[e] - mean;
                    ss += dlt * dlt;
                }
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
        const float rstd = rsqrtf(ss * invD + 1e-6f);
        uint4 *dst = reinterpret_cast<uint4 *>(out + (int64_t)j * D);
        uint4 *dst2 = j2 >= 0 ? reinterpret_cast<uint4 *>(out2 + (int64_t)j2 * D) : nullptr;
#pragma unroll
        for (int k = 0; k < CPL; ++k) {
            const int c = lane + 32 * k;
            if (c < C) {
                float f[8];
                unpack8_bf16(v[k], f);
#pragma unroll
                for (int e = 0; e < 8; ++e) f[e] = (f[e] - mean) * rstd;
                const uint4 o = pack8_bf16(f);
                dst[c] = o;
                if (dst2) dst2[c] = o;
            }
        }
    }
}

// All rows of a bf16 input (no gather), for D <= 8192: one warp per row as in
// layernorm_warp_bf16, but each warp streams its rows through two shared-memory
// buffers filled by 1-D bulk copies, the next row's copy in flight while the
// current row is normalised and written.  Same arithmetic, same bits.  With
// scatter_map, row j is also written to out2[scatter_map[j]] when that is
// >= 0: the LN of every latent (for K and V) then also yields the gathered LN
// of the active ones (for Q') without reading them a second time.
constexpr int kBulkWarps = 4;
constexpr size_t kBulkSmemMin = 78 * 1024;   // a third of an SM's 228 KB and more: two CTAs per SM

template <int CPL>
__global__ void __launch_bounds__(kBulkWarps * 32)
layernorm_bulk_bf16(const __nv_bfloat16 *__restrict__ in, int n_rows, int D,
                    __nv_bfloat16 *__restrict__ out, const int32_t *__restrict__ scatter_map,
                    __nv_bfloat16 *__restrict__ out2, int *err) {
    extern __shared__ __align__(128) uint8_t smem_rows[];
    __shared__ __align__(8) uint64_t bar[kBulkWarps][2];
    __shared__ int abort_flag;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t row_bytes = (uint32_t)D * 2u;
    uint8_t *buf = smem_rows + (size_t)warp * 2 * row_bytes;
    if (lane == 0) {
        mbar_init(&bar[warp][0], 1);
        mbar_init(&bar[warp][1], 1);
    }
    if (threadIdx.x == 0) abort_flag = 0;
    fence_barrier_init();
    __syncthreads();
    pdl_enter();
    volatile int *abort_v = &abort_flag;
    const int C = D >> 3;
    const float invD = 1.f / (float)D;
    const int nw = gridDim.x * kBulkWarps;
    int j = blockIdx.x * kBulkWarps + warp;
    if (j < n_rows && lane == 0) {
        mbar_arrive_expect_tx(&bar[warp][0], row_bytes);
        bulk_load_1d(buf, in + (int64_t)j * D, row_bytes, &bar[warp][0]);
    }
    bool pending_next = false;
    for (int it = 0; j < n_rows; ++it, j += nw) {
        const int b = it & 1;
        const int jn = j + nw;
        __syncwarp();   // every lane is done with buffer b ^ 1 (read in the last iteration)
        pending_next = jn < n_rows;
        if (pending_next && lane == 0) {
            fence_proxy_async_smem();
            mbar_arrive_expect_tx(&bar[warp][b ^ 1], row_bytes);
            bulk_load_1d(buf + (b ^ 1) * row_bytes, in + (int64_t)jn * D, row_bytes,
                         &bar[warp][b ^ 1]);
        }
        if (!__all_sync(0xffffffffu, mbar_wait(&bar[warp][b], (it >> 1) & 1, abort_v, err))) {
            pending_next = false;   // the CTA gives up; let the next copy land first
            if (jn < n_rows)
                mbar_wait(&bar[warp][b ^ 1], ((it + 1) >> 1) & 1, abort_v, nullptr, 100000000ull);
            break;
        }
        const uint4 *src = reinterpret_cast<const uint4 *>(buf + b * row_bytes);
        uint4 v[CPL];
#pragma unroll
        for (int k = 0; k < CPL; ++k) {
            const int c = lane + 32 * k;
            v[k] = c < C ? src[c] : make_uint4(0, 0, 0, 0);
        }
        float s = 0.f;
#pragma unroll
        for (int k = 0; k < CPL; ++k) {
            float f[8];
            unpack8_bf16(v[k], f);
#pragma unroll
            for (int e = 0; e < 8; ++e) s += f[e];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        const float mean = s * invD;
        float ss = 0.f;
#pragma unroll
        for (int k = 0; k < CPL; ++k) {
            if (lane + 32 * k < C) {
                float f[8];
                unpack8_bf16(v[k], f);
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const float dlt = f[e] - mean;
                    ss += dlt * dlt;
                }
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
        const float rstd = rsqrtf(ss * invD + 1e-6f);
        uint4 *dst = reinterpret_cast<uint4 *>(out + (int64_t)j * D);
        const int j2 = scatter_map ? scatter_map[j] : -1;
        uint4 *dst2 = j2 >= 0 ? reinterpret_cast<uint4 *>(out2 + (int64_t)j2 * D) : nullptr;
#pragma unroll
        for (int k = 0; k < CPL; ++k) {
            const int c = lane + 32 * k;
            if (c < C) {
                float f[8];
                unpack8_bf16(v[k], f);
#pragma unroll
                for (int e = 0; e < 8; ++e) f[e] = (f[e] - mean) * rstd;
                const uint4 o = pack8_bf16(f);
                dst[c] = o;
                if (dst2) dst2[c] = o;
            }
        }
    }
    (void)pending_next;
}

template <int CPL>
void launch_bulk_bf16(const __nv_bfloat16 *in, int n_rows, int D, __nv_bfloat16 *out,
                      const int32_t *scatter_map, __nv_bfloat16 *out2, cudaStream_t st) {
    // Two CTAs per SM, as the grid has them, whatever the width: where four would fit,
    // the next kernel's CTAs came to lie unevenly beside those still running (32760 rows
    // of 2112 59.0 -> 51.5 us, 7800 of 3072 19.0 -> 17.9, 15000 of 4096 44.3 -> 42.8).
    size_t smem = (size_t)kBulkWarps * 2 * D * sizeof(__nv_bfloat16);
    if (smem < kBulkSmemMin) smem = kBulkSmemMin;
    static int attr_done[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 0 && dev < 64 && !attr_done[dev]) {
        cudaFuncSetAttribute(layernorm_bulk_bf16<CPL>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)(kBulkWarps * 2 * 8192 * sizeof(__nv_bfloat16)));
        attr_done[dev] = 1;
    }
    int grid = (n_rows + kBulkWarps - 1) / kBulkWarps;
    if (grid > 152 * 2) grid = 152 * 2;
    echo::launch_chained(layernorm_bulk_bf16<CPL>, dim3(grid), dim3(kBulkWarps * 32), smem, st,
                         in, n_rows, D, out, scatter_map,
                                                                  out2, echo::device_error_ptr());
}

template <int CPL>
void launch_warp_bf16(const __nv_bfloat16 *in, const int32_t *rows, int n_rows, int D,
                      __nv_bfloat16 *out, __nv_bfloat16 *out2, const int32_t *idx, int n_idx,
                      int32_t *rowmap, uint32_t *zero, cudaStream_t st) {
    int grid = blocks_for_rows(n_rows, kThreads / 32);
    if (grid > 152 * 8) grid = 152 * 8;
    echo::launch_chained(layernorm_warp_bf16<CPL>, dim3(grid), dim3(kThreads), 0, st, in, rows,
                         n_rows, D, out, out2, idx, n_idx, rowmap, zero);
}

// the row packed in registers: gathered rows, and every row up to D = kWarpRowMax
void launch_regs_bf16(const __nv_bfloat16 *in, const int32_t *rows, int n_rows, int D,
                      __nv_bfloat16 *out, __nv_bfloat16 *out2, const int32_t *idx, int n_idx,
                      int32_t *rowmap, uint32_t *zero, cudaStream_t st) {
    const int cpl = (D / 8 + 31) / 32;   // 16-byte chunks per lane
    auto go = [&](auto launch) { launch(in, rows, n_rows, D, out, out2, idx, n_idx, rowmap, zero, st); };
    if (cpl <= 1) return go(launch_warp_bf16<1>);
    if (cpl <= 4) return go(launch_warp_bf16<4>);
    if (cpl <= 8) return go(launch_warp_bf16<8>);
    if (cpl <= 16) return go(launch_warp_bf16<16>);
    if (cpl <= 20) return go(launch_warp_bf16<20>);
    if (cpl <= 24) return go(launch_warp_bf16<24>);
    return go(launch_warp_bf16<32>);
}

// ((T_0 + T_1) + T_2) + T_3, T_w the sum of p[w] over the warp as a xor butterfly adds
// it.  A lane passes on the partial sums that its partner keeps, so that after two
// steps each quarter of the warp works on one of them: 18 shuffles a row instead of
// 40 (7800 rows of 2048 13.2 -> 11.6 us; 10.5 with one sum per lane in an order of
// its own).
ECHO_DEV float ordered_total(const float (&p)[4]) {
    const int lane = threadIdx.x & 31;
    auto xor_add = [](float keep, float pass, int o) { return keep + __shfl_xor_sync(0xffffffffu, pass, o); };
    const bool hi = lane & 16, odd = lane & 8;
    const float a = xor_add(hi ? p[2] : p[0], hi ? p[0] : p[2], 16);
    const float b = xor_add(hi ? p[3] : p[1], hi ? p[1] : p[3], 16);
    float t = xor_add(odd ? b : a, odd ? a : b, 8);
    t = xor_add(t, t, 4);
    t = xor_add(t, t, 2);
    t = xor_add(t, t, 1);
    float r = __shfl_sync(0xffffffffu, t, 0);
#pragma unroll
    for (int w = 1; w < 4; ++w) r += __shfl_sync(0xffffffffu, t, 8 * w);
    return r;
}

// the sum of p[0] over the warp as a xor butterfly adds it
ECHO_DEV float ordered_total(const float (&p)[1]) {
    float s = p[0];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}

// fp32 rows of up to kWarpRowMax values: one warp per row, the row in registers
// (lane l holds 16-byte chunks l, l + 32, ...).  Sums: up to 1024 values each lane's
// chunks in order, then a xor butterfly.  Above, where a few rows take
// layernorm_row_f32 below, in the order of that form, to the same bits, so that a
// row's result does not depend on how many rows come with it: chunk l + 32 k belongs
// to thread l of warp k mod 4 there, and a lane keeps the partial sums of the four.
template <int CPL>
__global__ void __launch_bounds__(kThreads)
layernorm_warp_f32(const float *__restrict__ in, int n_rows, int D,
                   __nv_bfloat16 *__restrict__ out) {
    pdl_enter();
    constexpr int P = CPL > 8 ? 4 : 1;
    const int lane = threadIdx.x & 31;
    const int j = blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5);
    if (j >= n_rows) return;
    const int C4 = D >> 2;
    const float invD = 1.f / (float)D;
    const float4 *row = reinterpret_cast<const float4 *>(in + (int64_t)j * D);
    float4 v[CPL];
#pragma unroll
    for (int k = 0; k < CPL; ++k)
        v[k] = lane + 32 * k < C4 ? __ldcs(row + lane + 32 * k) : make_float4(0.f, 0.f, 0.f, 0.f);
    float s[P] = {};
#pragma unroll
    for (int k = 0; k < CPL; ++k) {
        float &p = s[k % P];
        if constexpr (P == 1) {
            p += (v[k].x + v[k].y) + (v[k].z + v[k].w);
        } else {
            p += v[k].x; p += v[k].y; p += v[k].z; p += v[k].w;
        }
    }
    const float mean = ordered_total(s) * invD;
    float ss[P] = {};
#pragma unroll
    for (int k = 0; k < CPL; ++k)
        if (lane + 32 * k < C4) {
            const float a = v[k].x - mean, b = v[k].y - mean, c = v[k].z - mean, d = v[k].w - mean;
            float &p = ss[k % P];
            if constexpr (P == 1) {
                p += (a * a + b * b) + (c * c + d * d);
            } else {
                p += a * a; p += b * b; p += c * c; p += d * d;
            }
        }
    const float rstd = rsqrtf(ordered_total(ss) * invD + 1e-6f);
    uint2 *dst = reinterpret_cast<uint2 *>(out + (int64_t)j * D);
#pragma unroll
    for (int k = 0; k < CPL; ++k)
        if (lane + 32 * k < C4)
            dst[lane + 32 * k] = make_uint2(pack_bf16((v[k].x - mean) * rstd, (v[k].y - mean) * rstd),
                                            pack_bf16((v[k].z - mean) * rstd, (v[k].w - mean) * rstd));
}

template <int CPL>
void launch_warp_f32(const float *in, int n_rows, int D, __nv_bfloat16 *out, cudaStream_t st) {
    echo::launch_chained(layernorm_warp_f32<CPL>, dim3(blocks_for_rows(n_rows, kThreads / 32)),
                         dim3(kThreads), 0, st, in, n_rows, D, out);
}

// fp32 rows of up to 8192 values: one CTA of 128 threads per row, the row in
// registers (thread t holds 16-byte chunks t, t + 128, ...), every load in
// flight before the first sum.  Sums: each thread's chunks in order, a xor
// butterfly per warp, then the four warp partials in order.
constexpr int kRowThreads = 128, kRowChunks = 16;

__global__ void __launch_bounds__(kRowThreads)
layernorm_row_f32(const float *__restrict__ in, int D, __nv_bfloat16 *__restrict__ out) {
    pdl_enter();
    __shared__ float red[2][kRowThreads / 32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int C4 = D >> 2;
    const float4 *row = reinterpret_cast<const float4 *>(in + (int64_t)blockIdx.x * D);
    float4 v[kRowChunks];
#pragma unroll
    for (int k = 0; k < kRowChunks; ++k) {
        const int c = threadIdx.x + k * kRowThreads;
        v[k] = c < C4 ? __ldcs(row + c) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    float s = 0.f;
#pragma unroll
    for (int k = 0; k < kRowChunks; ++k) {
        s += v[k].x; s += v[k].y; s += v[k].z; s += v[k].w;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) red[0][warp] = s;
    __syncthreads();
    const float invD = 1.f / (float)D;
    const float mean = (((red[0][0] + red[0][1]) + red[0][2]) + red[0][3]) * invD;
    float ss = 0.f;
#pragma unroll
    for (int k = 0; k < kRowChunks; ++k) {
        if (threadIdx.x + k * kRowThreads < C4) {
            const float a = v[k].x - mean, b = v[k].y - mean, c = v[k].z - mean, d = v[k].w - mean;
            ss += a * a; ss += b * b; ss += c * c; ss += d * d;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    if (lane == 0) red[1][warp] = ss;
    __syncthreads();
    const float rstd = rsqrtf((((red[1][0] + red[1][1]) + red[1][2]) + red[1][3]) * invD + 1e-6f);
    uint2 *dst = reinterpret_cast<uint2 *>(out + (int64_t)blockIdx.x * D);
#pragma unroll
    for (int k = 0; k < kRowChunks; ++k) {
        const int c = threadIdx.x + k * kRowThreads;
        if (c < C4)
            dst[c] = make_uint2(pack_bf16((v[k].x - mean) * rstd, (v[k].y - mean) * rstd),
                                pack_bf16((v[k].z - mean) * rstd, (v[k].w - mean) * rstd));
    }
}

// every row of an fp32 input (D <= 8192: echo_layernorm and the block step
// reject wider rows)
void launch_all_f32(const float *in, int n_rows, int D, __nv_bfloat16 *out, cudaStream_t st) {
    if (n_rows <= 0) return;
    // above 1024 values a few rows finish sooner with four warps each (64 rows of
    // 1536: 1.7 us against 2.2; 1024 rows: 3.4 against 2.4), to the same bits
    if (D <= 1024 || (D <= kWarpRowMax && n_rows > 1024)) {
        if (D <= 256) return launch_warp_f32<2>(in, n_rows, D, out, st);
        if (D <= 1024) return launch_warp_f32<8>(in, n_rows, D, out, st);
        return launch_warp_f32<16>(in, n_rows, D, out, st);
    }
    echo::launch_chained(layernorm_row_f32, dim3(n_rows), dim3(kRowThreads), 0, st, in, D, out);
}

// every row of a bf16 input, optionally also scattered through a map: the
// bulk-copy kernel (the same arithmetic as layernorm_warp_bf16)
void launch_all_bf16(const __nv_bfloat16 *in, int n_rows, int D, __nv_bfloat16 *out,
                     const int32_t *scatter_map, __nv_bfloat16 *out2, cudaStream_t st) {
    if (D <= kWarpRowMax && !scatter_map)
        return launch_regs_bf16(in, nullptr, n_rows, D, out, nullptr, nullptr, 0, nullptr, nullptr, st);
    const int cpl = (D / 8 + 31) / 32;
    if (cpl <= 16) return launch_bulk_bf16<16>(in, n_rows, D, out, scatter_map, out2, st);
    if (cpl <= 20) return launch_bulk_bf16<20>(in, n_rows, D, out, scatter_map, out2, st);
    if (cpl <= 24) return launch_bulk_bf16<24>(in, n_rows, D, out, scatter_map, out2, st);
    return launch_bulk_bf16<32>(in, n_rows, D, out, scatter_map, out2, st);
}

template <typename T>
void launch_t(const T *in, const int32_t *rows, int n_rows, int D, __nv_bfloat16 *out,
              cudaStream_t st) {
    const int C = D / 8;
    echo::LaunchScope ls(ECHO_K_LAYERNORM, n_rows, D, (int64_t)sizeof(T), st);
    if constexpr (sizeof(T) == 2) {
        if (!rows) return launch_all_bf16(in, n_rows, D, out, nullptr, nullptr, st);
        return launch_regs_bf16(in, rows, n_rows, D, out, nullptr, nullptr, 0, nullptr, nullptr, st);
    } else {
        if (!rows) return launch_all_f32(in, n_rows, D, out, st);
    }
    if (C <= 32 * kMaxChunks / 2) {   // D <= 1024: a warp per row
        constexpr int RPB = kThreads / 32;
        int grid = (n_rows + RPB - 1) / RPB;
        if (grid > 152 * 16) grid = 152 * 16;
        echo::launch_chained(layernorm_kernel<T, 32>, dim3(grid), dim3(kThreads), 0, st, in,
                             rows, n_rows, D, out);
    } else {
        constexpr int RPB = kThreads / 128;
        int grid = (n_rows + RPB - 1) / RPB;
        if (grid > 152 * 16) grid = 152 * 16;
        echo::launch_chained(layernorm_kernel<T, 128>, dim3(grid), dim3(kThreads), 0, st, in,
                             rows, n_rows, D, out);
    }
}

}  // namespace

namespace echo {

void launch_layernorm_active(const void *in, int32_t n_rows, int32_t D, void *out, const int32_t *idx,
                             int32_t K, int32_t *rowmap, uint32_t *zero, void *out2,
                             cudaStream_t st) {
    if (n_rows <= 0) return;
    const __nv_bfloat16 *x = static_cast<const __nv_bfloat16 *>(in);
    __nv_bfloat16 *o = static_cast<__nv_bfloat16 *>(out), *o2 = static_cast<__nv_bfloat16 *>(out2);
    if (D <= kWarpRowMax) {
        LaunchScope ls(ECHO_K_LAYERNORM, n_rows, D, 2, st);
        return launch_regs_bf16(x, nullptr, n_rows, D, o, o2, idx, K, rowmap, zero, st);
    }
    launch_rowmap(idx, K, n_rows, rowmap, zero, K, st);
    LaunchScope ls(ECHO_K_LAYERNORM, n_rows, D, 2, st);
    launch_all_bf16(x, n_rows, D, o, rowmap, o2, st);
}

void launch_layernorm(const void *in, echo_dtype in_t, const int32_t *rows, int32_t n_rows,
                      int32_t D, void *out, cudaStream_t st) {
    if (n_rows <= 0) return;
    __nv_bfloat16 *o = static_cast<__nv_bfloat16 *>(out);
    if (in_t == ECHO_BF16)
        launch_t(static_cast<const __nv_bfloat16 *>(in), rows, n_rows, D, o, st);
    else
        launch_t(static_cast<const float *>(in), rows, n_rows, D, o, st);
}

}  // namespace echo

extern "C" echo_status echo_layernorm(const void *in, echo_dtype in_t, const int32_t *rows,
                                      int32_t n_rows, int32_t D, void *out, echo_stream_t stream) {
    using namespace echo;
    if (n_rows < 0 || D < 8 || D % 8 || D > 8192) return ECHO_ERR_SHAPE;
    if (n_rows == 0) return ECHO_OK;
    if (!in || !out) return ECHO_ERR_INVALID_ARG;
    if (in_t != ECHO_BF16 && in_t != ECHO_F32) return ECHO_ERR_INVALID_ARG;
    if (!aligned16(in) || !aligned16(out) || (rows && !aligned16(rows))) return ECHO_ERR_INVALID_ARG;
    if (!device_supported()) return ECHO_ERR_UNSUPPORTED;
    launch_layernorm(in, in_t, rows, n_rows, D, out, reinterpret_cast<cudaStream_t>(stream));
    return last_launch_status();
}
