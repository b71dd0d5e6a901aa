// Cache forms of Sec. 3.4 beyond the plain int8 cache: the reference plus
// int8 residual manager (ECHO_CACHE_REF) and the full-precision ablation form
// (ECHO_CACHE_BF16).
//
// A REF write is four stream-ordered kernels:
//   ref_release  every written token drops its old reference (atomic
//                decrement of the slot's count) and the bounds of each scan
//                segment's written rows are recorded;
//   ref_scan     one CTA per scan segment walks its written rows in token
//                order, 6 or 12 rows a round: the rows are staged in shared memory,
//                two warps per row compute the fp32 cosines the walk is likely to need
//                (each row against the entering reference and against the row
//                before it, canonical order), then one thread walks the rows,
//                asking for others where it must, and the last new reference
//                carries into the next round;
//   ref_alloc    one CTA ranks the new references in token order and hands
//                them the free slots in slot order (block scans);
//   ref_store    one CTA per written row (a warp above D = 8192): a reference
//                copies its row into its slot, a residual quantises x - r by the
//                int8 rule, a run without a slot quantises x itself.
// Reconstruction (read, merge) is one thread per 16 values: bf16(r + q s).
#include <mutex>

#include "common.cuh"
#include "internal.h"

namespace {

// Rows of a scan window: 6, or 12 where every segment has an SM to itself and the time
// is one segment's walk.  A write of 7800 rows in 150 segments of 52, six rows against
// twelve: 43 and 39 us at 128 values, 117 and 89 at 5120 (nearly every row a reference:
// 49 and 45, 125 and 97); 9000 rows in 174 segments: 47 and 58, 126 and 131.
constexpr int kWin = 6, kWinWide = 12, kWideSegments = 152;
constexpr int kAllocThreads = 1024;
constexpr int kStoreThreads = 256;
constexpr int kVec = 256;

size_t al256(size_t b) { return (b + 255) & ~(size_t)255; }

int grid_for(int64_t work, int threads) {
    int64_t g = (work + threads - 1) / threads;
    const int64_t cap = 152 * 32;
    if (g > cap) g = cap;
    return (int)(g < 1 ? 1 : g);
}

ECHO_DEV bool bf16_nonfinite(uint32_t two) {
    return ((two & 0x7F80u) == 0x7F80u) || ((two & 0x7F800000u) == 0x7F800000u);
}

// ---------------------------------------------------------------- release
// every written token drops its reference (when a pool exists); the written
// rows of scan segment s are positions [seg_lo[s], seg_hi[s]) of rows (seg_lo
// stays -1 for a segment with none; rows ascending)
__global__ void ref_release_kernel(const int32_t *__restrict__ rows, int n, int seg_len,
                                   const int32_t *__restrict__ ref, int32_t *refcount,
                                   int32_t *__restrict__ seg_lo, int32_t *__restrict__ seg_hi) {
    pdl_enter();
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < n) {
        const int i = rows[j];
        if (refcount) {
            const int old = ref[i];
            if (old >= 0) atomicSub(&refcount[old], 1);
        }
        const int sg = i / seg_len;
        if (j == 0 || rows[j - 1] / seg_len != sg) seg_lo[sg] = j;
        if (j == n - 1 || rows[j + 1] / seg_len != sg) seg_hi[sg] = j + 1;
    }
}

// ---------------------------------------------------------------- scan
// The canonical-order fp32 sums <a, b> (and <a, a> when `norm`) of two bf16
// rows in shared memory: lane l owns 8-element chunks l, l+32, ..., adds each
// chunk's sum left to right into its accumulator in chunk order, then an xor
// butterfly 16..1.  Every lane returns the same sums.
ECHO_DEV void warp_dot(const uint4 *a, const uint4 *b, int C, int lane, bool norm, float &dot,
                       float &na) {
    dot = 0.f;
    na = 0.f;
    for (int c = lane; c < C; c += 32) {
        float fa[8], fb[8];
        unpack8_bf16(a[c], fa);
        unpack8_bf16(b[c], fb);
        float cd = __fmul_rn(fa[0], fb[0]);
        float cn = __fmul_rn(fa[0], fa[0]);
#pragma unroll
        for (int k = 1; k < 8; ++k) {
            cd = __fadd_rn(cd, __fmul_rn(fa[k], fb[k]));
            if (norm) cn = __fadd_rn(cn, __fmul_rn(fa[k], fa[k]));
        }
        dot = __fadd_rn(dot, cd);
        if (norm) na = __fadd_rn(na, cn);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        dot = __fadd_rn(dot, __shfl_xor_sync(0xffffffffu, dot, o));
        na = __fadd_rn(na, __shfl_xor_sync(0xffffffffu, na, o));
    }
}

// src_pos[j] = position (in rows) of row j's reference; j itself for a reference.
//
// One CTA per scan segment.  The segment's written rows are taken WIN at a
// time: the window's rows are staged in shared memory, then every row is compared
// with the reference that the window was entered with and with the row before it,
// one similarity per warp, and one thread walks the window in order.  Those two
// suffice while the reference stays or changes at every row; a row that follows a
// change by two or more also needs its similarity to the row of the change, which
// is then computed for the rest of the window at once before the walk goes on.
// Dynamic shared memory: WIN window rows, then the current reference row (bf16, D
// each); six rows leave room for three CTAs per SM at D = 5120.  6552 rows of 5120:
// 70 us with all 36 similarities of windows of eight rows and two CTAs per SM, 49 us.
template <int WIN>
__global__ void __launch_bounds__(2 * WIN * 32)
ref_scan_kernel(const __nv_bfloat16 *__restrict__ src, const int32_t *__restrict__ seg_lo,
                const int32_t *__restrict__ seg_hi, float tau, int D,
                int32_t *__restrict__ src_pos) {
    pdl_enter();
    extern __shared__ uint4 s_buf[];
    __shared__ float s_dref[WIN], s_dprev[WIN], s_dcur[WIN];   // <w, ref>, <w, w - 1>, <w, s_cur>
    __shared__ float s_nv[WIN];
    __shared__ float s_nr;
    __shared__ int s_jr, s_cur, s_w, s_more;   // walk: reference row of the window (-1: entering), row
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int C = D >> 3;
    uint4 *ref = s_buf + (size_t)WIN * C;
    const int lo = seg_lo[blockIdx.x];
    if (lo < 0) return;
    const int hi = seg_hi[blockIdx.x];
    if (threadIdx.x == 0) {
        src_pos[lo] = lo;
        s_jr = lo;
    }
    // the segment's first written row is its first reference
    {
        const uint4 *v = reinterpret_cast<const uint4 *>(src + (int64_t)lo * D);
        for (int c = threadIdx.x; c < C; c += blockDim.x) ref[c] = __ldg(v + c);
    }
    __syncthreads();
    if (warp == 0) {
        float d, nr;
        warp_dot(ref, ref, C, lane, true, d, nr);
        if (lane == 0) s_nr = nr;
    }
    __syncthreads();
    for (int j = lo + 1; j < hi; j += WIN) {
        const int nvalid = hi - j < WIN ? hi - j : WIN;
        // stage the window's rows (consecutive in src), eight 16-byte loads in flight
        const int total = nvalid * C;
        const uint4 *win = reinterpret_cast<const uint4 *>(src + (int64_t)j * D);
        for (int b = threadIdx.x; b < total; b += 8 * (int)blockDim.x) {
            uint4 u[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int e = b + k * blockDim.x;
                if (e < total) u[k] = __ldg(win + e);
            }
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int e = b + k * blockDim.x;
                if (e < total) s_buf[e] = u[k];
            }
        }
        if (threadIdx.x == 0) {
            s_cur = -1;
            s_w = 0;
        }
        __syncthreads();
        {
            const int w = warp < WIN ? warp : warp - WIN;
            const bool vs_ref = warp < WIN;
            if (w < nvalid && (vs_ref || w > 0)) {
                const uint4 *a = s_buf + (size_t)w * C;
                float dot, nv;
                warp_dot(a, vs_ref ? ref : a - C, C, lane, vs_ref, dot, nv);
                if (lane == 0) {
                    (vs_ref ? s_dref : s_dprev)[w] = dot;
                    if (vs_ref) s_nv[w] = nv;
                }
            }
        }
        int have = -1;   // the row that s_dcur holds the similarities to
        for (;;) {
            __syncthreads();
            if (threadIdx.x == 0) {
                int cur = s_cur, w = s_w;
                const int jr = s_jr;
                int more = 0;
                for (; w < nvalid; ++w) {
                    float dot;
                    if (cur < 0) dot = s_dref[w];
                    else if (cur == w - 1) dot = s_dprev[w];
                    else if (cur == have) dot = s_dcur[w];
                    else {
                        more = 1;
                        break;
                    }
                    const float nv = s_nv[w], ncur = cur < 0 ? s_nr : s_nv[cur];
                    float sim = 0.f;
                    if (nv > 0.f && ncur > 0.f)
                        sim = __fdiv_rn(dot, __fmul_rn(__fsqrt_rn(nv), __fsqrt_rn(ncur)));
                    if (sim > tau) {
                        src_pos[j + w] = cur < 0 ? jr : j + cur;
                    } else {
                        src_pos[j + w] = j + w;
                        cur = w;
                    }
                }
                s_cur = cur;
                s_w = w;
                s_more = more;
            }
            __syncthreads();
            if (!s_more) break;
            const int cur = s_cur, w = s_w + warp;
            if (w < nvalid) {
                float dot, nv;
                warp_dot(s_buf + (size_t)w * C, s_buf + (size_t)cur * C, C, lane, false, dot, nv);
                if (lane == 0) s_dcur[w] = dot;
            }
            have = cur;
        }
        const int nr = s_cur;   // the last new reference carries into the next window
        if (nr >= 0) {
            if (threadIdx.x == 0) {
                s_jr = j + nr;
                s_nr = s_nv[nr];
            }
            for (int c = threadIdx.x; c < C; c += blockDim.x) ref[c] = s_buf[(size_t)nr * C + c];
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------- alloc
// exclusive block scan of one value per thread; *total gets the block sum
ECHO_DEV int block_scan(int v, int *warp_sums, int *total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
    }
    if (lane == 31) warp_sums[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        const int w = lane < (int)(blockDim.x >> 5) ? warp_sums[lane] : 0;
        int wi = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o) wi += t;
        }
        warp_sums[lane] = wi - w;
        if (lane == 31) warp_sums[32] = wi;
    }
    __syncthreads();
    const int r = warp_sums[warp] + inc - v;
    *total = warp_sums[32];
    __syncthreads();
    return r;
}

// slot_of[j] = pool slot of the reference at position j (-1: none or not a reference)
__global__ void __launch_bounds__(kAllocThreads)
ref_alloc_kernel(const int32_t *__restrict__ src_pos, int n, const int32_t *__restrict__ refcount,
                 int R_cap, int32_t *__restrict__ free_list, int32_t *__restrict__ slot_of) {
    pdl_enter();
    __shared__ int warp_sums[33];
    // rank the references in token order
    int run = 0;
    for (int base = 0; base < n; base += kAllocThreads) {
        const int j = base + threadIdx.x;
        const int is_ref = j < n && src_pos[j] == j;
        int tot;
        const int r = run + block_scan(is_ref, warp_sums, &tot);
        if (j < n) slot_of[j] = is_ref ? r : -1;
        run += tot;
    }
    const int n_new = run;
    // the first n_new free slots in slot order
    int nfree = 0;
    for (int base = 0; base < R_cap && nfree < n_new; base += kAllocThreads) {
        const int sl = base + threadIdx.x;
        const int fr = sl < R_cap && refcount[sl] == 0;
        int tot;
        const int m = nfree + block_scan(fr, warp_sums, &tot);
        if (fr && m < n_new) free_list[m] = sl;
        nfree += tot;
    }
    const int avail = nfree < n_new ? nfree : n_new;
    __syncthreads();
    for (int j = threadIdx.x; j < n; j += kAllocThreads) {
        const int r = slot_of[j];
        if (r >= 0) slot_of[j] = r < avail ? free_list[r] : -1;
    }
}

// ---------------------------------------------------------------- store
__global__ void __launch_bounds__(kStoreThreads)
ref_store_kernel(const __nv_bfloat16 *__restrict__ src, const int32_t *__restrict__ rows, int n,
                 int D, const int32_t *__restrict__ src_pos, const int32_t *__restrict__ slot_of,
                 int8_t *__restrict__ q, float *__restrict__ scale, int32_t *__restrict__ ref,
                 int32_t *refcount, __nv_bfloat16 *__restrict__ pool, int *err) {
    pdl_enter();
    const int lane = threadIdx.x & 31;
    const int warps = blockDim.x >> 5;
    const int C = D >> 3;
    for (int j = blockIdx.x * warps + (threadIdx.x >> 5); j < n; j += gridDim.x * warps) {
        const int i = rows[j];
        const int jr = src_pos[j];
        const int sl = slot_of[jr];
        const __nv_bfloat16 *v = src + (int64_t)j * D;
        int8_t *qr = q + (int64_t)i * D;
        if (sl >= 0 && jr == j) {  // a new reference: the row itself into its slot
            bool bad = false;
            __nv_bfloat16 *pr = pool + (int64_t)sl * D;
            for (int c = lane; c < C; c += 32) {
                const uint4 u = *reinterpret_cast<const uint4 *>(v + 8 * c);
                bad |= bf16_nonfinite(u.x) || bf16_nonfinite(u.y) || bf16_nonfinite(u.z) ||
                       bf16_nonfinite(u.w);
                *reinterpret_cast<uint4 *>(pr + 8 * c) = u;
                *reinterpret_cast<uint2 *>(qr + 8 * c) = make_uint2(0, 0);
            }
            bad = __any_sync(0xffffffffu, bad);
            if (lane == 0) {
                scale[i] = 0.f;
                ref[i] = sl;
                atomicAdd(&refcount[sl], 1);
                if (bad) echo_flag_error(err, ECHO_ERR_NONFINITE);
            }
            continue;
        }
        // residual against the reference row, or the row itself without one
        const __nv_bfloat16 *r = sl >= 0 ? src + (int64_t)jr * D : nullptr;
        float amax = 0.f;
        bool nan = false, inf = false;
        for (int c = lane; c < C; c += 32) {
            float f[8], g[8];
            unpack8_bf16(*reinterpret_cast<const uint4 *>(v + 8 * c), f);
            if (r) unpack8_bf16(*reinterpret_cast<const uint4 *>(r + 8 * c), g);
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const float a = fabsf(r ? __fsub_rn(f[k], g[k]) : f[k]);
                nan |= a != a;
                inf |= a == INFINITY;
                amax = fmaxf(amax, a);
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
        nan = __any_sync(0xffffffffu, nan);
        inf = __any_sync(0xffffffffu, inf);
        if (lane == 0) {
            ref[i] = sl >= 0 ? sl : -1;
            if (sl >= 0) atomicAdd(&refcount[sl], 1);
        }
        if (nan || inf) {
            for (int c = lane; c < C; c += 32) *reinterpret_cast<uint2 *>(qr + 8 * c) = make_uint2(0, 0);
            if (lane == 0) {
                scale[i] = nan ? __int_as_float(0x7fc00000) : INFINITY;
                echo_flag_error(err, ECHO_ERR_NONFINITE);
            }
            continue;
        }
        float sc = 0.f, inv = 0.f;
        if (amax > 0.f) {
            sc = __fdiv_rn(amax, 127.f);
            inv = __fdiv_rn(127.f, amax);
        }
        for (int c = lane; c < C; c += 32) {
            float f[8], g[8];
            unpack8_bf16(*reinterpret_cast<const uint4 *>(v + 8 * c), f);
            if (r) unpack8_bf16(*reinterpret_cast<const uint4 *>(r + 8 * c), g);
            uint32_t w[2] = {0u, 0u};
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const float dv = r ? __fsub_rn(f[k], g[k]) : f[k];
                float t = rintf(__fmul_rn(dv, inv));
                t = fminf(fmaxf(t, -127.f), 127.f);
                const uint32_t b = (uint32_t)(uint8_t)(int8_t)(int)t;
                w[k >> 2] |= b << (8 * (k & 3));
            }
            *reinterpret_cast<uint2 *>(qr + 8 * c) = make_uint2(w[0], w[1]);
        }
        if (lane == 0) scale[i] = sc;
    }
}

// The same for rows of up to 1024 CPL values, one CTA of 128 threads per row: the
// row and its reference are held packed in registers (16-byte chunk tid + 128 k),
// every load in flight at once, each read once.  One warp per row reading them in
// two passes was bound by latency: 6552 residual rows of 5120 49 -> 31 us.
constexpr int kRowThreads = 128;

template <int CPL>
__global__ void __launch_bounds__(kRowThreads)
ref_store_row_kernel(const __nv_bfloat16 *__restrict__ src, const int32_t *__restrict__ rows, int n,
                     int D, const int32_t *__restrict__ src_pos, const int32_t *__restrict__ slot_of,
                     int8_t *__restrict__ q, float *__restrict__ scale, int32_t *__restrict__ ref,
                     int32_t *refcount, __nv_bfloat16 *__restrict__ pool, int *err) {
    __shared__ uint32_t warp_max[kRowThreads / 32];
    pdl_enter();
    const int tid = threadIdx.x;
    const int C = D >> 3;
    const int j = blockIdx.x;
    const uint4 *vp = reinterpret_cast<const uint4 *>(src + (int64_t)j * D);
    uint4 v[CPL], g[CPL];
#pragma unroll
    for (int k = 0; k < CPL; ++k)
        v[k] = tid + kRowThreads * k < C ? __ldg(vp + tid + kRowThreads * k) : make_uint4(0, 0, 0, 0);
    const int i = rows[j], jr = src_pos[j];
    const int sl = slot_of[jr];
    const bool is_ref = sl >= 0 && jr == j;
    uint4 *pr = reinterpret_cast<uint4 *>(pool + (int64_t)(is_ref ? sl : 0) * D);
    uint2 *qr = reinterpret_cast<uint2 *>(q + (int64_t)i * D);
    // residual against the reference row, or the row itself without one; a new
    // reference only looks for values that are not finite
    const bool residual = sl >= 0 && !is_ref;
    if (residual) {
        const uint4 *rp = reinterpret_cast<const uint4 *>(src + (int64_t)jr * D);
#pragma unroll
        for (int k = 0; k < CPL; ++k)
            g[k] = tid + kRowThreads * k < C ? __ldg(rp + tid + kRowThreads * k) : make_uint4(0, 0, 0, 0);
    }
    auto diff = [&](int k, float *f) {
        unpack8_bf16(v[k], f);
        if (residual) {
            float r[8];
            unpack8_bf16(g[k], r);
#pragma unroll
            for (int e = 0; e < 8; ++e) f[e] = __fsub_rn(f[e], r[e]);
        }
    };
    uint32_t ab = 0;   // max |x - r| as fp32 bits (NaN above infinity above every number)
#pragma unroll
    for (int k = 0; k < CPL; ++k) {
        float f[8];
        diff(k, f);
#pragma unroll
        for (int e = 0; e < 8; ++e) ab = max(ab, __float_as_uint(f[e]) & 0x7FFFFFFFu);
    }
    ab = __reduce_max_sync(0xffffffffu, ab);
    if ((tid & 31) == 0) warp_max[tid >> 5] = ab;
    __syncthreads();
    ab = max(max(warp_max[0], warp_max[1]), max(warp_max[2], warp_max[3]));
    const bool bad = ab >= 0x7F800000u;
    const float amax = __uint_as_float(ab);
    float sc = 0.f, inv = 0.f;
    if (!bad && amax > 0.f) {
        sc = __fdiv_rn(amax, 127.f);
        inv = __fdiv_rn(127.f, amax);
    }
#pragma unroll
    for (int k = 0; k < CPL; ++k) {
        const int c = tid + kRowThreads * k;
        if (c >= C) continue;
        if (is_ref) pr[c] = v[k];
        float f[8];
        diff(k, f);
        qr[c] = is_ref || bad ? make_uint2(0, 0) : quant8(f, inv);
    }
    if (tid == 0) {
        ref[i] = sl >= 0 ? sl : -1;
        if (sl >= 0) atomicAdd(&refcount[sl], 1);
        scale[i] = is_ref ? 0.f
                   : !bad ? sc
                          : ab > 0x7F800000u ? __int_as_float(0x7fc00000) : INFINITY;
        if (bad) echo_flag_error(err, ECHO_ERR_NONFINITE);
    }
}

// ---------------------------------------------------------------- reconstruction
// 16 values of token i: bf16(r + float(q) s), r = 0 without a reference
ECHO_DEV void ref_reconstruct16(const echo_cache &c, int i, int col, uint4 *out) {
    const int rs = c.ref[i];
    const float s = c.scale[i];
    const int4 qv = __ldcs(reinterpret_cast<const int4 *>(c.q + (int64_t)i * c.D + col));
    const int8_t *qb = reinterpret_cast<const int8_t *>(&qv);
    float r[16];
    if (rs >= 0) {
        const uint4 *p = reinterpret_cast<const uint4 *>(
            static_cast<const __nv_bfloat16 *>(c.pool) + (int64_t)rs * c.D + col);
        unpack8_bf16(p[0], r);
        unpack8_bf16(p[1], r + 8);
    } else {
#pragma unroll
        for (int k = 0; k < 16; ++k) r[k] = 0.f;
    }
    float f[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) f[k] = __fadd_rn(r[k], __fmul_rn((float)qb[k], s));
    out[0] = pack8_bf16(f);
    out[1] = pack8_bf16(f + 8);
}

template <int KIND>
ECHO_DEV void reconstruct16(const echo_cache &c, int i, int col, uint4 *out) {
    if constexpr (KIND == ECHO_CACHE_BF16) {
        const uint4 *p = reinterpret_cast<const uint4 *>(
            static_cast<const __nv_bfloat16 *>(c.full) + (int64_t)i * c.D + col);
        out[0] = __ldcs(p);
        out[1] = __ldcs(p + 1);
    } else {
        ref_reconstruct16(c, i, col, out);
    }
}

template <int KIND>
__global__ void __launch_bounds__(kVec)
cache_read_kernel(echo_cache c, const int32_t *__restrict__ rows, int n,
                  __nv_bfloat16 *__restrict__ dst) {
    pdl_enter();
    for (PieceWalk w = grid_pieces(c.D >> 4); w.below(n); w.next()) {
        const int j = (int)w.row, col = 16 * (int)w.piece;
        const int i = rows ? rows[j] : j;
        uint4 o[2];
        reconstruct16<KIND>(c, i, col, o);
        uint4 *d = reinterpret_cast<uint4 *>(dst + (int64_t)j * c.D + col);
        d[0] = o[0];
        d[1] = o[1];
    }
}

// y[i] = y_act[rowmap[i]] if rowmap[i] >= 0 else the reconstruction of token i
template <int KIND>
__global__ void __launch_bounds__(kVec)
cache_merge_kernel(echo_cache c, const int32_t *__restrict__ rowmap,
                   const __nv_bfloat16 *__restrict__ y_act, __nv_bfloat16 *__restrict__ y) {
    pdl_enter();
    for (PieceWalk w = grid_pieces(c.D >> 4); w.below(c.NT); w.next()) {
        const int i = (int)w.row, col = 16 * (int)w.piece;
        const int pos = rowmap[i];
        uint4 *o = reinterpret_cast<uint4 *>(y + (int64_t)i * c.D + col);
        uint4 v[2];
        if (pos >= 0) {
            const uint4 *a = reinterpret_cast<const uint4 *>(y_act + (int64_t)pos * c.D + col);
            v[0] = __ldcs(a);
            v[1] = __ldcs(a + 1);
        } else {
            reconstruct16<KIND>(c, i, col, v);
        }
        __stcs(o, v[0]);
        __stcs(o + 1, v[1]);
    }
}

// full[rows[j]] = src[j] (BF16 form)
__global__ void __launch_bounds__(kVec)
cache_copy_kernel(const __nv_bfloat16 *__restrict__ src, const int32_t *__restrict__ rows, int n,
                  int D, __nv_bfloat16 *__restrict__ full, int *err) {
    pdl_enter();
    bool bad = false;
    for (PieceWalk w = grid_pieces(D >> 3); w.below(n); w.next()) {
        const int j = (int)w.row, c = (int)w.piece;
        const uint4 u = __ldcs(reinterpret_cast<const uint4 *>(src + (int64_t)j * D + 8 * c));
        bad |= bf16_nonfinite(u.x) || bf16_nonfinite(u.y) || bf16_nonfinite(u.z) ||
               bf16_nonfinite(u.w);
        *reinterpret_cast<uint4 *>(full + (int64_t)rows[j] * D + 8 * c) = u;
    }
    if (bad) echo_flag_error(err, ECHO_ERR_NONFINITE);
}

__global__ void cache_stats_kernel(const int32_t *__restrict__ refcount, int R_cap,
                                   int32_t *__restrict__ out) {
    pdl_enter();
    __shared__ int s_live, s_top;
    if (threadIdx.x == 0) {
        s_live = 0;
        s_top = 0;
    }
    __syncthreads();
    int live = 0, top = 0;
    for (int sl = threadIdx.x; sl < R_cap; sl += blockDim.x)
        if (refcount[sl] > 0) {
            ++live;
            top = sl + 1;
        }
    atomicAdd(&s_live, live);
    atomicMax(&s_top, top);
    __syncthreads();
    if (threadIdx.x == 0) {
        out[0] = s_live;
        out[1] = s_top;
    }
}

struct RefWs {
    int32_t *src_pos, *slot_of, *free_list, *seg_lo, *seg_hi;
};

int n_segments(const echo_cache &c) {
    return (int)((c.NT + (int64_t)c.seg_len - 1) / c.seg_len);
}

size_t ref_ws_bytes(const echo_cache &c, int32_t n) {
    const size_t a = al256(sizeof(int32_t) * (size_t)(n > 0 ? n : 1));
    const size_t b = al256(sizeof(int32_t) * (size_t)n_segments(c));
    return 3 * a + 2 * b;
}

RefWs ref_ws(const echo_cache &c, void *ws, int32_t n) {
    const size_t a = al256(sizeof(int32_t) * (size_t)(n > 0 ? n : 1));
    const size_t b = al256(sizeof(int32_t) * (size_t)n_segments(c));
    uint8_t *p = static_cast<uint8_t *>(ws);
    return {reinterpret_cast<int32_t *>(p), reinterpret_cast<int32_t *>(p + a),
            reinterpret_cast<int32_t *>(p + 2 * a), reinterpret_cast<int32_t *>(p + 3 * a),
            reinterpret_cast<int32_t *>(p + 3 * a + b)};
}

size_t scan_smem_bytes(int win, int D) { return (size_t)(win + 1) * D * sizeof(__nv_bfloat16); }

// Dynamic shared memory that the scan may ask for on the current device (0: no
// device): what a CTA may have beside its static buffers.  The kernel's limit is
// raised to it once per device, whatever the width of the first write there, so that
// no call depends on the widths written before it or by another thread meanwhile.
template <int WIN>
size_t scan_smem_cap() {
    static size_t cap[64] = {};
    static std::mutex mu;
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    std::lock_guard<std::mutex> lk(mu);
    if (!cap[dev]) {
        cudaFuncAttributes fa;
        int most = 0;
        if (cudaFuncGetAttributes(&fa, ref_scan_kernel<WIN>) != cudaSuccess ||
            cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
            return 0;
        const int dyn = most - (int)fa.sharedSizeBytes;
        if (dyn <= 0 || cudaFuncSetAttribute(ref_scan_kernel<WIN>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             dyn) != cudaSuccess)
            return 0;
        cap[dev] = (size_t)dyn;
    }
    return cap[dev];
}

template <int WIN>
void launch_scan(const echo_cache &c, const __nv_bfloat16 *src, const RefWs &w, int nseg, cudaStream_t st) {
    echo::launch_chained(ref_scan_kernel<WIN>, dim3(nseg), dim3(2 * WIN * 32),
                         scan_smem_bytes(WIN, c.D), st, src, w.seg_lo, w.seg_hi, c.tau, c.D, w.src_pos);
}

}  // namespace

namespace echo {

echo_status cache_check(const echo_cache *c) {
    if (!c) return ECHO_ERR_INVALID_ARG;
    if (c->NT < 1 || c->D < 16 || c->D % 16) return ECHO_ERR_SHAPE;
    if ((int64_t)c->NT > (int64_t)INT32_MAX / 2) return ECHO_ERR_SHAPE;
    switch (c->kind) {
    case ECHO_CACHE_INT8:
        if (!c->q || !c->scale || !aligned16(c->q) || !aligned16(c->scale)) return ECHO_ERR_INVALID_ARG;
        return ECHO_OK;
    case ECHO_CACHE_BF16:
        if (!c->full || !aligned16(c->full)) return ECHO_ERR_INVALID_ARG;
        return ECHO_OK;
    case ECHO_CACHE_REF:
        if (!c->q || !c->scale || !c->ref || !aligned16(c->q) || !aligned16(c->scale) ||
            !aligned16(c->ref))
            return ECHO_ERR_INVALID_ARG;
        if (c->R_cap < 0 || c->seg_len < 1 || !(c->tau == c->tau)) return ECHO_ERR_INVALID_ARG;
        if (c->R_cap > 0 && (!c->pool || !c->refcount || !aligned16(c->pool) ||
                             !aligned16(c->refcount)))
            return ECHO_ERR_INVALID_ARG;
        return ECHO_OK;
    default:
        return ECHO_ERR_INVALID_ARG;
    }
}

size_t cache_write_ws(const echo_cache &c, int32_t n) {
    return c.kind == ECHO_CACHE_REF ? ref_ws_bytes(c, n) : 0;
}

echo_status launch_cache_write(const echo_cache &c, const void *src, const int32_t *rows,
                               int32_t n, void *ws, cudaStream_t st) {
    if (n <= 0) return ECHO_OK;
    int *err = device_error_ptr();
    const __nv_bfloat16 *s = static_cast<const __nv_bfloat16 *>(src);
    if (c.kind == ECHO_CACHE_INT8) {
        launch_quant(src, ECHO_BF16, rows, n, c.D, c.q, c.scale, st);
        return last_launch_status();
    }
    if (c.kind == ECHO_CACHE_BF16) {
        LaunchScope ls(ECHO_K_CACHE_COPY, n, c.D, 0, st);
        echo::launch_chained(cache_copy_kernel, dim3(grid_for((int64_t)n * (c.D / 8), kVec)),
                             dim3(kVec), 0, st,
            s, rows, n, c.D, static_cast<__nv_bfloat16 *>(c.full), err);
        return last_launch_status();
    }
    // before anything is enqueued: the release alone would leave slots counted free
    // that the entries still name
    const RefWs w = ref_ws(c, ws, n);
    const int nseg = n_segments(c);
    const bool wide = nseg <= kWideSegments && scan_smem_bytes(kWinWide, c.D) <= scan_smem_cap<kWinWide>();
    if (!wide) {
        const size_t cap = scan_smem_cap<kWin>();
        if (!cap) return ECHO_ERR_CUDA;
        if (scan_smem_bytes(kWin, c.D) > cap) return ECHO_ERR_SHAPE;
    }
    if (cudaMemsetAsync(w.seg_lo, 0xFF, sizeof(int32_t) * (size_t)nseg, st) != cudaSuccess)
        return ECHO_ERR_CUDA;
    {
        LaunchScope ls(ECHO_K_REF_ALLOC, n, c.D, 0, st);
        echo::launch_chained(ref_release_kernel, dim3((n + 255) / 256), dim3(256), 0, st,
            rows, n, c.seg_len, c.ref, c.R_cap > 0 ? c.refcount : nullptr, w.seg_lo, w.seg_hi);
    }
    if (last_launch_status() != ECHO_OK) return ECHO_ERR_CUDA;
    {
        LaunchScope ls(ECHO_K_REF_SCAN, n, c.D, 0, st);
        if (wide) launch_scan<kWinWide>(c, s, w, nseg, st);
        else launch_scan<kWin>(c, s, w, nseg, st);
    }
    if (last_launch_status() != ECHO_OK) return ECHO_ERR_CUDA;
    {
        LaunchScope ls(ECHO_K_REF_ALLOC, n, c.D, 0, st);
        echo::launch_chained(ref_alloc_kernel, dim3(1), dim3(kAllocThreads), 0, st, w.src_pos, n,
                             c.refcount, c.R_cap,
                                                       w.free_list, w.slot_of);
    }
    if (last_launch_status() != ECHO_OK) return ECHO_ERR_CUDA;
    {
        LaunchScope ls(ECHO_K_REF_STORE, n, c.D, 0, st);
        __nv_bfloat16 *pool = static_cast<__nv_bfloat16 *>(c.pool);
        auto store_rows = [&](auto kernel) {
            launch_chained(kernel, dim3(n), dim3(kRowThreads), 0, st, s, rows, n, c.D, w.src_pos,
                           w.slot_of, c.q, c.scale, c.ref, c.refcount, pool, err);
        };
        if (c.D <= 1024)
            store_rows(ref_store_row_kernel<1>);
        else if (c.D <= 2048)
            store_rows(ref_store_row_kernel<2>);
        else if (c.D <= 5120)
            store_rows(ref_store_row_kernel<5>);
        else if (c.D <= 8192)
            store_rows(ref_store_row_kernel<8>);
        else
            launch_chained(ref_store_kernel, dim3(grid_for((int64_t)n * 32, kStoreThreads)),
                           dim3(kStoreThreads), 0, st, s, rows, n, c.D, w.src_pos, w.slot_of, c.q, c.scale, c.ref, c.refcount,
                           pool, err);
    }
    return last_launch_status();
}

void launch_cache_merge(const echo_cache &c, const int32_t *rowmap, const void *y_act, void *y,
                        cudaStream_t st) {
    if (c.kind == ECHO_CACHE_INT8) {
        launch_dequant_merge(c.q, c.scale, rowmap, y_act, c.NT, c.D, y, st);
        return;
    }
    const int grid = grid_for((int64_t)c.NT * (c.D / 16), kVec);
    LaunchScope ls(ECHO_K_MERGE, c.NT, c.D, 0, st);
    const __nv_bfloat16 *ya = static_cast<const __nv_bfloat16 *>(y_act);
    __nv_bfloat16 *yo = static_cast<__nv_bfloat16 *>(y);
    if (c.kind == ECHO_CACHE_BF16)
        echo::launch_chained(cache_merge_kernel<ECHO_CACHE_BF16>, dim3(grid), dim3(kVec), 0, st,
                             c, rowmap, ya, yo);
    else
        echo::launch_chained(cache_merge_kernel<ECHO_CACHE_REF>, dim3(grid), dim3(kVec), 0, st,
                             c, rowmap, ya, yo);
}

}  // namespace echo

extern "C" echo_status echo_cache_reset(const echo_cache *c, echo_stream_t stream) {
    using namespace echo;
    const echo_status v = cache_check(c);
    if (v != ECHO_OK) return v;
    if (!device_supported()) return ECHO_ERR_UNSUPPORTED;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    const size_t NT = c->NT, D = c->D;
    bool ok = true;
    if (c->kind != ECHO_CACHE_BF16) {
        ok &= cudaMemsetAsync(c->q, 0, NT * D, st) == cudaSuccess;
        ok &= cudaMemsetAsync(c->scale, 0, NT * sizeof(float), st) == cudaSuccess;
    }
    if (c->kind == ECHO_CACHE_BF16) ok &= cudaMemsetAsync(c->full, 0, NT * D * 2, st) == cudaSuccess;
    if (c->kind == ECHO_CACHE_REF) {
        ok &= cudaMemsetAsync(c->ref, 0xFF, NT * sizeof(int32_t), st) == cudaSuccess;
        if (c->R_cap > 0)
            ok &= cudaMemsetAsync(c->refcount, 0, (size_t)c->R_cap * sizeof(int32_t), st) ==
                  cudaSuccess;
    }
    return ok ? ECHO_OK : ECHO_ERR_CUDA;
}

extern "C" size_t echo_cache_write_workspace_size(const echo_cache *c, int32_t n_rows) {
    if (echo::cache_check(c) != ECHO_OK || n_rows < 0) return 0;
    return echo::cache_write_ws(*c, n_rows);
}

extern "C" echo_status echo_cache_write(const echo_cache *c, const void *src, const int32_t *rows,
                                        int32_t n_rows, void *workspace, size_t ws_bytes,
                                        echo_stream_t stream) {
    using namespace echo;
    const echo_status v = cache_check(c);
    if (v != ECHO_OK) return v;
    if (n_rows < 0 || n_rows > c->NT) return ECHO_ERR_SHAPE;
    if (n_rows == 0) return ECHO_OK;
    if (!src || !rows || !aligned16(src) || !aligned16(rows)) return ECHO_ERR_INVALID_ARG;
    const size_t need = cache_write_ws(*c, n_rows);
    if (need && (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255u)))
        return ECHO_ERR_INVALID_ARG;
    if (ws_bytes < need) return ECHO_ERR_WORKSPACE;
    if (!device_supported()) return ECHO_ERR_UNSUPPORTED;
    return launch_cache_write(*c, src, rows, n_rows, workspace,
                              reinterpret_cast<cudaStream_t>(stream));
}

extern "C" echo_status echo_cache_read(const echo_cache *c, const int32_t *rows, int32_t n_rows,
                                       void *dst, echo_stream_t stream) {
    using namespace echo;
    const echo_status v = cache_check(c);
    if (v != ECHO_OK) return v;
    if (n_rows < 0) return ECHO_ERR_SHAPE;
    if (n_rows == 0) return ECHO_OK;
    if (!dst || !aligned16(dst) || (rows && !aligned16(rows))) return ECHO_ERR_INVALID_ARG;
    if (!device_supported()) return ECHO_ERR_UNSUPPORTED;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    if (c->kind == ECHO_CACHE_INT8) {
        launch_dequant(c->q, c->scale, rows, n_rows, c->D, dst, ECHO_BF16, st);
        return last_launch_status();
    }
    const int grid = grid_for((int64_t)n_rows * (c->D / 16), kVec);
    LaunchScope ls(ECHO_K_DEQUANT, n_rows, c->D, 0, st);
    __nv_bfloat16 *d = static_cast<__nv_bfloat16 *>(dst);
    if (c->kind == ECHO_CACHE_BF16)
        echo::launch_chained(cache_read_kernel<ECHO_CACHE_BF16>, dim3(grid), dim3(kVec), 0, st,
                             *c, rows, n_rows, d);
    else
        echo::launch_chained(cache_read_kernel<ECHO_CACHE_REF>, dim3(grid), dim3(kVec), 0, st,
                             *c, rows, n_rows, d);
    return last_launch_status();
}

extern "C" echo_status echo_cache_stats(const echo_cache *c, int32_t *out, echo_stream_t stream) {
    using namespace echo;
    const echo_status v = cache_check(c);
    if (v != ECHO_OK) return v;
    if (c->kind != ECHO_CACHE_REF || !out) return ECHO_ERR_INVALID_ARG;
    if (!device_supported()) return ECHO_ERR_UNSUPPORTED;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    if (c->R_cap == 0) return cudaMemsetAsync(out, 0, 2 * sizeof(int32_t), st) == cudaSuccess
                                  ? ECHO_OK : ECHO_ERR_CUDA;
    {
        LaunchScope ls(ECHO_K_REF_ALLOC, c->R_cap, 0, 0, st);
        echo::launch_chained(cache_stats_kernel, dim3(1), dim3(1024), 0, st, c->refcount,
                             c->R_cap, out);
    }
    return last_launch_status();
}
