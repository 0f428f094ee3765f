// The search of arXiv 2510.18136 Sec. 2.2 for short windows (up to 64 samples: the 25-sample
// real-time block, the 75-fold binned window, injection campaigns), candidate records only.
//
// A pixel of such a window is a few kilobytes and a DM row a few dozen samples, so a warp per DM row
// (the kernels for longer windows) leaves lanes idle and spends its time in warp scans, warp
// maxima and per-pixel hand-overs.  Here a lane is a pixel: a CTA takes 32 consecutive pixels, and each
// of its warps a contiguous group of the distinct DM rows of all 32.
//  * The pixels' samples are copied to shared memory (widened to FP32) at an odd pixel pitch, so that
//    the 32 lanes reading one (subband, sample) hit 32 banks whatever the shift, which is the same
//    for all lanes.
//  * A thread holds its pixel's de-dispersed row D[t] and prefix P[t] in registers and updates D from one
//    row to the next by the subbands whose shift changed, as the other kernels do.  Prefix,
//    boxcars and maxima need no communication between lanes.  Pairs of samples (w = 2) are summed
//    without the prefix: a sample that is not a number, or a bright one, does not reach those after it.
//  * D past the valid range is set to -inf; later rows of a group have shorter ranges (delays
//    grow with the DM), so an element once out of range stays out, and every trial that reads
//    it is -inf or NaN and drops out of the maximum.
//  * Only the best (row, width) is tracked.  At the end each pixel's best row is rebuilt from all
//    subbands (the samples shared out over the warps), and the earliest sample reaching its
//    maximum, with that maximum's S/N, goes to the record, the quotient corrected once.
// Bound by instruction issue: per sample and row 1.5 operations per width, one for the prefix and
// three per changed subband.  301 x 301 pixels x 16 subbands x 25 samples in FP32, 16 DM, 5 widths:
// 106 us (1.4 TB/s), where the warp-per-row kernel with CTA barriers takes 3119 us; 16 binned samples,
// one DM: 37 us (387 us in the barrier-free kernel).
#include <algorithm>
#include <climits>

#include "nsfrb.h"
#include "nsfrb_internal.h"
#include "plan_internal.h"
#include "search_impl.cuh"

namespace nsfrb {
namespace dev {

constexpr int kShortPix = 32;    // pixels per CTA, one per lane
constexpr int kShortPad = 128;   // words after the tile: a row is read up to max(NT) + shift past its start

__host__ __device__ inline int short_pitch(int n_sub, int n_t) { return (n_sub * n_t) | 1; }

struct ShortLayout {
    size_t table, xs, sinv, best, total;
};

__host__ __device__ inline ShortLayout short_layout(const SearchParams &p, int n_warps) {
    ShortLayout L{};
    size_t o = 0;
    L.table = o;
    o += align_up(sizeof(int32_t) * ((size_t)p.n_u * kInfo + p.n_deltas + (size_t)p.n_u * p.n_sub), 16);
    L.xs = o;
    // the tile; afterwards the same words hold the rebuilt rows [n_t + 1][kShortPix]
    size_t words = (size_t)kShortPix * short_pitch(p.n_sub, p.n_t) + kShortPad;
    const size_t rows = (size_t)kShortPix * (p.n_t + 1);
    o += align_up(sizeof(float) * (words > rows ? words : rows), 16);
    L.sinv = o;
    o += sizeof(float) * (size_t)p.n_w * kShortPix;
    L.best = o;
    o += (sizeof(float) + sizeof(int32_t)) * (size_t)n_warps * kShortPix;
    L.total = align_up(o, 16);
    return L;
}

// Maximum over t of the boxcars of width W: D itself for W = 1, D[t] + D[t + 1] for W = 2, else P[t + W] - P[t].
template <int NT, int W>
__device__ __forceinline__ float short_max(const float2 (&D)[NT / 2], const float2 (&P)[NT / 2 + 1]) {
    float acc[3] = {neg_inf(), neg_inf(), neg_inf()};
    if constexpr (W == 1) {
#pragma unroll
        for (int m = 0; m < NT / 2; ++m) acc[m % 3] = fmax3(acc[m % 3], D[m].x, D[m].y);
    } else if constexpr (W == 2) {
#pragma unroll
        for (int t = 0; t + 2 < NT; t += 2)
            acc[(t >> 1) % 3] = fmax3(acc[(t >> 1) % 3], pget(D, t) + pget(D, t + 1), pget(D, t + 1) + pget(D, t + 2));
        acc[2] = fmaxf(acc[2], pget(D, NT - 2) + pget(D, NT - 1));
    } else if constexpr (W % 2 == 0) {
        constexpr int N = NT - W + 1;   // trials t = 0 .. NT - W
#pragma unroll
        for (int m = 0; m < N / 2; ++m) {
            const float2 b = sub2(P[m + W / 2], P[m]);
            acc[m % 3] = fmax3(acc[m % 3], b.x, b.y);
        }
        acc[2] = fmaxf(acc[2], pget(P, NT) - pget(P, NT - W));   // N is odd
    } else {
        constexpr int N = NT - W + 1;
#pragma unroll
        for (int t = 0; t + 1 < N; t += 2)
            acc[(t >> 1) % 3] = fmax3(acc[(t >> 1) % 3], pget(P, t + W) - pget(P, t), pget(P, t + 1 + W) - pget(P, t + 1));
        if constexpr (N & 1) acc[2] = fmaxf(acc[2], pget(P, NT) - pget(P, NT - W));
    }
    return fmax3(acc[0], acc[1], acc[2]);
}

#define NSFRB_SHORT_W8(X, B) X(B + 1) X(B + 2) X(B + 3) X(B + 4) X(B + 5) X(B + 6) X(B + 7) X(B + 8)

// The width is the same for every lane; each has compile-time code (register arrays).
template <int NT>
__device__ __forceinline__ float short_max_any(int w, const float2 (&D)[NT / 2], const float2 (&P)[NT / 2 + 1]) {
    switch (w) {
#define NSFRB_SHORT_CASE(W)                                     \
    case W:                                                     \
        if constexpr ((W) <= NT) return short_max<NT, (W)>(D, P); \
        break;
        NSFRB_SHORT_W8(NSFRB_SHORT_CASE, 0)
        NSFRB_SHORT_W8(NSFRB_SHORT_CASE, 8)
        NSFRB_SHORT_W8(NSFRB_SHORT_CASE, 16)
        NSFRB_SHORT_W8(NSFRB_SHORT_CASE, 24)
        NSFRB_SHORT_W8(NSFRB_SHORT_CASE, 32)
        NSFRB_SHORT_W8(NSFRB_SHORT_CASE, 40)
        NSFRB_SHORT_W8(NSFRB_SHORT_CASE, 48)
        NSFRB_SHORT_W8(NSFRB_SHORT_CASE, 56)
#undef NSFRB_SHORT_CASE
        default:
            break;
    }
    return neg_inf();
}

template <int NT>
__global__ void __launch_bounds__(NT > 32 ? 256 : 128, NT > 32 ? 1 : 4)
search_kernel_short(const __grid_constant__ SearchParams p) {
    extern __shared__ __align__(128) unsigned char smem[];
    const int n_warps = blockDim.x >> 5;
    const ShortLayout lay = short_layout(p, n_warps);
    int32_t *s_table = reinterpret_cast<int32_t *>(smem + lay.table);
    float *xs = reinterpret_cast<float *>(smem + lay.xs);
    float *s_inv = reinterpret_cast<float *>(smem + lay.sinv);                       // [n_w][32]
    float *s_bs = reinterpret_cast<float *>(smem + lay.best);                        // [n_warps][32]
    int32_t *s_buw = reinterpret_cast<int32_t *>(s_bs + (size_t)n_warps * kShortPix);   // row * kMaxW + width index

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n_sub = p.n_sub, n_t = p.n_t, ne = n_sub * n_t;
    const int pitch = short_pitch(n_sub, n_t);
    int64_t n_items = p.n_items;
    if (p.n_items_dev) n_items = *p.n_items_dev;
    auto item_pixel = [&](int64_t it) -> int64_t {
        return p.pix_list ? static_cast<int64_t>(p.pix_list[it]) : p.pix0 + it;
    };
    const int table_words = p.n_u * kInfo + p.n_deltas + p.n_u * n_sub;
    for (int i = tid; i < table_words; i += blockDim.x) s_table[i] = p.table[i];
    const int32_t *s_info = s_table;
    const int32_t *s_delta = s_table + p.n_u * kInfo;
    const int32_t *s_shift = s_delta + p.n_deltas;
    // one set of pixels per CTA, or, where a device count says how many there are (re-scoring), several
    for (int64_t it0 = static_cast<int64_t>(blockIdx.x) * kShortPix; it0 < n_items;
         it0 += static_cast<int64_t>(gridDim.x) * kShortPix) {
        const int n_here = static_cast<int>(min(static_cast<int64_t>(kShortPix), n_items - it0));

        // ---- samples, 1 / (sigma sqrt(w))
        for (int q = warp; q < kShortPix; q += n_warps) {
            float *dst = xs + (size_t)q * pitch;
            const int64_t from = q < n_here ? (item_pixel(it0 + q) - p.cube_pix0) * ne : 0;
            if (q >= n_here) {
                for (int e = lane; e < ne; e += 32) dst[e] = 0.0f;
            } else if (p.dtype == 0) {
                const float *src = static_cast<const float *>(p.cube) + from;
                for (int e = lane; e < ne; e += 32)
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst + e)), "l"(src + e) : "memory");
            } else {
                const unsigned short *src = static_cast<const unsigned short *>(p.cube) + from;
#pragma unroll 8
                for (int e = lane; e < ne; e += 32) dst[e] = widen16(src[e], p.dtype);
            }
        }
        for (int i = tid; i < kShortPad; i += blockDim.x) xs[(size_t)kShortPix * pitch + i] = 0.0f;
        {
            const float sg = (p.sigma && lane < n_here) ? p.sigma[item_pixel(it0 + lane)] : p.sigma_default;
            for (int wi = warp; wi < p.n_w; wi += n_warps)
                s_inv[wi * kShortPix + lane] = 1.0f / (sg * sqrtf(static_cast<float>(p.widths[wi])));
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();

        // ---- the warp's rows of all 32 pixels
        const int n_ua = p.n_u_active;
        const int n_grp = min(n_warps, n_ua);
        float bs = neg_inf();
        int buw = -1;
        if (warp < n_grp) {
            const int u_lo = (warp * n_ua) / n_grp, u_hi = ((warp + 1) * n_ua) / n_grp;
            const float *xp = xs + (size_t)lane * pitch;
            float2 D[NT / 2];
            int L_prev = NT + 1;
#pragma unroll 1
            for (int u = u_lo; u < u_hi; ++u) {
                const int32_t *info = s_info + u * kInfo;
                if (u == u_lo) {
#pragma unroll
                    for (int m = 0; m < NT / 2; ++m) D[m] = make_float2(0.0f, 0.0f);
                    const int32_t *sh = s_shift + u * n_sub;
#pragma unroll 1
                    for (int k = 0; k < n_sub; ++k) {
                        const float *x = xp + k * n_t + sh[k];
#pragma unroll
                        for (int m = 0; m < NT / 2; ++m) D[m] = add2(D[m], make_float2(x[2 * m], x[2 * m + 1]));
                    }
                } else {
                    const int d0 = info[UI_DOFF], nd = info[UI_ND];
#pragma unroll 1
                    for (int e = d0; e < d0 + nd; ++e) {
                        const uint32_t pk = static_cast<uint32_t>(s_delta[e]);
                        const int k = pk & 63u, so = (pk >> 6) & 0x1fffu, sn = pk >> 19;
                        const float *xo = xp + k * n_t + so;
                        if (sn == so + 1) {   // both values from one read of the row
                            float a = xo[0];
#pragma unroll
                            for (int m = 0; m < NT / 2; ++m) {
                                const float b = xo[2 * m + 1], c = xo[2 * m + 2];
                                D[m] = add2(D[m], make_float2(b - a, c - b));
                                a = c;
                            }
                        } else {
                            const float *xn = xp + k * n_t + sn;
#pragma unroll
                            for (int m = 0; m < NT / 2; ++m)
                                D[m] = sub2(add2(D[m], make_float2(xn[2 * m], xn[2 * m + 1])),
                                            make_float2(xo[2 * m], xo[2 * m + 1]));
                        }
                    }
                }
                const int L = n_t - info[UI_SMAX];
                if (L != L_prev) {
#pragma unroll
                    for (int m = 0; m < NT / 2; ++m) {
                        if (2 * m >= L) D[m].x = neg_inf();
                        if (2 * m + 1 >= L) D[m].y = neg_inf();
                    }
                    L_prev = L;
                }
                float2 P[NT / 2 + 1];
                float run = 0.0f;
                P[0].x = 0.0f;
#pragma unroll
                for (int t = 0; t < NT; ++t) {
                    run += pget(D, t);
                    pset(P, t + 1, run);
                }
#pragma unroll 1
                for (int wi = 0; wi < p.n_w; ++wi) {
                    const int w = p.widths[wi];
                    if (w > L) break;
                    const float s = short_max_any<NT>(w, D, P) * s_inv[wi * kShortPix + lane];
                    if (s > bs) {   // ascending rows and widths: ties keep the smallest
                        bs = s;
                        buw = u * kMaxW + wi;
                    }
                }
            }
            s_bs[warp * kShortPix + lane] = bs;
            s_buw[warp * kShortPix + lane] = buw;
        }
        __syncthreads();

        // ---- the pixel's best row, rebuilt from all subbands: warp q takes samples q, q + n_warps, ...
        for (int g = 0; g < n_grp; ++g) {
            const float s = s_bs[g * kShortPix + lane];
            if (g == 0 || s > bs) {
                bs = s;
                buw = s_buw[g * kShortPix + lane];
            }
        }
        if (n_grp == 0) buw = -1;
        const bool any = buw >= 0;
        const int bu = any ? buw / kMaxW : 0, bwi = any ? buw % kMaxW : 0;
        const int L = n_t - s_info[bu * kInfo + UI_SMAX];
        constexpr int kW = NT > 32 ? 8 : 4;          // = n_warps
        constexpr int kMine = (NT + kW - 1) / kW;   // samples per thread
        float d[kMine];
#pragma unroll
        for (int j = 0; j < kMine; ++j) d[j] = 0.0f;
        if (any) {
            const float *xp = xs + (size_t)lane * pitch + warp;
            const int32_t *sh = s_shift + bu * n_sub;
#pragma unroll 2
            for (int k = 0; k < n_sub; ++k) {
                const float *x = xp + k * n_t + sh[k];
#pragma unroll
                for (int j = 0; j < kMine; ++j) d[j] += x[j * kW];
            }
        }
        __syncthreads();   // the last reads of the samples: their words take the rows now
#pragma unroll
        for (int j = 0; j < kMine; ++j)
            if (warp + j * kW < n_t) xs[(warp + j * kW) * kShortPix + lane] = d[j];
        __syncthreads();
        if (warp == 0 && lane < n_here) {
            PixRec r{neg_inf(), -1, -1, -1};
            if (any) {
                const int w = p.widths[bwi];
                const float inv = s_inv[bwi * kShortPix + lane];
                float *col = xs + lane;   // D[t] at col[t * 32]; P[t] in its place for w > 2
                if (w > 2) {
                    float run = 0.0f;
                    for (int t = 0; t <= L; ++t) {
                        const float v = t < L ? col[t * kShortPix] : 0.0f;
                        col[t * kShortPix] = run;
                        run += v;
                    }
                }
                // boxcar t = b[t] + ca a[t] (exact product): D[t] + 0 for w = 1, D[t + 1] + D[t], P[t + w] - P[t]; lanes
                // differ in w, so no branches
                const float *b = col + (w == 1 ? 0 : w == 2 ? 1 : w) * kShortPix;
                const float *a = w == 1 ? xs + (size_t)kShortPix * pitch + kShortPad - 1 : col;
                const int sa = w == 1 ? 0 : kShortPix;
                const float ca = w <= 2 ? 1.0f : -1.0f;
                auto box = [&](int t) { return fmaf(ca, a[t * sa], b[t * kShortPix]); };
                float m = neg_inf();
                for (int t = 0; t + w <= L; ++t) m = fmaxf(m, box(t));
                for (int t = L - w; t >= 0; --t)
                    if (box(t) * inv == m * inv) r.t_idx = t;
                r.snr = record_snr(m, p.sigma ? p.sigma[item_pixel(it0 + lane)] : p.sigma_default, w, inv);
                r.dm_idx = s_info[bu * kInfo + UI_FIRST_D];
                r.w_idx = bwi;
            }
            const int64_t pix = item_pixel(it0 + lane);
            if (p.bad_pix && p.bad_pix[pix]) {
                r = PixRec{neg_inf(), -1, -1, -1};
                atomicOr(p.err, ERR_ZERO_MAD);
            }
            p.rec[pix] = r;
        }
        __syncthreads();   // everything of this set has been read
    }
}

}  // namespace dev

// Warps per CTA for a window this kernel takes (0: another kernel): candidate records of a contiguous
// pixel-major cube with a known noise, up to 64 samples, whose tile fits in shared memory.
int short_warps(const SearchParams &p, int max_smem) {
    if (p.n_t > kShortT || p.full_snr || p.noise_mode != 0 || p.t_wrap || p.t_stride || p.t_off || p.t_off_dev ||
        p.new_blk || p.row_len != p.n_t)
        return 0;
    const int w = p.n_t > 32 ? 8 : 4;
    return dev::short_layout(p, w).total <= static_cast<size_t>(max_smem) ? w : 0;
}

size_t short_smem(const SearchParams &p, int n_warps) { return dev::short_layout(p, n_warps).total; }

cudaError_t launch_search_short(const SearchParams &p, int grid_sm, size_t smem, cudaStream_t s) {
    // where only the device knows the count, as many CTAs as can run at once (at most) loop over it
    const int64_t sets = (p.n_items + dev::kShortPix - 1) / dev::kShortPix;
    const unsigned grid = static_cast<unsigned>(p.n_items_dev ? std::min<int64_t>(sets, 4 * grid_sm) : sets);
    const unsigned threads = 32u * static_cast<unsigned>(p.short_w);
    if (p.n_items <= 0) return cudaSuccess;
    if (p.n_t <= 16)
        dev::search_kernel_short<16><<<grid, threads, smem, s>>>(p);
    else if (p.n_t <= 26)
        dev::search_kernel_short<26><<<grid, threads, smem, s>>>(p);
    else if (p.n_t <= 32)
        dev::search_kernel_short<32><<<grid, threads, smem, s>>>(p);
    else if (p.n_t <= 48)
        dev::search_kernel_short<48><<<grid, threads, smem, s>>>(p);
    else
        dev::search_kernel_short<64><<<grid, threads, smem, s>>>(p);
    return cudaGetLastError();
}

cudaError_t prepare_search_short(size_t smem) {
    const int sm = static_cast<int>(smem);
    const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
    cudaError_t e = cudaFuncSetAttribute(dev::search_kernel_short<16>, attr, sm);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(dev::search_kernel_short<26>, attr, sm);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(dev::search_kernel_short<32>, attr, sm);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(dev::search_kernel_short<48>, attr, sm);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(dev::search_kernel_short<64>, attr, sm);
    return e;
}

}  // namespace nsfrb
