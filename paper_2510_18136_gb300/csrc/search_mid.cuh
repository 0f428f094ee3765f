// The search of arXiv 2510.18136 Sec. 2.2 for windows of 65 to 607 samples, candidate records only
// (the 5-fold binned window of 240 samples, the 256-sample cubes of the classifier's data).
//
// A warp per DM row of such a window leaves a lane 3 to 19 samples, and the row costs what its
// dependent chain costs (warp scan, shared-memory round trip, warp maxima), whatever its length.
// Here a warp searches the same DM row of 32 / S pixels at once, S lanes to a pixel, and a lane owns a
// chunk of C samples as long as the full window's kernel gives it: sample pairs, widths up to 16 by doubling
// in registers (small_sums: the kernels before had chunks of 3 to 17 samples, and an in-lane prefix over 22
// to 38 would put a bright or invalid sample into more of them), P to shared memory, lane-strided
// widths from there.
//  * A CTA takes 32 / S consecutive pixels, its warps contiguous groups of the distinct DM rows.  A
//    pixel's rows lie packed in shared memory as stored (16-bit rows read in place), one
//    bulk copy per pixel.  The pixel pitch is C S modulo 32 words: the lanes' chunks then go on from
//    pixel to pixel in steps of C words modulo 32 (C = 2 modulo 4), and the 64-bit reads of 16
//    lanes hit 32 banks.
//  * De-dispersed samples past the valid range are set to -inf when it changes; ranges shrink as
//    the DM grows, so they stay out, and trials that read them are -inf or NaN and drop out.
//  * Lane-strided widths read P in pairs, lane j of a pixel the pairs (2 S m + 2 j, + 1), so that
//    P[t + w] is a register of the same lane for every power of two w >= 2 S.
//  * Each lane tracks its own best (S/N, row, width) over all rows: no warp maxima per row.  At the end
//    a warp per pixel rebuilds the best row from all subbands, and takes the record's S/N and the
//    earliest sample reaching it from that row: widths up to 16 by doubling, others from a prefix
//    kept as a value and its rounding error (over chunks of 3 to 19 samples a plain one is off by up to three times
//    what the kernels before it were beside bright features), the quotient corrected once.
// Bound by instruction issue and, for few rows, by the copies (two or three CTAs fit on an SM, so
// copy and search overlap only between them).  C and S are the smallest of the compiled windows S C
// that hold the samples; the rows are split over as many warps as keep the SM's register file full.
// 301 x 301 pixels x 16 subbands, 40 distinct DM rows, power-of-two widths, against the kernels
// with a warp per row: FP32 100 samples 539 us (2873), 240 1324 us (2947), 400 2270 us (3261), 600
// 3059 us (4409); BF16 240 1127 us (4887), 300 1630 us (9300), 600 2638 us (7077).  With plain prefixes
// for every width: 521, 1295, 2178, 3001; 1098, 1540, 2561 us.
#pragma once

#include <algorithm>
#include <climits>

#include "nsfrb.h"
#include "nsfrb_internal.h"
#include "plan_internal.h"
#include "search_impl.cuh"

namespace nsfrb {
namespace dev {

struct MidLayout {
    int pitch;   // elements from pixel to pixel
    size_t table, xs, pbuf, sinv, best, bar, total;
};

__host__ __device__ inline MidLayout mid_layout(const SearchParams &p, int C, int S, int n_warps) {
    MidLayout L{};
    const int es = p.dtype == 0 ? 4 : 2, mod = p.dtype == 0 ? 32 : 64;
    const int pw = 32 / S, ne = p.n_sub * p.n_t;
    L.pitch = ne + ((C * S - ne) % mod + mod) % mod;
    size_t o = 0;
    L.table = o;
    o += align_up(sizeof(int32_t) * ((size_t)p.n_u * kInfo + p.n_deltas + (size_t)p.n_u * p.n_sub), 16);
    L.xs = o;
    // chunks past the end of the last pixel's last row are read (and masked): S C + 16 elements more
    o += align_up((size_t)es * ((size_t)pw * L.pitch + S * C + 16), 128);
    L.pbuf = o;
    o += sizeof(float) * (size_t)n_warps * 32 * C;
    L.sinv = o;
    o += sizeof(float) * (size_t)p.n_w * pw;
    L.best = o;
    o += (sizeof(float) + sizeof(int32_t)) * (size_t)n_warps * pw;
    L.bar = align_up(o, 8);
    L.total = L.bar + 16;
    return L;
}

// D += / -= the row at element e of the pixel (any parity); D += x(t + 1) - x(t).
template <int C, bool SUB, int ST>
__device__ __forceinline__ void mid_acc(float2 (&D)[C / 2], const void *xs, int e) {
    acc_row<C, SUB, ST>(D, xs, 0, 0, e);
}
template <int C, int ST>
__device__ __forceinline__ void mid_step1(float2 (&D)[C / 2], const void *xs, int e) {
    if constexpr (ST == 0)
        acc_step1<C>(D, static_cast<const float *>(xs) + e, e & 1);
    else
        acc_step1_16<C, ST>(D, static_cast<const uint16_t *>(xs), e);
}

// Width w = 2 S M from the lane-strided pairs of P.
template <int C, int M>
__device__ __forceinline__ float mid_large(const float2 (&Ps)[C / 2]) {
    float acc[3] = {neg_inf(), neg_inf(), neg_inf()};
#pragma unroll
    for (int m = 0; m < C / 2 - M; ++m) {
        const float2 b = sub2(Ps[m + M], Ps[m]);
        acc[m % 3] = fmax3(acc[m % 3], b.x, b.y);
    }
    return fmax3(acc[0], acc[1], acc[2]);
}

template <int C, int S, int ST>
__global__ void __launch_bounds__(C > 26 ? 192 : 256, 2) search_kernel_mid(const __grid_constant__ SearchParams p) {
    static_assert(C % 4 == 2 && C >= kSmallMax, "pairs without bank conflicts; the halo is one chunk at most");
    extern __shared__ __align__(128) unsigned char smem[];
    constexpr int PW = 32 / S, kEs = (ST == 0) ? 4 : 2;
    const int n_warps = blockDim.x >> 5;
    const MidLayout lay = mid_layout(p, C, S, n_warps);
    int32_t *s_table = reinterpret_cast<int32_t *>(smem + lay.table);
    unsigned char *s_xs = smem + lay.xs;
    float *s_inv = reinterpret_cast<float *>(smem + lay.sinv);              // [n_w][PW]
    float *s_bs = reinterpret_cast<float *>(smem + lay.best);               // [n_warps][PW]
    int32_t *s_buw = reinterpret_cast<int32_t *>(s_bs + (size_t)n_warps * PW);   // row * kMaxW + width index
    unsigned long long *s_bar = reinterpret_cast<unsigned long long *>(smem + lay.bar);

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int q = lane / S, j = lane % S;   // pixel of the warp's set, chunk of the pixel
    const int n_sub = p.n_sub, n_t = p.n_t, ne = n_sub * n_t;
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
    if (p.stage == 1 && tid == 0) {
        mbar_init(s_bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_proxy_async();
    }
    const int top = small_top<26>(p);   // (32 samples are lane-strided here, whatever the chunk)
    uint32_t phase = 0;
    // one set of pixels per CTA, or, where a device count says how many there are (re-scoring), several
    for (int64_t it0 = static_cast<int64_t>(blockIdx.x) * PW; it0 < n_items;
         it0 += static_cast<int64_t>(gridDim.x) * PW) {
        const int n_here = static_cast<int>(min(static_cast<int64_t>(PW), n_items - it0));
        const unsigned char *cube = static_cast<const unsigned char *>(p.cube);

        // ---- samples as stored, 1 / (sigma sqrt(w))
        if (p.stage == 1) {
            if (tid == 0) {
                const uint32_t bytes = static_cast<uint32_t>(ne * kEs);
                mbar_expect_tx(s_bar, bytes * static_cast<uint32_t>(n_here));
                for (int i = 0; i < n_here; ++i)
                    bulk_g2s(s_xs + (size_t)i * lay.pitch * kEs,
                             cube + (item_pixel(it0 + i) - p.cube_pix0) * static_cast<int64_t>(bytes), bytes, s_bar);
            }
        } else {
            for (int i = 0; i < n_here; ++i) {
                const int64_t from = (item_pixel(it0 + i) - p.cube_pix0) * ne;
                for (int e = tid; e < ne; e += blockDim.x) {
                    const size_t at = (size_t)i * lay.pitch + e;
                    if constexpr (ST == 0)
                        reinterpret_cast<float *>(s_xs)[at] = reinterpret_cast<const float *>(cube)[from + e];
                    else
                        reinterpret_cast<uint16_t *>(s_xs)[at] = reinterpret_cast<const uint16_t *>(cube)[from + e];
                }
            }
        }
        for (int i = tid; i < p.n_w * PW; i += blockDim.x) {
            const float sg = (p.sigma && i % PW < n_here) ? p.sigma[item_pixel(it0 + i % PW)] : p.sigma_default;
            s_inv[i] = 1.0f / (sg * sqrtf(static_cast<float>(p.widths[i / PW])));
        }
        __syncthreads();
        const int landed = p.stage == 1 ? mbar_wait(s_bar, phase) : 1;
        phase ^= 1u;
        if (!__syncthreads_and(landed)) {
            if (tid == 0) {
                atomicOr(p.err, ERR_WAIT_TIMEOUT);
                mbar_wait(s_bar, phase ^ 1u);   // the copies in flight, bounded, before the CTA leaves
            }
            return;
        }

        // ---- the warp's rows
        const int n_ua = p.n_u_active;
        float *Pw = reinterpret_cast<float *>(smem + lay.pbuf) + (size_t)warp * 32 * C;
        const void *xp = s_xs + (size_t)(q < n_here ? q : 0) * lay.pitch * kEs;
        const int t0 = j * C;
        const int u_lo = (warp * n_ua) / n_warps, u_hi = ((warp + 1) * n_ua) / n_warps;
        float bs = neg_inf();
        int buw = -1;
        float2 D[C / 2];
        int L_prev = -1;
#pragma unroll 1
        for (int u = u_lo; u < u_hi; ++u) {
            const int32_t *info = s_info + u * kInfo;
            if (u == u_lo) {
#pragma unroll
                for (int m = 0; m < C / 2; ++m) D[m] = make_float2(0.0f, 0.0f);
                const int32_t *sh = s_shift + u * n_sub;
#pragma unroll 1
                for (int k = 0; k < n_sub; ++k) mid_acc<C, false, ST>(D, xp, k * n_t + t0 + sh[k]);
            } else {
                const int d0 = info[UI_DOFF], nd = info[UI_ND];
#pragma unroll 1
                for (int e = d0; e < d0 + nd; ++e) {
                    const uint32_t pk = static_cast<uint32_t>(s_delta[e]);
                    const int k = pk & 63u, so = (pk >> 6) & 0x1fffu, sn = pk >> 19;
                    const int at = k * n_t + t0;
                    if (sn == so + 1) {
                        mid_step1<C, ST>(D, xp, at + so);
                    } else {
                        mid_acc<C, false, ST>(D, xp, at + sn);
                        mid_acc<C, true, ST>(D, xp, at + so);
                    }
                }
            }
            const int L = n_t - info[UI_SMAX];
            if (L != L_prev) {
#pragma unroll
                for (int m = 0; m < C / 2; ++m) {
                    if (t0 + 2 * m >= L) D[m].x = neg_inf();
                    if (t0 + 2 * m + 1 >= L) D[m].y = neg_inf();
                }
                L_prev = L;
            }
            // ascending widths with a strict '>' keep the smallest index on ties
            const int uw = u * kMaxW;
            auto consider = [&](int wi, float m) {
                const float s = m * s_inv[wi * PW + q];
                if (s > bs) {
                    bs = s;
                    buw = uw + wi;
                }
            };
            {
                float2 Hd[kSmallMax / 2];
                halo_samples<C>(D, Hd);   // a pixel's last lane takes the next pixel's: see there
                small_sums<C>(D, Hd, top, [&](int b, float m) {
                    if (p.pow2_wi[b] >= 0) consider(p.pow2_wi[b], m);
                });
            }
            {
                float2 Lp[C / 2];
                const float tot = prefix_pairs<C>(D, Lp);
                float inc = tot;
#pragma unroll
                for (int o = 1; o < S; o <<= 1) {
                    const float y = __shfl_up_sync(kFull, inc, o, S);
                    if (j >= o) inc += y;
                }
                float carry = __shfl_up_sync(kFull, inc, 1, S);
                if (j == 0) carry = 0.0f;
                store_p<C>(Pw, lane * C, carry, Lp);
            }
            __syncwarp();
            if (p.has_large) {
                float2 Ps[C / 2];
                const float2 *src2 = reinterpret_cast<const float2 *>(Pw + q * S * C) + j;
#pragma unroll
                for (int m = 0; m < C / 2; ++m) Ps[m] = src2[S * m];
#define NSFRB_MID_LARGE(J)                                                                     \
    if constexpr ((1 << J) > kSmallMax && (1 << J) < S * C) {                                         \
        if (p.pow2_wi[J] >= 0) consider(p.pow2_wi[J], mid_large<C, (1 << J) / (2 * S)>(Ps));  \
    }
                NSFRB_POW2(NSFRB_MID_LARGE)
#undef NSFRB_MID_LARGE
            }
#pragma unroll 1
            for (int g = 0; g < p.n_gen; ++g) {
                const int wi = p.gen_wi[g], w = p.widths[wi];
                const float *Pq = Pw + q * S * C;
                float m = neg_inf();
                for (int t = j; t + w <= L; t += S) m = fmaxf(m, Pq[t + w] - Pq[t]);
                const float s = m * s_inv[wi * PW + q];
                if (s > bs || (s == bs && uw + wi < buw)) {
                    bs = s;
                    buw = uw + wi;
                }
            }
            __syncwarp();
        }
        // the pixel's best over its lanes: ties go to the smallest row, then width
#pragma unroll
        for (int o = S / 2; o > 0; o >>= 1) {
            const float os = __shfl_xor_sync(kFull, bs, o);
            const int ob = __shfl_xor_sync(kFull, buw, o);
            if (os > bs || (os == bs && ob >= 0 && ob < buw)) {
                bs = os;
                buw = ob;
            }
        }
        if (j == 0) {
            s_bs[warp * PW + q] = bs;
            s_buw[warp * PW + q] = buw;
        }
        __syncthreads();

        // ---- records: a warp per pixel rebuilds its best row
        for (int i = warp; i < n_here; i += n_warps) {
            float best = neg_inf();
            int uw = -1;
            for (int g = 0; g < n_warps; ++g)
                if (s_bs[g * PW + i] > best) {
                    best = s_bs[g * PW + i];
                    uw = s_buw[g * PW + i];
                }
            PixRec r{neg_inf(), -1, -1, -1};
            if (uw >= 0) {
                const int u = uw / kMaxW, wi = uw % kMaxW, w = p.widths[wi];
                const int32_t *sh = s_shift + u * n_sub;
                const int L = n_t - s_info[u * kInfo + UI_SMAX];
                const unsigned char *row = s_xs + (size_t)i * lay.pitch * kEs;
                const float inv = s_inv[wi * PW + i];
                // lane l takes samples [l CC, l CC + CC), CC odd: no bank conflicts
                constexpr int CC = ((S * C + 31) / 32) | 1;
                const int t1 = lane * CC;
                float d[CC];
#pragma unroll
                for (int c = 0; c < CC; ++c) d[c] = 0.0f;
                if (t1 < L) {
#pragma unroll 2
                    for (int k = 0; k < n_sub; ++k) {
                        const int e = k * n_t + t1 + sh[k];
#pragma unroll
                        for (int c = 0; c < CC; ++c) {
                            if constexpr (ST == 0)
                                d[c] += reinterpret_cast<const float *>(row)[e + c];
                            else
                                d[c] += widen16(reinterpret_cast<const uint16_t *>(row)[e + c], ST);
                        }
                    }
                }
                // widths of the in-lane path: the samples in the buffer, boxcars by doubling as in small_sums;
                // others: P as a value and its rounding error in the buffer (each S C words of the 32 C), P[t1 + c]
                // kept in d[c], dl[c].  The error is left out where it is not a number (an infinite sample).
                static_assert(2 * S <= 32, "value and error of the prefix");
                float *Pl = Pw + S * C, dl[CC];
                const bool small = w <= kSmallMax && (w & (w - 1)) == 0;
                __syncwarp();
                if (small) {
#pragma unroll
                    for (int c = 0; c < CC; ++c)
                        if (t1 + c < L) Pw[t1 + c] = d[c];
                } else {
                    float tot = 0.0f, tot_l = 0.0f;
#pragma unroll
                    for (int c = 0; c < CC; ++c) {
                        const float v = t1 + c < L ? d[c] : 0.0f;
                        d[c] = tot;
                        dl[c] = tot_l;
                        pair_add(tot, tot_l, v, 0.0f);
                    }
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const float yh = __shfl_up_sync(kFull, tot, o), yl = __shfl_up_sync(kFull, tot_l, o);
                        if (lane >= o) pair_add(tot, tot_l, yh, yl);
                    }
                    float ch = __shfl_up_sync(kFull, tot, 1), cl = __shfl_up_sync(kFull, tot_l, 1);
                    if (lane == 0) ch = cl = 0.0f;
#pragma unroll
                    for (int c = 0; c < CC; ++c) {
                        pair_add(d[c], dl[c], ch, cl);
                        if (t1 + c <= L) {
                            Pw[t1 + c] = d[c];
                            Pl[t1 + c] = dl[c];
                        }
                    }
                }
                __syncwarp();
                if (small) {
                    constexpr int N = CC + kSmallMax - 1;
                    float x[N];
#pragma unroll
                    for (int c = 0; c < N; ++c) x[c] = c < CC ? d[c] : (c < CC + w - 1 && t1 + c < L) ? Pw[t1 + c] : 0.0f;
#pragma unroll
                    for (int h = 1; h < kSmallMax; h *= 2) {
                        if (w <= h) break;
#pragma unroll
                        for (int c = 0; c + h < N; ++c) x[c] += x[c + h];
                    }
#pragma unroll
                    for (int c = 0; c < CC; ++c) d[c] = x[c];
                }
                float m = neg_inf();
#pragma unroll
                for (int c = 0; c < CC; ++c) {
                    if (t1 + c + w <= L) {
                        if (!small) {
                            const float b = Pw[t1 + c + w] - d[c], e = Pl[t1 + c + w] - dl[c];
                            d[c] = e == e ? b + e : b;
                        }
                        m = fmaxf(m, d[c]);
                    }
                }
                m = warp_max(m);
                int at = INT_MAX;
#pragma unroll
                for (int c = CC - 1; c >= 0; --c)
                    if (t1 + c + w <= L && d[c] * inv == m * inv) at = t1 + c;
                at = warp_min(at);
                r.snr = record_snr(m, p.sigma ? p.sigma[item_pixel(it0 + i)] : p.sigma_default, w, inv);
                r.t_idx = at == INT_MAX ? -1 : at;
                r.dm_idx = s_info[u * kInfo + UI_FIRST_D];
                r.w_idx = wi;
                __syncwarp();
            }
            if (lane == 0) {
                const int64_t pix = item_pixel(it0 + i);
                if (p.bad_pix && p.bad_pix[pix]) {
                    r = PixRec{neg_inf(), -1, -1, -1};
                    atomicOr(p.err, ERR_ZERO_MAD);
                }
                p.rec[pix] = r;
            }
        }
        fence_proxy_async();
        __syncthreads();   // everything of this set has been read
    }
}

template <int C, int S, int ST>
cudaError_t mid_launch(const SearchParams &p, int grid_sm, size_t smem, cudaStream_t s) {
    // where only the device knows the count, as many CTAs as can run at once (at most) loop over it
    const int64_t sets = (p.n_items + 32 / S - 1) / (32 / S);
    const unsigned grid = static_cast<unsigned>(p.n_items_dev ? std::min<int64_t>(sets, 2 * grid_sm) : sets);
    const cudaError_t e = raise_smem_limit(reinterpret_cast<const void *>(search_kernel_mid<C, S, ST>));
    if (e != cudaSuccess) return e;
    search_kernel_mid<C, S, ST><<<grid, 32 * p.mid_w, smem, s>>>(p);
    return cudaGetLastError();
}

}  // namespace dev

// (C, S) with compiled kernels, the windows they hold ascending.
#define NSFRB_MID_TILES(X) X(22, 4) X(26, 4) X(34, 4) X(22, 8) X(26, 8) X(34, 8) X(22, 16) X(26, 16) X(34, 16) X(38, 16)

#define NSFRB_INSTANTIATE_MID(ST)                                                                     \
    cudaError_t launch_search_mid_s##ST(const SearchParams &p, int grid_sm, size_t smem, cudaStream_t s) { \
        switch (100 * p.mid_c + p.mid_s) {                                                            \
            NSFRB_MID_TILES(NSFRB_MID_CASE_##ST)                                                      \
            default:                                                                                  \
                return cudaErrorInvalidValue;                                                         \
        }                                                                                             \
    }
#define NSFRB_MID_CASE_0(C, S) case 100 * C + S: return dev::mid_launch<C, S, 0>(p, grid_sm, smem, s);
#define NSFRB_MID_CASE_1(C, S) case 100 * C + S: return dev::mid_launch<C, S, 1>(p, grid_sm, smem, s);
#define NSFRB_MID_CASE_2(C, S) case 100 * C + S: return dev::mid_launch<C, S, 2>(p, grid_sm, smem, s);

}  // namespace nsfrb
