// The search of arXiv 2510.18136 Sec. 2.2 for windows of 1248 to 4096 samples whose pixels fit in shared
// memory, candidate records only: V = 2, 3 or 4 warps search one DM row together.
//
// The long-window kernel (search_long.cu) reads the cube through L1 and L2, scans every 32 samples and
// evaluates each trial with four shared-memory reads.  Here a pixel's rows lie in shared memory as
// stored (16-bit rows read in place) and each lane of the V warps owns a chunk of C samples with the
// full window's per-lane code: sample pairs, in-lane prefix and halo, lane-strided widths.
//  * Warp v holds the samples [32 C v, 32 C (v + 1)) of the row.  Its prefix q starts at zero there, so a
//    boxcar inside one segment has the rounding of a prefix over at most 1216 samples, and one that ends in
//    another segment is (q' - q) plus the sum of the segments between, added in warp order.
//  * Per row the warps exchange their segments' sums and the first 15 prefix values of each segment (the halo
//    of the last lane before it), and read each other's q for the trials that cross; two
//    barriers of the row's warps.
//  * Each lane tracks its own best (S/N, row, width) over all rows.  At the end of a pixel all
//    warps rebuild the best row from all subbands and find the earliest sample reaching its
//    maximum; the S/N is the tracked one.
//  * One persistent CTA of 12 warps per SM; the next pixel's copy overlaps the search where two pixels
//    fit (16-bit rows, shorter FP32 windows), else it starts when the rows have been read for the last time.
// Bound by instruction issue (FP32 and BF16 rows take the same time).  9696 pixels x 16 subbands, 40 distinct
// DM rows, power-of-two widths, against the long-window kernel: 1250 samples FP32 1.19 ms (7.44), 2048
// 1.54 ms (11.95), BF16 1.53 ms (16.4); V = 3 and 4 evaluate the 2048-sample width from shared
// memory: BF16 3000 samples 5.06 ms (27.7), 4096 7.78 ms (39.1).  Error against 64 bits on
// 193 x 193 pixels of 2048 samples: 9.4e-8 (long-window kernel 9.5e-8).
#pragma once

#include <climits>

#include "nsfrb.h"
#include "nsfrb_internal.h"
#include "plan_internal.h"
#include "search_impl.cuh"

namespace nsfrb {
namespace dev {

constexpr int kWideHalo = 16;   // prefix values a segment hands to the one before it

struct WideLayout {
    size_t buf_bytes;   // a pixel's rows and the samples read past them
    size_t table, xs, pbuf, halo, sums, sinv, best, red, bar, total;
};

__host__ __device__ inline WideLayout wide_layout(const SearchParams &p, int C, int V, int nb) {
    WideLayout L{};
    const size_t es = p.dtype == 0 ? 4 : 2;
    L.buf_bytes = align_up(es * ((size_t)p.n_sub * p.n_t + (size_t)V * 32 * C + 16), 128);
    size_t o = 0;
    L.table = o;
    o += align_up(sizeof(int32_t) * ((size_t)p.n_u * kInfo + p.n_deltas + (size_t)p.n_u * p.n_sub), 128);
    L.xs = o;
    o += L.buf_bytes * nb;
    L.pbuf = o;   // [kWarps][32 C]; at the end of a pixel its best row's prefix
    o += sizeof(float) * (size_t)kWarps * 32 * C;
    L.halo = o;   // [kWarps + 1][16]: the row after the last stays zero
    o += sizeof(float) * (kWarps + 1) * kWideHalo;
    L.sums = o;   // [kWarps] segment sums; at the end of a pixel the warps' sums
    o += sizeof(float) * 16;
    L.sinv = o;
    o += sizeof(float) * kMaxW;
    L.best = o;   // [kWarps] S/N, row * kMaxW + width index
    o += (sizeof(float) + sizeof(int32_t)) * kWarps;
    L.red = o;    // [kWarps] maximum, earliest sample
    o += (sizeof(float) + sizeof(int32_t)) * kWarps;
    L.bar = align_up(o, 8);
    L.total = L.bar + 16;
    return L;
}

template <int THREADS>
__device__ __forceinline__ void team_sync(int team) {
    asm volatile("bar.sync %0, %1;" ::"r"(team + 1), "n"(THREADS) : "memory");
}

template <int C, int V, int ST>
__global__ void __launch_bounds__(kThreads, 1) search_kernel_wide(const __grid_constant__ SearchParams p) {
    static_assert(C % 4 == 2 && C >= kSmallMax && kWarps % V == 0, "chunk of sample pairs; whole teams");
    extern __shared__ __align__(128) unsigned char smem[];
    constexpr int SH = kSmallMax, kEs = (ST == 0) ? 4 : 2, G = kWarps / V, kSeg = 32 * C;
    const int nb = p.nb;
    const WideLayout lay = wide_layout(p, C, V, nb);
    int32_t *s_table = reinterpret_cast<int32_t *>(smem + lay.table);
    float *s_p = reinterpret_cast<float *>(smem + lay.pbuf);
    float *s_halo = reinterpret_cast<float *>(smem + lay.halo);
    float *s_sums = reinterpret_cast<float *>(smem + lay.sums);
    float *s_inv = reinterpret_cast<float *>(smem + lay.sinv);
    float *s_bs = reinterpret_cast<float *>(smem + lay.best);
    int32_t *s_buw = reinterpret_cast<int32_t *>(s_bs + kWarps);
    float *s_rm = reinterpret_cast<float *>(smem + lay.red);
    int32_t *s_rt = reinterpret_cast<int32_t *>(s_rm + kWarps);
    unsigned long long *s_bar = reinterpret_cast<unsigned long long *>(smem + lay.bar);

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int team = warp / V, v = warp % V;
    const int n_sub = p.n_sub, n_t = p.n_t, ne = n_sub * n_t;
    const int table_words = p.n_u * kInfo + p.n_deltas + p.n_u * n_sub;
    for (int i = tid; i < table_words; i += kThreads) s_table[i] = p.table[i];
    const int32_t *s_info = s_table;
    const int32_t *s_delta = s_table + p.n_u * kInfo;
    const int32_t *s_shift = s_delta + p.n_deltas;
    if (tid < kWideHalo) s_halo[kWarps * kWideHalo + tid] = 0.0f;
    if (tid == 0) {
        mbar_init(&s_bar[0], 1);
        mbar_init(&s_bar[1], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_proxy_async();
    }
    __syncthreads();
    int64_t n_items = p.n_items;
    if (p.n_items_dev) n_items = *p.n_items_dev;
    auto item_pixel = [&](int64_t it) -> int64_t {
        return p.pix_list ? static_cast<int64_t>(p.pix_list[it]) : p.pix0 + it;
    };
    const uint32_t bytes = static_cast<uint32_t>(ne * kEs);
    auto issue = [&](int64_t it, int b) {   // one thread
        const unsigned char *src =
            static_cast<const unsigned char *>(p.cube) + (item_pixel(it) - p.cube_pix0) * static_cast<int64_t>(bytes);
        mbar_expect_tx(&s_bar[b], bytes);
        bulk_g2s(smem + lay.xs + b * lay.buf_bytes, src, bytes, &s_bar[b]);
    };
    if (tid == 0 && blockIdx.x < n_items) issue(blockIdx.x, 0);

    const int n_ua = p.n_u_active;
    const int n_grp = min(G, n_ua);
    const int u_lo = team < n_grp ? (team * n_ua) / n_grp : 0, u_hi = team < n_grp ? ((team + 1) * n_ua) / n_grp : 0;
    float *Pt = s_p + (size_t)team * V * kSeg;   // the team's q, segment after segment
    float *Pw = Pt + v * kSeg;
    float *halo_out = s_halo + warp * kWideHalo;
    // the segment after this one; the last one's last chunk ends past the window (its total is -inf or NaN)
    const float *halo_in = s_halo + (v + 1 < V ? warp + 1 : kWarps) * kWideHalo;
    float *sums = s_sums + team * V;
    const int t0 = (v * 32 + lane) * C;

    int i = 0;
    for (int64_t it = blockIdx.x; it < n_items; it += gridDim.x, ++i) {
        const int64_t pix = item_pixel(it), nxt = it + gridDim.x;
        const int b = nb == 2 ? (i & 1) : 0;
        const unsigned char *xs = smem + lay.xs + b * lay.buf_bytes;
        // the other buffer was read for the last time before the barriers of the previous pixel's end
        if (nb == 2 && tid == 0 && nxt < n_items) issue(nxt, b ^ 1);
        if (tid < p.n_w) {
            const float sg = p.sigma ? p.sigma[pix] : p.sigma_default;
            s_inv[tid] = 1.0f / (sg * sqrtf(static_cast<float>(p.widths[tid])));
        }
        const int landed = mbar_wait(&s_bar[b], static_cast<uint32_t>(nb == 2 ? i >> 1 : i) & 1u);
        if (!__syncthreads_and(landed)) {
            if (tid == 0) {
                atomicOr(p.err, ERR_WAIT_TIMEOUT);
                // the copy ahead is waited for (bounded) before the CTA leaves
                if (nb == 2 && nxt < n_items) mbar_wait(&s_bar[b ^ 1], static_cast<uint32_t>((i + 1) >> 1) & 1u);
            }
            return;
        }

        // ---- the team's rows
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
                for (int k = 0; k < n_sub; ++k) acc_row<C, false, ST>(D, xs, 0, 0, k * n_t + t0 + sh[k]);
            } else {
                const int d0 = info[UI_DOFF], nd = info[UI_ND];
#pragma unroll 1
                for (int e = d0; e < d0 + nd; ++e) {
                    const uint32_t pk = static_cast<uint32_t>(s_delta[e]);
                    const int k = pk & 63u, so = (pk >> 6) & 0x1fffu, sn = pk >> 19;
                    const int at = k * n_t + t0 + so;
                    if (sn == so + 1) {
                        if constexpr (ST == 0)
                            acc_step1<C>(D, reinterpret_cast<const float *>(xs) + at, at & 1);
                        else
                            acc_step1_16<C, ST>(D, reinterpret_cast<const uint16_t *>(xs), at);
                    } else {
                        acc_row<C, false, ST>(D, xs, 0, 0, at - so + sn);
                        acc_row<C, true, ST>(D, xs, 0, 0, at);
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
            const int uw = u * kMaxW;
            auto consider = [&](int wi, float m) {
                const float s = m * s_inv[wi];
                if (s > bs) {   // ascending widths: ties keep the smallest index
                    bs = s;
                    buw = uw + wi;
                }
            };
            {
                float2 Lp[C / 2], Hh[SH / 2];
                const float tot = prefix_pairs<C>(D, Lp);
                const float carry = lane_carry(tot, lane);
                if (lane == 31) sums[v] = carry + tot;
                if (lane == 0) {
                    float2 *h2 = reinterpret_cast<float2 *>(halo_out);
#pragma unroll
                    for (int m = 0; m < kWideHalo / 2; ++m) h2[m] = Lp[m];
                }
                store_p<C>(Pw, lane * C, carry, Lp);
                team_sync<32 * V>(team);
                halo_pairs<C, SH>(Lp, tot, Hh);
                if (lane == 31) {
                    const float2 *h2 = reinterpret_cast<const float2 *>(halo_in);
                    const float2 tt = make_float2(tot, tot);
#pragma unroll
                    for (int m = 0; m < SH / 2; ++m) Hh[m] = add2(tt, h2[m]);   // h[0] = 0
                }
#define NSFRB_WIDE_SMALL(J) \
    if (p.pow2_wi[J] >= 0) consider(p.pow2_wi[J], small_max_pk<C, SH, (1 << J)>(D, Lp, Hh));
                NSFRB_WIDE_SMALL(0) NSFRB_WIDE_SMALL(1) NSFRB_WIDE_SMALL(2) NSFRB_WIDE_SMALL(3) NSFRB_WIDE_SMALL(4)
#undef NSFRB_WIDE_SMALL
            }
            // sums of the segments from this one on: s1 to the next segment's start, s2 to the one after
            const float s1 = sums[v], s2 = v + 1 < V ? s1 + sums[v + 1] : 0.0f;
            if (p.has_large) {
                float2 Ps[C / 2];
                load_ps<C>(Pw, lane, Ps);
#define NSFRB_WIDE_LARGE(J)                                                                        \
    if constexpr ((1 << J) > SH && ((1 << J) >> 5) < 2 * C) {                                      \
        if (p.pow2_wi[J] >= 0) {                                                                   \
            constexpr int M = (1 << J) >> 5;                                                       \
            float m = neg_inf();                                                                   \
            if constexpr (M < C) m = large_max_pk<C, M>(Ps);                                       \
            if (v + 1 < V) {                                                                       \
                float a[2] = {neg_inf(), neg_inf()};                                               \
                _Pragma("unroll") for (int r = (M > C ? M - C : 0); r < (M < C ? M : C); ++r)      \
                    a[r & 1] = fmaxf(a[r & 1], (Pw[kSeg + 32 * r + lane] - pget(Ps, r + C - M)) + s1); \
                m = fmax3(m, a[0], a[1]);                                                          \
            }                                                                                      \
            if constexpr (M > C) {                                                                 \
                if (v + 2 < V) {                                                                   \
                    _Pragma("unroll") for (int r = 0; r < M - C; ++r)                              \
                        m = fmaxf(m, (Pw[2 * kSeg + 32 * r + lane] - pget(Ps, r + 2 * C - M)) + s2); \
                }                                                                                  \
            }                                                                                      \
            consider(p.pow2_wi[J], m);                                                             \
        }                                                                                          \
    }
                NSFRB_POW2(NSFRB_WIDE_LARGE)
#undef NSFRB_WIDE_LARGE
            }
#pragma unroll 1
            for (int g = 0; g < p.n_gen; ++g) {
                const int wi = p.gen_wi[g], w = p.widths[wi];
                float m = neg_inf();
                // this warp's trials: those that start in its segment
                for (int t = v * kSeg + lane; t < (v + 1) * kSeg && t + w <= L; t += 32) {
                    const int e = t + w, se = min(e / kSeg, V - 1);
                    float add = 0.0f;
                    for (int q = v; q < se; ++q) add += sums[q];
                    m = fmaxf(m, (Pt[e] - Pt[t]) + add);
                }
                const float s = m * s_inv[wi];
                if (s > bs || (s == bs && uw + wi < buw)) {
                    bs = s;
                    buw = uw + wi;
                }
            }
            team_sync<32 * V>(team);   // the row's q, halos and sums have been read
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float os = __shfl_xor_sync(kFull, bs, o);
            const int ob = __shfl_xor_sync(kFull, buw, o);
            if (os > bs || (os == bs && ob >= 0 && ob < buw)) {
                bs = os;
                buw = ob;
            }
        }
        if (lane == 0) {
            s_bs[warp] = bs;
            s_buw[warp] = buw;
        }
        __syncthreads();

        // ---- the pixel's record: ties go to the smallest row, then width
        bs = neg_inf();
        buw = -1;
        for (int g = 0; g < kWarps; ++g) {
            const float os = s_bs[g];
            const int ob = s_buw[g];
            if (os > bs || (os == bs && ob >= 0 && ob < buw)) {
                bs = os;
                buw = ob;
            }
        }
        const bool any = buw >= 0;
        const int u = any ? buw / kMaxW : 0, wi = any ? buw % kMaxW : 0, w = p.widths[wi];
        const int L = any ? n_t - s_info[u * kInfo + UI_SMAX] : 0;
        constexpr int CC = ((32 * C * V + kThreads - 1) / kThreads) | 1;   // samples per thread, odd
        const int t1 = tid * CC;
        float d[CC];
#pragma unroll
        for (int c = 0; c < CC; ++c) d[c] = 0.0f;
        if (t1 < L) {
            const int32_t *sh = s_shift + u * n_sub;
#pragma unroll 2
            for (int k = 0; k < n_sub; ++k) {
                const int e = k * n_t + t1 + sh[k];
#pragma unroll
                for (int c = 0; c < CC; ++c) {
                    if constexpr (ST == 0)
                        d[c] += reinterpret_cast<const float *>(xs)[e + c];
                    else
                        d[c] += widen16(reinterpret_cast<const uint16_t *>(xs)[e + c], ST);
                }
            }
        }
        float tot = 0.0f;
#pragma unroll
        for (int c = 0; c < CC; ++c) {
            const float x = t1 + c < L ? d[c] : 0.0f;
            if (w > 1) d[c] = tot;   // prefix; w = 1 keeps the samples
            tot += x;
        }
        float carry = lane_carry(tot, lane);
        if (lane == 31) s_sums[warp] = carry + tot;
        fence_proxy_async();
        __syncthreads();   // the rows have been read for the last time
        if (nb == 1 && tid == 0 && nxt < n_items) issue(nxt, 0);
        for (int g = 0; g < warp; ++g) carry += s_sums[g];
#pragma unroll
        for (int c = 0; c < CC; ++c) {
            if (w > 1) d[c] += carry;
            if (t1 + c <= L) s_p[t1 + c] = d[c];
        }
        __syncthreads();
        float m = neg_inf();
#pragma unroll
        for (int c = 0; c < CC; ++c) {
            if (any && t1 + c + w <= L) {
                if (w > 1) d[c] = s_p[t1 + c + w] - d[c];
                m = fmaxf(m, d[c]);
            }
        }
        m = warp_max(m);
        int at = INT_MAX;
#pragma unroll
        for (int c = CC - 1; c >= 0; --c)
            if (any && t1 + c + w <= L && d[c] == m) at = t1 + c;
        at = warp_min(at);
        if (lane == 0) {
            s_rm[warp] = m;
            s_rt[warp] = at;
        }
        __syncthreads();
        if (tid == 0) {
            PixRec r{neg_inf(), -1, -1, -1};
            if (any) {
                float best = neg_inf();
                int t = INT_MAX;
                for (int g = 0; g < kWarps; ++g)   // ascending samples: the earliest on ties
                    if (s_rm[g] > best) {
                        best = s_rm[g];
                        t = s_rt[g];
                    }
                r = PixRec{bs, s_info[u * kInfo + UI_FIRST_D], wi, t == INT_MAX ? -1 : t};
            }
            if (p.bad_pix && p.bad_pix[pix]) {
                r = PixRec{neg_inf(), -1, -1, -1};
                atomicOr(p.err, ERR_ZERO_MAD);
            }
            p.rec[pix] = r;
        }
    }
}

template <int C, int V, int ST>
cudaError_t wide_launch(const SearchParams &p, int grid, size_t smem, cudaStream_t s) {
    const cudaError_t e = raise_smem_limit(reinterpret_cast<const void *>(search_kernel_wide<C, V, ST>));
    if (e != cudaSuccess) return e;
    search_kernel_wide<C, V, ST><<<grid, kThreads, smem, s>>>(p);
    return cudaGetLastError();
}

}  // namespace dev

// (C, V) with compiled kernels, the windows they hold ascending: 1407, 1663, 2175, 2431, 3263, 4351 samples.
#define NSFRB_WIDE_TILES(X) X(22, 2) X(26, 2) X(34, 2) X(38, 2) X(34, 3) X(34, 4)

#define NSFRB_INSTANTIATE_WIDE(ST)                                                                      \
    cudaError_t launch_search_wide_s##ST(const SearchParams &p, int grid, size_t smem, cudaStream_t s) { \
        switch (10 * p.mid_c + p.mid_s) {                                                               \
            NSFRB_WIDE_TILES(NSFRB_WIDE_CASE_##ST)                                                      \
            default:                                                                                    \
                return cudaErrorInvalidValue;                                                           \
        }                                                                                               \
    }
#define NSFRB_WIDE_CASE_0(C, V) case 10 * C + V: return dev::wide_launch<C, V, 0>(p, grid, smem, s);
#define NSFRB_WIDE_CASE_1(C, V) case 10 * C + V: return dev::wide_launch<C, V, 1>(p, grid, smem, s);
#define NSFRB_WIDE_CASE_2(C, V) case 10 * C + V: return dev::wide_launch<C, V, 2>(p, grid, smem, s);

}  // namespace nsfrb
