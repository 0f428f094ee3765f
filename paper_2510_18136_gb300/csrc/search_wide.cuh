// The search of arXiv 2510.18136 Sec. 2.2 for windows of 1248 to 4096 samples whose pixels fit in shared
// memory, candidate records only: V = 2, 3 or 4 warps search one DM row together.
//
// The long-window kernel (search_long.cu) reads the cube through L1 and L2, scans every 32 samples and
// evaluates each trial with four shared-memory reads.  Here a pixel's rows lie in shared memory as
// stored (16-bit rows read in place) and each lane of the V warps owns a chunk of C samples in registers.
//  * No boxcar is the difference of two long prefixes (over thousands of samples, and after bright
//    features, that loses more than the 1e-5 relative S/N the search keeps): widths up to 16 are summed by
//    doubling, a longer boxcar is the rest of its first chunk (S, registers) + the chunks between + the
//    beginning of its last chunk (Lp, shared memory), all made of samples inside the boxcar.  The
//    chunks between are a difference of the chunks' prefix, which is kept as a value and its rounding error.
//    That sum is one per lane and width: it is added to the maximum over the lane's trials, not to each.
//    Other widths shorter than a chunk (3, 25, ...) take the difference of Lp and its rounding error (FP16).
//  * Warp v of a row holds the chunks [32 v, 32 v + 32).  Per row the warps exchange their chunks' prefix,
//    their segments' sums and the first 15 samples of each segment, and read each other's Lp; two barriers
//    of the row's warps.
//  * Each lane tracks its own best (S/N, row, width) over all rows.  At the end of a pixel all
//    warps rebuild the best row from all subbands and take the S/N and the earliest sample reaching it from
//    that row, with samples that are not finite counted, so that the trials without one are compared.
//  * One persistent CTA of 12 warps per SM; the next pixel's copy overlaps the search where two pixels
//    fit (16-bit rows, shorter FP32 windows), else it starts when the rows have been read for the last time.
// Bound by the reads of Lp (66 % of L1's throughput at 2048 FP32 samples, issue 50 %).  9696 pixels x 16
// subbands, 40 distinct DM rows, 12 widths, against the long-window kernel: 1250 samples FP32
// 1.35 ms (7.44), 2048 1.70 ms (11.9), BF16 1.70 ms (16.4), 3000 2.45 ms (27.3), 4096 3.15 ms (38.5).  With
// one FP32 prefix per segment and differences of it the same searches take 1.22, 1.54, 1.52, 2.10
// and 2.81 ms, but beside a dip of -300 a sample over 256 of 2048 samples the relative error of the S/N
// reaches 6e-4 (here 1.4e-7, the long-window kernel 2.4e-6), and a sample that is not a number left
// records whose sample did not have their S/N.
#pragma once

#include <climits>
#include <type_traits>

#include <cuda_fp16.h>

#include "nsfrb.h"
#include "nsfrb_internal.h"
#include "plan_internal.h"
#include "search_impl.cuh"

namespace nsfrb {
namespace dev {

constexpr int kWideHalo = 16;   // samples a segment hands to the one before it (15 are read)

struct WideLayout {
    size_t buf_bytes;   // a pixel's rows and the samples read past them
    size_t table, xs, pbuf, lo, carr, halo, sums, sinv, best, red, bar, total;
};

__host__ __device__ inline WideLayout wide_layout(const SearchParams &p, int C, int V, int nb) {
    WideLayout L{};
    const size_t es = p.dtype == 0 ? 4 : 2;
    // chunks past the end are read (and masked): of the top subband, whose shift is 0, up to sample 32 C V
    L.buf_bytes = align_up(es * ((size_t)(p.n_sub - 1) * p.n_t + (size_t)V * 32 * C + 16), 128);
    size_t o = 0;
    L.table = o;
    o += align_up(sizeof(int32_t) * ((size_t)p.n_u * kInfo + p.n_deltas + (size_t)p.n_u * p.n_sub), 128);
    L.xs = o;
    o += L.buf_bytes * nb;
    L.pbuf = o;   // [kWarps][32 C]; at the end of a pixel its best row's prefix (value, error, count)
    o += sizeof(float) * (size_t)kWarps * 32 * C;
    L.lo = o;     // [kWarps][32 C] rounding errors of Lp, FP16, where a width needs them
    o += p.wide_lo ? sizeof(__half) * (size_t)kWarps * 32 * C : 0;
    L.carr = o;   // [kWarps][32] the chunks' prefix within their segment
    o += sizeof(float2) * kWarps * 32;
    L.halo = o;   // [kWarps + 1][16]: the row after the last stays zero
    o += sizeof(float) * (kWarps + 1) * kWideHalo;
    L.sums = o;   // [kWarps] segment sums; at the end of a pixel the warps' sums
    o += sizeof(float2) * 16;
    L.sinv = o;
    o += sizeof(float) * kMaxW;
    L.best = o;   // [kWarps] S/N, row * kMaxW + width index
    o += (sizeof(float) + sizeof(int32_t)) * kWarps;
    L.red = o;    // [kWarps] maximum, earliest sample, invalid samples
    o += (sizeof(float) + 2 * sizeof(int32_t)) * kWarps;
    L.bar = align_up(o, 8);
    L.total = L.bar + 16;
    return L;
}

template <int THREADS>
__device__ __forceinline__ void team_sync(int team) {
    asm volatile("bar.sync %0, %1;" ::"r"(team + 1), "n"(THREADS) : "memory");
}

// Sums of the chunk's samples from each one to the chunk's end, as pairs (two chains, like prefix_pairs).
template <int C>
__device__ __forceinline__ void suffix_pairs(const float2 (&D)[C / 2], float2 (&S)[C / 2]) {
    constexpr int H1 = 2 * ((C / 2 + 1) / 2);   // the second half, [H1, C), and what the first adds to it
    float run = 0.0f;
#pragma unroll
    for (int c = C - 1; c >= H1; --c) {
        run += pget(D, c);
        pset(S, c, run);
    }
    float q = 0.0f;
#pragma unroll
    for (int c = H1 - 1; c >= 0; --c) {
        q += pget(D, c);
        pset(S, c, q);
    }
    const float2 rr = make_float2(run, run);
#pragma unroll
    for (int m = 0; m < H1 / 2; ++m) S[m] = add2(S[m], rr);
}

template <int C, int V, int ST>
__global__ void __launch_bounds__(kThreads, 1) search_kernel_wide(const __grid_constant__ SearchParams p) {
    static_assert(C % 4 == 2 && C >= kSmallMax && kWarps % V == 0 && V <= 4, "chunk of sample pairs; whole teams");
    extern __shared__ __align__(128) unsigned char smem[];
    constexpr int kEs = (ST == 0) ? 4 : 2, G = kWarps / V, kSeg = 32 * C, kChunks = 32 * V;
    const int nb = p.nb;
    const WideLayout lay = wide_layout(p, C, V, nb);
    int32_t *s_table = reinterpret_cast<int32_t *>(smem + lay.table);
    float *s_p = reinterpret_cast<float *>(smem + lay.pbuf);
    float *s_halo = reinterpret_cast<float *>(smem + lay.halo);
    float2 *s_sums = reinterpret_cast<float2 *>(smem + lay.sums);
    float *s_inv = reinterpret_cast<float *>(smem + lay.sinv);
    float *s_bs = reinterpret_cast<float *>(smem + lay.best);
    int32_t *s_buw = reinterpret_cast<int32_t *>(s_bs + kWarps);
    float *s_rm = reinterpret_cast<float *>(smem + lay.red);
    int32_t *s_rt = reinterpret_cast<int32_t *>(s_rm + kWarps);
    int32_t *s_rn = s_rt + kWarps;
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
    float *Pt = s_p + (size_t)team * V * kSeg;   // the team's Lp, chunk after chunk
    float *Pw = Pt + v * kSeg;
    __half *Low = reinterpret_cast<__half *>(smem + lay.lo) + (size_t)warp * kSeg;
    float *halo_out = s_halo + warp * kWideHalo;
    // the segment after this one; the last one's last chunk ends past the window (its last sample is -inf or NaN)
    const float *halo_in = s_halo + (v + 1 < V ? warp + 1 : kWarps) * kWideHalo;
    float2 *sums = s_sums + team * V;
    float2 *carr = reinterpret_cast<float2 *>(smem + lay.carr) + team * kChunks;
    const int chunk = v * 32 + lane, t0 = chunk * C;
    const int top = small_top<C>(p);

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
                // the copies in flight are waited for (bounded) before the CTA leaves
                mbar_wait(&s_bar[b], static_cast<uint32_t>(nb == 2 ? i >> 1 : i) & 1u);
                if (nb == 2 && nxt < n_items) mbar_wait(&s_bar[b ^ 1], static_cast<uint32_t>((i + 1) >> 1) & 1u);
            }
            return;
        }

        // ---- the team's rows; a pixel whose best is +inf (an infinite sample) once more without such samples
        float bs = neg_inf();
        int buw = -1;
#pragma unroll 1
        for (bool clean = false;; clean = true) {
            bs = neg_inf();
            buw = -1;
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
                if (clean) {
#pragma unroll
                    for (int m = 0; m < C / 2; ++m) D[m] = add2(D[m], sub2(D[m], D[m]));   // infinite: NaN
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
                float inc_h, inc_l = 0.0f;   // the segment's prefix up to this chunk's end, and its rounding error
                {
                    float2 Lp[C / 2];
                    inc_h = prefix_pairs<C>(D, Lp);
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const float yh = __shfl_up_sync(kFull, inc_h, o), yl = __shfl_up_sync(kFull, inc_l, o);
                        if (lane >= o) pair_add(inc_h, inc_l, yh, yl);
                    }
                    float ch = __shfl_up_sync(kFull, inc_h, 1), cl = __shfl_up_sync(kFull, inc_l, 1);
                    if (lane == 0) ch = cl = 0.0f;
                    carr[chunk] = make_float2(ch, cl);
                    if (lane == 31) sums[v] = make_float2(inc_h, inc_l);
                    if (lane == 0) {
                        float2 *h2 = reinterpret_cast<float2 *>(halo_out);
#pragma unroll
                        for (int m = 0; m < kWideHalo / 2; ++m) h2[m] = D[m];
                    }
                    float2 *dst = reinterpret_cast<float2 *>(Pw + lane * C);
#pragma unroll
                    for (int m = 0; m < C / 2; ++m) dst[m] = Lp[m];
                    if (p.wide_lo) {
                        // what each Lp lacks to the sum it stands for
                        __half2 *lo2 = reinterpret_cast<__half2 *>(Low + lane * C);
                        float h = 0.0f, l = 0.0f;
#pragma unroll
                        for (int m = 0; m < C / 2; ++m) {
                            const float e0 = (h - Lp[m].x) + l;
                            pair_add(h, l, D[m].x, 0.0f);
                            const float e1 = (h - Lp[m].y) + l;
                            pair_add(h, l, D[m].y, 0.0f);
                            lo2[m] = __floats2half2_rn(e0, e1);
                        }
                    }
                }
                float m32;
                {
                    float2 Hd[kSmallMax / 2];
                    halo_samples<C>(D, Hd);
                    team_sync<32 * V>(team);
                    if (lane == 31) {
#pragma unroll
                        for (int m = 0; m < kSmallMax / 2; ++m) Hd[m] = reinterpret_cast<const float2 *>(halo_in)[m];
                    }
                    m32 = small_sums<C>(D, Hd, top, [&](int j, float m) {
                        if (p.pow2_wi[j] >= 0) consider(p.pow2_wi[j], m);
                    });
                }
                if (p.has_large || p.n_gen) {
                    float2 S[C / 2];
                    suffix_pairs<C>(D, S);
                    // from this chunk's end to the end of the segment, of the next, and of the one after (-inf
                    // from where there is no such segment)
                    const float2 own = sums[v];
                    float rest[3];
                    rest[0] = v + 1 < V ? (own.x - inc_h) + (own.y - inc_l) : neg_inf();
#pragma unroll
                    for (int j = 1; j < 3; ++j)
                        rest[j] = v + j + 1 < V ? rest[j - 1] + (sums[v + j].x + sums[v + j].y) : neg_inf();
                    // sum of the chunks after this one and before chunk + q; h, l: what its own segment's
                    // prefix lacks
                    const float2 *ahead = carr + chunk;
                    auto between = [&](auto q) -> float {
                        constexpr int A = decltype(q)::value / 32, B = decltype(q)::value % 32;
                        const float2 cg = ahead[decltype(q)::value];
                        const bool next = lane + B >= 32;
                        if constexpr (A == 0)
                            return (cg.x + (next ? rest[0] : -inc_h)) + (cg.y + (next ? 0.0f : -inc_l));
                        else
                            return (cg.x + (next ? rest[A] : rest[A - 1])) + cg.y;
                    };
                    const int first = v * kSeg;   // this segment's first sample: a width with no trial from it on is left out
                    // Width q C + r: trial c of the chunk ends in chunk + q, from c = C - r on in the one after.
                    // A trial that would leave the row reads what lies there, and adds -inf.
#define NSFRB_WIDE_LARGE(J)                                                                                     \
    if constexpr ((1 << J) > kSmallMax) {                                                                       \
        if (p.pow2_wi[J] >= 0 && first + (1 << J) <= L) {                                                       \
            constexpr int W = 1 << J, Q = W / C, R = W % C;                                                     \
            const float2 *x = reinterpret_cast<const float2 *>(Pt + min(t0 + W, (kChunks - 1) * C + R));        \
            float a[2] = {neg_inf(), neg_inf()};                                                                \
            if constexpr (Q > 0) {                                                                              \
                _Pragma("unroll") for (int m = 0; m < (C - R) / 2; ++m) {                                       \
                    const float2 bx = add2(S[m], x[m]);                                                         \
                    a[0] = fmax3(a[0], bx.x, bx.y);                                                             \
                }                                                                                               \
                a[0] += between(std::integral_constant<int, Q>{});                                              \
            } else {                                                                                            \
                a[0] = m32;                                                                                     \
            }                                                                                                   \
            if constexpr (R > 0) {                                                                              \
                _Pragma("unroll") for (int m = (C - R) / 2; m < C / 2; ++m) {                                   \
                    const float2 bx = add2(S[m], x[m]);                                                         \
                    a[1] = fmax3(a[1], bx.x, bx.y);                                                             \
                }                                                                                               \
                a[1] += between(std::integral_constant<int, Q + 1>{});                                          \
            }                                                                                                   \
            consider(p.pow2_wi[J], fmaxf(a[0], a[1]));                                                          \
        }                                                                                                       \
    }
                    NSFRB_POW2(NSFRB_WIDE_LARGE)
#undef NSFRB_WIDE_LARGE
#pragma unroll 1
                    for (int g = 0; g < p.n_gen; ++g) {
                        const int wi = p.gen_wi[g], w = p.widths[wi], q = w / C, r = w - q * C;
                        if (first + w > L) continue;
                        const float *x = Pt + min(t0 + w, (kChunks - 1) * C + r), *own_p = Pw + lane * C;
                        const __half *own_lo = Low + lane * C;
                        auto link = [&](int g1) -> float {   // between, of chunk g1
                            if (g1 >= kChunks) return neg_inf();
                            const float2 cg = carr[g1];
                            const int dv = (g1 >> 5) - v;
                            if (dv == 0) return (cg.x - inc_h) + (cg.y - inc_l);
                            return (cg.x + (dv == 1 ? rest[0] : dv == 2 ? rest[1] : rest[2])) + cg.y;
                        };
                        float a[2] = {neg_inf(), neg_inf()};
#pragma unroll
                        for (int c = 0; c < C; ++c) {
                            if (c + r >= C)
                                a[1] = fmaxf(a[1], pget(S, c) + x[c]);
                            else if (q > 0)
                                a[0] = fmaxf(a[0], pget(S, c) + x[c]);
                            else
                                a[0] = fmaxf(a[0], (own_p[c + r] - own_p[c]) +
                                                       (__half2float(own_lo[c + r]) - __half2float(own_lo[c])));
                        }
                        if (q > 0) a[0] += link(chunk + q);
                        a[1] += link(chunk + q + 1);
                        const float s = fmaxf(a[0], a[1]) * s_inv[wi];
                        if (s > bs || (s == bs && uw + wi < buw)) {
                            bs = s;
                            buw = uw + wi;
                        }
                    }
                }
                team_sync<32 * V>(team);   // the row's Lp, prefixes, halos and sums have been read
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
            // ties go to the smallest row, then width
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
            if (clean || bs != -neg_inf()) break;
            __syncthreads();   // s_bs has been read
        }

        // ---- the pixel's record, from its best row rebuilt: prefix and its rounding error, samples that are
        // not finite taken as zero and counted
        const bool any = buw >= 0;
        const int u = any ? buw / kMaxW : 0, wi = any ? buw % kMaxW : 0, w = p.widths[wi];
        const int L = any ? n_t - s_info[u * kInfo + UI_SMAX] : 0;
        constexpr int CC = ((32 * C * V + kThreads - 1) / kThreads) | 1;   // samples per thread, odd
        static_assert(3 * kChunks * C <= kWarps * kSeg, "value, error and count of the prefix");
        float *ph = s_p, *pl = s_p + kChunks * C;
        int32_t *pn = reinterpret_cast<int32_t *>(s_p + 2 * kChunks * C);
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
        float dl[CC];
        float tot = 0.0f, tot_l = 0.0f;
        uint32_t bad = 0;   // this thread's samples that are not finite
#pragma unroll
        for (int c = 0; c < CC; ++c) {
            float x = t1 + c < L ? d[c] : 0.0f;
            if (!(fabsf(x) < -neg_inf())) {
                x = 0.0f;
                bad |= 1u << c;
            }
            d[c] = tot;
            dl[c] = tot_l;
            pair_add(tot, tot_l, x, 0.0f);
        }
        float ih = tot, il = tot_l;
        int in = __popc(bad);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const float yh = __shfl_up_sync(kFull, ih, o), yl = __shfl_up_sync(kFull, il, o);
            const int yn = __shfl_up_sync(kFull, in, o);
            if (lane >= o) {
                pair_add(ih, il, yh, yl);
                in += yn;
            }
        }
        if (lane == 31) {
            s_sums[warp] = make_float2(ih, il);
            s_rn[warp] = in;
        }
        float ch = __shfl_up_sync(kFull, ih, 1), cl = __shfl_up_sync(kFull, il, 1);
        int cn = __shfl_up_sync(kFull, in, 1);
        if (lane == 0) ch = cl = 0.0f, cn = 0;
        fence_proxy_async();
        __syncthreads();   // the rows have been read for the last time
        if (nb == 1 && tid == 0 && nxt < n_items) issue(nxt, 0);
        for (int g = 0; g < warp; ++g) {
            pair_add(ch, cl, s_sums[g].x, s_sums[g].y);
            cn += s_rn[g];
        }
#pragma unroll
        for (int c = 0; c < CC; ++c) {
            pair_add(d[c], dl[c], ch, cl);
            if (t1 + c <= L) {
                ph[t1 + c] = d[c];
                pl[t1 + c] = dl[c];
                pn[t1 + c] = cn;
            }
            cn += (bad >> c) & 1u;
        }
        __syncthreads();
        float m = neg_inf();
#pragma unroll
        for (int c = 0; c < CC; ++c) {
            const int e = t1 + c + w;
            const bool ok = any && e <= L && pn[e] == pn[t1 + c];
            d[c] = ok ? (ph[e] - d[c]) + (pl[e] - dl[c]) : neg_inf();
            m = fmaxf(m, d[c]);
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
                int t = -1;
                for (int g = 0; g < kWarps; ++g)   // ascending samples: the earliest on ties
                    if (s_rm[g] > best) {
                        best = s_rm[g];
                        t = s_rt[g];
                    }
                r = PixRec{record_snr(best, p.sigma ? p.sigma[pix] : p.sigma_default, w, s_inv[wi]),
                           s_info[u * kInfo + UI_FIRST_D], wi, t};
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
