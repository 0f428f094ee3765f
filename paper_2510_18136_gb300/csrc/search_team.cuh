// The search of arXiv 2510.18136 Sec. 2.2 for windows of 608 to 1215 samples, candidate records only: the full
// 1200-sample window (FP32, BF16, FP16, and the FP32 slabs of MAD normalisation), a warp per DM row.
//
// The row search and the hand-over of pixels are those of the barrier-free kernel (search_impl.cuh); this
// kernel differs in what its warps share and carry:
//  * A pixel's rows lie packed in shared memory as they do in the cube, one bulk copy per pixel; the samples past
//    the valid range are set to -inf in registers when the range changes (ranges shrink as the DM
//    grows), so rows need no -inf tail.
//  * Of the delay tables only the row infos, the changes and the first row of each group are kept in
//    shared memory, and the earliest-sample search borrows the warp's prefix buffer.  What that
//    frees, and registers held below 144 a thread, lets more than 12 warps run: the search is bound by
//    the latency of its dependent chains (prefix, scan, shared-memory round trip) at three warps a
//    scheduler.
//  * The warps of a pixel share the best S/N found so far: a row whose maximum is below it cannot
//    be the record, and skips the search for its earliest sample.
//  * 1 / (sigma sqrt(w)) of the power-of-two widths is kept in width order (NaN where a width is
//    absent): a row reads it in vector loads, takes one maximum over its widths, and looks for
//    the width that has it only when the row beats the pixel's best.
//  * The copy of a team's next pixel starts as soon as its warps have read the rows for the last time,
//    for every storage type.
// 40401 pixels x 16 subbands, 12 widths, against the barrier-free kernel's default tile: FP32 1200 samples, 40
// DM rows 2395 us (2592), 101 rows 4750 us (5264), 640 samples 1251 us (1929); BF16 1200 samples 1965 us
// (2203), 101 rows 4409 us (4877), 640 samples 1266 us (3087).  Not kept: fourteen warps of 128 registers for
// FP32 (2525 us), and reading the next row's infos and first change ahead (2386 -> 2447 us).
#pragma once

#include <algorithm>
#include <climits>

#include "nsfrb.h"
#include "nsfrb_internal.h"
#include "plan_internal.h"
#include "search_impl.cuh"

namespace nsfrb {
namespace dev {

struct TeamLayout {
    size_t buf_bytes;
    size_t table, first, xs, pbuf, wbest, sinv, cnt, bar, total;
};

// teams x warps: the CTA's shape.
__host__ __device__ inline TeamLayout team_layout(const SearchParams &p, int C, int teams, int warps) {
    TeamLayout L{};
    const size_t es = p.dtype == 0 ? 4 : 2;
    L.buf_bytes = es * (size_t)p.n_sub * p.n_t;   // a multiple of 16 bytes
    size_t o = 0;
    L.table = o;
    o += align_up(sizeof(int32_t) * ((size_t)p.n_u * kInfo + p.n_deltas), 16);
    L.first = o;
    o += align_up(sizeof(int32_t) * (size_t)warps * p.n_sub, 128);
    L.xs = o;
    // a chunk past the window reads on into the next buffer, after the last one into its tail (masked)
    o += align_up(L.buf_bytes * teams + es * (size_t)(32 * C + 16), 16);
    L.pbuf = o;
    o += sizeof(float) * (size_t)teams * warps * 32 * C;
    L.wbest = o;
    o += sizeof(PixRec) * 2 * (size_t)teams * warps;
    L.sinv = o;   // [teams][2]: [16] in power-of-two order, [16] by width index
    o += sizeof(float) * 4 * kMaxW * (size_t)teams;
    L.cnt = o;    // [teams][2] done, [teams][2] best so far, [teams] rows read, error
    o += sizeof(int32_t) * (5 * (size_t)teams + 1);
    L.bar = align_up(o, 8);
    L.total = L.bar + sizeof(unsigned long long) * teams;
    return L;
}

template <int C, int ST, int TEAMS, int W>
__global__ void __launch_bounds__(TEAMS * W * 32, 1) search_kernel_team(const __grid_constant__ SearchParams p) {
    static_assert(C % 4 == 2 && C >= kSmallMax && C + kSmallMax <= kFindScr, "chunk of sample pairs");
    extern __shared__ __align__(128) unsigned char smem[];
    constexpr int SH = kSmallMax, kEs = (ST == 0) ? 4 : 2, kThr = TEAMS * W * 32;
    const TeamLayout lay = team_layout(p, C, TEAMS, W);
    int32_t *s_table = reinterpret_cast<int32_t *>(smem + lay.table);
    int32_t *s_first = reinterpret_cast<int32_t *>(smem + lay.first);               // [W][n_sub]
    PixRec *s_wbest = reinterpret_cast<PixRec *>(smem + lay.wbest);                 // [TEAMS][2][W]
    float *s_inv = reinterpret_cast<float *>(smem + lay.sinv);                      // [TEAMS][2][2][kMaxW]
    int32_t *s_cnt = reinterpret_cast<int32_t *>(smem + lay.cnt);                   // [TEAMS][2]
    volatile uint32_t *s_top = reinterpret_cast<uint32_t *>(s_cnt + 2 * TEAMS);     // [TEAMS][2]
    int32_t *s_rd = s_cnt + 4 * TEAMS;                                              // [TEAMS]
    int32_t *s_flag = s_rd + TEAMS;
    unsigned long long *s_bar = reinterpret_cast<unsigned long long *>(smem + lay.bar);

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int team = warp / W, wt = warp % W;
    const int n_sub = p.n_sub, n_t = p.n_t, n_ua = p.n_u_active;
    const int table_words = p.n_u * kInfo + p.n_deltas;
    for (int i = tid; i < table_words; i += kThr) s_table[i] = p.table[i];
    const int32_t *s_info = s_table;
    const int32_t *s_delta = s_table + p.n_u * kInfo;
    // the first row of each group of rows, row by row of the unique-row shifts
    for (int i = tid; i < W * n_sub; i += kThr) {
        const int u = ((i / n_sub) * n_ua) / W;
        s_first[i] = p.table[table_words + u * n_sub + i % n_sub];
    }
    constexpr uint32_t kNone = 0x007fffffu;   // f2key(-inf)
    if (tid == 0) {
        for (int t = 0; t < TEAMS; ++t) {
            mbar_init(&s_bar[t], 1);
            s_rd[t] = 0;
        }
        for (int r = 0; r < 2 * TEAMS; ++r) {
            s_cnt[r] = 0;
            s_top[r] = kNone;
        }
        s_flag[0] = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_proxy_async();
    }
    int64_t n_items = p.n_items;
    if (p.n_items_dev) n_items = *p.n_items_dev;
    auto item_pixel = [&](int64_t it) -> int64_t {
        return p.pix_list ? static_cast<int64_t>(p.pix_list[it]) : p.pix0 + it;
    };
    unsigned char *xs = smem + lay.xs + team * lay.buf_bytes;
    // one warp: 1 / (sigma sqrt(w)) of item `it` into record slot rs, then its rows into the team's buffer
    auto issue_warp = [&](int64_t it, int rs) {
        const int64_t pix = item_pixel(it);
        const float sigma = p.sigma ? p.sigma[pix] : p.sigma_default;
        if (lane < kMaxW) {
            const float by_pow2 = lane < kPow2 && p.pow2_wi[lane] >= 0
                                      ? 1.0f / (sigma * sqrtf(static_cast<float>(1 << lane)))
                                      : qnan();
            s_inv[rs * 2 * kMaxW + lane] = by_pow2;
            if (lane < p.n_w)
                s_inv[(rs * 2 + 1) * kMaxW + lane] = 1.0f / (sigma * sqrtf(static_cast<float>(p.widths[lane])));
        }
        __syncwarp();
        if (lane == 0) {
            const uint32_t bytes = static_cast<uint32_t>(lay.buf_bytes);
            mbar_expect_tx(&s_bar[team], bytes);
            bulk_g2s(xs, static_cast<const unsigned char *>(p.cube) + (pix - p.cube_pix0) * static_cast<int64_t>(bytes),
                     bytes, &s_bar[team]);
        }
    };
    __syncthreads();
    const int64_t G = static_cast<int64_t>(gridDim.x) * TEAMS;
    const int64_t it0 = static_cast<int64_t>(blockIdx.x) * TEAMS + team;
    int issued_last = -1;   // local index of the last item whose copy this warp started
    if (wt == 0 && it0 < n_items) {
        issue_warp(it0, 2 * team);
        issued_last = 0;
    }

    float *Pw = reinterpret_cast<float *>(smem + lay.pbuf) + (size_t)warp * 32 * C;
    const int t0 = lane * C;
    int i = 0;
    for (int64_t it = it0; it < n_items; it += G, ++i) {
        const int rs = 2 * team + (i & 1);
        if (*reinterpret_cast<volatile int32_t *>(s_flag)) break;
        if (!mbar_wait(&s_bar[team], static_cast<uint32_t>(i) & 1u)) {
            if (lane == 0) {
                atomicOr(s_flag, ERR_WAIT_TIMEOUT);
                atomicOr(p.err, ERR_WAIT_TIMEOUT);
            }
            break;
        }
        const int64_t pix = item_pixel(it);
        const int g = (wt + i) % W;   // the groups that hold one row more rotate over the warps
        const int u_lo = (g * n_ua) / W, u_hi = ((g + 1) * n_ua) / W;
        // the last warp of the team to read the buffer for this pixel starts the copy of its next pixel
        auto read_done = [&]() {
            fence_proxy_async();
            int lastr = 0;
            if (lane == 0) {
                __threadfence_block();
                lastr = atomicAdd(&s_rd[team], 1) == W - 1;
                __threadfence_block();
            }
            lastr = __shfl_sync(kFull, lastr, 0);
            if (lastr) {
                if (lane == 0) s_rd[team] = 0;
                __syncwarp();
                if (it + G < n_items) {
                    issue_warp(it + G, 2 * team + ((i + 1) & 1));
                    issued_last = i + 1;
                }
            }
            __syncwarp();
        };
        const float4 *inv4 = reinterpret_cast<const float4 *>(s_inv + rs * 2 * kMaxW);
        const float *inv_w = s_inv + (rs * 2 + 1) * kMaxW;
        float bsnr = neg_inf();
        int bu = -1, bwi = -1, bt = -1;
        float2 D[C / 2];
        int L_prev = -1;
        if (u_lo >= u_hi) read_done();
#pragma unroll 1
        for (int u = u_lo; u < u_hi; ++u) {
            const int32_t *info = s_info + u * kInfo;
            if (u == u_lo) {
#pragma unroll
                for (int m = 0; m < C / 2; ++m) D[m] = make_float2(0.0f, 0.0f);
                const int32_t *sh = s_first + g * n_sub;
                int at = sh[0];
#pragma unroll 1
                for (int k = 0; k < n_sub; ++k) {
                    const int e = k * n_t + t0 + at;
                    if (k + 1 < n_sub) at = sh[k + 1];
                    acc_row<C, false, ST>(D, xs, 0, 0, e);
                }
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
                        continue;
                    }
                    acc_row<C, false, ST>(D, xs, 0, 0, at - so + sn);
                    acc_row<C, true, ST>(D, xs, 0, 0, at);
                }
            }
            if (u == u_hi - 1) read_done();
            const int L = n_t - info[UI_SMAX];
            if (L != L_prev) {
#pragma unroll
                for (int m = 0; m < C / 2; ++m) {
                    if (t0 + 2 * m >= L) D[m].x = neg_inf();
                    if (t0 + 2 * m + 1 >= L) D[m].y = neg_inf();
                }
                L_prev = L;
            }
            const float top = key2f(s_top[rs]);   // the pixel's best so far, of any of its warps
            float s[kPow2];   // this lane's best S/N of each power-of-two width, NaN where absent
            {
                float2 Lp[C / 2], Hh[SH / 2];
                const float tot = prefix_pairs<C>(D, Lp);
                halo_pairs<C, SH>(Lp, tot, Hh);
                const float carry = lane_carry(tot, lane);
                const float4 ia = inv4[0];
                const float ib = inv4[1].x;
                s[0] = small_max_pk<C, SH, 1>(D, Lp, Hh) * ia.x;
                s[1] = small_max_pk<C, SH, 2>(D, Lp, Hh) * ia.y;
                s[2] = small_max_pk<C, SH, 4>(D, Lp, Hh) * ia.z;
                s[3] = small_max_pk<C, SH, 8>(D, Lp, Hh) * ia.w;
                s[4] = small_max_pk<C, SH, 16>(D, Lp, Hh) * ib;
                store_p<C>(Pw, t0, carry, Lp);
            }
            __syncwarp();
#pragma unroll
            for (int j = 5; j < kPow2; ++j) s[j] = qnan();
            if (p.has_large) {
                float2 Ps[C / 2];
                load_ps<C>(Pw, lane, Ps);
                const float4 ib = inv4[1], ic = inv4[2];
                s[5] = large_max_pk<C, 1>(Ps) * ib.y;
                s[6] = large_max_pk<C, 2>(Ps) * ib.z;
                s[7] = large_max_pk<C, 4>(Ps) * ib.w;
                s[8] = large_max_pk<C, 8>(Ps) * ic.x;
                s[9] = large_max_pk<C, 16>(Ps) * ic.y;
                if constexpr (C > 32) s[10] = large_max_pk<C, 32>(Ps) * ic.z;
            }
            float sg = neg_inf();   // the other widths
            int wg = INT_MAX;
#pragma unroll 1
            for (int q = 0; q < p.n_gen; ++q) {
                const int wi = p.gen_wi[q];
                const float v = generic_max(Pw, p.widths[wi], L, 0, lane) * inv_w[wi];
                if (v > sg) {
                    sg = v;
                    wg = wi;
                }
            }
            float ls = fmax3(fmax3(s[0], s[1], s[2]), fmax3(s[3], s[4], s[5]), fmax3(s[6], s[7], s[8]));
            ls = fmaxf(fmax3(ls, s[9], s[10]), sg);
            // a row that beats the warp's own best and is not below the pixel's
            if (__any_sync(kFull, ls > bsnr && ls >= top)) {
                bsnr = warp_max(ls);
                // the smallest width index that reaches it, and the lanes whose own best that is
                unsigned lw = sg == bsnr ? static_cast<unsigned>(wg) : 0xffffffffu;
#pragma unroll
                for (int j = kPow2 - 1; j >= 0; --j)
                    if (s[j] == bsnr) lw = min(lw, static_cast<unsigned>(p.pow2_wi[j]));
                bwi = static_cast<int>(__reduce_min_sync(kFull, lw));
                const unsigned match = __ballot_sync(kFull, static_cast<int>(lw) == bwi);
                bt = find_t_even<C>(p, D, Pw, bwi, inv_w[bwi], bsnr, L, lane, false, match, Pw);
                bu = u;
                if (lane == 0) atomicMax(const_cast<uint32_t *>(&s_top[rs]), f2key(bsnr));
            }
            __syncwarp();
        }
        // publish; this warp's reads of the buffer are done before the copy that refills it
        fence_proxy_async();
        int last = 0;
        if (lane == 0) {
            s_wbest[rs * W + g] = PixRec{bsnr, bu, bwi, bt};
            __threadfence_block();
            last = atomicAdd(&s_cnt[rs], 1) == W - 1;
            __threadfence_block();
        }
        last = __shfl_sync(kFull, last, 0);
        if (last) {
            if (lane == 0) {
                PixRec best{neg_inf(), -1, -1, -1};
                for (int q = 0; q < W; ++q) {
                    const PixRec r = s_wbest[rs * W + q];
                    if (r.snr > best.snr) best = r;
                }
                if (best.dm_idx >= 0) best.dm_idx = s_info[best.dm_idx * kInfo + UI_FIRST_D];
                if (p.bad_pix && p.bad_pix[pix]) {
                    best = PixRec{neg_inf(), -1, -1, -1};
                    atomicOr(p.err, ERR_ZERO_MAD);
                }
                p.rec[pix] = best;
                s_cnt[rs] = 0;
                s_top[rs] = kNone;
            }
        }
        __syncwarp();
    }
    // after an error: wait (bounded) for a copy this warp started that may still be in flight
    if (*reinterpret_cast<volatile int32_t *>(s_flag) && lane == 0 && issued_last >= 0)
        mbar_wait(&s_bar[team], static_cast<uint32_t>(issued_last) & 1u);
}

template <int C, int ST, int TEAMS, int W>
cudaError_t team_launch(const SearchParams &p, int n_sm, size_t smem, cudaStream_t s) {
    const cudaError_t e = raise_smem_limit(reinterpret_cast<const void *>(search_kernel_team<C, ST, TEAMS, W>));
    if (e != cudaSuccess) return e;
    search_kernel_team<C, ST, TEAMS, W><<<n_sm, TEAMS * W * 32, smem, s>>>(p);
    return cudaGetLastError();
}

}  // namespace dev

// Samples per lane, and teams x warps, with compiled kernels.
#define NSFRB_TEAM_CHUNKS(X) X(22) X(26) X(34) X(38)
#define NSFRB_TEAM_SHAPES(X, C) X(C, 4, 4) X(C, 4, 3) X(C, 3, 5) X(C, 2, 8) X(C, 2, 6)

#define NSFRB_TEAM_CASE(C, T, W) \
    case 100 * C + 10 * T + W: return dev::team_launch<C, kSt, T, W>(p, n_sm, smem, s);
#define NSFRB_TEAM_CASES(C) NSFRB_TEAM_SHAPES(NSFRB_TEAM_CASE, C)
#define NSFRB_INSTANTIATE_TEAM(ST)                                                                       \
    cudaError_t launch_search_team_s##ST(const SearchParams &p, int n_sm, size_t smem, cudaStream_t s) { \
        constexpr int kSt = ST;                                                                          \
        switch (100 * p.mid_c + 10 * p.teams + p.mid_s) {                                                \
            NSFRB_TEAM_CHUNKS(NSFRB_TEAM_CASES)                                                          \
            default:                                                                                     \
                return cudaErrorInvalidValue;                                                            \
        }                                                                                                \
    }

}  // namespace nsfrb
