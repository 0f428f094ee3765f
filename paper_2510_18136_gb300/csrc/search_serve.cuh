// The serving search of arXiv 2510.18136 Sec. 2.2 (only trials that end in the newest block, at most 32 samples)
// of rolling windows up to 1215 samples, stored as rows of a ring.
//
// The newest block leaves at most 32 ends per DM row, so a lane is an end e and holds the boxcars b[w] that
// end there, one per width.  Going from one row to the next, a subband whose shift grows by one sample moves
// every boxcar by one sample of that subband:
//     b[w] += x_k[e + s] - x_k[e - w + s],
// so a row costs one read per width and changed subband, not the de-dispersion and prefix of the whole
// window.  Only a group's first row (and a row whose ends have moved out of the 32 lanes) is built
// from all samples: de-dispersed in chunks of C samples per lane, prefix to shared memory, b[w] = P[e] - P[e - w].
//  * Ends: lane j holds e = E - j, E the last end of the row that was built.  Rows of larger delay end
//    earlier (the newest block begins earlier in the top subband's frame), so the row's ends are
//    the lanes with n_t - smax - new_blk < e <= n_t - smax; a lane past the end of the
//    range never comes back, whatever its boxcars read.
//  * Trials, S/N and ties are those of the other kernels: t = e - w >= 0, the smallest DM row, width index
//    and sample of the largest S/N.
//  * Precision: a boxcar keeps the rounding of its updates, relative to the largest value it had since the row was
//    built, as the masked search of the other kernels keeps that of the prefixes and samples it
//    updates: beside a sample of -1e4 (u = 2^-10 its unit) 0.34 u rms here and 0.36 u there.
// Pixels are handed over between the teams of a persistent CTA as in search_team.cuh.  A row's window starts
// anywhere in its ring row; it is copied from the 16-byte boundary below.
// Bound by instruction issue at 12 warps an SM.  301 x 301 pixels, BF16 window of 1200 samples, 25-sample
// block, 40 DM rows, 12 widths: 1.88 ms, against 3.30 ms for the barrier-free kernel, which
// de-disperses and sums the whole window for every row (3.15 ms with boxcar starts recomputed and
// a branch per width; three teams of five warps 2.14 ms, two of six 2.66 ms).
#pragma once

#include <algorithm>
#include <climits>

#include "nsfrb.h"
#include "nsfrb_internal.h"
#include "plan_internal.h"
#include "search_impl.cuh"

namespace nsfrb {
namespace dev {

constexpr int kRebuild = 20;   // a moved sample costs about 75 instructions, a built row 1500

struct ServeLayout {
    int pitch;   // elements from row to row of a buffer
    size_t buf_bytes;
    size_t table, xs, pbuf, wbest, sinv, cnt, bar, total;
};

__host__ __device__ inline ServeLayout serve_layout(const SearchParams &p, int C, int teams, int warps) {
    ServeLayout L{};
    const size_t es = p.dtype == 0 ? 4 : 2;
    const int epv = static_cast<int>(16 / es);
    L.pitch = static_cast<int>(align_up(static_cast<size_t>(p.n_t + epv - 1), epv));
    L.buf_bytes = es * (size_t)p.n_sub * L.pitch;
    size_t o = 0;
    L.table = o;
    o += align_up(sizeof(int32_t) * ((size_t)p.n_u * kInfo + p.n_deltas + (size_t)p.n_u * p.n_sub), 16);
    o = align_up(o, 128);
    L.xs = o;
    // chunks and ends past the window read on into the next buffer, after the last one into its tail
    o += align_up(L.buf_bytes * teams + es * (size_t)(32 * C + 16), 16);
    L.pbuf = o;
    o += sizeof(float) * (size_t)teams * warps * 32 * C;
    L.wbest = o;
    o += sizeof(PixRec) * 2 * (size_t)teams * warps;
    L.sinv = o = align_up(o, 16);   // [teams][2][kMaxW]
    o += sizeof(float) * 2 * kMaxW * (size_t)teams;
    L.cnt = o;    // [teams][2] done, error
    o += sizeof(int32_t) * (2 * (size_t)teams + 1);
    L.bar = align_up(o, 8);
    L.total = L.bar + sizeof(unsigned long long) * teams;
    return L;
}

// The sample at byte `at` of a buffer in storage ST, widened.
template <int ST>
__device__ __forceinline__ float buf_x(const unsigned char *xs, int at) {
    if constexpr (ST == 0)
        return *reinterpret_cast<const float *>(xs + at);
    else
        return widen16(*reinterpret_cast<const uint16_t *>(xs + at), ST);
}

// v - the sample at byte `at`: for 16-bit storage the mixed-precision fma of v and -1 (the product is exact).
template <int ST>
__device__ __forceinline__ float sub_buf(float v, const unsigned char *xs, int at) {
    if constexpr (ST == 0) {
        return v - *reinterpret_cast<const float *>(xs + at);
    } else {
        const uint16_t x = *reinterpret_cast<const uint16_t *>(xs + at);
        float r;
        if constexpr (ST == 1)
            asm("{\n\t.reg .b16 m;\n\tmov.b16 m, 0xBF80;\n\tfma.rn.f32.bf16 %0, %1, m, %2;\n\t}" : "=f"(r) : "h"(x), "f"(v));
        else
            asm("{\n\t.reg .b16 m;\n\tmov.b16 m, 0xBC00;\n\tfma.rn.f32.f16 %0, %1, m, %2;\n\t}" : "=f"(r) : "h"(x), "f"(v));
        return r;
    }
}

template <int C, int ST, int TEAMS, int W>
__global__ void __launch_bounds__(TEAMS * W * 32, 1) search_kernel_serve(const __grid_constant__ SearchParams p) {
    static_assert(C % 4 == 2, "chunk of sample pairs");
    extern __shared__ __align__(128) unsigned char smem[];
    constexpr int kEs = (ST == 0) ? 4 : 2, kEpv = 16 / kEs, kThr = TEAMS * W * 32;
    const ServeLayout lay = serve_layout(p, C, TEAMS, W);
    int32_t *s_table = reinterpret_cast<int32_t *>(smem + lay.table);
    PixRec *s_wbest = reinterpret_cast<PixRec *>(smem + lay.wbest);   // [TEAMS][2][W]
    float *s_inv = reinterpret_cast<float *>(smem + lay.sinv);        // [TEAMS][2][kMaxW]
    int32_t *s_cnt = reinterpret_cast<int32_t *>(smem + lay.cnt);     // [TEAMS][2]
    int32_t *s_flag = s_cnt + 2 * TEAMS;
    unsigned long long *s_bar = reinterpret_cast<unsigned long long *>(smem + lay.bar);

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int team = warp / W, wt = warp % W;
    const int n_sub = p.n_sub, n_t = p.n_t, n_ua = p.n_u_active, nb = p.new_blk, n_w = p.n_w;
    const int t_off = p.t_off_dev ? *p.t_off_dev : p.t_off;
    const int eoff = t_off & (kEpv - 1);
    const int row_elems = static_cast<int>(align_up(static_cast<size_t>(eoff + n_t), kEpv));
    const int table_words = p.n_u * kInfo + p.n_deltas + p.n_u * n_sub;
    for (int i = tid; i < table_words; i += kThr) s_table[i] = p.table[i];
    const int32_t *s_info = s_table;
    const int32_t *s_delta = s_table + p.n_u * kInfo;
    const int32_t *s_shift = s_delta + p.n_deltas;
    if (tid == 0) {
        for (int t = 0; t < TEAMS; ++t) mbar_init(&s_bar[t], 1);
        for (int r = 0; r < 2 * TEAMS; ++r) s_cnt[r] = 0;
        s_flag[0] = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_proxy_async();
    }
    const int64_t n_items = p.n_items;
    unsigned char *xs = smem + lay.xs + team * lay.buf_bytes;
    // one warp: 1 / (sigma sqrt(w)) of item `it` into record slot rs, then its rows into the team's buffer
    auto issue_warp = [&](int64_t it, int rs) {
        const int64_t pix = p.pix0 + it;
        if (lane < kMaxW) {   // (a boxcar past the last width is -inf: its S/N is NaN and never the largest)
            const float sg = p.sigma ? p.sigma[pix] : p.sigma_default;
            s_inv[rs * kMaxW + lane] = lane < n_w ? 1.0f / (sg * sqrtf(static_cast<float>(p.widths[lane]))) : qnan();
        }
        __syncwarp();
        const uint32_t bytes = static_cast<uint32_t>(row_elems * kEs);
        if (lane == 0) mbar_expect_tx(&s_bar[team], bytes * static_cast<uint32_t>(n_sub));
        __syncwarp();
        const unsigned char *src = static_cast<const unsigned char *>(p.cube);
        const int64_t row0 = (pix - p.cube_pix0) * n_sub;
        for (int k = lane; k < n_sub; k += 32)
            bulk_g2s(xs + (size_t)k * lay.pitch * kEs, src + ((row0 + k) * p.row_len + t_off - eoff) * kEs, bytes,
                     &s_bar[team]);
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
        const int64_t pix = p.pix0 + it;
        const int g = (wt + i) % W;
        const int u_lo = (g * n_ua) / W, u_hi = ((g + 1) * n_ua) / W;
        const float4 *inv4 = reinterpret_cast<const float4 *>(s_inv + rs * kMaxW);
        float bsnr = neg_inf();
        int bu = -1, bwi = -1, bt = -1;
        // per width: the boxcar that ends at e (-inf where it would start before the window: it stays -inf),
        // and the byte it starts at in a row
        float b[kMaxW];
        int st[kMaxW];
        int e = 0, e_at = 0, e_last = -1;   // this lane's end, its byte; the smallest end the lanes hold
#pragma unroll 1
        for (int u = u_lo; u < u_hi; ++u) {
            const int32_t *info = s_info + u * kInfo;
            const int L = n_t - info[UI_SMAX];
            const int lo = max(0, L - nb + 1);   // the row's ends are lo .. L
            // samples by which the row's subbands move: more than kRebuild cost more than building the row
            const int d0 = info[UI_DOFF], nd = info[UI_ND];
            const uint32_t mine = lane < nd ? static_cast<uint32_t>(s_delta[d0 + lane]) : 0u;
            const int steps = __reduce_add_sync(kFull, (mine >> 19) - ((mine >> 6) & 0x1fffu));
            if (u == u_lo || lo < e_last || steps > kRebuild) {
                {
                    float2 D[C / 2];
#pragma unroll
                    for (int m = 0; m < C / 2; ++m) D[m] = make_float2(0.0f, 0.0f);
                    const int32_t *sh = s_shift + u * n_sub;
                    int at = sh[0];
#pragma unroll 1
                    for (int k = 0; k < n_sub; ++k) {
                        const int x = k * lay.pitch + eoff + t0 + at;
                        if (k + 1 < n_sub) at = sh[k + 1];
                        acc_row<C, false, ST>(D, xs, 0, 0, x);
                    }
                    // samples at or past L only reach prefixes past P[L], which nothing reads
                    float2 Lp[C / 2];
                    const float tot = prefix_pairs<C>(D, Lp);
                    store_p<C>(Pw, t0, lane_carry(tot, lane), Lp);
                }
                __syncwarp();
                e = L - lane;
                e_at = max(e, 0) * kEs;
                e_last = max(0, L - 31);
                const float pe = Pw[max(e, 0)];
#pragma unroll
                for (int wi = 0; wi < kMaxW; ++wi) {
                    const int t = wi < n_w ? e - p.widths[wi] : -1;
                    st[wi] = max(t, 0) * kEs;
                    b[wi] = t >= 0 ? pe - Pw[max(t, 0)] : neg_inf();
                }
                __syncwarp();
            } else {
#pragma unroll 1
                for (int q = d0; q < d0 + nd; ++q) {
                    const uint32_t pk = static_cast<uint32_t>(s_delta[q]);
                    const int k = pk & 63u, sn = pk >> 19;
                    // delays grow with the DM: from the old shift up to the new one, sample by sample
                    int s = (pk >> 6) & 0x1fffu;
                    const unsigned char *row = xs + (k * lay.pitch + eoff + s) * kEs;
#pragma unroll 1
                    for (; s < sn; ++s, row += kEs) {
                        const float in = buf_x<ST>(row, e_at);
#pragma unroll
                        for (int w4 = 0; w4 < kMaxW; w4 += 4)
                            if (w4 < n_w) {
#pragma unroll
                                for (int wi = w4; wi < w4 + 4; ++wi) b[wi] = sub_buf<ST>(b[wi] + in, row, st[wi]);
                            }
                    }
                }
            }
            // the row's largest S/N of this lane; the width only where the warp's best is beaten
            float ls = neg_inf();
#pragma unroll
            for (int w4 = 0; w4 < kMaxW; w4 += 4)
                if (w4 < n_w) {
                    const float4 iv = inv4[w4 / 4];
                    ls = fmax3(ls, b[w4] * iv.x, b[w4 + 1] * iv.y);
                    ls = fmax3(ls, b[w4 + 2] * iv.z, b[w4 + 3] * iv.w);
                }
            if (e < lo || e > L) ls = neg_inf();
            if (__any_sync(kFull, ls > bsnr)) {
                bsnr = warp_max(ls);
                unsigned lw = 0xffffffffu;
                if (ls == bsnr) {
                    const float *inv = reinterpret_cast<const float *>(inv4);
#pragma unroll
                    for (int wi = kMaxW - 1; wi >= 0; --wi)
                        if (b[wi] * inv[wi] == bsnr) lw = wi;
                }
                bwi = static_cast<int>(__reduce_min_sync(kFull, lw));
                bt = warp_min(static_cast<int>(lw) == bwi ? e - p.widths[bwi] : INT_MAX);
                bu = u;
            }
        }
        // publish; the last warp of the pixel combines the groups in row order and starts the next copy
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
            if (it + G < n_items) {
                issue_warp(it + G, 2 * team + ((i + 1) & 1));
                issued_last = i + 1;
            }
            if (lane == 0) {
                PixRec best{neg_inf(), -1, -1, -1};
                for (int q = 0; q < W; ++q) {
                    const PixRec r = s_wbest[rs * W + q];
                    if (r.snr > best.snr) best = r;
                }
                if (best.dm_idx >= 0) best.dm_idx = s_info[best.dm_idx * kInfo + UI_FIRST_D];
                p.rec[pix] = best;
                s_cnt[rs] = 0;
            }
        }
        __syncwarp();
    }
    // after an error: wait (bounded) for a copy this warp started that may still be in flight
    if (*reinterpret_cast<volatile int32_t *>(s_flag) && lane == 0 && issued_last >= 0)
        mbar_wait(&s_bar[team], static_cast<uint32_t>(issued_last) & 1u);
}

template <int C, int ST, int TEAMS, int W>
cudaError_t serve_launch(const SearchParams &p, int n_sm, size_t smem, cudaStream_t s) {
    const cudaError_t e = raise_smem_limit(reinterpret_cast<const void *>(search_kernel_serve<C, ST, TEAMS, W>));
    if (e != cudaSuccess) return e;
    search_kernel_serve<C, ST, TEAMS, W><<<n_sm, TEAMS * W * 32, smem, s>>>(p);
    return cudaGetLastError();
}

}  // namespace dev

// Samples per lane, and teams x warps, with compiled kernels.
#define NSFRB_SERVE_CHUNKS(X) X(22) X(38)
#define NSFRB_SERVE_SHAPES(X, C) X(C, 4, 4) X(C, 4, 3) X(C, 3, 5) X(C, 2, 6)

#define NSFRB_SERVE_CASE(C, T, W) \
    case 100 * C + 10 * T + W: return dev::serve_launch<C, kSt, T, W>(p, n_sm, smem, s);
#define NSFRB_SERVE_CASES(C) NSFRB_SERVE_SHAPES(NSFRB_SERVE_CASE, C)
#define NSFRB_INSTANTIATE_SERVE(ST)                                                                       \
    cudaError_t launch_search_serve_s##ST(const SearchParams &p, int n_sm, size_t smem, cudaStream_t s) { \
        constexpr int kSt = ST;                                                                           \
        switch (100 * p.mid_c + 10 * p.teams + p.mid_s) {                                                 \
            NSFRB_SERVE_CHUNKS(NSFRB_SERVE_CASES)                                                         \
            default:                                                                                      \
                return cudaErrorInvalidValue;                                                             \
        }                                                                                                 \
    }

}  // namespace nsfrb
