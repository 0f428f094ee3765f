// Mid-window search kernels for FP32 rows, and the choice among the mid-window tiles.
#include "search_mid.cuh"

namespace nsfrb {

NSFRB_INSTANTIATE_MID(0)
cudaError_t launch_search_mid_s1(const SearchParams &, int, size_t, cudaStream_t);
cudaError_t launch_search_mid_s2(const SearchParams &, int, size_t, cudaStream_t);

bool choose_mid(SearchParams &p, int max_smem, size_t &smem) {
    if (p.n_t <= kShortT || p.full_snr || p.noise_mode != 0 || p.t_wrap || p.t_stride || p.t_off || p.t_off_dev ||
        p.new_blk || p.row_len != p.n_t || p.n_u_active < 1)
        return false;
    int C = 0, S = 0;
#define NSFRB_MID_PICK(CC, SS)            \
    if (C == 0 && CC * SS > p.n_t) {      \
        C = CC;                           \
        S = SS;                           \
    }
    NSFRB_MID_TILES(NSFRB_MID_PICK)
#undef NSFRB_MID_PICK
    if (C == 0) return false;
    // Warps per CTA (row groups, the first row of each built from all subbands): those that keep the most
    // warps on the SM (its 228 KB of shared memory, 1 KB of it per CTA; 12 warps of 168 registers or 16
    // of 128), the fewest groups on ties.
    const int most = C > 26 ? 12 : 16;
    int best = 0, best_w = 0;
    size_t best_smem = 0;
    for (const int w : {2, 3, 4, 6, 8}) {
        if (w > p.n_u_active && w > 2) break;
        if (32 * w > (C > 26 ? 192 : 256)) break;
        const size_t sm = dev::mid_layout(p, C, S, w).total;
        if (sm > static_cast<size_t>(max_smem)) break;
        const int ctas = std::min(static_cast<int>((228u * 1024u) / (sm + 1024u)), most / w);
        if (ctas * w > best) {
            best = ctas * w;
            best_w = w;
            best_smem = sm;
        }
    }
    // FP32 pixels so large that few warps stay resident are left to the barrier-free kernel where its buffers hold more
    // of them (24 subbands, 9000 pixels: 520 samples 52 rows 671 us against 471; from 544 samples on they
    // do not: 32 subbands, 600 samples 544 us against 2118)
    if (best == 0 || (best < 8 && p.dtype == NSFRB_F32 && p.n_t > 415 && p.n_t <= 543 && p.n_t % 4 == 0 &&
                      reinterpret_cast<uintptr_t>(p.cube) % 16 == 0))
        return false;
    p.pipe = 0;
    p.mid_c = C;
    p.mid_s = S;
    p.mid_w = best_w;
    smem = best_smem;
    // one bulk copy per pixel where its bytes and address allow it, else plain loads
    const size_t pix_bytes = static_cast<size_t>(p.n_sub) * p.n_t * (p.dtype == NSFRB_F32 ? 4 : 2);
    p.stage = (reinterpret_cast<uintptr_t>(p.cube) % 16 == 0 && pix_bytes % 16 == 0) ? 1 : 0;
    // power-of-two widths have their own code at every size here
    p.n_gen = p.has_large = 0;
    for (int j = 0; j < kPow2; ++j) p.pow2_wi[j] = -1;
    for (int i = 0; i < p.n_w; ++i) {
        int j = -1;
        for (int b = 0; b < kPow2; ++b)
            if (p.widths[i] == (1 << b)) j = b;
        if (j >= 0) {
            p.pow2_wi[j] = i;
            p.has_large |= p.widths[i] > kSmallMax;
        } else {
            p.gen_wi[p.n_gen++] = i;
        }
    }
    return true;
}

cudaError_t launch_search_mid(const SearchParams &p, int grid, size_t smem, cudaStream_t s) {
    if (p.n_items <= 0) return cudaSuccess;
    if (p.dtype == NSFRB_F32) return launch_search_mid_s0(p, grid, smem, s);
    return p.dtype == NSFRB_BF16 ? launch_search_mid_s1(p, grid, smem, s) : launch_search_mid_s2(p, grid, smem, s);
}

}  // namespace nsfrb
