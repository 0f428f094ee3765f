// Wide-window search kernels for FP32 rows, and the choice among the wide-window tiles.
#include "search_wide.cuh"

namespace nsfrb {

NSFRB_INSTANTIATE_WIDE(0)
cudaError_t launch_search_wide_s1(const SearchParams &, int, size_t, cudaStream_t);
cudaError_t launch_search_wide_s2(const SearchParams &, int, size_t, cudaStream_t);

bool choose_wide(SearchParams &p, int max_smem, size_t &smem) {
    if (p.n_t <= kMaxTRegs || p.full_snr || p.noise_mode != 0 || p.t_wrap || p.t_stride || p.t_off || p.t_off_dev ||
        p.new_blk || p.row_len != p.n_t || p.n_u_active < 1)
        return false;
    // one bulk copy per pixel: whole 16-byte units
    const size_t pix_bytes = static_cast<size_t>(p.n_sub) * p.n_t * (p.dtype == NSFRB_F32 ? 4 : 2);
    if (reinterpret_cast<uintptr_t>(p.cube) % 16 != 0 || pix_bytes % 16 != 0) return false;
    int C = 0, V = 0;
#define NSFRB_WIDE_PICK(CC, VV)              \
    if (C == 0 && 32 * CC * VV > p.n_t) {    \
        C = CC;                              \
        V = VV;                              \
    }
    NSFRB_WIDE_TILES(NSFRB_WIDE_PICK)
#undef NSFRB_WIDE_PICK
    if (C == 0) return false;
    // power-of-two widths have their own code; the others, where shorter than a chunk, need the rounding
    // errors of the chunks' prefixes
    p.n_gen = p.has_large = p.wide_lo = 0;
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
            p.wide_lo |= p.widths[i] < C;
        }
    }
    int nb = 2;
    while (nb > 0 && dev::wide_layout(p, C, V, nb).total > static_cast<size_t>(max_smem)) --nb;
    if (nb == 0) return false;
    p.pipe = 0;
    p.stage = 1;
    p.mid_c = C;
    p.mid_s = V;
    p.wide = 1;
    p.nb = nb;
    smem = dev::wide_layout(p, C, V, nb).total;
    return true;
}

cudaError_t launch_search_wide(const SearchParams &p, int grid, size_t smem, cudaStream_t s) {
    if (p.dtype == NSFRB_F32) return launch_search_wide_s0(p, grid, smem, s);
    return p.dtype == NSFRB_BF16 ? launch_search_wide_s1(p, grid, smem, s) : launch_search_wide_s2(p, grid, smem, s);
}

}  // namespace nsfrb
