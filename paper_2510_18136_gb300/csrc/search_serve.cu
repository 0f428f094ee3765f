// Serving search kernels, and the choice of their shape.
#include "search_serve.cuh"

namespace nsfrb {

NSFRB_INSTANTIATE_SERVE(0)
NSFRB_INSTANTIATE_SERVE(1)
NSFRB_INSTANTIATE_SERVE(2)

bool choose_serve(SearchParams &p, int max_smem, size_t &smem) {
    if (p.new_blk < 1 || p.new_blk > 32 || p.n_t > 1215 || p.full_snr || p.noise_mode != 0 || p.t_wrap || p.t_stride ||
        p.pix_list || p.n_items_dev || p.bad_pix || p.n_u_active < 1)
        return false;
    // blocks of nearly 32 samples have almost every row built from the whole window, and on few pixels that takes longer
    // than the masked search's rows (64 pixels of 400 FP32 samples, blocks of 32, 70 rows: 54 us against 43)
    if (p.new_blk > 28 && p.n_pix <= kSms) return false;
    // rows are copied from the 16-byte boundary below the window, which may start anywhere below n_t
    const int epv = p.dtype == NSFRB_F32 ? 4 : 8;
    if (reinterpret_cast<uintptr_t>(p.cube) % 16 != 0 || p.row_len % epv != 0 || !p.t_off_dev ||
        p.row_len < 2 * static_cast<int64_t>(p.n_t) + 8)
        return false;
    const int C = p.n_t < 704 ? 22 : 38;
    const int shapes[] = {44, 43, 35, 26};   // the most pixels, then the most warps that fit
    for (const int t : shapes) {
        const size_t sm = dev::serve_layout(p, C, t / 10, t % 10).total;
        if (sm > static_cast<size_t>(max_smem)) continue;
        p.pipe = 0;
        p.stage = 1;
        p.serve = 1;
        p.mid_c = C;
        p.teams = t / 10;
        p.mid_s = t % 10;
        smem = sm;
        return true;
    }
    return false;
}

cudaError_t launch_search_serve(const SearchParams &p, int grid, size_t smem, cudaStream_t s) {
    if (p.dtype == NSFRB_F32) return launch_search_serve_s0(p, grid, smem, s);
    return p.dtype == NSFRB_BF16 ? launch_search_serve_s1(p, grid, smem, s) : launch_search_serve_s2(p, grid, smem, s);
}

}  // namespace nsfrb
