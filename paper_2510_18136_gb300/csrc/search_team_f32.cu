// Team search kernels for FP32 rows, and the choice of their shape.
#include "search_team.cuh"

namespace nsfrb {

NSFRB_INSTANTIATE_TEAM(0)
cudaError_t launch_search_team_s1(const SearchParams &, int, size_t, cudaStream_t);
cudaError_t launch_search_team_s2(const SearchParams &, int, size_t, cudaStream_t);

bool choose_team(SearchParams &p, int max_smem, size_t &smem) {
    if (p.n_t <= 607 || p.n_t > 1215 || p.full_snr || p.noise_mode != 0 || p.t_wrap || p.t_stride || p.t_off ||
        p.t_off_dev || p.new_blk || p.row_len != p.n_t || p.n_u_active < 1)
        return false;
    const size_t pix_bytes = static_cast<size_t>(p.n_sub) * p.n_t * (p.dtype == NSFRB_F32 ? 4 : 2);
    if (reinterpret_cast<uintptr_t>(p.cube) % 16 != 0 || pix_bytes % 16 != 0) return false;
    int C = 0;
#define NSFRB_TEAM_PICK(CC) \
    if (C == 0 && 32 * CC > p.n_t) C = CC;
    NSFRB_TEAM_CHUNKS(NSFRB_TEAM_PICK)
#undef NSFRB_TEAM_PICK
    // The most pixels in shared memory first, then the most warps.  6080 pixels, 4 to 24 subbands, 608 to 1200 samples:
    // sixteen warps in four teams against four teams of three 0.94 of the time at 608 samples (16 subbands, 40 rows:
    // 202 us against 214; 10 subbands 167, 176), 0.97 at 1000 (273, 283), and 1.1 with very few rows (4 subbands, 5
    // rows, 1200 samples: 66, 60); three teams of five or two of eight against two of six 0.80 with seven rows
    // (20 subbands, 700 FP32 samples: 113 us, 145), 0.93 with 52 (294, 315), but 1.06 for 12 subbands of 1200 (336,
    // 316).  Over all of them this order is 1 to 2 % faster than leaving out any of the shapes.
    const int shapes[] = {44, 43, 35, 28, 26};
    for (const int t : shapes) {
        const size_t sm = dev::team_layout(p, C, t / 10, t % 10).total;
        if (sm > static_cast<size_t>(max_smem)) continue;
        p.pipe = 0;
        p.stage = 1;
        p.team = 1;
        p.mid_c = C;
        p.teams = t / 10;
        p.mid_s = t % 10;
        smem = sm;
        return true;
    }
    return false;
}

cudaError_t launch_search_team(const SearchParams &p, int grid, size_t smem, cudaStream_t s) {
    if (p.dtype == NSFRB_F32) return launch_search_team_s0(p, grid, smem, s);
    return p.dtype == NSFRB_BF16 ? launch_search_team_s1(p, grid, smem, s) : launch_search_team_s2(p, grid, smem, s);
}

}  // namespace nsfrb
