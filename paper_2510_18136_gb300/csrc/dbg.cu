// Test hook for the kernels' bounded waits: a kernel waits on an mbarrier that no thread ever
// arrives at, gives up after the limit like every wait in the library, latches the error bit
// and returns; the host reads the bit and reports NSFRB_ETIMEOUT.  Nothing traps or hangs.
#include <cuda_runtime.h>

#include "async_copy.cuh"
#include "nsfrb_debug.h"
#include "nsfrb_internal.h"
#include "plan_internal.h"

namespace nsfrb {
namespace {

__global__ void stalled_wait_kernel(int32_t *err, unsigned long long limit_ns) {
    __shared__ unsigned long long bar;
    if (threadIdx.x == 0) {
        dev::mbar_init(&bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    // phase 0 never completes: nothing arrives
    if (!dev::mbar_wait_for(&bar, 0, limit_ns) && threadIdx.x == 0) atomicOr(err, ERR_WAIT_TIMEOUT);
}

}  // namespace
}  // namespace nsfrb

extern "C" nsfrb_status nsfrb_dbg_wait_timeout(int32_t limit_ms) {
    using namespace nsfrb;
    if (limit_ms < 1 || limit_ms > 5000) return NSFRB_EINVAL;
    int32_t *d_err = nullptr;
    if (cudaMalloc(&d_err, sizeof(int32_t)) != cudaSuccess) return NSFRB_ENOMEM;
    int32_t h_err = 0;
    cudaError_t e = cudaMemset(d_err, 0, sizeof(int32_t));
    if (e == cudaSuccess) {
        stalled_wait_kernel<<<1, 32>>>(d_err, static_cast<unsigned long long>(limit_ms) * 1000000ull);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(&h_err, d_err, sizeof(int32_t), cudaMemcpyDeviceToHost);
    cudaFree(d_err);
    if (e != cudaSuccess) return NSFRB_ECUDA;
    return (h_err & ERR_WAIT_TIMEOUT) ? NSFRB_ETIMEOUT : NSFRB_OK;
}

extern "C" nsfrb_status nsfrb_dbg_plan_by_length(nsfrb_plan_t plan, int32_t on) {
    if (!plan) return NSFRB_EINVAL;
    plan->by_length = on != 0;
    return NSFRB_OK;
}

extern "C" int32_t nsfrb_dbg_search_kernel(nsfrb_plan_t plan, int32_t dtype, int64_t n_items, int32_t offset,
                                           int32_t new_blk, int32_t tile, int32_t tuned) {
    using namespace nsfrb;
    if (!plan || dtype < NSFRB_F32 || dtype > NSFRB_F16 || n_items < 1 || new_blk < 0) return -1;
    const nsfrb_config &c = plan->cfg;
    SearchParams sp;
    base_params(plan, sp);
    // addresses that nothing reads: the choice looks at their alignment and at whether they are there
    static char somewhere[64];
    const uintptr_t base = (reinterpret_cast<uintptr_t>(somewhere) + 15) / 16 * 16;
    sp.cube = reinterpret_cast<const void *>(base + offset);
    sp.dtype = dtype;
    sp.n_items = sp.n_pix = n_items;
    sp.row_len = c.n_t;
    sp.new_blk = new_blk;
    if (new_blk > 0) {   // a ring row, its window start on the device
        sp.row_len = static_cast<int64_t>(align_up(static_cast<size_t>(2 * c.n_t + 8), dtype == NSFRB_F32 ? 4 : 8));
        sp.t_off_dev = reinterpret_cast<const int32_t *>(base);
    }
    if (c.out_mode == NSFRB_OUT_FULL) sp.full_snr = reinterpret_cast<float *>(base);
    if (mad_slabs_apply(plan)) sp.noise_mode = NSFRB_NOISE_KNOWN;
    size_t smem = 0;
    if (!choose_stage_for(plan->C, 227 * 1024, sp, smem, tile, tuned != 0)) return 0;
    if (sp.short_w > 0) return 4;
    if (sp.mid_w > 0) return 5;
    if (sp.wide) return 6;
    if (sp.team) return 7;
    if (sp.serve) return 8;
    if (plan->C == kLongC) return 3;
    return sp.pipe ? 2 : 1;
}

extern "C" nsfrb_status nsfrb_dbg_mad_normalise(const void *d_in, int32_t dtype, int64_t n_rows, int32_t n_t,
                                                float *d_out, uint8_t *d_bad, void *stream) {
    using namespace nsfrb;
    if (!d_in || !d_out || !d_bad || n_rows < 1 || n_t < 1 || n_t > kMaxT || dtype < NSFRB_F32 || dtype > NSFRB_F16)
        return NSFRB_EINVAL;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int dev = 0, n_sm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return NSFRB_ECUDA;
    // rows as pixels of one subband: bad[] is then per row
    if (cudaMemsetAsync(d_bad, 0, static_cast<size_t>(n_rows), s) != cudaSuccess) return NSFRB_ECUDA;
    if (launch_mad_normalise(d_in, dtype, 0, n_rows, 1, n_t, d_out, d_bad, n_sm, s) != cudaSuccess) return NSFRB_ECUDA;
    return NSFRB_OK;
}
