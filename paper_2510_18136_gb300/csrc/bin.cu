// Time binning for the longer search timescales of arXiv 2510.18136 Sec. 2.2
// (0.67 s = 5 samples and 10.05 s = 75 samples of 134 ms): each (pixel,
// subband) row of n_t samples becomes n_t / factor sums of `factor`
// consecutive samples (a trailing remainder is dropped).  FP32 output.
//
// Bound by HBM: every sample is read once.  bin_tile_kernel streams tiles of whole rows through a ring of
// shared-memory stages by bulk copies and sums from there; bin_kernel reads global memory in place
// and takes small factors and what the copies cannot (a cube off a 16-byte boundary, rows too long for
// a stage).  In place, the 32 lanes of a load of the 75-fold sums touch 32 lines, and L1 rather than
// HBM sets the rate: 301 x 301 x 16 rows of 1200 FP32 samples take 2301 us in place and 1066 us
// through the tiles (6.6 TB/s); BF16 1962 and 700 us.
#include <algorithm>
#include <numeric>

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "async_copy.cuh"
#include "nsfrb_debug.h"
#include "plan_internal.h"

namespace nsfrb {
namespace {

template <typename T>
__device__ __forceinline__ float widen(T v);
template <>
__device__ __forceinline__ float widen<float>(float v) { return v; }
template <>
__device__ __forceinline__ float widen<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }
template <>
__device__ __forceinline__ float widen<__half>(__half v) { return __half2float(v); }

// One thread per output sample; consecutive threads read consecutive input runs.
template <typename T>
__global__ void bin_kernel(const T *__restrict__ in, int64_t n_rows, int n_t, int factor, float *__restrict__ out) {
    const int n_out = n_t / factor;
    const int64_t total = n_rows * n_out;
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < total;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int64_t r = i / n_out;
        const int j = static_cast<int>(i - r * n_out);
        const T *src = in + r * n_t + static_cast<int64_t>(j) * factor;
        float acc = 0.0f;
        for (int q = 0; q < factor; ++q) acc += widen<T>(src[q]);
        out[i] = acc;
    }
}

constexpr int kBinThreads = 256;
constexpr int kBinStages = 5;          // per CTA, two CTAs on an SM
constexpr int kBinStageBytes = 20480;  // at most
constexpr int kBinTileFactor = 32;     // smallest factor

// Tiles of `rows` whole rows (contiguous in memory), tile i to CTA i mod gridDim.  An output's samples are split
// into `parts` runs, one thread each, thread part * outputs + output: a warp's lanes then read runs
// `factor` samples apart, and where that stride shares a power of two with the banks, lane o starts its run
// `rot` samples late (and wraps), so that the lanes spread over all banks.
// Once a copy has not landed within its wait's limit, no other is started: this tile (whose sums are written again) and
// every later one is read in place, and the copies in flight are waited for (bounded) before the CTA leaves.  TEST: the odd
// warps take the wait for this CTA's tile give_up as run out (looked at in the loop of the others it costs 5 %).
template <typename T, bool TEST>
__global__ void __launch_bounds__(kBinThreads, 2)
bin_tile_kernel(const T *__restrict__ in, int64_t n_rows, int n_t, int factor, int rows, int parts,
                float *__restrict__ out, int give_up) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ __align__(8) unsigned long long s_full[kBinStages];
    __shared__ float s_part[kBinThreads];
    const int n_out = n_t / factor;
    const uint32_t tile_bytes = static_cast<uint32_t>(rows) * n_t * sizeof(T);
    const int64_t n_tiles = n_rows / rows;   // whole tiles; the rows left over are read in place
    const int tid = threadIdx.x;
    auto issue = [&](int64_t tile, int st) {
        dev::mbar_expect_tx(&s_full[st], tile_bytes);
        dev::bulk_g2s(smem + static_cast<size_t>(st) * tile_bytes, in + tile * rows * n_t, tile_bytes, &s_full[st]);
    };
    if (tid == 0) {
        for (int st = 0; st < kBinStages; ++st) dev::mbar_init(&s_full[st], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        dev::fence_proxy_async();
        for (int st = 0; st < kBinStages; ++st) {
            const int64_t tile = blockIdx.x + static_cast<int64_t>(st) * gridDim.x;
            if (tile < n_tiles) issue(tile, st);
        }
    }
    __syncthreads();
    // samples per 32-bank sweep of the stride, and the start offset that undoes its conflicts
    constexpr int kSweep = 128 / static_cast<int>(sizeof(T)), kWord = 4 / static_cast<int>(sizeof(T));
    int g = 1;
    while (g < kSweep && factor % (2 * g) == 0) g *= 2;
    const int rot_step = g > kWord ? kSweep / g : 0;   // lanes per sweep
    const int per_pass = kBinThreads / parts;          // outputs a pass of the CTA sums
    const int part = tid / per_pass, slot = tid % per_pass;
    const int lo = (part * factor) / parts, len = ((part + 1) * factor) / parts - lo;
    const int rot = rot_step ? min((slot % 32) / rot_step * kWord, len - 1) : 0;
    auto sum_rows = [&](const T *src, int64_t row0, int n) {
        const int total = n * n_out;
        for (int o0 = 0; o0 < total; o0 += per_pass) {
            const int o = o0 + slot;
            float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
            if (o < total) {
                const int r = o / n_out;
                const T *x = src + static_cast<size_t>(r) * n_t + static_cast<size_t>(o - r * n_out) * factor + lo;
                auto run = [&](int q, int end) {
                    for (; q + 3 < end; q += 4) {
#pragma unroll
                        for (int a = 0; a < 4; ++a) acc[a] += widen<T>(x[q + a]);
                    }
                    for (; q < end; ++q) acc[0] += widen<T>(x[q]);
                };
                run(rot, len);
                run(0, rot);
            }
            const float v = (acc[0] + acc[1]) + (acc[2] + acc[3]);
            if (parts == 1) {
                if (o < total) out[row0 * n_out + o] = v;
            } else {
                s_part[tid] = v;
                __syncthreads();
                if (part == 0 && o < total) {
                    float t = v;
                    for (int q = 1; q < parts; ++q) t += s_part[q * per_pass + slot];
                    out[row0 * n_out + o] = t;
                }
                __syncthreads();
            }
        }
    };
    int st = 0, mine = 0;   // the tile's stage and ordinal among this CTA's
    uint32_t parity = 0;
    int64_t tile = blockIdx.x;
    for (; tile < n_tiles; tile += gridDim.x, ++mine) {
        bool stuck = false;
        if constexpr (TEST) stuck = mine == give_up && (tid & 32);
        if (!stuck) stuck = !dev::mbar_wait(&s_full[st], parity);
        sum_rows(reinterpret_cast<const T *>(smem + static_cast<size_t>(st) * tile_bytes), tile * rows, rows);
        dev::fence_proxy_async();
        if (__syncthreads_or(stuck)) break;   // (the stage has been read)
        const int64_t next = tile + static_cast<int64_t>(kBinStages) * gridDim.x;
        if (tid == 0 && next < n_tiles) issue(next, st);
        if (++st == kBinStages) {
            st = 0;
            parity ^= 1u;
        }
    }
    if (tile < n_tiles && tid == 0)
        // copies of the tiles up to kBinStages - 1 ahead, this one's among them
        for (int o = mine; o < mine + kBinStages; ++o)
            if (blockIdx.x + static_cast<int64_t>(o) * gridDim.x < n_tiles)
                dev::mbar_wait(&s_full[o % kBinStages], static_cast<uint32_t>(o / kBinStages) & 1u);
    // in place: the tiles left after a wait that ran out, and the last CTA the rows that fill no tile
    const int64_t left = n_tiles * rows;
    bool rest = left < n_rows && blockIdx.x == gridDim.x - 1;
    while (tile < n_tiles || rest) {
        const bool whole = tile < n_tiles;
        const int64_t row = whole ? tile * rows : left;
        sum_rows(in + row * n_t, row, whole ? rows : static_cast<int>(n_rows - left));
        if (whole)
            tile += gridDim.x;
        else
            rest = false;
    }
}

template <typename T>
cudaError_t launch_bin(const void *d_in, int64_t n_rows, int n_t, int factor, float *d_out, cudaStream_t s,
                       int give_up) {
    const T *in = static_cast<const T *>(d_in);
    const int64_t total = n_rows * (n_t / factor);
    // rows per tile: whole 16-byte units of contiguous memory, up to a stage
    const int row_bytes = static_cast<int>(std::min<int64_t>(static_cast<int64_t>(sizeof(T)) * n_t, 1 << 20));
    const int unit = 16 / std::gcd(16, row_bytes);
    const int rows = kBinStageBytes / row_bytes / unit * unit;
    // Small factors give a tile thousands of outputs, and their index arithmetic costs more than the loads
    // in place (301 x 301 x 16 x 1200, FP32: factor 5 2207 us by tiles, 1317 in place, factor 8 2910
    // and 1451); from 32 samples on the tiles win (32: 3455 and 4819 us, 64: 2625 and 4048).
    if (factor >= kBinTileFactor && rows >= unit && reinterpret_cast<uintptr_t>(in) % 16 == 0 && n_rows >= rows) {
        int dev_id = 0, n_sm = 0;
        cudaError_t e = cudaGetDevice(&dev_id);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev_id);
        if (e != cudaSuccess) return e;
        const int n_out = n_t / factor, resident = 2 * n_sm;
        const int64_t n_tiles = n_rows / rows;
        int parts = 1;   // threads per output, while they and the samples last
        while (parts < 32 && 2 * parts * rows * n_out <= kBinThreads && factor >= 16 * parts) parts *= 2;
        // In place all the same:
        //  * fewer tiles than resident CTAs and a thread per output: a tile's chain of copy and sums takes longer
        //    than the loads of as many threads over the whole chip (1024 rows of 100 samples by 33, FP32: 6.2 us by
        //    tiles, 4.2 in place; 16384 rows of 64 BF16 samples by 32: 8.3 and 6.2), unless the factor is a
        //    multiple of 64, where a load's lanes fall on the same banks of L1 (16 x 1200 BF16 by 64: 6.2, 10.3);
        //  * many tiles of few outputs that leave a good part of the samples out: they are copied all the
        //    same, and a quarter of the threads sum (65536 rows of 3000 FP32 samples by 1024: 435 us by
        //    tiles, 271 in place; 4096 rows 33 and 78).
        const bool few = parts == 1 && n_tiles < resident && factor % 64 != 0;
        const bool loose = sizeof(T) == 4 && 4 * parts * rows * n_out <= kBinThreads &&
                           4 * (n_t - n_out * factor) > n_t && n_tiles >= 40 * resident;
        if (!few && !loose) {
            const auto kernel = give_up < 0 ? bin_tile_kernel<T, false> : bin_tile_kernel<T, true>;
            // every call's limit: see raise_smem_limit
            e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kBinStages * kBinStageBytes);
            if (e != cudaSuccess) return e;
            const int smem = kBinStages * rows * row_bytes;
            const int grid = static_cast<int>(std::min<int64_t>(n_tiles, resident));
            kernel<<<grid, kBinThreads, smem, s>>>(in, n_rows, n_t, factor, rows, parts, d_out, give_up);
            return cudaGetLastError();
        }
    }
    const int bs = 256;
    const int grid = static_cast<int>(std::min<int64_t>((total + bs - 1) / bs, 152 * 64));
    bin_kernel<T><<<grid, bs, 0, s>>>(in, n_rows, n_t, factor, d_out);
    return cudaGetLastError();
}

nsfrb_status bin_time(const void *d_in, int32_t dtype, int64_t n_rows, int32_t n_t, int32_t factor, float *d_out,
                      void *stream, int give_up) {
    if (!d_in || !d_out || n_rows < 0 || n_t < 1 || factor < 1 || factor > n_t || dtype < NSFRB_F32 ||
        dtype > NSFRB_F16)
        return fail(nullptr, NSFRB_EINVAL, "bad argument");
    if (n_rows * (n_t / factor) == 0) return NSFRB_OK;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const cudaError_t e = dtype == NSFRB_F32    ? launch_bin<float>(d_in, n_rows, n_t, factor, d_out, s, give_up)
                          : dtype == NSFRB_BF16 ? launch_bin<__nv_bfloat16>(d_in, n_rows, n_t, factor, d_out, s, give_up)
                                                : launch_bin<__half>(d_in, n_rows, n_t, factor, d_out, s, give_up);
    return cuda_check(nullptr, e, "bin launch");
}

}  // namespace
}  // namespace nsfrb

using namespace nsfrb;

extern "C" nsfrb_status nsfrb_bin_time(const void *d_in, int32_t dtype, int64_t n_rows, int32_t n_t, int32_t factor,
                                       float *d_out, void *stream) {
    return bin_time(d_in, dtype, n_rows, n_t, factor, d_out, stream, -1);
}

extern "C" nsfrb_status nsfrb_dbg_bin_time(const void *d_in, int32_t dtype, int64_t n_rows, int32_t n_t, int32_t factor,
                                           int32_t give_up, float *d_out, void *stream) {
    return bin_time(d_in, dtype, n_rows, n_t, factor, d_out, stream, give_up);
}
