// Internal host-side interface between the C ABI (tq_api.cu) and the kernel files.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "tq.h"

namespace tq {

// Layer groups (Section 5 quantizes groups of layers independently): every worker's row is cut into the same
// n segments, and a (worker, segment) pair is handled like a worker of its own ("job" = worker * n + segment).
// n = 0: no segments, a job is a worker and its row is the whole slice.
struct SegTable {
    uint32_t n;
    uint32_t pad;
    uint64_t off[TQ_MAX_SEGMENTS];    // first element of the segment in the row
    uint64_t len[TQ_MAX_SEGMENTS];    // elements
    uint64_t woff[TQ_MAX_SEGMENTS];   // first word of the segment's packed bits in the worker's packed row
};

// All jobs' tiles, numbered worker after worker and segment after segment, cut into one contiguous range per block.
// A block's share of one job is a "piece"; a range that crosses a job's end consists of several.  Block b and job j
// have at most one piece, and b + j is different for every piece.
//
// Why ranges and not a grid row per job: jobs differ in length (layer groups by a factor of 75 and more) and rarely
// divide the resident blocks evenly; a range is within one tile of every other.  Measured on
// 25.6 M x 16 cut into 16 groups of unequal size: statistics 1142 -> 274 us, compress 1076 -> 402 us.
struct TilePlan {
    uint64_t per_worker;          // tiles of one worker's row
    uint64_t per_block;           // block b starts at tile floor(b * total / blocks) = b * per_block + floor(b * rest / blocks)
    uint32_t rest, blocks;
    double rows_per_tile, blocks_per_tile;   // 1 / per_worker, blocks / total: estimates of quotients, corrected by the user
    SegTable segs;                // without segments: one that covers the row
    uint64_t begin[TQ_MAX_SEGMENTS + 1];   // first tile of each segment within the worker's tiles
};
// segs may be null: one segment of d elements per worker.  At least one tile per job, at most `resident` blocks.
// Equal rows get a whole number of blocks each where that leaves at most 1/24 of the resident blocks out: a block with two
// pieces pays the end of a piece twice, and all wait for it (11.2 M x 8: statistics 75.7 us with, 73 us without such blocks).
// Where the start of a job costs as much as `start_tiles` tiles, each job has that many more, in front: ranges are then even in what they cost, and
// the caller takes them off a piece's tiles again.
inline void plan_tiles(TilePlan* plan, const SegTable* segs, uint64_t d, uint32_t n_workers, uint64_t tile_elems, uint64_t resident, uint64_t start_tiles = 0) {
    if (segs) plan->segs = *segs;
    else { plan->segs.n = 1; plan->segs.off[0] = 0; plan->segs.len[0] = d; plan->segs.woff[0] = 0; }
    uint64_t tiles = 0;
    for (uint32_t s = 0; s < plan->segs.n; ++s) {
        plan->begin[s] = tiles;
        const uint64_t t = (plan->segs.len[s] + tile_elems - 1) / tile_elems;
        tiles += (t ? t : 1) + start_tiles;
    }
    plan->begin[plan->segs.n] = tiles;
    plan->per_worker = tiles;
    const uint64_t total = tiles * n_workers;
    uint64_t blocks = total < resident ? total : resident;
    const uint64_t even = blocks / n_workers * n_workers;
    if (plan->segs.n == 1 && even > 0 && (blocks - even) * 24 <= blocks) blocks = even;
    plan->blocks = static_cast<uint32_t>(blocks);
    plan->per_block = total / blocks;
    plan->rest = static_cast<uint32_t>(total % blocks);
    plan->rows_per_tile = 1.0 / static_cast<double>(tiles);
    plan->blocks_per_tile = static_cast<double>(blocks) / static_cast<double>(total);
}

// SMs of the current device.
inline int sm_count() {
    static std::atomic<int> known[64];           // per device, 0: not asked yet
    int dev = 0, sms = 148;
    if (cudaGetDevice(&dev) != cudaSuccess) return sms;
    if (dev >= 0 && dev < 64 && (sms = known[dev].load(std::memory_order_relaxed)) > 0) return sms;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 148;
    if (dev >= 0 && dev < 64) known[dev].store(sms, std::memory_order_relaxed);
    return sms;
}

// Every kernel is launched through this: it may be set up (blocks placed, barriers initialised, tables built from kernel
// parameters) while the kernel before it on the stream is still running, and waits for that one's results at its
// pdl_wait().  Without it each launch of a round's chain begins about 1 us after the end of the one before it.
//
// A grid that does not fill the GPU is better placed late where its blocks have much to do: blocks that come early are put
// where the kernel before has left room, as many as fit on one SM while others get none, and stay there (aggregation of
// 250 k x 64 behind its compression: 63.1 us a round with an early start, 49.6 without).
enum class Start { kEarly, kLate };
template <class T> struct Same { using type = T; };
template <class... P>
inline cudaError_t launch_kernel(Start start, void (*kernel)(P...), dim3 grid, unsigned threads, size_t smem, cudaStream_t stream,
                                 const typename Same<P>::type&... args) {
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid; cfg.blockDim = dim3(threads); cfg.dynamicSmemBytes = smem; cfg.stream = stream; cfg.attrs = &attr; cfg.numAttrs = start == Start::kEarly ? 1 : 0;
    void* ptrs[] = {const_cast<void*>(static_cast<const void*>(&args))...};
    return cudaLaunchKernelExC(&cfg, reinterpret_cast<const void*>(kernel), ptrs);
}
template <class... P>
inline cudaError_t launch_kernel(void (*kernel)(P...), dim3 grid, unsigned threads, size_t smem, cudaStream_t stream,
                                 const typename Same<P>::type&... args) {
    return launch_kernel(Start::kEarly, kernel, grid, threads, smem, stream, args...);
}

struct CompressCall {
    const void* grad; bool bf16; uint64_t d, grad_stride; uint32_t n_workers;
    const tq_params_t* params;       // host array, or
    const tq_params_t* params_dev;   // device array (then bits / nonuniform come from the caller)
    uint32_t bits; bool nonuniform;
    uint64_t seed; uint32_t first_worker;
    uint32_t* packed; uint64_t words_stride, words_out;
    cudaStream_t stream;
    const SegTable* segs = nullptr;  // device parameters only: params_dev[n_workers * segs->n]; d and words_out are then unused
    int* launches = nullptr;         // device parameters only: receives the number of kernels launched
};
cudaError_t launch_compress(const CompressCall& c);
// bf16 rows through the per-bit-pattern decision table; *applied is false (and nothing is launched) when the
// table form does not fit the call, which then takes the element-wise kernels.
cudaError_t launch_compress_lut(const CompressCall& c, bool* applied);

struct DecompressCall {
    const uint32_t* packed; uint64_t words_stride, words_valid; uint32_t n_workers; uint64_t d;
    const tq_params_t* params;       // host array, or
    const tq_params_t* params_dev;   // device array (then bits comes from the caller)
    const float* weights; uint32_t bits;
    float* out; cudaStream_t stream;
    float* theta = nullptr; float* momentum_buf = nullptr; float lr = 0.0f, mu = 0.0f, wd = 0.0f;   // fused model update
    const uint32_t* const* rows = nullptr;   // host array of n_workers row pointers; when set, packed / words_stride are unused
    const SegTable* segs = nullptr;          // device parameters only: params_dev[n_workers * segs->n]; d and words_valid are then unused
};
cudaError_t launch_decompress(const DecompressCall& c);
cudaError_t read_wait_expired(unsigned int* count);           // give-ups of bounded barrier waits on the current device

struct StatsCall {
    const void* grad; bool bf16; uint64_t d, grad_stride; uint32_t n_workers;
    float g_min, kappa; tq_stats_t* stats; void* workspace; cudaStream_t stream;
    const SegTable* segs = nullptr;          // stats[n_workers * segs->n], workspace for that many jobs; d is then unused
};
// Enqueues the reduction; *launches receives the number of kernels launched.
cudaError_t launch_stats(const StatsCall& c, int* launches);
size_t stats_workspace_bytes(uint32_t n_workers);
// One-pass reduction with a power-of-two threshold and a caller-kept hint, plus the tail pass that
// runs only when the hint missed (two launches, the second usually returning at once).
cudaError_t launch_stats_hinted(const StatsCall& c, tq_gmin_hint_t* hint, int* launches);
// Same reduction with the library's built-in scratch array as workspace (c.workspace is ignored).
// *limit is set when n_workers exceeds what the array holds; nothing is launched then.
cudaError_t launch_stats_static(const StatsCall& c, int* launches, bool* limit);

// Parameter design on the device (one warp per worker); request already validated by params_request_ok.
bool params_request_ok(uint32_t num_levels, int mode, int rule, uint32_t* bits);
cudaError_t launch_params_device(const tq_stats_t* stats_dev, uint32_t n, uint32_t num_levels, uint32_t bits, uint32_t mode,
                                 double gamma, int rule, double alpha_user, tq_params_t* params_dev, cudaStream_t stream);

}  // namespace tq
