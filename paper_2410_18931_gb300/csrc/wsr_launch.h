// Host-side launch interface between the C ABI (api.cu) and the kernels.
#pragma once

#include <atomic>

#include <cuda_runtime.h>

#include "wsr_common.cuh"

namespace wsr {

// What a launcher asks the runtime for once per kernel and device: a number that does not change afterwards (SMs,
// resident blocks), kept per device (0: not asked yet; two threads may both ask and store the same).
struct PerDevice {
    std::atomic<int> value[64] = {};
    template <typename F>
    cudaError_t get(int& out, F&& ask) {
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        if (dev < 0 || dev >= 64) return ask(dev, out);
        out = value[dev].load(std::memory_order_relaxed);
        if (out == 0) {
            e = ask(dev, out);
            if (e == cudaSuccess) value[dev].store(out, std::memory_order_relaxed);
        }
        return e;
    }
};

// SMs of the current device.
cudaError_t sm_count(int& sms);

struct GaussPtrs {
    long long n;
    int deg;       // 0..3
    int vd;        // opacity from SH (Eq. 11) instead of a logit
    int red;       // reduced-precision storage (bf16 scales/quats, f16 SH/opacity)
    const float* means;
    const void* log_scales;
    const void* quats;
    const void* sh;
    const void* opacity;
    const float* lc_v;
};

struct WeightDev {
    int kind;
    const float* params;   // device [6]: sigma, beta, w_B, c_B
};

cudaError_t launch_project(const GaussPtrs& g, const Views& vs, WeightDev w, float* records,
                           cudaStream_t s);
// det_sb: nullptr, or (deterministic mode) room for kDetBlocks pairs of sigma/beta block sums; the
// records are then WSR_GRAD_RECORD_FLOATS_DET floats of fixed-point sums and their scales
cudaError_t launch_project_bwd(const GaussPtrs& g, const Views& vs, WeightDev w,
                               const float* grad_records, const wsr_grads& out, float* det_sb, cudaStream_t s);

// Binning with per-block counters in shared memory (k_bin_local): views of up to kLocalTiles tiles; up to
// kLocalTilesTwo, two blocks of 768 threads fit on an SM, beyond that one of 1024.  The grid is the same
// whatever the device, since the workspace holds a row of counters per block.
constexpr int kLocalTilesTwo = 12288;
constexpr int kLocalTiles = 40960;
constexpr int kLocalSMs = 152;
// Its scatter fills a run of a tile's segment per block, so every run's line stays open for the whole pass: past the
// size of L2 it loses to the scatter with global counters.  At two blocks per SM that is a list of 2^25 entries.  At
// one the runs count too, a third of their 32-byte sectors beside the list: both take as long at 27M entries in 14400
// tiles and at 20M to 22M in 32400 (the rule: 26.8M and 20.4M).  Whole binning, us, these counters and the global
// ones: 1920x1080 410 and 509 for 25M, 661 and 649 for 33M, 645 and 524 for 38M; 2560x1440 268 and 331 for 20M, 587
// and 488 for 33M; 3840x2160 120 and 156 for 10M, 270 and 264 for 20M, 377 and 329 for 25M, 678 and 435 for 33M (2^25
// entries whatever the tiles: 657, 447 with global counters in both passes).  The list's length is not known when the
// launch is made: its capacity is taken as a quarter above it there, as callers leave it room to grow.
constexpr unsigned long long kLocalList = 1ull << 25;
inline bool scatter_local(int t_max, unsigned long long capacity) {
    if (t_max <= kLocalTilesTwo) return capacity <= kLocalList;
    const unsigned long long l2 = 134000000ull, runs = 32ull * kLocalSMs * (unsigned)t_max;
    return capacity <= kLocalList && capacity / 5 * 16 <= l2 - runs / 3;
}

// Blocks per view of k_bin_local for views of at most t_max tiles (0: not used)
inline int bin_blocks_per_view(int n_views, int t_max) {
    if (t_max > kLocalTiles) return 0;
    const int all = t_max <= kLocalTilesTwo ? 2 * kLocalSMs : kLocalSMs;
    return all / n_views > 1 ? all / n_views : 1;
}

// A small scene's whole binning in one launch (k_bin_one): beyond these sizes its eight blocks take longer than the
// launches they save.  Clear, count, scan and scatter -> one kernel, us, over all views together: 17.8 -> 8.5 at 1000
// Gaussians and 104 tiles, 18.4 -> 12.5 at 8000 and 104, 21.3 -> 18.5 at 8000 and 920, 18.6 -> 20.6 at 16000 and 920;
// 31.1 -> 26.0 at 3000 and 3600, 30.8 -> 33.0 at 8000 and 3600; 42.0 -> 39.1 at 1000 and 8160 (not taken).
constexpr int kOneBlocks = 8;               // blocks of its cluster, the largest portable one
inline bool bin_in_one(long long n, int n_views, int total_tiles) {
    return total_tiles <= WSR_BIN_ONE_TILES &&
           n * n_views <= (total_tiles <= 1024 ? WSR_BIN_ONE_GAUSSIANS : WSR_BIN_ONE_GAUSSIANS / 2);
}
cudaError_t launch_bin_one(const float* records, long long n, const Views& vs, unsigned* offsets, unsigned* tile_list,
                           unsigned long long capacity, WsHeader* hdr, unsigned* order, cudaStream_t s);

// base: nullptr (global counters only), or total_tiles x bin_blocks_per_view words that carry each block's
// places from the count to the scatter (pass the same base and capacity to both; a count that no scatter follows
// passes the largest capacity)
cudaError_t launch_bin_count(const float* records, long long n, const Views& vs, unsigned* cursor, unsigned* base,
                             unsigned long long capacity, cudaStream_t s);
// the scan of the per-tile counts into offsets (and the scatter's cursors); with `order`, also
// the persistent schedule's longest-first tile order (`buckets`: 66 words of scratch)
cudaError_t launch_scan(const Views& vs, unsigned* cursor, unsigned* block_sums,
                        unsigned* tile_offsets, unsigned long long capacity, WsHeader* hdr,
                        unsigned* buckets, unsigned* order, cudaStream_t s);
cudaError_t launch_bin_scatter(const float* records, long long n, const Views& vs,
                               unsigned* cursor, unsigned* base, unsigned* tile_list,
                               unsigned long long capacity, WsHeader* hdr, cudaStream_t s);

// deterministic mode: each tile's list sorted by record index
cudaError_t launch_sort_segments(const Views& vs, const unsigned* tile_offsets, unsigned* tile_list,
                                 WsHeader* hdr, cudaStream_t s);

// Views of at most this many tiles (four per SM) leave SMs idle with a block per tile: the forward then splits each
// tile's list in two, and the backward takes smaller chunks.  (It needs no order up to WSR_ORDER_MIN_TILES: few blocks
// take a second tile, and idle ones look at every tile's parts.  640 tiles of 10000 Gaussians 31 -> 20 us, of which
// the order was 4.)
constexpr int kFewTiles = 608;

// Work distribution of a forward launch: order == nullptr means one block per
// tile; otherwise a persistent grid takes tiles order[0..total) via *counter
// (reset by the launcher).
struct Sched {
    const unsigned* order;
    unsigned* counter;
};

cudaError_t launch_render_fwd(const float* records, long long n, const unsigned* tile_offsets,
                              const unsigned* tile_list, const Views& vs, WeightDev w,
                              float* out_rgb, float* out_den, Sched sched, cudaStream_t s);

// The longest-first tile order of a binning's offsets (`buckets`: 66 words, zero).
cudaError_t launch_tile_order(const Views& vs, const unsigned* tile_offsets, unsigned* buckets, unsigned* order,
                              cudaStream_t s);

// Work distribution of a backward launch: the tile order (nullptr: as numbered), and total_tiles + 1 words, zero: the
// counter of tiles taken past the blocks' first ones, then each tile's counter of parts taken.
struct BwdSched {
    const unsigned* order;
    unsigned* counter;
};

// Float atomics into WSR_GRAD_RECORD_FLOATS records and grad_wparams; or (det, the deterministic mode,
// WSR_GRAD_RECORD_FLOATS_DET records) the record terms added as fixed point in units set by a per-Gaussian bound from
// *det_pmax (launch_det_pmax first), each tile's background terms stored in bg_tiles[4 tile + c].
cudaError_t launch_render_bwd(const float* records, const unsigned* tile_offsets,
                              const unsigned* tile_list, const Views& vs, WeightDev w,
                              const float* out_rgb, const float* out_den, const float* grad_rgb,
                              float* grad_records, float* grad_wparams, bool det, float* bg_tiles,
                              const unsigned* det_pmax, const BwdSched& sched, cudaStream_t s);
// deterministic mode: grad_wparams[2..5] = the tiles' background terms summed in tile order
cudaError_t launch_det_pmax(const float* out_rgb, const float* out_den, const float* grad_rgb, long long npix,
                            unsigned* pmax, cudaStream_t s);
cudaError_t launch_det_bg_reduce(const float* bg_tiles, int n_tiles, float* grad_wparams, cudaStream_t s);

cudaError_t launch_count_pairs(const float* records, long long n, const unsigned* tile_offsets, const unsigned* tile_list,
                               const Views& vs, unsigned long long* count, cudaStream_t s);

cudaError_t launch_loss_l1(const float* rgb, const float* target, long long count,
                           float* loss, float* grad, cudaStream_t s);

// Views of the 3DGS loss: strips (tiles_x of them) and segments of `rows` rows
// per view, in view order (loss_plan); the Gaussian window taps g[] are normalised
// to sum 1.
struct LossViews {
    int n;
    int rows;
    int tile_off[WSR_MAX_VIEWS + 1];
    int tiles_x[WSR_MAX_VIEWS];
    int w[WSR_MAX_VIEWS];
    int h[WSR_MAX_VIEWS];
    long long pix_off[WSR_MAX_VIEWS];
    float g[11];
    float lam, inv_count, c1, c2;
};

bool loss_plan(LossViews& L);
cudaError_t launch_loss_3dgs(const float* rgb, const float* target, const LossViews& L, float* loss,
                             float* grad, cudaStream_t s);

// Adam groups in float4 units: group k covers units [ubase[k], ubase[k+1])
// and elements [off[k], off[k] + cnt[k]) of the flat buffers.
struct AdamGroups {
    int n;
    long long ubase[WSR_ADAM_MAX_GROUPS + 1];
    long long off[WSR_ADAM_MAX_GROUPS];
    unsigned cnt[WSR_ADAM_MAX_GROUPS];
    float lr[WSR_ADAM_MAX_GROUPS];
    float lr_tail[WSR_ADAM_MAX_GROUPS];
    int period[WSR_ADAM_MAX_GROUPS];
    int head[WSR_ADAM_MAX_GROUPS];
    float b1, omb1, b2, omb2, eps;
};

// Device-resident Adam state (the wsr_adam_state of the C ABI).
struct AdamState {
    int step;
    float c1;      // 1 / (1 - beta1^step)
    float c2;      // 1 / sqrt(1 - beta2^step)
    int skipped;
};
static_assert(sizeof(AdamState) == sizeof(wsr_adam_state), "Adam state layout");

cudaError_t launch_adam(float* p, const float* g, float* m, float* v, const AdamGroups& G, double beta1,
                        double beta2, AdamState* st, const WsHeader* guard, cudaStream_t s);

}  // namespace wsr
