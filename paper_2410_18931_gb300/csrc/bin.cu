// Sort-free tile binning.
//
// 3DGS replicates each Gaussian into every tile its footprint touches and
// then sorts each tile's list by depth (Sec. 4.1, Fig. 2).  Eq. 7 is a sum,
// so the order inside a tile does not matter and the sort goes away; what is
// left is a counting pass, an exclusive scan over tiles and an unordered
// scatter (a counting sort by tile with arbitrary order inside each tile).
//
//   k_bin<false>   count: atomicAdd into every tile the footprint reaches
//   k_scan_*       exclusive scan of the per-tile counts (three phases; one
//                  block, with the persistent schedule's tile order, for up
//                  to kSmallScanTiles tiles)
//   k_bin<true>    scatter: claim a slot per (Gaussian, tile) and store
//   k_bin_one      all of these in one launch, for small scenes
// A tile is listed when a pixel-centre column of it meets the footprint
// q <= 9 within the tile's band of pixel-centre rows (the ellipse's exact
// extent per tile row), not merely when it meets the bounding box.
#include <cooperative_groups.h>

#include <mutex>

#include "wsr_launch.h"

namespace wsr {
namespace {

// Pixel rectangle of a record: pixels whose centre lies within the 3-sigma
// extents, clipped to the image.  Returns false when it misses the image.
__device__ __forceinline__ bool pixel_rect(const float4 r0, const float4 r2, const View& V, int& jx0, int& jx1,
                                           int& jy0, int& jy1) {
    if (!(r2.y >= 0.0f)) return false;          // culled (or NaN)
    if (!(fabsf(r0.x) < 1e30f) || !(fabsf(r0.y) < 1e30f) || !(r2.y < 1e30f) || !(r2.z < 1e30f)) return false;
    // pixel j is inside when |j + 0.5 - mu| <= extent; bounds kept within [-1, W]
    const float fw = (float)V.W, fh = (float)V.H;
    const float xlo = fminf(fmaxf(r0.x - r2.y - 0.5f, -1.0f), fw), xhi = fmaxf(fminf(r0.x + r2.y - 0.5f, fw), -1.0f);
    const float ylo = fminf(fmaxf(r0.y - r2.z - 0.5f, -1.0f), fh), yhi = fmaxf(fminf(r0.y + r2.z - 0.5f, fh), -1.0f);
    jx0 = max((int)ceilf(xlo), 0);
    jx1 = min((int)floorf(xhi), V.W - 1);
    jy0 = max((int)ceilf(ylo), 0);
    jy1 = min((int)floorf(yhi), V.H - 1);
    return jx0 <= jx1 && jy0 <= jy1;
}

// Binning pass.  Each warp takes 32 consecutive Gaussians of one view.  A
// Gaussian's work is cut into segments, one per tile row of its pixel
// rectangle (and, for footprints wider than kPiece tiles, one per kPiece
// tiles of that row); the warp lays its segments end to end and takes them
// 32 at a time, one per lane, so a large footprint is spread over the warp.
//
// A segment needs no per-tile test: the footprint q' <= QM is an ellipse, and
// its part inside the row's band of pixel-centre rows [y_a, y_b] is convex,
// so the tiles of the row it reaches are those whose pixel-centre columns
// meet that part's x-extent [x_l, x_r].  With A' = qw^2 + qd, B' = qs qw,
// C' = qs^2 the right edge of the ellipse at height dy is
//     x(dy) = (-B' dy + sqrt(A' QM - qd C' dy^2)) / A',
// a concave function whose maximum sqrt(QM / qd) lies at dy* = -(qw/qs)
// sqrt(QM / qd); x_r is x at the point of the band nearest dy*, and x_l
// follows by symmetry.  The extent is widened by a margin far above its FP32
// rounding error, so every pixel centre with q' <= QM is kept (a tile the
// ellipse only passes near is listed at worst).
//
// The 32 segments' tile ranges are then laid end to end again and the lanes
// take consecutive tiles, so the atomics of a warp fall on neighbouring
// counters of a few rows.  COUNT: atomicAdd per tile.  SCATTER: claim a slot
// in the tile's segment and write the record index.
constexpr int kPiece = 8;

// A warp's scratch: 32 Gaussians, and the segments of a batch that hold tiles.
struct BinScratch {
    int start[32];        // each Gaussian's first segment (exclusive prefix of segment counts)
    int gown[32];         // the lanes of the Gaussians with segments, in order
    int4 rect[32];        // pixel rectangle: jx0, jx1, jy0, jy1
    float4 geo[32][2];    // mu_x, mu_y, B'/A', A' QM | det', 1/A', dy*, margin
    int2 run[32];         // per segment with tiles, in order: its first tile, less its first position in the
                          // batch, and the owning lane
};

// One warp's 32 Gaussians i0 .. i0 + 31 of view v: emit(tile, owner) for every tile of the view (counted
// from the view's first) that a footprint reaches; owner is the Gaussian's place among the 32.
template <typename F>
__device__ __forceinline__ void bin_batch(const float4* __restrict__ rec, const long long n, const View& V,
                                          const int v, const long long i0, const int lw, const int lh,
                                          BinScratch& sc, F&& emit) {
    const int lane = threadIdx.x & 31;
    const long long i = i0 + lane;
    const float QM = kQMax * 1.0001f + 1e-4f;
    int nseg = 0, jx0 = 0, jx1 = -1, jy0 = 0, jy1 = -1;
    float4 g0 = make_float4(0.f, 0.f, 0.f, 0.f), g1 = g0;
    if (i < n) {
        const long long r = (long long)v * n + i;
        const float4 r0 = __ldg(rec + 3 * r);
        const float qd = __ldg(reinterpret_cast<const float*>(rec + 3 * r + 1));
        const float4 r2 = __ldg(rec + 3 * r + 2);
        if (pixel_rect(r0, r2, V, jx0, jx1, jy0, jy1)) {
            const float qs = r0.z, qw = r0.w;
            // hardware reciprocal and square root (relative error ~2^-22, far below the margin below)
            const float A = fmaf(qw, qw, qd), ia = rcp_approx(A);
            const float dxm = sqrt_approx(QM * rcp_approx(qd));  // half-width of the ellipse
            g0 = make_float4(r0.x, r0.y, qs * qw * ia, A * QM);
            g1 = make_float4(qd * qs * qs, ia, -(qw * rcp_approx(qs)) * dxm, fminf(2e-3f * dxm, 1e6f) + 0.01f);
            const int pcs = ((jx1 >> lw) - (jx0 >> lw) + kPiece) / kPiece;
            nseg = ((jy1 >> lh) - (jy0 >> lh) + 1) * pcs;
        }
    }
    int inc = nseg;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, inc, off);
        if (lane >= off) inc += y;
    }
    const int gex = inc - nseg;                          // this Gaussian's first segment
    // the Gaussians with segments, in lane order: a segment's owner is found by counting starts (below)
    const unsigned gmask = __ballot_sync(0xffffffffu, nseg > 0);
    if (nseg > 0) sc.gown[__popc(gmask & ((1u << lane) - 1u))] = lane;
    sc.start[lane] = gex;
    sc.rect[lane] = make_int4(jx0, jx1, jy0, jy1);
    sc.geo[lane][0] = g0;
    sc.geo[lane][1] = g1;
    __syncwarp();
    const int total = __shfl_sync(0xffffffffu, inc, 31);
    for (int c0 = 0; c0 < total; c0 += 32) {
        // ---- this lane's segment c0 + lane: its owner is the last Gaussian with segments whose first
        // segment is at or before it (those starting before c0, plus the starts in the batch up to it) ----
        const unsigned gst = __reduce_or_sync(0xffffffffu, nseg > 0 && gex >= c0 && gex < c0 + 32 ? 1u << (gex - c0)
                                                                                               : 0u);
        const int gbefore = __popc(__ballot_sync(0xffffffffu, nseg > 0 && gex < c0));
        const int c = c0 + lane;
        int ta = 0, tb = -1, lo = 0, row = 0;
        if (c < total) {
            lo = sc.gown[gbefore + __popc(gst & ((2u << lane) - 1u)) - 1];
            const int k = c - sc.start[lo];                     // segment index within the owner
            const int4 rc = sc.rect[lo];
            const float4 a = sc.geo[lo][0], b = sc.geo[lo][1];
            const int np = ((rc.y >> lw) - (rc.x >> lw) + kPiece) / kPiece;
            const int kr = np == 1 ? k : k / np, kp = k - kr * np;
            const int ty = (rc.z >> lh) + kr;
            // the row's band of pixel-centre rows, inside the footprint's rows
            const float dya = (float)max(ty << lh, rc.z) + 0.5f - a.y;
            const float dyb = (float)min(((ty + 1) << lh) - 1, rc.w) + 0.5f - a.y;
            auto edge = [&](float dy, float side) {
                return fmaf(-a.z, dy, side * sqrt_approx(fmaxf(fmaf(-b.x * dy, dy, a.w), 0.0f)) * b.y);
            };
            const float xr = edge(fminf(fmaxf(b.z, dya), dyb), 1.0f);
            const float xl = edge(fminf(fmaxf(-b.z, dya), dyb), -1.0f);
            // pixel columns whose centre lies in [mu_x + x_l, mu_x + x_r] (widened), clipped to the rectangle
            const float fa = fmaxf(ceilf(a.x + xl - b.w - 0.5f), (float)rc.x);
            const float fb = fminf(floorf(a.x + xr + b.w - 0.5f), (float)rc.y);
            if (fa <= fb) {
                const int p0 = (rc.x >> lw) + kp * kPiece;       // this segment's tiles of the row
                ta = max((int)fa >> lw, p0);
                tb = min((int)fb >> lw, p0 + kPiece - 1);
                row = ty * V.tiles_x;
            }
        }
        // ---- the batch's tiles end to end, consecutive tiles to consecutive lanes; a tile's segment is
        // found the same way, by counting the segments that start at or before it ----
        const int wdt = max(tb - ta + 1, 0);   // a piece the band does not reach has none
        int winc = wdt;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, winc, off);
            if (lane >= off) winc += y;
        }
        const int nt = __shfl_sync(0xffffffffu, winc, 31);
        const int wex = winc - wdt;                      // this segment's first position in the batch
        const unsigned smask = __ballot_sync(0xffffffffu, wdt > 0);
        if (wdt > 0) sc.run[__popc(smask & ((1u << lane) - 1u))] = make_int2(row + ta - wex, lo);
        __syncwarp();
        for (int j0 = 0; j0 < nt; j0 += 32) {
            const unsigned sst = __reduce_or_sync(0xffffffffu, wdt > 0 && wex >= j0 && wex < j0 + 32 ? 1u << (wex - j0)
                                                                                                  : 0u);
            const int sbefore = __popc(__ballot_sync(0xffffffffu, wdt > 0 && wex < j0));
            const int j = j0 + lane;
            if (j < nt) {
                const int2 run = sc.run[sbefore + __popc(sst & ((2u << lane) - 1u)) - 1];
                emit(run.x + j, run.y);
            }
        }
        __syncwarp();
    }
}

// The pass with global counters: one block per 256 Gaussians of a view.
template <bool SCATTER>
__global__ void __launch_bounds__(256) k_bin(const float4* __restrict__ rec, long long n, const Views vs,
                                             unsigned* __restrict__ cursor, unsigned* __restrict__ list,
                                             unsigned long long capacity, WsHeader* hdr) {
    __shared__ BinScratch scratch[8];
    const int v = blockIdx.y;
    const View& V = vs.v[v];
    const int warp = threadIdx.x >> 5;
    const long long i0 = (long long)blockIdx.x * blockDim.x + warp * 32;
    unsigned* const cur = cursor + V.tile_base;
    bin_batch(rec, n, V, v, i0, __ffs(vs.tile_w) - 1, __ffs(vs.tile_h) - 1, scratch[warp], [&](int tile, int owner) {
        if constexpr (SCATTER) {
            const unsigned slot = atomicAdd(cur + tile, 1u);
            if (slot < capacity) list[slot] = (unsigned)((long long)v * n + i0 + owner);
            else set_error(hdr, WSR_ERR_CAPACITY);
        } else {
            atomicAdd(cur + tile, 1u);
        }
    });
}

// The pass with counters in shared memory: a few blocks per SM over all views, each with a counter for
// every tile of its view.  Block b of a view takes the batches of 32 Gaussians b, b + B, ... (its warps
// one after another as they come free) in both passes.  COUNT: the block's counts per tile, then one
// global atomic per tile that it reaches; what that returns, the block's first place among the tile's
// instances, is kept in `base` (a row of T entries per block; nullptr: not asked for).  SCATTER: the block's cursors start
// at the tile's offset plus that place, so a slot costs one shared atomic.
//   The global counters bound the plain pass: neighbouring tiles share 32-byte sectors, and a view's
// counters are only a few kilobytes, so the atomics of all SMs queue at a few L2 lines.  Measured, count,
// scan and scatter: 171 -> 87 us for 1M Gaussians at 1920x1080 (6.3M instances), 392 -> 126 us for 300k
// in six views (6.3M instances, the smallest view 920 tiles), 21 -> 15 us for 10000 at 979x543.  What
// is left is the latency of a warp's chain (records, prefix, segments, tiles) at 48 warps per SM.
template <int NT, bool SCATTER>
__global__ void __launch_bounds__(NT, NT > 768 ? 1 : 2)
    k_bin_local(const float4* __restrict__ rec, long long n, const Views vs, unsigned* __restrict__ cursor,
                unsigned* __restrict__ base, unsigned* __restrict__ list, unsigned long long capacity,
                WsHeader* hdr) {
    extern __shared__ __align__(16) unsigned char s_dyn[];
    __shared__ int s_next;
    BinScratch* const scratch = reinterpret_cast<BinScratch*>(s_dyn);
    unsigned* const cnt = reinterpret_cast<unsigned*>(s_dyn + sizeof(BinScratch) * (NT / 32));
    const int v = blockIdx.y;
    const View& V = vs.v[v];
    const int T = V.tiles_x * V.tiles_y;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int lw = __ffs(vs.tile_w) - 1, lh = __ffs(vs.tile_h) - 1;   // tile sides are powers of two
    cursor += V.tile_base;
    if (base) base += (size_t)V.tile_base * gridDim.x + (size_t)blockIdx.x * T;
    if (threadIdx.x == 0) s_next = 0;
    // (four tiles per thread at a time, so that their loads, or below their atomics, are in flight together)
    for (int t0 = threadIdx.x; t0 < T; t0 += 4 * NT) {
        unsigned c[4] = {0u, 0u, 0u, 0u};
        if constexpr (SCATTER) {
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (t0 + k * NT < T) c[k] = cursor[t0 + k * NT] + base[t0 + k * NT];
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (t0 + k * NT < T) cnt[t0 + k * NT] = c[k];
    }
    __syncthreads();
    const long long nb = (n + 31) >> 5;                               // batches of the view
    for (;;) {
        int k = 0;
        if (lane == 0) k = atomicAdd(&s_next, 1);
        const long long b = blockIdx.x + (long long)__shfl_sync(0xffffffffu, k, 0) * gridDim.x;
        if (b >= nb) break;
        bin_batch(rec, n, V, v, b << 5, lw, lh, scratch[warp], [&](int tile, int owner) {
            const unsigned slot = atomicAdd(cnt + tile, 1u);
            if constexpr (SCATTER) {
                if (slot < capacity) list[slot] = (unsigned)((long long)v * n + (b << 5) + owner);
                else set_error(hdr, WSR_ERR_CAPACITY);
            }
        });
    }
    if constexpr (!SCATTER) {
        __syncthreads();
        if (base == nullptr) {
            for (int t = threadIdx.x; t < T; t += NT)
                if (const unsigned c = cnt[t]) atomicAdd(cursor + t, c);
            return;
        }
        for (int t0 = threadIdx.x; t0 < T; t0 += 4 * NT) {
            unsigned c[4], b[4] = {0u, 0u, 0u, 0u};
#pragma unroll
            for (int k = 0; k < 4; ++k) c[k] = t0 + k * NT < T ? cnt[t0 + k * NT] : 0u;
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (c[k]) b[k] = atomicAdd(cursor + t0 + k * NT, c[k]);
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (c[k]) base[t0 + k * NT] = b[k];
        }
    }
}

// --------------------------------------------------------------------------
// Exclusive scan over tiles: (1) per-block totals, (2) one block scans the
// totals and writes the grand total, (3) per-block scan plus block offset.
// --------------------------------------------------------------------------
__device__ __forceinline__ unsigned long long block_exclusive_scan(unsigned long long x, unsigned long long* s_warp,
                                                                   unsigned long long& total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long inc = x;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, inc, off);
        if (lane >= off) inc += y;
    }
    if (lane == 31) s_warp[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        const int nw = blockDim.x >> 5;
        unsigned long long t = lane < nw ? s_warp[lane] : 0ull;
        unsigned long long ti = t;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xffffffffu, ti, off);
            if (lane >= off) ti += y;
        }
        if (lane < nw) s_warp[lane] = ti - t;
        if (lane == 31) s_warp[32] = ti;
    }
    __syncthreads();
    total = s_warp[32];
    const unsigned long long r = s_warp[warp] + inc - x;
    __syncthreads();
    return r;
}

__global__ void __launch_bounds__(kScanBlock) k_scan_reduce(const unsigned* __restrict__ cnt, int n,
                                                            unsigned long long* __restrict__ bsum) {
    __shared__ unsigned long long s_warp[33];
    const long long base = (long long)blockIdx.x * kScanTile + (long long)threadIdx.x * kScanItems;
    unsigned long long x = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k)
        if (base + k < n) x += cnt[base + k];
    unsigned long long tot;
    block_exclusive_scan(x, s_warp, tot);
    if (threadIdx.x == 0) bsum[blockIdx.x] = tot;
}

__global__ void __launch_bounds__(kScanBlock) k_scan_top(unsigned long long* __restrict__ bsum, int nb,
                                                         unsigned* __restrict__ offsets, int n_tiles,
                                                         unsigned long long capacity, WsHeader* hdr) {
    __shared__ unsigned long long s_warp[33];
    unsigned long long carry = 0;
    for (int base = 0; base < nb; base += kScanBlock) {
        const int j = base + threadIdx.x;
        const unsigned long long x = j < nb ? bsum[j] : 0ull;
        unsigned long long tot;
        const unsigned long long ex = block_exclusive_scan(x, s_warp, tot);
        if (j < nb) bsum[j] = carry + ex;
        carry += tot;
    }
    if (threadIdx.x == 0) {
        // offsets never exceed the list capacity, so the renderers stay in
        // bounds even when the list overflowed; the true total goes to the
        // workspace header for the caller to size a larger list
        const unsigned long long lim = capacity < 0xffffffffull ? capacity : 0xffffffffull;
        offsets[n_tiles] = (unsigned)(carry < lim ? carry : lim);
        hdr->total = carry;
        hdr->err = carry > lim ? WSR_ERR_CAPACITY : 0;      // a binning starts from no error
    }
}

__global__ void __launch_bounds__(kScanBlock) k_scan_apply(unsigned* __restrict__ cursor, int n,
                                                           const unsigned long long* __restrict__ bsum,
                                                           unsigned* __restrict__ offsets,
                                                           unsigned long long capacity) {
    const unsigned long long lim = capacity < 0xffffffffull ? capacity : 0xffffffffull;
    __shared__ unsigned long long s_warp[33];
    const long long base = (long long)blockIdx.x * kScanTile + (long long)threadIdx.x * kScanItems;
    unsigned c[kScanItems];
    unsigned long long x = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        c[k] = (base + k < n) ? cursor[base + k] : 0u;
        x += c[k];
    }
    unsigned long long tot;
    unsigned long long run = bsum[blockIdx.x] + block_exclusive_scan(x, s_warp, tot);
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        if (base + k < n) {
            const unsigned o = (unsigned)(run < lim ? run : lim);
            offsets[base + k] = o;
            cursor[base + k] = o;   // scatter cursor starts at the tile's offset
        }
        run += c[k];
    }
}

// Longest-first tile order for the persistent schedule: tiles are bucketed by
// the magnitude of their instance count (floor(log2)), buckets taken from the
// largest down; the order inside a bucket is arbitrary.
__device__ __forceinline__ int cost_bucket(unsigned c) { return c ? 32 - __clz(c) : 0; }   // 0..32

// Exclusive scan over the tiles and, for the persistent schedule, the longest-first
// tile order (the buckets of k_order_*), in one block: for views of at most
// kSmallScanTiles tiles.  The counts pass through shared memory (dynamic, n + 1
// words) so that every global access is coalesced.  Warp w scans the
// consecutive tiles [w seg, (w + 1) seg), 32 at a time (lane l on tile 32 i + l
// of its range: no bank conflicts), after one block scan of the warps' totals.
constexpr int kSmallScanTiles = WSR_SCAN_ONE_BLOCK_TILES;
static_assert(kSmallScanTiles % kScanBlock == 0, "whole segments");

__global__ void __launch_bounds__(kScanBlock) k_scan_order_small(unsigned* __restrict__ cursor, int n,
                                                                 unsigned* __restrict__ offsets,
                                                                 unsigned long long capacity, WsHeader* hdr,
                                                                 unsigned* __restrict__ order) {
    extern __shared__ unsigned s_off[];         // [n + 1]: the counts, then the offsets
    __shared__ unsigned long long s_warp[33];
    __shared__ unsigned s_hist[33];
    const unsigned long long lim = capacity < 0xffffffffull ? capacity : 0xffffffffull;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int t = threadIdx.x; t < n; t += kScanBlock) s_off[t] = cursor[t];
    if (threadIdx.x < 33) s_hist[threadIdx.x] = 0u;
    __syncthreads();
    const int seg = (n + kScanBlock - 1) / kScanBlock * 32;             // tiles per warp, a multiple of 32
    const int w0 = min(warp * seg, n), w1 = min(w0 + seg, n);
    unsigned long long x = 0;
    for (int t = w0 + lane; t < w1; t += 32) x += s_off[t];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
    unsigned long long tot;
    unsigned long long carry = block_exclusive_scan(lane == 0 ? x : 0ull, s_warp, tot);   // ends with a barrier
    carry = __shfl_sync(0xffffffffu, carry, 0);
    for (int t0 = w0; t0 < w1; t0 += 32) {
        const int t = t0 + lane;
        const unsigned c = t < w1 ? s_off[t] : 0u;
        unsigned long long inc = c;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xffffffffu, inc, off);
            if (lane >= off) inc += y;
        }
        const unsigned long long run = carry + inc - c;
        if (t < w1) s_off[t] = (unsigned)(run < lim ? run : lim);
        carry += __shfl_sync(0xffffffffu, inc, 31);
    }
    if (threadIdx.x == 0) {
        s_off[n] = (unsigned)(tot < lim ? tot : lim);
        hdr->total = tot;
        hdr->err = tot > lim ? WSR_ERR_CAPACITY : 0;        // a binning starts from no error
    }
    __syncthreads();
    for (int t = threadIdx.x; t <= n; t += kScanBlock) {
        const unsigned o = s_off[t];
        offsets[t] = o;
        if (t < n) cursor[t] = o;       // the scatter's cursor starts at the tile's offset
    }
    if (!order) return;
    for (int t = threadIdx.x; t < n; t += kScanBlock) atomicAdd(&s_hist[cost_bucket(s_off[t + 1] - s_off[t])], 1u);
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned r = 0;                 // bucket starts, largest bucket first
        for (int b = 32; b >= 0; --b) {
            const unsigned h = s_hist[b];
            s_hist[b] = r;
            r += h;
        }
    }
    __syncthreads();
    for (int t = threadIdx.x; t < n; t += kScanBlock)
        order[atomicAdd(&s_hist[cost_bucket(s_off[t + 1] - s_off[t])], 1u)] = (unsigned)t;
}

// The same for up to 1024 I tiles, each thread's tiles in registers: warp w scans the tiles [32 I w, 32 I (w + 1))
// as I rows of 32, the rows' shuffles independent of one another, and ranks a tile among its warp's tiles of the
// same bucket by matching lanes, so that neither pass over the tiles queues on a bucket's counter.  It is bound by
// the latency of its chain of loads, shuffles and three barriers: 12 -> 6 us for 8160 tiles with the order.
// With SCAN false it only orders the tiles of given offsets.
struct ScanShared {
    unsigned long long sum[32];
    unsigned hist[32][33];              // per warp and bucket: tiles, then the first place among the bucket's
    unsigned total[33];                 // per bucket: tiles, then the bucket's first place in the order
};

// load(t): a tile's count; SCAN: store(t, o) takes its offset (at most lim), finish(total) the sum, once
template <int I, bool SCAN, typename Load, typename Store, typename Finish>
__device__ __forceinline__ void scan_order_rows(const int n, const unsigned long long lim, unsigned* __restrict__ order,
                                                ScanShared& sh, Load&& load, Store&& store, Finish&& finish) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned below = (1u << lane) - 1u;
    const int t0 = warp * 32 * I + lane;
    unsigned c[I], rank[I];
#pragma unroll
    for (int r = 0; r < I; ++r) {
        const int t = t0 + 32 * r;
        c[r] = t >= n ? 0u : load(t);
    }
    if (order) {
        sh.hist[warp][lane] = 0u;
        if (lane == 0) sh.hist[warp][32] = 0u;
        __syncwarp();
#pragma unroll
        for (int r = 0; r < I; ++r) {
            const int b = t0 + 32 * r < n ? cost_bucket(c[r]) : 33;
            const unsigned same = __match_any_sync(0xffffffffu, b);
            unsigned h = 0u;
            if (b < 33) h = sh.hist[warp][b];
            __syncwarp();
            if (b < 33 && (same & below) == 0u) sh.hist[warp][b] = h + __popc(same);
            __syncwarp();
            rank[r] = h + __popc(same & below);
        }
    }
    if constexpr (SCAN) {
        unsigned long long inc[I], sum = 0;
#pragma unroll
        for (int r = 0; r < I; ++r) inc[r] = c[r];
#pragma unroll
        for (int off = 1; off < 32; off <<= 1)
#pragma unroll
            for (int r = 0; r < I; ++r) {
                const unsigned long long y = __shfl_up_sync(0xffffffffu, inc[r], off);
                if (lane >= off) inc[r] += y;
            }
#pragma unroll
        for (int r = 0; r < I; ++r) {
            const unsigned long long row = __shfl_sync(0xffffffffu, inc[r], 31);
            inc[r] += sum - c[r];                   // exclusive within the warp's tiles
            sum += row;
        }
        if (lane == 0) sh.sum[warp] = sum;
        __syncthreads();
        unsigned long long x = sh.sum[lane], scan = x;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xffffffffu, scan, off);
            if (lane >= off) scan += y;
        }
        const unsigned long long tot = __shfl_sync(0xffffffffu, scan, 31);
        const unsigned long long first = __shfl_sync(0xffffffffu, scan - x, warp);
#pragma unroll
        for (int r = 0; r < I; ++r) {
            const int t = t0 + 32 * r;
            const unsigned long long run = first + inc[r];
            const unsigned o = (unsigned)(run < lim ? run : lim);
            if (t < n) store(t, o);
        }
        if (threadIdx.x == 0) finish(tot);
    } else {
        __syncthreads();
    }
    if (!order) return;
    // warp b takes bucket b (warp 0 also bucket 32), a lane per warp's count; then warp 0 the buckets
    for (int b = warp; b < 33; b += 32) {
        const unsigned h = sh.hist[lane][b];
        unsigned hi = h;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, hi, off);
            if (lane >= off) hi += y;
        }
        sh.hist[lane][b] = hi - h;
        if (lane == 31) sh.total[b] = hi;
    }
    __syncthreads();
    if (warp == 0) {
        const unsigned most = sh.total[32], h = sh.total[lane];   // bucket 32 comes first
        unsigned hi = h;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const unsigned y = __shfl_down_sync(0xffffffffu, hi, off);
            if (lane + off < 32) hi += y;
        }
        sh.total[lane] = most + hi - h;
        if (lane == 0) sh.total[32] = 0u;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < I; ++r) {
        const int t = t0 + 32 * r;
        if (t < n) {
            const int b = cost_bucket(c[r]);
            order[sh.total[b] + sh.hist[warp][b] + rank[r]] = (unsigned)t;
        }
    }
}

template <int I, bool SCAN>
__global__ void __launch_bounds__(kScanBlock) k_scan_order_rows(unsigned* __restrict__ cursor, int n,
                                                                unsigned* __restrict__ offsets,
                                                                unsigned long long capacity, WsHeader* hdr,
                                                                unsigned* __restrict__ order) {
    __shared__ ScanShared sh;
    const unsigned long long lim = capacity < 0xffffffffull ? capacity : 0xffffffffull;
    scan_order_rows<I, SCAN>(
        n, lim, order, sh, [&](int t) { return SCAN ? cursor[t] : offsets[t + 1] - offsets[t]; },
        [&](int t, unsigned o) {
            offsets[t] = o;
            cursor[t] = o;                          // the scatter's cursor starts at the tile's offset
        },
        [&](unsigned long long tot) {
            offsets[n] = (unsigned)(tot < lim ? tot : lim);
            hdr->total = tot;
            hdr->err = tot > lim ? WSR_ERR_CAPACITY : 0;        // a binning starts from no error
        });
}

// Count, scan, order and scatter of a small scene in one launch: a cluster of kOneBlocks blocks, every tile's counter
// in each block's shared memory.  Warp w of block r takes the batches of 32 Gaussians r + kOneBlocks (w + 32 i) of all
// views in both passes; between them each block reads all blocks' counters (distributed shared memory) and scans
// them, so that its cursors start at a tile's offset plus what the blocks before it hold there.  Nothing else than
// the list, the offsets, the header and the order is written.
//   Latency bounds it (launch, records, prefix, segments, tiles, twice): 1000 Gaussians at 128x128, 17.7 us for the
// clear and three kernels -> 8.4; bin_in_one has the limits.
template <int I>
__global__ void __cluster_dims__(kOneBlocks, 1, 1) __launch_bounds__(1024, 1)
    k_bin_one(const float4* __restrict__ rec, long long n, const Views vs, unsigned* __restrict__ offsets,
              unsigned* __restrict__ list, unsigned long long capacity, WsHeader* hdr, unsigned* __restrict__ order) {
    namespace cg = cooperative_groups;
    extern __shared__ __align__(16) unsigned char s_dyn[];
    __shared__ ScanShared sh;
    BinScratch* const scratch = reinterpret_cast<BinScratch*>(s_dyn);
    const int T = vs.total_tiles;
    unsigned* const cnt = reinterpret_cast<unsigned*>(s_dyn + sizeof(BinScratch) * 32);
    unsigned* const cur = cnt + T;
    const cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank(), warp = threadIdx.x >> 5;
    const int lw = __ffs(vs.tile_w) - 1, lh = __ffs(vs.tile_h) - 1;     // tile sides are powers of two
    const unsigned long long lim = capacity < 0xffffffffull ? capacity : 0xffffffffull;
    for (int t = threadIdx.x; t < T; t += 1024) cnt[t] = 0u;
    __syncthreads();
    const long long nb = (n + 31) >> 5;                                 // batches per view
    auto pass = [&](auto&& emit) {
        for (long long b = rank + kOneBlocks * warp; b < nb * vs.n; b += kOneBlocks * 32) {
            const int v = (int)(b / nb);
            const long long i0 = (b - v * nb) << 5;
            const View& V = vs.v[v];
            bin_batch(rec, n, V, v, i0, lw, lh, scratch[warp],
                      [&](int tile, int owner) { emit(V.tile_base + tile, (unsigned)(v * n + i0 + owner)); });
        }
    };
    pass([&](int tile, unsigned) { atomicAdd(cnt + tile, 1u); });
    cluster.sync();
    const unsigned* all[kOneBlocks];
#pragma unroll
    for (int c = 0; c < kOneBlocks; ++c) all[c] = cluster.map_shared_rank(cnt, c);
    scan_order_rows<I, true>(
        T, lim, rank == kOneBlocks - 1 ? order : nullptr, sh,
        [&](int t) {
            unsigned sum = 0u, before = 0u;
#pragma unroll
            for (int c = 0; c < kOneBlocks; ++c) {
                if (c == rank) before = sum;
                sum += all[c][t];
            }
            cur[t] = before;
            return sum;
        },
        [&](int t, unsigned o) {
            cur[t] += o;
            if (rank == 0) offsets[t] = o;
        },
        [&](unsigned long long tot) {
            if (rank != 0) return;
            offsets[T] = (unsigned)(tot < lim ? tot : lim);
            hdr->total = tot;
            hdr->err = tot > lim ? WSR_ERR_CAPACITY : 0;                // a binning starts from no error
        });
    cluster.sync();                 // the cursors stand, every block is done with the others' counters
    pass([&](int tile, unsigned at) {
        const unsigned slot = atomicAdd(cur + tile, 1u);
        if (slot < capacity) list[slot] = at;
        else set_error(hdr, WSR_ERR_CAPACITY);
    });
}

__global__ void __launch_bounds__(256) k_order_hist(const unsigned* __restrict__ offsets, int n,
                                                    unsigned* __restrict__ hist) {
    __shared__ unsigned h[33];
    if (threadIdx.x < 33) h[threadIdx.x] = 0;
    __syncthreads();
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x)
        atomicAdd(&h[cost_bucket(offsets[t + 1] - offsets[t])], 1u);
    __syncthreads();
    if (threadIdx.x < 33 && h[threadIdx.x]) atomicAdd(hist + threadIdx.x, h[threadIdx.x]);
}

// hist[0..32]: tiles per bucket; hist[33..65]: taken of each so far (zero at the start).  A block claims its tiles'
// places of a bucket at once: with an atomic per tile the scatter queued on the buckets' few words (32400 tiles: 24 us
// for the order in three kernels, 4 in two).
__global__ void __launch_bounds__(256) k_order_scatter(const unsigned* __restrict__ offsets, int n,
                                                       unsigned* __restrict__ hist, unsigned* __restrict__ order) {
    __shared__ unsigned s_start[33], s_count[33], s_base[33];
    if (threadIdx.x < 32) {                         // each bucket's start, largest bucket first
        const int lane = threadIdx.x;
        const unsigned most = hist[32], h = hist[lane];
        unsigned hi = h;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const unsigned y = __shfl_down_sync(0xffffffffu, hi, off);
            if (lane + off < 32) hi += y;
        }
        s_start[lane] = most + hi - h;
        if (lane == 0) s_start[32] = 0u;
    }
    for (int t0 = blockIdx.x * 256; t0 < n; t0 += gridDim.x * 256) {
        const int t = t0 + (int)threadIdx.x;
        if (threadIdx.x < 33) s_count[threadIdx.x] = 0u;
        __syncthreads();
        int b = 0;
        unsigned rank = 0u;
        if (t < n) {
            b = cost_bucket(offsets[t + 1] - offsets[t]);
            rank = atomicAdd(&s_count[b], 1u);
        }
        __syncthreads();
        if (threadIdx.x < 33 && s_count[threadIdx.x])
            s_base[threadIdx.x] = s_start[threadIdx.x] + atomicAdd(hist + 33 + threadIdx.x, s_count[threadIdx.x]);
        __syncthreads();
        if (t < n) order[s_base[b] + rank] = (unsigned)t;
    }
}

// Deterministic mode: each tile's list sorted by record index, so that the
// per-pixel sums of the forward and the chunks of the backward do not depend
// on the order of the scatter's atomics.  A bitonic sort of T R keys held in
// the registers of T threads, thread t's at the places t R + i: exchanges at
// a distance below R stay within a thread, below 32 R within a warp
// (shuffles), and only those beyond pass through shared memory.  Lists of up
// to 1024 entries are sorted by a warp each, longer ones by the block; one
// longer than kDetMaxSegment is left as it is and reported.
constexpr int kSortThreads = 256;

template <int T, int R>
__device__ __forceinline__ void sort_list(unsigned* __restrict__ list, const unsigned len, unsigned* __restrict__ sm) {
    const int t = threadIdx.x & (T - 1);
    unsigned v[R];
    // which key starts where does not matter: consecutive threads load consecutive entries
#pragma unroll
    for (int i = 0; i < R; ++i) v[i] = (unsigned)(i * T + t) < len ? list[i * T + t] : 0xffffffffu;
#pragma unroll
    for (int k = 2; k < R; k <<= 1)                             // runs within a thread
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1)
#pragma unroll
            for (int i = 0; i < R; ++i)
                if ((i & j) == 0) {
                    const unsigned lo = min(v[i], v[i | j]), hi = max(v[i], v[i | j]);
                    v[i] = (i & k) ? hi : lo;
                    v[i | j] = (i & k) ? lo : hi;
                }
#pragma unroll 1
    for (int k = R; k <= T * R; k <<= 1) {
        const bool up = ((t * R) & k) == 0;                     // the run this thread's keys belong to ascends
#pragma unroll 1
        for (int j = k >> 1; j >= R; j >>= 1) {
            const int d = j / R;
            const bool low = ((t & d) == 0) == up;              // keep the smaller of the two
            if (T > 32 && d >= 32) {
                __syncthreads();
#pragma unroll
                for (int i = 0; i < R; ++i) sm[i * T + t] = v[i];
                __syncthreads();
#pragma unroll
                for (int i = 0; i < R; ++i) {
                    const unsigned o = sm[i * T + (t ^ d)];
                    v[i] = low ? min(v[i], o) : max(v[i], o);
                }
            } else {
#pragma unroll
                for (int i = 0; i < R; ++i) {
                    const unsigned o = __shfl_xor_sync(0xffffffffu, v[i], d);
                    v[i] = low ? min(v[i], o) : max(v[i], o);
                }
            }
        }
#pragma unroll
        for (int j = R >> 1; j > 0; j >>= 1)
#pragma unroll
            for (int i = 0; i < R; ++i)
                if ((i & j) == 0) {
                    const unsigned lo = min(v[i], v[i | j]), hi = max(v[i], v[i | j]);
                    v[i] = up ? lo : hi;
                    v[i | j] = up ? hi : lo;
                }
    }
#pragma unroll
    for (int i = 0; i < R; ++i)
        if ((unsigned)(t * R + i) < len) list[t * R + i] = v[i];
}

// A block takes as many tiles as it has warps.  It is bound by the exchanges' instructions: 70 -> 23 us for 250k
// Gaussians at 1280x720 (3600 lists of 267 entries), where 512 threads per list sorted it in shared memory with a
// barrier per exchange (41 us with neighbouring tiles in one block).
__global__ void __launch_bounds__(kSortThreads, 3) k_sort_segments(const unsigned* __restrict__ offsets, int n_tiles,
                                                                unsigned* __restrict__ list, WsHeader* hdr) {
    constexpr int W = kSortThreads / 32;
    __shared__ unsigned sm[kDetMaxSegment];
    static_assert(kDetMaxSegment == 32 * kSortThreads, "the longest list: 32 keys per thread");
    // neighbouring tiles, whose lists are about as long, go to different blocks
    const int warp = threadIdx.x >> 5, stride = (int)gridDim.x;
    const int mine = (int)blockIdx.x + warp * stride;
    if (mine < n_tiles) {
        const unsigned a = offsets[mine], len = offsets[mine + 1] - a;
        if (len > 1u && len <= 1024u) {
            if (len <= 256u) sort_list<32, 8>(list + a, len, sm);
            else if (len <= 512u) sort_list<32, 16>(list + a, len, sm);
            else sort_list<32, 32>(list + a, len, sm);
        }
    }
    for (int t = blockIdx.x; t < n_tiles; t += stride) {
        const unsigned a = offsets[t], len = offsets[t + 1] - a;
        if (len <= 1024u) continue;                             // the whole block alike
        if (len <= 2048u) sort_list<kSortThreads, 8>(list + a, len, sm);
        else if (len <= 4096u) sort_list<kSortThreads, 16>(list + a, len, sm);
        else if (len <= (unsigned)kDetMaxSegment) sort_list<kSortThreads, 32>(list + a, len, sm);
        else if (threadIdx.x == 0) set_error(hdr, WSR_ERR_UNSUPPORTED);
    }
}

}  // namespace

cudaError_t launch_tile_order(const Views& vs, const unsigned* offsets, unsigned* buckets, unsigned* order,
                              cudaStream_t s) {
    const int n = vs.total_tiles;
    unsigned* const off = const_cast<unsigned*>(offsets);       // read only
    static_assert(WSR_ORDER_ONE_BLOCK_TILES == 16 * kScanBlock, "sixteen tiles per thread at most");
    if (n <= WSR_ORDER_ONE_BLOCK_TILES) {
        if (n <= 4 * kScanBlock) k_scan_order_rows<4, false><<<1, kScanBlock, 0, s>>>(nullptr, n, off, 0, nullptr, order);
        else if (n <= 8 * kScanBlock) k_scan_order_rows<8, false><<<1, kScanBlock, 0, s>>>(nullptr, n, off, 0, nullptr, order);
        else k_scan_order_rows<16, false><<<1, kScanBlock, 0, s>>>(nullptr, n, off, 0, nullptr, order);
        return cudaGetLastError();
    }
    const int nb = min((n + 255) / 256, 1024);
    k_order_hist<<<nb, 256, 0, s>>>(offsets, n, buckets);
    k_order_scatter<<<nb, 256, 0, s>>>(offsets, n, buckets, order);
    return cudaGetLastError();
}

// Blocks per view and threads of k_bin_local, 0 blocks when its counters do not fit in shared memory.
struct LocalBin {
    int blocks, threads;
    bool scatter;               // the scatter too takes its counters (scatter_local)
    size_t smem;
};

static LocalBin local_bin(const Views& vs, long long n, unsigned long long capacity) {
    LocalBin L{0, 0, false, 0};
    int t_max = 0;
    for (int v = 0; v < vs.n; ++v) t_max = max(t_max, vs.v[v].tiles_x * vs.v[v].tiles_y);
    L.blocks = bin_blocks_per_view(vs.n, t_max);
    if (L.blocks == 0) return L;
    L.threads = t_max <= kLocalTilesTwo ? 768 : 1024;
    L.scatter = scatter_local(t_max, capacity);
    // a small scene is spread over more SMs: eight batches of 32 per block
    const long long want = (n + 255) / 256;
    if (want < L.blocks) L.blocks = (int)max(want, 1ll);
    L.smem = sizeof(BinScratch) * (L.threads / 32) + sizeof(unsigned) * (size_t)t_max;
    return L;
}

template <int NT, bool SCATTER>
static cudaError_t launch_bin_local(const LocalBin& L, const float* records, long long n, const Views& vs,
                                    unsigned* cursor, unsigned* base, unsigned* list, unsigned long long capacity,
                                    WsHeader* hdr, cudaStream_t s) {
    // the shared-memory opt-in is a per-device function attribute: set once per device (thread-safe)
    static std::once_flag once[64];
    static cudaError_t once_err[64];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    std::call_once(once[dev], [&] {
        const size_t most = sizeof(BinScratch) * (NT / 32) + sizeof(unsigned) * (size_t)(NT == 768 ? kLocalTilesTwo
                                                                                                   : kLocalTiles);
        once_err[dev] = cudaFuncSetAttribute(k_bin_local<NT, SCATTER>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)most);
    });
    if (once_err[dev] != cudaSuccess) return once_err[dev];
    k_bin_local<NT, SCATTER><<<dim3((unsigned)L.blocks, (unsigned)vs.n), NT, L.smem, s>>>(
        reinterpret_cast<const float4*>(records), n, vs, cursor, base, list, capacity, hdr);
    return cudaGetLastError();
}

template <int I>
static cudaError_t launch_one(const float* records, long long n, const Views& vs, unsigned* offsets, unsigned* list,
                              unsigned long long capacity, WsHeader* hdr, unsigned* order, cudaStream_t s) {
    // the shared-memory opt-in is a per-device function attribute: set once per device (thread-safe)
    static std::once_flag once[64];
    static cudaError_t once_err[64];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    constexpr size_t fixed = sizeof(BinScratch) * 32;
    std::call_once(once[dev], [&] {
        once_err[dev] = cudaFuncSetAttribute(k_bin_one<I>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)(fixed + 2 * sizeof(unsigned) * 1024 * I));
    });
    if (once_err[dev] != cudaSuccess) return once_err[dev];
    k_bin_one<I><<<kOneBlocks, 1024, fixed + 2 * sizeof(unsigned) * (size_t)vs.total_tiles, s>>>(
        reinterpret_cast<const float4*>(records), n, vs, offsets, list, capacity, hdr, order);
    return cudaGetLastError();
}

cudaError_t launch_bin_one(const float* records, long long n, const Views& vs, unsigned* offsets, unsigned* list,
                           unsigned long long capacity, WsHeader* hdr, unsigned* order, cudaStream_t s) {
    static_assert(WSR_BIN_ONE_TILES == 4096, "four tiles per thread at most");
    return (vs.total_tiles <= 1024 ? launch_one<1> : launch_one<4>)(records, n, vs, offsets, list, capacity, hdr, order, s);
}

cudaError_t launch_bin_count(const float* records, long long n, const Views& vs, unsigned* cursor, unsigned* base,
                             unsigned long long capacity, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(cursor, 0, sizeof(unsigned) * (size_t)vs.total_tiles, s);
    if (e != cudaSuccess || n == 0) return e;
    const LocalBin L = local_bin(vs, n, capacity);
    if (base && L.blocks) {
        if (!L.scatter) base = nullptr;
        return L.threads == 768
                   ? launch_bin_local<768, false>(L, records, n, vs, cursor, base, nullptr, 0ull, nullptr, s)
                   : launch_bin_local<1024, false>(L, records, n, vs, cursor, base, nullptr, 0ull, nullptr, s);
    }
    dim3 grid((unsigned)((n + 255) / 256), (unsigned)vs.n);
    k_bin<false><<<grid, 256, 0, s>>>(reinterpret_cast<const float4*>(records), n, vs, cursor, nullptr, 0ull,
                                      nullptr);
    return cudaGetLastError();
}

cudaError_t launch_scan(const Views& vs, unsigned* cursor, unsigned* block_sums, unsigned* offsets,
                        unsigned long long capacity, WsHeader* hdr, unsigned* buckets, unsigned* order,
                        cudaStream_t s) {
    const int n = vs.total_tiles;
    if (n <= 16 * kScanBlock) {
        if (n <= kScanBlock) k_scan_order_rows<1, true><<<1, kScanBlock, 0, s>>>(cursor, n, offsets, capacity, hdr, order);
        else if (n <= 4 * kScanBlock) k_scan_order_rows<4, true><<<1, kScanBlock, 0, s>>>(cursor, n, offsets, capacity, hdr, order);
        else if (n <= 8 * kScanBlock) k_scan_order_rows<8, true><<<1, kScanBlock, 0, s>>>(cursor, n, offsets, capacity, hdr, order);
        else k_scan_order_rows<16, true><<<1, kScanBlock, 0, s>>>(cursor, n, offsets, capacity, hdr, order);
        return cudaGetLastError();
    }
    if (n <= kSmallScanTiles) {
        const size_t smem = sizeof(unsigned) * ((size_t)n + 1);
        if (smem > 48 * 1024) {
            // the dynamic shared-memory opt-in is a per-device attribute: set once per device (thread-safe)
            static std::once_flag once[64];
            static cudaError_t once_err[64];
            int dev = 0;
            cudaError_t e = cudaGetDevice(&dev);
            if (e != cudaSuccess) return e;
            if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
            std::call_once(once[dev], [&] {
                once_err[dev] = cudaFuncSetAttribute(k_scan_order_small, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                     (int)(sizeof(unsigned) * (kSmallScanTiles + 1)));
            });
            if (once_err[dev] != cudaSuccess) return once_err[dev];
        }
        k_scan_order_small<<<1, kScanBlock, smem, s>>>(cursor, n, offsets, capacity, hdr, order);
        return cudaGetLastError();
    }
    const int nb = (n + kScanTile - 1) / kScanTile;
    unsigned long long* bsum = reinterpret_cast<unsigned long long*>(block_sums);
    k_scan_reduce<<<nb, kScanBlock, 0, s>>>(cursor, n, bsum);
    k_scan_top<<<1, kScanBlock, 0, s>>>(bsum, nb, offsets, n, capacity, hdr);
    k_scan_apply<<<nb, kScanBlock, 0, s>>>(cursor, n, bsum, offsets, capacity);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || !order) return e;
    e = cudaMemsetAsync(buckets, 0, sizeof(unsigned) * 66, s);
    if (e != cudaSuccess) return e;
    return launch_tile_order(vs, offsets, buckets, order, s);
}

cudaError_t launch_bin_scatter(const float* records, long long n, const Views& vs, unsigned* cursor,
                               unsigned* base, unsigned* list, unsigned long long capacity, WsHeader* hdr,
                               cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    const LocalBin L = local_bin(vs, n, capacity);
    if (base && L.blocks && L.scatter) {
        return L.threads == 768 ? launch_bin_local<768, true>(L, records, n, vs, cursor, base, list, capacity, hdr, s)
                                : launch_bin_local<1024, true>(L, records, n, vs, cursor, base, list, capacity, hdr, s);
    }
    dim3 grid((unsigned)((n + 255) / 256), (unsigned)vs.n);
    k_bin<true><<<grid, 256, 0, s>>>(reinterpret_cast<const float4*>(records), n, vs, cursor, list, capacity, hdr);
    return cudaGetLastError();
}

cudaError_t launch_sort_segments(const Views& vs, const unsigned* offsets, unsigned* list, WsHeader* hdr,
                                 cudaStream_t s) {
    if (vs.total_tiles == 0) return cudaSuccess;
    const int per = kSortThreads / 32;
    k_sort_segments<<<(unsigned)((vs.total_tiles + per - 1) / per), kSortThreads, 0, s>>>(offsets, vs.total_tiles, list,
                                                                                          hdr);
    return cudaGetLastError();
}

}  // namespace wsr
