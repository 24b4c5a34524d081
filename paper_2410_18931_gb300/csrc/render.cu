// Per-pixel Weighted Sum Rendering, forward and backward (Eq. 7).
//
// One thread block per tile (or, with the persistent schedule, one per
// resident slot taking tiles longest first).  A warp takes an 8x8 region of
// the tile and walks the Gaussians of the tile's list (unordered: Eq. 7 is a
// sum) that reach it, a quarter warp per Gaussian; every thread owns 2x4
// pixels (two columns share each paired float2 FP32 instruction) and
// accumulates, in FP32 registers,
//     N += (c u w) e,   D += (u w) e,   e = exp(-q/2) = 2^(-q'),   q <= 9
// with q' = q log2(e)/2 evaluated from the record's sum of squares
// q' = (qs dy + qw dx)^2 + qd dx^2, which has no cancellation even for
// needle-like footprints.
// There is no early termination (App. D: every covering Gaussian counts).
// The epilogue writes C = (c_B w_B + N) / (w_B + D) and the denominator.
//
// The backward recomputes every (pixel, Gaussian) term from the records and
// the stored C and denominator (no per-pixel lists are kept).  It walks the
// pixels of each Gaussian's footprint row by row (per-row spans), a group of
// lanes per Gaussian, and per Gaussian adds d/d(u w), d/d(c u w) and moments
// of dL/dq' to a gradient record.
#include "wsr_launch.h"

namespace wsr {
namespace {

struct TileCoord {
    int v, tx, ty;
};

__device__ __forceinline__ TileCoord tile_coord(const Views& vs, int tile) {
    TileCoord t;
    t.v = view_of_tile(vs, tile);
    const View& V = vs.v[t.v];
    const int lt = tile - V.tile_base;
    t.ty = lt / V.tiles_x;
    t.tx = lt - t.ty * V.tiles_x;
    return t;
}

// Threads per block of the backward for chunks of CH Gaussians: 2 CH, at most 256.
template <int CH>
struct BwdThreads {
    static constexpr int value = CH < 128 ? 2 * CH : 256;
};

// Lane counts as a type, to instantiate one walk of the backward per group shape: lanes across a row's column
// pairs, and rows walked side by side.
template <int N, int R>
struct Lanes {
    static constexpr int value = N, rows = R;
};

// The part of a footprint q' <= QM inside a tile, as the backward walks it.  On row dy the footprint is
// dx = -(B'/A') dy +- sqrt(QM / A' - (det'/A'^2) dy^2) with A' = qw^2 + qd, B' = qs qw, det' = qd qs^2 (no
// cancellation); on column dx it is dy = (-qw dx +- sqrt(QM - qd dx^2)) / qs.  `rows` gives the tile's rows that
// it can reach between the tile's first and last columns (from the second form, at the columns of the tile
// nearest its highest and lowest points) and whether a row can need more than half the tile's width.  Both
// are widened far beyond their rounding; NaN widens them to the whole tile.
struct Footprint {
    float h0, h1, slope;                // half-width^2 = h0 - h1 dy^2, centre = -slope dy
    __device__ __forceinline__ Footprint(const float4 a, const float qd) {
        const float QM = kQMax * 1.0001f + 1e-4f;
        const float ia = rcp_approx(fmaf(a.w, a.w, qd));
        slope = a.z * a.w * ia;
        h0 = QM * ia;
        h1 = qd * a.z * a.z * ia * ia;
    }
    // (gx, gy): the tile's first pixel centre less the mean; x_lim, y_lim: its pixels inside the image
    template <int TW>
    __device__ __forceinline__ void rows(const float4 a, const float qd, const float gx, const float gy, const int x_lim,
                                         const int y_lim, int& first, int& count, bool& wide) const {
        const float QM = kQMax * 1.0001f + 1e-4f;
        const float iqs = rcp_approx(a.z), xm = sqrt_approx(QM * rcp_approx(qd));       // half-width of the box
        const float xt = -a.w * xm * sqrt_approx(rcp_approx(fmaf(a.w, a.w, qd)));       // dx of the highest point
        const float xl = gx, xr = gx + (float)(x_lim - 1);
        const float x1 = fminf(fmaxf(xt, xl), xr), x0 = fminf(fmaxf(-xt, xl), xr);
        const float y1 = fmaf(-a.w, x1, sqrt_approx(fmaxf(fmaf(-qd * x1, x1, QM), 0.0f))) * iqs;
        const float y0 = fmaf(-a.w, x0, -sqrt_approx(fmaxf(fmaf(-qd * x0, x0, QM), 0.0f))) * iqs;
        const float margin = fmaf(1e-3f, fabsf(y1) + fabsf(y0), 0.02f);
        int lo = 0, hi = y_lim - 1;
        if (y0 - margin - gy > 0.0f) lo = (int)fminf(ceilf(y0 - margin - gy), 64.0f);
        if (y1 + margin - gy < (float)hi) hi = (int)fmaxf(floorf(y1 + margin - gy), -1.0f);
        first = min(lo, y_lim - 1);
        count = max(hi - lo + 1, 0);
        // narrow: the widest row has at most TW / 2 - 1 pixel centres (one more may go before an even first
        // column), or the whole box lies in one half of the tile
        const float yc = fminf(fmaxf(0.0f, gy + (float)lo), gy + (float)hi);
        const float h = sqrt_approx(fmaxf(fmaf(-h1 * yc, yc, h0), 0.0f));
        wide = !(2.0f * h < (float)(TW / 2 - 1) - 0.1f || xm < gx + (float)(TW / 2) - 0.1f ||
                 -xm > gx + (float)(TW / 2 - 1) + 0.1f);
    }
};

// Pixel-per-thread layout of the pair-count diagnostic.
template <int TW, int TH, int PPT>
struct TileShape {
    static constexpr int NT = TW * TH / PPT;
    static_assert(TH % PPT == 0 && NT % 32 == 0, "whole warps");
};

// Forward.  A tile is cut into 8x8 regions, one warp each, and its list into S slices, each walked by a group of
// one warp per region.  The warps of a group stage a batch together, each thread one record: the walk constants
// into shared memory and, per region, whether the footprint reaches it.  Each warp then lists its region's
// Gaussians and walks them four at a time, one per quarter warp: eight threads with 2x4 pixels each cover the
// region, so the walk constants and the terms of a column pair are read and formed once for eight pixels, and
// the quarters' sums are added once per tile.
//   It is bound by the FP32 pipe (its paired instructions issue every 2.4 cycles from distinct registers, not
// every 2) and by the shared loads beside them.  16x16 tiles at 1M Gaussians and 1920x1080, persistent: 457 us
// with a warp per 16x8 pixels, 2x2 pixels per thread and a Gaussian per warp (1.96 pixel slots per pair, each
// warp staging the whole list); 414 us with that split and quarter warps on 8x8 regions; 363 us with the shared
// staging and a warp per region.  One block per tile: 566 -> 399 us, 95 -> 60 us for 200k at 1280x720.
//   20 warps per SM (at most 96 registers a thread): 363 us against 367 at 16, 379 at 24 and 389 at 28.
constexpr int kFwdWarpsPerSM = 20;
// The kernel for sparse views, 64 registers a thread: with 40 warps (48 registers, 8 bytes spilled) 8000 Gaussians at
// 1920x1080 take 13.2 us instead of 12.1, wide ones 65 instead of 57.
constexpr int kLightWarpsPerSM = 32;

template <int TW, int TH>
struct FwdShape {
    static constexpr int RX = TW / 8, RY = TH / 8, NR = RX * RY;
    static_assert(TW % 8 == 0 && TH % 8 == 0 && NR <= 4, "whole regions");
};

// Which of RX x RY regions of RW x 8 pixels a footprint q' <= kQMax can reach, one bit each (row by row); (gx, gy) is
// the first region's first pixel centre less the mean.  Eight pixel rows cut the ellipse in a convex part whose x-extent
// [x_l, x_r] has a closed form (as in the binning: x(dy) = (-B' dy +- sqrt(A' QM - det' dy^2)) / A' at the row
// of the band nearest the ellipse's rightmost and leftmost point); a region is reached when that extent,
// widened far beyond its rounding, meets the region's pixel-centre columns.  Every comparison is "not outside":
// NaN counts as reached.
template <int RX, int RY, int RW = 8>
__device__ __forceinline__ unsigned regions_hit(const float4 a, const float qd, const float gx, const float gy) {
    const float QM = kQMax * 1.0001f + 1e-4f;
    const float A = fmaf(a.w, a.w, qd), ia = rcp_approx(A), det = qd * a.z * a.z, aq = A * QM;
    const float dxm = sqrt_approx(QM * rcp_approx(qd));         // half-width of the ellipse
    const float dys = -(a.w * rcp_approx(a.z)) * dxm;           // dy of its rightmost point
    const float slope = a.z * a.w * ia, margin = fminf(2e-3f * dxm, 1e6f) + 0.01f;
    unsigned hit = 0u;
#pragma unroll
    for (int b = 0; b < RY; ++b) {
        const float ya = gy + (float)(8 * b), yb = ya + 7.0f;   // the band's pixel-centre rows
        const float dn = fminf(fmaxf(0.0f, ya), yb);
        const float dr = fminf(fmaxf(dys, ya), yb), dl = fminf(fmaxf(-dys, ya), yb);
        const float xr = fmaf(-slope, dr, sqrt_approx(fmaxf(fmaf(-det * dr, dr, aq), 0.0f)) * ia) + margin;
        const float xl = fmaf(-slope, dl, -sqrt_approx(fmaxf(fmaf(-det * dl, dl, aq), 0.0f)) * ia) - margin;
        const bool out = det * dn * dn > aq * 1.001f;
#pragma unroll
        for (int c = 0; c < RX; ++c)
            if (!(out || xl > gx + (float)(RW * c + RW - 1) || xr < gx + (float)(RW * c))) hit |= 1u << (b * RX + c);
    }
    return hit;
}

// A group's shared memory: two batches of 32 list entries per warp, and each warp's list of the batch's
// Gaussians that reach its region.  Walk constants, 48 bytes per Gaussian: (qs, qw, r_0, qd),
// (qd g_x^2, 2 qd g_x, c_r u w, c_g u w), (c_b u w, u w), with g the tile's first pixel centre less the mean and
// r_0 = qs g_y + qw g_x.  The last entry lies outside every pixel's cutoff.
template <int NR>
struct FwdStage {
    float4 g[2][32 * NR + 1][3];
    unsigned hits[2][NR][NR];                       // per region: which of each warp's 32 entries reach it
    unsigned short list[NR][4][8 * NR + 2];         // per region and quarter warp: byte offsets into g
};

// C = (c_B w_B + N) / D and D = w_B + sum of a pixel, from its sums (N, D) = (x, y, z, w)
__device__ __forceinline__ float4 pixel_out(const float4 n, const float* __restrict__ wparams) {
    const float wB = __ldg(wparams + 2), D = wB + n.w, inv = 1.0f / D;
    return make_float4((__ldg(wparams + 3) * wB + n.x) * inv, (__ldg(wparams + 4) * wB + n.y) * inv,
                       (__ldg(wparams + 5) * wB + n.z) * inv, D);
}

// Whether two neighbouring pixels, the first at an even column, start on eight bytes in every row of the view.
__device__ __forceinline__ bool pairs_aligned(const View& V, const float* out_rgb, const float* out_den) {
    return (((V.pix_base | V.W) & 1) | ((reinterpret_cast<size_t>(out_rgb) | reinterpret_cast<size_t>(out_den)) & 7)) == 0;
}

// Two neighbouring pixels of a row, the first at an even column, in eight-byte stores where they are aligned: the
// stores of a sparse view bound it otherwise (an empty 1920x1920 image 33 -> 25 us, 200k at 1280x720 58 -> 57).
__device__ __forceinline__ void store_pair(const View& V, const bool aligned, const int x, const int y, const float4 p0,
                                           const float4 p1, float* __restrict__ out_rgb, float* __restrict__ out_den) {
    if (x >= V.W || y >= V.H) return;
    const long long pix = V.pix_base + (long long)y * V.W + x;
    float* const o = out_rgb + 3 * pix;
    if (aligned) {                                  // (the width is even: both pixels exist)
        reinterpret_cast<float2*>(o)[0] = f2(p0.x, p0.y);
        reinterpret_cast<float2*>(o)[1] = f2(p0.z, p1.x);
        reinterpret_cast<float2*>(o)[2] = f2(p1.y, p1.z);
        *reinterpret_cast<float2*>(out_den + pix) = f2(p0.w, p1.w);
        return;
    }
    o[0] = p0.x;
    o[1] = p0.y;
    o[2] = p0.z;
    out_den[pix] = p0.w;
    if (x + 1 < V.W) {
        o[3] = p1.x;
        o[4] = p1.y;
        o[5] = p1.z;
        out_den[pix + 1] = p1.w;
    }
}

// The same where not every row starts on eight bytes (an odd width or an odd first pixel), by all lanes of a warp: rows
// that start at an odd pixel pair their columns one further on.  `next` is the lane that holds the columns to the
// right, and for the last lane of a row (`last`) the first, WIDTH columns before those.
template <int WIDTH>
__device__ __forceinline__ void store_shifted(const View& V, const int next, const bool last, const int x, const int y,
                                              const float4 p0, const float4 p1, float* __restrict__ out_rgb,
                                              float* __restrict__ out_den) {
    const long long row = V.pix_base + (long long)y * V.W;
    const bool aligned = ((reinterpret_cast<size_t>(out_rgb) | reinterpret_cast<size_t>(out_den)) & 7) == 0;
    const bool off = ((row + x) & 1) != 0;
    const float4 nx = make_float4(__shfl_sync(0xffffffffu, p0.x, next), __shfl_sync(0xffffffffu, p0.y, next),
                                  __shfl_sync(0xffffffffu, p0.z, next), __shfl_sync(0xffffffffu, p0.w, next));
    if (y >= V.H) return;
    const float4 a = off ? p1 : p0, b = off ? nx : p1;
    const int xa = off ? x + 1 : x, xb = off ? (last ? x + 2 - WIDTH : x + 2) : x + 1;
    if (aligned && xb == xa + 1 && xb < V.W) {
        float2* const o = reinterpret_cast<float2*>(out_rgb + 3 * (row + xa));
        o[0] = f2(a.x, a.y);
        o[1] = f2(a.z, b.x);
        o[2] = f2(b.y, b.z);
        *reinterpret_cast<float2*>(out_den + row + xa) = f2(a.w, b.w);
        return;
    }
    if (xa < V.W) {
        float* const o = out_rgb + 3 * (row + xa);
        o[0] = a.x;
        o[1] = a.y;
        o[2] = a.z;
        out_den[row + xa] = a.w;
    }
    if (xb < V.W) {
        float* const o = out_rgb + 3 * (row + xb);
        o[0] = b.x;
        o[1] = b.y;
        o[2] = b.z;
        out_den[row + xb] = b.w;
    }
}

template <int TW, int TH, int S>
__device__ __forceinline__ void fwd_tile(const int tile, const float4* __restrict__ rec,
                                         const unsigned* __restrict__ offsets, const unsigned* __restrict__ list,
                                         const Views& vs, const float* __restrict__ wparams,
                                         float* __restrict__ out_rgb, float* __restrict__ out_den) {
    using F = FwdShape<TW, TH>;
    constexpr int RX = F::RX, NR = F::NR, BATCH = 32 * NR;
    union GroupMem {
        FwdStage<NR> st;
        float4 px[TW * TH];             // the slice's sums, at the end
    };
    __shared__ __align__(16) unsigned char s_mem[S][sizeof(GroupMem)];

    // The slice's batches of list entries, each thread staging one; the next batch's records are loaded while
    // this one is walked, and the list entries of the one after that.
    const unsigned start = offsets[tile], end = offsets[tile + 1];
    const TileCoord tc = tile_coord(vs, tile);
    const View& V = vs.v[tc.v];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, quarter = lane >> 3, o8 = lane & 7;
    const int w = warp % NR, slice = warp / NR;     // the warp's region, and its group
    const int x_org = tc.tx * TW, y_org = tc.ty * TH;
    FwdStage<NR>& st = reinterpret_cast<GroupMem*>(s_mem[slice])->st;
    auto group_sync = [&] {
        if constexpr (NR == 1) __syncwarp();
        else if constexpr (S == 1) __syncthreads();
        else asm volatile("bar.sync %0, %1;" ::"r"(1 + slice), "n"(32 * NR) : "memory");
    };
    // a thread's 2x4 pixels (columns, rows) of the region, as offsets from the tile's first pixel
    const float2 ox = f2((float)(8 * (w % RX) + 2 * (o8 & 3)), (float)(8 * (w % RX) + 2 * (o8 & 3) + 1));
    const float oy0 = (float)(8 * (w / RX) + 4 * (o8 >> 2));

    // accumulators per pixel (row r, column c): (N_r, N_g) and (N_b, D)
    float2 rg[4][2], bd[4][2];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 2; ++c) rg[r][c] = bd[r][c] = f2(0.f, 0.f);

    if (w == 0 && lane < 2) {
        st.g[lane][BATCH][0] = make_float4(0.f, 0.f, 1e4f, 0.f);
        st.g[lane][BATCH][1] = st.g[lane][BATCH][2] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    unsigned base = start + (unsigned)(BATCH * slice);
    const int me = 32 * w + lane;
    unsigned nidx = base + me < end ? list[base + me] : 0u;
    float4 na, nb;
    float ncb;
    auto fetch = [&](unsigned b) {
        na = nb = make_float4(0.f, 0.f, 0.f, 0.f);
        ncb = 0.f;
        if (b + me < end) {
            const float4* p = rec + 3ull * nidx;
            na = __ldg(p);
            nb = __ldg(p + 1);
            ncb = __ldg(reinterpret_cast<const float*>(p + 2));
        }
        nidx = b + BATCH * S + me < end ? list[b + BATCH * S + me] : 0u;
    };
    fetch(base);
    int buf = 0;
    for (; base < end; base += BATCH * S, buf ^= 1) {
        {
            const float4 a = na, b = nb;
            const float gx = (float)x_org + 0.5f - a.x, gy = (float)y_org + 0.5f - a.y;
            st.g[buf][me][0] = make_float4(a.z, a.w, fmaf(a.z, gy, a.w * gx), b.x);
            st.g[buf][me][1] = make_float4(b.x * gx * gx, 2.0f * b.x * gx, b.z, b.w);
            *reinterpret_cast<float2*>(&st.g[buf][me][2]) = f2(ncb, b.y);
            const unsigned hit = base + me < end ? regions_hit<RX, F::RY>(a, b.x, gx, gy) : 0u;
#pragma unroll
            for (int k = 0; k < NR; ++k) {
                const unsigned bal = __ballot_sync(0xffffffffu, (hit >> k) & 1u);
                if (lane == 0) st.hits[buf][k][w] = bal;
            }
        }
        fetch(base + BATCH * S);
        // The batch is staged, and every warp has walked the one before: the buffer written next is free
        group_sync();
        // the region's Gaussians by turns to the four quarter warps; the last round is filled with the entry
        // that lies outside
        int n = 0;
#pragma unroll
        for (int k = 0; k < NR; ++k) {
            const unsigned bal = st.hits[buf][w][k];
            const int pos = n + __popc(bal & ((1u << lane) - 1u));
            if ((bal >> lane) & 1u) st.list[w][pos & 3][pos >> 2] = (unsigned short)((32 * k + lane) * 48);
            n += __popc(bal);
        }
        if (lane < 3) st.list[w][(n + lane) & 3][(n + lane) >> 2] = (unsigned short)(BATCH * 48);
        __syncwarp();
        const char* const gbase = reinterpret_cast<const char*>(st.g[buf]);
        const unsigned short* const lk = st.list[w][quarter];
        const int nj = (n + 3) >> 2;
#pragma unroll 4
        for (int j = 0; j < nj; ++j) {
            const float4* g = reinterpret_cast<const float4*>(gbase + lk[j]);
            const float4 u = g[0], t = g[1];
            const float2 cbuw = *reinterpret_cast<const float2*>(g + 2);
            const float2 crg = f2(t.z, t.w);
            // q' = r^2 + qd dx^2 with dx = g_x + o_x: qd dx^2 = qd g_x^2 + o_x (2 qd g_x + o_x qd) and
            // r = r_0 + qs o_y + qw o_x from the values at the tile's first pixel centre (8-wide tiles
            // add the two products the other way round)
            const float2 P = __ffma2_rn(ox, __ffma2_rn(ox, f2(u.w, u.w), f2(t.y, t.y)), f2(t.x, t.x));
            const float2 rx = __ffma2_rn(f2(u.y, u.y), ox, f2(u.z, u.z));       // TW == 8 only
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const float oy = oy0 + (float)r;
                float2 rr;
                if constexpr (TW == 8) {
                    rr = __ffma2_rn(f2(u.x, u.x), f2(oy, oy), rx);
                } else {
                    const float ry = fmaf(u.x, oy, u.z);
                    rr = __ffma2_rn(f2(u.y, u.y), ox, f2(ry, ry));
                }
                const float2 q = __ffma2_rn(rr, rr, P);
                if (q.x <= kQMax) {
                    const float e = ex2_approx(-q.x);
                    rg[r][0] = __ffma2_rn(crg, f2(e, e), rg[r][0]);
                    bd[r][0] = __ffma2_rn(cbuw, f2(e, e), bd[r][0]);
                }
                if (q.y <= kQMax) {
                    const float e = ex2_approx(-q.y);
                    rg[r][1] = __ffma2_rn(crg, f2(e, e), rg[r][1]);
                    bd[r][1] = __ffma2_rn(cbuw, f2(e, e), bd[r][1]);
                }
            }
        }
        __syncwarp();                                   // the list is read: the next batch's may be written
    }

    // The quarter warps' sums: a lane keeps row `quarter` of its 2x4 pixels (two exchanges, each handing over
    // half of what is left)
    const bool up = quarter & 2, odd = quarter & 1;
    auto pass = [&](float lo, float hi, bool keep_hi, int mask) {
        const float mine = keep_hi ? hi : lo, give = keep_hi ? lo : hi;
        return mine + __shfl_xor_sync(0xffffffffu, give, mask);
    };
    float4 sum[2];
    sum[0] = sum[1] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (start != end)
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        float o[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            auto val = [&](int r) {
                const float2 x = e < 2 ? rg[r][c] : bd[r][c];
                return e & 1 ? x.y : x.x;
            };
            o[e] = pass(pass(val(0), val(2), up, 16), pass(val(1), val(3), up, 16), odd, 8);
        }
        sum[c] = make_float4(o[0], o[1], o[2], o[3]);
    }
    const int ly = 8 * (w / RX) + 4 * (o8 >> 2) + quarter, lx = 8 * (w % RX) + 2 * (o8 & 3);
    if (S > 1 && start != end) {
        // the slices' sums, added by the first group in their order
        if (slice > 0) {
            group_sync();                               // the stage is read: it may hold the sums
            float4* const px = reinterpret_cast<GroupMem*>(s_mem[slice])->px;
            px[32 * w + lane] = sum[0];
            px[32 * w + lane + 32 * NR] = sum[1];
        }
        __syncthreads();
        if (slice > 0) return;                          // (back to the tile loop)
#pragma unroll
        for (int k = 1; k < S; ++k)
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const float4 o = reinterpret_cast<const GroupMem*>(s_mem[k])->px[32 * w + lane + 32 * NR * c];
                sum[c].x += o.x;
                sum[c].y += o.y;
                sum[c].z += o.z;
                sum[c].w += o.w;
            }
    }
    if (S > 1 && slice > 0) return;
    store_pair(V, pairs_aligned(V, out_rgb, out_den), x_org + lx, y_org + ly, pixel_out(sum[0], wparams),
               pixel_out(sum[1], wparams), out_rgb, out_den);
}

// The kernel for sparse views: a warp per 16x8 pixels (8x8 in tiles of that width).
template <int TW, int TH>
struct LightShape {
    static constexpr int RW = TW == 8 ? 8 : 16, RX = TW / RW, NR = RX * (TH / 8);
    static constexpr int COLS = RW / 8;     // columns per thread, of two rows; eight lanes across
    static_assert(TW % RW == 0 && TH % 8 == 0, "whole regions");
};

// Forward for sparse views, where a tile's time is the latency of its chain (offsets, list, records, pixels) and not
// its arithmetic: a warp per region, each staging the tile's list on its own (no barrier between warps), two rows and
// one or two columns per thread, the Gaussians that reach the region one after another.  A quarter to a half of the
// kernel above's accumulators, so that 32 warps fit on an SM.
//   With a warp per 8x8 pixels, two columns of one row per thread and batches staged by the block it took 1920x1080,
// us: 8000 Gaussians 15.7 -> 12.1, 16000 19.7 -> 16.4 (and 22.2 -> 17.8 at 1919x1079), 4.5 times as wide 70 -> 57 and
// 133 -> 108, 12 times as wide 394 -> 303; 16000 at 3840x2160 66 -> 48; in 8x8 tiles 16000 22 -> 19.3, wide 144 -> 109.
template <int TW, int TH>
__device__ __forceinline__ void fwd_tile_light(const int tile, const float4* __restrict__ rec,
                                               const unsigned* __restrict__ offsets, const unsigned* __restrict__ list,
                                               const Views& vs, const float* __restrict__ wparams,
                                               float* __restrict__ out_rgb, float* __restrict__ out_den) {
    using F = LightShape<TW, TH>;
    constexpr int COLS = F::COLS;
    __shared__ float4 s_g[F::NR][32][3];                // walk constants, as in FwdStage
    const unsigned start = offsets[tile], end = offsets[tile + 1];
    const TileCoord tc = tile_coord(vs, tile);
    const View& V = vs.v[tc.v];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float4(*const g)[3] = s_g[w];
    const int x_org = tc.tx * TW, y_org = tc.ty * TH;
    const int rx = F::RW * (w % F::RX), ry = 8 * (w / F::RX);               // the warp's region
    const int lx = rx + COLS * (lane & 7), ly = ry + 2 * (lane >> 3);
    const float2 ox = f2((float)lx, (float)(lx + 1));
    const float oy = (float)ly;
    float2 rg[2][COLS], bd[2][COLS];                    // per row and column: (N_r, N_g) and (N_b, D)
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int c = 0; c < COLS; ++c) rg[r][c] = bd[r][c] = f2(0.f, 0.f);
    auto add = [&](const float q, const float2 crg, const float2 cbuw, float2& o_rg, float2& o_bd) {
        if (q <= kQMax) {
            const float e = ex2_approx(-q);
            o_rg = __ffma2_rn(crg, f2(e, e), o_rg);
            o_bd = __ffma2_rn(cbuw, f2(e, e), o_bd);
        }
    };
    // the next batch's records are loaded while this one is walked, and the list entries of the one after that
    unsigned nidx = start + lane < end ? list[start + lane] : 0u;
    float4 na, nb;
    float ncb;
    auto fetch = [&](unsigned b) {
        na = nb = make_float4(0.f, 0.f, 0.f, 0.f);
        ncb = 0.f;
        if (b + lane < end) {
            const float4* p = rec + 3ull * nidx;
            na = __ldg(p);
            nb = __ldg(p + 1);
            ncb = __ldg(reinterpret_cast<const float*>(p + 2));
        }
        nidx = b + 32 + lane < end ? list[b + 32 + lane] : 0u;
    };
    fetch(start);
    for (unsigned base = start; base < end; base += 32) {
        const float4 a = na, b = nb;
        const float gx = (float)x_org + 0.5f - a.x, gy = (float)y_org + 0.5f - a.y;
        // (the binning has tested a tile that is one region)
        const bool hit = base + lane < end &&
                         (F::NR == 1 || regions_hit<1, 1, F::RW>(a, b.x, gx + (float)rx, gy + (float)ry));
        const unsigned bal = __ballot_sync(0xffffffffu, hit);
        if (hit) {
            float4* const o = g[__popc(bal & ((1u << lane) - 1u))];
            o[0] = make_float4(a.z, a.w, fmaf(a.z, gy, a.w * gx), b.x);
            o[1] = make_float4(b.x * gx * gx, 2.0f * b.x * gx, b.z, b.w);
            *reinterpret_cast<float2*>(o + 2) = f2(ncb, b.y);
        }
        fetch(base + 32);
        __syncwarp();
        const int nj = __popc(bal);
#pragma unroll 4
        for (int j = 0; j < nj; ++j) {
            const float4 u = g[j][0], t = g[j][1];
            const float2 cbuw = *reinterpret_cast<const float2*>(&g[j][2]);
            const float2 crg = f2(t.z, t.w);
            // q' by the operations of the kernel above (and so the same pairs): there the columns are paired in tiles
            // of every width, here the rows where a thread has one column
            if constexpr (COLS == 1) {
                const float P = fmaf(ox.x, fmaf(ox.x, u.w, t.y), t.x), rx = fmaf(u.y, ox.x, u.z);
                const float2 rr = __ffma2_rn(f2(u.x, u.x), f2(oy, oy + 1.0f), f2(rx, rx));
                const float2 q = __ffma2_rn(rr, rr, f2(P, P));
                add(q.x, crg, cbuw, rg[0][0], bd[0][0]);
                add(q.y, crg, cbuw, rg[1][0], bd[1][0]);
            } else {
                const float2 P = __ffma2_rn(ox, __ffma2_rn(ox, f2(u.w, u.w), f2(t.y, t.y)), f2(t.x, t.x));
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    const float ry = fmaf(u.x, oy + (float)r, u.z);
                    const float2 rr = __ffma2_rn(f2(u.y, u.y), ox, f2(ry, ry));
                    const float2 q = __ffma2_rn(rr, rr, P);
                    add(q.x, crg, cbuw, rg[r][0], bd[r][0]);
                    add(q.y, crg, cbuw, rg[r][COLS - 1], bd[r][COLS - 1]);
                }
            }
        }
        __syncwarp();                                   // the batch is walked: the next may be written
    }
    const bool pairs = pairs_aligned(V, out_rgb, out_den);
    float4 px[2][COLS];
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int c = 0; c < COLS; ++c)
            px[r][c] = pixel_out(make_float4(rg[r][c].x, rg[r][c].y, bd[r][c].x, bd[r][c].y), wparams);
    if constexpr (COLS == 1) {
        // two lanes side by side: the even one takes both columns of the first row, the odd one of the second
        const bool odd = lane & 1;
        const float4 give = odd ? px[0][0] : px[1][0], mine = odd ? px[1][0] : px[0][0];
        const float4 got = make_float4(__shfl_xor_sync(0xffffffffu, give.x, 1), __shfl_xor_sync(0xffffffffu, give.y, 1),
                                       __shfl_xor_sync(0xffffffffu, give.z, 1), __shfl_xor_sync(0xffffffffu, give.w, 1));
        const float4 p0 = odd ? got : mine, p1 = odd ? mine : got;
        const int x = x_org + (lx & ~1), y = y_org + ly + odd;
        if (pairs) store_pair(V, true, x, y, p0, p1, out_rgb, out_den);
        else store_shifted<8>(V, (lane & ~7) | ((lane + 2) & 7), (lane & 7) >= 6, x, y, p0, p1, out_rgb, out_den);
    } else {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const float4 p0 = px[r][0], p1 = px[r][COLS - 1];
            const int x = x_org + lx, y = y_org + ly + r;
            if (pairs) store_pair(V, true, x, y, p0, p1, out_rgb, out_den);
            else store_shifted<16>(V, (lane & ~7) | ((lane + 1) & 7), (lane & 7) == 7, x, y, p0, p1, out_rgb, out_den);
        }
    }
}

// Persistent schedule: block i takes the tile order[i], and then the others through *counter.  Dealt by their numbers
// the longest tiles spread over the SMs where every block has one (claimed through the counter they lie anywhere: 2108
// tiles of wide Gaussians in the sparse kernel, 979x543, 39 -> 23 us), and views of no more tiles than blocks need
// neither counter nor clear (1000 Gaussians at 200x120 8.4 -> 4.1 us, at 500x313 8.4 -> 4.2).
template <typename F>
__device__ __forceinline__ void for_each_tile(const unsigned* __restrict__ order, unsigned* __restrict__ counter,
                                              int n_tiles, F&& body) {
    if (order == nullptr) {
        body((int)blockIdx.x);
        return;
    }
    __shared__ int s_item;
    for (int item = (int)blockIdx.x; item < n_tiles;) {
        body((int)order[item]);
        if ((int)gridDim.x >= n_tiles) break;
        __syncthreads();                      // the tile is done with shared memory
        if (threadIdx.x == 0) s_item = (int)(gridDim.x + atomicAdd(counter, 1u));
        __syncthreads();
        item = s_item;
    }
}

template <int TW, int TH, int S>
__global__ void __launch_bounds__(32 * S * FwdShape<TW, TH>::NR, kFwdWarpsPerSM / (S * FwdShape<TW, TH>::NR))
    k_render_fwd(const float4* __restrict__ rec, const unsigned* __restrict__ offsets,
                 const unsigned* __restrict__ list, const Views vs, const float* __restrict__ wparams,
                 float* __restrict__ out_rgb, float* __restrict__ out_den, const unsigned* __restrict__ order,
                 unsigned* __restrict__ counter) {
    for_each_tile(order, counter, vs.total_tiles, [&](int tile) {
        fwd_tile<TW, TH, S>(tile, rec, offsets, list, vs, wparams, out_rgb, out_den);
    });
}

template <int TW, int TH>
__global__ void __launch_bounds__(32 * LightShape<TW, TH>::NR, kLightWarpsPerSM / LightShape<TW, TH>::NR)
    k_render_fwd_light(const float4* __restrict__ rec, const unsigned* __restrict__ offsets,
                       const unsigned* __restrict__ list, const Views vs, const float* __restrict__ wparams,
                       float* __restrict__ out_rgb, float* __restrict__ out_den, const unsigned* __restrict__ order,
                       unsigned* __restrict__ counter) {
    for_each_tile(order, counter, vs.total_tiles, [&](int tile) {
        fwd_tile_light<TW, TH>(tile, rec, offsets, list, vs, wparams, out_rgb, out_den);
    });
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}

// x 2^s rounded to the nearest integer (halves to even), as __double2ll_rn(ldexp((double)x, s)) gives it, from the
// float's bits: the deterministic mode forms nine of them per Gaussian and tile, and the double-precision pipe is 64
// times slower than the others.  With the sums added by consecutive lanes: 237 -> 185 us for 250k Gaussians at
// 1280x720 (each lane adding its Gaussian's nine words took 237 us with either conversion).
__device__ __forceinline__ long long fixed_point(const float x, const int s) {
    const unsigned bits = __float_as_uint(x);
    const int ex = (int)((bits >> 23) & 0xffu);
    if (ex == 0xff) return __double2ll_rn(ldexp((double)x, s));         // infinities and NaN
    const unsigned m = (bits & 0x7fffffu) | (ex ? 0x800000u : 0u);
    const int sh = (ex ? ex : 1) - 150 + s;                             // |x| 2^s = m 2^sh
    long long q;
    if (sh >= 0) {
        if (sh > 38) return __double2ll_rn(ldexp((double)x, s));        // beyond 2^62
        q = (long long)((unsigned long long)m << sh);
    } else {
        const int n = min(-sh, 31);                                     // from 26 on everything rounds to zero
        const unsigned r = m >> n, rest = m & ((1u << n) - 1u), half = 1u << (n - 1);
        q = (long long)(r + ((rest > half || (rest == half && (r & 1u))) ? 1u : 0u));
    }
    return (bits >> 31) ? -q : q;
}

// Backward, one block per tile, a group of lanes per Gaussian.
//
// The tile's pixel terms P = (G/D, -(G.C)/D) sit in shared memory by column
// pairs, two float4 planes (x0, x1, y0, y1) and (z0, z1, w0, w1), with zero
// pairs past the tile's right edge as far as a lane reads.  For each chunk of
// CH Gaussians of the tile:
//   A. a thread per Gaussian finds the rows of the tile that its footprint
//      reaches and whether a row may need more than TW / 2 pixels (closed
//      forms, Footprint), and takes its rank in its bucket of the sort below;
//   B. the chunk's Gaussians are ordered wide ones first (more than TW / 2
//      pixels on a row), each class by its number of rows, longest first
//      (a counting sort: the buckets' starts from one warp suffix scan); each
//      warp takes the next Gaussians of a class whenever it is free (a shared
//      counter per class), so that the groups of a warp walk for the same
//      number of steps and the warps stay busy;
//   C. a group of L consecutive lanes takes one Gaussian at a time and walks
//      its rows one per step, L = TW / (2 M) for the wide class and TW / (4 M)
//      for the narrow one (whose spans all fit in 2 M L columns), M = 4 column
//      pairs per lane and row (2 for 8-pixel-wide tiles); lane k takes column
//      pairs start / 2 + k + m L (m < M) of the row, start being the first
//      column the footprint can reach there, rounded down to even, so the
//      lanes of a group read consecutive entries of each plane, 2 M pixels
//      per step from one start, every quantity of a column pair in one paired
//      FP32 op.  The nine record terms stay in registers until
//      the Gaussian's last row; then log2(L) shuffle steps sum them over the
//      group and its first lane adds them to the Gaussian's global record (in
//      the deterministic mode: as fixed point, in units that a per-Gaussian
//      bound fixes).  A Gaussian's sums over a tile are thus formed in one
//      fixed order, whichever group takes it.
// Every pair is tested against the forward's cutoff (q' <= kQMax, FP32, from
// the same record values).  The forward forms q' from values at the tile's
// first pixel centre, the walk from each pixel's own offsets, so a pair
// within rounding of the cutoff (a tie: its term is e^-4.5 of the
// Gaussian's peak there) may be counted by one and not the other.
// Gaussians per chunk: CH, a template parameter (64, 128, 256 or 512); threads
// per block: BwdThreads<CH> (2 CH up to 256).
//   It is bound by the shared-memory data path (76% busy: two 16-byte loads per
// column pair and lane, a quarter of the wavefronts bank conflicts) and the FP32
// pipe (63%).  1M Gaussians at 1920x1080, 512 per chunk, persistent: 1008 us and
// 7.9e8 warp instructions when step A found every row's span (two threads per
// Gaussian, a table of spans in shared memory), 931 us and 6.7e8 with the rows in
// closed form and a row's start formed as it is walked; three blocks per SM at 80
// registers, without spills, took 960 us.
constexpr float kMagic = 12582912.0f;       // 1.5 x 2^23
// Up to this many Gaussians of a class in a chunk are walked by twice the lanes, two rows side by side, so that more
// warps have some: 915 -> 905 us at 1M Gaussians and 1920x1080, 84 -> 80 us at 150k and 979x543 (more lanes for
// larger classes cost more bank conflicts than they save: 1111 us with two rows throughout).
constexpr int kFewWalk = 64;
// Chunks per part of a tile's list (1 for few tiles): claiming each chunk on its own costs 20 us at 1M Gaussians.
constexpr unsigned kPartChunks = 4;
// Deterministic mode: a bound's exponent in a byte, kExpBias above frexpf's (-148 for the smallest subnormal, at most
// 100 here), and the byte of a bound of zero.
constexpr int kExpBias = 24, kNoBound = 127;
static_assert(-148 + kExpBias >= -128 && 100 + kExpBias < kNoBound, "exponents and kNoBound fit in a byte");
constexpr int kHelpTiles = 1024;            // tiles whose chunks idle blocks look for (a power of two)
// Tiles a block claims at once after one of at most kShortList entries.  Claims of 8 gain and lose 1 % against 4.
constexpr unsigned kShortList = 64u;
constexpr int kClaim = 4;

// Schedule: as many blocks as fit on the device take the tiles in the order given (longest first, or as they are
// numbered), each the tile of its own number and then through *counter.  A tile's list is cut into parts of part_chunks chunks; those of a tile with several are
// handed out one by one (parts[tile], zero at the start), and a block that finds no tile left looks for parts nobody
// has taken among the first tiles of the order, picking its tile at random among those that have any, so that the
// longest lists do not hold up the end.  Nothing waits for another block: a part is done by whoever takes it, and the
// block that took the tile itself takes parts until none is left.
//   Measured against a block per tile and chunks of 128, and against the longest-first order with 512: 1301 and
// 931 -> 905 us at 1M Gaussians and 1920x1080, 187 and 135 -> 128 us for 200k at 1280x720, 58 -> 22 us for 5000 at
// 200x120 (104 tiles).  Taking the next tile while one is walked made it slower, 35 us at 1M: a block then holds a
// tile that others could start.
//   Where lists are short a tile's time is its chain of loads, and the claim of the next one (counter, order, offsets)
// a third of it: there a block claims up to kClaim tiles at once, fewer as the end comes near.  A block looks for
// others' parts only if a list has several.  With a claim per tile, the first one too, and a search by every block,
// 1920x1080 and 1000 Gaussians took 78 instead of 72 us and in 8x8 tiles 193 instead of 172, 979x543 28 instead of 24,
// 200x120 16.9 instead of 12.4 (a clear less among them), 500x313 and 10000 27 instead of 20.
template <int TW, int TH, int CH, bool DET>
__global__ void __launch_bounds__(BwdThreads<CH>::value, 1024 / BwdThreads<CH>::value)
    k_render_bwd(const float4* __restrict__ rec, const unsigned* __restrict__ offsets,
                 const unsigned* __restrict__ list, const Views vs, const float* __restrict__ wparams,
                 const float* __restrict__ out_rgb, const float* __restrict__ out_den,
                 const float* __restrict__ grad_rgb, float* __restrict__ grec, float* __restrict__ gw,
                 float* __restrict__ bg_tiles, const unsigned* __restrict__ det_pmax,
                 const unsigned* __restrict__ order, unsigned* __restrict__ counter, unsigned* __restrict__ parts,
                 const unsigned part_chunks) {
    constexpr int NT = BwdThreads<CH>::value;
    constexpr int NW = NT / 32;
    // pixel-table row pitch in column pairs: the row's TW / 2 pairs, then zero pairs up to the farthest pair a
    // lane reads (start / 2 + k + m L <= (TW / 2 - 1) + (TW / 2 - 1)), so no index needs a clamp; odd, so that
    // the rows start in different banks
    constexpr int PP = TW - 1;
    constexpr int NB = TH + 1;                          // row counts 0 .. TH
    constexpr int NK = 2 * NB;                          // sort keys: narrow 0 .. TH, wide NB .. NB + TH
    static_assert(CH % 32 == 0 && TW % 8 == 0 && TW <= 64 && CH <= 512 && NK <= NT, "layout");
    static_assert((TW * TH) % NT == 0 || NT % (TW * TH) == 0, "whole pixels per thread");
    constexpr int M = TW >= 16 ? 4 : 2;                 // column pairs per lane and row in step C
    // per pixel: G/D (3), -(G.C)/D, stored per column pair as (x0, x1, y0, y1) and (z0, z1, w0, w1)
    __shared__ float4 spA[PP * TH];
    __shared__ float4 spB[PP * TH];
    __shared__ float4 s0[CH];                   // mu_x, mu_y, qs, qw
    __shared__ float4 s1[CH];                   // qd, u w, c_r u w, c_g u w
    __shared__ float2 s2[CH];                   // c_b u w, u w
    __shared__ unsigned sidx[CH];
    __shared__ unsigned char sfirst[CH];        // first row of the tile that the footprint reaches
    __shared__ unsigned char snst[CH];          // rows from there to the last one
    __shared__ unsigned char skey[CH];          // sort key: rows, plus NB when wide
    __shared__ unsigned short srank[CH];        // rank among the chunk's Gaussians of the same key
    __shared__ unsigned short sord[CH];         // the chunk's Gaussians: wide ones first, most rows first
    __shared__ unsigned shist[NK];
    __shared__ unsigned snext[2];               // per class: the next position of the order a warp takes
    __shared__ float4 sbg[NW];                  // background terms per warp
    // deterministic mode: a warp's Gaussians' sums on their way out, the exponents of their bounds, their records
    __shared__ float s_val[DET ? NW : 1][DET ? 32 : 1][9];
    __shared__ signed char s_exp[DET ? NW : 1][DET ? 32 : 1][9];
    __shared__ unsigned s_rec[DET ? NW : 1][DET ? 32 : 1];
    __shared__ int4 s_cur, s_next[kClaim];      // a tile (-1: none left) and its ends; and those claimed with it,
    __shared__ int s_left, s_seen;              // of which s_left are to come; how far the order was claimed then
    __shared__ unsigned s_part;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n = vs.total_tiles;
    const float wB = __ldg(wparams + 2);
    const float pmax = DET ? __int_as_float(*det_pmax) : 0.0f;    // deterministic mode
    auto item_tile = [&](unsigned item) { return item < (unsigned)n ? order ? (int)order[item] : (int)item : -1; };
    auto load_tile = [&](int t) {
        return t < 0 ? make_int4(-1, 0, 0, 0) : make_int4(t, (int)offsets[t], (int)offsets[t + 1], 0);
    };
    // a block's first tile is its own, the others follow in order
    if (tid == 0) {
        s_cur = load_tile(item_tile(blockIdx.x));
        s_left = 0;
        s_seen = (int)gridDim.x;
    }
    bool split = false;                         // the first tiles of the order: any list of several parts?
    for (int pos = tid; pos < min(n, kHelpTiles); pos += NT) {
        const unsigned t = order ? order[pos] : (unsigned)pos;
        split |= offsets[t + 1] - offsets[t] > CH * part_chunks;
    }
    if (tid < NK) shist[tid] = 0u;
    for (int p = tid; p < PP * TH; p += NT) spA[p] = spB[p] = make_float4(0.f, 0.f, 0.f, 0.f);
    const bool any_split = __syncthreads_or(split);

    for (;;) {
        int tile = s_cur.x;
        unsigned start = (unsigned)s_cur.y, end = (unsigned)s_cur.z;
        const bool first = tile >= 0;                   // this block took the tile: it sums its background terms
        if (!first) {
            if (!any_split) break;
            __syncthreads();
            if (tid == 0) s_part = 0u;
            __syncthreads();
            unsigned best = 0u;                         // a random number and the position, 0: none
            for (int pos = tid; pos < min(n, kHelpTiles); pos += NT) {
                const unsigned t = order ? order[pos] : (unsigned)pos;
                const unsigned np = (offsets[t + 1] - offsets[t] + CH * part_chunks - 1) / (CH * part_chunks);
                if (np > 1 && __ldcg(parts + t) < np) {
                    const unsigned h = ((unsigned)pos * 2654435761u ^ (blockIdx.x + 1u) * 2246822519u) * 3266489917u;
                    best = max(best, (h & ~(unsigned)(kHelpTiles - 1)) | (unsigned)pos | (unsigned)kHelpTiles);
                }
            }
            best = __reduce_max_sync(0xffffffffu, best);
            if (lane == 0 && best) atomicMax(&s_part, best);
            __syncthreads();
            best = s_part;
            if (best == 0u) break;
            __syncthreads();                            // s_part is read: the parts below write it again
            best &= (unsigned)(kHelpTiles - 1);
            tile = order ? (int)order[best] : (int)best;
            start = offsets[tile];
            end = offsets[tile + 1];
        }
        const TileCoord tc = tile_coord(vs, tile);
        const View& V = vs.v[tc.v];
        const int x_org = tc.tx * TW, y_org = tc.ty * TH;
        const int x_lim = min(TW, V.W - x_org);         // pixels of the tile inside the image
        const int y_lim = min(TH, V.H - y_org);

        const unsigned per_part = CH * part_chunks, n_parts = (end - start + per_part - 1) / per_part;
        float4 bg = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int k = 0; k < (TW * TH > NT ? TW * TH / NT : 1); ++k) {
            const int p = tid + k * NT, ly = p / TW, lx = p - ly * TW;
            float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
            if (lx < x_lim && ly < y_lim) {
                const long long pix = V.pix_base + (long long)(y_org + ly) * V.W + x_org + lx;
                const float inv = 1.0f / out_den[pix];
                const float G0 = grad_rgb[3 * pix], G1 = grad_rgb[3 * pix + 1], G2 = grad_rgb[3 * pix + 2];
                const float C0 = out_rgb[3 * pix], C1 = out_rgb[3 * pix + 1], C2 = out_rgb[3 * pix + 2];
                f = make_float4(G0 * inv, G1 * inv, G2 * inv, -(G0 * C0 + G1 * C1 + G2 * C2) * inv);
                // dL/dw_B = G.(c_B - C)/D,  dL/dc_B = G w_B / D
                bg.x += f.x * __ldg(wparams + 3) + f.y * __ldg(wparams + 4) + f.z * __ldg(wparams + 5) + f.w;
                bg.y += f.x * wB;
                bg.z += f.y * wB;
                bg.w += f.z * wB;
            }
            if (TW * TH >= NT || p < TW * TH) {
                const int pi = 4 * (ly * PP + (lx >> 1)) + (lx & 1);
                reinterpret_cast<float*>(spA)[pi] = f.x;
                reinterpret_cast<float*>(spA)[pi + 2] = f.y;
                reinterpret_cast<float*>(spB)[pi] = f.z;
                reinterpret_cast<float*>(spB)[pi + 2] = f.w;
            }
        }
        if (first) {
            bg = make_float4(warp_sum(bg.x), warp_sum(bg.y), warp_sum(bg.z), warp_sum(bg.w));
            if (lane == 0) sbg[warp] = bg;
        }
        for (unsigned part = 0;; ++part) {
            if (n_parts > 1) {
                if (tid == 0) s_part = atomicAdd(parts + tile, 1u);
                __syncthreads();
                part = s_part;
            }
            if (part >= n_parts) break;
            const unsigned part_end = min(end, start + (part + 1) * per_part);
            for (unsigned base = start + part * per_part; base < part_end; base += CH) {
                const int cnt = (int)min((unsigned)CH, part_end - base);
                // ---- A: record, rows and class of a Gaussian per thread ----
#pragma unroll 1
                for (int gj = tid; gj < cnt; gj += NT) {
                    const unsigned r = list[base + gj];
                    const float4* pr = rec + 3ull * r;
                    const float4 a = __ldg(pr), b = __ldg(pr + 1);
                    const float cb = __ldg(reinterpret_cast<const float*>(pr + 2));
                    s0[gj] = a;
                    s1[gj] = b;
                    s2[gj] = f2(cb, b.y);
                    sidx[gj] = r;
                    int row, nst;
                    bool wide;
                    Footprint(a, b.x).rows<TW>(a, b.x, (float)x_org + 0.5f - a.x, (float)y_org + 0.5f - a.y, x_lim, y_lim,
                                               row, nst, wide);
                    const int key = nst + (wide ? NB : 0);
                    sfirst[gj] = (unsigned char)row;
                    snst[gj] = (unsigned char)nst;
                    skey[gj] = (unsigned char)key;
                    srank[gj] = (unsigned short)atomicAdd(&shist[key], 1u);
                }
                if (tid < 2) snext[tid] = 0u;
                __syncthreads();
                // ---- B: the chunk's order, wide first, most rows first: each warp forms the buckets' starts (the
                // counts of all larger keys, a suffix scan over the NK <= 64 keys held two per lane), and a
                // Gaussian's position is its bucket's start plus its rank in the bucket ----
                const unsigned h0 = lane < NK ? shist[lane] : 0u, h1 = lane + 32 < NK ? shist[lane + 32] : 0u;
                unsigned s0i = h0, s1i = h1;                    // inclusive suffix sums of keys lane and lane + 32
#pragma unroll
                for (int off = 1; off < 32; off <<= 1) {
                    const unsigned y0 = __shfl_down_sync(0xffffffffu, s0i, off), y1 = __shfl_down_sync(0xffffffffu, s1i, off);
                    if (lane + off < 32) {
                        s0i += y0;
                        s1i += y1;
                    }
                }
                s0i += __shfl_sync(0xffffffffu, s1i, 0);        // keys 32.. lie above every key of the first half
                const unsigned start0 = s0i - h0, start1 = s1i - h1;
                const int nwide = (int)__shfl_sync(0xffffffffu, s0i, NB);   // Gaussians with keys NB and up: the wide
                static_assert(NB < 32, "the wide class starts in the first half of the keys");
                for (int g0 = warp * 32; g0 < cnt; g0 += NT) {
                    const int gj = g0 + lane;
                    const int key = gj < cnt ? (int)skey[gj] : 0;
                    const unsigned a0 = __shfl_sync(0xffffffffu, start0, key & 31);
                    const unsigned a1 = __shfl_sync(0xffffffffu, start1, key & 31);
                    if (gj < cnt) sord[(key < 32 ? a0 : a1) + srank[gj]] = (unsigned short)gj;
                }
                __syncthreads();
                if (tid < NK) shist[tid] = 0u;                  // for the next chunk (step C does not read it)
                // ---- C: a group per Gaussian; each warp takes the next 32 / L Gaussians of a class ----
                auto walk = [&](auto lanes, const int lo, const int hi, unsigned* next) {
                    constexpr int L = decltype(lanes)::value, RP = decltype(lanes)::rows, LT = L * RP;
                    constexpr int GW = 32 / LT;                 // groups per warp
                    const int grp = lane / LT, gk = lane % L, rp = lane % LT / L;    // group, column lane and row lane
                    for (;;) {
                        unsigned at0 = 0;
                        if (lane == 0) at0 = atomicAdd(next, (unsigned)GW);
                        at0 = __shfl_sync(0xffffffffu, at0, 0);
                        if (lo + (int)at0 >= hi) break;
                        const int so = lo + (int)at0 + grp;
                        const bool act = so < hi;
                        const int j = act ? (int)sord[so] : 0;
                        const int steps = act ? (int)snst[j] : 0;
                        const int r0 = act ? (int)sfirst[j] : 0;
                        const float4 a = s0[j], b = s1[j];
                        const float2 c2 = s2[j];
                        const float gx0 = (float)x_org + 0.5f - a.x;                 // dx of column 0
                        const float gy0 = (float)y_org + 0.5f - a.y;                 // dy of row 0
                        const float qs = a.z;
                        const float2 qw2 = f2(a.w, a.w), qd2 = f2(b.x, b.x), gx2 = f2(gx0, gx0);
                        // dL/dq' = e (P . cw) with cw = -ln2 u w (c, 1): the walk uses the colour c = (c u w) / (u w)
                        // (in both halves of a pair) and applies the factor -ln2 u w to the moments once, after it
                        const float iuw = c2.y != 0.0f ? 1.0f / c2.y : 0.0f;
                        const float2 ccr = f2(b.z * iuw, b.z * iuw), ccg = f2(b.w * iuw, b.w * iuw);
                        const float2 ccb = f2(c2.x * iuw, c2.x * iuw);
                        // accumulators, each over the two pixels of a column pair: d/d(c u w) per channel, d/d(u w);
                        // and the moments of gq = dL/dq' in the record's own frame (r = qs dy + qw dx, dx):
                        // sum gq r^2, sum gq r dx, sum gq dx^2, sum gq r, sum gq dx.  Kept apart, a thin
                        // footprint's small along-axis terms (dx) are not rounded away under its large r terms.
                        float2 gr = f2(0.f, 0.f), gg = gr, gb = gr, gu = gr;
                        float2 srr = f2(0.f, 0.f), srx = srr, sxx = srr, sr = srr, sx = srr;
                        // dx of this lane's first column pair (2 k, 2 k + 1) from the row's even first column, less that column
                        const float2 gxb = __fadd2_rn(f2((float)(2 * gk), (float)(2 * gk + 1)), gx2);
                        const Footprint fp(a, b.x);
                        const float left = -gx0 - 0.025f;                               // columns, with a little slack
                        int row = (r0 + rp) * PP + gk - __float_as_int(kMagic);
                        const float yend = (float)(r0 + steps);
                        for (float yf = (float)(r0 + rp); yf < yend; row += RP * PP, yf += (float)RP) {
                            const float dy = yf + gy0, rb = qs * dy;
                            // the row's first column v (not beyond the last pair), rounded up and then down to even:
                            // round(v / 2), by adding a number whose last bit weighs one
                            const float v = fmaf(-fp.slope, dy, left) - sqrt_approx(fmaxf(fmaf(-fp.h1 * dy, dy, fp.h0), 0.0f));
                            const float w = fmaf(fminf(fmaxf(v, 0.0f), (float)(TW - 2)), 0.5f, kMagic);
                            const int pb = row + __float_as_int(w);
                            const float xsf = fmaf(w, 2.0f, -2.0f * kMagic);
                            const float2 xb = __fadd2_rn(f2(xsf, xsf), gxb);             // dx of the lane's first pair
                            const float2 rb2 = f2(rb, rb);
#pragma unroll
                            for (int m = 0; m < M; ++m) {
                                // Columns outside the footprint evaluate q > 9, so the cutoff test zeroes them; pairs past
                                // the tile and rows past the image read zero pairs.  No per-pixel mask is needed.
                                const int pi = pb + m * L;
                                const float4 A = spA[pi], B = spB[pi];          // (x0, x1, y0, y1), (z0, z1, w0, w1)
                                const float2 dx = m == 0 ? xb : __fadd2_rn(xb, f2((float)(2 * m * L), (float)(2 * m * L)));
                                const float2 rr = __ffma2_rn(qw2, dx, rb2);
                                const float2 q = __ffma2_rn(rr, rr, __fmul2_rn(__fmul2_rn(qd2, dx), dx));
                                const float2 e = f2(ex2_approx(q.x <= kQMax ? -q.x : -256.0f),      // 2^-256 flushes to 0
                                                    ex2_approx(q.y <= kQMax ? -q.y : -256.0f));
                                // d/d(c u w) and d/d(u w) at fixed c u w
                                gr = __ffma2_rn(f2(A.x, A.y), e, gr);
                                gg = __ffma2_rn(f2(A.z, A.w), e, gg);
                                gb = __ffma2_rn(f2(B.x, B.y), e, gb);
                                gu = __ffma2_rn(f2(B.z, B.w), e, gu);
                                // dL/dq' per pixel, less the factor -ln2 u w: e * (P_w + c . P_rgb)
                                const float2 pc = __ffma2_rn(f2(B.x, B.y), ccb, __ffma2_rn(f2(A.z, A.w), ccg,
                                                             __ffma2_rn(f2(A.x, A.y), ccr, f2(B.z, B.w))));
                                const float2 gq = __fmul2_rn(e, pc);
                                const float2 tr = __fmul2_rn(gq, rr), tx = __fmul2_rn(gq, dx);
                                srr = __ffma2_rn(tr, rr, srr);
                                srx = __ffma2_rn(tr, dx, srx);
                                sxx = __ffma2_rn(tx, dx, sxx);
                                sr = __fadd2_rn(sr, tr);
                                sx = __fadd2_rn(sx, tx);
                            }
                        }
                        // the group's sums: record order sum gq r, sum gq dx, sum gq r^2, sum gq r dx, sum gq dx^2,
                        // d/d(u w), d/d(c u w)
                        const float fq = -kLn2 * c2.y;
                        float vals[9] = {fq * (sr.x + sr.y), fq * (sx.x + sx.y), fq * (srr.x + srr.y), fq * (srx.x + srx.y),
                                         fq * (sxx.x + sxx.y), gu.x + gu.y, gr.x + gr.y, gg.x + gg.y, gb.x + gb.y};
                        __syncwarp();
#pragma unroll
                        for (int off = LT / 2; off > 0; off >>= 1)
#pragma unroll
                            for (int c = 0; c < 9; ++c) vals[c] += __shfl_xor_sync(0xffffffffu, vals[c], off);
                        const bool add = act && lane % LT == 0 && steps > 0;        // the group's lane with its sums
                        if constexpr (!DET) {
                            if (add) {
                                float4* o = reinterpret_cast<float4*>(grec + (size_t)WSR_GRAD_RECORD_FLOATS * sidx[j]);
                                atomicAdd(o, make_float4(vals[0], vals[1], vals[2], vals[3]));
                                atomicAdd(o + 1, make_float4(vals[4], vals[5], vals[6], vals[7]));
                                atomicAdd(reinterpret_cast<float*>(o + 2), vals[8]);
                            }
                        } else {
                            // deterministic mode: a 128-byte record holds 9 int64 sums, then the 9 bounds (float
                            // bits) that fix their units.  A term's bound caps the sum of its absolute pixel
                            // terms over the whole footprint, the same in every tile of the Gaussian: at most
                            // (2 hx + 2)(2 hy + 2) pixels (hx, hy its half-extents), each with e <= 1, every
                            // pixel-table entry at most pmax, |r| <= sqrt(QM), |dx| <= hx inside the cutoff.
                            // The sums go out through shared memory, so that consecutive lanes form and add consecutive
                            // words of a record.
                            if (add) {
                                constexpr float QM = kQMax * 1.0001f + 1e-4f;
                                const float qd = b.x, hx = sqrtf(QM / qd);
                                const float hy = sqrtf(QM * fmaf(a.w, a.w, qd) / (qd * a.z * a.z));
                                const float npx = fminf((2.0f * hx + 2.0f) * (2.0f * hy + 2.0f), 1e12f);
                                const float gqm = pmax * kLn2 * 1.0001f * (fabsf(b.z) + fabsf(b.w) + fabsf(c2.x) + fabsf(b.y));
                                const float sq = sqrtf(QM);
                                float* const o = grec + (size_t)kDetRecordFloats * sidx[j] + 18;
                                auto bound = [&](int c, float m) {
                                    m = fminf(m, 1e30f);
                                    int e = kNoBound - kExpBias;
                                    if (m > 0.0f) frexpf(m, &e);    // m < 2^e
                                    e += kExpBias;
                                    s_exp[warp][grp][c] = (signed char)e;
                                    return m;
                                };
#pragma unroll
                                for (int c = 0; c < 9; ++c) s_val[warp][grp][c] = vals[c];
                                // every tile of the Gaussian writes the same bounds (and a zero in the padding)
                                *reinterpret_cast<float2*>(o) = f2(bound(0, npx * gqm * sq), bound(1, npx * gqm * hx));
                                *reinterpret_cast<float4*>(o + 2) = make_float4(bound(2, npx * gqm * QM),
                                                                                bound(3, npx * gqm * sq * hx),
                                                                                bound(4, npx * gqm * hx * hx),
                                                                                bound(5, npx * pmax));
                                const float m = bound(6, npx * pmax);
                                *reinterpret_cast<float4*>(o + 6) = make_float4(m, bound(7, npx * pmax), bound(8, npx * pmax),
                                                                                0.0f);
                            }
                            if (lane % LT == 0) s_rec[warp][grp] = add ? sidx[j] : 0xffffffffu;
                            __syncwarp();
                            for (int k = lane; k < 9 * GW; k += 32) {
                                const int gi = k / 9, c = k - 9 * gi, e = s_exp[warp][gi][c];
                                const unsigned ri = s_rec[warp][gi];
                                if (ri != 0xffffffffu && e != kNoBound)
                                    atomicAdd(reinterpret_cast<unsigned long long*>(grec + (size_t)kDetRecordFloats * ri) + c,
                                              (unsigned long long)fixed_point(s_val[warp][gi][c], kDetBits + kExpBias - e));
                            }
                            __syncwarp();
                        }
                    }
                };
                // few Gaussians: more lanes each, so that every warp has some
                if (nwide > kFewWalk) walk(Lanes<TW / (2 * M), 1>(), 0, nwide, &snext[0]);        // the wide class
                else walk(Lanes<TW / (2 * M), 2>(), 0, nwide, &snext[0]);
                if (cnt - nwide > kFewWalk) walk(Lanes<TW / (4 * M), 1>(), nwide, cnt, &snext[1]);   // the narrow class
                else walk(Lanes<TW / (4 * M), 2>(), nwide, cnt, &snext[1]);
                __syncthreads();                                // this chunk is done with shared memory
            }
        }
        if (n_parts == 0) __syncthreads();                      // every thread has read s_cur, sbg is written
        if (first && warp == 0) {
            // the next tile: claimed already, or the next of the order, several at once while lists are short and many
            // tiles are left
            const int left = s_left, seen = s_seen;
            __syncwarp();
            if (left > 0) {
                if (lane == 0) {
                    s_cur = s_next[left - 1];
                    s_left = left - 1;
                }
            } else {
                const int count = end - start > kShortList ? 1 : min(max((n - seen) / (4 * (int)gridDim.x), 1), kClaim);
                int item = n;
                if (lane == 0 && (int)gridDim.x < n) item = (int)(gridDim.x + atomicAdd(counter, (unsigned)count));
                item = __shfl_sync(0xffffffffu, item, 0);
                if (lane < count) {
                    const int4 t = load_tile(item_tile((unsigned)(item + lane)));
                    if (lane == 0) s_cur = t;
                    else s_next[count - 1 - lane] = t;
                }
                if (lane == 0) {
                    s_left = count - 1;
                    s_seen = item;
                }
            }
        }
        if (first && tid >= 32 && tid < 36) {
            const int c = tid - 32;
            float t = 0.0f;
            for (int w = 0; w < NW; ++w) t += reinterpret_cast<const float*>(&sbg[w])[c];
            if constexpr (DET) bg_tiles[4 * (size_t)tile + c] = t;      // summed in tile order afterwards
            else if (t != 0.0f) atomicAdd(gw + 2 + c, t);
        }
        __syncthreads();                                        // s_cur is written, s_part and sbg read
    }
}

// Deterministic mode: the largest magnitude of the backward's pixel terms, G / D per channel and
// (G.C) / D, over all pixels (the same expressions as the backward's pixel table), as float bits
// with an order-independent integer atomicMax.
__global__ void __launch_bounds__(256) k_det_pmax(const float* __restrict__ out_rgb,
                                                  const float* __restrict__ out_den,
                                                  const float* __restrict__ grad_rgb, long long npix,
                                                  unsigned* __restrict__ pmax) {
    float m = 0.0f;
    for (long long pix = (long long)blockIdx.x * blockDim.x + threadIdx.x; pix < npix;
         pix += (long long)gridDim.x * blockDim.x) {
        const float inv = 1.0f / out_den[pix];
        const float G0 = grad_rgb[3 * pix], G1 = grad_rgb[3 * pix + 1], G2 = grad_rgb[3 * pix + 2];
        const float C0 = out_rgb[3 * pix], C1 = out_rgb[3 * pix + 1], C2 = out_rgb[3 * pix + 2];
        m = fmaxf(m, fmaxf(fmaxf(fabsf(G0 * inv), fabsf(G1 * inv)),
                           fmaxf(fabsf(G2 * inv), fabsf(-(G0 * C0 + G1 * C1 + G2 * C2) * inv))));
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
    if ((threadIdx.x & 31) == 0 && m > 0.0f) atomicMax(pmax, __float_as_uint(m));
}

// Deterministic mode: the tiles' background terms summed in a fixed order.
__global__ void __launch_bounds__(256) k_det_bg_reduce(const float* __restrict__ bg, int n_tiles,
                                                       float* __restrict__ gw) {
    __shared__ float part[4][8];
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 8
    for (int t = threadIdx.x; t < n_tiles; t += 256) {
        const float4 v = reinterpret_cast<const float4*>(bg)[t];
        acc[0] += v.x;
        acc[1] += v.y;
        acc[2] += v.z;
        acc[3] += v.w;
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const float t = warp_sum(acc[c]);
        if ((threadIdx.x & 31) == 0) part[c][threadIdx.x >> 5] = t;
    }
    __syncthreads();
    if (threadIdx.x < 4) {
        float sum = 0.0f;
#pragma unroll
        for (int k = 0; k < 8; ++k) sum += part[threadIdx.x][k];
        gw[2 + threadIdx.x] = sum;
    }
}

// As many blocks as fit on the device at once, kept in `known` (one per kernel).
template <typename K>
cudaError_t resident_blocks(PerDevice& known, K kernel, int threads, int& blocks) {
    return known.get(blocks, [&](int dev, int& out) {
        int sms = 0, per_sm = 0;
        cudaError_t e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, 0);
        out = max(1, sms * max(per_sm, 1));
        return e;
    });
}

// Records per 1024 pixels up to which the kernel for sparse views is taken (the lists' lengths are not known on the
// host).  It and the other, us, for Gaussians of size exp(-4), five units away, and wider ones:
//   1920x1080   500 (0.25 per 1024)   9.4, 17.5   exp(-2.5) 11.4, 24   exp(-1.5) 26.5, 36
//               8000 (4)             12.1, 23     exp(-2.5) 57, 56     exp(-1.5) 303, 264
//               20000 (10)           18.7, 27     exp(-3.5) 31, 35
//               32000 (16)           25.7, 31     exp(-2.5) 213, 174
//               50000 (25)           35.9, 37                           (not taken)
//   1280x720    10000 (11)            8.5, 12.7   exp(-3) 21.1, 20.7
//   979x543     8000 (15)             7.7, 9.8    exp(-2.5) 27, 21
//               10000 (19)            8.4, 9.8    exp(-3) 18.0, 15.2    (not taken)
// In 8x8 tiles, whose lists are shorter, 32000 at 1920x1080 take 26 and 32, 50000 at 1280x720 (56) 21.9 and 22.4, of
// exp(-3) 10000 at 979x543 (19) 17.1 and 16.4.  So near the limits Gaussians of a trained scene's size gain a fifth,
// and wide ones lose up to a third (the two cases of 27 and 213 took 30 and 214 before there were two kernels).  16000
// in two clusters of a hundred tiles take 151 and 85.  Deciding per tile (lists past 64 entries left to a second launch
// of the other kernel) gives the clusters 79 us, and takes 1.7 to 2 us from every sparse view.
//   A view with many records for its pixels has long lists, and they set the end of the whole batch: the sparse
// kernel's time lost there is about 0.5 us per record and 256 pixels of the densest view, and what it gains elsewhere
// 1.4 us per 1000 times 256 pixels, so in wide tiles it also needs 480 n <= all pixels / 256 times the densest view's
// / 256.  Frames of 2832 Gaussians in 846x566, 667x375 and 148x83 104 and 81 us, 4796 in 1334x750 and 222x222 97 and
// 83, 8569 in 1805x1015 and 539x539 80 and 88 (taken), 1037 in 1389x1389, 1098x1098 and 145x108 105 and 115 (taken).
constexpr long long kSparse = 16, kSparse8 = 40, kDenseView = 480;
inline bool sparse_view(const Views& vs, const long long n) {
    const long long pixels = vs.tile_w * vs.tile_h, all = vs.total_tiles * pixels;
    if (vs.total_tiles <= kFewTiles || n * vs.n * 1024 > (pixels == 64 ? kSparse8 : kSparse) * all) return false;
    if (pixels == 64) return true;
    long long least = all;
    for (int v = 0; v < vs.n; ++v) least = min(least, vs.v[v].tiles_x * vs.v[v].tiles_y * pixels);
    return kDenseView * n <= (all / 256) * (least / 256);
}

// S slices, or 0: the kernel for sparse views
template <int TW, int TH, int S>
cudaError_t fwd_s(const float* rec, const unsigned* off, const unsigned* list, const Views& vs, WeightDev w,
                  float* rgb, float* den, Sched sched, cudaStream_t s) {
    constexpr int NT = S ? 32 * S * FwdShape<TW, TH>::NR : 32 * LightShape<TW, TH>::NR;
    auto kernel = [] {
        if constexpr (S == 0) return k_render_fwd_light<TW, TH>;
        else return k_render_fwd<TW, TH, S>;
    }();
    static PerDevice known;
    int grid = vs.total_tiles;
    if (sched.order) {
        int most = 0;
        cudaError_t e = resident_blocks(known, kernel, NT, most);
        if (e == cudaSuccess && most < grid) e = cudaMemsetAsync(sched.counter, 0, sizeof(unsigned), s);
        if (e != cudaSuccess) return e;
        grid = min(grid, most);
    }
    kernel<<<(unsigned)grid, NT, 0, s>>>(reinterpret_cast<const float4*>(rec), off, list, vs, w.params, rgb, den, sched.order,
                                         sched.counter);
    return cudaGetLastError();
}

template <int TW, int TH>
cudaError_t fwd_t(const float* rec, long long n, const unsigned* off, const unsigned* list, const Views& vs, WeightDev w,
                  float* rgb, float* den, Sched sched, cudaStream_t s) {
    // Two slices where the tiles alone leave the SMs idle: 14.4 -> 10.4 us at 240 tiles, 14.5 -> 13.7 at 475
    // (40k Gaussians), 14.4 -> 15.1 at 920, 39 -> 70 at 8160.
    if (sparse_view(vs, n))
        return fwd_s<TW, TH, 0>(rec, off, list, vs, w, rgb, den, sched, s);
    return vs.total_tiles <= kFewTiles ? fwd_s<TW, TH, 2>(rec, off, list, vs, w, rgb, den, sched, s)
                                            : fwd_s<TW, TH, 1>(rec, off, list, vs, w, rgb, den, sched, s);
}

template <int TW, int TH, int CH>
cudaError_t bwd_chunk(const float* rec, const unsigned* off, const unsigned* list, const Views& vs, WeightDev w,
                      const float* rgb, const float* den, const float* grgb, float* grec, float* gw, bool det,
                      float* bg_tiles, const unsigned* det_pmax, const BwdSched& sched, cudaStream_t s) {
    constexpr int NT = BwdThreads<CH>::value;
    auto kernel = det ? k_render_bwd<TW, TH, CH, true> : k_render_bwd<TW, TH, CH, false>;
    static PerDevice known[2];
    int most = 0;
    cudaError_t e = resident_blocks(known[det], kernel, NT, most);
    if (e != cudaSuccess) return e;
    const long long want = 4ll * vs.total_tiles;
    kernel<<<(unsigned)min((long long)most, want), NT, 0, s>>>(reinterpret_cast<const float4*>(rec), off, list, vs, w.params, rgb,
                                                    den, grgb, grec, gw, bg_tiles, det_pmax, sched.order,
                                                    sched.counter, sched.counter + 1,
                                                    vs.total_tiles <= kFewTiles ? 1u : kPartChunks);
    return cudaGetLastError();
}

template <int TW, int TH>
cudaError_t bwd_t(const float* rec, const unsigned* off, const unsigned* list, const Views& vs, WeightDev w,
                  const float* rgb, const float* den, const float* grgb, float* grec, float* gw, bool det,
                  float* bg_tiles, const unsigned* det_pmax, const BwdSched& sched, cudaStream_t s) {
    const int ch = vs.chunk ? vs.chunk : vs.total_tiles <= kFewTiles ? 128 : 512;
    auto k = ch == 64 ? bwd_chunk<TW, TH, 64> : ch == 256 ? bwd_chunk<TW, TH, 256>
                                              : ch == 512 ? bwd_chunk<TW, TH, 512> : bwd_chunk<TW, TH, 128>;
    return k(rec, off, list, vs, w, rgb, den, grgb, grec, gw, det, bg_tiles, det_pmax, sched, s);
}

// Diagnostic: the work of the render kernels, three counts added to count[0..2]:
//   [0] (pixel, Gaussian) pairs inside the cutoff, i.e. the algorithmic work
//       (q' from each pixel's own dx, dy; the renderers may decide pairs
//       within rounding of the cutoff differently);
//   [1] the (pixel, Gaussian) slots the forward evaluates: per batch of a
//       tile's list and 8x8 region, rounds of four Gaussians that reach the
//       region (its own test), 256 slots each, in 8x8 tiles without the idle
//       quarters of the last one; in sparse views (`light`) the pixels of
//       each region of that kernel that a Gaussian reaches;
//   [2] the backward's pixel slots (per tile instance, the rows its footprint
//       reaches, TW columns each, or TW / 2 when no row needs more), from the
//       backward's own arithmetic.
template <int TW, int TH, int PPT>
__global__ void __launch_bounds__(TileShape<TW, TH, PPT>::NT)
    k_count_pairs(const float4* __restrict__ rec, const unsigned* __restrict__ offsets,
                  const unsigned* __restrict__ list, const Views vs, const bool light,
                  unsigned long long* __restrict__ count) {
    using S = TileShape<TW, TH, PPT>;
    using G = LightShape<TW, TH>;
    constexpr int NT = S::NT;
    using F = FwdShape<TW, TH>;
    static_assert(NT == 32 * F::NR, "the forward's batches");
    __shared__ float4 s0[NT];
    __shared__ float s1[NT];
    __shared__ unsigned s_n[F::NR];
    const int tile = blockIdx.x;
    const TileCoord tc = tile_coord(vs, tile);
    const View& V = vs.v[tc.v];
    const int tid = threadIdx.x;
    const int lx = tid % TW, ly = tid / TW;
    const int x = tc.tx * TW + lx;
    const int y0 = tc.ty * TH + ly * PPT;
    const float px = (float)x + 0.5f;
    const int x_org = tc.tx * TW, y_org = tc.ty * TH;
    const int x_lim = min(TW, V.W - x_org), y_lim = min(TH, V.H - y_org);
    unsigned long long cnt_pairs = 0, cnt_fwd = 0, cnt_bwd = 0;
    const unsigned start = offsets[tile], end = offsets[tile + 1];
    for (unsigned base = start; base < end; base += NT) {
        const int cnt = (int)min((unsigned)NT, end - base);
        __syncthreads();
        unsigned hit = 0u;
        if (tid < F::NR) s_n[tid] = 0u;
        if (tid < cnt) {
            const float4* p = rec + 3ull * list[base + tid];
            const float4 a = __ldg(p);
            const float qd = __ldg(reinterpret_cast<const float*>(p + 1));
            s0[tid] = a;
            s1[tid] = qd;
            const float gx = (float)x_org + 0.5f - a.x, gy = (float)y_org + 0.5f - a.y;
            if (!light) hit = regions_hit<F::RX, F::RY>(a, qd, gx, gy);
            else if (G::NR == 1) cnt_fwd += G::RW * 8;
            else
                for (int k = 0; k < G::NR; ++k)         // one region at a time, as its warps do
                    cnt_fwd += G::RW * 8 * regions_hit<1, 1, G::RW>(a, qd, gx + (float)(G::RW * (k % G::RX)),
                                                                    gy + (float)(8 * (k / G::RX)));
            // the backward's pixel slots: the rows its footprint reaches, TW or TW / 2 columns each
            int first, nst;
            bool wide;
            Footprint(a, qd).rows<TW>(a, qd, (float)x_org + 0.5f - a.x, (float)y_org + 0.5f - a.y, x_lim, y_lim, first,
                                      nst, wide);
            cnt_bwd += (unsigned long long)(nst * (wide ? TW : TW / 2));
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < F::NR; ++k) {
            const unsigned bal = __ballot_sync(0xffffffffu, (hit >> k) & 1u);
            if ((tid & 31) == 0 && bal) atomicAdd(&s_n[k], (unsigned)__popc(bal));
        }
        __syncthreads();
        // the forward's rounds over this batch: 256 slots each (one region per tile: 64 per Gaussian; none if light)
        if (tid < F::NR) cnt_fwd += F::NR > 1 ? 256ull * ((s_n[tid] + 3u) >> 2) : 64ull * s_n[tid];
        if (x >= V.W) continue;
        for (int j = 0; j < cnt; ++j) {
            const float4 a = s0[j];
            const float dx = px - a.x;
            const float P = s1[j] * dx * dx;
            const float Q = a.w * dx;
#pragma unroll
            for (int k = 0; k < PPT; ++k) {
                const float dy = (float)(y0 + k) + 0.5f - a.y;
                const float rr = fmaf(a.z, dy, Q);
                const float q = fmaf(rr, rr, P);
                if (q <= kQMax && y0 + k < V.H) ++cnt_pairs;
            }
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        cnt_pairs += __shfl_xor_sync(0xffffffffu, cnt_pairs, off);
        cnt_fwd += __shfl_xor_sync(0xffffffffu, cnt_fwd, off);
        cnt_bwd += __shfl_xor_sync(0xffffffffu, cnt_bwd, off);
    }
    if ((tid & 31) == 0) {
        if (cnt_pairs) atomicAdd(count, cnt_pairs);
        if (cnt_fwd) atomicAdd(count + 1, cnt_fwd);
        if (cnt_bwd) atomicAdd(count + 2, cnt_bwd);
    }
}

// Mean absolute error and its gradient: float4 loads and stores (the arrays are 16-byte aligned;
// a scalar tail covers count % 4), then a block reduction and one atomic per block.
__global__ void __launch_bounds__(256) k_loss_l1(const float* __restrict__ rgb, const float* __restrict__ target,
                                                 long long count, float* __restrict__ loss,
                                                 float* __restrict__ grad) {
    __shared__ float red[8];
    const float inv = 1.0f / (float)count;
    auto sgn = [&](float d) { return d > 0.0f ? inv : (d < 0.0f ? -inv : 0.0f); };
    float acc = 0.0f;
    const long long n4 = count >> 2;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += stride) {
        const float4 a = reinterpret_cast<const float4*>(rgb)[i];
        const float4 b = reinterpret_cast<const float4*>(target)[i];
        const float4 d = make_float4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w);
        acc += (fabsf(d.x) + fabsf(d.y)) + (fabsf(d.z) + fabsf(d.w));
        reinterpret_cast<float4*>(grad)[i] = make_float4(sgn(d.x), sgn(d.y), sgn(d.z), sgn(d.w));
    }
    for (long long i = 4 * n4 + (long long)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += stride) {
        const float d = rgb[i] - target[i];
        acc += fabsf(d);
        grad[i] = sgn(d);
    }
    acc = warp_sum(acc);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        float t = 0.0f;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
        atomicAdd(loss, t * inv);
    }
}

}  // namespace

cudaError_t sm_count(int& sms) {
    static PerDevice known;
    return known.get(sms, [](int dev, int& out) {
        return cudaDeviceGetAttribute(&out, cudaDevAttrMultiProcessorCount, dev);
    });
}

cudaError_t launch_render_fwd(const float* rec, long long n, const unsigned* off, const unsigned* list, const Views& vs,
                              WeightDev w, float* rgb, float* den, Sched sc, cudaStream_t s) {
    if (vs.total_tiles == 0) return cudaSuccess;
    if (vs.tile_w == 16 && vs.tile_h == 16) return fwd_t<16, 16>(rec, n, off, list, vs, w, rgb, den, sc, s);
    if (vs.tile_w == 8 && vs.tile_h == 8) return fwd_t<8, 8>(rec, n, off, list, vs, w, rgb, den, sc, s);
    if (vs.tile_w == 32 && vs.tile_h == 8) return fwd_t<32, 8>(rec, n, off, list, vs, w, rgb, den, sc, s);
    if (vs.tile_w == 16 && vs.tile_h == 8) return fwd_t<16, 8>(rec, n, off, list, vs, w, rgb, den, sc, s);
    return cudaErrorInvalidValue;
}

cudaError_t launch_render_bwd(const float* rec, const unsigned* off, const unsigned* list, const Views& vs,
                              WeightDev w, const float* rgb, const float* den, const float* grgb, float* grec,
                              float* gw, bool det, float* bg_tiles, const unsigned* det_pmax, const BwdSched& sc,
                              cudaStream_t s) {
    if (vs.total_tiles == 0) return cudaSuccess;
    if (vs.tile_w == 16 && vs.tile_h == 16)
        return bwd_t<16, 16>(rec, off, list, vs, w, rgb, den, grgb, grec, gw, det, bg_tiles, det_pmax, sc, s);
    if (vs.tile_w == 8 && vs.tile_h == 8)
        return bwd_t<8, 8>(rec, off, list, vs, w, rgb, den, grgb, grec, gw, det, bg_tiles, det_pmax, sc, s);
    if (vs.tile_w == 32 && vs.tile_h == 8)
        return bwd_t<32, 8>(rec, off, list, vs, w, rgb, den, grgb, grec, gw, det, bg_tiles, det_pmax, sc, s);
    if (vs.tile_w == 16 && vs.tile_h == 8)
        return bwd_t<16, 8>(rec, off, list, vs, w, rgb, den, grgb, grec, gw, det, bg_tiles, det_pmax, sc, s);
    return cudaErrorInvalidValue;
}

cudaError_t launch_det_pmax(const float* out_rgb, const float* out_den, const float* grad_rgb, long long npix,
                            unsigned* pmax, cudaStream_t s) {
    if (npix == 0) return cudaSuccess;
    int sms = 0;
    cudaError_t e = sm_count(sms);
    if (e != cudaSuccess) return e;
    const long long blocks = min((npix + 255) / 256, (long long)sms * 8);
    k_det_pmax<<<(unsigned)blocks, 256, 0, s>>>(out_rgb, out_den, grad_rgb, npix, pmax);
    return cudaGetLastError();
}

cudaError_t launch_det_bg_reduce(const float* bg_tiles, int n_tiles, float* gw, cudaStream_t s) {
    k_det_bg_reduce<<<1, 256, 0, s>>>(bg_tiles, n_tiles, gw);
    return cudaGetLastError();
}

cudaError_t launch_count_pairs(const float* rec, long long n, const unsigned* off, const unsigned* list, const Views& vs,
                               unsigned long long* count, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(count, 0, 3 * sizeof(unsigned long long), s);
    if (e != cudaSuccess || vs.total_tiles == 0) return e;
    const float4* r = reinterpret_cast<const float4*>(rec);
    const bool light = sparse_view(vs, n);
    if (vs.tile_w == 16 && vs.tile_h == 16) k_count_pairs<16, 16, 2><<<vs.total_tiles, 128, 0, s>>>(r, off, list, vs, light, count);
    else if (vs.tile_w == 8 && vs.tile_h == 8) k_count_pairs<8, 8, 2><<<vs.total_tiles, 32, 0, s>>>(r, off, list, vs, light, count);
    else if (vs.tile_w == 32 && vs.tile_h == 8) k_count_pairs<32, 8, 2><<<vs.total_tiles, 128, 0, s>>>(r, off, list, vs, light, count);
    else if (vs.tile_w == 16 && vs.tile_h == 8) k_count_pairs<16, 8, 2><<<vs.total_tiles, 64, 0, s>>>(r, off, list, vs, light, count);
    else return cudaErrorInvalidValue;
    return cudaGetLastError();
}

cudaError_t launch_loss_l1(const float* rgb, const float* target, long long count, float* loss, float* grad,
                           cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(loss, 0, sizeof(float), s);
    if (e != cudaSuccess || count == 0) return e;
    int sms = 0;
    e = sm_count(sms);
    if (e != cudaSuccess) return e;
    long long nb = (count / 4 + 255) / 256;
    const long long cap = 4ll * sms;
    if (nb > cap) nb = cap;
    if (nb < 1) nb = 1;
    k_loss_l1<<<(unsigned)nb, 256, 0, s>>>(rgb, target, count, loss, grad);
    return cudaGetLastError();
}

}  // namespace wsr
