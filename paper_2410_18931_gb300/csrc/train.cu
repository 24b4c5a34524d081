// Training step around the renderer: the 3DGS rendering loss the paper
// trains with (Sec. 4.4: L1 + 0.2 D-SSIM) with its gradient, and the Adam
// update of the parameters.
//
// Loss.  A block per strip of pixel columns and segment of rows of one view
// filters the local statistics (mu_x, mu_y, E[x^2 + y^2], E[xy]) separably
// with the 11-tap Gaussian (zero outside the image), forms the SSIM map and
// the three partials of the loss with respect to (mu_x, E[x^2], E[xy]), and
// filters those back (the window is symmetric, so the filter is its own
// adjoint) to the gradient of the segment's pixels.  L1 and SSIM sums go to the
// loss with one atomic per block and quantity.
//
// Adam.  One pass over a flat parameter buffer in float4 units, groups of
// contiguous elements with their own learning rates.  The step count and the
// bias corrections live in device memory (a one-thread kernel advances them),
// so a captured CUDA graph replays correct steps; both kernels leave
// everything untouched when a guard workspace recorded an error (a tile list
// that overflowed in the same step).
#include <mutex>

#include "wsr_common.cuh"
#include "wsr_launch.h"

namespace wsr {
namespace {

// Loss: the images are taken as rows of 3 W floats (the channels interleaved, as stored).  A block walks down a strip
// of kOP pixel columns, kTap rows at a time:
//   1. a thread per staged float column reads its next rows (coalesced) and filters x, y, x^2 + y^2 and (x - y)^2
//      vertically, eleven partial sums per quantity in registers.  SSIM's factor (2 cov + c2) / (var + var + c2) is
//      1 - D / (var + var + c2) with D the variance of x - y, so these four are enough, and where the images are
//      alike the cancellation in the variances hardly reaches it (gradient against 64 bits on smooth images: 1.3e-5
//      relative with the covariance, 1.1e-5 so; on noise 1.3e-7 either way);
//   2. the rows' horizontal filter, five neighbouring pixels of a channel per item, gives the statistics; the SSIM map
//      and its three partials follow;
//   3. a thread per statistics column filters the partials vertically, as in 1;
//   4. their horizontal filter, as in 2; 5. the gradient, a thread per output column.
// The strip's halo is 20 pixel columns (85 for 65) and the segment's 20 rows, where a 32x32 tile needed 52x52 staged
// pixels, staged through shared memory once per channel.  Bound by instruction issue (61 % of the cycles of two blocks
// of eight warps, the rest the batch's five barriers): a filter's tap on two quantities is one instruction, and the
// instructions fell from 9.4e7 to 6.8e7 at 1920x1080.  Tiles -> strips, us: 1080p 127 -> 96, 720p 66 -> 56,
// 979x543 43 -> 40, 640x360 24.7 -> 24.5, 320x180 18.1 -> 16.5, 3840x2160 474 -> 352.
constexpr int kTap = 11;                    // taps of the window, and rows per batch
constexpr int kOP = 65, kTP = kOP + 10, kSP = kOP + 20;     // output, statistics and staged pixels of a strip
constexpr int kVW = 91, kPW = 75;           // pixels per channel and row in shared memory (3 mod 8: a thread per
                                            // column writes three channels side by side without bank conflicts)
constexpr int kLossThreads = 256;
constexpr int kLossSmem = (kTap * 3 * (kVW + kPW)) * (int)sizeof(float4);
static_assert(3 * kSP <= kLossThreads && kTP % 5 == 0 && kOP % 5 == 0 && kVW >= kSP && kPW >= kTP, "layout");

__device__ __forceinline__ float block_sum_to(float x, float* red) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
    const int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) red[w] = x;
    __syncthreads();
    float t = 0.f;
    if (threadIdx.x == 0)
        for (int k = 0; k < (int)(blockDim.x >> 5); ++k) t += red[k];
    return t;   // valid in thread 0
}

__global__ void __launch_bounds__(kLossThreads, 2) k_loss_3dgs(const float* __restrict__ rgb,
                                                               const float* __restrict__ tgt, const LossViews L,
                                                               float* __restrict__ loss, float* __restrict__ grad) {
    extern __shared__ __align__(16) float4 sm[];
    float4* const sv = sm;                          // [kTap][3][kVW] vertically filtered; at the end F of the outputs
    float4* const sp = sm + kTap * 3 * kVW;         // [kTap][3][kPW] partials, then vertically filtered
    __shared__ float red[kLossThreads / 32];
    const int tid = threadIdx.x;
    int v = 0;
    while (v + 1 < L.n && (int)blockIdx.x >= L.tile_off[v + 1]) ++v;
    const int t = (int)blockIdx.x - L.tile_off[v];
    const int W = L.w[v], H = L.h[v];
    const int seg = t / L.tiles_x[v], x0 = (t - seg * L.tiles_x[v]) * kOP;
    const int r0 = seg * L.rows, rows = min(L.rows, H - r0);        // output rows r0 .. r0 + rows - 1
    const float* const img = rgb + L.pix_off[v] * 3;
    const float* const ref = tgt + L.pix_off[v] * 3;
    float* const out = grad + L.pix_off[v] * 3;
    const float gs = -L.lam * L.inv_count;                 // dL / d(SSIM map value)
    const float gl1 = (1.0f - L.lam) * L.inv_count;        // dL / d|x - y|
    const int px = tid / 3, ch = tid - 3 * px;             // this thread's column in steps 1, 3 and 5
    const int in_x = x0 - 10 + px;
    const bool in_col = px < kSP && in_x >= 0 && in_x < W;
    const long long in_at = 3ll * in_x + ch;
    const long long pitch = 3ll * W;
    float g[kTap];
#pragma unroll
    for (int k = 0; k < kTap; ++k) g[k] = L.g[k];
    // row q's partial sums lie in slot q mod 11; a batch's first row is a multiple of 11, so every slot is known here
    float2 a01[kTap], a23[kTap], b01[kTap];
    float b2[kTap];
#pragma unroll
    for (int k = 0; k < kTap; ++k) {
        a01[k] = a23[k] = b01[k] = f2(0.f, 0.f);
        b2[k] = 0.f;
    }
    float l1 = 0.f, ss = 0.f;
    const int batches = (rows + 20 + kTap - 1) / kTap;
    // a batch's first rows are loaded before the last one's steps 4 and 5, the others while the first are filtered
    constexpr int kAhead = 5;
    float2 xy[kTap];
    auto load_row = [&](int t) {
        const int y = r0 - 10 + t;
        if (!in_col || y < 0 || y >= H) return f2(0.f, 0.f);
        return f2(__ldg(img + (y * pitch + in_at)), __ldg(ref + (y * pitch + in_at)));
    };
#pragma unroll
    for (int i = 0; i < kAhead; ++i) xy[i] = load_row(i);
    for (int b = 0; b < batches; ++b) {
        const int t0 = kTap * b;                    // input row t is image row r0 - 10 + t
        // ---- 1: input row t adds g[d] times itself to statistics row t - d; row t - 10 is then complete ----
#pragma unroll
        for (int i = kAhead; i < kTap; ++i) xy[i] = load_row(t0 + i);
#pragma unroll
        for (int i = 0; i < kTap; ++i) {
            const float2 x = xy[i];
            const float dif = x.x - x.y;
            const float2 m = f2(fmaf(x.x, x.x, x.y * x.y), dif * dif);
#pragma unroll
            for (int d = 0; d < kTap; ++d) {
                const int k = (i - d + kTap) % kTap;
                a01[k] = d == 0 ? __fmul2_rn(f2(g[0], g[0]), x) : __ffma2_rn(f2(g[d], g[d]), x, a01[k]);
                a23[k] = d == 0 ? __fmul2_rn(f2(g[0], g[0]), m) : __ffma2_rn(f2(g[d], g[d]), m, a23[k]);
            }
            const int k = (i + 1) % kTap;
            if (px < kSP) sv[(i * 3 + ch) * kVW + px] = make_float4(a01[k].x, a01[k].y, a23[k].x, a23[k].y);
        }
        __syncthreads();
        // ---- 2: statistics row q (image row r0 - 5 + q), pixel j (image column x0 - 5 + j) ----
        for (int it = tid; it < kTap * 3 * (kTP / 5); it += kLossThreads) {
            const int i = it / (3 * (kTP / 5)), rest = it - i * (3 * (kTP / 5));
            const int c = rest / (kTP / 5), j0 = 5 * (rest - c * (kTP / 5));
            const int q = t0 + i - 10, y = r0 - 5 + q;
            const bool row_in = q >= 0 && q < rows + 10 && y >= 0 && y < H;
            float4* const dst = sp + (i * 3 + c) * kPW + j0;
            if (!row_in) {
#pragma unroll
                for (int o = 0; o < 5; ++o) dst[o] = make_float4(0.f, 0.f, 0.f, 0.f);
                continue;
            }
            float2 s01[5], s23[5];
#pragma unroll
            for (int o = 0; o < 5; ++o) s01[o] = s23[o] = f2(0.f, 0.f);
            const float4* const src = sv + (i * 3 + c) * kVW + j0;
#pragma unroll
            for (int k = 0; k < kTap + 4; ++k) {
                const float4 w = src[k];
#pragma unroll
                for (int o = 0; o < 5; ++o)
                    if (k - o >= 0 && k - o < kTap) {
                        s01[o] = __ffma2_rn(f2(g[k - o], g[k - o]), f2(w.x, w.y), s01[o]);
                        s23[o] = __ffma2_rn(f2(g[k - o], g[k - o]), f2(w.z, w.w), s23[o]);
                    }
            }
#pragma unroll
            for (int o = 0; o < 5; ++o) {
                const int x = x0 - 5 + j0 + o;
                float4 p = make_float4(0.f, 0.f, 0.f, 0.f);
                if (x >= 0 && x < W) {
                    const float mx = s01[o].x, my = s01[o].y, md = mx - my, mm = fmaf(mx, mx, my * my);
                    const float a1 = fmaf(2.f, mx * my, L.c1), b1 = mm + L.c1;
                    const float b2_ = (s23[o].x - mm) + L.c2, a2 = b2_ - fmaf(-md, md, s23[o].y);
                    const float ib1 = rcp_approx(b1), ib2 = rcp_approx(b2_), i12 = ib1 * ib2;
                    const float sval = a1 * a2 * i12;
                    p.x = 2.f * gs * fmaf(my * (a2 - a1), i12, mx * sval * (ib2 - ib1));
                    p.y = -gs * sval * ib2;
                    p.z = 2.f * gs * a1 * i12;
                    if (j0 + o >= 5 && j0 + o < 5 + kOP && q >= 5 && q < 5 + rows) ss += sval;
                }
                dst[o] = p;
            }
        }
        __syncthreads();
        // ---- 3: statistics row q adds to output row q - d; row q - 10 is then complete (in place) ----
        if (px < kTP) {
#pragma unroll
            for (int i = 0; i < kTap; ++i) {
                float4* const at = sp + (i * 3 + ch) * kPW + px;
                const float4 p = *at;
#pragma unroll
                for (int d = 0; d < kTap; ++d) {
                    const int k = (i + 1 - d + kTap) % kTap;            // q = 11 b + i - 10 is i + 1 mod 11
                    b01[k] = d == 0 ? __fmul2_rn(f2(g[0], g[0]), f2(p.x, p.y))
                                    : __ffma2_rn(f2(g[d], g[d]), f2(p.x, p.y), b01[k]);
                    b2[k] = d == 0 ? g[0] * p.z : fmaf(g[d], p.z, b2[k]);
                }
                const int k = (i + 2) % kTap;
                *at = make_float4(b01[k].x, b01[k].y, b2[k], 0.f);
            }
        }
#pragma unroll
        for (int i = 0; i < kAhead; ++i) xy[i] = load_row(t0 + kTap + i);
        if (t0 + kTap <= 20) continue;              // the first batch completes no output row
        __syncthreads();
        // ---- 4: output row n (image row r0 + n), pixel j (image column x0 + j) ----
        for (int it = tid; it < kTap * 3 * (kOP / 5); it += kLossThreads) {
            const int i = it / (3 * (kOP / 5)), rest = it - i * (3 * (kOP / 5));
            const int c = rest / (kOP / 5), j0 = 5 * (rest - c * (kOP / 5));
            const int n = t0 + i - 20;
            if (n < 0 || n >= rows) continue;
            float2 f01[5];
            float fz[5];
#pragma unroll
            for (int o = 0; o < 5; ++o) f01[o] = f2(0.f, 0.f), fz[o] = 0.f;
            const float4* const src = sp + (i * 3 + c) * kPW + j0;
#pragma unroll
            for (int k = 0; k < kTap + 4; ++k) {
                const float4 w = src[k];
#pragma unroll
                for (int o = 0; o < 5; ++o)
                    if (k - o >= 0 && k - o < kTap) {
                        f01[o] = __ffma2_rn(f2(g[k - o], g[k - o]), f2(w.x, w.y), f01[o]);
                        fz[o] = fmaf(g[k - o], w.z, fz[o]);
                    }
            }
            float4* const dst = sv + (i * 3 + c) * kVW + j0;
#pragma unroll
            for (int o = 0; o < 5; ++o) dst[o] = make_float4(f01[o].x, f01[o].y, fz[o], 0.f);
        }
        const bool out_col = px < kOP && x0 + px < W;
        const long long out_at = 3ll * (x0 + px) + ch;
        float2 ab[kTap];                                // step 5's pixels, loaded across the barrier
#pragma unroll
        for (int i = 0; i < kTap; ++i) {
            const int n = t0 + i - 20;
            ab[i] = f2(0.f, 0.f);
            if (out_col && n >= 0 && n < rows)
                ab[i] = f2(__ldg(img + ((r0 + n) * pitch + out_at)), __ldg(ref + ((r0 + n) * pitch + out_at)));
        }
        __syncthreads();
        // ---- 5: the gradient ----
        if (out_col) {
#pragma unroll
            for (int i = 0; i < kTap; ++i) {
                const int n = t0 + i - 20;
                if (n < 0 || n >= rows) continue;
                const float4 f = sv[(i * 3 + ch) * kVW + px];
                const float x = ab[i].x, y = ab[i].y, d = x - y;
                l1 += fabsf(d);
                const float gd = d > 0.f ? gl1 : (d < 0.f ? -gl1 : 0.f);
                out[(r0 + n) * pitch + out_at] = f.x + 2.f * x * f.y + y * f.z + gd;
            }
        }
        __syncthreads();
    }
    const float tl1 = block_sum_to(l1, red);
    __syncthreads();
    const float tss = block_sum_to(ss, red);
    if (tid == 0) {
        atomicAdd(loss, gl1 * tl1 + gs * tss + (blockIdx.x == 0 ? L.lam : 0.f));
        atomicAdd(loss + 1, tl1 * L.inv_count);
        atomicAdd(loss + 2, tss * L.inv_count);
    }
}

// The next step's number and bias corrections 1 / (1 - b1^t) and 1 / sqrt(1 - b2^t), a lane each.  One chain of FP64
// operations bounds it, so the powers are formed by squaring (2 log2 t products) beside each other: 9.4 us with two calls
// of pow() one after the other, 3.5 us.  A power's relative error grows as t 2^-53, and b^t damps it in 1 - b^t: below
// 2^-52 / (1 - b), 2e-13 for b = 0.999 and 2e-12 for 0.9999, far under the float results' 6e-8.
__global__ void k_adam_tick(AdamState* st, const WsHeader* guard, double b1, double b2) {
    if (guard && guard->err != 0) {
        if (threadIdx.x == 0) st->skipped += 1;
        return;
    }
    const int t = st->step + 1;
    double p = 1.0, b = threadIdx.x == 0 ? b1 : b2;
    for (unsigned k = (unsigned)t;; b *= b) {
        if (k & 1u) p *= b;
        if ((k >>= 1) == 0u) break;
    }
    const double d = 1.0 - p;
    const float c = (float)(1.0 / (threadIdx.x == 0 ? d : sqrt(d)));
    __syncwarp(3u);
    if (threadIdx.x == 0) {
        st->step = t;
        st->c1 = c;
    } else {
        st->c2 = c;
    }
}

__global__ void __launch_bounds__(256) k_adam(float* __restrict__ p, const float* __restrict__ g,
                                              float* __restrict__ m, float* __restrict__ v, const AdamGroups G,
                                              const AdamState* __restrict__ st, const WsHeader* guard) {
    if (guard && guard->err != 0) return;
    const float c1 = st->c1, c2 = st->c2;
    const long long units = G.ubase[G.n];
    for (long long u = (long long)blockIdx.x * blockDim.x + threadIdx.x; u < units;
         u += (long long)gridDim.x * blockDim.x) {
        int gi = 0;
        while (u >= G.ubase[gi + 1]) ++gi;
        const unsigned e0 = (unsigned)(u - G.ubase[gi]) * 4u;
        const long long at = G.off[gi] + e0;
        const unsigned left = G.cnt[gi] - e0;
        const unsigned per = (unsigned)G.period[gi];
        const unsigned r0 = per ? e0 % per : 0u;
        float lr[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            unsigned r = r0 + (unsigned)k;
            if (per) r = (r >= per) ? r - per * (r / per) : r;
            lr[k] = (per && r >= (unsigned)G.head[gi]) ? G.lr_tail[gi] : G.lr[gi];
        }
        if (left >= 4) {
            float4 pp = *reinterpret_cast<const float4*>(p + at);
            const float4 gg = *reinterpret_cast<const float4*>(g + at);
            float4 mv = *reinterpret_cast<const float4*>(m + at);
            float4 vv = *reinterpret_cast<const float4*>(v + at);
            float* P = &pp.x;
            const float* Gr = &gg.x;
            float* M = &mv.x;
            float* V = &vv.x;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                M[k] = fmaf(G.b1, M[k], G.omb1 * Gr[k]);
                V[k] = fmaf(G.b2, V[k], G.omb2 * Gr[k] * Gr[k]);
                P[k] -= lr[k] * c1 * M[k] / (sqrtf(V[k]) * c2 + G.eps);
            }
            *reinterpret_cast<float4*>(p + at) = pp;
            *reinterpret_cast<float4*>(m + at) = mv;
            *reinterpret_cast<float4*>(v + at) = vv;
        } else {
            for (unsigned k = 0; k < left; ++k) {
                const float gk = g[at + k];
                const float mk = fmaf(G.b1, m[at + k], G.omb1 * gk);
                const float vk = fmaf(G.b2, v[at + k], G.omb2 * gk * gk);
                m[at + k] = mk;
                v[at + k] = vk;
                p[at + k] -= lr[k] * c1 * mk / (sqrtf(vk) * c2 + G.eps);
            }
        }
    }
}

}  // namespace

cudaError_t launch_loss_3dgs(const float* rgb, const float* target, const LossViews& L, float* loss, float* grad,
                             cudaStream_t s) {
    constexpr int smem = kLossSmem;
    // the shared-memory opt-in is a per-device function attribute: set it once per device (thread-safe)
    static std::once_flag once[64];
    static cudaError_t once_err[64];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    std::call_once(once[dev], [&] {
        once_err[dev] = cudaFuncSetAttribute(k_loss_3dgs, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    });
    if (once_err[dev] != cudaSuccess) return once_err[dev];
    e = cudaMemsetAsync(loss, 0, 3 * sizeof(float), s);
    if (e != cudaSuccess) return e;
    const int tiles = L.tile_off[L.n];
    if (tiles == 0) return cudaSuccess;
    k_loss_3dgs<<<tiles, kLossThreads, smem, s>>>(rgb, target, L, loss, grad);
    return cudaGetLastError();
}

// Strips and segments of the views (tiles_x, tile_off, rows).  A segment takes as many batches of 11 rows as its
// rows and 20 more need, so the rows are 11 k - 20; k is the one whose last wave of 304 blocks (two per SM) ends
// first: a batch of 11 rows costs about the same wherever it lies, 8.0 us for two blocks on an SM and 4.9 for one
// (and 2.5 to begin with), which a last wave of at most 152 blocks has.  Weighed as whole waves, 640x360 took 24.8
// instead of 22.7 us (k 3 instead of 4), 801x601 40.5 instead of 37.0 (5, 7), 65x5000 33 instead of 27 (4, 5), 32
// views of 64x64 24.8 instead of 22.7 (3, 4).  False when the views hold too many.
bool loss_plan(LossViews& L) {
    long long best = 0;
    for (int k = 3; k <= 32; ++k) {
        const int rows = kTap * k - 20;
        long long blocks = 0;
        for (int v = 0; v < L.n; ++v)
            blocks += (long long)((L.w[v] + kOP - 1) / kOP) * ((L.h[v] + rows - 1) / rows);
        const long long rest = blocks % 304;
        const long long cost = (blocks / 304 + (rest > 152)) * 80 * k + (rest > 0 && rest <= 152 ? 49 * k + 25 : 0);
        if (best == 0 || cost < best) {
            best = cost;
            L.rows = rows;
        }
    }
    long long blocks = 0;
    for (int v = 0; v < L.n; ++v) {
        L.tiles_x[v] = (L.w[v] + kOP - 1) / kOP;
        L.tile_off[v] = (int)blocks;
        blocks += (long long)L.tiles_x[v] * ((L.h[v] + L.rows - 1) / L.rows);
        if (blocks > (1ll << 30)) return false;
    }
    L.tile_off[L.n] = (int)blocks;
    return true;
}

cudaError_t launch_adam(float* p, const float* g, float* m, float* v, const AdamGroups& G, double beta1,
                        double beta2, AdamState* st, const WsHeader* guard, cudaStream_t s) {
    k_adam_tick<<<1, 2, 0, s>>>(st, guard, beta1, beta2);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const long long units = G.ubase[G.n];
    if (units == 0) return cudaSuccess;
    int sms = 0;
    e = sm_count(sms);
    if (e != cudaSuccess) return e;
    const long long want = (units + 255) / 256;
    const long long cap = (long long)sms * 8;
    k_adam<<<(unsigned)(want < cap ? want : cap), 256, 0, s>>>(p, g, m, v, G, st, guard);
    return cudaGetLastError();
}

}  // namespace wsr
