// Per-Gaussian projection (forward) and its gradient chain (backward).
//
// Forward, one thread per Gaussian, looping over the views so the parameters
// are read from HBM once per call:
//   Sec. 3 Eq. 3   Sigma_3D = R S S^t R^t          (R from the normalised quaternion)
//   Sec. 3 Eq. 5   Sigma_2D = J W Sigma_3D W^t J^t  (+ 0.3 I, J clamped at 1.3 tan(fov))
//   Sec. 3 Eq. 4   c = max(0, Y(dir) . H + 0.5)
//   Eq. 11 / Eq. 3 u = Y(dir) . H^alpha (unclamped) or sigmoid(o)
//   Eqs. 8-10      w(d) with d = camera z
// and writes the 48-byte render record {mu, qs, qw, qd, u w, c u w, extents}
// with the footprint's quadratic form, prescaled by log2(e)/2, as the sum of
// squares q' = (qs dy + qw dx)^2 + qd dx^2.
//
// Backward, one thread per Gaussian: the render backward's record of each
// (view, Gaussian) holds moments of dL/dq' in that sum-of-squares frame plus
// d/d(u w) and d/d(c u w); they are chained to the mean, the 2D covariance
// (in factored form), the colour and opacity SH, the depth weight and the
// stored parameters, summed over views.
//
// The 2D covariance is formed as T T^t with T = J W R S (2x3), so its
// determinant is the squared norm of the cross product of T's rows (plus the
// dilation terms): a sum of squares with no cancellation.  For strongly
// anisotropic footprints (det < 1e-3 a c) the conic is recomputed in FP64
// from the same rows.
#include <mutex>

#include "wsr_launch.h"

namespace wsr {
namespace {

struct Geom {
    float tx, ty, tz;
    float M[9];            // W R diag(s), row-major
    float J00, J02, J11, J12;
    float rxc, ryc;        // clamped x/z and y/z
    bool freex, freey;     // not clamped
    float r0[3], r1[3];    // rows of T = J W R S
    float a, b, c;         // Sigma_2D with dilation
    float A, B, C;         // conic
    // the same quadratic form as a sum of squares, prescaled by log2(e)/2:
    // q' = (qs dy + qw dx)^2 + qd dx^2, i.e. q = (a/det)(dy - (b/a) dx)^2 + dx^2 / a
    float qs, qw, qd;
};

__device__ __forceinline__ void geometry(const View& V, const float* Rg, const float* s, float px,
                                         float py, float pz, Geom& G) {
    G.tx = V.R[0] * px + V.R[1] * py + V.R[2] * pz + V.T[0];
    G.ty = V.R[3] * px + V.R[4] * py + V.R[5] * pz + V.T[1];
    G.tz = V.R[6] * px + V.R[7] * py + V.R[8] * pz + V.T[2];
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int c = 0; c < 3; ++c)
            G.M[3 * r + c] =
                (V.R[3 * r] * Rg[c] + V.R[3 * r + 1] * Rg[3 + c] + V.R[3 * r + 2] * Rg[6 + c]) * s[c];
    const float iz = 1.0f / G.tz;
    const float ux = G.tx * iz, uy = G.ty * iz;
    G.rxc = fminf(fmaxf(ux, -V.limx), V.limx);
    G.ryc = fminf(fmaxf(uy, -V.limy), V.limy);
    G.freex = (ux >= -V.limx) && (ux <= V.limx);
    G.freey = (uy >= -V.limy) && (uy <= V.limy);
    G.J00 = V.fx * iz;
    G.J02 = -V.fx * G.rxc * iz;
    G.J11 = V.fy * iz;
    G.J12 = -V.fy * G.ryc * iz;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        G.r0[k] = G.J00 * G.M[k] + G.J02 * G.M[6 + k];
        G.r1[k] = G.J11 * G.M[3 + k] + G.J12 * G.M[6 + k];
    }
    const float a0 = G.r0[0] * G.r0[0] + G.r0[1] * G.r0[1] + G.r0[2] * G.r0[2];
    const float c0 = G.r1[0] * G.r1[0] + G.r1[1] * G.r1[1] + G.r1[2] * G.r1[2];
    const float b0 = G.r0[0] * G.r1[0] + G.r0[1] * G.r1[1] + G.r0[2] * G.r1[2];
    const float x0 = G.r0[1] * G.r1[2] - G.r0[2] * G.r1[1];
    const float x1 = G.r0[2] * G.r1[0] - G.r0[0] * G.r1[2];
    const float x2 = G.r0[0] * G.r1[1] - G.r0[1] * G.r1[0];
    G.a = a0 + kDilation;
    G.c = c0 + kDilation;
    G.b = b0;
    const float det = (x0 * x0 + x1 * x1 + x2 * x2) + kDilation * (a0 + c0) + kDilation * kDilation;
    if (det < 1e-3f * G.a * G.c) {
        // strongly anisotropic footprint: conic in FP64 from the same rows
        const double p0 = G.r0[0], p1 = G.r0[1], p2 = G.r0[2];
        const double q0 = G.r1[0], q1 = G.r1[1], q2 = G.r1[2];
        const double ad = p0 * p0 + p1 * p1 + p2 * p2, cd = q0 * q0 + q1 * q1 + q2 * q2;
        const double bd = p0 * q0 + p1 * q1 + p2 * q2;
        const double y0 = p1 * q2 - p2 * q1, y1 = p2 * q0 - p0 * q2, y2 = p0 * q1 - p1 * q0;
        const double dd = (y0 * y0 + y1 * y1 + y2 * y2) + 0.3 * (ad + cd) + 0.09;
        G.A = (float)((cd + 0.3) / dd);
        G.B = (float)(-bd / dd);
        G.C = (float)((ad + 0.3) / dd);
        const double k = (double)kHalfLog2e, a_ = ad + 0.3;
        const double qs = sqrt(k * a_ / dd);
        G.qs = (float)qs;
        G.qw = (float)(-(bd / a_) * qs);
        G.qd = (float)(k / a_);
    } else {
        const float id = 1.0f / det;
        G.A = G.c * id;
        G.B = -G.b * id;
        G.C = G.a * id;
        G.qs = sqrtf(kHalfLog2e * G.a * id);
        G.qw = -(G.b / G.a) * G.qs;
        G.qd = kHalfLog2e / G.a;
    }
}

template <int DEG, bool VD, bool RED>
struct Params {
    static constexpr int K = (DEG + 1) * (DEG + 1);
    float p[3], ls[3], q[4];
    float H[K * 3];
    float Ha[VD ? K : 1];
    float lcv;
};

template <int DEG, bool VD, bool RED>
__device__ __forceinline__ void load_params(const GaussPtrs& g, long long i, int wkind,
                                            Params<DEG, VD, RED>& P) {
    using sq_t = typename Store<RED>::sq_t;
    using sh_t = typename Store<RED>::sh_t;
    constexpr int K = Params<DEG, VD, RED>::K;
    P.p[0] = __ldg(g.means + 3 * i);
    P.p[1] = __ldg(g.means + 3 * i + 1);
    P.p[2] = __ldg(g.means + 3 * i + 2);
    load_n<sq_t, 3>(reinterpret_cast<const sq_t*>(g.log_scales) + 3 * i, P.ls);
    load_n<sq_t, 4>(reinterpret_cast<const sq_t*>(g.quats) + 4 * i, P.q);
    load_n<sh_t, K * 3>(reinterpret_cast<const sh_t*>(g.sh) + (long long)K * 3 * i, P.H);
    if constexpr (VD) {
        load_n<sh_t, K>(reinterpret_cast<const sh_t*>(g.opacity) + (long long)K * i, P.Ha);
    } else {
        load_n<sh_t, 1>(reinterpret_cast<const sh_t*>(g.opacity) + i, P.Ha);
    }
    P.lcv = (wkind == WSR_WEIGHT_LC) ? __ldg(g.lc_v + i) : 0.0f;
}

// Normalised quaternion, rotation and scales.
__device__ __forceinline__ void rot_scale(const float* qr, const float* ls, float* qn, float& qlen,
                                          float* Rg, float* s) {
    const float n2 = qr[0] * qr[0] + qr[1] * qr[1] + qr[2] * qr[2] + qr[3] * qr[3];
    qlen = sqrtf(n2);
    const float inv = 1.0f / qlen;
#pragma unroll
    for (int k = 0; k < 4; ++k) qn[k] = qr[k] * inv;
    quat_rot(qn[0], qn[1], qn[2], qn[3], Rg);
#pragma unroll
    for (int k = 0; k < 3; ++k) s[k] = expf(ls[k]);
}

// The depth factor of the weight (Eqs. 8-10): w = factor for DIR and EXP, w = factor * v_i for LC.
// A Gaussian is culled only where the factor is 0 (LC beyond sigma, EXP underflow): there neither
// Eq. 7 nor its gradient depends on it.  Where only v_i is 0, w = 0 but dw/dv_i is not, so it stays.
__device__ __forceinline__ float depth_factor(int kind, float d, float sigma, float beta) {
    if (kind == WSR_WEIGHT_EXP) return expf(-sigma * powf(d, beta));
    if (kind == WSR_WEIGHT_LC) return fmaxf(0.0f, 1.0f - d / sigma);
    return 1.0f;
}

template <int DEG, bool VD, bool RED>
__global__ void __launch_bounds__(256) k_project(const GaussPtrs g, const Views vs, const WeightDev wd,
                                                 float4* __restrict__ rec) {
    constexpr int K = (DEG + 1) * (DEG + 1);
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.n) return;
    Params<DEG, VD, RED> P;
    load_params<DEG, VD, RED>(g, i, wd.kind, P);
    const float sigma = __ldg(wd.params + 0), beta = __ldg(wd.params + 1);
    float qn[4], qlen, Rg[9], s[3];
    rot_scale(P.q, P.ls, qn, qlen, Rg, s);

    for (int v = 0; v < vs.n; ++v) {
        const View& V = vs.v[v];
        float4* o = rec + 3 * ((long long)v * g.n + i);
        const float tz = V.R[6] * P.p[0] + V.R[7] * P.p[1] + V.R[8] * P.p[2] + V.T[2];
        float wf = 0.0f;
        if (tz > V.znear) wf = depth_factor(wd.kind, tz, sigma, beta);
        if (!(tz > V.znear) || wf == 0.0f) {
            // culled: behind the near plane (App. C), or a zero depth factor
            // (LC beyond sigma), which contributes nothing to Eq. 7 or its gradient
            o[0] = make_float4(0.f, 0.f, 0.f, 0.f);
            o[1] = make_float4(0.f, 0.f, 0.f, 0.f);
            o[2] = make_float4(0.f, -1.f, -1.f, tz);
            continue;
        }
        const float w = (wd.kind == WSR_WEIGHT_LC) ? wf * P.lcv : wf;
        Geom G;
        geometry(V, Rg, s, P.p[0], P.p[1], P.p[2], G);
        const float mx = V.fx * G.tx / G.tz + V.cx;
        const float my = V.fy * G.ty / G.tz + V.cy;
        // 3-sigma half extents, slightly widened so that binning stays
        // conservative with respect to the FP32 cutoff test of the renderer
        const float rx = 3.0f * sqrtf(G.a) * 1.0001f + 0.01f;
        const float ry = 3.0f * sqrtf(G.c) * 1.0001f + 0.01f;

        float dx = P.p[0] - V.campos[0], dy = P.p[1] - V.campos[1], dz = P.p[2] - V.campos[2];
        const float il = rsqrtf(dx * dx + dy * dy + dz * dz);
        dx *= il; dy *= il; dz *= il;
        float Y[K];
        sh_basis<DEG>(dx, dy, dz, Y);
        float col[3];
#pragma unroll
        for (int ch = 0; ch < 3; ++ch) {
            float r = 0.0f;
#pragma unroll
            for (int k = 0; k < K; ++k) r += Y[k] * P.H[3 * k + ch];
            col[ch] = fmaxf(r + 0.5f, 0.0f);
        }
        float u;
        if constexpr (VD) {
            u = 0.0f;
#pragma unroll
            for (int k = 0; k < K; ++k) u += Y[k] * P.Ha[k];
        } else {
            u = 1.0f / (1.0f + expf(-P.Ha[0]));
        }
        const float uw = u * w;
        o[0] = make_float4(mx, my, G.qs, G.qw);
        o[1] = make_float4(G.qd, uw, col[0] * uw, col[1] * uw);
        o[2] = make_float4(col[2] * uw, rx, ry, G.tz);
    }
}

// ---------------------------------------------------------------------------
// Backward chain: grad record {dmu, dA, dB, dC, d(uw), d(c uw)} per view ->
// parameters.  Recomputes every forward intermediate from the parameters.
// ---------------------------------------------------------------------------
template <int N>
__device__ __forceinline__ void store_n(float* __restrict__ p, const float* v) {
    if constexpr ((N * 4) % 16 == 0) {
        float4* q = reinterpret_cast<float4*>(p);
#pragma unroll
        for (int k = 0; k < N / 4; ++k) q[k] = make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
    } else {
#pragma unroll
        for (int k = 0; k < N; ++k) p[k] = v[k];
    }
}

// A block's SH rows in shared memory: R floats per Gaussian, P apart.  Rows that are whole float4s are padded so
// that a row per lane falls on distinct banks; other rows (odd lengths do already) lie as in global memory.
template <int R>
struct Rows {
    static constexpr int P = R % 4 ? R : (R / 4 + 1) % 2 ? R + 4 : (R / 4) % 2 ? R : R + 8;
    static_assert(R % 4 || (P / 4) % 2, "an odd number of float4s apart");
};

// Whether rows of R stored as T lie in shared memory as they are stored (else as floats): halfs in whole 16 bytes.
template <int R, typename T>
constexpr bool kRawHalfs = sizeof(T) == 2 && R % 8 == 0;

// A thread's own row as floats: 16 bytes at a time where the rows are padded for it.
template <int R, typename T>
__device__ __forceinline__ void row_get(const float* __restrict__ row, float (&v)[R]) {
    if constexpr (kRawHalfs<R, T>) {
#pragma unroll
        for (int c = 0; c < R / 8; ++c) {
            const uint4 x = reinterpret_cast<const uint4*>(row)[c];
            const T* e = reinterpret_cast<const T*>(&x);
#pragma unroll
            for (int j = 0; j < 8; ++j) v[8 * c + j] = to_f(e[j]);
        }
    } else if constexpr (R % 4 == 0) {
#pragma unroll
        for (int c = 0; c < R / 4; ++c) {
            const float4 x = reinterpret_cast<const float4*>(row)[c];
            v[4 * c] = x.x, v[4 * c + 1] = x.y, v[4 * c + 2] = x.z, v[4 * c + 3] = x.w;
        }
    } else {
#pragma unroll
        for (int e = 0; e < R; ++e) v[e] = row[e];
    }
}
template <int R>
__device__ __forceinline__ void row_put(float* __restrict__ row, const float (&v)[R]) {
    if constexpr (R % 4 == 0) {
#pragma unroll
        for (int c = 0; c < R / 4; ++c)
            reinterpret_cast<float4*>(row)[c] = make_float4(v[4 * c], v[4 * c + 1], v[4 * c + 2], v[4 * c + 3]);
    } else {
#pragma unroll
        for (int e = 0; e < R; ++e) row[e] = v[e];
    }
}

// Rows [0, cnt) of R consecutive T each from global memory (16-byte aligned) to shared memory, consecutive lanes on
// consecutive 16 bytes; asynchronous copies where nothing is converted.
template <int R, typename T>
__device__ __forceinline__ void rows_in(float* __restrict__ sm, const T* __restrict__ g, const int cnt) {
    constexpr int PER = 16 / (int)sizeof(T), P = Rows<R>::P;
    constexpr bool RAW = sizeof(T) == 4 || kRawHalfs<R, T>;
    const int total = cnt * R, whole = total / PER;
    if constexpr (RAW) {
        for (int c = threadIdx.x; c < whole; c += blockDim.x) {
            float* const o = sm + (sizeof(T) == 4 ? P == R ? 4 * c : 4 * c / R * P + 4 * c % R
                                                  : 8 * c / R * P + 8 * c % R / 2);
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(o)),
                         "l"(reinterpret_cast<const uint4*>(g) + c) : "memory");
        }
        // (rows of halfs are whole 16 bytes: nothing is left over)
        for (int k = whole * PER + threadIdx.x; k < total; k += blockDim.x) sm[k / R * P + k % R] = to_f(g[k]);
    } else {
#pragma unroll 4
        for (int c = threadIdx.x; c < whole; c += blockDim.x) {
            const uint4 u = __ldg(reinterpret_cast<const uint4*>(g) + c);
            const T* e = reinterpret_cast<const T*>(&u);
#pragma unroll
            for (int j = 0; j < PER; ++j) sm[(c * PER + j) / R * P + (c * PER + j) % R] = to_f(e[j]);
        }
        for (int k = whole * PER + threadIdx.x; k < total; k += blockDim.x) sm[k / R * P + k % R] = to_f(g[k]);
    }
}

// The way back, floats: 16 bytes per lane when the output allows it (only its elements' alignment is asked for).
template <int R>
__device__ __forceinline__ void rows_out(float* __restrict__ g, const float* __restrict__ sm, const int cnt) {
    constexpr int P = Rows<R>::P;
    const int total = cnt * R, whole = (reinterpret_cast<uintptr_t>(g) & 15u) ? 0 : total / 4;
#pragma unroll 4
    for (int c = threadIdx.x; c < whole; c += blockDim.x)
        reinterpret_cast<float4*>(g)[c] = *reinterpret_cast<const float4*>(sm + (P == R ? 4 * c : 4 * c / R * P + 4 * c % R));
    for (int k = 4 * whole + threadIdx.x; k < total; k += blockDim.x) g[k] = sm[k / R * P + k % R];
}

// From degree 2 up the SH coefficients and their gradients go through shared memory, a row per thread there and 16
// bytes per lane in global memory: a row per thread in global memory puts each lane of an access on a line of its
// own, and the lines, not the bytes, bound the kernel.  Neither then stays in registers.  The copies in and the
// gradient record's loads are all in flight at once (with a round of loads at a time the kernel took 200 us).
// ONE: a single view, whose SH gradients are final as soon as they are formed and take the coefficients' place;
// several views add theirs in rows beside them.  Below degree 2 the rows are short and stay in registers.
//   One view, 1M Gaussians of degree 3 with view-dependent opacity: 138 -> 117 us (636 MB, 80% of the copy rate);
// 400k of degree 2: 82 -> 37 us (rows of 27 floats took 4-byte accesses); six views of 300k, degree 2: 128 -> 84 us.
// Blocks per SM: at degree 3 four, which spills up to 36 bytes with view-dependent opacity; five spill more (136 us).
// Small scenes of degree 3 pay for the way through shared memory: one view of 2000 6.0 -> 6.5 us, of 100k 16.4 -> 17.7
// (three views 26 -> 23.6); 20k 8.1 -> 7.4.
//   The deterministic mode's records are a kernel of their own (DET): as a branch they cost the others 0.3 to 1.5 us,
// 2000 of degree 0 in three views 7.3 -> 6.6, 100k of degree 1 12.2 -> 10.7.
template <int DEG, bool VD, bool RED, bool ONE, bool DET>
__global__ void __launch_bounds__(128, ONE ? (DEG == 3 ? 4 : DEG == 2 ? 6 : 3) : (DEG == 3 ? 3 : DEG == 2 ? 4 : 1))
    k_project_bwd(const GaussPtrs g, const Views vs, const WeightDev wd, const float* __restrict__ grec,
                  const wsr_grads out, float* __restrict__ det_sb) {
    using sq_t = typename Store<RED>::sq_t;
    using sh_t = typename Store<RED>::sh_t;
    constexpr int K = (DEG + 1) * (DEG + 1), KA = VD ? K : 1;
    constexpr bool ROWS = DEG >= 2;
    constexpr int PH = Rows<3 * K>::P, PA = Rows<KA>::P;
    extern __shared__ __align__(16) float s_rows[];
    float* const s_h = s_rows;                                  // coefficients, or (ONE) at the end gradients
    float* const s_a = s_h + 128 * PH;                          // opacity likewise
    float* const s_gh = ONE ? s_h : s_a + 128 * PA;             // gradients
    float* const s_ga = ONE ? s_a : s_gh + 128 * PH;
    // deterministic mode: a view's records (27 words used of 32), 28 words apart: 67 -> 44 us for 250k Gaussians
    // against a record per thread in global memory
    float* const s_det = ROWS ? s_ga + 128 * PA : s_rows;
    float gsig = 0.0f, gbeta = 0.0f;
    const float sigma = __ldg(wd.params + 0), beta = __ldg(wd.params + 1);
    // DET: deterministic mode (fixed-point records, a bounded grid striding over the Gaussians, sigma/beta
    // summed per block in a fixed order into det_sb)
    for (long long i0 = 128ll * blockIdx.x; i0 < g.n; i0 += 128ll * gridDim.x) {
        const int cnt = (int)min(128ll, g.n - i0);
        const long long i = i0 + threadIdx.x;
        const bool mine = (int)threadIdx.x < cnt;
        float p[3] = {0.f, 0.f, 0.f}, ls[3] = {0.f, 0.f, 0.f}, q[4] = {1.f, 0.f, 0.f, 0.f}, lcv = 0.0f;
        if (mine) {
#pragma unroll
            for (int k = 0; k < 3; ++k) p[k] = __ldg(g.means + 3 * i + k);
            load_n<sq_t, 3>(reinterpret_cast<const sq_t*>(g.log_scales) + 3 * i, ls);
            load_n<sq_t, 4>(reinterpret_cast<const sq_t*>(g.quats) + 4 * i, q);
            if (wd.kind == WSR_WEIGHT_LC) lcv = __ldg(g.lc_v + i);
        }
        float rh[ROWS ? 1 : 3 * K], ra_[ROWS ? 1 : KA];             // short rows, in registers
        float rgh[ROWS ? 1 : 3 * K], rga[ROWS ? 1 : KA];
        if constexpr (ROWS) {
            rows_in<3 * K>(s_h, reinterpret_cast<const sh_t*>(g.sh) + 3ll * K * i0, cnt);
            rows_in<KA>(s_a, reinterpret_cast<const sh_t*>(g.opacity) + (long long)KA * i0, cnt);
        } else if (mine) {
            load_n<sh_t, 3 * K>(reinterpret_cast<const sh_t*>(g.sh) + 3ll * K * i, rh);
            load_n<sh_t, KA>(reinterpret_cast<const sh_t*>(g.opacity) + (long long)KA * i, ra_);
        }
        float4 ra = make_float4(0.f, 0.f, 0.f, 0.f), rb = ra;       // a gradient record (not the deterministic mode's)
        float rc = 0.0f;
        auto load_record = [&](int v) {
            const float4* r = reinterpret_cast<const float4*>(grec + WSR_GRAD_RECORD_FLOATS * ((long long)v * g.n + i));
            ra = __ldg(r);
            rb = __ldg(r + 1);
            rc = __ldg(reinterpret_cast<const float*>(r + 2));
        };
        auto copy_det = [&](int v) {
            const uint4* from = reinterpret_cast<const uint4*>(grec) + 8ll * ((long long)v * g.n + i0);
            for (int c = threadIdx.x; c < 7 * cnt; c += 128) {
                float* const o = s_det + 4 * c;
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(o)),
                             "l"(from + (c / 7 * 8 + c % 7)) : "memory");
            }
        };
        if constexpr (DET) copy_det(0);
        else if (mine) load_record(0);
        auto get_h = [&](float (&h)[3 * K], float (&ha)[KA]) {
            if constexpr (ROWS) {
                row_get<3 * K, sh_t>(s_h + PH * threadIdx.x, h);
                row_get<KA, sh_t>(s_a + PA * threadIdx.x, ha);
            } else {
#pragma unroll
                for (int e = 0; e < 3 * K; ++e) h[e] = rh[e];
#pragma unroll
                for (int e = 0; e < KA; ++e) ha[e] = ra_[e];
            }
        };
        auto get_g = [&](float (&h)[3 * K], float (&ha)[KA]) {
            if constexpr (ROWS) {
                row_get<3 * K, float>(s_gh + PH * threadIdx.x, h);
                row_get<KA, float>(s_ga + PA * threadIdx.x, ha);
            } else {
#pragma unroll
                for (int e = 0; e < 3 * K; ++e) h[e] = rgh[e];
#pragma unroll
                for (int e = 0; e < KA; ++e) ha[e] = rga[e];
            }
        };
        auto put_g = [&](const float (&h)[3 * K], const float (&ha)[KA]) {
            if constexpr (ROWS) {
                row_put<3 * K>(s_gh + PH * threadIdx.x, h);
                row_put<KA>(s_ga + PA * threadIdx.x, ha);
            } else {
#pragma unroll
                for (int e = 0; e < 3 * K; ++e) rgh[e] = h[e];
#pragma unroll
                for (int e = 0; e < KA; ++e) rga[e] = ha[e];
            }
        };
        const float zero_h[3 * K] = {}, zero_a[KA] = {};
        if constexpr (!ONE || !ROWS) put_g(zero_h, zero_a);
        if constexpr (ROWS || DET) {
            asm volatile("cp.async.wait_all;" ::: "memory");
            __syncthreads();
        }

        float qn[4], qlen, Rg[9], s[3];
        rot_scale(q, ls, qn, qlen, Rg, s);
        float gp[3] = {0.f, 0.f, 0.f}, gs[3] = {0.f, 0.f, 0.f}, gR[9];
#pragma unroll
        for (int e = 0; e < 9; ++e) gR[e] = 0.f;
        float glcv = 0.f;
        bool sh_done = false;           // ONE: the rows hold the gradients

        const int nv = ONE ? 1 : vs.n;
        for (int v = 0; v < nv; ++v) {
            if (DET && v > 0) {
                __syncthreads();                // the last view's records are read
                copy_det(v);
                asm volatile("cp.async.wait_all;" ::: "memory");
                __syncthreads();
            }
            if (!mine) continue;
            const View& V = vs.v[v];
            float g9[9];
            bool any = false;
            if constexpr (!DET) {
                g9[0] = ra.x, g9[1] = ra.y, g9[2] = ra.z, g9[3] = ra.w;
                g9[4] = rb.x, g9[5] = rb.y, g9[6] = rb.z, g9[7] = rb.w;
                g9[8] = rc;
                if (!ONE && v + 1 < nv) load_record(v + 1);         // the next view's, while this one is chained
#pragma unroll
                for (int e = 0; e < 9; ++e) any |= (g9[e] != 0.0f);
            } else {
                // 9 int64 sums in units of 2^(e - kDetBits), 2^e above the term's bound (stored beside them)
                const float* const gr = s_det + 28 * threadIdx.x;
                const long long* sums = reinterpret_cast<const long long*>(gr);
                const int* mag = reinterpret_cast<const int*>(gr + 18);
#pragma unroll
                for (int c = 0; c < 9; ++c) {
                    const float m = __int_as_float(mag[c]);
                    float val = 0.0f;
                    if (m > 0.0f) {
                        int e;
                        frexpf(m, &e);
                        val = ldexpf(__ll2float_rn(sums[c]), e - kDetBits);
                    }
                    g9[c] = val;
                    any |= (val != 0.0f);
                }
            }
            if (!any) continue;
            const float tz0 = V.R[6] * p[0] + V.R[7] * p[1] + V.R[8] * p[2] + V.T[2];
            if (!(tz0 > V.znear)) continue;
            const float wf = depth_factor(wd.kind, tz0, sigma, beta);
            if (wf == 0.0f) continue;
            const float w = (wd.kind == WSR_WEIGHT_LC) ? wf * lcv : wf;
            Geom G;
            geometry(V, Rg, s, p[0], p[1], p[2], G);
            const float tx = G.tx, ty = G.ty, tz = G.tz;

            float vx = p[0] - V.campos[0], vy = p[1] - V.campos[1], vz = p[2] - V.campos[2];
            const float il = rsqrtf(vx * vx + vy * vy + vz * vz);
            const float dx = vx * il, dy = vy * il, dz = vz * il;
            float Y[K];
            sh_basis<DEG>(dx, dy, dz, Y);
            float raw[3] = {0.f, 0.f, 0.f}, col[3], u = 0.0f;
            {
                float h[3 * K], ha[KA];
                get_h(h, ha);
#pragma unroll
                for (int k = 0; k < K; ++k) {
#pragma unroll
                    for (int ch = 0; ch < 3; ++ch) raw[ch] += Y[k] * h[3 * k + ch];
                    if constexpr (VD) u += Y[k] * ha[k];
                }
                if constexpr (!VD) u = 1.0f / (1.0f + expf(-ha[0]));
            }
#pragma unroll
            for (int ch = 0; ch < 3; ++ch) col[ch] = fmaxf(raw[ch] + 0.5f, 0.0f);
            const float uw = u * w;

            // Eq. 7 record terms -> colour, opacity, weight
            const float gcuw[3] = {g9[6], g9[7], g9[8]};
            const float guw = g9[5] + gcuw[0] * col[0] + gcuw[1] * col[1] + gcuw[2] * col[2];
            const float gu = guw * w, gw = guw * u;
            float graw[3];
#pragma unroll
            for (int ch = 0; ch < 3; ++ch) graw[ch] = (raw[ch] + 0.5f > 0.0f) ? gcuw[ch] * uw : 0.0f;
            float wk[K];
            if constexpr (ROWS) asm volatile("" ::: "memory");      // read the rows again rather than keep them in registers
            {
                float h[3 * K], ha[KA];
                get_h(h, ha);
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    wk[k] = graw[0] * h[3 * k] + graw[1] * h[3 * k + 1] + graw[2] * h[3 * k + 2];
                    if constexpr (VD) wk[k] += gu * ha[k];
                }
                if constexpr (!ONE) {
                    get_g(h, ha);
                }
#pragma unroll
                for (int k = 0; k < K; ++k) {
#pragma unroll
                    for (int ch = 0; ch < 3; ++ch) h[3 * k + ch] = (ONE ? 0.0f : h[3 * k + ch]) + graw[ch] * Y[k];
                    if constexpr (VD) ha[k] = (ONE ? 0.0f : ha[k]) + gu * Y[k];
                }
                if constexpr (!VD) ha[0] = (ONE ? 0.0f : ha[0]) + gu * u * (1.0f - u);
                put_g(h, ha);
            }
            sh_done = true;
            // direction dir = (p - f)/|p - f|: tangential part of the SH gradient
            float gdx = 0.f, gdy = 0.f, gdz = 0.f;
            sh_grad_dot<DEG>(dx, dy, dz, wk, gdx, gdy, gdz);
            const float dd = dx * gdx + dy * gdy + dz * gdz;
            gp[0] += (gdx - dx * dd) * il;
            gp[1] += (gdy - dy * dd) * il;
            gp[2] += (gdz - dz * dd) * il;

            // depth weight, d = t_z
            float gt[3] = {0.f, 0.f, 0.f};
            if (wd.kind == WSR_WEIGHT_EXP) {
                const float db = powf(tz, beta);
                gsig += gw * (-db) * w;
                gbeta += gw * (-sigma * db * logf(tz)) * w;
                gt[2] += gw * (-sigma * beta * db / tz) * w;
            } else if (wd.kind == WSR_WEIGHT_LC) {
                const float lin = 1.0f - tz / sigma;
                glcv += gw * lin;
                gsig += gw * lcv * tz / (sigma * sigma);
                gt[2] += gw * (-lcv / sigma);
            }
            // The record holds moments of gq = dL/dq' over the Gaussian's pixels in the sum-of-squares
            // frame of q' = r^2 + qd dx^2, r = qs dy + qw dx (qs, qw, qd exactly as rendered):
            // Sr = sum gq r, Sx = sum gq dx, Srr = sum gq r^2, Srx = sum gq r dx, Sxx = sum gq dx^2.
            const float Sr = g9[0], Sx = g9[1], Srr = g9[2], Srx = g9[3], Sxx = g9[4];
            const float qs = G.qs, qw = G.qw, qd = G.qd;
            // projected mean: dq'/dmu_x = -2 (r qw + qd dx), dq'/dmu_y = -2 r qs
            const float gmx = -2.0f * fmaf(qw, Sr, qd * Sx), gmy = -2.0f * qs * Sr;
            const float iz = 1.0f / tz, iz2 = iz * iz;
            gt[0] += gmx * V.fx * iz;
            gt[1] += gmy * V.fy * iz;
            gt[2] += -(gmx * V.fx * tx + gmy * V.fy * ty) * iz2;

            // Sigma_2D = T T^t + 0.3 I with rows r0, r1 of T = J W R S.  With v = k Sigma_2D^{-1} d =
            // r w + qd dx e1 (w = (qw, qs), e1 = (1, 0), k = log2(e)/2), dq'/dSigma_2D = -v v^t / k, so
            //   dL/dSigma_2D = -(Srr w w^t + qd Srx (w e1^t + e1 w^t) + qd^2 Sxx e1 e1^t) / k
            // and dL/dT = 2 dL/dSigma_2D T is taken in that factored form: with z = w^t T = qw r0 + qs r1,
            //   dL/dr0 = -2/k (qw P1 + P2),  dL/dr1 = -2/k qs P1,
            //   P1 = Srr z + qd Srx r0,  P2 = qd Srx z + qd^2 Sxx r0.
            // For a thin footprint z is nearly orthogonal to the long axis, so the large Srr terms
            // stay off that axis instead of cancelling there in FP32.
            const float c2 = -2.0f / kHalfLog2e, qsx = qd * Srx, qxx = qd * qd * Sxx;
            float gr0[3], gr1[3];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const float z = fmaf(qw, G.r0[k], qs * G.r1[k]);
                const float P1 = fmaf(Srr, z, qsx * G.r0[k]);
                const float P2 = fmaf(qsx, z, qxx * G.r0[k]);
                gr0[k] = c2 * fmaf(qw, P1, P2);
                gr1[k] = c2 * qs * P1;
            }
            // r0 = J00 m0 + J02 m2,  r1 = J11 m1 + J12 m2  (m_k: rows of M = W R S)
            float gJ00 = 0.f, gJ02 = 0.f, gJ11 = 0.f, gJ12 = 0.f, gM[9];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                gJ00 += gr0[k] * G.M[k];
                gJ02 += gr0[k] * G.M[6 + k];
                gJ11 += gr1[k] * G.M[3 + k];
                gJ12 += gr1[k] * G.M[6 + k];
                gM[k] = G.J00 * gr0[k];
                gM[3 + k] = G.J11 * gr1[k];
                gM[6 + k] = G.J02 * gr0[k] + G.J12 * gr1[k];
            }
            // J(t): J00 = fx/tz, J02 = -fx rx/tz, J11 = fy/tz, J12 = -fy ry/tz
            gt[2] += -(gJ00 * V.fx + gJ11 * V.fy) * iz2 + (gJ02 * V.fx * G.rxc + gJ12 * V.fy * G.ryc) * iz2;
            if (G.freex) {
                gt[0] += -gJ02 * V.fx * iz2;
                gt[2] += gJ02 * V.fx * tx * iz2 * iz;
            }
            if (G.freey) {
                gt[1] += -gJ12 * V.fy * iz2;
                gt[2] += gJ12 * V.fy * ty * iz2 * iz;
            }
            // t = W p + T
#pragma unroll
            for (int k = 0; k < 3; ++k) gp[k] += V.R[k] * gt[0] + V.R[3 + k] * gt[1] + V.R[6 + k] * gt[2];
            // M = W N, N = R diag(s):  gN = W^t gM
#pragma unroll
            for (int r = 0; r < 3; ++r)
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    const float gN = V.R[r] * gM[c] + V.R[3 + r] * gM[3 + c] + V.R[6 + r] * gM[6 + c];
                    gR[3 * r + c] += gN * s[c];
                    gs[c] += gN * Rg[3 * r + c];
                }
        }

        // rotation <- normalised quaternion <- raw quaternion
        const float w_ = qn[0], x_ = qn[1], y_ = qn[2], z_ = qn[3];
        float gqn[4];
        gqn[0] = -2.f * z_ * gR[1] + 2.f * y_ * gR[2] + 2.f * z_ * gR[3] - 2.f * x_ * gR[5] - 2.f * y_ * gR[6] +
                 2.f * x_ * gR[7];
        gqn[1] = 2.f * y_ * gR[1] + 2.f * z_ * gR[2] + 2.f * y_ * gR[3] - 4.f * x_ * gR[4] - 2.f * w_ * gR[5] +
                 2.f * z_ * gR[6] + 2.f * w_ * gR[7] - 4.f * x_ * gR[8];
        gqn[2] = -4.f * y_ * gR[0] + 2.f * x_ * gR[1] + 2.f * w_ * gR[2] + 2.f * x_ * gR[3] + 2.f * z_ * gR[5] -
                 2.f * w_ * gR[6] + 2.f * z_ * gR[7] - 4.f * y_ * gR[8];
        gqn[3] = -4.f * z_ * gR[0] - 2.f * w_ * gR[1] + 2.f * x_ * gR[2] + 2.f * w_ * gR[3] - 4.f * z_ * gR[4] +
                 2.f * y_ * gR[5] + 2.f * x_ * gR[6] + 2.f * y_ * gR[7];
        const float qd = gqn[0] * qn[0] + gqn[1] * qn[1] + gqn[2] * qn[2] + gqn[3] * qn[3];
        float gq[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) gq[k] = (gqn[k] - qn[k] * qd) / qlen;
        float gls[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) gls[k] = gs[k] * s[k];

        if (mine) {
            if (out.means) { out.means[3 * i] = gp[0]; out.means[3 * i + 1] = gp[1]; out.means[3 * i + 2] = gp[2]; }
            if (out.log_scales) {
                out.log_scales[3 * i] = gls[0]; out.log_scales[3 * i + 1] = gls[1]; out.log_scales[3 * i + 2] = gls[2];
            }
            if (out.quats) store_n<4>(out.quats + 4 * i, gq);
            if (out.lc_v) out.lc_v[i] = glcv;
            if (ONE && ROWS && !sh_done) put_g(zero_h, zero_a);         // a view that added nothing
            if constexpr (!ROWS) {
                if (out.sh) store_n<3 * K>(out.sh + 3ll * K * i, rgh);
                if (out.opacity) store_n<KA>(out.opacity + (long long)KA * i, rga);
            }
        }
        if constexpr (ROWS) {
            __syncthreads();
            if (out.sh) rows_out<3 * K>(out.sh + 3ll * K * i0, s_gh, cnt);
            if (out.opacity) rows_out<KA>(out.opacity + (long long)KA * i0, s_ga, cnt);
        }
        if constexpr (ROWS || DET) __syncthreads();    // the rows and records are read
    }
    // global weight parameters: warp reduce, then one atomic per warp, or (deterministic) the block's sums
    // in warp order
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        gsig += __shfl_xor_sync(0xffffffffu, gsig, off);
        gbeta += __shfl_xor_sync(0xffffffffu, gbeta, off);
    }
    if constexpr (DET) {
        __shared__ float swb[2][4];
        if ((threadIdx.x & 31) == 0) {
            swb[0][threadIdx.x >> 5] = gsig;
            swb[1][threadIdx.x >> 5] = gbeta;
        }
        __syncthreads();
        if (threadIdx.x < 2) {
            float t = 0.0f;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += swb[threadIdx.x][w];
            det_sb[2 * blockIdx.x + threadIdx.x] = t;
        }
    } else if (out.weight_params && wd.kind != WSR_WEIGHT_DIR && (threadIdx.x & 31) == 0) {
        if (gsig != 0.0f) atomicAdd(out.weight_params + 0, gsig);
        if (gbeta != 0.0f) atomicAdd(out.weight_params + 1, gbeta);
    }
}

// Deterministic mode: the blocks' sigma/beta sums added in block order.
__global__ void __launch_bounds__(256) k_det_sb_reduce(const float* __restrict__ sb, int nb, float* __restrict__ gw) {
    __shared__ float part[2][8];
    float a0 = 0.0f, a1 = 0.0f;
    for (int b = threadIdx.x; b < nb; b += 256) {
        a0 += sb[2 * b];
        a1 += sb[2 * b + 1];
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        a0 += __shfl_xor_sync(0xffffffffu, a0, off);
        a1 += __shfl_xor_sync(0xffffffffu, a1, off);
    }
    if ((threadIdx.x & 31) == 0) {
        part[0][threadIdx.x >> 5] = a0;
        part[1][threadIdx.x >> 5] = a1;
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        float t = 0.0f;
#pragma unroll
        for (int k = 0; k < 8; ++k) t += part[threadIdx.x][k];
        gw[threadIdx.x] = t;
    }
}

template <int DEG, bool VD, bool RED>
cudaError_t project_t(const GaussPtrs& g, const Views& vs, WeightDev w, float* rec, cudaStream_t s) {
    const int bs = 256;
    const long long nb = (g.n + bs - 1) / bs;
    k_project<DEG, VD, RED><<<(unsigned)nb, bs, 0, s>>>(g, vs, w, reinterpret_cast<float4*>(rec));
    return cudaGetLastError();
}

template <int DEG, bool VD, bool RED>
cudaError_t project_bwd_t(const GaussPtrs& g, const Views& vs, WeightDev w, const float* grec,
                          const wsr_grads& out, float* det_sb, cudaStream_t s) {
    constexpr int bs = 128, K = (DEG + 1) * (DEG + 1);
    long long nb = (g.n + bs - 1) / bs;
    // one sigma/beta slot per block, and the blocks that fit on the device at once: 608 at four per SM
    if (det_sb && nb > kDetBlocks) nb = kDetBlocks;
    // the shared-memory opt-in is a per-device function attribute: set once per device (thread-safe)
    constexpr int rows = DEG < 2 ? 0 : sizeof(float) * bs * (Rows<3 * K>::P + Rows<VD ? K : 1>::P);
    constexpr int det_rows = sizeof(float) * bs * 28;
    const int more = det_sb ? det_rows : 0;
    static std::once_flag once[64];
    static cudaError_t once_err[64];
    int dev = 0;
    cudaError_t e0 = cudaGetDevice(&dev);
    if (e0 != cudaSuccess) return e0;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    std::call_once(once[dev], [&] {
        auto most = [&](auto kernel, int bytes) {
            if (once_err[dev] == cudaSuccess && bytes)
                once_err[dev] = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        };
        once_err[dev] = cudaSuccess;
        most(k_project_bwd<DEG, VD, RED, true, false>, rows);
        most(k_project_bwd<DEG, VD, RED, false, false>, 2 * rows);
        most(k_project_bwd<DEG, VD, RED, true, true>, rows + det_rows);
        most(k_project_bwd<DEG, VD, RED, false, true>, 2 * rows + det_rows);
    });
    if (once_err[dev] != cudaSuccess) return once_err[dev];
    auto kernel = vs.n == 1 ? det_sb ? k_project_bwd<DEG, VD, RED, true, true> : k_project_bwd<DEG, VD, RED, true, false>
                            : det_sb ? k_project_bwd<DEG, VD, RED, false, true> : k_project_bwd<DEG, VD, RED, false, false>;
    kernel<<<(unsigned)nb, bs, (vs.n == 1 ? rows : 2 * rows) + more, s>>>(g, vs, w, grec, out, det_sb);
    if (det_sb) {
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        k_det_sb_reduce<<<1, 256, 0, s>>>(det_sb, (int)nb, out.weight_params);
    }
    return cudaGetLastError();
}

template <bool VD, bool RED>
cudaError_t project_deg(const GaussPtrs& g, const Views& vs, WeightDev w, float* rec, cudaStream_t s) {
    switch (g.deg) {
        case 0: return project_t<0, VD, RED>(g, vs, w, rec, s);
        case 1: return project_t<1, VD, RED>(g, vs, w, rec, s);
        case 2: return project_t<2, VD, RED>(g, vs, w, rec, s);
        default: return project_t<3, VD, RED>(g, vs, w, rec, s);
    }
}

template <bool VD, bool RED>
cudaError_t project_bwd_deg(const GaussPtrs& g, const Views& vs, WeightDev w, const float* grec,
                            const wsr_grads& out, float* det_sb, cudaStream_t s) {
    switch (g.deg) {
        case 0: return project_bwd_t<0, VD, RED>(g, vs, w, grec, out, det_sb, s);
        case 1: return project_bwd_t<1, VD, RED>(g, vs, w, grec, out, det_sb, s);
        case 2: return project_bwd_t<2, VD, RED>(g, vs, w, grec, out, det_sb, s);
        default: return project_bwd_t<3, VD, RED>(g, vs, w, grec, out, det_sb, s);
    }
}

}  // namespace

cudaError_t launch_project(const GaussPtrs& g, const Views& vs, WeightDev w, float* rec, cudaStream_t s) {
    if (g.n == 0) return cudaSuccess;
    if (g.vd) return g.red ? project_deg<true, true>(g, vs, w, rec, s) : project_deg<true, false>(g, vs, w, rec, s);
    return g.red ? project_deg<false, true>(g, vs, w, rec, s) : project_deg<false, false>(g, vs, w, rec, s);
}

cudaError_t launch_project_bwd(const GaussPtrs& g, const Views& vs, WeightDev w, const float* grec,
                               const wsr_grads& out, float* det_sb, cudaStream_t s) {
    if (g.n == 0) return cudaSuccess;
    if (g.vd)
        return g.red ? project_bwd_deg<true, true>(g, vs, w, grec, out, det_sb, s)
                     : project_bwd_deg<true, false>(g, vs, w, grec, out, det_sb, s);
    return g.red ? project_bwd_deg<false, true>(g, vs, w, grec, out, det_sb, s)
                 : project_bwd_deg<false, false>(g, vs, w, grec, out, det_sb, s);
}

}  // namespace wsr
