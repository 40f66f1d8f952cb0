// DeepFlow (Sec. 4.3): variational refinement of a flow field with the
// DeepMatching matches as one of its terms.
//
// Energy E = int delta Psi(theta0 (grad3 I . w)^2) + gamma Psi(normalised
// gradient constancy) + alpha(x) Psi(|grad u|^2 + |grad v|^2) + beta_k c phi
// Psi(|w - w'|^2), Psi(s^2) = sqrt(s^2 + eps^2), minimised coarse to fine
// (factor eta) with warping; per level n_fixed fixed-point steps (the robust
// weights recomputed from the current increment), each solved approximately
// by n_sor red-black SOR sweeps.  Every step is a data-parallel pass over the
// pixels of one level; the arithmetic is FP32 with one fixed order of
// correctly rounded operations, the same as the FP32 reference.  The
// choices the paper leaves open (resampling, stencils, border rules, where a
// match lands on a coarse level, SOR ordering) are stated at each kernel.
//
// The SOR sweeps are sequential in time (each half-sweep needs the other
// colour's previous values), so the latency of a half-sweep and the launches,
// not the arithmetic, bound the solver: the smaller levels (up to 1024 pairs of pixels) run
// entirely in one CTA; larger levels run 8 half-sweeps per launch, temporally blocked
// (a tile plus an 8-pixel halo), which gives the same bits as 8 global half-sweeps.
// In both a thread keeps the edge weights and increments of its pixels in registers and reads
// its neighbours' current values and the constants of its own update from shared memory.
#include <math.h>

#include "dm_internal.cuh"

namespace {

struct DfConst {
    float scale, kappa, gamma, delta, zeta2, eps2, omega, one_m_omega, sigma_m, two_sigma_m, norm;
};

__device__ __forceinline__ float df_at(const float* f, int W, int x, int y) { return f[(size_t)y * W + x]; }

// Central differences with a replicated border.
__device__ __forceinline__ float df_dx(const float* f, int W, int x, int y) {
    return __fmul_rn(0.5f, __fsub_rn(df_at(f, W, x + 1 < W ? x + 1 : W - 1, y), df_at(f, W, x > 0 ? x - 1 : 0, y)));
}
__device__ __forceinline__ float df_dy(const float* f, int W, int H, int x, int y) {
    return __fmul_rn(0.5f, __fsub_rn(df_at(f, W, x, y + 1 < H ? y + 1 : H - 1), df_at(f, W, x, y > 0 ? y - 1 : 0)));
}

// Bilinear sample at (xs, ys), coordinates clamped to the image.
__device__ __forceinline__ float df_bilinear(const float* f, int W, int H, float xs, float ys) {
    xs = xs < 0.0f ? 0.0f : xs;
    ys = ys < 0.0f ? 0.0f : ys;
    xs = xs > (float)(W - 1) ? (float)(W - 1) : xs;
    ys = ys > (float)(H - 1) ? (float)(H - 1) : ys;
    const float fx0 = floorf(xs), fy0 = floorf(ys);
    const int x0 = (int)fx0, y0 = (int)fy0;
    const int x1 = x0 + 1 < W ? x0 + 1 : W - 1, y1 = y0 + 1 < H ? y0 + 1 : H - 1;
    const float fx = __fsub_rn(xs, fx0), fy = __fsub_rn(ys, fy0);
    const float p00 = df_at(f, W, x0, y0), p10 = df_at(f, W, x1, y0), p01 = df_at(f, W, x0, y1), p11 = df_at(f, W, x1, y1);
    const float top = __fadd_rn(p00, __fmul_rn(fx, __fsub_rn(p10, p00)));
    const float bot = __fadd_rn(p01, __fmul_rn(fx, __fsub_rn(p11, p01)));
    return __fadd_rn(top, __fmul_rn(fy, __fsub_rn(bot, top)));
}

// Psi'(s2) = 1 / (2 sqrt(s2 + eps^2)).
__device__ __forceinline__ float df_dpsi(float s2, float eps2) { return __fdiv_rn(0.5f, __fsqrt_rn(__fadd_rn(s2, eps2))); }

// Level resampling: dst pixel x samples src at (x + 1/2) / s - 1/2 (down,
// s = eta: the next coarser level) or (x + 1/2) s - 1/2 (up, s = eta: the
// flow carried to the finer level), times mul.
__global__ void k_df_resample(const float* __restrict__ src, int Ws, int Hs, float* __restrict__ dst, int Wd, int Hd,
                              float s, int down, float mul) {
    const long long n = (long long)Wd * Hd;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(i % Wd), y = (int)(i / Wd);
        const float cx = __fadd_rn((float)x, 0.5f), cy = __fadd_rn((float)y, 0.5f);
        const float xs = down ? __fsub_rn(__fdiv_rn(cx, s), 0.5f) : __fsub_rn(__fmul_rn(cx, s), 0.5f);
        const float ys = down ? __fsub_rn(__fdiv_rn(cy, s), 0.5f) : __fsub_rn(__fmul_rn(cy, s), 0.5f);
        dst[i] = __fmul_rn(df_bilinear(src, Ws, Hs, xs, ys), mul);
    }
}

__device__ __forceinline__ int df_clampi(int v, int lo, int hi) { return v < lo ? lo : (v > hi ? hi : v); }

__device__ __forceinline__ int df_count(const int* d_count, int capacity) {
    const int n = *d_count;
    return n < 0 ? 0 : (n > capacity ? capacity : n);
}

// Weight phi of each match at full resolution: lambda~ = 10 x the smaller
// eigenvalue of the 3x3 sum of gradient products of I1 around x1; Delta =
// |I1(x1) - I2(x2)| + |dx I1(x1) - dx I2(x2)| + |dy I1(x1) - dy I2(x2)|;
// phi = sqrt(lambda~) / (sigma_M sqrt(2 pi)) exp(-Delta / (2 sigma_M)).
__global__ void k_df_phi(const float* __restrict__ I1, const float* __restrict__ I2, int W, int H,
                         const dm_match_t* __restrict__ m, const int* __restrict__ d_count, int capacity, DfConst k,
                         float* __restrict__ phi) {
    const int n = df_count(d_count, capacity);
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int x1 = df_clampi((int)m[i].x1, 0, W - 1), y1 = df_clampi((int)m[i].y1, 0, H - 1);
        const int x2 = df_clampi((int)m[i].x2, 0, W - 1), y2 = df_clampi((int)m[i].y2, 0, H - 1);
        float a = 0.0f, b = 0.0f, c = 0.0f;
        for (int dy = -1; dy <= 1; dy++)
            for (int dx = -1; dx <= 1; dx++) {
                const int xx = df_clampi(x1 + dx, 0, W - 1), yy = df_clampi(y1 + dy, 0, H - 1);
                const float gx = df_dx(I1, W, xx, yy), gy = df_dy(I1, W, H, xx, yy);
                a = __fadd_rn(a, __fmul_rn(gx, gx));
                b = __fadd_rn(b, __fmul_rn(gx, gy));
                c = __fadd_rn(c, __fmul_rn(gy, gy));
            }
        const float h = __fmul_rn(__fsub_rn(a, c), 0.5f);
        float lmin = __fsub_rn(__fmul_rn(__fadd_rn(a, c), 0.5f), __fsqrt_rn(__fadd_rn(__fmul_rn(h, h), __fmul_rn(b, b))));
        if (lmin < 0.0f) lmin = 0.0f;
        const float lt = __fmul_rn(10.0f, lmin);
        float d = fabsf(__fsub_rn(df_at(I1, W, x1, y1), df_at(I2, W, x2, y2)));
        d = __fadd_rn(d, fabsf(__fsub_rn(df_dx(I1, W, x1, y1), df_dx(I2, W, x2, y2))));
        d = __fadd_rn(d, fabsf(__fsub_rn(df_dy(I1, W, H, x1, y1), df_dy(I2, W, H, x2, y2))));
        const float z = -__fdiv_rn(d, k.two_sigma_m);
        phi[i] = __fmul_rn(__fmul_rn(__fdiv_rn(__fsqrt_rn(lt), k.sigma_m), k.norm), dm_expf(z));
    }
}

// Matches on level k: match i lands on pixel round((x1 + 1/2) s_k - 1/2)
// (clamped); a pixel keeps the match with the higher DeepMatching score, then
// the lower index (64-bit key: order-preserving score bits, then ~index).
__device__ __forceinline__ unsigned int df_score_key(float s) {
    const unsigned int b = __float_as_uint(s);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

__global__ void k_df_raster(const dm_match_t* __restrict__ m, const int* __restrict__ d_count, int capacity, int w, int h,
                            float sk, unsigned long long* __restrict__ owner) {
    const int n = df_count(d_count, capacity);
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const float fx = __fsub_rn(__fmul_rn(__fadd_rn(m[i].x1, 0.5f), sk), 0.5f);
        const float fy = __fsub_rn(__fmul_rn(__fadd_rn(m[i].y1, 0.5f), sk), 0.5f);
        const int px = df_clampi((int)floorf(__fadd_rn(fx, 0.5f)), 0, w - 1);
        const int py = df_clampi((int)floorf(__fadd_rn(fy, 0.5f)), 0, h - 1);
        const unsigned long long key = ((unsigned long long)df_score_key(m[i].score) << 32) | (0xffffffffu - (unsigned int)i);
        atomicMax(owner + (size_t)py * w + px, key);
    }
}

// Per pixel: beta_k phi, u', v' of the winning match (0 where none).
__global__ void k_df_match_fields(const unsigned long long* __restrict__ owner, const dm_match_t* __restrict__ m,
                                  const float* __restrict__ phi, int n_px, float beta_k, float sk, float* __restrict__ mc,
                                  float* __restrict__ mu, float* __restrict__ mv) {
    for (int o = blockIdx.x * blockDim.x + threadIdx.x; o < n_px; o += gridDim.x * blockDim.x) {
        const unsigned long long key = owner[o];
        float c = 0.0f, a = 0.0f, b = 0.0f;
        if (key != 0ull) {
            const int i = (int)(0xffffffffu - (unsigned int)key);
            c = __fmul_rn(beta_k, phi[i]);
            a = __fmul_rn(__fsub_rn(m[i].x2, m[i].x1), sk);
            b = __fmul_rn(__fsub_rn(m[i].y2, m[i].y1), sk);
        }
        mc[o] = c;
        mu[o] = a;
        mv[o] = b;
    }
}

// Linearisation around the current flow, step 1: alpha(x) = exp(-kappa
// |grad I1| / 255), the warped I2w = I2(x + w) (bilinear, clamped) and the
// mean Im = (I1 + I2w) / 2.
__global__ void k_df_prep1(const float* __restrict__ I1, const float* __restrict__ I2, const float* __restrict__ u,
                           const float* __restrict__ v, int w, int h, DfConst k, float* __restrict__ alpha,
                           float* __restrict__ I2w, float* __restrict__ Im) {
    const long long n = (long long)w * h;
    for (long long o = (long long)blockIdx.x * blockDim.x + threadIdx.x; o < n; o += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(o % w), y = (int)(o / w);
        const float gx = __fdiv_rn(df_dx(I1, w, x, y), k.scale), gy = __fdiv_rn(df_dy(I1, w, h, x, y), k.scale);
        alpha[o] = dm_expf(-__fmul_rn(k.kappa, __fsqrt_rn(__fadd_rn(__fmul_rn(gx, gx), __fmul_rn(gy, gy)))));
        const float wv = df_bilinear(I2, w, h, __fadd_rn((float)x, u[o]), __fadd_rn((float)y, v[o]));
        I2w[o] = wv;
        Im[o] = __fmul_rn(0.5f, __fadd_rn(I1[o], wv));
    }
}

// Step 2: first derivatives of the mean image.
__global__ void k_df_prep2(const float* __restrict__ Im, int w, int h, float* __restrict__ Ix, float* __restrict__ Iy) {
    const long long n = (long long)w * h;
    for (long long o = (long long)blockIdx.x * blockDim.x + threadIdx.x; o < n; o += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(o % w), y = (int)(o / w);
        Ix[o] = df_dx(Im, w, x, y);
        Iy[o] = df_dy(Im, w, h, x, y);
    }
}

// Step 3: the 11 per-pixel data-term quantities D = (Ix, Iy, Iz, Ixx, Ixy,
// Iyy, Ixz, Iyz, theta0, thetax, thetay), structure-of-arrays with stride n:
// Iz = I2w - I1; Ixx = dx(Ix), Ixy = dy(Ix), Iyy = dy(Iy); Ixz = dx(I2w) -
// dx(I1), Iyz = dy(I2w) - dy(I1); theta0 = 1 / (Ix^2 + Iy^2 + zeta^2),
// thetax = 1 / (Ixx^2 + Ixy^2 + zeta^2), thetay = 1 / (Ixy^2 + Iyy^2 + zeta^2).
__global__ void k_df_prep3(const float* __restrict__ I1, const float* __restrict__ I2w, const float* __restrict__ Ixa,
                           const float* __restrict__ Iya, int w, int h, DfConst k, float* __restrict__ D,
                           unsigned int* __restrict__ published) {
    const long long n = (long long)w * h;
    if (blockIdx.x == 0 && threadIdx.x == 0) *published = 0u;        // for the level's fixed-point steps (k_df_weights)
    for (long long o = (long long)blockIdx.x * blockDim.x + threadIdx.x; o < n; o += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(o % w), y = (int)(o / w);
        const float Ix = Ixa[o], Iy = Iya[o];
        const float Ixx = df_dx(Ixa, w, x, y), Ixy = df_dy(Ixa, w, h, x, y), Iyy = df_dy(Iya, w, h, x, y);
        D[o] = Ix;
        D[n + o] = Iy;
        D[2 * n + o] = __fsub_rn(I2w[o], I1[o]);
        D[3 * n + o] = Ixx;
        D[4 * n + o] = Ixy;
        D[5 * n + o] = Iyy;
        D[6 * n + o] = __fsub_rn(df_dx(I2w, w, x, y), df_dx(I1, w, x, y));
        D[7 * n + o] = __fsub_rn(df_dy(I2w, w, h, x, y), df_dy(I1, w, h, x, y));
        D[8 * n + o] = __fdiv_rn(1.0f, __fadd_rn(__fadd_rn(__fmul_rn(Ix, Ix), __fmul_rn(Iy, Iy)), k.zeta2));
        D[9 * n + o] = __fdiv_rn(1.0f, __fadd_rn(__fadd_rn(__fmul_rn(Ixx, Ixx), __fmul_rn(Ixy, Ixy)), k.zeta2));
        D[10 * n + o] = __fdiv_rn(1.0f, __fadd_rn(__fadd_rn(__fmul_rn(Ixy, Ixy), __fmul_rn(Iyy, Iyy)), k.zeta2));
    }
}

// Fixed-point step, per pixel o: the smoothness weight psi_s = alpha
// Psi'(|grad(u + du)|^2 + |grad(v + dv)|^2) from forward differences (0 at the
// last column / row), the robust data and matching weights at the current
// increment, and the 2x2 system A = (A11, A12, A22, b1, b2) (structure of
// arrays, stride n).
struct DfLevel {
    int w, h;
    long long n;
    const float* D;        // [11][n]
    const float* alpha;
    const float* mc;       // beta_k phi at matched pixels, else 0
    const float* mu;
    const float* mv;
    const float* u;
    const float* v;
    float* du;
    float* dv;
    float* A;              // [5][n]
    float* ps;
};

// The fixed-point step's arithmetic for one pixel, on values: the
// smoothness weight from the forward differences of u + du, v + dv (has_r /
// has_d: the right / lower neighbour exists), the data and matching weights
// and the 2x2 system (A11, A12, A22, b1, b2).
struct DfPix {
    float ps, a11, a12, a22, b1, b2;
};

__device__ __forceinline__ DfPix df_weights_vals(float u, float du, float v, float dv, bool has_r, float Ur, float Vr,
                                                 bool has_d, float Ud, float Vd, const float* d, float alpha, float mc, float mu, float mv,
                                                 const DfConst& k) {
    const float U = __fadd_rn(u, du), V = __fadd_rn(v, dv);
    float ux = 0.0f, uy = 0.0f, vx = 0.0f, vy = 0.0f;
    if (has_r) {
        ux = __fsub_rn(Ur, U);
        vx = __fsub_rn(Vr, V);
    }
    if (has_d) {
        uy = __fsub_rn(Ud, U);
        vy = __fsub_rn(Vd, V);
    }
    DfPix r;
    const float s2 = __fadd_rn(__fadd_rn(__fadd_rn(__fmul_rn(ux, ux), __fmul_rn(uy, uy)), __fmul_rn(vx, vx)), __fmul_rn(vy, vy));
    r.ps = __fmul_rn(alpha, df_dpsi(s2, k.eps2));
    const float d0 = d[0], d1 = d[1], d2 = d[2], d3 = d[3], d4 = d[4], d5 = d[5], d6 = d[6], d7 = d[7], d8 = d[8];
    const float d9 = d[9], d10 = d[10];
    float a0 = 0.0f;
    if (k.delta > 0.0f) {
        const float r0 = __fadd_rn(__fadd_rn(__fmul_rn(d0, du), __fmul_rn(d1, dv)), d2);
        a0 = __fmul_rn(__fmul_rn(k.delta, df_dpsi(__fmul_rn(d8, __fmul_rn(r0, r0)), k.eps2)), d8);
    }
    const float rx = __fadd_rn(__fadd_rn(__fmul_rn(d3, du), __fmul_rn(d4, dv)), d6);
    const float ry = __fadd_rn(__fadd_rn(__fmul_rn(d4, du), __fmul_rn(d5, dv)), d7);
    const float ag = __fmul_rn(k.gamma, df_dpsi(__fadd_rn(__fmul_rn(d9, __fmul_rn(rx, rx)), __fmul_rn(d10, __fmul_rn(ry, ry))), k.eps2));
    float mw = 0.0f;
    if (mc > 0.0f) {
        const float eu = __fsub_rn(U, mu), ev = __fsub_rn(V, mv);
        mw = __fmul_rn(mc, df_dpsi(__fadd_rn(__fmul_rn(eu, eu), __fmul_rn(ev, ev)), k.eps2));
    }
    const float gx = __fmul_rn(ag, d9), gy = __fmul_rn(ag, d10);
    const float a0x = __fmul_rn(a0, d0), a0y = __fmul_rn(a0, d1);
    r.a11 = __fadd_rn(__fadd_rn(__fmul_rn(a0x, d0), __fadd_rn(__fmul_rn(__fmul_rn(gx, d3), d3), __fmul_rn(__fmul_rn(gy, d4), d4))), mw);
    r.a12 = __fadd_rn(__fmul_rn(a0x, d1), __fadd_rn(__fmul_rn(__fmul_rn(gx, d3), d4), __fmul_rn(__fmul_rn(gy, d4), d5)));
    r.a22 = __fadd_rn(__fadd_rn(__fmul_rn(a0y, d1), __fadd_rn(__fmul_rn(__fmul_rn(gx, d4), d4), __fmul_rn(__fmul_rn(gy, d5), d5))), mw);
    r.b1 = __fsub_rn(-__fadd_rn(__fmul_rn(a0x, d2), __fadd_rn(__fmul_rn(__fmul_rn(gx, d3), d6), __fmul_rn(__fmul_rn(gy, d4), d7))),
                     __fmul_rn(mw, __fsub_rn(u, mu)));
    r.b2 = __fsub_rn(-__fadd_rn(__fmul_rn(a0y, d2), __fadd_rn(__fmul_rn(__fmul_rn(gx, d4), d6), __fmul_rn(__fmul_rn(gy, d5), d7))),
                     __fmul_rn(mw, __fsub_rn(v, mv)));
    return r;
}

__device__ __forceinline__ void df_load_d(const float* D, long long n, long long o, float* d) {
#pragma unroll
    for (int j = 0; j < 11; j++) d[j] = D[j * n + o];
}

__device__ __forceinline__ void df_weights_at(const DfLevel& L, const DfConst& k, long long o) {
    const int x = (int)(o % L.w), y = (int)(o / L.w);
    const bool hr = x + 1 < L.w, hd = y + 1 < L.h;
    const long long r = hr ? o + 1 : o, dn = hd ? o + L.w : o;
    float d[11];
    df_load_d(L.D, L.n, o, d);
    const DfPix q = df_weights_vals(L.u[o], L.du[o], L.v[o], L.dv[o], hr, __fadd_rn(L.u[r], L.du[r]),
                                    __fadd_rn(L.v[r], L.dv[r]), hd, __fadd_rn(L.u[dn], L.du[dn]),
                                    __fadd_rn(L.v[dn], L.dv[dn]), d, L.alpha[o], L.mc[o], L.mu[o], L.mv[o], k);
    const long long n = L.n;
    L.ps[o] = q.ps;
    L.A[o] = q.a11;
    L.A[n + o] = q.a12;
    L.A[2 * n + o] = q.a22;
    L.A[3 * n + o] = q.b1;
    L.A[4 * n + o] = q.b2;
}

// ---------------------------------------------------------------------------
// Red-black SOR in a CTA.  One relaxation of a pixel o from its existing
// 4-neighbours p (left, right, up, down), edge weights w_p = (ps_o + ps_p) / 2:
//   du = (1 - omega) du + omega (b1 + sum w_p ((du_p + u_p) - u_o) - A12 dv) / (A11 + sum w_p),
// then dv the same way with the new du.
//
// A thread owns pairs of horizontally neighbouring pixels, one of each colour, so
// every thread updates a pixel in every half-sweep.  What does not change during
// the sweeps is formed once: the edge weights (0 for a missing neighbour: the
// terms it adds are zeros, which leave the sums unchanged), the two diagonals and
// their reciprocals.  Shared memory holds, in one plane per colour (a warp's
// accesses are then consecutive), the sums (du + u, dv + v) that the neighbours
// read -- one 8-byte load each -- and the constants of the pixel's own update.
// Against reading ps, du, u, dv, v of every neighbour
// and two divisions per update this shortens the chain of an update to less than half:
// the blocked launch of a level of a few tiles 12.6 -> 7.4 us, of 1024x436 45.7 -> 29.1,
// a one-CTA level 220 -> 100 us; with the launches of a fixed-point step overlapped
// (programmatic dependence) a 1024x436 pair 39.2 -> 26.3 -> 20.3 ms.
constexpr int SOR_INV = 7;       // planes of constants: A12, b1, b2, A11 + w, 1 / that, A22 + w, 1 / that

struct SorPx {
    float wl, wr, wu, wd;        // edge weights
    float u, v, du, dv;
};

// a / d correctly rounded, y = RN(1 / d): the quotient estimate with two remainder
// corrections (Markstein: the remainder of an fma is exact, and with a correctly
// rounded reciprocal the correction of a quotient that is off by less than an ulp
// rounds correctly).  Outside the range where no remainder can underflow -- and
// for the d that sor_setup marks with lo = infinity -- the division itself.
__device__ __forceinline__ float df_div(float a, float d, float y, float lo) {
    const float m = fabsf(a);
    if (!(m >= lo && m <= 1.0e24f)) return __fdiv_rn(a, d);
    float q = __fmul_rn(a, y);
    q = __fmaf_rn(__fmaf_rn(-d, q, a), y, q);
    return __fmaf_rn(__fmaf_rn(-d, q, a), y, q);
}

// The constants of one pixel from its system and its neighbours' ps (has_*: the
// neighbour exists); returns false where a diagonal lies outside df_div's range.
__device__ __forceinline__ bool sor_setup(SorPx& p, float* inv, int stride, float pso, bool hl, float psl, bool hr, float psr,
                                          bool hu, float psu, bool hd, float psd, float a11, float a12, float a22, float b1,
                                          float b2) {
    p.wl = hl ? __fmul_rn(0.5f, __fadd_rn(pso, psl)) : 0.0f;
    p.wr = hr ? __fmul_rn(0.5f, __fadd_rn(pso, psr)) : 0.0f;
    p.wu = hu ? __fmul_rn(0.5f, __fadd_rn(pso, psu)) : 0.0f;
    p.wd = hd ? __fmul_rn(0.5f, __fadd_rn(pso, psd)) : 0.0f;
    const float sw = __fadd_rn(__fadd_rn(__fadd_rn(p.wl, p.wr), p.wu), p.wd);
    const float d1 = __fadd_rn(a11, sw), d2 = __fadd_rn(a22, sw);
    inv[0] = a12;
    inv[stride] = b1;
    inv[2 * stride] = b2;
    inv[3 * stride] = d1;
    inv[4 * stride] = __frcp_rn(d1);
    inv[5 * stride] = d2;
    inv[6 * stride] = __frcp_rn(d2);
    return fminf(d1, d2) >= 1.0e-12f && fmaxf(d1, d2) <= 1.0e12f;
}

// The other colour's neighbours of a pixel of pair e (planes of `pw` pairs per row): the
// pixel of colour c lies at column 2 i + off of its row, its left and right
// neighbours in pairs e - 1 + off and e + off, the upper and lower ones in e -+ pw.
// A neighbour that does not exist has weight 0 and its element holds zeros: the planes have
// guard elements before and after, and where a row could run into the next one (its end is
// its successor's left neighbour) an element of padding.  (Weight 0 times whatever lies
// there would carry a NaN or an infinity from one border to the other.)
__device__ __forceinline__ void sor_update(SorPx& p, float2* mine, const float2* other, int off, int pw, const float* inv,
                                           int stride, float lo, const DfConst& k) {
    const float2 l = other[off - 1], r = other[off], t = other[-pw], b = other[pw];
    const float a12 = inv[0], b1 = inv[stride], b2 = inv[2 * stride];
    const float d1 = inv[3 * stride], y1 = inv[4 * stride], d2 = inv[5 * stride], y2 = inv[6 * stride];
    float su = __fmul_rn(p.wl, __fsub_rn(l.x, p.u)), sv = __fmul_rn(p.wl, __fsub_rn(l.y, p.v));
    su = __fadd_rn(su, __fmul_rn(p.wr, __fsub_rn(r.x, p.u)));
    sv = __fadd_rn(sv, __fmul_rn(p.wr, __fsub_rn(r.y, p.v)));
    su = __fadd_rn(su, __fmul_rn(p.wu, __fsub_rn(t.x, p.u)));
    sv = __fadd_rn(sv, __fmul_rn(p.wu, __fsub_rn(t.y, p.v)));
    su = __fadd_rn(su, __fmul_rn(p.wd, __fsub_rn(b.x, p.u)));
    sv = __fadd_rn(sv, __fmul_rn(p.wd, __fsub_rn(b.y, p.v)));
    const float nu = __fsub_rn(__fadd_rn(b1, su), __fmul_rn(a12, p.dv));
    p.du = __fadd_rn(__fmul_rn(k.one_m_omega, p.du), __fmul_rn(k.omega, df_div(nu, d1, y1, lo)));
    const float nv = __fsub_rn(__fadd_rn(b2, sv), __fmul_rn(a12, p.du));
    p.dv = __fadd_rn(__fmul_rn(k.one_m_omega, p.dv), __fmul_rn(k.omega, df_div(nv, d2, y2, lo)));
    *mine = make_float2(__fadd_rn(p.du, p.u), __fadd_rn(p.dv, p.v));
}

// The systems and smoothness weights of a fixed-point step; every CTA publishes its share by a
// release (its threads' writes are ordered before it by the barrier), so that whoever
// acquires the count of all CTAs may read them, and what this kernel found written (u, v).
__global__ void k_df_weights(DfLevel L, DfConst k, unsigned int* published) {
    for (long long o = (long long)blockIdx.x * blockDim.x + threadIdx.x; o < L.n; o += (long long)gridDim.x * blockDim.x)
        df_weights_at(L, k, o);
    __syncthreads();
    if (threadIdx.x == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" :: "l"(published) : "memory");
}

__device__ __forceinline__ bool df_acquired(const unsigned int* published, unsigned int count) {
    unsigned int c;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(c) : "l"(published) : "memory");
    return c == count;
}

// Temporally blocked red-black SOR: a CTA owns a TB_W x TB_H tile and stages
// it with a halo of S pixels (S = the half-sweeps of this launch, even, <= TB_S) in
// shared memory and registers, then runs S half-sweeps there, colours 0, 1, 0, ...
// Half-sweep j updates the pixels of its colour in the staged region shrunk by
// j + 1 on every side that is not the image border: their neighbours then
// hold exactly the values the global sweep would give them, so after S
// half-sweeps the tile itself is exact and is written back -- the same bits
// as S global half-sweeps, with one launch and no global barrier between them.
// The halos of other CTAs overlap this tile, so the increments are read from
// L.du / L.dv and written to a second pair of buffers (ping-pong between
// launches): no CTA ever sees another's updates of the same launch.
constexpr int TB_W = 32, TB_H = 16, TB_S = 8;
constexpr int TB_LW = TB_W + 2 * TB_S, TB_LH = TB_H + 2 * TB_S;
constexpr int TB_PW = TB_LW / 2, TB_PAIRS = TB_PW * TB_LH;       // 24 x 32 pairs, one per thread
constexpr int TB_THREADS = TB_PAIRS;
constexpr int TB_PLANE = TB_PAIRS + 2 * TB_PW;                   // with guards
constexpr size_t TB_SMEM = (size_t)(4 * TB_PLANE + 2 * SOR_INV * TB_PAIRS) * sizeof(float);
static_assert(TB_S % 2 == 0 && TB_W % 2 == 0, "a launch starts with colour 0 and the staged region at an even column");

// Every launch depends programmatically on the one before it (dm_launch_pdl): its CTAs become
// resident while that one's last ones run.  What it reads that its predecessor does not
// write (u, v, ps, A) it stages meanwhile, and only its increments after the wait.  The wait
// covers the predecessor alone, so the early reads are ordered by the count that
// k_df_weights publishes: a thread that acquires `count` (the CTAs of all weights launches
// of the level so far) reads what that kernel wrote or found written; any other value --
// and count = 0, the first launch of a step, whose predecessor is the weights kernel
// -- and it waits first.
// (Everything staged after the wait: a 1024x436 pair 22.3 ms instead of 20.4.)
__global__ void __launch_bounds__(TB_THREADS, 2) k_df_sor_tb(DfLevel L, DfConst k, int S, const unsigned int* published,
                                                             unsigned int count, float* __restrict__ out_du,
                                                             float* __restrict__ out_dv) {
    extern __shared__ __align__(16) float sm[];
    // per colour: the sums, the constants of this thread's pixel
    float2* cur[2] = {reinterpret_cast<float2*>(sm) + TB_PW + threadIdx.x,
                      reinterpret_cast<float2*>(sm) + TB_PLANE + TB_PW + threadIdx.x};
    float* inv[2] = {sm + 4 * TB_PLANE + threadIdx.x, sm + 4 * TB_PLANE + SOR_INV * TB_PAIRS + threadIdx.x};
    float* sps = sm;                                     // [TB_LH][TB_LW], before the sums take its place
    const int tiles_x = (L.w + TB_W - 1) / TB_W;
    const int tx0 = (blockIdx.x % tiles_x) * TB_W, ty0 = (blockIdx.x / tiles_x) * TB_H;
    const int tx1 = min(tx0 + TB_W, L.w), ty1 = min(ty0 + TB_H, L.h);
    const int lx0 = max(tx0 - S, 0) & ~1, ly0 = max(ty0 - S, 0);
    const int lx1 = min(tx1 + S, L.w), ly1 = min(ty1 + S, L.h);
    const int lw = lx1 - lx0, lh = ly1 - ly0;
    const long long n = L.n;
    const int i = threadIdx.x % TB_PW, y = threadIdx.x / TB_PW, gy = ly0 + y;
    const int flip = (lx0 + gy) & 1;                     // offset of colour 0 in this row's pairs
    // colour c of the pair lies at column 2 i + (c ^ flip)
    SorPx px[2];
    int act[2];                                          // half-sweeps in which the pixel is updated: j < act
    float ps[2], A[2][5];
    bool in[2];
    const bool early = count != 0u && df_acquired(published, count);
    if (!early) dm_pdl_wait();
#pragma unroll
    for (int c = 0; c < 2; c++) {
        const int x = 2 * i + (c ^ flip);
        in[c] = x < lw && y < lh;
        const long long o = in[c] ? (long long)gy * L.w + (lx0 + x) : 0;
        px[c].u = L.u[o];
        px[c].v = L.v[o];
        ps[c] = L.ps[o];
#pragma unroll
        for (int j = 0; j < 5; j++) A[c][j] = L.A[j * n + o];
        sps[y * TB_LW + x] = ps[c];
    }
    __syncthreads();
    bool ok = true;
#pragma unroll
    for (int c = 0; c < 2; c++) {
        const int x = 2 * i + (c ^ flip), gx = lx0 + x;
        const bool hl = gx > 0, hr = gx + 1 < L.w, hu = gy > 0, hd = gy + 1 < L.h;
        auto at = [&](int yy, int xx) { return xx >= 0 && xx < TB_LW && yy >= 0 && yy < TB_LH ? sps[yy * TB_LW + xx] : 0.0f; };
        // half-sweep j updates the staged region shrunk by j + 1 on sides that are not
        // the image border
        act[c] = in[c] ? S : 0;
        if (lx0 > 0) act[c] = min(act[c], x);
        if (ly0 > 0) act[c] = min(act[c], y);
        if (lx1 < L.w) act[c] = min(act[c], lw - 1 - x);
        if (ly1 < L.h) act[c] = min(act[c], lh - 1 - y);
        const bool good = sor_setup(px[c], inv[c], TB_PAIRS, ps[c], hl, at(y, x - 1), hr, at(y, x + 1), hu, at(y - 1, x),
                                    hd, at(y + 1, x), A[c][0], A[c][1], A[c][2], A[c][3], A[c][4]);
        ok = ok && (good || act[c] <= 0);
    }
    __syncthreads();                                     // ps read
    if (early) dm_pdl_wait();
#pragma unroll
    for (int c = 0; c < 2; c++) {
        const long long o = in[c] ? (long long)gy * L.w + (lx0 + 2 * i + (c ^ flip)) : 0;
        px[c].du = L.du[o];
        px[c].dv = L.dv[o];
        // (zeros past the image's right and lower border; a staged region that has none to spare
        // there ends 8 columns or rows past its tile, and what its last ones read does not
        // reach the tile in 8 half-sweeps)
        cur[c][0] = in[c] ? make_float2(__fadd_rn(px[c].du, px[c].u), __fadd_rn(px[c].dv, px[c].v)) : make_float2(0.0f, 0.0f);
        if (threadIdx.x < TB_PW) cur[c][-TB_PW] = cur[c][TB_PAIRS] = make_float2(0.0f, 0.0f);
    }
    const float lo = ok ? 1.0e-24f : INFINITY;
    __syncthreads();
    for (int j = 0; j < S; j += 2) {
        if (j < act[0]) sor_update(px[0], cur[0], cur[1], flip, TB_PW, inv[0], TB_PAIRS, lo, k);
        __syncthreads();
        if (j + 1 < act[1]) sor_update(px[1], cur[1], cur[0], flip ^ 1, TB_PW, inv[1], TB_PAIRS, lo, k);
        __syncthreads();
    }
#pragma unroll
    for (int c = 0; c < 2; c++) {
        const int gx = lx0 + 2 * i + (c ^ flip);
        if (gx >= tx0 && gx < tx1 && gy >= ty0 && gy < ty1) {
            const long long o = (long long)gy * L.w + gx;
            out_du[o] = px[c].du;
            out_dv[o] = px[c].dv;
        }
    }
}

__global__ void k_df_update(float* __restrict__ u, float* __restrict__ v, const float* __restrict__ du,
                            const float* __restrict__ dv, long long n) {
    for (long long o = (long long)blockIdx.x * blockDim.x + threadIdx.x; o < n; o += (long long)gridDim.x * blockDim.x) {
        u[o] = __fadd_rn(u[o], du[o]);
        v[o] = __fadd_rn(v[o], dv[o]);
    }
}

// A whole small level in one CTA: n_fixed x (weights, then n_sor red-black sweeps)
// with block barriers between the passes, then w += dw.  The same per-pixel
// arithmetic as the multi-launch path.  One pair of pixels per thread.
constexpr int DF_SMALL_THREADS = 1024;
// Pairs of a level solved by one CTA (a row of w pixels holds (w + 1) / 2): with two
// pairs per thread, up to 2048, a 1024x436 pair took 0.4 ms longer (spilled registers).
constexpr int DF_SMALL_PAIRS = DF_SMALL_THREADS;
// sums (two planes of h + 2 rows of pw + 1 elements, the guards and the padding among them: at most
// 3 pairs + 3 for pw h <= pairs), constants, psi_s
constexpr size_t DF_SMALL_SMEM = (size_t)(4 * (3 * DF_SMALL_PAIRS + 3) + 2 * (SOR_INV + 1) * DF_SMALL_PAIRS) * sizeof(float);

__global__ void __launch_bounds__(DF_SMALL_THREADS) k_df_level_small(DfLevel L, DfConst k, int n_fixed, int n_sor) {
    extern __shared__ __align__(16) float sm[];
    const int w = L.w, h = L.h, pw = (w + 1) / 2, np = pw * h, row = pw + 1, plane = row * (h + 2);
    const long long n = L.n;
    float2* cur[2] = {reinterpret_cast<float2*>(sm) + row, reinterpret_cast<float2*>(sm) + plane + row};
    float* inv[2] = {sm + 4 * plane, sm + 4 * plane + SOR_INV * np};
    float* sps[2] = {sm + 4 * plane + 2 * SOR_INV * np, sm + 4 * plane + (2 * SOR_INV + 1) * np};      // psi_s per colour
    const int e = threadIdx.x, y = e / pw, i = e - y * pw, flip = y & 1, at = y * row + i;      // the pair, its sums
    SorPx px[2];                                         // per colour, at column 2 i + (c ^ flip)
    bool in[2];
#pragma unroll
    for (int c = 0; c < 2; c++) {
        SorPx& p = px[c];
        const int x = 2 * i + (c ^ flip);
        in[c] = e < np && x < w;
        p.u = p.v = p.du = p.dv = p.wl = p.wr = p.wu = p.wd = 0.0f;
        if (in[c]) {
            p.u = L.u[(long long)y * w + x];
            p.v = L.v[(long long)y * w + x];
        }
        if (e < np) cur[c][at] = make_float2(p.u, p.v);  // du = dv = 0
        if (e < np && i == pw - 1) cur[c][at + 1] = make_float2(0.0f, 0.0f);
        for (int g = e; g < row; g += blockDim.x) cur[c][g - row] = cur[c][row * h + g] = make_float2(0.0f, 0.0f);
    }
    __syncthreads();
    for (int it = 0; it < n_fixed; it++) {
        // systems and smoothness weights: u + du and v + dv of the right and lower
        // neighbours are the sums in `cur`
        DfPix a[2];
#pragma unroll
        for (int c = 0; c < 2; c++) {
            if (!in[c]) continue;
            const SorPx& p = px[c];
            const int x = 2 * i + (c ^ flip);
            const long long o = (long long)y * w + x;
            const float2 r = cur[c ^ 1][at + (c ^ flip)], b = cur[c ^ 1][at + row];
            float d[11];
            df_load_d(L.D, n, o, d);
            a[c] = df_weights_vals(p.u, p.du, p.v, p.dv, x + 1 < w, r.x, r.y, y + 1 < h, b.x, b.y, d, L.alpha[o], L.mc[o],
                                   L.mu[o], L.mv[o], k);
            sps[c][e] = a[c].ps;
        }
        __syncthreads();
        bool ok = true;
#pragma unroll
        for (int c = 0; c < 2; c++) {
            if (!in[c]) continue;
            const int x = 2 * i + (c ^ flip), off = c ^ flip;
            const float* ps = sps[c ^ 1];
            const bool hl = x > 0, hr = x + 1 < w, hu = y > 0, hd = y + 1 < h;
            const bool good = sor_setup(px[c], inv[c] + e, np, a[c].ps, hl, hl ? ps[e - 1 + off] : 0.0f, hr, hr ? ps[e + off] : 0.0f,
                                        hu, hu ? ps[e - pw] : 0.0f, hd, hd ? ps[e + pw] : 0.0f, a[c].a11, a[c].a12, a[c].a22,
                                        a[c].b1, a[c].b2);
            ok = ok && good;
        }
        const float lo = ok ? 1.0e-24f : INFINITY;
        for (int s = 0; s < n_sor; s++) {
            if (in[0]) sor_update(px[0], cur[0] + at, cur[1] + at, flip, row, inv[0] + e, np, lo, k);
            __syncthreads();
            if (in[1]) sor_update(px[1], cur[1] + at, cur[0] + at, flip ^ 1, row, inv[1] + e, np, lo, k);
            __syncthreads();
        }
    }
    float* u = const_cast<float*>(L.u);
    float* v = const_cast<float*>(L.v);
#pragma unroll
    for (int c = 0; c < 2; c++)
        if (in[c]) {
            const long long o = (long long)y * w + 2 * i + (c ^ flip);
            u[o] = __fadd_rn(px[c].u, px[c].du);
            v[o] = __fadd_rn(px[c].v, px[c].dv);
        }
}

}  // namespace

// ---------------------------------------------------------------------------
// Host side: the plan (level sizes, constants, workspace) and the launches.
// ---------------------------------------------------------------------------
namespace {
constexpr double kPi = 3.14159265358979323846;
inline unsigned df_blocks(long long n) {
    const long long b = (n + 255) / 256;
    return (unsigned)(b < 4096 ? (b > 0 ? b : 1) : 4096);
}
}  // namespace

void dm_flow_plan(int W, int H, int capacity, const dm_flow_params& p, DmFlowPlan* q) {
    memset(q, 0, sizeof(*q));
    q->ws[0] = W;
    q->hs[0] = H;
    int n = 1;
    while (n < DM_DF_MAXLEVELS) {
        const int w = (int)floor(p.eta * q->ws[n - 1] + 0.5), h = (int)floor(p.eta * q->hs[n - 1] + 0.5);
        if (w < p.min_size || h < p.min_size) break;
        q->ws[n] = w;
        q->hs[n] = h;
        n++;
    }
    q->nl = n;
    const int kmax = n - 1;
    for (int k = 0; k < n; k++) {
        q->beta_k[k] = (float)(kmax > 0 ? p.beta * pow((double)k / (double)kmax, p.b) : p.beta);
        q->sk[k] = (float)pow(p.eta, (double)k);
    }
    q->eta = (float)p.eta;
    q->inv_eta = 1.0f / q->eta;
    q->scale = (float)p.image_scale;
    q->kappa = (float)p.kappa;
    q->gamma = (float)p.gamma;
    q->delta = (float)p.delta;
    q->zeta2 = (float)(p.zeta * p.zeta);
    q->eps2 = (float)(p.eps * p.eps);
    q->omega = (float)p.omega;
    q->one_m_omega = 1.0f - q->omega;
    q->sigma_m = (float)p.sigma_m;
    q->two_sigma_m = 2.0f * q->sigma_m;
    q->norm = (float)(1.0 / sqrt(2.0 * kPi));
    q->n_fixed = p.n_fixed;
    q->n_sor = p.n_sor;
    q->capacity = capacity;
    // workspace (floats unless stated): both pyramids, flow ping-pong, per-level scratch
    const size_t N0 = (size_t)W * H;
    size_t off = 0;
    for (int k = 0; k < n; k++) {
        const size_t Nk = (size_t)q->ws[k] * q->hs[k];
        q->P1[k] = off; off = dm_align(off + Nk * 4);
        q->P2[k] = off; off = dm_align(off + Nk * 4);
    }
    size_t* one[] = {&q->tmp, &q->fa_u, &q->fa_v, &q->fb_u, &q->fb_v, &q->du, &q->dv, &q->du2, &q->dv2, &q->alpha, &q->I2w, &q->Im,
                     &q->Ix, &q->Iy, &q->ps, &q->mc, &q->mu, &q->mv};
    for (size_t* f : one) { *f = off; off = dm_align(off + N0 * 4); }
    q->D = off; off = dm_align(off + N0 * 11 * 4);
    q->A = off; off = dm_align(off + N0 * 5 * 4);
    q->owner = off; off = dm_align(off + N0 * 8);
    q->phi = off; off = dm_align(off + (size_t)(capacity > 0 ? capacity : 1) * 4);
    q->bytes = off;
}

cudaError_t dm_launch_deepflow(const DmFlowPlan& q, const DmTaps& taps, const float* img1, const float* img2,
                               const dm_match_t* m, const int* d_count, float* out_u, float* out_v, char* ws,
                               cudaStream_t st) {
    auto F = [&](size_t off) { return reinterpret_cast<float*>(ws + off); };
    DfConst k;
    k.scale = q.scale; k.kappa = q.kappa; k.gamma = q.gamma; k.delta = q.delta; k.zeta2 = q.zeta2; k.eps2 = q.eps2;
    k.omega = q.omega; k.one_m_omega = q.one_m_omega; k.sigma_m = q.sigma_m; k.two_sigma_m = q.two_sigma_m;
    k.norm = q.norm;
    const int W = q.ws[0], H = q.hs[0];
    long long launches = 0;
    cudaError_t e;
    static std::atomic<unsigned long long> tb_done{0}, small_done{0};
    if ((e = dm_smem_opt_in(reinterpret_cast<const void*>(k_df_sor_tb), (int)TB_SMEM, tb_done)) != cudaSuccess) return e;
    if ((e = dm_smem_opt_in(reinterpret_cast<const void*>(k_df_level_small), (int)DF_SMALL_SMEM, small_done)) != cudaSuccess)
        return e;
    if ((e = dm_launch_smooth1(img1, W, H, q.scale, taps, F(q.P1[0]), F(q.tmp), st)) != cudaSuccess) return e;
    if ((e = dm_launch_smooth1(img2, W, H, q.scale, taps, F(q.P2[0]), F(q.tmp), st)) != cudaSuccess) return e;
    for (int l = 1; l < q.nl; l++) {
        const long long n = (long long)q.ws[l] * q.hs[l];
        k_df_resample<<<df_blocks(n), 256, 0, st>>>(F(q.P1[l - 1]), q.ws[l - 1], q.hs[l - 1], F(q.P1[l]), q.ws[l], q.hs[l],
                                                    q.eta, 1, 1.0f);
        k_df_resample<<<df_blocks(n), 256, 0, st>>>(F(q.P2[l - 1]), q.ws[l - 1], q.hs[l - 1], F(q.P2[l]), q.ws[l], q.hs[l],
                                                    q.eta, 1, 1.0f);
        launches += 2;
    }
    const bool has_m = m != nullptr && d_count != nullptr && q.capacity > 0;
    if (has_m) {
        k_df_phi<<<df_blocks(q.capacity), 256, 0, st>>>(F(q.P1[0]), F(q.P2[0]), W, H, m, d_count, q.capacity, k, F(q.phi));
        launches++;
    }
    float* cu = F(q.fa_u);
    float* cv = F(q.fa_v);
    float* nu = F(q.fb_u);
    float* nv = F(q.fb_v);
    for (int l = q.nl - 1; l >= 0; l--) {
        const int w = q.ws[l], h = q.hs[l];
        const long long n = (long long)w * h;
        if (l == q.nl - 1) {
            if ((e = cudaMemsetAsync(cu, 0, n * 4, st)) != cudaSuccess) return e;
            if ((e = cudaMemsetAsync(cv, 0, n * 4, st)) != cudaSuccess) return e;
        } else {
            k_df_resample<<<df_blocks(n), 256, 0, st>>>(cu, q.ws[l + 1], q.hs[l + 1], nu, w, h, q.eta, 0, q.inv_eta);
            k_df_resample<<<df_blocks(n), 256, 0, st>>>(cv, q.ws[l + 1], q.hs[l + 1], nv, w, h, q.eta, 0, q.inv_eta);
            launches += 2;
            float* t = cu; cu = nu; nu = t;
            t = cv; cv = nv; nv = t;
        }
        // matches on this level
        if ((e = cudaMemsetAsync(ws + q.owner, 0, n * 8, st)) != cudaSuccess) return e;
        unsigned long long* owner = reinterpret_cast<unsigned long long*>(ws + q.owner);
        if (has_m) {
            k_df_raster<<<df_blocks(q.capacity), 256, 0, st>>>(m, d_count, q.capacity, w, h, q.sk[l], owner);
            launches++;
        }
        k_df_match_fields<<<df_blocks(n), 256, 0, st>>>(owner, m, F(q.phi), (int)n, q.beta_k[l], q.sk[l], F(q.mc), F(q.mu),
                                                         F(q.mv));
        // linearisation around the current flow (Im is free after the second step: its first word counts
        // the CTAs of the weights launches)
        unsigned int* published = reinterpret_cast<unsigned int*>(F(q.Im));
        k_df_prep1<<<df_blocks(n), 256, 0, st>>>(F(q.P1[l]), F(q.P2[l]), cu, cv, w, h, k, F(q.alpha), F(q.I2w), F(q.Im));
        k_df_prep2<<<df_blocks(n), 256, 0, st>>>(F(q.Im), w, h, F(q.Ix), F(q.Iy));
        k_df_prep3<<<df_blocks(n), 256, 0, st>>>(F(q.P1[l]), F(q.I2w), F(q.Ix), F(q.Iy), w, h, k, F(q.D),
                                                   published);
        launches += 4;
        if ((e = cudaMemsetAsync(F(q.du), 0, n * 4, st)) != cudaSuccess) return e;
        if ((e = cudaMemsetAsync(F(q.dv), 0, n * 4, st)) != cudaSuccess) return e;
        DfLevel L;
        L.w = w; L.h = h; L.n = n;
        L.D = F(q.D); L.alpha = F(q.alpha); L.mc = F(q.mc); L.mu = F(q.mu); L.mv = F(q.mv);
        L.u = cu; L.v = cv; L.du = F(q.du); L.dv = F(q.dv); L.A = F(q.A); L.ps = F(q.ps);
        if ((long long)((w + 1) / 2) * h <= DF_SMALL_PAIRS) {
            // one warp per 32 pairs: fewer warps meet at the barriers sooner
            const int threads = ((w + 1) / 2 * h + 31) / 32 * 32;
            k_df_level_small<<<1, threads, DF_SMALL_SMEM, st>>>(L, k, q.n_fixed, q.n_sor);
            launches++;
        } else {
            const unsigned tiles = (unsigned)(((w + TB_W - 1) / TB_W) * ((h + TB_H - 1) / TB_H));
            float* alt_u = F(q.du2);
            float* alt_v = F(q.dv2);
            for (int it = 0; it < q.n_fixed; it++) {
                k_df_weights<<<df_blocks(n), 256, 0, st>>>(L, k, published);
                launches++;
                for (int j = 0; j < 2 * q.n_sor; j += TB_S) {
                    const int S = 2 * q.n_sor - j < TB_S ? 2 * q.n_sor - j : TB_S;
                    const unsigned int count = j > 0 ? df_blocks(n) * (unsigned int)(it + 1) : 0u;
                    if ((e = dm_launch_pdl(k_df_sor_tb, tiles, TB_THREADS, TB_SMEM, st, L, k, S, published, count, alt_u, alt_v)) !=
                        cudaSuccess)
                        return e;
                    launches++;
                    float* t = L.du; L.du = alt_u; alt_u = t;
                    t = L.dv; L.dv = alt_v; alt_v = t;
                }
            }
            k_df_update<<<df_blocks(n), 256, 0, st>>>(cu, cv, L.du, L.dv, n);
            launches++;
        }
    }
    dm_count_launches(launches);
    if ((e = cudaMemcpyAsync(out_u, cu, (size_t)W * H * 4, cudaMemcpyDeviceToDevice, st)) != cudaSuccess) return e;
    if ((e = cudaMemcpyAsync(out_v, cv, (size_t)W * H * 4, cudaMemcpyDeviceToDevice, st)) != cudaSuccess) return e;
    return cudaGetLastError();
}

