// Pixel descriptors (Sec. 3.2 "Pixel descriptor").
//
// Pipeline per image: s = image_scale * I; Gaussian nu1 (horizontal pass,
// then vertical); central-difference gradient with replicated border;
// non-negative projections on the directions k*pi/4, k = 0..7; Gaussian nu2
// on each channel; sigmoid 2/(1+exp(-slope x)) - 1; Gaussian nu3; append mu
// and L2-normalise the 9-vector.  The operation order inside each output is fixed
// (an fma chain over taps j = -R..R from 0) so the FP32 result is reproducible bit
// for bit.  Smoothings of radius 3 (widths in (2/3, 1], the defaults) run the whole
// chain in one kernel on a tile in shared memory; other widths run one simple kernel
// per pass.
#include "dm_internal.cuh"

#include <algorithm>
#include <cstring>

namespace {

__device__ __forceinline__ int clampi(int v, int lo, int hi) { return v < lo ? lo : (v > hi ? hi : v); }

// Horizontal pass of one channel plane set.  in: [H][W][C] (C = 1 or 8);
// scale applied to the input value first when `scale_in` != 1 (first pass).
template <int C>
__device__ __forceinline__ void smooth_h(const float* __restrict__ in, float* __restrict__ out, int W, int H,
                                         const DmTaps& t, float scale_in, int apply_scale, long long idx) {
    long long n = (long long)W * H * C;
    if (idx >= n) return;
    int c = (int)(idx % C);
    long long pix = idx / C;
    int x = (int)(pix % W), y = (int)(pix / W);
    const float* row = in + (long long)y * W * C;
    float acc = 0.0f;
    for (int j = -t.R; j <= t.R; j++) {
        float v = row[(long long)clampi(x + j, 0, W - 1) * C + c];
        if (apply_scale) v = __fmul_rn(v, scale_in);
        acc = __fmaf_rn(t.w[j + t.R], v, acc);
    }
    out[idx] = acc;
}

// Vertical pass; post = 0 none, 1 sigmoid, 2 normalise into [H][W][9] output.
template <int C, int POST>
__device__ __forceinline__ void smooth_v(const float* __restrict__ in, float* __restrict__ out, int W, int H,
                                         const DmTaps& t, float slope, float mu, long long gidx) {
    if (POST == 2) {
        // one thread per pixel: smooth its C channels, then normalise
        long long pix = gidx;
        if (pix >= (long long)W * H) return;
        int x = (int)(pix % W), y = (int)(pix / W);
        float v[C];
#pragma unroll
        for (int c = 0; c < C; c++) {
            float acc = 0.0f;
            for (int j = -t.R; j <= t.R; j++)
                acc = __fmaf_rn(t.w[j + t.R], in[((long long)clampi(y + j, 0, H - 1) * W + x) * C + c], acc);
            v[c] = acc;
        }
        float acc = 0.0f;
#pragma unroll
        for (int c = 0; c < C; c++) acc = __fmaf_rn(v[c], v[c], acc);
        acc = __fmaf_rn(mu, mu, acc);
        float nrm = __fsqrt_rn(acc);
        float* o = out + pix * 9;
#pragma unroll
        for (int c = 0; c < C; c++) o[c] = __fdiv_rn(v[c], nrm);
        o[8] = __fdiv_rn(mu, nrm);
        return;
    }
    const long long idx = gidx;
    long long n = (long long)W * H * C;
    if (idx >= n) return;
    int c = (int)(idx % C);
    long long pix = idx / C;
    int x = (int)(pix % W), y = (int)(pix / W);
    float acc = 0.0f;
    for (int j = -t.R; j <= t.R; j++)
        acc = __fmaf_rn(t.w[j + t.R], in[((long long)clampi(y + j, 0, H - 1) * W + x) * C + c], acc);
    if (POST == 1) {
        float tt = __fmul_rn(slope, acc);
        float e = dm_expf(-tt);
        float d = __fadd_rn(1.0f, e);
        acc = __fsub_rn(__fdiv_rn(2.0f, d), 1.0f);
    }
    out[idx] = acc;
}

// Elementwise sigmoid (used when nu2 = 0, i.e. no vertical pass to fuse into).
__global__ void k_sigmoid(float* __restrict__ buf, long long n, float slope) {
    long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= n) return;
    float tt = __fmul_rn(slope, buf[idx]);
    float e = dm_expf(-tt);
    float d = __fadd_rn(1.0f, e);
    buf[idx] = __fsub_rn(__fdiv_rn(2.0f, d), 1.0f);
}

// Scale without smoothing (nu1 = 0).
__global__ void k_scale(const float* __restrict__ in, float* __restrict__ out, long long n, float s) {
    long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx < n) out[idx] = __fmul_rn(in[idx], s);
}

// Gradient + 8 non-negative projections.  dir_k = (cos k pi/4, sin k pi/4)
// with the exact table {1, r, 0, -r, -1, -r, 0, r} / {0, r, 1, r, 0, -r, -1, -r},
// r = sqrt(1/2) rounded to float; v_k = fma(gx, cos_k, gy * sin_k), then max(v, 0).
__device__ __forceinline__ void project8(float gx, float gy, float* o) {
    const float r = 0.70710678118654752f;
    const float dc[8] = {1.0f, r, 0.0f, -r, -1.0f, -r, 0.0f, r};
    const float ds[8] = {0.0f, r, 1.0f, r, 0.0f, -r, -1.0f, -r};
#pragma unroll
    for (int k = 0; k < 8; k++) {
        float v = __fmaf_rn(gx, dc[k], __fmul_rn(gy, ds[k]));
        o[k] = v > 0.0f ? v : 0.0f;
    }
}

__device__ __forceinline__ void grad_proj(const float* __restrict__ s, float* __restrict__ o8, int W, int H, long long pix) {
    if (pix >= (long long)W * H) return;
    int x = (int)(pix % W), y = (int)(pix / W);
    float gx = __fmul_rn(__fsub_rn(s[(long long)y * W + clampi(x + 1, 0, W - 1)], s[(long long)y * W + clampi(x - 1, 0, W - 1)]), 0.5f);
    float gy = __fmul_rn(__fsub_rn(s[(long long)clampi(y + 1, 0, H - 1) * W + x], s[(long long)clampi(y - 1, 0, H - 1) * W + x]), 0.5f);
    project8(gx, gy, o8 + pix * 8);
}

__device__ __forceinline__ long long gtid() { return (long long)blockIdx.x * blockDim.x + threadIdx.x; }

template <int C>
__global__ void k_smooth_h(const float* __restrict__ in, float* __restrict__ out, int W, int H, DmTaps t, float scale_in,
                           int apply_scale) {
    smooth_h<C>(in, out, W, H, t, scale_in, apply_scale, gtid());
}
template <int C, int POST>
__global__ void k_smooth_v(const float* __restrict__ in, float* __restrict__ out, int W, int H, DmTaps t, float slope,
                           float mu) {
    smooth_v<C, POST>(in, out, W, H, t, slope, mu, gtid());
}
__global__ void k_grad_proj(const float* __restrict__ s, float* __restrict__ o8, int W, int H) { grad_proj(s, o8, W, H, gtid()); }

// Cross-pair form: the same passes for every image of a wave of the batched
// form in one launch each, image blockIdx.y (its buffers in the parameters).
struct IoBatch {
    const float* in[2 * DM_BATCH_MAX];
    float* out[2 * DM_BATCH_MAX];
    int W[2 * DM_BATCH_MAX], H[2 * DM_BATCH_MAX];
    int n;
};
template <int C>
__global__ void k_smooth_h_b(const __grid_constant__ IoBatch B, DmTaps t, float scale_in, int apply_scale) {
    const int i = blockIdx.y;
    smooth_h<C>(B.in[i], B.out[i], B.W[i], B.H[i], t, scale_in, apply_scale, gtid());
}
template <int C, int POST>
__global__ void k_smooth_v_b(const __grid_constant__ IoBatch B, DmTaps t, float slope, float mu) {
    const int i = blockIdx.y;
    smooth_v<C, POST>(B.in[i], B.out[i], B.W[i], B.H[i], t, slope, mu, gtid());
}
__global__ void k_grad_proj_b(const __grid_constant__ IoBatch B) {
    const int i = blockIdx.y;
    grad_proj(B.in[i], B.out[i], B.W[i], B.H[i], gtid());
}

// The whole chain for a TX x TY tile of one image, every smoothing of radius R.  Each
// pass forms its result on the tile and the border that the passes after it read, in
// shared memory.  A position outside the image holds the value of the nearest one
// inside, so that the replicated border costs one clamp per output instead of one per
// tap.  Channels go in fours (one 16-byte load per tap, two packed fmas); the vertical
// passes form two rows per thread from eight loads.
//
// What bounds it: shared-memory loads (56 % of the pipe) and instruction issue (58 %), on
// a 32x16 tile 1.6 times the tile's own work for the borders; before, each of the seven
// passes went through memory with one scalar load and index arithmetic per tap.  Both
// images: 1024x436 311 -> 86 us, 512x224 115 -> 40, 64x48 63 -> 23.
constexpr int FR = 3;                                // the radius
struct Taps7 {
    float w[2 * FR + 1];
};

template <int TX, int TY>
struct DescTile {
    static constexpr int IW = TX + 6 * FR + 2, IH = TY + 6 * FR + 2;     // image
    static constexpr int SW = TX + 4 * FR + 2, SH = TY + 4 * FR + 2;     // smoothed image (h: IH rows)
    static constexpr int GW = TX + 4 * FR, GH = TY + 4 * FR;             // projections
    static constexpr int PW = TX + 2 * FR, PH = TY + 2 * FR;             // after the sigmoid (h: GH rows)
    static constexpr int A = GW * GH * 8, B = PW * GH * 8;               // floats of the two buffers
    static_assert(IW * IH + SW * IH + SW * SH <= B && TX * PH * 8 <= B && PW * PH * 8 <= A && TX * TY * 9 <= A, "buffers");
    static constexpr size_t SMEM = (size_t)(A + B) * sizeof(float);
};

__device__ __forceinline__ float4 fma4(float w, float4 v, float4 a) {
    const float2 ww = make_float2(w, w);
    const float2 lo = __ffma2_rn(ww, make_float2(v.x, v.y), make_float2(a.x, a.y));
    const float2 hi = __ffma2_rn(ww, make_float2(v.z, v.w), make_float2(a.z, a.w));
    return make_float4(lo.x, lo.y, hi.x, hi.y);
}

__device__ __forceinline__ float sigmoid1(float v, float slope) {
    const float e = dm_expf(-__fmul_rn(slope, v));
    return __fsub_rn(__fdiv_rn(2.0f, __fadd_rn(1.0f, e)), 1.0f);
}

// Horizontal pass of eight channels: OW x OH outputs at (ox, oy), inputs of IW columns at (ox - FR, oy).
template <int OW, int OH>
__device__ __forceinline__ void tile_h(const float* in, float* out, int ox, int oy, int W, int H, const Taps7& t) {
    constexpr int IW = OW + 2 * FR;
    for (int i = threadIdx.x; i < OW * OH * 2; i += blockDim.x) {
        const int half = i & 1, x = (i >> 1) % OW, y = (i >> 1) / OW;
        const int xi = clampi(ox + x, 0, W - 1) - ox, yi = clampi(oy + y, 0, H - 1) - oy;
        const float4* p = reinterpret_cast<const float4*>(in) + (yi * IW + xi) * 2 + half;
        float4 acc = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
        for (int j = 0; j <= 2 * FR; j++) acc = fma4(t.w[j], p[2 * j], acc);
        reinterpret_cast<float4*>(out)[i] = acc;
    }
}

// Vertical pass, two rows (y, y + 1) of four channels: inputs of IW columns at (.., oy - FR).
template <int IW>
__device__ __forceinline__ void tile_v2(const float* in, int x, int y, int half, int oy, int H, const Taps7& t, float4& r0,
                                        float4& r1) {
    const int y0 = clampi(oy + y, 0, H - 1) - oy, y1 = clampi(oy + y + 1, 0, H - 1) - oy;
    const float4* p = reinterpret_cast<const float4*>(in) + (y0 * IW + x) * 2 + half;
    float4 v[2 * FR + 2];
#pragma unroll
    for (int j = 0; j < 2 * FR + 2; j++) v[j] = p[2 * IW * j];
    r0 = r1 = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
    for (int j = 0; j <= 2 * FR; j++) {
        r0 = fma4(t.w[j], v[j], r0);
        r1 = fma4(t.w[j], v[j + 1], r1);
    }
    if (y1 == y0) r1 = r0;                           // (both beyond the image's edge, or on it)
}

template <int TX, int TY>
__device__ __forceinline__ void desc_tile(const float* __restrict__ img, float* __restrict__ desc, int W, int H, int tile,
                                          const Taps7& t1, const Taps7& t2, const Taps7& t3, float scale, float slope,
                                          float mu) {
    using T = DescTile<TX, TY>;
    extern __shared__ __align__(16) float dsm[];
    float* A = dsm;
    float* B = dsm + T::A;
    const int tx = (W + TX - 1) / TX;
    const int x0 = (tile % tx) * TX, y0 = (tile / tx) * TY;
    if (y0 >= H) return;                             // (the same for the whole block)
    const int tid = threadIdx.x, nt = blockDim.x;

    // s = scale * I, smoothed by t1
    float* im = B;
    float* h1 = im + T::IW * T::IH;
    float* sm = h1 + T::SW * T::IH;
    for (int i = tid; i < T::IW * T::IH; i += nt) {
        const int x = clampi(x0 - 3 * FR - 1 + i % T::IW, 0, W - 1), y = clampi(y0 - 3 * FR - 1 + i / T::IW, 0, H - 1);
        im[i] = __fmul_rn(__ldg(img + (long long)y * W + x), scale);
    }
    __syncthreads();
    {
        const int ox = x0 - 2 * FR - 1, oy = y0 - 3 * FR - 1;
        for (int i = tid; i < T::SW * T::IH; i += nt) {
            const int xi = clampi(ox + i % T::SW, 0, W - 1) - ox, yi = clampi(oy + i / T::SW, 0, H - 1) - oy;
            float acc = 0.0f;
#pragma unroll
            for (int j = 0; j <= 2 * FR; j++) acc = __fmaf_rn(t1.w[j], im[yi * T::IW + xi + j], acc);
            h1[i] = acc;
        }
    }
    __syncthreads();
    {
        const int oy = y0 - 2 * FR - 1;
        for (int i = tid; i < T::SW * T::SH; i += nt) {
            const int x = i % T::SW, yi = clampi(oy + i / T::SW, 0, H - 1) - oy;
            float acc = 0.0f;
#pragma unroll
            for (int j = 0; j <= 2 * FR; j++) acc = __fmaf_rn(t1.w[j], h1[(yi + j) * T::SW + x], acc);
            sm[i] = acc;
        }
    }
    __syncthreads();
    // gradient projections -> A
    for (int i = tid; i < T::GW * T::GH; i += nt) {
        const int ox = x0 - 2 * FR, oy = y0 - 2 * FR;
        const int xi = clampi(ox + i % T::GW, 0, W - 1) - ox + 1, yi = clampi(oy + i / T::GW, 0, H - 1) - oy + 1;
        const float* c = sm + yi * T::SW + xi;
        const float gx = __fmul_rn(__fsub_rn(c[1], c[-1]), 0.5f), gy = __fmul_rn(__fsub_rn(c[T::SW], c[-T::SW]), 0.5f);
        float o[8];
        project8(gx, gy, o);
        reinterpret_cast<float4*>(A)[2 * i] = make_float4(o[0], o[1], o[2], o[3]);
        reinterpret_cast<float4*>(A)[2 * i + 1] = make_float4(o[4], o[5], o[6], o[7]);
    }
    __syncthreads();
    // t2 and the sigmoid -> A
    tile_h<T::PW, T::GH>(A, B, x0 - FR, y0 - 2 * FR, W, H, t2);
    __syncthreads();
    for (int i = tid; i < T::PW * T::PH; i += nt) {          // two rows x two halves
        const int half = i & 1, x = (i >> 1) % T::PW, y = (i >> 1) / T::PW * 2;
        float4 r[2];
        tile_v2<T::PW>(B, x, y, half, y0 - FR, H, t2, r[0], r[1]);
#pragma unroll
        for (int k = 0; k < 2; k++)
            reinterpret_cast<float4*>(A)[((y + k) * T::PW + x) * 2 + half] =
                make_float4(sigmoid1(r[k].x, slope), sigmoid1(r[k].y, slope), sigmoid1(r[k].z, slope), sigmoid1(r[k].w, slope));
    }
    __syncthreads();
    // t3 and the normalisation -> A as [TY][TX][9]
    tile_h<TX, T::PH>(A, B, x0, y0 - FR, W, H, t3);
    __syncthreads();
    static_assert(TX * TY % 32 == 0, "whole warps below");
    for (int i = tid; i < TX * TY; i += nt) {
        const int half = i & 1, x = (i >> 1) % TX, y = (i >> 1) / TX * 2;
        float4 r[2];
        tile_v2<TX>(B, x, y, half, y0, H, t3, r[0], r[1]);
#pragma unroll
        for (int k = 0; k < 2; k++) {
            // the sum of squares runs over the channels in order: the first half's lane, then the second's
            auto squares = [&](float a) {
                a = __fmaf_rn(r[k].x, r[k].x, a);
                a = __fmaf_rn(r[k].y, r[k].y, a);
                a = __fmaf_rn(r[k].z, r[k].z, a);
                return __fmaf_rn(r[k].w, r[k].w, a);
            };
            const float first = __shfl_xor_sync(0xffffffffu, squares(0.0f), 1);
            float nrm = __fsqrt_rn(__fmaf_rn(mu, mu, squares(first)));   // (the second half's)
            const float other = __shfl_xor_sync(0xffffffffu, nrm, 1);
            if (half == 0) nrm = other;
            float* o = A + ((y + k) * TX + x) * 9 + 4 * half;
            o[0] = __fdiv_rn(r[k].x, nrm);
            o[1] = __fdiv_rn(r[k].y, nrm);
            o[2] = __fdiv_rn(r[k].z, nrm);
            o[3] = __fdiv_rn(r[k].w, nrm);
            if (half) o[4] = __fdiv_rn(mu, nrm);
        }
    }
    __syncthreads();
    const int cols = min(TX, W - x0) * 9, rows = min(TY, H - y0);
    for (int i = tid; i < TX * TY * 9; i += nt) {
        const int c = i % (TX * 9), y = i / (TX * 9);
        if (c < cols && y < rows) desc[((long long)(y0 + y) * W + x0) * 9 + c] = A[i];
    }
}

constexpr int DESC_THREADS = 256;

template <int TX, int TY>
__global__ void __launch_bounds__(DESC_THREADS) k_descriptors(const float* __restrict__ img, float* __restrict__ desc, int W,
                                                              int H, Taps7 t1, Taps7 t2, Taps7 t3, float scale, float slope,
                                                              float mu) {
    dm_pdl_wait();
    desc_tile<TX, TY>(img, desc, W, H, blockIdx.x, t1, t2, t3, scale, slope, mu);
}

template <int TX, int TY>
__global__ void __launch_bounds__(DESC_THREADS) k_descriptors_b(const __grid_constant__ IoBatch B, Taps7 t1, Taps7 t2,
                                                                Taps7 t3, float scale, float slope, float mu) {
    const int i = blockIdx.y;
    desc_tile<TX, TY>(B.in[i], B.out[i], B.W[i], B.H[i], blockIdx.x, t1, t2, t3, scale, slope, mu);
}

bool fused_taps(const DmDescParams& prm, Taps7 t[3]) {
    const DmTaps* src[3] = {&prm.t1, &prm.t2, &prm.t3};
    for (int i = 0; i < 3; i++) {
        if (src[i]->R != FR) return false;
        for (int j = 0; j <= 2 * FR; j++) t[i].w[j] = src[i]->w[j];
    }
    return true;
}

template <int TX, int TY>
cudaError_t launch_fused(const DmDescParams& prm, const Taps7 t[3], const IoBatch& b, cudaStream_t st) {
    static std::atomic<unsigned long long> done{0}, done_b{0};      // > 48 KB dynamic shared memory opted in, per device
    const int smem = (int)DescTile<TX, TY>::SMEM;
    cudaError_t e;
    unsigned tiles = 0;
    for (int i = 0; i < b.n; i++) tiles = std::max(tiles, (unsigned)((b.W[i] + TX - 1) / TX) * (unsigned)((b.H[i] + TY - 1) / TY));
    if (b.n == 1) {
        if ((e = dm_smem_opt_in(reinterpret_cast<const void*>(k_descriptors<TX, TY>), smem, done)) != cudaSuccess) return e;
        e = dm_launch_pdl(k_descriptors<TX, TY>, tiles, DESC_THREADS, smem, st, b.in[0], b.out[0], b.W[0], b.H[0], t[0], t[1], t[2],
                          prm.scale, prm.slope, prm.mu);
        if (e != cudaSuccess) return e;
    } else {
        if ((e = dm_smem_opt_in(reinterpret_cast<const void*>(k_descriptors_b<TX, TY>), smem, done_b)) != cudaSuccess) return e;
        k_descriptors_b<TX, TY><<<dim3(tiles, (unsigned)b.n), DESC_THREADS, smem, st>>>(b, t[0], t[1], t[2], prm.scale,
                                                                                       prm.slope, prm.mu);
    }
    dm_count_launches(1);
    return cudaGetLastError();
}

// Tiles of 32x16 do the least work twice; images of few such tiles take tiles of a
// quarter of that, which spread over more SMs and are each done sooner.
cudaError_t launch_fused(const DmDescParams& prm, const Taps7 t[3], const IoBatch& b, cudaStream_t st) {
    long long px = 0;
    for (int i = 0; i < b.n; i++) px += (long long)b.W[i] * b.H[i];
    if (px >= 32LL * 16 * dm_sm_count()) return launch_fused<32, 16>(prm, t, b, st);
    return launch_fused<16, 8>(prm, t, b, st);
}

inline unsigned nblk(long long n, int b) { return (unsigned)((n + b - 1) / b); }

}  // namespace

// tmpA, tmpB: [H][W][8] float each.
cudaError_t dm_launch_descriptors(const DmDescParams& prm, const float* img, int W, int H, float* desc,
                                  float* tmpA, float* tmpB, cudaStream_t st) {
    Taps7 t[3];
    if (fused_taps(prm, t)) {
        IoBatch one;
        one.in[0] = img, one.out[0] = desc, one.W[0] = W, one.H[0] = H, one.n = 1;
        return launch_fused(prm, t, one, st);
    }
    const int B = 256;
    long long n1 = (long long)W * H, n8 = n1 * 8;
    // s = scale * I, smoothed by nu1 -> tmpB (1 channel)
    if (prm.t1.R > 0) {
        k_smooth_h<1><<<nblk(n1, B), B, 0, st>>>(img, tmpA, W, H, prm.t1, prm.scale, 1);
        k_smooth_v<1, 0><<<nblk(n1, B), B, 0, st>>>(tmpA, tmpB, W, H, prm.t1, 0.f, 0.f);
    } else {
        k_scale<<<nblk(n1, B), B, 0, st>>>(img, tmpB, n1, prm.scale);
    }
    // gradient projections -> tmpA [H][W][8]
    k_grad_proj<<<nblk(n1, B), B, 0, st>>>(tmpB, tmpA, W, H);
    // nu2 smoothing + sigmoid -> tmpA
    if (prm.t2.R > 0) {
        k_smooth_h<8><<<nblk(n8, B), B, 0, st>>>(tmpA, tmpB, W, H, prm.t2, 1.f, 0);
        k_smooth_v<8, 1><<<nblk(n8, B), B, 0, st>>>(tmpB, tmpA, W, H, prm.t2, prm.slope, 0.f);
    } else {
        k_sigmoid<<<nblk(n8, B), B, 0, st>>>(tmpA, n8, prm.slope);
    }
    // nu3 smoothing + normalisation -> desc [H][W][9]
    const float* src = tmpA;
    if (prm.t3.R > 0) {
        k_smooth_h<8><<<nblk(n8, B), B, 0, st>>>(tmpA, tmpB, W, H, prm.t3, 1.f, 0);
        src = tmpB;
    }
    DmTaps id;
    id.R = 0;
    id.w[0] = 1.0f;
    k_smooth_v<8, 2><<<nblk(n1, B), B, 0, st>>>(src, desc, W, H, prm.t3.R > 0 ? prm.t3 : id, 0.f, prm.mu);
    dm_count_launches((prm.t1.R > 0 ? 2 : 1) + 1 + (prm.t2.R > 0 ? 2 : 1) + (prm.t3.R > 0 ? 1 : 0) + 1);
    return cudaGetLastError();
}

// One image scaled by `scale` and smoothed by taps t (horizontal pass, then
// vertical), as the first step of the descriptors; R = 0: scaled only.
cudaError_t dm_launch_smooth1(const float* img, int W, int H, float scale, const DmTaps& t, float* out, float* tmp,
                              cudaStream_t st) {
    const int B = 256;
    const long long n1 = (long long)W * H;
    if (t.R > 0) {
        k_smooth_h<1><<<nblk(n1, B), B, 0, st>>>(img, tmp, W, H, t, scale, 1);
        k_smooth_v<1, 0><<<nblk(n1, B), B, 0, st>>>(tmp, out, W, H, t, 0.f, 0.f);
        dm_count_launches(2);
    } else {
        k_scale<<<nblk(n1, B), B, 0, st>>>(img, out, n1, scale);
        dm_count_launches(1);
    }
    return cudaGetLastError();
}

// Descriptors of n <= 2 DM_BATCH_MAX images (a wave of the batched form): one
// launch (or one per pass) for all of them.  (With a zero smoothing width the scaling
// and sigmoid passes run image by image.)
cudaError_t dm_launch_descriptors_batch(const DmDescParams& prm, int n, const float* const* imgs, const int* Ws,
                                        const int* Hs, float* const* descs, float* const* tmpAs, float* const* tmpBs,
                                        cudaStream_t st) {
    if (n < 1 || n > 2 * DM_BATCH_MAX) return cudaErrorInvalidValue;
    if (prm.t1.R == 0 || prm.t2.R == 0 || prm.t3.R == 0) {
        for (int i = 0; i < n; i++) {
            cudaError_t e = dm_launch_descriptors(prm, imgs[i], Ws[i], Hs[i], descs[i], tmpAs[i], tmpBs[i], st);
            if (e != cudaSuccess) return e;
        }
        return cudaSuccess;
    }
    Taps7 t[3];
    if (fused_taps(prm, t)) {
        IoBatch b;
        memset(&b, 0, sizeof(b));
        b.n = n;
        for (int i = 0; i < n; i++) b.in[i] = imgs[i], b.out[i] = descs[i], b.W[i] = Ws[i], b.H[i] = Hs[i];
        return launch_fused(prm, t, b, st);
    }
    const int B = 256;
    long long n1 = 0;
    for (int i = 0; i < n; i++) n1 = std::max(n1, (long long)Ws[i] * Hs[i]);
    const long long n8 = 8 * n1;
    auto io = [&](int step) {
        IoBatch b;
        memset(&b, 0, sizeof(b));
        b.n = n;
        for (int i = 0; i < n; i++) {
            b.W[i] = Ws[i];
            b.H[i] = Hs[i];
            switch (step) {
                case 0: b.in[i] = imgs[i]; b.out[i] = tmpAs[i]; break;     // nu1, horizontal
                case 1: b.in[i] = tmpAs[i]; b.out[i] = tmpBs[i]; break;    // nu1, vertical
                case 2: b.in[i] = tmpBs[i]; b.out[i] = tmpAs[i]; break;    // gradient projections
                case 3: b.in[i] = tmpAs[i]; b.out[i] = tmpBs[i]; break;    // nu2, horizontal
                case 4: b.in[i] = tmpBs[i]; b.out[i] = tmpAs[i]; break;    // nu2, vertical + sigmoid
                case 5: b.in[i] = tmpAs[i]; b.out[i] = tmpBs[i]; break;    // nu3, horizontal
                default: b.in[i] = tmpBs[i]; b.out[i] = descs[i]; break;   // nu3, vertical + normalisation
            }
        }
        return b;
    };
    const dim3 g1(nblk(n1, B), (unsigned)n), g8(nblk(n8, B), (unsigned)n);
    k_smooth_h_b<1><<<g1, B, 0, st>>>(io(0), prm.t1, prm.scale, 1);
    k_smooth_v_b<1, 0><<<g1, B, 0, st>>>(io(1), prm.t1, 0.f, 0.f);
    k_grad_proj_b<<<g1, B, 0, st>>>(io(2));
    k_smooth_h_b<8><<<g8, B, 0, st>>>(io(3), prm.t2, 1.f, 0);
    k_smooth_v_b<8, 1><<<g8, B, 0, st>>>(io(4), prm.t2, prm.slope, 0.f);
    k_smooth_h_b<8><<<g8, B, 0, st>>>(io(5), prm.t3, 1.f, 0);
    k_smooth_v_b<8, 2><<<g1, B, 0, st>>>(io(6), prm.t3, 0.f, prm.mu);
    dm_count_launches(7);
    return cudaGetLastError();
}
