// Bottom-level correlation (Eq. 3-4) on the FP32 SIMT pipes, with the first
// max-pooling + subsampling (Eq. 8-9) and rectification (Eq. 11) fused into
// the epilogue.  The unpooled level-0 volume (P0 x W2 x H2 values) is never
// written to memory: only P_0(p, r) = (max_{m} C0(p, 2r+m))^lambda and its
// argmax code.
//
// Tiling.  A CTA owns 32 atomic patches (8 warps x 4) and a band of 8 pooled rows,
// and walks along it in tiles of 32 pooled columns, i.e. C0 at 17 rows x 64 columns.
// Lane j of a warp owns the C0 columns 2j and 2j + 1 of the tile for its warp's 4
// patches and all 17 rows: 136 accumulators, held as 68 float2 pairs of neighbouring
// columns, so that one packed FP32x2 fma (__ffma2_rn) updates two columns.  The image-2
// descriptors of the tile are staged channel by channel, so that a pair of
// neighbouring columns is one 8-byte load, free of bank conflicts; a second copy,
// shifted by one column, serves the odd offsets dx.  The patch vectors are staged with
// every value twice.  So the main loop is packed fmas and loads alone: per (dx,
// channel) 20 + 8 loads for 272 fmas, no moves to pair operands.  The next tile is
// staged into a second buffer meanwhile (asynchronous 4-byte copies, zero-filled
// outside the images: a pixel's nine floats allow no wider ones).
//
// The bands of a patch group lie side by side in one row of tiles, so that a map's last
// columns and the next band's first ones share a tile: one empty lane after each band, whose
// pixels are zeros, is border enough for both (a position needs two pixels to the left and one
// to the right).  Where the columns fill whole tiles, or on small inputs where that makes no
// SM's tiles fewer, a band takes whole tiles instead.  With whole tiles for every width up to
// 62 % of the lanes were idle.  dm_correlate_pyramid, whole tiles / so / tiles of 15 columns with
// one lane per column: 256x256 against 24x200 (map of 12 columns) 521 / 353 / 445 us, 200x200 1091
// / 903 / 1058, 512x224 5701 / 5714 / 7085.
//
// Work of a CTA: an equal range of the tiles in the order (patch group, band, column),
// about one CTA per SM and at most RANGE tiles each, so that the last wave is a full
// one (13.5 waves of whole bands took 14).  Small inputs have fewer tiles than SMs: they
// take lower bands and 2 patches per warp (two CTAs per SM, one buffer), by the cost
// rule at the launch.
//
// What bounds it: the FMA pipe and the operand reads of the packed fmas (the main loop
// alone runs at 77 % of the pipe's rate).  Measured (start: one lane per column, patch
// pairs packed, operands paired by moves, 13 % overlapping tiles, 46 % of the FMA peak):
// 512x224 6.43 -> 5.20 ms (49 % of the peak in useful fmas), 256x256 2.11 -> 1.74,
// 64x48 25.7 -> 15.2 us.  Two CTAs of 2 patches per warp throughout: 5.43 ms (all nine
// channels unrolled); 4 patches without the second buffer: 5.45; main loop by dy
// instead of by staged row: 5.87; 3 channels unrolled: 5.58.
//
// Summation order (identical to the FP32 reference): per output,
// acc = fma(a, b, acc) over dx = 0..3, then channel c = 0..8, then dy = 0..3,
// starting from 0, then acc * (1/16).  Terms outside either image are zero
// and leave acc unchanged (all operands are non-negative).  The loop order
// (dx, c) outer / dy inner lets a staged column pair feed all 4 dy offsets: staged row
// hr goes to the output rows hr - dy.
//
// Epilogue, in registers: x1/16, out-of-domain positions masked to -inf, 3x3/2
// max-pool with the first strict maximum in scan order (row-major in the window),
// i.e. (no NaN occurs) the smallest scan index among the positions equal to the
// maximum.  A lane reduces each of its two columns over the three rows of every
// pooled row (maximum and the first row reaching it), then pools column j: the left
// column of its window is the second column of lane j - 1, and for lane 0 the last
// column of the tile before, which the warp keeps (so tiles do not overlap).  Then the
// power of two rows' maxima at once and coalesced stores of 32 columns.
#include "dm_internal.cuh"

namespace {

constexpr int WARPS = 8;                      // of a CTA, NP patches each
constexpr int PWT = 32;                       // pooled columns per tile
constexpr int HCOLS = 2 * PWT + 3;            // pixels 64 t - 2 .. 64 t + 64
constexpr int HPITCH = 66;                    // columns of a staged row (either copy)
constexpr int LEFT = 12;                      // a patch's column kept for the next tile: 8 maxima, their rows, padding
constexpr int RANGE = 32;                     // tiles of a CTA, at most

// A band of PH pooled rows, NP patches per warp.
template <int PH, int NP>
struct Band {
    static constexpr int PATCHES = WARPS * NP;
    static constexpr int CTAS_SM = NP == 2 ? 2 : 1, BUFS = NP == 2 ? 1 : 2;
    static constexpr int CROWS = 2 * PH + 1, HROWS = CROWS + 3;
    // floats of a channel's plane: even, and a multiple of the banks plus 10, so that the
    // nine channels of a pixel, which the staging writes together, fall in distinct banks
    static constexpr int PLANE = (HROWS * HPITCH - 10 + 31) / 32 * 32 + 10;
    static constexpr int COPY = 9 * PLANE;
    static constexpr size_t SMEM_BYTES =
        (size_t)(BUFS * 2 * COPY + 144 * PATCHES * 2 + WARPS * NP * LEFT + 9 * HROWS) * 4;
    static_assert(SMEM_BYTES <= 227 * 1024 && (SMEM_BYTES + 1024) * CTAS_SM <= 228 * 1024, "shared memory");
};

// 4-byte asynchronous global -> shared copy; n = 0 writes a zero and reads nothing.
__device__ __forceinline__ void cp_async4(float* dst, const float* src, int n) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;"
                 :: "r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "r"(n) : "memory");
}

__device__ __forceinline__ float fmax3(float a, float b, float c) {
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// Tiles of a patch group's row of bands, `bl` lanes each.
__host__ __device__ inline int band_tiles(int bands, int bl) { return (bands * bl + PWT - 1) / PWT; }

// The maximum of a column over the three rows of a pooled row, and 3 x the first row
// reaching it, shifted by sh.
__device__ __forceinline__ float col_max(float v0, float v1, float v2, int sh, uint32_t& y3) {
    const float m = fmax3(v0, v1, v2);
    y3 = v0 == m ? 0u : (v1 == m ? 3u << sh : 6u << sh);
    return m;
}

template <int PH, int NP>
__global__ void __launch_bounds__(256, Band<PH, NP>::CTAS_SM)
k_corr0_f32(DmGeom g, const float* __restrict__ d1, const float* __restrict__ d2, float lam,
            float* __restrict__ pooled0, unsigned char* __restrict__ amax0, const float* __restrict__ amat, int n0,
            long long units, int bl) {
    using B = Band<PH, NP>;
    constexpr int CROWS = B::CROWS, HROWS = B::HROWS, PLANE = B::PLANE, COPY = B::COPY, PATCHES = B::PATCHES;
    extern __shared__ __align__(16) float sm[];
    // a buffer: even [9][HROWS][HPITCH], the pixels of lane j at columns 2 j + 2 and 2 j + 3, two more before
    // and one after them, and odd, the same shifted by one
    float2* a_s = reinterpret_cast<float2*>(sm + B::BUFS * 2 * COPY);    // [(dx*9+c)*4+dy][patch], value twice
    float* left_s = sm + B::BUFS * 2 * COPY + 144 * PATCHES * 2;         // [warp][patch][LEFT]
    float* edge = left_s + WARPS * NP * LEFT;                            // [9][HROWS]: the pixel before those of the first tile

    const int W2 = g.W2, H2 = g.H2, mw = g.dw[1], mh = g.dh[1], pitch = g.pitch(1);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int bands = (mh + PH - 1) / PH, tiles = band_tiles(bands, bl);
    const long long u0 = units * blockIdx.x / gridDim.x;
    int todo = (int)(units * (blockIdx.x + 1) / gridDim.x - u0);
    int t = (int)(u0 % tiles), p_base = (int)(u0 / tiles) * PATCHES;
    int b0 = PWT * t / bl, c0 = PWT * t - b0 * bl;       // lane 0's band and its pooled column
    // stage the patch vectors; form the column before the first tile, where that begins inside a band
    bool load = true, edged = c0 > 0 && c0 < mw;
    const DmPow pr = dm_pow_setup(lam);
    dm_pdl_wait();

    // band and pooled column of a lane past the end of band b
    auto wrap = [&](int& b, int& c) {
        while (c >= bl) {
            c -= bl;
            b++;
        }
    };

    // image-2 descriptors of a tile, zero outside I': the pixels of lane j and one row of them per
    // staged row of its band (a band's first row is 3 above its C0 rows' centres)
    auto stage = [&](int b0, int c0, float* even) {
        const int y00 = 2 * PH * b0 - 3;
        // a tile inside a band and inside I': a row of it is 603 consecutive floats
        const bool full = c0 > 0 && 2 * (c0 + PWT) + 1 <= W2 && y00 >= 0 && y00 + HROWS <= H2;
        for (int q = tid; q < HCOLS * 9; q += 256) {
            const int col = q / 9, c = q - 9 * col;
            float* e = even + c * PLANE + col;
            float* o = even + COPY + c * PLANE + col - 1;
            if (full && col >= 1 && col < HPITCH) {
                const float* src = d2 + (long long)y00 * W2 * 9 + (2 * c0 - 2) * 9 + q;
#pragma unroll
                for (int r = 0; r < HROWS; r++) {
                    cp_async4(e + r * HPITCH, src, 4);
                    cp_async4(o + r * HPITCH, src, 4);
                    src += W2 * 9;
                }
                continue;
            }
            const int j = min(max((col - 2) >> 1, 0), PWT - 1);
            int b = b0, cj = c0 + j;
            wrap(b, cj);
            const int x = 2 * (cj - j) + col - 2, y0 = 2 * PH * b - 3;
            const float* src = d2 + ((long long)y0 * W2 + x) * 9 + c;
            const bool in = x >= 0 && x < W2;
#pragma unroll 4
            for (int r = 0; r < HROWS; r++) {
                const int y = y0 + r;
                const int n = in && y >= 0 && y < H2 ? 4 : 0;
                const float* s = n ? src : d2;
                if (col < HPITCH) cp_async4(e + r * HPITCH, s, n);
                if (col >= 1) cp_async4(o + r * HPITCH, s, n);
                src += W2 * 9;
            }
        }
    };

    float* left = left_s + warp * NP * LEFT;             // this warp's: the last column of the tile before
    float* even = sm;                                    // the tile's buffer
    if (B::BUFS == 2) stage(b0, c0, even);

    for (; todo > 0; todo--) {
        const int cy0 = 2 * PH * b0 - 1;                 // lane 0's first C0 row (may be -1)
        if (B::BUFS == 1) stage(b0, c0, even);
        if (load) {
            // (every warp has used the vectors before: with two buffers only the barrier here says so)
            if (B::BUFS == 2) __syncthreads();
            // patch vectors: window [p-2, p+1]^2 of I, zero outside I (partial
            // patches), or row p < n0 of amat (element (dy*4 + dx)*9 + c)
            load = false;
            for (int k = tid; k < 144 * PATCHES; k += 256) {
                const int pl = k % PATCHES, kk = k / PATCHES;
                const int dy = kk % 4, c = (kk / 4) % 9, dx = kk / 36;
                const int p = p_base + pl;
                const float* src = amat ? amat : d1;
                int n = 0;
                if (p < n0) {
                    if (amat) {
                        src = amat + (long long)p * 144 + (dy * 4 + dx) * 9 + c;
                        n = 4;
                    } else {
                        const int x = 4 * (p % g.P0x) + dx, y = 4 * (p / g.P0x) + dy;
                        if (x < g.W1 && y < g.H1) {
                            src = d1 + ((long long)y * g.W1 + x) * 9 + c;
                            n = 4;
                        }
                    }
                }
                cp_async4(&a_s[k].x, src, n);
                cp_async4(&a_s[k].y, src, n);
            }
        }
        if (edged)
            for (int k = tid; k < 9 * HROWS; k += 256) {
                const int c = k / HROWS, x = 2 * c0 - 3, y = cy0 - 2 + k % HROWS;
                const bool in = x >= 0 && y >= 0 && y < H2;
                cp_async4(edge + k, in ? d2 + ((long long)y * W2 + x) * 9 + c : d2, in ? 4 : 0);
            }
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();

        // the tile after this one is staged while this one is computed
        int bn = b0, cn = c0 + PWT;
        wrap(bn, cn);
        if (++t == tiles) t = bn = cn = 0;
        if (B::BUFS == 2 && todo > 1) stage(bn, cn, even == sm ? sm + 2 * COPY : sm);

        if (edged) {
            edged = false;
            // the first window needs the column before the tile: lane r computes its row r
            const int r = lane < CROWS ? lane : CROWS - 1;
            float sv[NP] = {};
#pragma unroll 1
            for (int k = 0; k < 36; k++) {
                const int dx = k / 9, c = k - 9 * dx;
                const float* hp = dx == 0 ? edge + c * HROWS + r : even + c * PLANE + r * HPITCH + dx - 1;
                const int step = dx == 0 ? 1 : HPITCH;
                const float2* ap = a_s + warp * NP + k * 4 * PATCHES;
#pragma unroll
                for (int dy = 0; dy < 4; dy++) {
                    const float h = hp[dy * step];
#pragma unroll
                    for (int q = 0; q < NP; q++) sv[q] = __fmaf_rn(ap[dy * PATCHES + q].x, h, sv[q]);
                }
            }
            const bool in = lane < CROWS && cy0 + lane >= 0 && cy0 + lane < H2;
#pragma unroll
            for (int q = 0; q < NP; q++) {
                const float v = in ? __fmul_rn(sv[q], 0.0625f) : -INFINITY;
                const int r3 = 2 * (lane & 7);           // lane i: pooled row i
                const float v0 = __shfl_sync(0xffffffffu, v, r3), v1 = __shfl_sync(0xffffffffu, v, r3 + 1);
                const float v2 = __shfl_sync(0xffffffffu, v, r3 + 2);
                uint32_t y3;
                const float m = col_max(v0, v1, v2, 0, y3);
                y3 = __reduce_or_sync(0xffffffffu, y3 << (4 * (lane & 7)));
                if (lane < PH) left[q * LEFT + lane] = m;
                if (lane == 8) left[q * LEFT + 8] = __uint_as_float(y3);
            }
            __syncwarp();
        }

        float2 acc[NP][CROWS];
#pragma unroll
        for (int q = 0; q < NP; q++)
#pragma unroll
            for (int r = 0; r < CROWS; r++) acc[q][r] = make_float2(0.0f, 0.0f);
        const float4* ap = reinterpret_cast<const float4*>(a_s) + warp * (NP / 2);      // 2 patches of this warp, each value twice
#pragma unroll 1
        for (int dx = 0; dx < 4; dx++) {
            const float2* hp = reinterpret_cast<const float2*>((dx & 1) ? even + COPY : even) + lane + (dx >> 1);
#pragma unroll 1
            for (int c = 0; c < 9; c++) {
                float2 av[4][NP];
#pragma unroll
                for (int dy = 0; dy < 4; dy++)
#pragma unroll
                for (int q = 0; q < NP; q += 2) {
                    const float4 a = ap[dy * (PATCHES / 2) + q / 2];
                    av[dy][q] = make_float2(a.x, a.y);
                    av[dy][q + 1] = make_float2(a.z, a.w);
                }
                // a staged row at a time: row hr feeds output row hr - dy with dy = 0..3, so each output
                // row gets its four in order and a value is dead as soon as it is used
#pragma unroll
                for (int hr = 0; hr < HROWS; hr++) {
                    const float2 h = hp[hr * (HPITCH / 2)];
#pragma unroll
                    for (int dy = 0; dy < 4; dy++) {
                        const int r = hr - dy;
                        if (r < 0 || r >= CROWS) continue;
#pragma unroll
                        for (int q = 0; q < NP; q++) acc[q][r] = __ffma2_rn(av[dy][q], h, acc[q][r]);
                    }
                }
                hp += PLANE / 2;
                ap += 4 * (PATCHES / 2);
            }
        }
        if (B::BUFS == 1) __syncthreads();   // the next tile's descriptors may be staged

        int band = b0, rx = c0 + lane;
        wrap(band, rx);
        const int x = 2 * rx, ry0 = band * PH;
        const bool inner = 2 * (c0 + PWT) <= W2 && cy0 >= 0 && cy0 + CROWS <= H2;
        const long long pstride = (long long)mh * pitch;
#pragma unroll
        for (int q = 0; q < NP; q++) {
            float2* v = acc[q];
#pragma unroll
            for (int r = 0; r < CROWS; r++) v[r] = __fmul2_rn(v[r], make_float2(0.0625f, 0.0625f));
            if (!inner) {
#pragma unroll
                for (int r = 0; r < CROWS; r++) {
                    const bool rin = 2 * ry0 - 1 + r >= 0 && 2 * ry0 - 1 + r < H2;
                    if (!(rin && x < W2)) v[r].x = -INFINITY;
                    if (!(rin && x + 1 < W2)) v[r].y = -INFINITY;
                }
            }
            // the second column's maxima go to the lane on the right, lane 31's to the next tile
            float right[PH], before[PH];
            uint32_t yr = 0;
#pragma unroll
            for (int i = 0; i < PH; i++) {
                uint32_t y3;
                right[i] = col_max(v[2 * i].y, v[2 * i + 1].y, v[2 * i + 2].y, 4 * i, y3);
                yr |= y3;
            }
#pragma unroll
            for (int i = 0; i < PH; i++) before[i] = __shfl_up_sync(0xffffffffu, right[i], 1);
            uint32_t yb = __shfl_up_sync(0xffffffffu, yr, 1);
            float* lq = left + q * LEFT;
            if (lane == 0) {
#pragma unroll
                for (int i = 0; i < PH; i++) before[i] = c0 > 0 ? lq[i] : -INFINITY;
                yb = __float_as_uint(lq[8]);
            }
            __syncwarp();
            if (lane == 31) {
#pragma unroll
                for (int i = 0; i < PH; i++) lq[i] = right[i];
                lq[8] = __uint_as_float(yr);
            }
            auto pool = [&](int i, int& code) -> float {
                uint32_t ym;
                const float mid = col_max(v[2 * i].x, v[2 * i + 1].x, v[2 * i + 2].x, 0, ym);
                const float best = fmax3(before[i], mid, right[i]);
                const int k0 = before[i] == best ? (int)((yb >> (4 * i)) & 15u) : 15;
                const int k1 = mid == best ? (int)ym + 1 : 15;
                const int k2 = right[i] == best ? (int)((yr >> (4 * i)) & 15u) + 2 : 15;
                code = min(k0, min(k1, k2));
                return best;
            };
            const int p = p_base + NP * warp + q;
            const bool st = rx < mw && p < n0;
            long long o = p * pstride + (long long)ry0 * pitch + rx;
#pragma unroll
            for (int i = 0; i < PH; i += 2) {
                int ca, cb;
                const float va = pool(i, ca), vb = pool(i + 1, cb);
                const bool out0 = st && ry0 + i < mh, out1 = st && ry0 + i + 1 < mh;
                // (lanes without an output evaluate the power of 1)
                const float2 pw = dm_powf2(make_float2(out0 ? va : 1.0f, out1 ? vb : 1.0f), pr);
                if (out0) {
                    pooled0[o] = pw.x;
                    amax0[o] = (unsigned char)ca;
                }
                if (out1) {
                    pooled0[o + pitch] = pw.y;
                    amax0[o + pitch] = (unsigned char)cb;
                }
                o += 2 * pitch;
            }
        }
        if (t == 0) p_base += PATCHES, load = true;
        b0 = bn;
        c0 = cn;
        if (B::BUFS == 2) even = even == sm ? sm + 2 * COPY : sm;
    }
}

template <int PH, int NP>
long long band_units(const DmGeom& g, int n_rows, int bl) {
    constexpr int P = Band<PH, NP>::PATCHES;
    return (long long)((n_rows + P - 1) / P) * band_tiles((g.dh[1] + PH - 1) / PH, bl);
}

// The time of a form: tiles of the busiest SM, each its C0 rows and what costs about four
// more of them besides, for the patches of a CTA; a quarter more where the CTAs of small
// inputs begin inside a band, at a window that needs a column of its own.
template <int PH, int NP>
long long band_cost(const DmGeom& g, int n_rows, int bl, int sms) {
    const long long c = (band_units<PH, NP>(g, n_rows, bl) + sms - 1) / sms * (2 * PH + 5) * NP;
    return NP == 2 && bl != PWT ? c + c / 4 : c;
}

template <int PH, int NP>
cudaError_t launch_band(const DmGeom& g, const float* d1, const float* d2, float lam, float* pooled0, unsigned char* amax0,
                        cudaStream_t st, const float* amat, int n_rows, int bl, int sms) {
    using B = Band<PH, NP>;
    static std::atomic<unsigned long long> smem_done{0};   // > 48 KB dynamic shared memory opted in, per device
    cudaError_t e = dm_smem_opt_in(reinterpret_cast<const void*>(k_corr0_f32<PH, NP>), (int)B::SMEM_BYTES, smem_done);
    if (e != cudaSuccess) return e;
    const long long units = band_units<PH, NP>(g, n_rows, bl), slots = (long long)sms * B::CTAS_SM;
    const long long waves = (units + slots * RANGE - 1) / (slots * RANGE);
    const long long grid = units < slots ? units : slots * waves;
    e = dm_launch_pdl(k_corr0_f32<PH, NP>, (unsigned)grid, 256, B::SMEM_BYTES, st, g, d1, d2, lam, pooled0, amax0, amat, n_rows,
                      units, bl);
    if (e != cudaSuccess) return e;
    dm_count_launches(1);
    return cudaGetLastError();
}

}  // namespace

cudaError_t dm_launch_corr0_f32(const DmGeom& g, const float* d1, const float* d2, float lam, float* pooled0,
                                unsigned char* amax0, cudaStream_t st, const float* amat, int n_rows) {
    if (n_rows < 0) n_rows = g.P0x * g.P0y;
    // The form with the shortest way: bands of 8 rows do the least extra work (17 C0 rows for
    // 16, against 9 for 8 and 5 for 4) and are taken by all but inputs of few tiles, whose
    // time is that of the busiest SM (64x48: 15.2 us with bands of 2, 29.5 with 8; 128x96: 83 us
    // with 8 rows and 4 patches, 88 with 2 patches).  Lanes of a band: whole tiles, or its
    // columns and one (see above), where that makes the tiles fewer.
    const int whole = (g.dw[1] + PWT - 1) / PWT * PWT, dense = g.dw[1] + 1, sms = dm_sm_count();
    int ph = 0, bl = 0;
    long long best = 0;
    auto consider = [&](int rows, int lanes, long long cost) {
        if (ph == 0 || cost < best) ph = rows, bl = lanes, best = cost;
    };
    for (int lanes : {whole, dense}) {
        consider(8, lanes, band_cost<8, 4>(g, n_rows, lanes, sms));
        consider(4, lanes, band_cost<4, 2>(g, n_rows, lanes, sms));
        consider(2, lanes, band_cost<2, 2>(g, n_rows, lanes, sms));
    }
    if (ph == 8) return launch_band<8, 4>(g, d1, d2, lam, pooled0, amax0, st, amat, n_rows, bl, sms);
    if (ph == 4) return launch_band<4, 2>(g, d1, d2, lam, pooled0, amax0, st, amat, n_rows, bl, sms);
    return launch_band<2, 2>(g, d1, d2, lam, pooled0, amax0, st, amat, n_rows, bl, sms);
}
