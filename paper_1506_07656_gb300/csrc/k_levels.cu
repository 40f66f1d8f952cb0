// Pyramid levels l >= 1 (Eq. 5-12, boundary rule of Sec. 3.2, Algorithm 1).
//
// For a lattice patch p at level l with existing children c_i = p + 2^l o_i:
//   C_l(p, q) = (1/n) sum_{existing i} P_{l-1}(c_i, q + o_i)      (0 outside the domain)
// and, below the top, the stored pooled map
//   P_l(p, r) = (max over in-domain m of C_l(p, 2r + m))^lambda   + argmax code,
// or at the top C_L(p, q) = (C_l(p, q))^lambda.
// The children's sum runs in child order i = 0..3, Knuth-TwoSum compensated
// and rounded once (default) or plain (one rounding per addition), then is
// divided by n; pooling is on the unrectified average and the power is
// applied to the pooled value (x -> x^lambda is increasing on [0,1]).
//
// The pass reads the pooled maps of the level below and does a fixed amount of
// arithmetic per stored output (~4 averages of 4 values, a 9-way max with argmax, one
// power).  Algorithmic bytes per stored output: 16 B of child values read (each child
// value is shared by 4 parents), 4 + 1 B written.  Two kernels do it, with the same bits;
// level_streams below says which takes a level, and with what times on either side:
//
// k_level_rows, the row-streaming kernel: a warp walks down the rows of its patches' maps
// in registers, in strips of 64 columns (or of 32, 16 or 8).  It takes the maps that fill
// its strips, those of at most 16 columns, and small images: every level of 1024x436 and
// of 512x224.  Described where it stands.
//
// k_level_sweep, the tiled kernel: the maps that leave strips part-empty (640x480 levels 1
// to 4, 1242x375 levels 2 to 5, 320x240 levels 1 to 3; of small images where the maps are
// wider than 64 columns or another tile than the default was set), and fault injection.  A CTA owns a tile of 32 x TH pooled outputs (TH = 8 by
// default on 4 warps; 16 on 8 or 4 on 2 as tuned shapes) of a run of up to 32 lattice
// patches on one row, spaced so that the right child column of one patch is the left
// child column of the next: the child windows (72 x (2 TH + 1) floats, which cover both
// shifts +-1 of a shared column) are staged in shared memory by 3-D TMA tensor
// loads into a ring of NR = 2 (or 3, as a tuned shape) columns; as soon as a patch's
// averages are formed its left column is released and one thread starts the
// loads of the column NR ahead, which overlap the pooling and rectification.
// Each child window reaches shared memory about twice per (up to) four parents
// instead of four times; the CTAs of one tile row and one row of patches run
// together, so the second staging (by the next row of patches) and the window
// edges shared by neighbouring tiles come from L2.
// Every thread forms the same number of averages and of pooled outputs per
// patch (the CTA meets a barrier after each phase).
// (Rows of the pooled maps are padded to 16 floats and the window's first
// column is a multiple of 4, so every load starts 16-byte aligned; the tensor
// map zero-fills whatever lies outside the domain.)
#include <algorithm>

#include "dm_internal.cuh"

namespace {

// valid[l][p] = 1 iff some child exists (Eq. 7 with the boundary rule; level 0: every
// atomic patch).  A patch's children are two columns times two rows, so it exists iff
// its column and its row do, and has 0, 1, 2 or 4 existing children, never 3.  Every CTA
// derives the columns' and rows' flags of all levels in shared memory and writes its share of
// the patches, all levels in one launch (one launch per level took 28 us at 1024x436 and, at
// 64x48, 15 of 157).
constexpr int VALID_SIDE = 8192;             // lattice columns + rows of a pair, at most; larger ones level by level
constexpr int VALID_THREADS = 1024;
struct ValidArgs {
    DmGeom g;
    unsigned char* v[DM_MAXL + 1];
};
struct ValidBatch {
    ValidArgs a[DM_BATCH_MAX];
};

inline bool valid_fits(const DmGeom& g) { return g.Lx + g.Ly <= VALID_SIDE; }

__device__ __forceinline__ void valid_all(const ValidArgs& a) {
    const DmGeom& g = a.g;
    __shared__ unsigned char flags[2][VALID_SIDE];       // columns, then rows
    const int n = g.Lx * g.Ly, n0 = g.npatch(0);
    const int first = blockIdx.x * blockDim.x + threadIdx.x, step = gridDim.x * blockDim.x;
    for (int p = first; p < n0; p += step) a.v[0][p] = 1;
    for (int i = threadIdx.x; i < g.Lx + g.Ly; i += blockDim.x) flags[0][i] = 1;
    for (int l = 1; l <= g.L; l++) {
        __syncthreads();
        const unsigned char* was = flags[(l & 1) ^ 1];
        unsigned char* now = flags[l & 1];
        for (int i = threadIdx.x; i < g.Lx + g.Ly; i += blockDim.x) {
            const bool row = i >= g.Lx;
            const int k = row ? i - g.Lx : i, at = row ? g.Lx : 0;
            const int m = l == 1 ? (row ? g.P0y : g.P0x) : (row ? g.Ly : g.Lx);   // the children's columns or rows
            const int lo = l == 1 ? k - 1 : k - (1 << (l - 2)), hi = l == 1 ? k : k + (1 << (l - 2));
            now[i] = (lo >= 0 && lo < m && was[at + lo]) || (hi >= 0 && hi < m && was[at + hi]);
        }
        __syncthreads();
        for (int p = first; p < n; p += step) a.v[l][p] = now[p % g.Lx] & now[g.Lx + p / g.Lx];
    }
}

__global__ void __launch_bounds__(VALID_THREADS) k_valid_all(const __grid_constant__ ValidArgs a) {
    dm_pdl_wait();
    valid_all(a);
}
__global__ void __launch_bounds__(VALID_THREADS) k_valid_all_b(const __grid_constant__ ValidBatch B) {
    valid_all(B.a[blockIdx.y]);
}

ValidArgs valid_args(const dm_pyramid& py) {
    ValidArgs a;
    a.g = py.g;
    for (int l = 0; l <= py.g.L; l++) a.v[l] = const_cast<unsigned char*>(py.valid[l]);
    return a;
}

unsigned valid_blocks(long long patches) { return (unsigned)((patches + VALID_THREADS - 1) / VALID_THREADS); }

// One level of it (pairs too large for the kernels above).
__global__ void k_valid(DmGeom g, int l, const unsigned char* __restrict__ vprev, unsigned char* __restrict__ v) {
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= g.Lx * g.Ly) return;
    int ix = p % g.Lx, iy = p / g.Lx;
    unsigned char any = 0;
    for (int i = 0; i < 4; i++) {
        int c = dm_child(g, l, ix, iy, i);
        if (c >= 0 && vprev[c]) any = 1;
    }
    v[p] = any;
}

__global__ void k_fill_u8(unsigned char* p, int n, unsigned char val) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) p[i] = val;
}

// Three-input maximum (one PTX max with three operands).
__device__ __forceinline__ float fmax3(float a, float b, float c) {
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

constexpr int TW = 32;                           // pooled columns per CTA tile (one per lane)
constexpr int AW = 2 * TW + 1;                   // average columns per CTA (65)
constexpr int KW = 72;                           // staged child columns (TMA box width)
constexpr int AWP = 68;                          // padded row of the averages (16-byte aligned rows)
constexpr int LEVEL_THREADS = 256;
// threads of a tiled level CTA for TH pooled rows: 8 warps for 16 rows, 4 for 8,
// 2 for 4 -- every thread forms two 4-column average groups and two pooled
// outputs per patch, and smaller CTAs wait less at their per-patch barriers.
// A BF16 pyramid (rows, ring columns; us): 640x480, four of seven levels tiled, 8 2 6279,
// 8 3 6547, 16 2 6606, 16 3 6884, 4 2 6763, 4 3 7121; 320x240 627, 643, 653, 666, 672, 695;
// 1242x375 14418, 14569, 14704, 14869, 14694, 14924 (row-streaming at every level: 6792, 659, 14790)
template <int TH>
__host__ __device__ constexpr int level_threads() { return TH == 16 ? 256 : (TH == 8 ? 128 : 64); }

// CTA tile of TW x TH pooled outputs (TH = 8, 16 or 4):
// AH rows of averages, child windows of KW x AH floats (KIDF with padding to
// 128 bytes), KID_BYTES delivered by one TMA window load.
template <int TH_>
struct LevelTile {
    static constexpr int TH = TH_;
    static constexpr int AH = 2 * TH + 1;
    static constexpr int KIDF = ((AH * KW + 31) / 32) * 32;
    static constexpr unsigned KID_BYTES = AH * KW * 4;
};
constexpr long long LEVEL_WAIT_CYCLES = 4000000000LL;   // ~2 s at 2 GHz

// Averages at staged row ay, columns ax .. ax+3 of child 0's frame, from the
// four child windows (a missing child's window holds zeros, which leave both
// the plain and the compensated sum of the others unchanged: s + 0 = s exactly,
// with a zero TwoSum error): child i contributes its column ax + o_x,i + 3.
// Children with o_x = -1 (left, windows lt / lb) read columns ax+2 .. ax+5 (two
// aligned float4 loads, which unlike 8-byte loads at a 16-byte stride are free
// of bank conflicts), children with o_x = +1 (right, rt / rb) columns
// ax+4 .. ax+7.  Then times w = 1/n (n is 1, 2 or 4: valid_all).  Two columns per packed
// FP32x2 operation: Knuth's TwoSum (6 additions, every step correctly rounded per lane)
// costs 3 instructions per column and step.
template <bool COMP>
__device__ __forceinline__ float4 avg_group(const float* lt, const float* lb, const float* rt, const float* rb, float w) {
    const float4 a0 = *reinterpret_cast<const float4*>(lt), b0 = *reinterpret_cast<const float4*>(lt + 4);
    const float4 a1 = *reinterpret_cast<const float4*>(lb), b1 = *reinterpret_cast<const float4*>(lb + 4);
    const float4 v2 = *reinterpret_cast<const float4*>(rt + 4);
    const float4 v3 = *reinterpret_cast<const float4*>(rb + 4);
    const float2 r0 = avg_pair4<COMP>(make_float2(a0.z, a0.w), make_float2(a1.z, a1.w), make_float2(v2.x, v2.y),
                                            make_float2(v3.x, v3.y), w);
    const float2 r1 = avg_pair4<COMP>(make_float2(b0.x, b0.y), make_float2(b1.x, b1.y), make_float2(v2.z, v2.w),
                                            make_float2(v3.z, v3.w), w);
    return make_float4(r0.x, r0.y, r1.x, r1.y);
}

// The same for two columns c, c+1 (c even: 8-byte loads at columns c+2 and
// c+4), or -- ONE -- for column c alone (the second lane's result unused).
template <bool COMP, bool ONE>
__device__ __forceinline__ float2 avg_two(const float* lt, const float* lb, const float* rt, const float* rb, float w) {
    float2 x[4];
    if constexpr (ONE) {
        x[0] = make_float2(lt[2], 0.0f);
        x[1] = make_float2(lb[2], 0.0f);
        x[2] = make_float2(rt[4], 0.0f);
        x[3] = make_float2(rb[4], 0.0f);
    } else {
        x[0] = *reinterpret_cast<const float2*>(lt + 2);
        x[1] = *reinterpret_cast<const float2*>(lb + 2);
        x[2] = *reinterpret_cast<const float2*>(rt + 4);
        x[3] = *reinterpret_cast<const float2*>(rb + 4);
    }
    return avg_pair4<COMP>(x[0], x[1], x[2], x[3], w);
}

// Sweep geometry of level l: a CTA owns one tile of TW x TH pooled outputs of a
// run of `run` lattice patches on one row iy, ix = r + (k0 + k) * S.  Patch ix
// has its children in the lattice (or atomic-grid) columns ix - d and ix + d'
// of level l-1 (level 1: ix - 1 and ix; level l >= 2: ix -+ 2^(l-2)), rows
// iy - e, iy + e' likewise; the stride S = 2^(l-1) (1 at level 1) makes the
// right column of one patch the left column of the next, so the run needs
// run + 1 columns of two child windows each instead of 4 windows per patch.
// Runs of 32 (measured at 1024x436 with 8-row tiles at every level wider than 16 columns,
// which the row-streaming kernel has taken over there, levels stage: 8 8.09 ms,
// 16 7.79, 32 7.66, 48 7.67, 64 7.63; 32 keeps more CTAs for small images;
// shorter runs on the small top levels gained nothing).
__host__ __device__ inline int level_run(int) { return 32; }

__device__ __forceinline__ void child_col_row(const DmGeom& g, int l, int ix, int iy, int* cx_left, int* cy_top, int* step) {
    if (l == 1) { *cx_left = ix - 1; *cy_top = iy - 1; *step = 1; }
    else { const int s = 1 << (l - 2); *cx_left = ix - s; *cy_top = iy - s; *step = 2 * s; }
}

// Index at level l-1 of the child at column cx, row cy, or -1 (outside the
// grid, or not existing).
__device__ __forceinline__ int child_at(const DmGeom& g, int l, int cx, int cy, const unsigned char* __restrict__ vprev) {
    const int gx = l == 1 ? g.P0x : g.Lx, gy = l == 1 ? g.P0y : g.Ly;
    if (cx < 0 || cy < 0 || cx >= gx || cy >= gy) return -1;
    const int c = cy * gx + cx;
    return vprev[c] ? c : -1;
}

// Level l in [1, L-1].  Work item = (tile row, row iy, tile column, residue r,
// run k0) with the residue and run fastest, so the CTAs whose windows overlap
// (neighbouring runs, neighbouring tiles of a tile row, and -- one row of
// patches later -- the rows that share child windows) run close together in
// time.  `tmap` maps the pooled maps of
// level l-1 as a 3-D array (columns dw[l], rows dh[l], patches) with a
// 72 x (2 TH + 1) x 1 box.  Dynamic shared memory: a ring of NR columns x 2
// child windows, then the averages.  Per patch of the run: form the averages
// from its two columns, release the left column (thread 0 starts the loads of
// the column NR ahead into it), pool, power, store, wait for the next patch's
// columns; two barriers per patch.
template <bool COMP, int TH, int NR, bool APPROX, int NT = LEVEL_THREADS>
__device__ __forceinline__ void level_sweep_body(const DmGeom& g, int l, const CUtensorMap* tmap_p,
                                                 const unsigned char* __restrict__ vprev, int runs_per_res, int run,
                                                 float* __restrict__ out, unsigned char* __restrict__ amax, float lam,
                                                 int* __restrict__ err, const int* __restrict__ proto_of, int n_maps,
                                                 long long inject_wait, int item) {
    using T = LevelTile<TH>;
    constexpr int AH = T::AH, KIDF = T::KIDF;
    extern __shared__ __align__(128) unsigned char lsm_raw[];
    // TMA destinations must be 128-byte aligned: round the dynamic base up (128 bytes are reserved for this)
    float* lsm = reinterpret_cast<float*>(lsm_raw + ((128u - ((uint32_t)__cvta_generic_to_shared(lsm_raw) & 127u)) & 127u));
    float* ring = lsm;                                       // [NR][2][KIDF]
    float (*avg)[AWP] = reinterpret_cast<float (*)[AWP]>(lsm + NR * 2 * KIDF);
    __shared__ __align__(8) uint64_t bars[NR + 1];          // ring slots, then one barrier nothing completes
    __shared__ int colc[NR][2];                              // child index per ring slot (top, bottom), -1 absent
    __shared__ int abort_s;

    const int ow = g.dw[l + 1], oh = g.dh[l + 1], opitch = g.pitch(l + 1);
    const int mw = g.dw[l], mh = g.dh[l];
    const int tiles_x = (ow + TW - 1) / TW;
    int cx0, cy0, S;
    child_col_row(g, l, 0, 0, &cx0, &cy0, &S);
    const int per_row = S * runs_per_res;
    // work item = (tile row, lattice row iy, tile column, run): the CTAs of one
    // tile row and one row of patches run together, so the window edges that
    // neighbouring tiles of the row share (64-byte memory granules at their x
    // edges) come from DRAM once, and the next row of patches, which stages the
    // same child rows again, follows within a few hundred CTAs, while they are
    // still in L2 (level 1 of 1024x436 on this kernel, tiles of 16 rows: DRAM reads
    // 1.14x the maps; all tiles of a row of patches together instead: 2.1x, their
    // child rows exceed the L2 before the next row of patches reads them again; the
    // tile as the slowest index: 1.83x at 512x224)
    const int rr = item % per_row;
    int t = item / per_row;
    const int tx = t % tiles_x;
    t /= tiles_x;
    const int iy = t % g.Ly;
    const int tile = (t / g.Ly) * tiles_x + tx;
    const int r = rr / runs_per_res, k0 = (rr - r * runs_per_res) * run;
    const int ix0 = r + k0 * S;                              // first patch of the run
    if (ix0 >= g.Lx) return;
    const int nrun = min(run, (g.Lx - 1 - ix0) / S + 1);    // patches in this run
    const int rx0 = (tile % tiles_x) * TW, ry0 = (tile / tiles_x) * TH;
    const int qx0 = 2 * rx0 - 1, qy0 = 2 * ry0 - 1;
    const int xa = 2 * rx0 - 4;                              // first staged child column (multiple of 4 floats)
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int cxl, cyt, st;
    child_col_row(g, l, ix0, iy, &cxl, &cyt, &st);
    const int cyb = cyt + (l == 1 ? 1 : S);                  // bottom child row

    // start the loads of column j (child column cxl + j*S) into slot j % NR (one thread);
    // a missing child's window is loaded from map index -1, outside the tensor,
    // which the TMA unit fills with zeros without reading memory
    auto stage = [&](int j) {
        const int slot = j % NR;
        const int cx = cxl + j * S;
        const int ct = child_at(g, l, cx, cyt, vprev), cb = child_at(g, l, cx, cyb, vprev);
        colc[slot][0] = ct;
        colc[slot][1] = cb;
        const uint32_t bar = (uint32_t)__cvta_generic_to_shared(&bars[slot]);
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" :: "r"(bar), "r"(2u * T::KID_BYTES) : "memory");
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(ring + slot * 2 * KIDF);
        // the map of an atomic child is its prototype's in the approximate form
        int zt = ct, zb = cb;
        if constexpr (APPROX) {
            // (an entry outside [0, maps) would only read the zero fill; it is
            // clamped like everywhere else)
            if (ct >= 0) zt = min(max(__ldg(proto_of + ct), 0), n_maps - 1);
            if (cb >= 0) zb = min(max(__ldg(proto_of + cb), 0), n_maps - 1);
        }
        asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
                     :: "r"(dst), "l"(reinterpret_cast<uint64_t>(tmap_p)), "r"(xa), "r"(qy0 - 1), "r"(zt), "r"(bar)
                     : "memory");
        asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
                     :: "r"(dst + KIDF * 4), "l"(reinterpret_cast<uint64_t>(tmap_p)), "r"(xa), "r"(qy0 + 1), "r"(zb), "r"(bar)
                     : "memory");
    };
    // wait for column j (the (j / NR)-th use of its slot); false on timeout
    auto wait_col = [&](int j) -> bool {
        const uint32_t bar = (uint32_t)__cvta_generic_to_shared(&bars[j % NR]);
        const uint32_t parity = (uint32_t)((j / NR) & 1);
        const long long t0 = clock64();
        while (true) {
            uint32_t done;
            asm volatile("{.reg .pred q; mbarrier.try_wait.parity.shared::cta.b64 q, [%1], %2, %3; selp.u32 %0, 1, 0, q;}"
                         : "=r"(done) : "r"(bar), "r"(parity), "n"(WAIT_HINT_NS) : "memory");
            if (done) return true;
            if (clock64() - t0 > LEVEL_WAIT_CYCLES) return false;
        }
    };

    if (tid == 0) {
        abort_s = 0;
        for (int b = 0; b <= NR; b++)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"((uint32_t)__cvta_generic_to_shared(&bars[b])) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        for (int j = 0; j < NR && j <= nrun; j++) stage(j);
        if (inject_wait > 0) {
            // fault injection: a bounded wait on a barrier nothing completes runs
            // out after inject_wait cycles, exactly like a wait for a load that
            // never lands; the CTA then takes its abort path below (which still
            // waits, with the normal limit, for the loads it has started)
            const uint32_t never = (uint32_t)__cvta_generic_to_shared(&bars[NR]);
            const long long t0 = clock64();
            uint32_t done = 0;
            while (!done && clock64() - t0 <= inject_wait)
                asm volatile("{.reg .pred q; mbarrier.try_wait.parity.shared::cta.b64 q, [%1], %2, %3; selp.u32 %0, 1, 0, q;}"
                             : "=r"(done) : "r"(never), "r"(0u), "n"(WAIT_HINT_NS) : "memory");
            if (!done) { atomicOr(err, 1); abort_s = 1; }
        }
    }
    __syncthreads();
    const DmPow pr = dm_pow_setup(lam);
    const bool interior = qx0 >= 0 && qy0 >= 0 && qx0 + AW <= mw && qy0 + AH <= mh;
    // thread 0 waits for the loads; the barrier after its wait passes their
    // data on to every thread of the CTA
    if (tid == 0 && (!wait_col(0) || !wait_col(1))) { atomicOr(err, 1); abort_s = 1; }
    __syncthreads();                                         // columns 0, 1 and their colc visible; abort agreed
    for (int k = 0; k < nrun; k++) {
        if (abort_s) {
            // let the loads already started finish (each wait bounded) before the CTA exits
            if (tid == 0)
                for (int j = k; j <= min(k + NR - 1, nrun); j++) wait_col(j);
            return;
        }
        const int sl = k % NR, sr = (k + 1) % NR;
        const int ci[4] = {colc[sl][0], colc[sl][1], colc[sr][0], colc[sr][1]};
        const int n = (ci[0] >= 0) + (ci[1] >= 0) + (ci[2] >= 0) + (ci[3] >= 0);
        const int ix = ix0 + k * S;
        const int p = iy * g.Lx + ix;
        if (n > 0) {
            // averages of the tile: rows 0 .. 2 TH - 1 in 16 groups of 4 columns
            // (columns 0 .. 63), 32 TH / NT groups per thread; then the last row's 32
            // column pairs and column 64 of every row, one item each for threads
            // from 64 on.  (A tile that reaches past the map holds -inf at the
            // positions outside the domain, which the pooling then never selects.)
            const float* lt = ring + (sl * 2) * KIDF;
            const float* rt = ring + (sr * 2) * KIDF;
            const float w = n == 4 ? 0.25f : (n == 2 ? 0.5f : 1.0f);
            auto mask = [&](float& v, int ay, int ax) {
                const int qy = qy0 + ay, qx = qx0 + ax;
                if (qy < 0 || qy >= mh || qx < 0 || qx >= mw) v = -INFINITY;
            };
#pragma unroll
            for (int u = 0; u < 32 * TH / NT; u++) {
                const int e = tid + u * NT;
                const int ay = e >> 4, ax = 4 * (e & 15);
                const int o = ay * KW + ax;
                float4 a = avg_group<COMP>(lt + o, lt + KIDF + o, rt + o, rt + KIDF + o, w);
                if (!interior) {
                    mask(a.x, ay, ax);
                    mask(a.y, ay, ax + 1);
                    mask(a.z, ay, ax + 2);
                    mask(a.w, ay, ax + 3);
                }
                *reinterpret_cast<float4*>(&avg[ay][ax]) = a;
            }
            constexpr int XB = NT >= 64 + 32 + AH ? 64 : NT - (32 + AH);   // first thread of the extra items
            const int x = tid - XB;
            if (x >= 0 && x < 32 + AH) {
                if (x < 32) {
                    // last row, columns 2x, 2x + 1
                    const int ay = AH - 1, ax = 2 * x, o = ay * KW + ax;
                    float2 a = avg_two<COMP, false>(lt + o, lt + KIDF + o, rt + o, rt + KIDF + o, w);
                    if (!interior) {
                        mask(a.x, ay, ax);
                        mask(a.y, ay, ax + 1);
                    }
                    *reinterpret_cast<float2*>(&avg[ay][ax]) = a;
                } else {
                    // column 64 of row x - 32
                    const int ay = x - 32, ax = AW - 1, o = ay * KW + ax;
                    float2 a = avg_two<COMP, true>(lt + o, lt + KIDF + o, rt + o, rt + KIDF + o, w);
                    if (!interior) mask(a.x, ay, ax);
                    avg[ay][ax] = a.x;
                }
            }
        }
        __syncthreads();                                     // averages ready; column k no longer needed
        // into the slot column k just released; issued from the last warp, so that
        // warp 0, whose thread 0 waits for the loads, does not carry both
        if (tid == NT - 32 && k + NR <= nrun) stage(k + NR);
        if (n > 0) {
            // 3x3 / 2 max-pool over in-domain averages, first strict maximum, power.
            // A thread owns R = 32 TH / NT vertically adjacent outputs (rows R*warp ..), so
            // the horizontal 3-maxima of the 2R+1 average rows it reads are formed
            // once (a row shared by two outputs serves both); rows are then merged in
            // scan order m_y = -1, 0, 1, which keeps the first strict maximum.
            constexpr int R = 32 * TH / NT;
            static_assert(R >= 1 && 32 + AH <= NT && 32 * TH % NT == 0, "tile rows and threads");
            const int rx = rx0 + lane;
            const int ty0 = R * warp;
            if (rx < ow) {
                float hv[2 * R + 1], h0[2 * R + 1], h1[2 * R + 1];
#pragma unroll
                for (int kk = 0; kk < 2 * R + 1; kk++) {
                    const int ay = 2 * ty0 + kk;             // average row; map row qy0 + ay
                    const float a0 = avg[ay][2 * lane], a1 = avg[ay][2 * lane + 1], a2 = avg[ay][2 * lane + 2];
                    hv[kk] = fmax3(a0, a1, a2);
                    h0[kk] = a0;
                    h1[kk] = a1;
                }
                float best[R], pw[R];
                int code[R];
#pragma unroll
                for (int j = 0; j < R; j++) {
                    // first row holding the maximum (m_y = -1, 0, 1), then the first column of
                    // that row holding it (m_x = -1, 0, 1): the first maximum in scan order
                    best[j] = fmax3(hv[2 * j], hv[2 * j + 1], hv[2 * j + 2]);
                    const bool r0 = hv[2 * j] == best[j], r1 = hv[2 * j + 1] == best[j];
                    const float x0 = r0 ? h0[2 * j] : (r1 ? h0[2 * j + 1] : h0[2 * j + 2]);
                    const float x1 = r0 ? h1[2 * j] : (r1 ? h1[2 * j + 1] : h1[2 * j + 2]);
                    code[j] = (r0 ? 0 : (r1 ? 3 : 6)) + (x0 == best[j] ? 0 : (x1 == best[j] ? 1 : 2));
                }
                // the power of two outputs per packed evaluation (rows past the map
                // are evaluated on whatever the tile holds there and not stored)
#pragma unroll
                for (int j = 0; j + 1 < R; j += 2) {
                    const float2 v = dm_powf2(make_float2(best[j], best[j + 1]), pr);
                    pw[j] = v.x;
                    pw[j + 1] = v.y;
                }
                if constexpr (R % 2 == 1) pw[R - 1] = dm_powf(best[R - 1], lam);
#pragma unroll
                for (int j = 0; j < R; j++) {
                    const int ry = ry0 + ty0 + j;
                    if (ry >= oh) break;
                    const long long o = ((long long)p * oh + ry) * opitch + rx;
                    out[o] = pw[j];
                    amax[o] = (unsigned char)code[j];
                }
            }
        }
        // the next patch's columns k+1, k+2 (waited for by thread 0), then one
        // barrier: averages consumed, those columns and their colc visible, abort agreed
        if (tid == 0 && k + 1 < nrun && (!wait_col(k + 1) || !wait_col(k + 2))) { atomicOr(err, 1); abort_s = 1; }
        __syncthreads();
    }
}

template <bool COMP, int TH, int NR, bool APPROX = false, int NT = level_threads<TH>()>
__global__ void __launch_bounds__(NT) k_level_sweep(DmGeom g, int l, const __grid_constant__ CUtensorMap tmap,
                                                               const unsigned char* __restrict__ vprev,
                                                               int runs_per_res, int run, float* __restrict__ out,
                                                               unsigned char* __restrict__ amax, float lam,
                                                               int* __restrict__ err, const int* __restrict__ proto_of,
                                                               int n_maps, long long inject_wait) {
    level_sweep_body<COMP, TH, NR, APPROX, NT>(g, l, &tmap, vprev, runs_per_res, run, out, amax, lam, err, proto_of, n_maps,
                                               inject_wait, (int)blockIdx.x);
}

// ---------------------------------------------------------------------------
// Row-streaming form of the same pass: a warp walks down the rows of its patches'
// maps in registers, with no shared memory and no barrier but a rare one.
//
// What bounds it: at level 1 of a 1024x436 pair 167 instructions per output at 66 %
// issue, the rest the latency of the child loads (62 % L1 hits; DRAM reads 1.19x the
// maps, 59 % of the copy bandwidth with the writes); 4.49 ms against 5.36 ms of the
// tiled kernel, whose averages go through shared memory between two barriers per patch.
// Also measured there (whole level pass, this form 6.24 ms): the next rows' loads held in
// registers (2 CTAs per SM) 7.8, the child rows staged by 4-D TMA loads of two rows of
// every map 8.2 (a load costs about 45 cycles per map it touches), staged by 16-byte
// asynchronous copies 8.9, all strips of a row in one CTA 6.7.
//
// Work split of level l.  A unit of LPP lanes (32, 16, 8 or 4) owns one lattice
// patch and a strip of 2 LPP pooled columns; a warp holds 32 / LPP units of
// neighbouring patches, so that narrow maps fill their lanes too.  A lane owns two
// neighbouring pooled columns and the four columns of averages they need (the fifth
// is the next lane's first).  A CTA of 4 x 2 warps owns a block of patches spaced
// S = 2^(l-1) apart (1 at level 1), which share their child maps: the right children
// of one patch are the left children of the next, likewise up and down, so 4 x 2
// patches read 15 maps instead of 32 and the rest hits in L1.  It walks down a
// segment of rows.  CTAs are numbered in groups of LV_GROUP along x, then the strips
// (which share the memory sectors at their edges), then the rows of patches, then the
// groups and the segments: the child rows that two rows of patches share are still in
// L2 when the second one reads them (level pass 6.60 ms with all of a row of patches
// first, 6.66 with the strips after the rows of patches, 6.34 so).
constexpr int LV_GROUP = 16;        // CTAs along x numbered together (see level_shape)
constexpr int LV_WX = 4, LV_WY = 2;  // warps of a CTA
constexpr int LV_THREADS = 32 * LV_WX * LV_WY;

__host__ __device__ constexpr int level_stride(int l) { return l == 1 ? 1 : 1 << (l - 1); }

// One row of averages of a lane: columns q0 - 1 .. q0 + 2, then the next
// lane's first (q0 + 3), and the horizontal 3-maxima of the two pooled columns.
struct LvRow {
    float a[5];
    float h0, h1;
};

// The child values of one row of averages: per child side the left pair of
// children's columns q0 - 2 .. q0 + 1 (o_x = -1) and the right pair's q0 .. q0 + 3.
struct LvKids {
    float2 lt0, lt1, lb0, lb1;
    float4 rt, rb;
};

// Average of the four children (child order: left top, left bottom, right top,
// right bottom; zeros for missing ones leave the sums unchanged: s + 0 = s, with
// a zero error) for two columns at once, times w = 1 / n.  The compensated sum's
// first FAST steps take Dekker's Fast2Sum on (max, min), the others Knuth's
// TwoSum: both give the exact rounding error of a sum of non-negative values,
// hence the same bits.  TwoSum costs 3 instructions per value and step on the
// FP32 pipe alone; Fast2Sum 3.5, 2 of them min / max on the integer pipe, which
// is idle here.
template <bool FAST>
__device__ __forceinline__ void lv_two_sum(float2& s, float2 x, float2& err) {
    if constexpr (FAST) {
        const float2 hi = make_float2(fmaxf(s.x, x.x), fmaxf(s.y, x.y)), lo = make_float2(fminf(s.x, x.x), fminf(s.y, x.y));
        const float2 t = __fadd2_rn(s, x);
        err = dm_fsub2(lo, dm_fsub2(t, hi));
        s = t;
    } else {
        dm_two_sum2(s, x, err);
    }
}

constexpr int LV_FAST_STEPS = 2;
template <bool COMP>
__device__ __forceinline__ float2 lv_avg2(float2 x0, float2 x1, float2 x2, float2 x3, float w) {
    float2 sv = x0;
    if constexpr (COMP) {
        float2 cp, err;
        lv_two_sum<(LV_FAST_STEPS > 0)>(sv, x1, cp);
        lv_two_sum<(LV_FAST_STEPS > 1)>(sv, x2, err);
        cp = __fadd2_rn(cp, err);
        lv_two_sum<(LV_FAST_STEPS > 2)>(sv, x3, err);
        cp = __fadd2_rn(cp, err);
        sv = __fadd2_rn(sv, cp);
    } else {
        sv = __fadd2_rn(__fadd2_rn(__fadd2_rn(sv, x1), x2), x3);
    }
    return __fmul2_rn(sv, make_float2(w, w));
}

// Per-lane state of the kernel.
struct LvLane {
    const char* kid[4];     // child maps (nullptr: missing)
    float w;                // 1 / number of children
    int mw, mh;             // child map domain (level l)
    uint32_t pitch4;        // row pitch in bytes
    int q0;                 // 2 x the lane's first pooled column
    bool first;             // q0 == 0: column -1 does not exist
};

// Child values of average row y; `off32` is the byte offset of (row y - 1,
// column q0) in a child map.  IN: every child exists, the rows y - 1, y + 1 and the lane's
// columns lie inside the maps (column -2 of the first lane is the padding before
// the row, whose values are replaced; y - 1 >= 1 there).  Otherwise missing
// children and rows and columns outside the domain read as zeros; a vector whose
// first element lies inside the domain lies inside the row's padded pitch, so it is
// loaded whole and its elements past the domain are replaced.
template <bool IN>
__device__ __forceinline__ LvKids lv_load(const LvLane& L, int y, uint32_t off32) {
    LvKids v;
    if constexpr (IN) {
        const uint32_t ot = off32, ob = ot + 2u * L.pitch4;
        v.lt0 = __ldg(reinterpret_cast<const float2*>(L.kid[0] + ot - 8));
        v.lt1 = __ldg(reinterpret_cast<const float2*>(L.kid[0] + ot));
        v.lb0 = __ldg(reinterpret_cast<const float2*>(L.kid[1] + ob - 8));
        v.lb1 = __ldg(reinterpret_cast<const float2*>(L.kid[1] + ob));
        v.rt = __ldg(reinterpret_cast<const float4*>(L.kid[2] + ot));
        v.rb = __ldg(reinterpret_cast<const float4*>(L.kid[3] + ob));
    } else {
        const size_t off = (size_t)((long long)(y - 1) * L.pitch4 + 4LL * L.q0), ob = off + 2u * (size_t)L.pitch4;
        const bool t = y >= 1 && y <= L.mh, b = y >= -1 && y + 1 < L.mh;
        const bool c0 = L.q0 < L.mw, cl = !L.first && L.q0 - 2 < L.mw;
        const float2 z2 = make_float2(0.0f, 0.0f);
        const float4 z4 = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        v.lt0 = t && cl && L.kid[0] ? __ldg(reinterpret_cast<const float2*>(L.kid[0] + off - 8)) : z2;
        v.lt1 = t && c0 && L.kid[0] ? __ldg(reinterpret_cast<const float2*>(L.kid[0] + off)) : z2;
        v.lb0 = b && cl && L.kid[1] ? __ldg(reinterpret_cast<const float2*>(L.kid[1] + ob - 8)) : z2;
        v.lb1 = b && c0 && L.kid[1] ? __ldg(reinterpret_cast<const float2*>(L.kid[1] + ob)) : z2;
        v.rt = t && c0 && L.kid[2] ? __ldg(reinterpret_cast<const float4*>(L.kid[2] + off)) : z4;
        v.rb = b && c0 && L.kid[3] ? __ldg(reinterpret_cast<const float4*>(L.kid[3] + ob)) : z4;
        if (L.q0 - 1 >= L.mw) { v.lt0.y = 0.0f; v.lb0.y = 0.0f; }
        if (L.q0 + 1 >= L.mw) { v.lt1.y = 0.0f; v.lb1.y = 0.0f; v.rt.y = 0.0f; v.rb.y = 0.0f; }
        if (L.q0 + 2 >= L.mw) { v.rt.z = 0.0f; v.rb.z = 0.0f; }
        if (L.q0 + 3 >= L.mw) { v.rt.w = 0.0f; v.rb.w = 0.0f; }
    }
    return v;
}

// The average at (x, y) (scalar, the same sums), -inf outside the domain: the
// column right of a unit's last lane (x >= 1), one row per lane.
template <bool COMP>
__device__ __forceinline__ float lv_extra(const LvLane& L, int y, int x) {
    const bool t = y >= 1, b = y + 1 < L.mh, r = x + 1 < L.mw;
    if (y < 0 || y >= L.mh || x >= L.mw) return -INFINITY;
    const size_t ot = (size_t)(y - 1) * L.pitch4 + (size_t)x * 4, ob = ot + 2u * (size_t)L.pitch4;
    const float v0 = t && L.kid[0] ? __ldg(reinterpret_cast<const float*>(L.kid[0] + ot - 4)) : 0.0f;
    const float v1 = b && L.kid[1] ? __ldg(reinterpret_cast<const float*>(L.kid[1] + ob - 4)) : 0.0f;
    const float v2 = t && r && L.kid[2] ? __ldg(reinterpret_cast<const float*>(L.kid[2] + ot + 4)) : 0.0f;
    const float v3 = b && r && L.kid[3] ? __ldg(reinterpret_cast<const float*>(L.kid[3] + ob + 4)) : 0.0f;
    float s = v0, comp = 0.0f;
    child_add<COMP>(s, comp, v1);
    child_add<COMP>(s, comp, v2);
    child_add<COMP>(s, comp, v3);
    return __fmul_rn(__fadd_rn(s, comp), L.w);
}

// Averages and horizontal maxima of one row from its child values; `ex` holds the
// unit's extra column for the row in lane `src` of the unit.
template <bool COMP, bool IN, int LPP>
__device__ __forceinline__ LvRow lv_row(const LvLane& L, LvKids v, int y, float ex, int src) {
    LvRow r;
    if constexpr (IN)
        if (L.first) { v.lt0.y = 0.0f; v.lb0.y = 0.0f; }
    const float2 a01 = lv_avg2<COMP>(v.lt0, v.lb0, make_float2(v.rt.x, v.rt.y), make_float2(v.rb.x, v.rb.y), L.w);
    const float2 a23 = lv_avg2<COMP>(v.lt1, v.lb1, make_float2(v.rt.z, v.rt.w), make_float2(v.rb.z, v.rb.w), L.w);
    r.a[0] = L.first ? -INFINITY : a01.x;
    r.a[1] = a01.y;
    r.a[2] = a23.x;
    r.a[3] = a23.y;
    if constexpr (!IN) {
        const bool in = y >= 0 && y < L.mh;
#pragma unroll
        for (int j = 0; j < 4; j++)
            if (!in || L.q0 - 1 + j >= L.mw) r.a[j] = -INFINITY;
    }
    const float nx = __shfl_down_sync(0xffffffffu, r.a[0], 1, LPP);
    const float e = __shfl_sync(0xffffffffu, ex, src, LPP);
    r.a[4] = (threadIdx.x & (LPP - 1)) == LPP - 1 ? e : nx;
    r.h0 = fmax3(r.a[0], r.a[1], r.a[2]);
    r.h1 = fmax3(r.a[2], r.a[3], r.a[4]);
    return r;
}

// Maximum of the 3x3 window whose columns start at a[C] of the rows r0, r1, r2, and
// its code: the first row holding the maximum (m_y = -1, 0, 1), then the first
// column of that row holding it: the first maximum in scan order.
template <int C>
__device__ __forceinline__ float lv_pool(const LvRow& r0, const LvRow& r1, const LvRow& r2, uint32_t& code) {
    const float h0 = C ? r0.h1 : r0.h0, h1 = C ? r1.h1 : r1.h0, h2 = C ? r2.h1 : r2.h0;
    const float b = fmax3(h0, h1, h2);
    const bool p0 = h0 == b, p1 = h1 == b;
    const float x0 = p0 ? r0.a[C] : (p1 ? r1.a[C] : r2.a[C]);
    const float x1 = p0 ? r0.a[C + 1] : (p1 ? r1.a[C + 1] : r2.a[C + 1]);
    code = (p0 ? 0u : (p1 ? 3u : 6u)) + (x0 == b ? 0u : (x1 == b ? 1u : 2u));
    return b;
}

template <bool COMP, int LPP>
__device__ __forceinline__ void level_rows_body(const DmGeom& g, int l, const float* __restrict__ prev,
                                                const unsigned char* __restrict__ vprev, int nbx, int nby, int seg_rows,
                                                float* __restrict__ out, unsigned char* __restrict__ amax, float lam,
                                                const int* __restrict__ proto_of, int n_maps, unsigned item) {
    constexpr int UPW = 32 / LPP;                            // units per warp
    const int lane = threadIdx.x & 31, ul = lane & (LPP - 1);
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);   // warp-uniform
    const int ow = g.dw[l + 1], oh = g.dh[l + 1], opitch = g.pitch(l + 1);

    const int S = level_stride(l), strips = (ow + 2 * LPP - 1) / (2 * LPP);
    // numbering of the CTAs: see level_shape
    const unsigned nbxs = (unsigned)(S * nbx), nbys = (unsigned)(S * nby), per = nbys * (unsigned)(strips * LV_GROUP);
    const unsigned groups = (nbxs + LV_GROUP - 1) / LV_GROUP;
    unsigned t = item;
    const int seg = (int)(t / (per * groups));
    t -= (unsigned)seg * per * groups;
    const unsigned grp = t / per;
    t -= grp * per;
    const int byi = (int)(t / (unsigned)(strips * LV_GROUP));
    t -= (unsigned)byi * (unsigned)(strips * LV_GROUP);
    const int strip = (int)(t / LV_GROUP), bxi = (int)(grp * LV_GROUP + t % LV_GROUP);
    if (bxi >= (int)nbxs) return;                            // (the whole CTA)
    // residues slowest: consecutive blocks of a residue share child maps
    const int res_x = bxi / nbx, res_y = byi / nby;
    const int ix = res_x + (((bxi - res_x * nbx) * LV_WX + (warp & (LV_WX - 1))) * UPW + (LPP == 32 ? 0 : lane / LPP)) * S;
    const int iy = res_y + ((byi - res_y * nby) * LV_WY + warp / LV_WX) * S;
    const int p = iy * g.Lx + ix;

    LvLane L;
    L.mw = g.dw[l];
    L.mh = g.dh[l];
    L.pitch4 = (uint32_t)g.pitch(l) * 4u;
    L.q0 = 4 * (strip * LPP + ul);
    L.first = L.q0 == 0;
    const size_t csize = (size_t)g.psize(l);
    int n = 0;
#pragma unroll
    for (int i = 0; i < 4; i++) {
        const int c = (ix < g.Lx && iy < g.Ly) ? dm_child(g, l, ix, iy, i) : -1;
        L.kid[i] = nullptr;
        if (c >= 0 && vprev[c]) {
            const int cm = proto_of ? min(max(__ldg(proto_of + c), 0), n_maps - 1) : c;
            L.kid[i] = reinterpret_cast<const char*>(prev + (size_t)cm * csize);
            n++;
        }
    }
    L.w = n == 4 ? 0.25f : (n == 2 ? 0.5f : 1.0f);
    const bool any = __any_sync(0xffffffffu, n > 0);
    // every unit of the warp has all its children and a complete strip (and byte
    // offsets within a map fit 32 bits): rows inside the map need no checks
    const bool full = __all_sync(0xffffffffu, n == 4) && 4 * LPP * (strip + 1) <= L.mw && csize < (1u << 29);
    const int xe = 4 * LPP * (strip + 1) - 1;                // the extra column
    const int ry0 = seg * seg_rows, ry1 = min(oh, ry0 + seg_rows);
    const int rx = 2 * (strip * LPP + ul);
    const bool st0 = n > 0 && rx < ow, st1 = n > 0 && rx + 1 < ow;
    const DmPow pr = dm_pow_setup(lam);

    // outputs: the patch's maps and the byte offset of (row ry, column rx) in the codes
    char* ovals = reinterpret_cast<char*>(out + (size_t)p * oh * opitch);
    unsigned char* ocodes = amax + (size_t)p * oh * opitch;
    uint32_t oo = (uint32_t)ry0 * (uint32_t)opitch + (uint32_t)rx;
    const uint32_t pitch4 = L.pitch4;
    uint32_t off = (uint32_t)(2 * ry0 - 2) * pitch4 + (uint32_t)L.q0 * 4u;   // (row y - 1, column q0) of y = 2 ry0 - 1
    LvRow r0;
    if (any) {
        const int y = 2 * ry0 - 1;
        const float ex = lv_extra<COMP>(L, y, xe);
        r0 = full && ry0 >= 2 && y + 1 < L.mh ? lv_row<COMP, true, LPP>(L, lv_load<true>(L, y, off), y, ex, 0)
                                              : lv_row<COMP, false, LPP>(L, lv_load<false>(L, y, off), y, ex, 0);
    }
    off += pitch4;
    for (int c0 = ry0; c0 < ry1; c0 += LPP / 2) {
        __syncthreads();                                     // keeps the warps that share child rows together
        if (!any) continue;
        const float ex = lv_extra<COMP>(L, 2 * c0 + ul, xe);  // the extra column of the next LPP rows
        const int c1 = min(ry1, c0 + LPP / 2);
        for (int ry = c0; ry < c1; ry++) {
            const int y = 2 * ry;
            uint32_t k0, k1;
            if (full && y >= 2 && y + 2 < L.mh) {
                const LvKids v1 = lv_load<true>(L, y, off), v2 = lv_load<true>(L, y + 1, off + pitch4);
                const LvRow r1 = lv_row<COMP, true, LPP>(L, v1, y, ex, y - 2 * c0);
                const LvRow r2 = lv_row<COMP, true, LPP>(L, v2, y + 1, ex, y + 1 - 2 * c0);
                const float b0 = lv_pool<0>(r0, r1, r2, k0), b1 = lv_pool<2>(r0, r1, r2, k1);
                *reinterpret_cast<float2*>(ovals + (size_t)(4u * oo)) = dm_powf2(make_float2(b0, b1), pr);
                *reinterpret_cast<unsigned short*>(ocodes + oo) = (unsigned short)(k0 | (k1 << 8));
                r0 = r2;
            } else {
                const LvKids v1 = lv_load<false>(L, y, off), v2 = lv_load<false>(L, y + 1, off + pitch4);
                const LvRow r1 = lv_row<COMP, false, LPP>(L, v1, y, ex, y - 2 * c0);
                const LvRow r2 = lv_row<COMP, false, LPP>(L, v2, y + 1, ex, y + 1 - 2 * c0);
                const float b0 = lv_pool<0>(r0, r1, r2, k0), b1 = lv_pool<2>(r0, r1, r2, k1);
                // (lanes without an output evaluate the power of 1; a last odd column's
                // partner lands in the row's padding)
                const float2 pw = dm_powf2(make_float2(st0 ? b0 : 1.0f, st1 ? b1 : 1.0f), pr);
                if (st0) {
                    *reinterpret_cast<float2*>(ovals + (size_t)4 * oo) = pw;
                    *reinterpret_cast<unsigned short*>(ocodes + oo) = (unsigned short)(k0 | (k1 << 8));
                }
                r0 = r2;
            }
            oo += (uint32_t)opitch;
            off += 2u * pitch4;
        }
    }
}

template <bool COMP, int LPP>
__global__ void __launch_bounds__(LV_THREADS, 4)
k_level_rows(DmGeom g, int l, const float* __restrict__ prev, const unsigned char* __restrict__ vprev, int nbx, int nby,
             int seg_rows, float* __restrict__ out, unsigned char* __restrict__ amax, float lam,
             const int* __restrict__ proto_of, int n_maps) {
    dm_pdl_wait();
    level_rows_body<COMP, LPP>(g, l, prev, vprev, nbx, nby, seg_rows, out, amax, lam, proto_of, n_maps, blockIdx.x);
}

// Top level L: C_L = (mean of children)^lambda over the domain of level L.
template <bool COMP>
__global__ void k_level_top(DmGeom g, int l, const unsigned char* __restrict__ vprev,
                            const unsigned char* __restrict__ vcur, const float* __restrict__ prev,
                            float* __restrict__ top, float lam, const int* __restrict__ proto_of, int n_maps) {
    const int p = blockIdx.y;
    dm_pdl_wait();
    if (!vcur[p]) return;
    const int mw = g.dw[l], mh = g.dh[l];
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= mw * mh) return;
    Kids k;
    load_kids(g, l, p, vprev, prev, k, proto_of, n_maps);
    float a = child_mean<COMP>(k, q % mw, q / mw, mw, mh, g.pitch(l));
    top[(long long)p * mw * mh + q] = dm_powf(a, lam);
}

template <bool COMP, int TH, int NR, bool APPROX = false, int NT = level_threads<TH>()>
cudaError_t launch_sweep(const DmGeom& g, int l, const CUtensorMap& tm, const dm_pyramid& py, int per_res, long long items,
                         float lam, int* status, cudaStream_t st) {
    const size_t smem = (size_t)(NR * 2 * LevelTile<TH>::KIDF + LevelTile<TH>::AH * AWP) * sizeof(float) + 128;
    static std::atomic<unsigned long long> smem_done{0};
    cudaError_t ea = dm_smem_opt_in(reinterpret_cast<const void*>(k_level_sweep<COMP, TH, NR, APPROX, NT>), (int)smem, smem_done);
    if (ea != cudaSuccess) return ea;
    if (items <= 0) return cudaSuccess;
    if (items > 0x7fffffffLL) return cudaErrorInvalidValue;
    k_level_sweep<COMP, TH, NR, APPROX, NT><<<(unsigned)items, NT, smem, st>>>(g, l, tm, py.valid[l - 1], per_res, level_run(l),
                                                                          const_cast<float*>(py.pooled[l]),
                                                                          const_cast<unsigned char*>(py.amax[l]), lam, status,
                                                                          APPROX ? py.proto_of : nullptr, py.n0_maps,
                                                                          py.inject_wait);
    return cudaGetLastError();
}

// Launch shape of the row-streaming kernel at level l.
struct LvShape {
    int lpp, nbx, nby, seg_rows;     // lanes per unit, blocks of patches per residue, rows per segment
    double fill;                     // share of the units' pooled columns that exist
    long long blocks;
};

LvShape level_shape(const DmGeom& g, int l, int sms) {
    LvShape s;
    const int ow = g.dw[l + 1], oh = g.dh[l + 1], S = level_stride(l);
    // lanes per unit: the least lanes per row, a unit's memory sectors past its edges
    // counted as 4 lanes
    s.lpp = 32;
    double best = 1e30;
    for (int lpp = 32; lpp >= 4; lpp /= 2) {
        const double cost = (double)((ow + 2 * lpp - 1) / (2 * lpp)) * (lpp + 4);
        if (cost < best) { best = cost; s.lpp = lpp; }
    }
    const int strips = (ow + 2 * s.lpp - 1) / (2 * s.lpp);
    s.fill = (double)ow / (2.0 * s.lpp * strips);
    const int px = LV_WX * (32 / s.lpp);                     // patches along x of a CTA
    s.nbx = ((g.Lx + S - 1) / S + px - 1) / px;
    s.nby = ((g.Ly + S - 1) / S + LV_WY - 1) / LV_WY;
    // segments of about 32 rows of outputs (each costs one more row of averages, and
    // a shorter one keeps more of the child rows that two rows of patches share in L2:
    // whole columns 6.34, 64 rows 6.34, 32 rows 6.34, 16 rows 6.50 ms for the levels of
    // 1024x436), shorter where the patches alone leave the GPU idle
    const long long per_seg = (long long)S * s.nby * strips * ((S * s.nbx + LV_GROUP - 1) / LV_GROUP) * LV_GROUP;
    const long long fit = 8LL * sms;
    const long long segs = std::max<long long>((oh + 31) / 32, std::min<long long>((oh + 2) / 3, (fit + per_seg - 1) / per_seg));
    s.seg_rows = (int)((oh + segs - 1) / segs);
    s.blocks = (long long)((oh + s.seg_rows - 1) / s.seg_rows) * per_seg;
    return s;
}

template <bool COMP, int LPP>
cudaError_t launch_rows_lpp(const DmGeom& g, int l, const dm_pyramid& py, const LvShape& s, float lam, cudaStream_t st) {
    static std::atomic<unsigned long long> l1_done{0};
    const cudaError_t e = dm_prefer_l1(reinterpret_cast<const void*>(k_level_rows<COMP, LPP>), l1_done);
    if (e != cudaSuccess) return e;
    return dm_launch_pdl(
        k_level_rows<COMP, LPP>, (unsigned)s.blocks, LV_THREADS, 0, st, g, l, py.pooled[l - 1], py.valid[l - 1], s.nbx, s.nby, s.seg_rows, const_cast<float*>(py.pooled[l]),
        const_cast<unsigned char*>(py.amax[l]), lam, l == 1 ? py.proto_of : nullptr, py.n0_maps);
}

template <bool COMP>
cudaError_t launch_rows(const DmGeom& g, int l, const dm_pyramid& py, const LvShape& s, float lam, cudaStream_t st) {
    if (s.blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
    if (s.lpp == 32) return launch_rows_lpp<COMP, 32>(g, l, py, s, lam, st);
    if (s.lpp == 16) return launch_rows_lpp<COMP, 16>(g, l, py, s, lam, st);
    if (s.lpp == 8) return launch_rows_lpp<COMP, 8>(g, l, py, s, lam, st);
    return launch_rows_lpp<COMP, 4>(g, l, py, s, lam, st);
}

// Which kernel takes level l.  The row-streaming one where the tuned shape asks for it
// (level_th = 0) and for maps of at most 16 columns; for maps of up to 64 columns, where
// they fill its strips (one of 64 or of 32) to 88 % or the image is small (the tiled
// kernel's per-patch pipeline is then latency-bound; not where another tile than the default
// was set, which is a request for it); for wider maps where they fill strips of 64 to
// 88 % and the patches (twice the columns) are enough to hide its loads: it moves less through L1 and L2 than
// the tiled kernel, which has no such granularity.  A fault-injection run takes the
// tiled kernel, which holds the bounded waits.
//   Measured (us, tiled / row-streaming; columns of the stored map in front): 1024x436 256
// 5362 / 4487, 128 1362 / 1137, 64 395 / 309, 32 117 / 113, 1242x375 311 (97 % filled) 6043 /
// 5484, 512x224 128 370 / 311, 256x256 64 132 / 113; 640x480 160 (in strips of 32) 2497 / 2806,
// 80 807 / 909, 20 80 / 115, 1242x375 156 1535 / 1790; 130x70 33 41 / 29.
//   Image 1 of few patches (what the tiled kernel adds to a call of dm_correlate_pyramid): maps
// of 40 columns, patches in front: 144 +9, 576 +10, 1024 +11, 1936 +13; 80 columns: 144 -15,
// 576 -24, 1024 -29, 1936 -21; 160: -42, -38, -41, -48; 128 (filled): 144 -2, 576 +8, 1024 +2;
// 256 (filled): 144 -19, 576 +11, 1024 +28; 311 (filled): 144 -36, 400 -26, 576 -14, 1024 +1, 1936 +28.
bool level_streams(const DmGeom& g, int l, const DmTune& tune, const LvShape& s) {
    const int ow = g.dw[l + 1], np = g.npatch(l);
    if (tune.level_th == 0 || ow <= 16) return true;
    const bool filled = s.fill >= 0.88, default_tile = tune.level_th == 8 && tune.level_ring == 2;
    if (ow <= 64) return (np <= 2048 && default_tile) || (filled && (s.lpp == 32 || ow <= 32));
    return filled && s.lpp == 32 && np >= 2 * ow;
}

// ---------------------------------------------------------------------------
// Cross-pair form: one launch per step of the pass for every pair of a wave
// of the batched form (dm_launch_levels_batch).  The per-pair arguments travel
// in the kernel parameters (a captured graph replays them as they were), and
// block b of a launch belongs to the pair j with first[j] <= b < first[j+1]
// (tiled and row-streaming kernels) or to pair blockIdx.y / blockIdx.z.
// ---------------------------------------------------------------------------
struct LvPair {
    CUtensorMap tmap;          // tiled kernel: the pooled maps of level l-1
    DmGeom g;
    const unsigned char* vprev;
    unsigned char* vcur;
    const float* prev;         // pooled maps of level l-1
    float* out;                // pooled maps of level l (or the top)
    unsigned char* amax;
    int* err;
    int a, b;                  // tiled: runs per residue; row-streaming: blocks per residue in x, y
    int seg_rows;              // row-streaming: rows per segment
    long long first;           // first block of this pair in the launch
};
struct LvBatch {
    LvPair p[DM_BATCH_MAX];
    int n;
};

__device__ __forceinline__ int lv_pair_of(const LvBatch& B, long long blk) {
    int j = 0;
    while (j + 1 < B.n && blk >= B.p[j + 1].first) j++;
    return j;
}

template <bool COMP, int TH, int NR>
__global__ void __launch_bounds__(level_threads<TH>()) k_level_sweep_b(const __grid_constant__ LvBatch B, int l, float lam) {
    const int j = lv_pair_of(B, blockIdx.x);
    const LvPair& P = B.p[j];
    level_sweep_body<COMP, TH, NR, false, level_threads<TH>()>(P.g, l, &P.tmap, P.vprev, P.a, level_run(l), P.out, P.amax,
                                                               lam, P.err, nullptr, 0, 0,
                                                               (int)((long long)blockIdx.x - P.first));
}

template <bool COMP, int LPP>
__global__ void __launch_bounds__(LV_THREADS, 4) k_level_rows_b(const __grid_constant__ LvBatch B, int l, float lam) {
    const int j = lv_pair_of(B, blockIdx.x);
    const LvPair& P = B.p[j];
    level_rows_body<COMP, LPP>(P.g, l, P.prev, P.vprev, P.a, P.b, P.seg_rows, P.out, P.amax, lam, nullptr, 0,
                               (unsigned)((long long)blockIdx.x - P.first));
}

__global__ void k_valid_b(const __grid_constant__ LvBatch B, int l) {
    const LvPair& P = B.p[blockIdx.y];
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (l == 0) {
        if (p < P.g.npatch(0)) P.vcur[p] = 1;
        return;
    }
    if (p >= P.g.Lx * P.g.Ly) return;
    const int ix = p % P.g.Lx, iy = p / P.g.Lx;
    unsigned char any = 0;
    for (int i = 0; i < 4; i++) {
        const int c = dm_child(P.g, l, ix, iy, i);
        if (c >= 0 && P.vprev[c]) any = 1;
    }
    P.vcur[p] = any;
}

template <bool COMP>
__global__ void k_level_top_b(const __grid_constant__ LvBatch B, int l, float lam) {
    const LvPair& P = B.p[blockIdx.z];
    const DmGeom& g = P.g;
    const int p = blockIdx.y;
    if (p >= g.npatch(l) || !P.vcur[p]) return;
    const int mw = g.dw[l], mh = g.dh[l];
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= mw * mh) return;
    Kids k;
    load_kids(g, l, p, P.vprev, P.prev, k, nullptr, g.npatch(0));
    const float a = child_mean<COMP>(k, q % mw, q / mw, mw, mh, g.pitch(l));
    P.out[(long long)p * mw * mh + q] = dm_powf(a, lam);
}

}  // namespace

bool dm_level_tiled(const DmGeom& g, int l, const DmTune& tune) {
    return l >= 1 && l < g.L && !level_streams(g, l, tune, level_shape(g, l, 1));   // (the rule does not depend on the SMs)
}

cudaError_t dm_launch_levels(const DmGeom& g, const dm_pyramid& py, float lam, int* status, cudaStream_t st) {
    const int B = 128;
    int n0 = g.npatch(0), np = g.npatch(1);
    const int sms = dm_sm_count();
    const bool whole = valid_fits(g);
    if (whole) dm_launch_pdl(k_valid_all, valid_blocks(max(n0, np)), VALID_THREADS, 0, st, valid_args(py));
    else k_fill_u8<<<(n0 + 255) / 256, 256, 0, st>>>(const_cast<unsigned char*>(py.valid[0]), n0, 1);
    for (int l = 1; l <= g.L; l++) {
        if (!whole) k_valid<<<(np + 255) / 256, 256, 0, st>>>(g, l, py.valid[l - 1], const_cast<unsigned char*>(py.valid[l]));
        const LvShape sh = l < g.L ? level_shape(g, l, sms) : LvShape();
        if (l < g.L && py.inject_wait == 0 && level_streams(g, l, py.tune, sh)) {
            const cudaError_t e = py.compensated ? launch_rows<true>(g, l, py, sh, lam, st) : launch_rows<false>(g, l, py, sh, lam, st);
            if (e != cudaSuccess) return e;
        } else if (l < g.L) {
            // pooled maps of level l-1: [npatch(l-1)][dh[l]][pitch(l)] floats
            // level 1 of an approximate pyramid reads the level-0 maps through the
            // prototype index: its own kernel instance, 16-row tiles, ring of 2
            const bool approx = l == 1 && py.proto_of != nullptr;
            const int th = approx ? 16 : (py.tune.level_th == 8 || py.tune.level_th == 4 ? py.tune.level_th : 16);
            CUtensorMap tm;
            // (level 0 holds n0_maps maps: one per atomic patch, or per prototype)
            const cuuint64_t dims[3] = {(cuuint64_t)g.dw[l], (cuuint64_t)g.dh[l],
                                        (cuuint64_t)(l == 1 ? py.n0_maps : g.npatch(l - 1))};
            const cuuint64_t strides[2] = {(cuuint64_t)g.pitch(l) * 4, (cuuint64_t)g.psize(l) * 4};
            const cuuint32_t box[3] = {KW, (cuuint32_t)(2 * th + 1), 1};
            if (!dm_encode_tiled(&tm, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<float*>(py.pooled[l - 1]), dims,
                                 strides, box))
                return cudaErrorNotSupported;
            const int tiles = ((g.dw[l + 1] + TW - 1) / TW) * ((g.dh[l + 1] + th - 1) / th);
            const int S = l == 1 ? 1 : 1 << (l - 1);
            const int run = level_run(l);
            const int per_res = ((g.Lx + S - 1) / S + run - 1) / run;    // runs per residue class
            const long long items = (long long)tiles * g.Ly * S * per_res;
            cudaError_t e;
            const bool r2 = py.tune.level_ring == 2;
            if (approx)
                e = py.compensated ? launch_sweep<true, 16, 2, true>(g, l, tm, py, per_res, items, lam, status, st)
                                   : launch_sweep<false, 16, 2, true>(g, l, tm, py, per_res, items, lam, status, st);
            else if (th == 8)
                e = py.compensated ? (r2 ? launch_sweep<true, 8, 2> : launch_sweep<true, 8, 3>)(g, l, tm, py, per_res, items, lam, status, st)
                                   : (r2 ? launch_sweep<false, 8, 2> : launch_sweep<false, 8, 3>)(g, l, tm, py, per_res, items, lam, status, st);
            else if (th == 4)
                e = py.compensated ? (r2 ? launch_sweep<true, 4, 2> : launch_sweep<true, 4, 3>)(g, l, tm, py, per_res, items, lam, status, st)
                                   : (r2 ? launch_sweep<false, 4, 2> : launch_sweep<false, 4, 3>)(g, l, tm, py, per_res, items, lam, status, st);
            else
                e = py.compensated ? (r2 ? launch_sweep<true, 16, 2> : launch_sweep<true, 16, 3>)(g, l, tm, py, per_res, items, lam, status, st)
                                   : (r2 ? launch_sweep<false, 16, 2> : launch_sweep<false, 16, 3>)(g, l, tm, py, per_res, items, lam, status, st);
            if (e != cudaSuccess) return e;
        } else {
            int n = g.dw[l] * g.dh[l];
            dim3 grid((n + B - 1) / B, np);
            auto kern = py.compensated ? k_level_top<true> : k_level_top<false>;
            dm_launch_pdl(kern, grid, B, 0, st, g, l, py.valid[l - 1], py.valid[l], py.pooled[l - 1], const_cast<float*>(py.top),
                          lam, l == 1 ? py.proto_of : nullptr, py.n0_maps);
        }
    }
    dm_count_launches(1 + (whole ? 1 : 2) * g.L);
    return cudaGetLastError();
}

// Levels >= 1 of the n <= DM_BATCH_MAX pyramids of a wave (level 0 computed):
// per level, one launch of the existence flags and one launch per kernel shape
// in use (tiled with each tuned (rows, ring), row-streaming, top) for all the
// pairs at that level; status[j] receives pair j's bounded-wait flag.
cudaError_t dm_launch_levels_batch(const dm_pyramid* const* pys, int n, float lam, int* const* status, cudaStream_t st) {
    if (n < 1 || n > DM_BATCH_MAX) return cudaErrorInvalidValue;
    const bool comp = pys[0]->compensated != 0;
    const int sms = dm_sm_count();
    int Lmax = 0;
    for (int j = 0; j < n; j++) Lmax = max(Lmax, pys[j]->g.L);
    long long launches = 0;
    auto base_pair = [&](int j, int l) {
        const dm_pyramid& py = *pys[j];
        LvPair q;
        memset(&q, 0, sizeof(q));
        q.g = py.g;
        q.vprev = l >= 1 ? py.valid[l - 1] : nullptr;
        q.vcur = const_cast<unsigned char*>(py.valid[l]);
        q.prev = l >= 1 ? py.pooled[l - 1] : nullptr;
        q.out = l < py.g.L ? const_cast<float*>(py.pooled[l]) : const_cast<float*>(py.top);
        q.amax = l < py.g.L ? const_cast<unsigned char*>(py.amax[l]) : nullptr;
        q.err = status[j];
        return q;
    };
    bool whole = true;
    for (int j = 0; j < n; j++) whole = whole && valid_fits(pys[j]->g);
    if (whole) {
        ValidBatch V;
        int maxp = 0;
        for (int j = 0; j < n; j++) {
            V.a[j] = valid_args(*pys[j]);
            maxp = max(maxp, max(pys[j]->g.npatch(0), pys[j]->g.npatch(1)));
        }
        k_valid_all_b<<<dim3(valid_blocks(maxp), (unsigned)n), VALID_THREADS, 0, st>>>(V);
        launches++;
    }
    for (int l = 0; l <= Lmax; l++) {
        // existence flags of level l (level 0: every atomic patch)
        if (!whole) {
            LvBatch B;
            memset(&B, 0, sizeof(B));
            int maxp = 0;
            for (int j = 0; j < n; j++)
                if (l <= pys[j]->g.L) {
                    B.p[B.n++] = base_pair(j, l);
                    maxp = max(maxp, pys[j]->g.npatch(l));
                }
            if (B.n == 0) break;
            k_valid_b<<<dim3((unsigned)((maxp + 255) / 256), (unsigned)B.n), 256, 0, st>>>(B, l);
            launches++;
        }
        if (l == 0) continue;
        // the pairs whose level l is the top
        {
            LvBatch B;
            memset(&B, 0, sizeof(B));
            int maxq = 0, maxp = 0;
            for (int j = 0; j < n; j++)
                if (l == pys[j]->g.L) {
                    B.p[B.n++] = base_pair(j, l);
                    maxq = max(maxq, pys[j]->g.dw[l] * pys[j]->g.dh[l]);
                    maxp = max(maxp, pys[j]->g.npatch(l));
                }
            if (B.n) {
                const dim3 grid((unsigned)((maxq + 127) / 128), (unsigned)maxp, (unsigned)B.n);
                if (comp) k_level_top_b<true><<<grid, 128, 0, st>>>(B, l, lam);
                else k_level_top_b<false><<<grid, 128, 0, st>>>(B, l, lam);
                launches++;
            }
        }
        // the pairs below their top: one launch per kernel shape in use.
        // shape 1 + 2 (rows 16 / 8 / 4 as 0 / 1 / 2) + (ring == 3): tiled; 7 .. 10:
        // row-streaming with units of 32, 16, 8 and 4 lanes
        for (int shape = 1; shape < 11; shape++) {
            LvBatch B;
            memset(&B, 0, sizeof(B));
            long long blocks = 0;
            for (int j = 0; j < n; j++) {
                const dm_pyramid& py = *pys[j];
                const DmGeom& g = py.g;
                if (l >= g.L) continue;
                const LvShape sh = level_shape(g, l, sms);
                const bool stream = level_streams(g, l, py.tune, sh);
                const int th = py.tune.level_th == 8 || py.tune.level_th == 4 ? py.tune.level_th : 16;
                const int nr = py.tune.level_ring == 3 ? 3 : 2;
                const int my = stream ? (sh.lpp == 32 ? 7 : sh.lpp == 16 ? 8 : sh.lpp == 8 ? 9 : 10) : 1 + 2 * (th == 16 ? 0 : (th == 8 ? 1 : 2)) + (nr == 3);
                if (my != shape) continue;
                LvPair q = base_pair(j, l);
                const int S = l == 1 ? 1 : 1 << (l - 1);
                long long items;
                if (stream) {
                    q.a = sh.nbx;
                    q.b = sh.nby;
                    q.seg_rows = sh.seg_rows;
                    items = sh.blocks;
                } else {
                    const cuuint64_t dims[3] = {(cuuint64_t)g.dw[l], (cuuint64_t)g.dh[l], (cuuint64_t)g.npatch(l - 1)};
                    const cuuint64_t strides[2] = {(cuuint64_t)g.pitch(l) * 4, (cuuint64_t)g.psize(l) * 4};
                    const cuuint32_t box[3] = {KW, (cuuint32_t)(2 * th + 1), 1};
                    if (!dm_encode_tiled(&q.tmap, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<float*>(py.pooled[l - 1]),
                                         dims, strides, box))
                        return cudaErrorNotSupported;
                    const int tiles = ((g.dw[l + 1] + TW - 1) / TW) * ((g.dh[l + 1] + th - 1) / th);
                    const int run = level_run(l);
                    q.a = ((g.Lx + S - 1) / S + run - 1) / run;
                    items = (long long)tiles * g.Ly * S * q.a;
                }
                q.first = blocks;
                blocks += items;
                B.p[B.n++] = q;
            }
            if (B.n == 0 || blocks == 0) continue;
            if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
            cudaError_t e = cudaSuccess;
            if (shape >= 7) {
                static std::atomic<unsigned long long> l1_done[8];
                auto go = [&](auto kern) -> cudaError_t {
                    const cudaError_t el = dm_prefer_l1(reinterpret_cast<const void*>(kern), l1_done[2 * (shape - 7) + comp]);
                    if (el == cudaSuccess) kern<<<(unsigned)blocks, LV_THREADS, 0, st>>>(B, l, lam);
                    return el;
                };
                if (shape == 7) e = comp ? go(k_level_rows_b<true, 32>) : go(k_level_rows_b<false, 32>);
                else if (shape == 8) e = comp ? go(k_level_rows_b<true, 16>) : go(k_level_rows_b<false, 16>);
                else if (shape == 9) e = comp ? go(k_level_rows_b<true, 8>) : go(k_level_rows_b<false, 8>);
                else e = comp ? go(k_level_rows_b<true, 4>) : go(k_level_rows_b<false, 4>);
            } else {
                auto launch = [&](auto kern, int TH, int NR) -> cudaError_t {
                    const int kidf = (((2 * TH + 1) * KW + 31) / 32) * 32;     // LevelTile<TH>::KIDF
                    const size_t smem = (size_t)(NR * 2 * kidf + (2 * TH + 1) * AWP) * sizeof(float) + 128;
                    const int nt = TH == 16 ? level_threads<16>() : (TH == 8 ? level_threads<8>() : level_threads<4>());
                    // (per kernel: this lambda has one instance, the kernels being of one type)
                    static std::atomic<unsigned long long> done[6][2];
                    cudaError_t ea = dm_smem_opt_in(reinterpret_cast<const void*>(kern), (int)smem, done[shape - 1][comp]);
                    if (ea != cudaSuccess) return ea;
                    kern<<<(unsigned)blocks, nt, smem, st>>>(B, l, lam);
                    return cudaSuccess;
                };
                switch (shape) {
                    case 1: e = comp ? launch(k_level_sweep_b<true, 16, 2>, 16, 2) : launch(k_level_sweep_b<false, 16, 2>, 16, 2); break;
                    case 2: e = comp ? launch(k_level_sweep_b<true, 16, 3>, 16, 3) : launch(k_level_sweep_b<false, 16, 3>, 16, 3); break;
                    case 3: e = comp ? launch(k_level_sweep_b<true, 8, 2>, 8, 2) : launch(k_level_sweep_b<false, 8, 2>, 8, 2); break;
                    case 4: e = comp ? launch(k_level_sweep_b<true, 8, 3>, 8, 3) : launch(k_level_sweep_b<false, 8, 3>, 8, 3); break;
                    case 5: e = comp ? launch(k_level_sweep_b<true, 4, 2>, 4, 2) : launch(k_level_sweep_b<false, 4, 2>, 4, 2); break;
                    default: e = comp ? launch(k_level_sweep_b<true, 4, 3>, 4, 3) : launch(k_level_sweep_b<false, 4, 3>, 4, 3); break;
                }
            }
            if (e != cudaSuccess) return e;
            launches++;
        }
    }
    dm_count_launches(launches);
    return cudaGetLastError();
}
