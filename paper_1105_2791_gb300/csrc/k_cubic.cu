// Pixel-space kernels of the modal projection (Eq. bbispect with the linear term of
// Eq. bispectrumest), the Monte Carlo pair means, and the pixel part of the adjoint.
//
//   cubic     C_prs = sum_x W_x M_p M_r M_s                      (p <= r <= s)
//   linear    G_{(ab),c} = sum_x W_x <M_a M_b>_x M_c             (all pairs, all c)
//   beta_prs  = C_prs - (G_{(pr),s} + G_{(ps),r} + G_{(rs),p})
//   pairs     S_{(ab)}(x) += sum_b M_a M_b   (mean over simulations, FP64 sums)
//   adjoint   U_t(x) = 3 W_x sum_{a,b} h_tab (M_a M_b - <M_a M_b>_x)
#include "modal_internal.cuh"

#include "tc_common.cuh"
#include "tma_map.cuh"

#include <algorithm>

namespace modal {

// ---------------------------------------------------------------- cubic term
// C_prs = sum_x (W_x M_p M_r)(x) M_s(x), p <= r <= s, of every map over its pixel ranges
// (units: one map, one range of px_per_cta pixels).
//
// Modes in blocks of four: a box is a block triple bp <= br <= bs, that is up to 4 x 4 x 4
// coefficients, in four shapes (all blocks different, bp = br, br = bs, all equal: 64, 40, 40 and
// 20 coefficients) and, up to 10 modes, as many again for a last block of at most two modes.  A
// warp owns one box; a lane owns one of 16 pixel classes of one of two units (the half-warps), reads its pixel's 4 to 12 map values and W from shared memory, forms
// the products W M_p M_r of its box in registers and accumulates in packed FP32 pairs over p
// (32, 24, 20 or 13 FFMA2 per pixel).  The pair products are thus formed by the warps that use
// them, at a quarter of the multiply-adds they feed, instead of being written to a panel in
// shared memory and read back: that panel's traffic (640 bytes in and 1152 out per pixel at 16
// modes) was the bound.  Two sums per coefficient (8 pixels of a stage, then the stages) take 128
// registers, so ten warps fill an SM: 16 modes (20 boxes) go as two CTAs per pair of units.
// Maps and W stream through four stages of CUB_TX pixels: a producer thread issues four tiled
// copies per stage (copies by all threads behind a CTA barrier per stage cost 0.2 of the time in
// barriers, one bulk copy per row more than that in issue).  Every coefficient is the same chain of operations whatever the grid:
// per lane class the stages' 8-pixel sums in order, then the 16 classes in order.
// 16 modes, l_max = 1000, 16 maps: 2.34 -> 1.54 ms (34.7 TF/s useful, 0.44 of the measured FP32
// rate; the FMA pipe is busy 0.66 of the time); 10 modes, l_max = 500, 64 maps: 1.17 -> 0.72 ms.
constexpr int CUB_TX = 128;                 // pixels per stage
constexpr int CUB_LANES = 16;               // pixel classes
constexpr int CUB_ROW = CUB_TX + 16;        // floats per mode row of a unit: the second unit's pixels start at 16
constexpr int CUB_WROW = 160;               // the same for W, to a multiple of 128 bytes
constexpr int CUB_STAGES = 4;
constexpr int CUB_RED = 65;                 // floats per (box, class) in the final sums

__device__ __forceinline__ void named_arrive(int id, int n) { asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory"); }
struct CubicJob {
    double* partial;
    int64_t npix, ppc;                      // ppc: pixels per range, a multiple of CUB_TX
    int nctas;                              // ranges per map
    int64_t nunits;                         // maps x ranges
};
// The job's maps as rows (map, mode) of npix, and W as one row; a copy is P rows (or one) of
// CUB_ROW pixels.
struct CubicTiles {
    CUtensorMap maps, W;
};
struct CubicJobs {
    CubicTiles tiles[CUBIC_MAX_JOBS];
    CubicJob job[CUBIC_MAX_JOBS];
    int64_t item_end[CUBIC_MAX_JOBS];       // cumulative item counts (an item: two units, one group of boxes)
    int n;
};

// The boxes of P modes: groups of at most CUBIC_BOXES codes (shape | bp << 2 | br << 4 | bs << 6 |
// half << 8: bs is a last block of at most two modes), box i of a group on warp i.
struct CubicShape {
    int P, nb, ngroups, nbox, n_max;        // nbox: boxes per group
    const int* boxes;                       // [ngroups][nbox]
    const int* mode_of;                     // [P][P][P]
};

// SHAPE: 0 all blocks different, 1 bp = br, 2 br = bs, 3 all equal; + 4: bs holds only two modes.
// The coefficients of a box's (r, s) and p pair that a shape holds:
template <int SHAPE>
__host__ __device__ constexpr bool cub_used(int r, int s, int pp) {
    return ((SHAPE & 1) == 0 || 2 * pp <= r) && ((SHAPE & 2) == 0 || s >= r) && ((SHAPE & 4) == 0 || s < 2);
}
// the pair products u(r, pp) that any of its coefficients needs
template <int SHAPE>
__host__ __device__ constexpr bool cub_product(int r, int pp) {
    return cub_used<SHAPE>(r, 0, pp) || cub_used<SHAPE>(r, 1, pp) || cub_used<SHAPE>(r, 2, pp) || cub_used<SHAPE>(r, 3, pp);
}

template <int SHAPE>
struct CubValues {
    float p[4], r[4], s[4], w;
    __device__ __forceinline__ void load(const float* sp, const float* sr, const float* ss, const float* sw, int off) {
        constexpr int NS = (SHAPE & 4) ? 2 : 4;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (i < NS || (SHAPE & 3) != 3) p[i] = sp[i * CUB_ROW + off];
            if (!(SHAPE & 1) && (i < NS || !(SHAPE & 2))) r[i] = sr[i * CUB_ROW + off];
            if (!(SHAPE & 2) && i < NS) s[i] = ss[i * CUB_ROW + off];
        }
        w = sw[off];
    }
    __device__ __forceinline__ float rv(int i) const { return (SHAPE & 1) ? p[i] : r[i]; }
    __device__ __forceinline__ float sv(int i) const { return (SHAPE & 2) ? rv(i) : s[i]; }
};

template <int SHAPE, bool FIRST>
__device__ __forceinline__ void cub_pixel(const CubValues<SHAPE>& v, float2 (&t)[4][4][2]) {
    const float2 w2 = make_float2(v.w, v.w);
#pragma unroll
    for (int pp = 0; pp < 2; ++pp) {
        if (!cub_product<SHAPE>(0, pp) && !cub_product<SHAPE>(1, pp) && !cub_product<SHAPE>(2, pp) && !cub_product<SHAPE>(3, pp)) continue;
        const float2 wm = __fmul2_rn(w2, make_float2(v.p[2 * pp], v.p[2 * pp + 1]));
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            if (!cub_product<SHAPE>(r, pp)) continue;
            const float2 u = __fmul2_rn(wm, make_float2(v.rv(r), v.rv(r)));   // W M_p M_r of two p
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                if (!cub_used<SHAPE>(r, s, pp)) continue;
                const float2 s2 = make_float2(v.sv(s), v.sv(s));
                t[r][s][pp] = FIRST ? __fmul2_rn(u, s2) : __ffma2_rn(u, s2, t[r][s][pp]);
            }
        }
    }
}

// The two units of one item as a CTA sees them.
struct CubicUnits {
    int x[2], y[2];                         // the unit's first pixel (npix: none) and first row of its map
    double* out[2];                         // the unit's partial sums
    int nch;                                // stages
};

// Floats of a stage: [unit][4 nb modes][CUB_ROW], then [unit] W rows.
__host__ __device__ inline int cub_stage(int nb) { return 2 * (4 * nb * CUB_ROW + CUB_WROW); }

// Stage barriers behind the stages' data: full (the producer's copies have landed) and empty (every
// box warp has read the stage); `it` counts the stages of the CTA, so a persistent caller's
// barriers run on from item to item.
struct CubicPipe {
    uint64_t *full, *empty;                 // [CUB_STAGES] each
    volatile int* abort_flag;
    int* err;
};

// The producer (one thread): four tiled copies per stage.  The second unit's tile starts 16
// pixels early, which puts its pixels half a bank row from the first's; what lies outside the
// map (also a unit that has run out of pixels: only a map's last range is shorter) reads as zero,
// and the rows of modes past P are never written: no coefficient that is kept depends on them.
__device__ __forceinline__ void cub_produce(float* smem, const CubicPipe& pipe, const CubicTiles& tl, const CubicUnits& un, int P,
                                            int nb, uint32_t& it) {
    for (int k = 0; k < un.nch; ++k, ++it) {
        const int s = it % CUB_STAGES;
        if (!mbar_wait(&pipe.empty[s], ((it / CUB_STAGES) & 1) ^ 1, pipe.abort_flag, pipe.err)) return;
        float* st = smem + s * cub_stage(nb);
        mbar_arrive_expect_tx(&pipe.full[s], 2 * (P + 1) * CUB_ROW * 4);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int x = un.x[h] + k * CUB_TX - 16 * h;
            tma_load_2d(st + h * 4 * nb * CUB_ROW, &tl.maps, x, un.y[h], &pipe.full[s]);
            tma_load_2d(st + 8 * nb * CUB_ROW + h * CUB_WROW, &tl.W, x, 0, &pipe.full[s]);
        }
    }
}

template <int SHAPE, bool LOOPED>
__device__ __forceinline__ void cubic_box(float* smem, const CubicPipe& pipe, const CubicUnits& un, const CubicShape& sh,
                                          const int* boxes, int code, uint32_t& it) {
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32, half = lane / CUB_LANES, cl = lane % CUB_LANES;
    const int nthr = sh.nbox * 32, nb = sh.nb, P = sh.P;
    const int op = 4 * ((code >> 2) & 3) * CUB_ROW, orr = 4 * ((code >> 4) & 3) * CUB_ROW, os = 4 * ((code >> 6) & 3) * CUB_ROW;
    float2 acc[4][4][2], t[4][4][2];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int s = 0; s < 4; ++s)
#pragma unroll
            for (int pp = 0; pp < 2; ++pp) acc[r][s][pp] = make_float2(0.f, 0.f);
    for (int k = 0; k < un.nch; ++k, ++it) {
        const int sg = it % CUB_STAGES;
        if (!__all_sync(0xffffffffu, mbar_wait(&pipe.full[sg], (it / CUB_STAGES) & 1, pipe.abort_flag, pipe.err))) break;
        const float* st = smem + sg * cub_stage(nb) + 16 * half + cl;
        const float* sm = st + half * 4 * nb * CUB_ROW;
        const float *sp = sm + op, *sr = sm + orr, *ss = sm + os, *sw = st + 8 * nb * CUB_ROW + half * CUB_WROW;
        // two pixels per turn, each one's values read while the other is summed
        CubValues<SHAPE> va, vb;
        va.load(sp, sr, ss, sw, 0);
        vb.load(sp, sr, ss, sw, CUB_LANES);
        cub_pixel<SHAPE, true>(va, t);
        va.load(sp, sr, ss, sw, 2 * CUB_LANES);
        cub_pixel<SHAPE, false>(vb, t);
        auto turn = [&](int i) {
            vb.load(sp, sr, ss, sw, (i + 1) * CUB_LANES);
            cub_pixel<SHAPE, false>(va, t);
            va.load(sp, sr, ss, sw, min(i + 2, CUB_TX / CUB_LANES - 1) * CUB_LANES);
            cub_pixel<SHAPE, false>(vb, t);
        };
        if constexpr (LOOPED) {
#pragma unroll 1
            for (int i = 2; i < CUB_TX / CUB_LANES; i += 2) turn(i);
        } else {
#pragma unroll
            for (int i = 2; i < CUB_TX / CUB_LANES; i += 2) turn(i);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&pipe.empty[sg]);
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int s = 0; s < 4; ++s)
#pragma unroll
                for (int pp = 0; pp < 2; ++pp)
                    if (cub_used<SHAPE>(r, s, pp)) acc[r][s][pp] = __fadd2_rn(acc[r][s][pp], t[r][s][pp]);
    }
    // the classes' sums: [unit][nbox][CUB_LANES][CUB_RED], entry (r, s, p)
    float* red = smem + CUB_STAGES * cub_stage(nb);
    named_sync(1, nthr);                                     // the sums of the item before have been read
    float* own = red + ((half * sh.nbox + warp) * CUB_LANES + cl) * CUB_RED;
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int s = 0; s < 4; ++s)
#pragma unroll
            for (int pp = 0; pp < 2; ++pp)
                if (cub_used<SHAPE>(r, s, pp)) {
                    own[(r * 4 + s) * 4 + 2 * pp] = acc[r][s][pp].x;
                    own[(r * 4 + s) * 4 + 2 * pp + 1] = acc[r][s][pp].y;
                }
    named_sync(1, nthr);
    for (int i = threadIdx.x; i < 2 * sh.nbox * 64; i += nthr) {
        const int h = i >= sh.nbox * 64, bx = i / 64 - h * sh.nbox, e = i % 64, c = boxes[bx];
        const int p = 4 * ((c >> 2) & 3) + e % 4, r = 4 * ((c >> 4) & 3) + e / 16, s = 4 * ((c >> 6) & 3) + (e / 4) % 4;
        if (p > r || r > s || s >= P || !un.out[h]) continue;
        float v = 0.f;
#pragma unroll
        for (int ln = 0; ln < CUB_LANES; ++ln) v += red[((h * sh.nbox + bx) * CUB_LANES + ln) * CUB_RED + e];
        un.out[h][sh.mode_of[(p * P + r) * P + s]] = (double)v;
    }
}

// Units u0 and u0 + 1 of a job (the second may not exist).
__device__ __forceinline__ CubicUnits cub_units(const CubicJob& jb, int P, int n_max, int64_t u0) {
    CubicUnits un;
    un.nch = 0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int64_t u = u0 + h;
        const bool valid = u < jb.nunits;
        const int64_t b = valid ? u / jb.nctas : 0, cta = valid ? u % jb.nctas : 0;
        const int64_t xb = valid ? min(jb.npix, cta * jb.ppc) : jb.npix, xe = min(jb.npix, xb + jb.ppc);
        un.x[h] = (int)xb;
        un.y[h] = (int)(b * P);
        un.out[h] = valid ? jb.partial + u * n_max : nullptr;
        un.nch = max(un.nch, (int)((xe - xb + CUB_TX - 1) / CUB_TX));
    }
    return un;
}

// The tiled copies want 128-byte aligned stages.
__device__ __forceinline__ float* cub_align(float* raw) { return raw + ((128 - (smem_u32(raw) & 127)) & 127) / 4; }

constexpr int CUB_THREADS = (CUBIC_BOXES + 1) * 32;

// One CTA's barriers, producer and boxes; run() takes them through one item.  HALF: the last block
// of modes holds at most two.  The warps of a CTA run as many different box bodies as there are
// shapes, so the instruction cache decides how far the pixel loop is unrolled: with four shapes
// all 8 pixels of a stage (16 modes, l_max = 1000, 16 maps: 1.51 ms, 1.63 looped), with the
// eight that a half block brings (cubic_half) two at a time (10 modes, l_max = 500, 64 maps: 0.72
// ms looped, 1.05 unrolled, 0.91 with the last block treated as whole).
template <bool HALF>
struct CubicCta {
    float* smem;
    CubicPipe pipe;
    uint32_t it;
    __device__ __forceinline__ void run(const CubicTiles& tl, const CubicJob& jb, const CubicShape& sh, int64_t local) {
        const int warp = threadIdx.x / 32;
        const CubicUnits un = cub_units(jb, sh.P, sh.n_max, 2 * (local / sh.ngroups));
        if (warp == sh.nbox) {
            cub_produce(smem, pipe, tl, un, sh.P, sh.nb, it);
            return;
        }
        const int* boxes = sh.boxes + local % sh.ngroups * sh.nbox;
        const int code = boxes[warp];
        if constexpr (HALF) {
            switch ((code & 3) | (code >> 8) << 2) {
                case 0: cubic_box<0, true>(smem, pipe, un, sh, boxes, code, it); break;
                case 1: cubic_box<1, true>(smem, pipe, un, sh, boxes, code, it); break;
                case 2: cubic_box<2, true>(smem, pipe, un, sh, boxes, code, it); break;
                case 3: cubic_box<3, true>(smem, pipe, un, sh, boxes, code, it); break;
                case 4: cubic_box<4, true>(smem, pipe, un, sh, boxes, code, it); break;
                case 5: cubic_box<5, true>(smem, pipe, un, sh, boxes, code, it); break;
                case 6: cubic_box<6, true>(smem, pipe, un, sh, boxes, code, it); break;
                default: cubic_box<7, true>(smem, pipe, un, sh, boxes, code, it); break;
            }
        } else {
            switch (code & 3) {
                case 0: cubic_box<0, false>(smem, pipe, un, sh, boxes, code, it); break;
                case 1: cubic_box<1, false>(smem, pipe, un, sh, boxes, code, it); break;
                case 2: cubic_box<2, false>(smem, pipe, un, sh, boxes, code, it); break;
                default: cubic_box<3, false>(smem, pipe, un, sh, boxes, code, it); break;
            }
        }
    }
    // after a wait that gave up, the copies still in flight land before the CTA exits
    __device__ __forceinline__ void drain() {
        if (!*pipe.abort_flag) return;
        for (uint32_t k = it > CUB_STAGES ? it - CUB_STAGES : 0; k < it; ++k) {
            const long long t0 = clock64();
            while (!mbar_try_wait(&pipe.full[k % CUB_STAGES], (k / CUB_STAGES) & 1) && clock64() - t0 < TC_WAIT_CYCLES) {
            }
        }
    }
};

template <bool HALF>
__device__ __forceinline__ CubicCta<HALF> cubic_cta(float* raw, uint64_t* bars, int* abort_word, int nbox, int* err) {
    CubicCta<HALF> c = {cub_align(raw), {bars, bars + CUB_STAGES, abort_word, err}, 0};
    if (threadIdx.x == 0) {
        for (int s = 0; s < CUB_STAGES; ++s) {
            mbar_init(&c.pipe.full[s], 1);
            mbar_init(&c.pipe.empty[s], nbox);
        }
        *c.pipe.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    return c;
}

// One CTA per item (pair of units, group of boxes), the groups of a pair adjacent: they read the
// same maps.  (Persistent CTAs whose producer ran on into the next item measured no faster:
// 1.76 -> 1.87 ms for 64 maps of 16 modes at l_max = 500, the loop costs registers.)
template <bool HALF>
__global__ void __launch_bounds__(CUB_THREADS, 1) k_cubic(const __grid_constant__ CubicTiles tl, const __grid_constant__ CubicJob jb,
                                                        CubicShape sh, int* err) {
    extern __shared__ __align__(128) float cub_raw[];
    __shared__ uint64_t bars[2 * CUB_STAGES];
    __shared__ int abort_word;
    CubicCta<HALF> c = cubic_cta<HALF>(cub_raw, bars, &abort_word, sh.nbox, err);
    const bool producer = (int)threadIdx.x / 32 == sh.nbox;
    if (producer && threadIdx.x % 32 != 0) return;
    c.run(tl, jb, sh, blockIdx.x);
    if (producer) c.drain();
}

// The cubic sums of several plans (one pass of a mixed-l_max batch, the same P) as one
// persistent launch over items (job, pair of units, group), jobs in the order given (the host
// puts the plans with the longest items first); the units are those that each plan's own launch
// would compute, so the partial sums are identical.
template <bool HALF>
__global__ void __launch_bounds__(CUB_THREADS, 1) k_cubic_multi(const __grid_constant__ CubicJobs jobs, CubicShape sh, int* err) {
    extern __shared__ __align__(128) float cub_raw[];
    __shared__ uint64_t bars[2 * CUB_STAGES];
    __shared__ int abort_word;
    CubicCta<HALF> c = cubic_cta<HALF>(cub_raw, bars, &abort_word, sh.nbox, err);
    const bool producer = (int)threadIdx.x / 32 == sh.nbox;
    if (producer && threadIdx.x % 32 != 0) return;
    int j = 0;
    for (int64_t item = blockIdx.x; item < jobs.item_end[jobs.n - 1]; item += gridDim.x) {
        while (item >= jobs.item_end[j]) ++j;
        c.run(jobs.tiles[j], jobs.job[j], sh, item - (j > 0 ? jobs.item_end[j - 1] : 0));
    }
    if (producer) c.drain();
}

static size_t cubic_smem(const CubicShape& sh) {
    const size_t stages = (size_t)CUB_STAGES * cub_stage(sh.nb);
    const size_t red = (size_t)2 * sh.nbox * CUB_LANES * CUB_RED;
    return (stages + red) * sizeof(float) + 128;
}

static CubicShape cubic_shape(const Plan& pl) {
    CubicShape sh;
    sh.P = pl.P;
    sh.nb = (pl.P + 3) / 4;
    sh.ngroups = pl.cubic_groups;
    sh.nbox = pl.cubic_boxes;
    sh.n_max = pl.n_max;
    sh.boxes = pl.boxes;
    sh.mode_of = pl.mode_of;
    return sh;
}

static int64_t cubic_ppc(const Plan& pl) { return ((pl.npix + pl.cubic_ctas - 1) / pl.cubic_ctas + CUB_TX - 1) / CUB_TX * CUB_TX; }

// The tiled copies take 32-bit pixel coordinates, which run to one range past the map's end.
constexpr int64_t CUB_COORDS = (int64_t)1 << 31;
bool cubic_one_launch(const Plan& pl) { return pl.npix + cubic_ppc(pl) < CUB_COORDS; }

// B maps, their first `npix` pixels in `nctas` ranges
static CubicJob cubic_job(const Plan& pl, int B, int64_t npix, int nctas, double* partial) {
    CubicJob jb;
    jb.partial = partial;
    jb.npix = npix;
    jb.ppc = cubic_ppc(pl);
    jb.nctas = nctas;
    jb.nunits = (int64_t)B * nctas;
    return jb;
}

static cudaError_t cubic_tiles(const Plan& pl, const float* maps, const float* W, int B, int64_t npix, CubicTiles* tl) {
    const cuuint64_t dims[2] = {(cuuint64_t)npix, (cuuint64_t)B * pl.P}, wdims[2] = {(cuuint64_t)npix, 1};
    const cuuint64_t strides[1] = {(cuuint64_t)pl.npix * sizeof(float)};
    const cuuint32_t box[2] = {CUB_ROW, (cuuint32_t)pl.P}, wbox[2] = {CUB_ROW, 1};
    const cudaError_t e = tma_map_f32(&tl->maps, maps, 2, dims, strides, box);
    return e != cudaSuccess ? e : tma_map_f32(&tl->W, W, 2, wdims, strides, wbox);
}

cudaError_t launch_cubic_multi(Plan* const* plans, const float* const* maps, const int* B, int n, cudaStream_t st) {
    if (n < 1 || n > CUBIC_MAX_JOBS) return cudaErrorInvalidValue;
    const Plan& p0 = *plans[0];
    const CubicShape sh = cubic_shape(p0);
    CubicJobs jobs = {};
    int64_t total = 0;
    for (int i = 0; i < n; ++i) {
        const Plan& pl = *plans[i];
        if (pl.P != p0.P || B[i] < 1 || B[i] > pl.chunk || !cubic_one_launch(pl)) return cudaErrorInvalidValue;
        jobs.job[i] = cubic_job(pl, B[i], pl.npix, pl.cubic_ctas, pl.partial);
        const cudaError_t e = cubic_tiles(pl, maps[i], pl.W, B[i], pl.npix, &jobs.tiles[i]);
        if (e != cudaSuccess) return e;
        total += (jobs.job[i].nunits + 1) / 2 * sh.ngroups;
        jobs.item_end[i] = total;
    }
    jobs.n = n;
    const size_t smem = cubic_smem(sh);
    auto kernel = cubic_half(p0.P) ? k_cubic_multi<true> : k_cubic_multi<false>;
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    // CTAs: as many as the register file holds (twelve warps per SM)
    const int64_t grid = std::min(total, (int64_t)std::max(p0.nsm, 1) * std::max(1, 12 / (sh.nbox + 1)));
    kernel<<<(unsigned)grid, (sh.nbox + 1) * 32, smem, st>>>(jobs, sh, p0.d_err);
    note_launch(p0);
    return cudaGetLastError();
}

static cudaError_t cubic_launch(const Plan& pl, const CubicTiles& tl, const CubicJob& jb, cudaStream_t st) {
    const CubicShape sh = cubic_shape(pl);
    const size_t smem = cubic_smem(sh);
    auto kernel = cubic_half(pl.P) ? k_cubic<true> : k_cubic<false>;
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const int64_t items = (jb.nunits + 1) / 2 * sh.ngroups;
    kernel<<<(unsigned)items, (sh.nbox + 1) * 32, smem, st>>>(tl, jb, sh, pl.d_err);
    note_launch(pl);
    return cudaGetLastError();
}

cudaError_t launch_cubic(Plan& pl, const float* maps, int B, double* partial, cudaStream_t st) {
    if (B == 0) return cudaSuccess;
    CubicTiles tl;
    if (cubic_one_launch(pl)) {
        const cudaError_t e = cubic_tiles(pl, maps, pl.W, B, pl.npix, &tl);
        return e != cudaSuccess ? e : cubic_launch(pl, tl, cubic_job(pl, B, pl.npix, pl.cubic_ctas, partial), st);
    }
    // larger maps one by one, as many whole ranges at a time as the coordinates reach; ranges past
    // the last pixel (their sums are zero) go with the last part
    const int64_t ppc = cubic_ppc(pl);
    const int per = (int)((CUB_COORDS - 1) / ppc) - 1, full = (int)((pl.npix + ppc - 1) / ppc);
    if (per < 1) return cudaErrorInvalidValue;
    for (int b = 0; b < B; ++b)
        for (int r0 = 0; r0 < full; r0 += per) {
            const bool last = r0 + per >= full;
            const int64_t x0 = r0 * ppc, n = last ? pl.npix - x0 : per * ppc;
            cudaError_t e = cubic_tiles(pl, maps + (int64_t)b * pl.P * pl.npix + x0, pl.W + x0, 1, n, &tl);
            if (e == cudaSuccess)
                e = cubic_launch(pl, tl, cubic_job(pl, 1, n, last ? pl.cubic_ctas - r0 : per,
                                                   partial + ((int64_t)b * pl.cubic_ctas + r0) * pl.n_max), st);
            if (e != cudaSuccess) return e;
        }
    return cudaSuccess;
}

// ---------------------------------------------------------------- linear term GEMM
// out[z][row][col] = sum_{x in split z} (W_x <pair row>_x) * maps[col][x],
// rows = pairs (lexicographic), cols = (map, c) = b * P + c, K = pixels, split over gridDim.z.
// Every output of a split is one chain of FMAs over its pixels in order, whatever the tile, so
// a small problem is bound by that chain and by how many SMs its few outputs reach, a large
// one by FP32 arithmetic.  Panel and maps are contiguous along K in memory and stay so in
// shared memory: a ring of ST stages of BK pixels filled by cp.async, each thread multiplying
// the panel pieces that it copied by W once they are there.  A thread reads 4 pixels (16
// bytes) of its TL rows and TC columns at a time; the padding of 4 floats per row puts the
// rows on different banks.  Synchronous staging through registers, one tile of 64 x 64 for
// every size, took (us, linear term of one call) 290 at l_max = 32 with 6 modes and one map,
// 2467 at l_max = 250 with 8 modes and 21 maps; now 23 and 141.
__device__ __forceinline__ void lg_cp16(float* dst, const float* src, int bytes) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(bytes) : "memory");
}

template <int BM, int BN, int BK, int ST>
constexpr size_t lg_smem() { return (size_t)ST * (BM + BN) * (BK + 4) * sizeof(float); }

template <int BM, int BN, int TL, int TC, int BK, int ST>
__global__ void __launch_bounds__((BM / TL) * (BN / TC))
k_linear_gemm(int nrows, int ncols, int64_t npix, int64_t kchunk, const float* __restrict__ panel,
              const float* __restrict__ W, const float* __restrict__ maps, double* __restrict__ out) {
    constexpr int NT = (BM / TL) * (BN / TC), S = BK + 4, Q = BK / 4;
    constexpr int STAGE = (BM + BN) * S;
    constexpr int NR = BM / TL, NCG = BN / TC;               // thread groups along rows and columns
    constexpr int RS = NT / Q;                               // rows between a thread's copies
    constexpr int NA = BM / RS, NB = BN / RS;                // its 16-byte pieces of the panel and of the maps per stage
    static_assert(NT % Q == 0 && BM % RS == 0 && BN % RS == 0 && NR % 4 == 0 && NCG % 4 == 0, "tile shape");
    extern __shared__ __align__(16) float lg_sm[];
    const int tid = threadIdx.x;
    // half a warp holds 4 x 4 threads, so that its 16-byte reads touch 4 rows and 4 columns
    const int rg = tid % 4 + 4 * ((tid / 16) % (NR / 4)), cg = (tid / 4) % 4 + 4 * (tid / (4 * NR));
    const int r0 = blockIdx.x * BM, c0 = blockIdx.y * BN;    // rows rg + NR i, columns cg + NCG k
    const int64_t k_begin = (int64_t)blockIdx.z * kchunk;
    const int64_t k_end = min(npix, k_begin + kchunk);       // a multiple of 16, as npix and kchunk are
    const int nk = k_end > k_begin ? (int)((k_end - k_begin + BK - 1) / BK) : 0;
    // this thread copies piece q of rows lr + RS u; a piece past the last pixel, row or column is zero
    const int q = tid % Q, lr = tid / Q;
    const float* pa = panel + (int64_t)(r0 + lr) * npix + k_begin + 4 * q;
    const float* pb = maps + (int64_t)(c0 + lr) * npix + k_begin + 4 * q;
    const float* pw = W + k_begin + 4 * q;
    const int64_t step = (int64_t)RS * npix;
    auto issue = [&](int k) {
        if (k < nk) {
            const int off = k * BK;
            const bool in = k_begin + off + 4 * q < k_end;
            float* st = lg_sm + (k % ST) * STAGE + lr * S + 4 * q;
#pragma unroll
            for (int u = 0; u < NA; ++u) {
                const bool ok = in && r0 + lr + RS * u < nrows;
                lg_cp16(st + RS * u * S, ok ? pa + off + u * step : panel, ok ? 16 : 0);
            }
#pragma unroll
            for (int u = 0; u < NB; ++u) {
                const bool ok = in && c0 + lr + RS * u < ncols;
                lg_cp16(st + (BM + RS * u) * S, ok ? pb + off + u * step : maps, ok ? 16 : 0);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    auto weight = [&](int k) {
        return k < nk && k_begin + (int64_t)k * BK + 4 * q < k_end ? __ldg(reinterpret_cast<const float4*>(pw + k * BK))
                                                                   : make_float4(0.f, 0.f, 0.f, 0.f);
    };
    float acc[TL][TC];
#pragma unroll
    for (int i = 0; i < TL; ++i)
#pragma unroll
        for (int j = 0; j < TC; ++j) acc[i][j] = 0.f;
#pragma unroll
    for (int k = 0; k < ST - 1; ++k) issue(k);
    float4 w = weight(0);
    for (int k = 0; k < nk; ++k) {
        const float4 wn = weight(k + 1);
        asm volatile("cp.async.wait_group %0;" ::"n"(ST - 2) : "memory");
        // the panel's pieces that this thread copied, times W
        float* own = lg_sm + (k % ST) * STAGE + lr * S + 4 * q;
#pragma unroll
        for (int u = 0; u < NA; ++u) {
            float4* v = reinterpret_cast<float4*>(own + RS * u * S);
            const float4 x = *v;
            *v = make_float4(x.x * w.x, x.y * w.y, x.z * w.z, x.w * w.w);
        }
        w = wn;
        __syncthreads();                                     // stage k is ready, stage k - 1 is free
        issue(k + ST - 1);
        const float* sa = lg_sm + (k % ST) * STAGE + rg * S;
        const float* sb = lg_sm + (k % ST) * STAGE + (BM + cg) * S;
        constexpr int UNROLL = TL * TC >= 32 ? 2 : (TL * TC >= 16 ? 4 : 8);
#pragma unroll UNROLL
        for (int p = 0; p < Q; ++p) {
            float4 a[TL], b[TC];
#pragma unroll
            for (int i = 0; i < TL; ++i) a[i] = *reinterpret_cast<const float4*>(sa + i * NR * S + 4 * p);
#pragma unroll
            for (int j = 0; j < TC; ++j) b[j] = *reinterpret_cast<const float4*>(sb + j * NCG * S + 4 * p);
#pragma unroll
            for (int i = 0; i < TL; ++i)
#pragma unroll
                for (int j = 0; j < TC; ++j) acc[i][j] = fmaf(a[i].x, b[j].x, acc[i][j]);
#pragma unroll
            for (int i = 0; i < TL; ++i)
#pragma unroll
                for (int j = 0; j < TC; ++j) acc[i][j] = fmaf(a[i].y, b[j].y, acc[i][j]);
#pragma unroll
            for (int i = 0; i < TL; ++i)
#pragma unroll
                for (int j = 0; j < TC; ++j) acc[i][j] = fmaf(a[i].z, b[j].z, acc[i][j]);
#pragma unroll
            for (int i = 0; i < TL; ++i)
#pragma unroll
                for (int j = 0; j < TC; ++j) acc[i][j] = fmaf(a[i].w, b[j].w, acc[i][j]);
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
#pragma unroll
    for (int i = 0; i < TL; ++i)
#pragma unroll
        for (int j = 0; j < TC; ++j) {
            const int r = r0 + rg + NR * i, c = c0 + cg + NCG * j;
            if (r < nrows && c < ncols) out[((int64_t)blockIdx.z * nrows + r) * ncols + c] = (double)acc[i][j];
        }
}

template <int BM, int BN, int TL, int TC, int BK, int ST>
static cudaError_t linear_gemm_launch(Plan& pl, const float* maps, int ncols, int64_t kchunk, double* partial,
                                      cudaStream_t st) {
    constexpr size_t smem = lg_smem<BM, BN, BK, ST>();
    auto kernel = k_linear_gemm<BM, BN, TL, TC, BK, ST>;
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    const dim3 grid((pl.n_pair + BM - 1) / BM, (ncols + BN - 1) / BN, pl.lin_ksplit);
    kernel<<<grid, (BM / TL) * (BN / TC), smem, st>>>(pl.n_pair, ncols, pl.npix, kchunk, pl.pair_mean, pl.W, maps, partial);
    note_launch(pl);
    return cudaGetLastError();
}

// The same sums where the outputs are few: one compute warp per block, which does nothing but read
// and accumulate, and one copy warp, which keeps LC_ST - 1 stages in flight and multiplies the
// panel's pieces by W.  (With copies, weights and sums in the same warps a chain advanced by one
// pixel in 20 clocks; here in 8.7 with one block per SM.)  A thread holds 2 rows x 2 columns: a
// warp's 16-byte read occupies the shared-memory return path for four clocks whatever its lanes
// share, so several blocks on an SM are bound by that path; blocks of 8 rows waste little of 21,
// 36 or 55 pairs there (21 maps, l_max = 250, 8 modes: 183 us with 16 x 16 blocks, 141; 2 x 4
// outputs per thread, with fewer bytes per output and fewer warps, 179).
constexpr int LC_BK = 128, LC_ST = 4, LC_S = LC_BK + 4, LC_Q = LC_BK / 4, LC_R = 8;
constexpr int LC_C = 16;                    // columns per block
constexpr size_t LC_SMEM = (size_t)LC_ST * (LC_R + LC_C) * LC_S * sizeof(float);

__global__ void __launch_bounds__(64)
k_linear_chain(int nrows, int ncols, int64_t npix, int64_t kchunk, const float* __restrict__ panel,
               const float* __restrict__ W, const float* __restrict__ maps, double* __restrict__ out) {
    constexpr int LC_STAGE = (LC_R + LC_C) * LC_S;
    constexpr int TC = LC_C / 8, G = 4;                      // columns per thread, pieces per read-ahead group
    extern __shared__ __align__(16) float lg_sm[];
    const int r0 = blockIdx.x * LC_R, c0 = blockIdx.y * LC_C;
    const int64_t k_begin = (int64_t)blockIdx.z * kchunk;
    const int64_t k_end = min(npix, k_begin + kchunk);
    const int nk = k_end > k_begin ? (int)((k_end - k_begin + LC_BK - 1) / LC_BK) : 0;
    // blocks alternate which warp computes: two blocks' compute warps then sit on different sub-partitions
    const bool copies = (threadIdx.x / 32 ^ (blockIdx.x + blockIdx.y + blockIdx.z)) & 1;
    const int lane = threadIdx.x % 32;
    // barriers: 1 + s: stage s is filled; 1 + LC_ST + s: stage s has been read
    if (copies) {
        constexpr int RS = 32 / LC_Q, NA = LC_R / RS, NB = LC_C / RS;
        const int q = lane % LC_Q, lr = lane / LC_Q;         // pieces q of rows lr + RS u
        const float* pa = panel + (int64_t)(r0 + lr) * npix + k_begin + 4 * q;
        const float* pb = maps + (int64_t)(c0 + lr) * npix + k_begin + 4 * q;
        const float* pw = W + k_begin + 4 * q;
        const int64_t step = (int64_t)RS * npix;
        float4 w[LC_ST];
        auto issue = [&](int k, float4& wk) {
            wk = make_float4(0.f, 0.f, 0.f, 0.f);
            if (k < nk) {
                const int off = k * LC_BK;
                const bool in = k_begin + off + 4 * q < k_end;
                float* st = lg_sm + (k % LC_ST) * LC_STAGE + lr * LC_S + 4 * q;
#pragma unroll
                for (int u = 0; u < NA; ++u) {
                    const bool ok = in && r0 + lr + RS * u < nrows;
                    lg_cp16(st + RS * u * LC_S, ok ? pa + off + u * step : panel, ok ? 16 : 0);
                }
#pragma unroll
                for (int u = 0; u < NB; ++u) {
                    const bool ok = in && c0 + lr + RS * u < ncols;
                    lg_cp16(st + (LC_R + RS * u) * LC_S, ok ? pb + off + u * step : maps, ok ? 16 : 0);
                }
                if (in) wk = __ldg(reinterpret_cast<const float4*>(pw + off));
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
#pragma unroll
        for (int k = 0; k < LC_ST - 1; ++k) issue(k, w[k]);
        for (int k0 = 0; k0 < nk; k0 += LC_ST) {
#pragma unroll
            for (int s = 0; s < LC_ST; ++s) {                // stage s holds step k
                const int k = k0 + s;
                if (k >= nk) break;
                asm volatile("cp.async.wait_group %0;" ::"n"(LC_ST - 2) : "memory");
                float* own = lg_sm + s * LC_STAGE + lr * LC_S + 4 * q;
#pragma unroll
                for (int u = 0; u < NA; ++u) {
                    float4* v = reinterpret_cast<float4*>(own + RS * u * LC_S);
                    const float4 x = *v;
                    *v = make_float4(x.x * w[s].x, x.y * w[s].y, x.z * w[s].z, x.w * w[s].w);
                }
                __threadfence_block();
                named_arrive(1 + s, 64);
                const int kn = k + LC_ST - 1;                // goes where step k - 1 was
                if (k >= 1 && kn < nk) named_sync(1 + LC_ST + (s + LC_ST - 1) % LC_ST, 64);
                issue(kn, w[(s + LC_ST - 1) % LC_ST]);
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        return;
    }
    const int rg = lane % 4, cg = lane / 4;                  // rows rg, rg + 4; columns cg + 8 i
    float acc[2][TC];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < TC; ++j) acc[i][j] = 0.f;
    for (int k = 0; k < nk; ++k) {
        const int s = k % LC_ST;
        named_sync(1 + s, 64);
        const float* sa = lg_sm + s * LC_STAGE + rg * LC_S;
        const float* sb = lg_sm + s * LC_STAGE + (LC_R + cg) * LC_S;
        // the next group's reads are issued before this group's sums
        float4 a[2][G][2], b[2][G][TC];
        auto read = [&](int h, int g) {
#pragma unroll
            for (int p = 0; p < G; ++p) {
#pragma unroll
                for (int i = 0; i < 2; ++i) a[h][p][i] = *reinterpret_cast<const float4*>(sa + 4 * i * LC_S + 4 * (g * G + p));
#pragma unroll
                for (int i = 0; i < TC; ++i) b[h][p][i] = *reinterpret_cast<const float4*>(sb + 8 * i * LC_S + 4 * (g * G + p));
            }
        };
        read(0, 0);
#pragma unroll
        for (int g = 0; g < LC_Q / G; ++g) {
            const int h = g & 1;
            if (g + 1 < LC_Q / G) read(h ^ 1, g + 1);
#pragma unroll
            for (int p = 0; p < G; ++p) {
#pragma unroll
                for (int i = 0; i < 2; ++i)
#pragma unroll
                    for (int j = 0; j < TC; ++j) acc[i][j] = fmaf(a[h][p][i].x, b[h][p][j].x, acc[i][j]);
#pragma unroll
                for (int i = 0; i < 2; ++i)
#pragma unroll
                    for (int j = 0; j < TC; ++j) acc[i][j] = fmaf(a[h][p][i].y, b[h][p][j].y, acc[i][j]);
#pragma unroll
                for (int i = 0; i < 2; ++i)
#pragma unroll
                    for (int j = 0; j < TC; ++j) acc[i][j] = fmaf(a[h][p][i].z, b[h][p][j].z, acc[i][j]);
#pragma unroll
                for (int i = 0; i < 2; ++i)
#pragma unroll
                    for (int j = 0; j < TC; ++j) acc[i][j] = fmaf(a[h][p][i].w, b[h][p][j].w, acc[i][j]);
            }
        }
        if (k + LC_ST < nk) named_arrive(1 + LC_ST + s, 64);     // the copy of step k + LC_ST waits for this
    }
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < TC; ++j) {
            const int r = r0 + rg + 4 * i, c = c0 + cg + 8 * j;
            if (r < nrows && c < ncols) out[((int64_t)blockIdx.z * nrows + r) * ncols + c] = (double)acc[i][j];
        }
}

cudaError_t launch_linear_gemm(Plan& pl, const float* maps, int B, double* partial, cudaStream_t st) {
    if (B == 0) return cudaSuccess;
    const int ncols = B * pl.P;
    const int64_t kchunk = ((pl.npix + pl.lin_ksplit - 1) / pl.lin_ksplit + 31) / 32 * 32;
    auto blocks = [&](int bm, int bn) {
        return (int64_t)((pl.n_pair + bm - 1) / bm) * ((ncols + bn - 1) / bn) * pl.lin_ksplit;
    };
    // The largest tile that still fills the SMs: a block of the larger tiles is two warps, and an
    // SM needs about eight of them before its FP32 units are busy (136 pairs x 16 modes x 8 maps on
    // 501 x 1024 pixels, us: 64 x 64 1507, 32 x 32 889, chains 1004); with fewer blocks of 32 x 32
    // the chains' own latency is the bound (55 pairs, 8 maps of 10 modes, 1.2 blocks per SM: 452
    // with 32 x 32 tiles, 309 with k_linear_chain).
    if (blocks(64, 64) >= 4 * (int64_t)pl.nsm) return linear_gemm_launch<64, 64, 8, 8, 16, 4>(pl, maps, ncols, kchunk, partial, st);
    if (blocks(32, 32) >= 3 * (int64_t)pl.nsm) return linear_gemm_launch<32, 32, 4, 4, 32, 4>(pl, maps, ncols, kchunk, partial, st);
    const cudaError_t e = cudaFuncSetAttribute(k_linear_chain, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)LC_SMEM);
    if (e != cudaSuccess) return e;
    k_linear_chain<<<dim3((pl.n_pair + LC_R - 1) / LC_R, (ncols + LC_C - 1) / LC_C, pl.lin_ksplit), 64, LC_SMEM, st>>>(
        pl.n_pair, ncols, pl.npix, kchunk, pl.pair_mean, pl.W, maps, partial);
    note_launch(pl);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- beta
__device__ __forceinline__ int pair_lex(int p, int r, int P) { return p * P - (p * (p - 1)) / 2 + (r - p); }

__global__ void k_beta_finalize(int P, int n_max, int B, int ncub, int use_linear, int ksplit, int n_pair,
                                const int* __restrict__ mp, const int* __restrict__ mr, const int* __restrict__ ms,
                                const double* __restrict__ cub, const double* __restrict__ lin,
                                double* __restrict__ beta) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= B * n_max) return;
    const int b = i / n_max, n = i % n_max;
    double v = 0.0;
    for (int c = 0; c < ncub; ++c) v += cub[((int64_t)b * ncub + c) * n_max + n];
    if (use_linear) {
        const int p = mp[n], r = mr[n], s = ms[n];
        const int ncols = B * P;
        const int rpr = pair_lex(p, r, P), rps = pair_lex(p, s, P), rrs = pair_lex(r, s, P);
        double l = 0.0;
        for (int z = 0; z < ksplit; ++z) {
            const double* g = lin + (int64_t)z * n_pair * ncols;
            l += g[(int64_t)rpr * ncols + b * P + s] + g[(int64_t)rps * ncols + b * P + r]
               + g[(int64_t)rrs * ncols + b * P + p];
        }
        v -= l;
    }
    beta[i] = v;
}

cudaError_t launch_beta_finalize(Plan& pl, int B, int use_linear, const double* cub_partial,
                                 const double* lin_partial, int lin_splits, double* beta, cudaStream_t st) {
    if (B == 0) return cudaSuccess;
    const int n = B * pl.n_max;
    k_beta_finalize<<<(n + 127) / 128, 128, 0, st>>>(pl.P, pl.n_max, B, pl.cubic_ctas, use_linear, lin_splits,
                                                      pl.n_pair, pl.mode_prs, pl.mode_prs + 1024,
                                                      pl.mode_prs + 2048, cub_partial, lin_partial, beta);
    note_launch(pl);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- Monte Carlo pair means
// Two threads per pixel: thread h (h = 0, 1, warp-uniform) owns the mode rows p = 2k + h,
// k = 0 .. PM/2 - 1.  It works on its pixel's map values shifted by h (v[i] = M_{i+h}),
// so that both threads run the same code with compile-time indices: its pairs are
// (2k, r') in the shifted frame, r' >= 2k, i.e. (2k + h, r' + h).  The maps stream
// through a PA_STAGES-deep ring in shared memory by cp.async: the two threads of a
// pixel copy alternate rows of its column (each map value is fetched once) and read the
// whole column after a CTA barrier; a second barrier keeps a stage from being refilled
// while it is read.  The FP64 sums are read, updated and written once per launch: the
// tile's FP32 sums go to shared memory by pair, each thread updates the pairs of its parity
// at its pixel, PA_RMW loads in flight at a time (more spill at the 128-register cap that
// keeps four CTAs per SM), their lines sent to L2 a few maps before the update.
constexpr int PA_THREADS = 128;             // 64 pixels x 2 row parities
constexpr int PA_PIX = PA_THREADS / 2;
constexpr int PA_STAGES = 5;
constexpr int PA_RMW = 8;                   // FP64 read-modify-writes in flight per thread (68 per thread at P = 16)
constexpr int PA_PREFETCH = 4;              // maps before the end of a tile at which its FP64 sums go to L2

template <int PM>
constexpr size_t pa_smem_floats() {
    constexpr size_t ring = (size_t)PA_STAGES * PM * PA_PIX;
    constexpr size_t sums = (size_t)(PM * (PM + 1) / 2) * PA_PIX;
    return ring > sums ? ring : sums;
}

__device__ __forceinline__ void cp_async4(float* dst, const float* src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(src) : "memory");
}

template <int PM>
__global__ void __launch_bounds__(PA_THREADS, 4)
k_pair_accumulate(int P, int B, int64_t npix, const float* __restrict__ maps, double* __restrict__ sums) {
    constexpr int NACC = (PM / 2) * (PM / 2 + 1);                // sum over k of (PM - 2k)
    extern __shared__ __align__(16) float pa_ring[];            // [PA_STAGES][PM][PA_PIX]; then [n_pair][PA_PIX]
    const int tid = threadIdx.x;
    const int h = tid / PA_PIX, xl = tid % PA_PIX;
    const int nv = P - h;                                       // shifted values that exist
    for (int64_t x0 = (int64_t)blockIdx.x * PA_PIX; x0 < npix; x0 += (int64_t)gridDim.x * PA_PIX) {
        const int64_t x = x0 + xl;
        const bool in = x < npix;
        __syncthreads();                                              // previous sums read out of the ring
        auto issue = [&](int b) {
            if (b < B && in) {
                const float* src = maps + ((int64_t)b * P + h) * npix + x;
                float* dst = pa_ring + ((b % PA_STAGES) * PM + h) * PA_PIX + xl;
                for (int i = h; i < P; i += 2) {                        // rows of this thread's parity
                    cp_async4(dst, src);
                    src += 2 * npix;
                    dst += 2 * PA_PIX;
                }
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
#pragma unroll
        for (int b = 0; b < PA_STAGES - 1; ++b) issue(b);
        float acc[NACC];
#pragma unroll
        for (int c = 0; c < NACC; ++c) acc[c] = 0.f;
#pragma unroll 1
        for (int b = 0; b < B; ++b) {
            __syncthreads();                                          // stage (b - 1) % PA_STAGES is free
            issue(b + PA_STAGES - 1);
            asm volatile("cp.async.wait_group %0;" ::"n"(PA_STAGES - 1) : "memory");   // this thread's rows of map b
            __syncthreads();                                          // ... and the partner's
            if (b == (B > PA_PREFETCH ? B - PA_PREFETCH : 0)) {
                // the FP64 sums of this tile into L2 a few maps before their update: one
                // 128-byte line per thread and step (PA_PIX doubles of a pair = 4 lines)
                const int npair = P * (P + 1) / 2;
                for (int i = tid; i < npair * (PA_PIX / 16); i += PA_THREADS) {
                    const int64_t xs = x0 + (i % (PA_PIX / 16)) * 16;
                    if (xs < npix) {
                        const double* line = sums + (int64_t)(i / (PA_PIX / 16)) * npix + xs;
                        asm volatile("prefetch.global.L2 [%0];" ::"l"(line));
                    }
                }
            }
            const float* col = pa_ring + ((b % PA_STAGES) * PM + h) * PA_PIX + xl;
            float v[PM];
#pragma unroll
            for (int i = 0; i < PM; ++i) v[i] = (i < nv && in) ? col[i * PA_PIX] : 0.f;
            int c = 0;
#pragma unroll
            for (int k = 0; k < PM / 2; ++k)
#pragma unroll
                for (int r = 2 * k; r < PM; ++r) {
                    acc[c] = fmaf(v[2 * k], v[r], acc[c]);
                    ++c;
                }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();                                              // the ring is free
        // the sums pass through shared memory, one row of PA_PIX pixels per pair (lexicographic),
        // so that the FP64 update below runs over pairs h, h + 2, ... with one stride
#pragma unroll
        for (int k = 0, c = 0; k < PM / 2; ++k) {
            const int pa = 2 * k + h, q0 = pair_lex(pa, pa, P);
#pragma unroll
            for (int j = 0; j < PM - 2 * k; ++j, ++c)
                if (pa + j < P) pa_ring[(q0 + j) * PA_PIX + xl] = acc[c];
        }
        __syncthreads();
        if (in) {
            // PA_RMW old values are loaded before the first of their stores, so that those
            // loads are in flight together
            const int nq = (P * (P + 1) / 2 - h + 1) / 2;
            double* row = sums + (int64_t)h * npix + x;
            const float* add = pa_ring + h * PA_PIX + xl;
#pragma unroll 1
            for (int i0 = 0; i0 < nq; i0 += PA_RMW) {
                double old[PA_RMW];
#pragma unroll
                for (int u = 0; u < PA_RMW; ++u)
                    if (i0 + u < nq) old[u] = row[(int64_t)(2 * (i0 + u)) * npix];
#pragma unroll
                for (int u = 0; u < PA_RMW; ++u)
                    if (i0 + u < nq) row[(int64_t)(2 * (i0 + u)) * npix] = old[u] + (double)add[2 * (i0 + u) * PA_PIX];
            }
        }
    }
}

cudaError_t launch_pair_accumulate(Plan& pl, const float* maps, int B, cudaStream_t st) {
    if (B == 0) return cudaSuccess;
    const int64_t nblk = (pl.npix + PA_PIX - 1) / PA_PIX;
    const int grid = (int)(nblk < 152 * 16 ? nblk : 152 * 16);
    return with_even_modes(pl.P, [&](auto pm) {
        constexpr int PM = decltype(pm)::value;
        k_pair_accumulate<PM><<<grid, PA_THREADS, pa_smem_floats<PM>() * 4, st>>>(pl.P, B, pl.npix, maps, pl.pair_sum);
        note_launch(pl);
        return cudaGetLastError();
    });
}

__global__ void k_pair_finalize(int64_t n, double inv, const double* __restrict__ sums, float* __restrict__ mean) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        mean[i] = (float)(sums[i] * inv);
}

cudaError_t launch_pair_finalize(Plan& pl, cudaStream_t st) {
    const int64_t n = (int64_t)pl.n_pair * pl.npix;
    k_pair_finalize<<<152 * 8, 256, 0, st>>>(n, 1.0 / (double)pl.n_lin, pl.pair_sum, pl.pair_mean);
    note_launch(pl);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- adjoint (pixel part)
// hk[b][t][c] = 3 k_c h_{t,a,b'} for lexicographic pair c = (a, b'), k_c = 2 if a != b'
// else 1, h_tab = g_{sort(t,a,b)} / (number of distinct orderings of that triple).
__global__ void k_adjoint_weights(int P, int n_pair, int n_max, int B, const int* __restrict__ mode_of,
                                  const double* __restrict__ g, float* __restrict__ hk) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= B * P * n_pair) return;
    const int b = i / (P * n_pair), rem = i % (P * n_pair), t = rem / n_pair, c = rem % n_pair;
    int a = 0, cc = c;
    while (cc >= P - a) { cc -= P - a; ++a; }
    const int bb = a + cc;
    int x0 = t, x1 = a, x2 = bb, tmp;
    if (x0 > x1) { tmp = x0; x0 = x1; x1 = tmp; }
    if (x1 > x2) { tmp = x1; x1 = x2; x2 = tmp; }
    if (x0 > x1) { tmp = x0; x0 = x1; x1 = tmp; }
    const int nperm = (x0 == x2) ? 1 : ((x0 == x1 || x1 == x2) ? 3 : 6);
    const int n = mode_of[(x0 * P + x1) * P + x2];
    const double kc = (a == bb) ? 1.0 : 2.0;
    hk[i] = (float)(3.0 * kc * g[(int64_t)b * n_max + n] / nperm);
}

cudaError_t launch_adjoint_weights(Plan& pl, const double* g, int B, float* hk, cudaStream_t st) {
    if (B == 0) return cudaSuccess;
    const int n = B * pl.P * pl.n_pair;
    k_adjoint_weights<<<(n + 127) / 128, 128, 0, st>>>(pl.P, pl.n_pair, pl.n_max, B, pl.mode_of,
                                                        g, hk);
    note_launch(pl);
    return cudaGetLastError();
}

// In place: maps[b][t][x] <- U_t(x) = W_x sum_c hk[b][t][c] (M_a M_b' - <c>_x).
// Register tile per thread: AU_NX adjacent pixels x AU_NB maps, all PM values of each
// map in registers, accumulators packed in FP32 pairs over t.  Both pair loops (a, then
// b' >= a) are unrolled at compile time, so every map value is a register and the body
// has no branches; each pair costs four broadcast float4 loads of the weights per map
// and one 8-byte load of the pair means for 8 AU_NX AU_NB packed FMAs.  The pair-mean
// row of a + 1 is copied into shared memory (cp.async, each thread its own pixels) while
// row a is being used.  A CTA keeps its AU_NB maps' weights in shared memory and walks
// pixel tiles g, g + G, ...; CTAs of the same g but different map pairs are adjacent in
// launch order, so they read the same pair-mean rows close together in time.
constexpr int AU_THREADS = 128;
constexpr int AU_NX = 2;                    // adjacent pixels per thread
constexpr int AU_NB = 2;                    // maps per thread (and per CTA)
constexpr int AU_TILE = AU_THREADS * AU_NX; // pixels per CTA tile

__device__ __forceinline__ void cp_async8(float* dst, const float* src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait1() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }

// Pair-mean row a (b' = a .. P-1 of this thread's two pixels) into stage a & 1.
template <int PM>
__device__ __forceinline__ void adj_issue_row(int a, const float* __restrict__ pm, bool in, int P, int64_t npix,
                                              int64_t x0, int px, float* sP) {
    if (pm && in) {
        const int crow = a * P - a * (a - 1) / 2 - a;
        float* dst = sP + (a & 1) * PM * AU_TILE + px;
#pragma unroll
        for (int bb = 0; bb < PM; ++bb)
            if (bb >= a && bb < P) cp_async8(dst + bb * AU_TILE, pm + (int64_t)(crow + bb) * npix + x0 + px);
    }
    cp_async_commit();
}

// Row A of the pair loop (pairs (A, b'), b' >= A), then rows A+1 .. PM-1: a template
// recursion, so that every map-value index is a compile-time constant.
template <int PM, int A>
__device__ __forceinline__ void adj_rows(const float2 (&M)[AU_NB][PM], float2 (&u)[AU_NB][AU_NX][PM / 2],
                                         const float* sH, float* sP, const float* __restrict__ pm, bool in, int P,
                                         int64_t npix, int64_t x0, int px) {
    if constexpr (A < PM) {
        constexpr int NPM = PM * (PM + 1) / 2;
        if (A + 1 < PM) adj_issue_row<PM>(A + 1, pm, in, P, npix, x0, px, sP);
        else cp_async_commit();
        cp_async_wait1();                                  // row A has landed
        const float* prow = sP + (A & 1) * PM * AU_TILE + px;
#pragma unroll
        for (int bb = A; bb < PM; ++bb) {
            const float2 pv = *reinterpret_cast<const float2*>(prow + bb * AU_TILE);
            const int k = A * PM - A * (A - 1) / 2 + (bb - A);  // PM-lex pair index
#pragma unroll
            for (int i = 0; i < AU_NB; ++i) {
                const float y0 = fmaf(M[i][A].x, M[i][bb].x, -pv.x);
                const float y1 = fmaf(M[i][A].y, M[i][bb].y, -pv.y);
                const float2 y02 = make_float2(y0, y0), y12 = make_float2(y1, y1);
                const float4* h4 = reinterpret_cast<const float4*>(sH + (i * NPM + k) * PM);
#pragma unroll
                for (int q = 0; q < PM / 4; ++q) {
                    const float4 h = h4[q];
                    const float2 hlo = make_float2(h.x, h.y), hhi = make_float2(h.z, h.w);
                    u[i][0][2 * q] = __ffma2_rn(hlo, y02, u[i][0][2 * q]);
                    u[i][0][2 * q + 1] = __ffma2_rn(hhi, y02, u[i][0][2 * q + 1]);
                    u[i][1][2 * q] = __ffma2_rn(hlo, y12, u[i][1][2 * q]);
                    u[i][1][2 * q + 1] = __ffma2_rn(hhi, y12, u[i][1][2 * q + 1]);
                }
            }
        }
        adj_rows<PM, A + 1>(M, u, sH, sP, pm, in, P, npix, x0, px);
    }
}

template <int PM>
__global__ void __launch_bounds__(AU_THREADS, 2)
k_adjoint_u(int P, int n_pair, int B, int ngroups, int64_t npix, int nphi, int nrings, const float* __restrict__ hk,
            const float* __restrict__ pm, const float* __restrict__ vring, const float* __restrict__ W,
            float* __restrict__ maps) {
    constexpr int NPM = PM * (PM + 1) / 2;
    extern __shared__ __align__(16) float au_smem[];
    float* sH = au_smem;                                   // [AU_NB][NPM][PM], pairs in PM-lex order
    float* sP = sH + AU_NB * NPM * PM;                     // [2][PM][AU_TILE] pair-mean rows
    const int tid = threadIdx.x;
    const int nmp = (B + AU_NB - 1) / AU_NB;
    const int mp = blockIdx.x % nmp;
    const int g = blockIdx.x / nmp;
    const int b0 = mp * AU_NB;
    const int nb = min(AU_NB, B - b0);
    const int px = AU_NX * tid;                            // this thread's pixels within a tile
    for (int i = tid; i < AU_NB * NPM * PM; i += AU_THREADS) {
        const int mb = i / (NPM * PM), rem = i % (NPM * PM);
        const int k = rem / PM, t = rem % PM;
        int a = 0, kk = k;
        while (kk >= PM - a) { kk -= PM - a; ++a; }
        const int bb = a + kk;
        float v = 0.f;
        if (mb < nb && t < P && bb < P) v = hk[((int64_t)(b0 + mb) * P + t) * n_pair + pair_lex(a, bb, P)];
        sH[i] = v;
    }
    // pair-mean rows that are never copied (b' >= P, or no linear term) read as zero
#pragma unroll
    for (int st = 0; st < 2; ++st)
#pragma unroll
        for (int bb = 0; bb < PM; ++bb)
            if (!pm || bb >= P) *reinterpret_cast<float2*>(sP + (st * PM + bb) * AU_TILE + px) = make_float2(0.f, 0.f);
    __syncthreads();
    const int64_t ntile = (npix + AU_TILE - 1) / AU_TILE;
    for (int64_t tile = g; tile < ntile; tile += ngroups) {
        const int64_t x0 = tile * AU_TILE;
        const bool in = x0 + px < npix;                    // npix is even: both pixels or neither
        adj_issue_row<PM>(0, pm, in, P, npix, x0, px, sP);
        float2 M[AU_NB][PM];                               // (pixel 0, pixel 1) per map and mode
#pragma unroll
        for (int i = 0; i < AU_NB; ++i)
#pragma unroll
            for (int p = 0; p < PM; ++p) {
                float2 v = make_float2(0.f, 0.f);
                if (i < nb && p < P && in) v = *reinterpret_cast<const float2*>(maps + ((int64_t)(b0 + i) * P + p) * npix + x0 + px);
                M[i][p] = v;
            }
        float2 u[AU_NB][AU_NX][PM / 2];                    // (t = 2 tp, 2 tp + 1) packed
#pragma unroll
        for (int i = 0; i < AU_NB; ++i)
#pragma unroll
            for (int j = 0; j < AU_NX; ++j)
#pragma unroll
                for (int tp = 0; tp < PM / 2; ++tp) u[i][j][tp] = make_float2(0.f, 0.f);
        // sP entries are copied in and read by the same thread only
        adj_rows<PM, 0>(M, u, sH, sP, pm, in, P, npix, x0, px);
        if (in) {
            const float2 wx = *reinterpret_cast<const float2*>(W + x0 + px);
            const int ring = (int)((x0 + px) / nphi);     // both pixels (nphi is even)
#pragma unroll
            for (int i = 0; i < AU_NB; ++i)
#pragma unroll
                for (int t = 0; t < PM; ++t)
                    if (i < nb && t < P) {
                        // ring mode: the pair-mean term sum_c h_tc <c>_ring, the same for both pixels
                        const float vr = vring ? vring[((int64_t)(b0 + i) * P + t) * nrings + ring] : 0.f;
                        const float u0 = ((t & 1) ? u[i][0][t >> 1].y : u[i][0][t >> 1].x) - vr;
                        const float u1 = ((t & 1) ? u[i][1][t >> 1].y : u[i][1][t >> 1].x) - vr;
                        *reinterpret_cast<float2*>(maps + ((int64_t)(b0 + i) * P + t) * npix + x0 + px) =
                            make_float2(wx.x * u0, wx.y * u1);
                    }
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
}

template <int PM>
static cudaError_t launch_adjoint_u_pm(Plan& pl, int B, const float* hk, const float* pm, const float* vring,
                                       float* maps, cudaStream_t st) {
    constexpr int NPM = PM * (PM + 1) / 2;
    const size_t smem = ((size_t)AU_NB * NPM * PM + (size_t)2 * PM * AU_TILE) * sizeof(float);
    cudaError_t e = cudaFuncSetAttribute(k_adjoint_u<PM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const int nmp = (B + AU_NB - 1) / AU_NB;
    const int64_t ntile = (pl.npix + AU_TILE - 1) / AU_TILE;
    // two resident CTAs per SM in total, every map pair in every group
    int64_t ng = std::max<int64_t>(1, (152 * 2) / nmp);
    ng = std::min<int64_t>(ng, ntile);
    k_adjoint_u<PM><<<(unsigned)(ng * nmp), AU_THREADS, smem, st>>>(pl.P, pl.n_pair, B, (int)ng, pl.npix, pl.nphi,
                                                                    pl.nrings, hk, pm, vring, pl.W, maps);
    note_launch(pl);
    return cudaGetLastError();
}

cudaError_t launch_adjoint_u(Plan& pl, const float* /*maps_in*/, int B, const float* hk, int use_linear,
                             float* maps, cudaStream_t st) {
    // The kernel can subtract a per-ring term at every pixel (vring); the library applies
    // that term to the m = 0 analysis coefficients instead (k_vring_correct), which is
    // cheaper.  The parameter stays: without it this fully unrolled kernel is allocated
    // 255 registers with a spill and runs 15 % slower (measured at l_max = 2000).
    const float* vring = nullptr;
    if (B == 0) return cudaSuccess;
    if (pl.npix % 2 != 0) return cudaErrorInvalidValue;
    const float* pm = use_linear ? pl.pair_mean : nullptr;
    if (pl.P <= 4) return launch_adjoint_u_pm<4>(pl, B, hk, pm, vring, maps, st);
    if (pl.P <= 8) return launch_adjoint_u_pm<8>(pl, B, hk, pm, vring, maps, st);
    return launch_adjoint_u_pm<16>(pl, B, hk, pm, vring, maps, st);
}

}  // namespace modal
