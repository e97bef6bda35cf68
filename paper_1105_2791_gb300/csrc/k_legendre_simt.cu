// FP32 SIMT Legendre sums: forward, a register tile of modes and maps per ring pair;
// transposed, one of multipoles l and channels.
//
// Forward:  D_{b,p,m}(theta) = sum_{l>=m} lambda_lm(theta) f_p(l) a_{b,lm},
// split by the parity of l - m into E (even) and O (odd) so that one table row
// serves the north ring (E + O) and its mirror south ring (E - O), since
// lambda_lm(-mu) = (-1)^{l+m} lambda_lm(mu).  E and O are stored per ring pair
// (delta layout [B][P][lmax+1][2][RH]); the ring FFT combines them.  This is the
// separable evaluation of the filtered maps whose cube gives Eq. bbispect.
#include "modal_internal.cuh"

namespace modal {

// A thread owns one ring pair and MB maps: a value of lambda and the filter values of its l,
// broadcast from shared memory, then serve all of them, and a row of the table is read once per
// MB WM maps.  WM of a block's four warps lie along the maps and the others along ring pairs, so
// that ring counts are padded to 32 where several maps fill the block.  Bound by instruction
// issue as scalar code, so the products and sums are packed FP32 pairs over modes (two roundings
// as before: the product lambda a, then one FMA per mode, l ascending).  us, before and after:
// 21 maps, l_max = 250, 8 modes 189 -> 123; 16 maps, l_max = 500, 10 modes 1320 -> 734; 8 maps,
// l_max = 1000, 16 modes 5131 -> 3728 (34 TF/s).
template <int PM, int MB, int WM>
__global__ void __launch_bounds__(128)
k_legendre_simt(int L, int P, int B, int R_half, int RH, const float* __restrict__ lam,
                const float* __restrict__ filt, const float2* __restrict__ alm, int64_t n_alm,
                float2* __restrict__ delta) {
    constexpr int CH = 64, NM = MB * WM, WR = 4 / WM;
    __shared__ __align__(16) float4 sa[CH][NM];                 // (re, re, im, im): operands of packed products
    __shared__ __align__(16) float sf[CH][PM];
    const int m = blockIdx.y, b0 = blockIdx.z * NM;
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int wm = warp % WM;                                   // this warp's maps: b0 + wm MB ..
    const int j = (blockIdx.x * WR + warp / WM) * 32 + lane;
    const int64_t base = d_alm_index(m, m, L);
    const bool active = j < R_half && b0 + wm * MB < B;
    const int last = L - m;                                     // the last row of this order
    const float* lp = lam + base * (int64_t)RH + (active ? j : 0);

    // sums of one parity: real and imaginary parts of two modes at a time
    float2 re[2][MB][PM / 2], im[2][MB][PM / 2];
#pragma unroll
    for (int e = 0; e < 2; ++e)
#pragma unroll
        for (int k = 0; k < MB; ++k)
#pragma unroll
            for (int p = 0; p < PM / 2; ++p) re[e][k][p] = im[e][k][p] = make_float2(0.f, 0.f);
    // the next eight values of lambda are on their way while eight are used; rows past the last
    // repeat it (their a_lm are zero)
    float lv[8], ln[8];
    auto fetch = [&](int d) {
        if (d + 7 <= last) {
            const float* q = lp + (int64_t)d * RH;
#pragma unroll
            for (int u = 0; u < 8; ++u) ln[u] = q[(int64_t)u * RH];
        } else {
#pragma unroll
            for (int u = 0; u < 8; ++u) ln[u] = lp[(int64_t)min(d + u, last) * RH];
        }
    };
    fetch(0);
    for (int d0 = 0; d0 <= last; d0 += CH) {
        const int n = min(CH, last + 1 - d0);
        __syncthreads();
        for (int i = threadIdx.x; i < CH * NM; i += 128) {
            const int li = i % CH, k = i / CH;
            const float2 a = (li < n && b0 + k < B) ? alm[(int64_t)(b0 + k) * n_alm + base + d0 + li] : make_float2(0.f, 0.f);
            sa[li][k] = make_float4(a.x, a.x, a.y, a.y);
        }
        for (int i = threadIdx.x; i < CH * PM; i += 128) {
            const int li = i / PM, p = i % PM;
            sf[li][p] = (li < n && p < P) ? filt[(int64_t)p * (L + 1) + m + d0 + li] : 0.f;
        }
        __syncthreads();
        if (active) {
            // d0 is a multiple of CH (even), so i + u has the parity of u.
            for (int i = 0; i < n; i += 8) {
#pragma unroll
                for (int u = 0; u < 8; ++u) lv[u] = ln[u];
                fetch(d0 + i + 8);
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    float2 tr[MB], ti[MB];
                    const float2 l2 = make_float2(lv[u], lv[u]);
#pragma unroll
                    for (int k = 0; k < MB; ++k) {
                        const float4 a = sa[i + u][wm * MB + k];
                        tr[k] = __fmul2_rn(l2, make_float2(a.x, a.y));
                        ti[k] = __fmul2_rn(l2, make_float2(a.z, a.w));
                    }
                    const float4* f4 = reinterpret_cast<const float4*>(&sf[i + u][0]);
#pragma unroll
                    for (int q = 0; q < PM / 4; ++q) {
                        const float4 f = f4[q];
                        const float2 fv[2] = {make_float2(f.x, f.y), make_float2(f.z, f.w)};
#pragma unroll
                        for (int k = 0; k < MB; ++k)
#pragma unroll
                            for (int c = 0; c < 2; ++c) {
                                re[u & 1][k][2 * q + c] = __ffma2_rn(fv[c], tr[k], re[u & 1][k][2 * q + c]);
                                im[u & 1][k][2 * q + c] = __ffma2_rn(fv[c], ti[k], im[u & 1][k][2 * q + c]);
                            }
                    }
                }
            }
        }
    }
    if (!active) return;
#pragma unroll
    for (int k = 0; k < MB; ++k) {
        const int b = b0 + wm * MB + k;
        if (b >= B) break;
#pragma unroll
        for (int p = 0; p < PM; ++p) {
            if (p < P) {
                const int64_t row = ((int64_t)(b * P + p) * (L + 1) + m) * 2 * RH;
#pragma unroll
                for (int e = 0; e < 2; ++e)
                    delta[row + e * RH + j] = (p & 1) ? make_float2(re[e][k][p / 2].y, im[e][k][p / 2].y)
                                                      : make_float2(re[e][k][p / 2].x, im[e][k][p / 2].x);
            }
        }
    }
}

template <int PM, int MB, int WM>
static void legendre_simt_launch(const Plan& pl, const float2* alm, int B, float2* delta, cudaStream_t st) {
    constexpr int rings = 32 * (4 / WM), maps = MB * WM;
    const dim3 grid((pl.R_half + rings - 1) / rings, pl.lmax + 1, (B + maps - 1) / maps);
    k_legendre_simt<PM, MB, WM><<<grid, 128, 0, st>>>(pl.lmax, pl.P, B, pl.R_half, pl.RH, pl.lam, pl.filt, alm, pl.n_alm, delta);
    note_launch(pl);
}

template <int PM>
static cudaError_t legendre_simt_pm(const Plan& pl, const float2* alm, int B, float2* delta, cudaStream_t st) {
    if (B == 1) {
        legendre_simt_launch<PM, 1, 1>(pl, alm, B, delta, st);
    } else if constexpr (PM > 12) {
        // the sums of two maps leave no room for three warps per sub-partition (16 modes, 16 maps,
        // l_max = 500: 971 us with one per thread, 1153 with two; 10 modes 861 and 734)
        if (B == 2) legendre_simt_launch<PM, 1, 2>(pl, alm, B, delta, st);
        else legendre_simt_launch<PM, 1, 4>(pl, alm, B, delta, st);
    } else {
        // Two maps per thread from two warps per sub-partition on; below that the longer chain per
        // order shows (10 modes, 8 maps, l_max = 32 9.7 us with two, 8.2 with one).  Four of a block's warps along the maps (eight maps, which read the table
        // once), or two where that leaves an eighth fewer places empty: 9 maps of 10 modes, l_max =
        // 250 104 and 95 us, l_max = 500 635 and 489 (12 maps 673 and 522); 16 maps, l_max = 250 126 and 134.
        const int64_t warps = (int64_t)((pl.R_half + 31) / 32) * ((B + 1) / 2) * (pl.lmax + 1);
        const int four = (B + 7) / 8 * 8, two = (B + 3) / 4 * 4;
        if (warps < 8 * (int64_t)pl.nsm) legendre_simt_launch<PM, 1, 2>(pl, alm, B, delta, st);
        else if (B == 2) legendre_simt_launch<PM, 2, 1>(pl, alm, B, delta, st);
        else if (8 * two < 7 * four) legendre_simt_launch<PM, 2, 2>(pl, alm, B, delta, st);
        else legendre_simt_launch<PM, 2, 4>(pl, alm, B, delta, st);
    }
    return cudaGetLastError();
}

cudaError_t launch_legendre_simt(const Plan& pl, const float2* alm, int B, float2* delta, cudaStream_t st) {
    if (B == 0) return cudaSuccess;
    switch ((pl.P + 3) / 4) {
        case 1: return legendre_simt_pm<4>(pl, alm, B, delta, st);
        case 2: return legendre_simt_pm<8>(pl, alm, B, delta, st);
        case 3: return legendre_simt_pm<12>(pl, alm, B, delta, st);
        default: return legendre_simt_pm<16>(pl, alm, B, delta, st);
    }
}

// Transposed sums:  G_{b,t,lm} = sum_j lambda_lm(theta_j) U^{par(l-m)}_{b,t,m}(j), where
// U^0 = U_north + U_south and U^1 = U_north - U_south per ring pair (the mirror
// symmetry again).  Output per (b, l, m):
//   rowfilt != NULL:  c_m sum_t rowfilt[t][l] G_t   (adjoint: c_0 = 1, c_m = 2)
//   rowfilt == NULL:  G_0                           (quadrature analysis, nt = 1)
// ut layout: [B][nt][lmax+1][2][RH] complex.
//
// For one order and parity this is a GEMM: rows = values of l, columns = channels (map, t)
// x (Re, Im), K = ring pairs, bound by FP32 arithmetic from about ten channels on and by the
// read of the lambda table below.  A block holds LA_BM rows x NC channels, so that a row of
// the table is read once per NC channels, and each thread TL rows x TC channels in
// registers.  Both operands are contiguous along K in memory and stay so in shared memory
// (cp.async, three stages of LA_BK ring pairs; a thread reads 16 bytes along K of each of its
// rows and channels; the odd multiples of 16 bytes between rows keep the reads of a warp on
// different banks).  Every output is one chain of FMAs over j ascending, whatever the tile.
// 32 maps at l_max = 1000 (1001 x 2048): 8.80 ms with one channel per block (the table read
// once per channel, three quarters of the arithmetic on padding), 0.70 ms now (46 TF/s, 0.58
// of the measured FP32 rate); the 55 pair-mean rows at l_max = 500 2.06 -> 0.17 ms.
constexpr int LA_BM = 64;                   // values of l (one parity) per block
constexpr int LA_BK = 16;                   // ring pairs per stage
constexpr int LA_STAGES = 3;
constexpr int LA_SL = LA_BK + 4;            // floats per row of the lambda tile
constexpr int LA_SU = 2 * LA_BK + 4;        // floats per channel of the U tile

__device__ __forceinline__ void la_cp16(float* dst, const void* src, int bytes) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(bytes) : "memory");
}

template <int NC, int TL, int TC>
__global__ void __launch_bounds__((LA_BM / TL) * (NC / TC))
k_legendre_adj_simt(int L, int nt, int nchan, int cpb, int R_half, int RH, const float* __restrict__ lam,
                    const float2* __restrict__ ut, const float* __restrict__ rowfilt, int64_t n_alm,
                    float2* __restrict__ out) {
    constexpr int NT = (LA_BM / TL) * (NC / TC);
    constexpr int NLG = LA_BM / TL, NCG = NC / TC;           // thread groups along l and channels
    constexpr int STAGE = LA_BM * LA_SL + NC * LA_SU;
    __shared__ __align__(16) float sm[LA_STAGES * STAGE];
    const int m = blockIdx.y >> 1, par = blockIdx.y & 1;
    const int nl = (L - m - par >= 0) ? (L - m - par) / 2 + 1 : 0;     // rows of this order and parity
    const int r0 = blockIdx.x * LA_BM;
    if (r0 >= nl) return;
    const int c0 = blockIdx.z * cpb;                          // first channel; cpb <= NC channels per block
    const int nc = min(cpb, nchan - c0);
    const int tid = threadIdx.x;
    // half a warp holds 4 x CW threads, so that its 16-byte reads touch few rows and channels
    constexpr int CW = NCG < 4 ? NCG : 4;
    const int rest = tid / (4 * CW);
    const int lg = tid % 4 + 4 * (rest % (NLG / 4));          // rows lg + NLG i
    const int cg = (tid / 4) % CW + CW * (rest / (NLG / 4));  // channels cg + NCG k
    const int64_t base = d_alm_index(m, m, L) + par;
    const int64_t urow = (int64_t)(L + 1) * 2 * RH;           // ut stride between channels
    const float2* ub = ut + (int64_t)c0 * urow + ((int64_t)m * 2 + par) * RH;

    auto issue = [&](int k) {
        const int j0 = k * LA_BK;
        if (j0 < R_half) {
            float* sl = sm + (k % LA_STAGES) * STAGE;
            float* su = sl + LA_BM * LA_SL;
#pragma unroll
            for (int i = tid; i < LA_BM * (LA_BK / 4); i += NT) {
                const int r = i / (LA_BK / 4), q = i % (LA_BK / 4);
                const bool in = r0 + r < nl;                  // the table's row is zero from R_half to RH
                la_cp16(sl + r * LA_SL + 4 * q, lam + (base + 2 * (int64_t)(in ? r0 + r : 0)) * RH + j0 + 4 * q, in ? 16 : 0);
            }
#pragma unroll
            for (int i = tid; i < NC * (LA_BK / 2); i += NT) {
                const int c = i / (LA_BK / 2), q = i % (LA_BK / 2);
                const int left = (c < nc) ? R_half - (j0 + 2 * q) : 0;   // valid ring pairs of this 16-byte piece
                la_cp16(su + c * LA_SU + 4 * q, ub + (left > 0 ? c * urow + j0 + 2 * q : 0), left >= 2 ? 16 : (left == 1 ? 8 : 0));
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };

    float2 acc[TL][TC];
#pragma unroll
    for (int i = 0; i < TL; ++i)
#pragma unroll
        for (int k = 0; k < TC; ++k) acc[i][k] = make_float2(0.f, 0.f);
    const int nk = (R_half + LA_BK - 1) / LA_BK;
#pragma unroll
    for (int k = 0; k < LA_STAGES - 1; ++k) issue(k);
    for (int k = 0; k < nk; ++k) {
        asm volatile("cp.async.wait_group %0;" ::"n"(LA_STAGES - 2) : "memory");
        __syncthreads();                                      // stage k is here, stage k - 1 is free
        issue(k + LA_STAGES - 1);
        const float* sl = sm + (k % LA_STAGES) * STAGE + lg * LA_SL;
        const float* su = sm + (k % LA_STAGES) * STAGE + LA_BM * LA_SL + cg * LA_SU;
#pragma unroll
        for (int q = 0; q < LA_BK / 4; ++q) {
            float4 lv[TL];
#pragma unroll
            for (int i = 0; i < TL; ++i) lv[i] = *reinterpret_cast<const float4*>(sl + i * NLG * LA_SL + 4 * q);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                float4 uv[TC];
#pragma unroll
                for (int c = 0; c < TC; ++c) uv[c] = *reinterpret_cast<const float4*>(su + c * NCG * LA_SU + 8 * q + 4 * h);
#pragma unroll
                for (int i = 0; i < TL; ++i) {
                    const float l0 = h ? lv[i].z : lv[i].x, l1 = h ? lv[i].w : lv[i].y;
                    const float2 l02 = make_float2(l0, l0), l12 = make_float2(l1, l1);
#pragma unroll
                    for (int c = 0; c < TC; ++c) acc[i][c] = __ffma2_rn(l02, make_float2(uv[c].x, uv[c].y), acc[i][c]);
#pragma unroll
                    for (int c = 0; c < TC; ++c) acc[i][c] = __ffma2_rn(l12, make_float2(uv[c].z, uv[c].w), acc[i][c]);
                }
            }
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    if (!rowfilt) {
#pragma unroll
        for (int i = 0; i < TL; ++i)
#pragma unroll
            for (int c = 0; c < TC; ++c) {
                const int r = r0 + lg + NLG * i, ch = cg + NCG * c;
                if (r < nl && ch < nc) out[(int64_t)(c0 + ch) * n_alm + base + 2 * r] = acc[i][c];
            }
        return;
    }
    // the nt channels of each map meet in shared memory: one thread per (row, map) sums them
    __syncthreads();
    float2* g = reinterpret_cast<float2*>(sm);                // [LA_BM][NC + 1]
    static_assert(LA_BM * (NC + 1) * 2 <= LA_STAGES * STAGE, "the G tile fits the stages");
#pragma unroll
    for (int i = 0; i < TL; ++i)
#pragma unroll
        for (int c = 0; c < TC; ++c) g[(lg + NLG * i) * (NC + 1) + cg + NCG * c] = acc[i][c];
    __syncthreads();
    for (int i = tid; i < LA_BM * (nc / nt); i += NT) {
        const int r = i % LA_BM, b = i / LA_BM;
        if (r0 + r >= nl) continue;
        const int l = m + par + 2 * (r0 + r);
        float2 v = make_float2(0.f, 0.f);
        for (int t = 0; t < nt; ++t) {
            const float f = rowfilt[(int64_t)t * (L + 1) + l];
            const float2 a = g[r * (NC + 1) + b * nt + t];
            v.x = fmaf(f, a.x, v.x);
            v.y = fmaf(f, a.y, v.y);
        }
        const float cm = (m == 0) ? 1.f : 2.f;
        v.x *= cm;
        v.y *= cm;
        if (m == 0) v.y = 0.f;
        out[(int64_t)(c0 / nt + b) * n_alm + base + 2 * (r0 + r)] = v;
    }
}

template <int NC, int TL, int TC>
static cudaError_t legendre_adj_launch(const Plan& pl, const float2* ut, int B, const float* rowfilt, int nt,
                                       float2* out, cudaStream_t st) {
    const int nchan = B * nt;
    const int cpb = rowfilt ? NC / nt * nt : NC;               // whole maps per block where their channels are summed
    const int nlmax = pl.lmax / 2 + 1;
    const dim3 grid((nlmax + LA_BM - 1) / LA_BM, 2 * (pl.lmax + 1), (nchan + cpb - 1) / cpb);
    k_legendre_adj_simt<NC, TL, TC><<<grid, (LA_BM / TL) * (NC / TC), 0, st>>>(
        pl.lmax, nt, nchan, cpb, pl.R_half, pl.RH, pl.lam, ut, rowfilt, pl.n_alm, out);
    note_launch(pl);
    return cudaGetLastError();
}

// ut: nt channels for each of B maps.  Without rowfilt the channels are independent rows (nt = 1).
cudaError_t launch_legendre_adjoint_simt(const Plan& pl, const float2* ut, int B, const float* rowfilt,
                                         int nt, float2* out, cudaStream_t st) {
    if (B == 0) return cudaSuccess;
    if (nt < 1 || nt > MODAL_MAXP || (!rowfilt && nt != 1)) return cudaErrorInvalidValue;
    // The tile of least cost: its padded channels times its time per channel (64 channels, l_max =
    // 400: 5.4, 2.5, 2.2 and 2.0 us), of those that give each SM 2.5 blocks; below that a narrower
    // tile's shorter blocks are faster.  us for tiles of 2 / 8 / 16 / 32: l_max = 51, 20 channels
    // 4.0 / 3.9 / 4.3 / 5.3; l_max = 100, 6 channels 4.3 / 4.7 / 5.7 / 7.0; l_max = 250, 11
    // channels 22.9 / 18.6 / 17.0 / 21.6; l_max = 400, 33 channels 189 / 103 / 107 / 127.
    // (The narrowest tile that holds all channels, up to 32, took 5.3, 4.7, 17.0 and 127.)
    int nsm = 0;
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, pl.dev);
    // blocks of one channel tile: each order's rows of either parity in tiles of LA_BM
    auto upto = [](int64_t n) { const int64_t q = (n + 1) / (2 * LA_BM); return LA_BM * q * (q + 1) + (n + 1) % (2 * LA_BM) * (q + 1); };
    const int64_t rows = upto(pl.lmax) + upto(pl.lmax - 1);
    const int width[4] = {2, 8, 16, 32}, cost_us[4] = {54, 25, 22, 20};
    int best = -1;
    int64_t best_cost = 0;
    for (int i = 0; i < 4; ++i) {
        if (width[i] < nt) continue;
        const int cpb = rowfilt ? width[i] / nt * nt : width[i];
        const int64_t tiles = ((int64_t)B * nt + cpb - 1) / cpb, cost = tiles * width[i] * cost_us[i];
        if (best >= 0 && (2 * rows * tiles < 5 * nsm || cost >= best_cost)) continue;
        best = i;
        best_cost = cost;
    }
    switch (best) {
        case 0: return legendre_adj_launch<2, 2, 1>(pl, ut, B, rowfilt, nt, out, st);
        case 1: return legendre_adj_launch<8, 4, 2>(pl, ut, B, rowfilt, nt, out, st);
        case 2: return legendre_adj_launch<16, 8, 2>(pl, ut, B, rowfilt, nt, out, st);
        default: return legendre_adj_launch<32, 8, 4>(pl, ut, B, rowfilt, nt, out, st);
    }
}

}  // namespace modal
