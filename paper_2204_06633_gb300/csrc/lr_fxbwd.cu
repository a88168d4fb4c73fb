// Adjoint kernels on the tensor cores: the transposes of the TDI and projection operators and the sky-angle
// gradient, for FP64 and mixed plans alike (FP64 accuracy).
//
// The gathers of lr_bwd.cu (FP64) and lr_bwdmx.cu (float-float) spend ~50 FP64 or ~1000 FP32 operations per
// tap on weights and sums.  Here the merged, expanded stencils of lr_fx64.cu are transposed: with
// W(t) = sum_q b_q T_q(nu(t)) the transpose of  y[j] = sum_c W(t_j)[c] x[j + c]  is
//      gx[i] = sum_q sum_c b_q[c] (T_q gy)[i - c],
// a contraction with constant stencils (taps in reverse) of the series T_q(nu_j) gy_j, formed in fixed point by
// Chebyshev's recurrence.  All orders, links and channels of one output meet in the same level sums.
//   K1  g_y = T^T g_xyz    blocks of link samples; three channels, four orders, stencils of the plan's table.
//   K2  g_h = P^T g_y      blocks of strain samples; six links, eight orders; h+ and hx are the columns' halves.
//   K3  dLoss/d(lambda, beta, psi)   blocks of link samples: with y[k] = sum_n V_n(k) h[k + c] over the
//       expansion nodes, the gradient is the inner product of dV_n/dtheta with the correlations
//       C_q[c] = sum_k T_q(nu_k) gy[k] h[k + c], which are contractions over the block's samples; the node
//       values (weights, their derivatives, geometry) are then needed 8 times per block, not per sample.
// Segments (stencil steps, spline knots), ranges and the blocks evaluated sample by sample are as in lr_fx64.cu; K3
// bounds the orders of its products from the geometry at the nodes (sky_series_fits).
//
// Measured (one year at order 41, mixed plan): K1 5.97 -> 1.65, K2 12.16 -> 4.45, K3 12.2 -> 6.34 ms;
// 65536 samples at order 25 (FP64 plan): K1 1.26 -> 0.063, K2 0.42 -> 0.116, K3 0.64 -> 0.175 ms.
// K3 is bound by the FP64 pipe (44 % busy: node weights with derivatives, level sums to FP64) and the barriers
// around it, with the tensor pipe at 20 %; integer conversion of its level sums was slower (0.914).
#include "lr_fx64.cuh"

#include "lr_bwd.h"

namespace lr {
namespace {

// digit planes of T_q g: digits that order q's products need (one more than its levels, up to seven)
__host__ __device__ constexpr int gdigits(bool tdi, int q) { return zq(tdi, q) ? 8 - zq(tdi, q) : 7; }
__host__ __device__ constexpr int gplane(bool tdi, int q)  // planes before order q
{
    return tdi ? (q == 0 ? 0 : q == 1 ? 7 : q == 2 ? 14 : q == 3 ? 19 : 22)
               : (q <= 3 ? 7 * q : q == 4 ? 27 : q == 5 ? 32 : q == 6 ? 37 : q == 7 ? 41 : 44);
}
constexpr int TQP = gplane(true, NT);                         // 22 planes of a channel
constexpr int QA = 3, PQA = gplane(false, QA), PQB = gplane(false, NN) - PQA;  // a link in two rounds: 21 and 23 planes
constexpr int GB = 520;                                       // bytes of a digit row of T_q g (K3): distinct banks per link
static_assert(GB % 4 == 0 && GB >= 4 + 12 + 16 * (NY / 16 - 1) + 8, "the last step's loads of a full block stay in the row");
constexpr int GROWS = gplane(false, NN);                      // 44 rows per link

constexpr int K1_PART = 3 * NY * 8, K1_PLANES = K1_PART + 6 * NY * 8;
// the node weights of blocks off the table share the sums' and planes' place
__host__ __device__ constexpr int k1_w(int T) { return K1_PART + (T * WTS * 8 > 6 * NY * 8 + TQP * DL * 2 ? T * WTS * 8 : 6 * NY * 8 + TQP * DL * 2); }
constexpr int K2_STENCILS = 6 * NY * 8, K2_PLANES = K2_STENCILS + FX_PROJ_W, K2_GROUP = PQB * DL * 2;  // one group of planes per 256 threads
constexpr int K3_G = FX_PROJ_PLANES, K3_PAIR = 2 * GROWS * GB;   // digit rows of a link pair per 256 threads
__host__ __device__ constexpr int k3_c(int T, int nthr)
{
    const int g = nthr / 256 * K3_PAIR, w = 16 * T * WNS;
    return K3_G + (((g > w ? g : w) + 15) & ~15);
}

// acc[L] += the level sums of order Q, its digit planes at `a_lane`, its digit rows at `w_lane`
template <int Q, bool TDI, bool LAST>
__device__ __forceinline__ void contract_order(float (&acc)[7][4], const unsigned char *a_lane, const unsigned char *w_lane,
                                               uint32_t sh, int nks)
{
    constexpr int Z = LAST ? 6 : zq(TDI, Q), Z0 = zq(TDI, Q), NA = Z ? 8 - Z : 7, RS = TDI ? 16 : 8;
#pragma unroll 1
    for (int ks = 0; ks < nks; ++ks, a_lane += 32, w_lane += 16) {
        uint32_t a[NA][4];
#pragma unroll
        for (int k = 0; k < NA; ++k) {
            const uint2 lo = *reinterpret_cast<const uint2 *>(a_lane + k * DL * 2);
            const uint2 hi = *reinterpret_cast<const uint2 *>(a_lane + k * DL * 2 + 8 * RS);
            a[k][0] = lo.x; a[k][1] = hi.x; a[k][2] = lo.y; a[k][3] = hi.y;
        }
#pragma unroll
        for (int d = Z; d < 7; ++d) {
            const uint32_t *w = reinterpret_cast<const uint32_t *>(w_lane + (d - Z0) * WS);
            const uint32_t u = __funnelshift_r(w[0], w[1], sh);
            const uint32_t b0 = digits_h2(u, 0x4140u), b1 = digits_h2(u, 0x4342u);
#pragma unroll
            for (int k = 0; k < 6 - d; ++k) mma_f16(acc[d + k], a[k], b0, b1);
            if (d == 0) {
                mma_f16(acc[6], a[6], b0, b1);
            } else {
                uint32_t x[4];
#pragma unroll
                for (int r = 0; r < 4; ++r) x[r] = extend_h2(a[6 - d][r], a[7 - d][r]);
                mma_f16(acc[6], x, b0, b1);
            }
        }
    }
}

// digits 0 .. N - 1 of X (units of 2^-55) into planes
template <int N>
__device__ __forceinline__ void put_digits(uint16_t *pl, int p, long long X)
{
    X += DIGIT_BIAS;
    const uint32_t lo = (uint32_t)X, hi = (uint32_t)(X >> 32);
    const uint32_t d[7] = {(uint32_t)((int)(X >> 48) + 128), (hi >> 8) & 255u, hi & 255u, lo >> 24, (lo >> 16) & 255u, (lo >> 8) & 255u, lo & 255u};
#pragma unroll
    for (int i = 0; i < N; ++i) {
        uint32_t r;
        asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(0x6400u + d[i]), "r"(0x6480u));
        pl[i * DL + p] = (uint16_t)r;
    }
}

__device__ __forceinline__ void lagrange_tables(Shared &S, int T)
{
    const int tid = threadIdx.x, h = (T - 2) / 2;
    if (tid < T) {
        S.lc1[tid] = 1.0 / (double)(tid + 1);
        S.lc0[tid] = (double)(h - tid) / (double)(tid + 1);
        S.rc1[tid] = 1.0 / (double)(T - tid);
        S.rc0[tid] = (double)(h - tid) / (double)(T - tid);
    }
}

// the sky frame of a single-source launch, by the first warp (the three angles' sines on three lanes); the same
// arithmetic as the batched launches' table
__device__ __forceinline__ void sky_by_warp(const lr_sky &sky, SkyConst *out)
{
    const int lane = threadIdx.x & 31;
    double s, c;
    sincos(lane == 0 ? sky.lam : lane == 1 ? sky.beta : 2.0 * sky.psi, &s, &c);
    const double sl = __shfl_sync(0xffffffffu, s, 0), cl = __shfl_sync(0xffffffffu, c, 0);
    const double sb = __shfl_sync(0xffffffffu, s, 1), cb = __shfl_sync(0xffffffffu, c, 1);
    const double s2 = __shfl_sync(0xffffffffu, s, 2), c2 = __shfl_sync(0xffffffffu, c, 2);
    if (lane == 0) {
        SkyConst k;
        k.k[0] = -cb * cl; k.k[1] = -cb * sl; k.k[2] = -sb;
        k.u[0] = sl;       k.u[1] = -cl;      k.u[2] = 0.0;
        k.v[0] = -sb * cl; k.v[1] = -sb * sl; k.v[2] = cb;
        k.c2p = c2; k.s2p = s2;
        *out = k;
    }
}

// ---------------------------------------------------------------- K1: TDI transpose
// Sample by sample, for blocks that the table or the fixed point does not cover: chunks of 64 outputs, the weights of
// two delayed reads at a time by 128 threads, then every link sample gathers from the chunk's rows whose stencils
// hold it, into a sum of its own.  Every link sample looking at all rows of a chunk, and adding to one of six
// registers by comparing the link, took 17.8 ms for 200 000 samples at order 25 (every block); 4.5 now.
constexpr int CR = 64;
__device__ void tdi_adj_scalar(const FwdParams &P, Shared &S, int T, int64_t k0, int nb, int rows, const double *gs, double *gy,
                               int64_t N, double *acc)
{
    const int tid = threadIdx.x, h = (T - 2) / 2, qn = P.q_terms;
    // sums [6][NY], the chunk's delays [6][CR], weights [T][2 CR], stencil positions [2 CR]
    double *L = acc + 6 * NY, *w = L + 6 * CR;
    int *M = reinterpret_cast<int *>(w + (size_t)2 * T * CR);
    __shared__ int lo[4], hi[4];
    __syncthreads();
    for (int i = tid; i < nb; i += blockDim.x) {
        for (int l = 0; l < 6; ++l) acc[l * NY + i] = 0.0;
        for (int cc = 0; cc < 6; ++cc) {   // the undelayed terms
            const double g = gs[(cc >> 1) * NY + i + h + 1];
            acc[c_tdifx.link[cc >> 1][cc & 1][0] * NY + i] += (cc & 1) ? -g : g;
        }
    }
    for (int p0 = 0; p0 < rows; p0 += CR) {
        __syncthreads();
        for (int i = tid; i < 6 * CR; i += blockDim.x) {
            const int l = i / CR, j = i % CR;
            double x;
            int piece;
            const Coef4 *row = row_at(P.to, P.t0 + (double)(k0 - h - 1 + p0 + j) * P.dt, -1, &x, &piece);
            L[i] = cubic(ldg4(row + 9 + l), x) * P.inv_dt;
        }
        for (int t = 0; t < 6 * qn; t += 2) {   // 18 or 42 delayed terms
            __syncthreads();
            if (tid < 2 * CR) {
                const int cc = (t + tid / CR) / qn, q = (t + tid / CR) % qn + 1, j = tid % CR;
                double D = 0.0;
                for (int k = 1; k <= q; ++k) D += L[c_tdifx.pair[cc >> 1][cc & 1][k] * CR + j];
                const int m = stencil_at(-D), a = __reduce_min_sync(0xffffffffu, m), b = __reduce_max_sync(0xffffffffu, m);
                M[tid] = m;
                if ((tid & 31) == 0) {
                    lo[tid >> 5] = a;
                    hi[tid >> 5] = b;
                }
                lagrange_to(S, T, -D - (double)m, w + tid, 2 * CR);
            }
            __syncthreads();
            for (int x = 0; x < 2; ++x) {
                const int cc = (t + x) / qn, q = (t + x) % qn + 1, l = c_tdifx.link[cc >> 1][cc & 1][q];
                const int mlo = min(lo[2 * x], lo[2 * x + 1]), mhi = max(hi[2 * x], hi[2 * x + 1]);
                const double *g = gs + (cc >> 1) * NY + p0;
                for (int i = tid; i < nb; i += blockDim.x) {
                    const int c = i + h + 1 - p0;   // rows j with c - h - 1 <= j + M[j] <= c + h
                    const int ja = max(c - h - 1 - mhi, 0), jb = min(c + h - mlo, CR - 1);
                    if (ja > jb) continue;
                    double sum = 0.0;
                    for (int j = ja; j <= jb; ++j) {
                        const int a = c - j - M[x * CR + j] + h;
                        if (a >= 0 && a < T) sum = fma(w[a * 2 * CR + x * CR + j], g[j], sum);
                    }
                    acc[l * NY + i] += (cc & 1) ? -sum : sum;
                }
            }
        }
    }
    for (int i = tid; i < nb; i += blockDim.x)
        for (int l = 0; l < 6; ++l) gy[l * N + k0 + i] = acc[l * NY + i];
    __syncthreads();
}
// its arrays fit in the place of the sums, the planes or node weights, and the stencils
constexpr int k1_scalar(int T) { return 6 * NY * 8 + 6 * CR * 8 + 2 * T * CR * 8 + 2 * CR * 4; }
static_assert(k1_scalar(32) <= k1_w(32) - K1_PART + FX_TDI_W && k1_scalar(42) <= k1_w(42) - K1_PART + FX_TDI_W, "tdi_adj_scalar's shared memory");

template <int NTHR>
__global__ void __launch_bounds__(NTHR, NTHR == 256 ? 2 : 1) k_fx_tdi_adj(FwdParams P, FxTab X, BwdParams B, int T)
{
    extern __shared__ __align__(16) unsigned char sm_raw[];
    double *gs = reinterpret_cast<double *>(sm_raw);
    long long *part = reinterpret_cast<long long *>(sm_raw + K1_PART);
    uint16_t *planes = reinterpret_cast<uint16_t *>(sm_raw + K1_PLANES);
    double *wt = reinterpret_cast<double *>(sm_raw + K1_PART);  // node weights, before the sums and planes
    unsigned char *W = sm_raw + k1_w(T);
    __shared__ Shared S;
    const int tid = threadIdx.x, h = (T - 2) / 2;
    const int lane = tid & 31, warp = tid >> 5, lr4 = lane >> 2, kp = lane & 3;
    const uint32_t sh = 8 * ((7 - lr4) & 3);
    lagrange_tables(S, T);
    const int64_t total = P.total_tiles >= 0 ? P.total_tiles : P.src.tile_off[P.src.S];
    for (int64_t g = blockIdx.x; g < total; g += gridDim.x) {
        int64_t src = 0;
        if (tid < 32 && P.src.tile_off) src = find_source(P, g);
        if (tid == 0) {
            S.ti = tile_info_of(P, g, src, 3);
            if (!S.ti.ok) atomicOr(P.err, ERR_OFFSETS);
            S.bad = 0;
        }
        __syncthreads();
        if (!S.ti.ok || S.ti.nb <= 0) {
            __syncthreads();
            continue;
        }
        const int64_t N = S.ti.N, k0 = S.ti.n0, n_lo = k0 - h - 1;
        const int nb = (int)S.ti.nb;
        const int rows = nb + X.tab_kw - 1 < NY ? nb + X.tab_kw - 1 : NY;
        const double t_lo = P.t0 + (double)n_lo * P.dt;
        const double *gx = B.g_xyz + (S.ti.out - P.out);
        double *gy = B.g_y + 2 * (S.ti.out - P.out);
        bool any = false;
#pragma unroll
        for (int r = 0; r < NY / NTHR; ++r) {
            const int p = tid + NTHR * r;
            const int64_t n = n_lo + p;
            unsigned w[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const double v = p < rows && n >= 0 && n < N ? __ldg(gx + c * N + n) : 0.0;
                gs[c * NY + p] = v;
                any |= v != 0.0;
                w[c] = warp_max(abs_hi(v));
            }
            if (lane == 0)   // a link sample gathers from two of the channels
#pragma unroll
                for (int c = 0; c < 3; ++c) S.st[c][p >> 5] = max(w[c], w[(c + 1) % 3]);
        }
        if (tid < NY / 32) S.brk[tid] = 0;
        if (tid == 0) {
            S.fast = table_segments(P, X, S, t_lo, rows);
            S.nlist = 0;
            S.mmin = 1 << 29;
            S.mmax = -(1 << 29);
        }
        if (!__syncthreads_or(any)) {
            for (int i = tid; i < nb; i += blockDim.x)
                for (int l = 0; l < 6; ++l) gy[l * N + k0 + i] = 0.0;
            __syncthreads();
            continue;
        }
        int eg = 0;
        const bool fast = S.fast != 0;
        if (!fast) find_tdi_segments(P, S, t_lo, rows);
        __syncthreads();
        unsigned vmax;
        bool bad = !range_ok<0>(S.st, 3, rows, X.tab_kw, X.range_adj, &vmax, &eg) || S.bad;
        const int nseg = S.nseg;
        for (int sg = 0; sg < nseg && !bad; ++sg) {
            const int piece = S.segm[sg][NTERM], mmin = fast ? X.meta[FX_META * piece + 1] : S.mmin, KW = T - mmin, nks = (KW + 7 + 15) / 16;
            const int js = S.segj[sg], je = S.segj[sg + 1];
            int ew;
            if (nks * 16 > 64 || nb + KW - 1 > rows || (!fast && S.mmax >= 0) ||
                !(fast ? tdi_stencils<true, NTHR>(P, X, S, t_lo, sg, KW, W, &ew)
                       : tdi_stencils_nodes<true, NTHR>(P, X, S, T, t_lo, sg, KW, mmin, W, wt, &ew))) {
                bad = true;
                break;
            }
            count_orders<NT>(S);
            const int nq = S.nq;
            const bool last = S.last;
            for (int ch = 0; ch < 3; ++ch) {
                // the channel's series times T_q in digits, zero outside the segment
                for (int p = tid; p < DL; p += blockDim.x) {
                    const bool in = p >= js && p < je;
                    const long long x0 = in ? to_fixed(gs[ch * NY + p], eg) : 0;
                    const int kappa = 2 * p + 1 - NY;
                    const long long x1 = in ? mul_nu<9>(x0, kappa) : 0;
                    const long long x2 = in ? mul_nu<8>(x1, kappa) - x0 : 0;
                    const long long x3 = in ? mul_nu<8>(x2, kappa) - x1 : 0;
                    put_digits<gdigits(true, 0)>(planes + gplane(true, 0) * DL, p, x0);
                    put_digits<gdigits(true, 1)>(planes + gplane(true, 1) * DL, p, x1);
                    put_digits<gdigits(true, 2)>(planes + gplane(true, 2) * DL, p, x2);
                    put_digits<gdigits(true, 3)>(planes + gplane(true, 3) * DL, p, x3);
                }
                __syncthreads();
                for (int it = warp; it < 16; it += blockDim.x >> 5) {
                    const int sl = it & 3, mb = it >> 2;
                    if (128 * mb >= nb) continue;
                    const int l = c_slots.link[ch][sl];
                    const unsigned char *a_lane = reinterpret_cast<const unsigned char *>(planes) + 16 * (16 * mb + lr4) + 8 * kp;
                    const unsigned char *w_lane = W + (ch * 4 + sl) * TD * WS + 4 * (kp + ((7 - lr4) >> 2));
                    float acc[7][4] = {};
                    contract_order<0, true, false>(acc, a_lane, w_lane, sh, nks);
                    if (last) {
                        if (nq > 1) contract_order<1, true, true>(acc, a_lane + gplane(true, 1) * DL * 2, w_lane + digit_row(true, 1) * WS, sh, nks);
                        if (nq > 2) contract_order<2, true, true>(acc, a_lane + gplane(true, 2) * DL * 2, w_lane + digit_row(true, 2) * WS, sh, nks);
                        if (nq > 3) contract_order<3, true, true>(acc, a_lane + gplane(true, 3) * DL * 2, w_lane + digit_row(true, 3) * WS, sh, nks);
                    } else {
                        if (nq > 1) contract_order<1, true, false>(acc, a_lane + gplane(true, 1) * DL * 2, w_lane + digit_row(true, 1) * WS, sh, nks);
                        if (nq > 2) contract_order<2, true, false>(acc, a_lane + gplane(true, 2) * DL * 2, w_lane + digit_row(true, 2) * WS, sh, nks);
                        if (nq > 3) contract_order<3, true, false>(acc, a_lane + gplane(true, 3) * DL * 2, w_lane + digit_row(true, 3) * WS, sh, nks);
                    }
                    bool first = true;   // each link is in two channels
                    for (int c2 = 0; c2 < ch; ++c2)
                        for (int s2 = 0; s2 < 4; ++s2) first &= c_slots.link[c2][s2] != l;
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        long long *o = part + l * NY + 128 * mb + 8 * (lr4 + (r >> 1) * 8) + 2 * kp + (r & 1);
                        const long long v = levels<0>(acc, r);
                        *o = first ? v : *o + v;
                    }
                }
                __syncthreads();
            }
            const int unit = eg + ew - 57;
            for (int i = tid; i < nb; i += blockDim.x)
#pragma unroll
                for (int l = 0; l < 6; ++l) {
                    const double v = from_fixed(part[l * NY + i], unit);
                    double *o = gy + l * N + k0 + i;
                    *o = sg ? *o + v : v;
                }
        }
        __syncthreads();
        if (bad) tdi_adj_scalar(P, S, T, k0, nb, rows, gs, gy, N, reinterpret_cast<double *>(sm_raw + K1_PART));
        __syncthreads();
    }
}

// ---------------------------------------------------------------- K2: projection transpose
// Sample by sample, for blocks that the expansion or the fixed point does not cover: chunks of 64 link samples,
// over all that the plan's bounds let the block's strain samples meet.  The reads' positions and coefficients of a
// chunk are shared between the threads by spacecraft and by link, the weights of two reads at a time are formed by
// 128 threads, and every strain sample gathers from the rows of the chunk whose stencils hold it.  Eight threads
// forming the reads of eight link samples, and every strain sample looking at all rows, took 5.07 ms for 200 000
// samples at order 25 (every block); 1.48 now.
__device__ void proj_adj_scalar(const FwdParams &P, const FxTab &X, Shared &S, int T, double u0, int64_t f0, int64_t i0, int nb,
                                const double *gy, double *ghp, double *ghc, double *w)
{
    const int tid = threadIdx.x, h = (T - 2) / 2;
    const int64_t N = S.ti.N;
    // weights [T][2 CR], before them the spacecraft's positions [9][CR]; the nine reads' positions and coefficients, whole parts
    double *pos = w, *U = w + (size_t)(2 * T > 9 ? 2 * T : 9) * CR, *CF = U + 9 * CR;
    int *M = reinterpret_cast<int *>(CF + 18 * CR);
    __shared__ int lo[9], hi[9];   // stencil positions of a chunk's reads
    double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
    const int64_t ka = i0 - f0 - P.sig_b - h - 3, kb = i0 + nb - f0 + P.sig_b + P.lproj_b + h + 3;
    const int64_t k_end = kb < N ? kb : N;
    for (int64_t k0 = ka > 0 ? ka : 0; k0 < k_end; k0 += CR) {
        __syncthreads();
        if (tid < 9) {
            lo[tid] = 1 << 29;
            hi[tid] = -(1 << 29);
        }
        for (int i = tid; i < 3 * CR; i += blockDim.x) {
            const int s = i / CR, j = i % CR;
            double x, u[3], ps[9];
            int piece;
            const Coef4 *row = row_at(P.po, P.t0 + (double)(k0 + j) * P.dt, -1, &x, &piece);
            reads_of(P, X, S.skc, row, x, s, u0, u, ps);
#pragma unroll
            for (int d = 0; d < 3; ++d) pos[(3 * s + d) * CR + j] = ps[3 * s + d];
            U[s * CR + j] = u[0];
#pragma unroll
            for (int e = 0; e < 2; ++e) U[(3 + c_by_emitter[s][e]) * CR + j] = u[1 + e];
        }
        __syncthreads();
        for (int i = tid; i < 6 * CR; i += blockDim.x) {
            const int l = i / CR, j = i % CR, r = c_lr[l], s = c_ls[l];
            const SkyConst &K = S.skc;
            double d0 = pos[3 * r * CR + j] - pos[3 * s * CR + j], d1 = pos[(3 * r + 1) * CR + j] - pos[(3 * s + 1) * CR + j],
                   d2 = pos[(3 * r + 2) * CR + j] - pos[(3 * s + 2) * CR + j];
            const double inv = 1.0 / sqrt(d0 * d0 + d1 * d1 + d2 * d2);
            d0 *= inv; d1 *= inv; d2 *= inv;
            const double un = K.u[0] * d0 + K.u[1] * d1 + K.u[2] * d2, vn = K.v[0] * d0 + K.v[1] * d1 + K.v[2] * d2;
            const double kn = K.k[0] * d0 + K.k[1] * d1 + K.k[2] * d2;
            const double xip = un * un - vn * vn, xic = 2.0 * un * vn;
            const double gl = k0 + j < k_end ? __ldg(gy + l * N + k0 + j) * (1.0 / (2.0 * (1.0 - kn))) : 0.0;
            CF[2 * (3 + l) * CR + j] = gl * (K.c2p * xip + K.s2p * xic);
            CF[(2 * (3 + l) + 1) * CR + j] = gl * (-K.s2p * xip + K.c2p * xic);
        }
        for (int i = tid; i < 9 * CR; i += blockDim.x) {   // a warp's lanes are of one read
            const int rd = i / CR;
            const double u = U[i];
            const int m = stencil_at(u);
            M[i] = m;
            const int a = __reduce_min_sync(0xffffffffu, m), b = __reduce_max_sync(0xffffffffu, m);
            if ((tid & 31) == 0) {
                atomicMin(&lo[rd], a);
                atomicMax(&hi[rd], b);
            }
            if (k0 + i % CR < k_end && (m > P.sig_b + 1 || m < -P.sig_b - P.lproj_b - 2)) atomicOr(P.err, ERR_WINDOW);
        }
        __syncthreads();
        for (int i = tid; i < 6 * CR; i += blockDim.x) {   // receptions: the two links of a receiver
            const int r = (i / CR) >> 1, pol = (i / CR) & 1, j = i % CR, l2 = r ? 6 - r : 3;
            CF[(2 * r + pol) * CR + j] = -(CF[(2 * (3 + r) + pol) * CR + j] + CF[(2 * (3 + l2) + pol) * CR + j]);
        }
        const int64_t at = k0 + f0 - i0;   // strain sample (within the block) that the chunk's first row reads at position 0
        for (int rd = 0; rd < 9; rd += 2) {
            bool any = false;
            for (int x = rd; x < rd + 2 && x < 9; ++x) any |= at + hi[x] + CR + h + 1 >= 0 && at + lo[x] - h < nb;
            if (!any) continue;   // uniform over the block
            __syncthreads();
            if (tid < 2 * CR && rd + tid / CR < 9) {
                const double u = U[rd * CR + tid];
                lagrange_to(S, T, u - (double)M[rd * CR + tid], w + tid, 2 * CR);
            }
            __syncthreads();
            for (int x = 0; x < 2 && rd + x < 9; ++x) {
                const double *cp = CF + 2 * (rd + x) * CR, *cc = cp + CR;
                const int *m = M + (rd + x) * CR;
#pragma unroll
                for (int o = 0; o < 2; ++o) {
                    const int i = tid + (int)blockDim.x * o;
                    const int64_t c = i - at;   // rows j with c - h - 1 <= j + m[j] <= c + h
                    const int64_t ja = c - h - 1 - hi[rd + x], jb = c + h - lo[rd + x];
                    if (i >= nb || jb < 0 || ja >= CR) continue;
                    for (int j = ja > 0 ? (int)ja : 0; j < CR && j <= jb; ++j) {
                        const int a = (int)(c - j) - m[j] + h;
                        if (a < 0 || a >= T) continue;
                        const double wt = w[a * 2 * CR + x * CR + j];
                        acc[o][0] = fma(wt, cp[j], acc[o][0]);
                        acc[o][1] = fma(wt, cc[j], acc[o][1]);
                    }
                }
            }
        }
    }
#pragma unroll
    for (int o = 0; o < 2; ++o)
        if (tid + (int)blockDim.x * o < nb) {
            ghp[i0 + tid + (int)blockDim.x * o] = acc[o][0];
            ghc[i0 + tid + (int)blockDim.x * o] = acc[o][1];
        }
    __syncthreads();
}
// its arrays fit in the stencils' and planes' place at every order compiled
static_assert((2 * 42 + 27) * CR * 8 + 9 * CR * 4 <= FX_PROJ_W + K2_GROUP, "proj_adj_scalar's shared memory");

// planes of T_q g for orders Q0 .. Q1 - 1 at row p, from x0 = g in fixed point
template <int Q0, int Q1>
__device__ __forceinline__ void order_planes(uint16_t *planes, int p, long long x0, int kappa, bool in)
{
    long long xa = x0, xb = in ? mul_nu<9>(x0, kappa) : 0;
#pragma unroll
    for (int q = 0; q < Q1; ++q) {
        // xa = T_q g, xb = T_{q+1} g
        uint16_t *pl = planes + (gplane(false, q) - gplane(false, Q0)) * DL;
        if (q >= Q0) {
            if (gdigits(false, q) == 7) put_digits<7>(pl, p, xa);
            else if (gdigits(false, q) == 6) put_digits<6>(pl, p, xa);
            else if (gdigits(false, q) == 5) put_digits<5>(pl, p, xa);
            else if (gdigits(false, q) == 4) put_digits<4>(pl, p, xa);
            else put_digits<3>(pl, p, xa);
        }
        const long long nx = in ? mul_nu<8>(xb, kappa) - xa : 0;
        xa = xb;
        xb = nx;
    }
}

template <int Q, bool LAST>
__device__ __forceinline__ void proj_order(float (&acc)[7][4], const unsigned char *a_lane, const unsigned char *w_lane,
                                           uint32_t sh, int nks)
{
    constexpr int base = Q < QA ? 0 : PQA;
    contract_order<Q, false, LAST>(acc, a_lane + (gplane(false, Q) - base) * DL * 2, w_lane + digit_row(false, Q) * WS, sh, nks);
}

template <int NTHR>
__global__ void __launch_bounds__(NTHR, NTHR == 256 ? 2 : 1) k_fx_proj_adj(FwdParams P, FxTab X, BwdParams B, int T)
{
    extern __shared__ __align__(16) unsigned char sm_raw[];
    double *gys = reinterpret_cast<double *>(sm_raw);
    constexpr int NGR = NTHR / 256;   // groups of eight warps: each takes every NGR-th link, in planes of its own
    unsigned char *W = sm_raw + K2_STENCILS;
    double *wn = reinterpret_cast<double *>(sm_raw + K2_PLANES);  // the node weights are done with before the planes
    __shared__ Shared S;
    __shared__ int nbs, umax;
    __shared__ double u0s;
    const int tid = threadIdx.x, h = (T - 2) / 2;
    const int lane = tid & 31, warp = (tid >> 5) & 7, grp = tid >> 8, lr4 = lane >> 2, kp = lane & 3;
    uint16_t *planes = reinterpret_cast<uint16_t *>(sm_raw + K2_PLANES + grp * K2_GROUP);
    const uint32_t sh = 8 * ((7 - lr4) & 3);
    lagrange_tables(S, T);
    if (tid < 32 && !B.h_tile_off) sky_by_warp(P.src.sky1, &S.skc);
    FwdParams Q = P;   // tiles over strain samples
    Q.src.tile_off = B.h_tile_off;
    Q.tile = B.tile_h;
    const int64_t total = B.h_total_tiles >= 0 ? B.h_total_tiles : B.h_tile_off[P.src.S];
    for (int64_t g = blockIdx.x; g < total; g += gridDim.x) {
        int64_t src = 0;
        if (tid < 32 && Q.src.tile_off) src = find_source(Q, g);
        if (tid == 0) {
            S.ti = tile_info_of(Q, g, src, 3);
            if (Q.src.tile_off) S.skc = P.src.skyc[src];
            if (!S.ti.ok) atomicOr(P.err, ERR_OFFSETS);
            const int64_t nbh = S.ti.nh - S.ti.n0;   // clipped against the strain, not the outputs
            nbs = !S.ti.ok || nbh <= 0 ? 0 : (int)(nbh < B.tile_h ? nbh : B.tile_h);
            u0s = (P.t0 - S.ti.t0h) / P.dt;
            umax = -(1 << 29);
        }
        __syncthreads();
        const int nb = nbs;
        if (nb <= 0) {
            __syncthreads();
            continue;
        }
        const int64_t i0 = S.ti.n0, N = S.ti.N, f0 = (int64_t)floor(u0s);
        const double u0 = u0s - floor(u0s);
        // the link samples whose reads can land on the tile: from the reads' positions near its centre
        if (tid < 9) {
            int piece;
            const double u = read_pos(P, X, S.skc, u0, P.t0 + (double)(i0 + nb / 2 - f0) * P.dt, tid, &piece);
            const int m = stencil_at(u + 0.25);   // beyond the plan's bounds: a window that holds no tile
            atomicMax(&umax, m > P.sig_b + 2 || m < -P.sig_b - P.lproj_b - 2 ? STENCIL_FAR : m);
        }
        __syncthreads();
        const int64_t k_lo = i0 - f0 - umax - (h + 1);
        const double t_lo = P.t0 + (double)k_lo * P.dt;
        projection_segments(P, X, S, t_lo, u0, NY);
        const double *gy = B.g_y + 2 * (S.ti.out - P.out);
        bool any = false;
#pragma unroll
        for (int r = 0; r < NY / NTHR; ++r) {
            const int j = tid + NTHR * r;
            const int64_t k = k_lo + j;
            unsigned w = 0;
            for (int l = 0; l < 6; ++l) {
                const double v = k >= 0 && k < N ? __ldg(gy + l * N + k) : 0.0;
                gys[l * NY + j] = v;
                any |= v != 0.0;
                w = max(w, abs_hi(v));
            }
            w = warp_max(w);
            if (lane == 0) S.st[0][j >> 5] = w;
        }
        double *ghp = B.g_hp + (S.ti.hp - P.hp), *ghc = B.g_hc + (S.ti.hp - P.hp);
        const int nseg = S.nseg, KW = S.mmax - S.mmin + T, nks = (KW + 3 + 15) / 16;
        const int j0 = umax - S.mmax;   // row of the first link sample that output 0 gathers from
        const bool lost = j0 < 0 || j0 + nb + KW - 1 > NY;   // link samples outside the rows may land on the tile
        if (!__syncthreads_or(any) && !lost) {
            for (int i = tid; i < nb; i += blockDim.x) ghp[i0 + i] = ghc[i0 + i] = 0.0;
            __syncthreads();
            continue;
        }
        int eg = 0;
        unsigned vmax;
        bool bad = !range_ok<0>(S.st, 1, NY, KW, X.range_adj, &vmax, &eg);
        bad |= S.bad || nks * 16 > 64 || lost;
        double out[4] = {0.0, 0.0, 0.0, 0.0};
        for (int sg = 0; sg < nseg && !bad; ++sg) {
            if (!projection_stencils<true>(P, X, S, T, t_lo, u0, sg, KW, W, wn)) {
                bad = true;
                break;
            }
            const int nq = S.nq, js = S.segj[sg], je = S.segj[sg + 1];
            const bool last = S.last;
            long long sum[4] = {0, 0, 0, 0};
            const unsigned char *a_lane = reinterpret_cast<const unsigned char *>(planes) + 8 * (16 * warp + lr4) + 8 * kp;
            for (int l = grp; l < 6; l += NGR) {
                const unsigned char *w_lane = W + (2 * l + (lr4 >> 2)) * PD * WS + 4 + 4 * kp;
                float acc[7][4] = {};
                for (int p = tid & 255; p < DL; p += 256) {
                    const int j = p + j0;
                    const bool in = j >= js && j < je;
                    order_planes<0, QA>(planes, p, in ? to_fixed(gys[l * NY + j], eg) : 0, 2 * j + 1 - NY, in);
                }
                __syncthreads();
                if (64 * warp < nb) {
                    proj_order<0, false>(acc, a_lane, w_lane, sh, nks);
                    if (last) {
                        if (nq > 1) proj_order<1, true>(acc, a_lane, w_lane, sh, nks);
                        if (nq > 2) proj_order<2, true>(acc, a_lane, w_lane, sh, nks);
                    } else {
                        if (nq > 1) proj_order<1, false>(acc, a_lane, w_lane, sh, nks);
                        if (nq > 2) proj_order<2, false>(acc, a_lane, w_lane, sh, nks);
                    }
                }
                __syncthreads();
                if (nq > QA) {
                    for (int p = tid & 255; p < DL; p += 256) {
                        const int j = p + j0;
                        const bool in = j >= js && j < je;
                        order_planes<QA, NN>(planes, p, in ? to_fixed(gys[l * NY + j], eg) : 0, 2 * j + 1 - NY, in);
                    }
                    __syncthreads();
                    if (64 * warp < nb) {
                        if (last) {
                            proj_order<3, true>(acc, a_lane, w_lane, sh, nks);
                            if (nq > 4) proj_order<4, true>(acc, a_lane, w_lane, sh, nks);
                            if (nq > 5) proj_order<5, true>(acc, a_lane, w_lane, sh, nks);
                            if (nq > 6) proj_order<6, true>(acc, a_lane, w_lane, sh, nks);
                            if (nq > 7) proj_order<7, true>(acc, a_lane, w_lane, sh, nks);
                        } else {
                            proj_order<3, false>(acc, a_lane, w_lane, sh, nks);
                            if (nq > 4) proj_order<4, false>(acc, a_lane, w_lane, sh, nks);
                            if (nq > 5) proj_order<5, false>(acc, a_lane, w_lane, sh, nks);
                            if (nq > 6) proj_order<6, false>(acc, a_lane, w_lane, sh, nks);
                            if (nq > 7) proj_order<7, false>(acc, a_lane, w_lane, sh, nks);
                        }
                    }
                    __syncthreads();
                }
#pragma unroll
                for (int r = 0; r < 4; ++r) sum[r] += levels<0>(acc, r);
            }
            const int unit = eg + S.wexp[0] - 57;
#pragma unroll
            for (int r = 0; r < 4; ++r) out[r] += from_fixed(sum[r], unit);
        }
        __syncthreads();
        double *parts = reinterpret_cast<double *>(sm_raw + K2_PLANES);   // the second group's sums
        if (NGR > 1) {
            if (grp == 1 && !bad)
                for (int r = 0; r < 4; ++r) parts[4 * (tid & 255) + r] = out[r];
            __syncthreads();
            if (grp == 0 && !bad)
                for (int r = 0; r < 4; ++r) out[r] += parts[4 * tid + r];
        }
        if (!bad && grp == 0) {
            double *o = (kp >> 1) ? ghc : ghp;
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int i = 64 * warp + 4 * (lr4 + (r >> 1) * 8) + 2 * (kp & 1) + (r & 1);
                if (i < nb) o[i0 + i] = out[r];
            }
        }
        if (bad) proj_adj_scalar(P, X, S, T, u0, f0, i0, nb, gy, ghp, ghc, reinterpret_cast<double *>(sm_raw + K2_STENCILS));
        __syncthreads();
    }
}

// ---------------------------------------------------------------- K3: sky-angle gradient
// derivatives of the frame (k, u, v) with respect to lambda (0) and beta (1), from the frame itself
__device__ __forceinline__ void frame_derivatives(const SkyConst &K, double dk[2][3], double du[2][3], double dv[2][3])
{
    const double sl = K.u[0], cl = -K.u[1], cb = K.v[2], sb = -K.k[2];
    dk[0][0] = cb * sl;  dk[0][1] = -cb * cl; dk[0][2] = 0.0;
    dk[1][0] = sb * cl;  dk[1][1] = sb * sl;  dk[1][2] = -cb;
    du[0][0] = cl;       du[0][1] = sl;       du[0][2] = 0.0;
    du[1][0] = 0.0;      du[1][1] = 0.0;      du[1][2] = 0.0;
    dv[0][0] = sb * sl;  dv[0][1] = -sb * cl; dv[0][2] = 0.0;
    dv[1][0] = -cb * cl; dv[1][1] = -cb * sl; dv[1][2] = -sb;
}

// link l's part of the gradient at positions x, angles a0 .. a1 - 1 of (lambda, beta); psi with beta.  e, r: the
// emission and reception reads summed against gy, (value, derivative) of h+ and hx.  geo, where not null, gets the
// link's coefficients of h+ and hx and their derivatives with respect to those angles: [6], two for the values
// (with the first angle), then two per angle.
__device__ __forceinline__ void sky_terms(const FwdParams &P, const SkyConst &K, const double *x, int l, const double *e,
                                          const double *r, int a0, int a1, double *G, double *geo)
{
    double dk[2][3], du[2][3], dv[2][3];
    frame_derivatives(K, dk, du, dv);
    const int ir = c_lr[l], is = c_ls[l];
    double n[3];
    for (int d = 0; d < 3; ++d) n[d] = x[3 * ir + d] - x[3 * is + d];
    const double inv = 1.0 / sqrt(n[0] * n[0] + n[1] * n[1] + n[2] * n[2]);
    for (int d = 0; d < 3; ++d) n[d] *= inv;
    auto dot = [&](const double *a) { return a[0] * n[0] + a[1] * n[1] + a[2] * n[2]; };
    const double un = dot(K.u), vn = dot(K.v), kn = dot(K.k);
    const double xip = un * un - vn * vn, xic = 2.0 * un * vn;
    const double xp = K.c2p * xip + K.s2p * xic, xc = -K.s2p * xip + K.c2p * xic;
    const double den = 1.0 / (2.0 * (1.0 - kn));
    const double dPp = e[0] - r[0], dPc = e[2] - r[2], dH = xp * dPp + xc * dPc;
    if (geo && a0 == 0) {
        geo[0] = den * xp;
        geo[1] = den * xc;
    }
    for (int th = a0; th < a1; ++th) {
        const double da = dot(du[th]), db = dot(dv[th]);
        const double dxip = 2.0 * (un * da - vn * db), dxic = 2.0 * (da * vn + un * db);
        const double dxp = K.c2p * dxip + K.s2p * dxic, dxc = -K.s2p * dxip + K.c2p * dxic;
        const double dden = 2.0 * den * den * dot(dk[th]);
        const double due = -(dk[th][0] * x[3 * is] + dk[th][1] * x[3 * is + 1] + dk[th][2] * x[3 * is + 2]) / C_LIGHT * P.inv_dt;
        const double dur = -(dk[th][0] * x[3 * ir] + dk[th][1] * x[3 * ir + 1] + dk[th][2] * x[3 * ir + 2]) / C_LIGHT * P.inv_dt;
        const double ddH = dxp * dPp + dxc * dPc + xp * (e[1] * due - r[1] * dur) + xc * (e[3] * due - r[3] * dur);
        G[th] += dden * dH + den * ddH;
        if (geo) {
            geo[2 + 2 * th] = fma(dden, xp, den * dxp);
            geo[3 + 2 * th] = fma(dden, xc, den * dxc);
        }
    }
    if (a1 == 2) G[2] += den * (2.0 * xc * dPp - 2.0 * xp * dPc);
}

// Whether the expansion of one coefficient series of a link over the block (g: its node values, a stride apart)
// holds, together with that of the reads' weights.  The gradient's products are taken at eight nodes, and the
// correlations of order q carry 8 zq(q) bits less than those of order 0, so the orders of (coefficient) x (weights)
// have to fall as the digits assume and the first one left out has to be small.  Orders of the coefficient relative
// to `scale`; those of the weights by those of sinc: with a drift of +-delta samples over the block the j-th is
// at most 2 (pi delta / 2)^j / (j! (j + 1)).  Checked against the exact terms of single blocks (a 3 mHz source, order
// 25): the bound of order 8 is 1e-11 at 0.01 rad from an arm, where the terms are 9e-12 off, 1.6e-9 at 5e-3 (1e-9),
// 5e-4 at 1e-3 (2e-4).  Far from the arms it is rounding: an arm's direction is the difference of positions sixty
// times its length, and the bound of 4000 random blocks is 6e-15 in the middle and 7e-14 at most.  A limit of 3e-14
// sent one block in a hundred to the sample form, and most launches waited for one (a year at order 41: 12.1 to
// 13.2 ms in one source's case).
__device__ __forceinline__ bool sky_series_fits(const FxTab &X, const double *g, int stride, float scale, float delta)
{
    double e[NN / 2], o[NN / 2];
#pragma unroll
    for (int n = 0; n < NN / 2; ++n) {
        const double a = g[n * stride], b = g[(NN - 1 - n) * stride];
        e[n] = a + b;
        o[n] = a - b;
    }
    float c[NN], w[NN + 1];
    const float inv = 1.0f / scale;
#pragma unroll
    for (int q = 0; q < NN; ++q) {
        double v = 0.0;
#pragma unroll
        for (int n = 0; n < NN / 2; ++n) v = fma((q & 1) ? o[n] : e[n], X.cheb[q][n], v);
        c[q] = fabsf((float)v) * inv;
    }
    float run = 2.0f;
    w[0] = 1.0f;
#pragma unroll
    for (int j = 1; j <= NN; ++j) {
        run *= 1.5707964f * delta / (float)j;
        w[j] = run / (float)(j + 1);
    }
    bool ok = true;
#pragma unroll
    for (int q = 1; q <= NN; ++q) {
        float p = 0.0f;
#pragma unroll
        for (int i = 0; i < NN && i <= q; ++i) p = fmaf(c[i], w[q - i], p);
        if (q < NN) {
            ok &= p <= 16.0f / (float)(1ull << (8 * zq(false, q)));
        } else {
            // the coefficient's own next order, from the decay over its last two pairs
            const float last = fmaxf(c[NN - 1], c[NN - 2]), before = fmaxf(c[NN - 3], c[NN - 4]);
            p += last <= before ? last * (last / fmaxf(before, 1e-30f)) : last;
            ok &= p <= 4.5e-13f;   // 2^-41: a source within about 0.016 rad of an arm
        }
    }
    return ok;   // false for NaN
}

// value and derivative of both polarisations at base + u, straight from memory (Horner form of read_scalar)
__device__ void read_vd_scalar(const Shared &S, int T, const double *hp, const double *hc, int64_t nh, int64_t base, double u,
                               double *v)
{
    const int h = (T - 2) / 2;
    const double fl = floor(u), e = u - fl;
    const int64_t st = base + (int64_t)fl - h;
    double L = -1.0, dL = 0.0;
    double a[4] = {0.0, 0.0, 0.0, 0.0};
    for (int j = 0; j < T; ++j) {
        const int64_t i = st + j;
        const double p = i >= 0 && i < nh ? __ldg(hp + i) : 0.0, c = i >= 0 && i < nh ? __ldg(hc + i) : 0.0;
        if (j) {
            const double f = fma(e, S.rc1[j], S.rc0[j]), f1 = S.rc1[j];
            const double q = -fma(e, S.lc1[j - 1], S.lc0[j - 1]), q1 = -S.lc1[j - 1];
            dL = fma(dL, q, L * q1);
            L *= q;
            a[1] = fma(a[1], f, fma(a[0], f1, dL * p));
            a[0] = fma(a[0], f, L * p);
            a[3] = fma(a[3], f, fma(a[2], f1, dL * c));
            a[2] = fma(a[2], f, L * c);
        } else {
            a[0] = L * p;
            a[2] = L * c;
        }
    }
    for (int i = 0; i < 4; ++i) v[i] = a[i];
}

// digit bytes of T_q g (K3's right operand) of one row
template <int N>
__device__ __forceinline__ void put_bytes(unsigned char *row, long long X)
{
    X += DIGIT_BIAS;
    row[0] = (unsigned char)((int)(X >> 48) + 128);   // |X| < 127.5 * 2^48
#pragma unroll
    for (int i = 1; i < N; ++i) row[i * GB] = (unsigned char)(X >> (8 * (6 - i)));
}

// correlations of order Q over k-steps [s0, s1): acc by level, the top one carrying the next
template <int Q>
__device__ __forceinline__ void correlate(float (&acc)[7][4], const unsigned char *a_lane, const unsigned char *g_lane,
                                          uint32_t sh, int s0, int s1)
{
    constexpr int n = 7 - zq(false, Q), NA = n < 7 ? n + 1 : 7, ND = gdigits(false, Q);
#pragma unroll 1
    for (int ks = s0; ks < s1; ++ks) {
        uint32_t a[NA][4];
#pragma unroll
        for (int k = 0; k < NA; ++k) {
            const uint2 p = *reinterpret_cast<const uint2 *>(a_lane + 32 * ks + k * DL * 2);
            const uint2 c = *reinterpret_cast<const uint2 *>(a_lane + 32 * ks + (7 + k) * DL * 2);
            a[k][0] = p.x; a[k][1] = c.x; a[k][2] = p.y; a[k][3] = c.y;
        }
#pragma unroll
        for (int d = 0; d < ND; ++d) {
            const uint32_t *w = reinterpret_cast<const uint32_t *>(g_lane + 16 * ks + (gplane(false, Q) + d) * GB);
            const uint32_t u = __funnelshift_r(w[0], w[1], sh);
            const uint32_t b0 = digits_h2(u, 0x4140u), b1 = digits_h2(u, 0x4342u);
            if (d < n) {
#pragma unroll
                for (int k = 0; k < n - 1 - d; ++k) mma_f16(acc[d + k], a[k], b0, b1);
                if (n - d < NA) {
                    uint32_t x[4];
#pragma unroll
                    for (int r = 0; r < 4; ++r) x[r] = extend_h2(a[n - 1 - d][r], a[n - d][r]);
                    mma_f16(acc[n - 1], x, b0, b1);
                } else {
                    mma_f16(acc[n - 1], a[n - 1 - d], b0, b1);
                }
            } else {  // digit n against the series' first digit: level n
                uint32_t x[4];
#pragma unroll
                for (int r = 0; r < 4; ++r) x[r] = extend_h2(0u, a[0][r]);
                mma_f16(acc[n - 1], x, b0, b1);
            }
        }
    }
}

template <int Q>
__device__ __forceinline__ void correlate_item(double *C, int LG, const unsigned char *a_lane, const unsigned char *g_lane,
                                               uint32_t sh, int s0, int s1, int lag0, int lane, int link0)
{
    constexpr int n = 7 - zq(false, Q);
    float acc[7][4] = {};
    correlate<Q>(acc, a_lane, g_lane, sh, s0, s1);
    const int lr4 = lane >> 2, kp = lane & 3, l = link0 + (kp >> 1);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        long long v = 0;
#pragma unroll
        for (int L = 0; L < n - 1; ++L) v = v * 256 + (long long)__float2int_rn(acc[L][r]);
        v += (long long)__float2int_rn(acc[n - 1][r] * (1.0f / 256.0f));
        const int lag = lag0 + 4 * lr4 + 2 * (kp & 1) + (r & 1), pol = r >> 1;
        // two contributions per place (the halves of the block), so the sum does not depend on their order
        if (lag < LG) atomicAdd(&C[((l * NN + Q) * 2 + pol) * LG + lag], (double)v * pow2(8 * zq(false, Q) - 54));
    }
}

// the (order, half of the block) items 2 q + half of each warp, balanced by issue slots per step (119, 119, 113,
// 94, 76, 76, 59, 43 for orders 0 .. 7: products, digit conversions and loads) over the warps (162 to 189) and
// over the schedulers, which have warps w and w + 4 (348 and 351)
__constant__ signed char c_items[8][2] = {{0, 12}, {1, 13}, {2, 14}, {3, 15}, {6, 10}, {7, 11}, {4, 8}, {5, 9}};

template <int NTHR>
__global__ void __launch_bounds__(NTHR, NTHR == 256 ? 2 : 1) k_fx_sky_adj(FwdParams P, FxTab X, BwdParams B, int T)
{
    extern __shared__ __align__(16) unsigned char sm_raw[];
    uint16_t *planes = reinterpret_cast<uint16_t *>(sm_raw);
    unsigned char *G = sm_raw + K3_G;
    double *wn = reinterpret_cast<double *>(sm_raw + K3_G), *dwn = wn + T * WNS;   // once the digit rows are done with
    double *C = reinterpret_cast<double *>(sm_raw + k3_c(T, NTHR));          // [link][order or node][pol][LG]
    const int LG = X.lags;
    __shared__ Shared S;
    __shared__ double dots[NN][6][2][4];   // node, link, (emission, reception): h+ value, derivative, hx value, derivative
    __shared__ double red[3][NTHR / 32];
    __shared__ int gscale[2];   // largest coefficient at the nodes, largest derivative (floats)
    const int tid = threadIdx.x, h = (T - 2) / 2;
    const int lane = tid & 31, warp = tid >> 5, lr4 = lane >> 2, kp = lane & 3;
    const uint32_t sh = 8 * ((7 - lr4) & 3);
    lagrange_tables(S, T);
    if (tid < 32 && !P.src.tile_off) sky_by_warp(P.src.sky1, &S.skc);
    const int64_t total = P.total_tiles >= 0 ? P.total_tiles : P.src.tile_off[P.src.S];
    for (int64_t g = blockIdx.x; g < total; g += gridDim.x) {
        int64_t src = 0;
        if (tid < 32 && P.src.tile_off) src = find_source(P, g);
        if (tid == 0) {
            S.ti = tile_info_of(P, g, src, 3);
            if (P.src.tile_off) S.skc = P.src.skyc[src];
            if (!S.ti.ok) atomicOr(P.err, ERR_OFFSETS);
        }
        __syncthreads();
        double Gs[3] = {0.0, 0.0, 0.0};
        if (S.ti.ok && S.ti.nb > 0) {
            const TileInfo &ti = S.ti;
            const int nb = (int)ti.nb;
            const int64_t k_lo = ti.n0, N = ti.N;
            const double u = (P.t0 - ti.t0h) / P.dt, u0 = u - floor(u), t_lo = P.t0 + (double)k_lo * P.dt;
            const int64_t f0 = (int64_t)floor(u);
            const double *gy = B.g_y + 2 * (ti.out - P.out);
            projection_segments(P, X, S, t_lo, u0, nb);
            const int nseg = S.nseg, mmin = S.mmin, KW = S.mmax - mmin + T, npass = (KW + 31) / 32;
            bool bad = S.bad || KW > LG;
            const int64_t w_lo = k_lo + f0 + mmin - h;
            const int WL = nb + KW - 1;
            bool anyg = false, anyh = false;
            constexpr int NV = (DL + NTHR - 1) / NTHR;
            double vp[NV], vc[NV];
            if (!bad) {
#pragma unroll
                for (int i = 0; i < NV; ++i) {
                    const int p = tid + i * NTHR;
                    const int64_t idx = w_lo + p;
                    vp[i] = vc[i] = 0.0;
                    if (p < WL && idx >= 0 && idx < ti.nh) {
                        vp[i] = __ldg(ti.hp + idx);
                        vc[i] = __ldg(ti.hc + idx);
                    }
                    anyh |= vp[i] != 0.0 || vc[i] != 0.0;
                    const unsigned a = abs_hi(vp[i]), b = abs_hi(vc[i]);
                    const unsigned w = warp_max(a > b ? a : b);
                    if (lane == 0 && p < DL) S.st[0][p >> 5] = w;
                }
#pragma unroll
                for (int r = 0; r < NY / NTHR; ++r) {
                    const int j = tid + NTHR * r;
                    unsigned w = 0;
                    for (int l = 0; l < 6; ++l) {
                        const double v = j < nb ? __ldg(gy + l * N + k_lo + j) : 0.0;
                        anyg |= v != 0.0;
                        w = max(w, abs_hi(v));
                    }
                    w = warp_max(w);
                    if (lane == 0) S.st[1][j >> 5] = w;
                }
            }
            const bool work = bad || (__syncthreads_or(anyg) && __syncthreads_or(anyh));
            int ex = 0, eg = 0;
            if (!bad && work) {
                unsigned hmax, gmax;
                bad = !range_ok<0>(S.st, 1, WL, KW, RANGE_SKY, &hmax, &ex);
                bad |= !range_ok<0>(S.st + 1, 1, nb, KW, RANGE_SKY, &gmax, &eg);
                eg += (gmax & 0xfffff) >= 0xfa000;   // the top byte's range is 127.5 / 128 of the scale
            }
            if (!bad && work) {
#pragma unroll
                for (int i = 0; i < NV; ++i) {
                    const int p = tid + i * NTHR;
                    if (p < DL) {
                        digits_to_planes(planes, p, vp[i], ex);
                        digits_to_planes(planes + 7 * DL, p, vc[i], ex);
                    }
                }
                const int steps = (nb + 3 + 15) / 16, mid = (steps + 1) / 2;
                for (int sg = 0; sg < nseg; ++sg) {
                    const int js = S.segj[sg], je = S.segj[sg + 1];
                    __syncthreads();
                    for (int i = tid; i < 12 * NN * LG; i += blockDim.x) C[i] = 0.0;
                    // link pairs one after the other (256 threads), or the first two side by side and then
                    // the third with an item per warp
                    constexpr int NGR = NTHR / 256, ROUNDS = NGR == 1 ? 3 : 2;
                    for (int round = 0; round < ROUNDS; ++round) {
                        const int lp0 = NGR * round, np = 3 - lp0 < NGR ? 3 - lp0 : NGR;
                        __syncthreads();
                        for (int i = tid; i < np * K3_PAIR / 4; i += NTHR) reinterpret_cast<uint32_t *>(G)[i] = 0x80808080u;
                        __syncthreads();
                        for (int i = tid; i < 2 * np * (je - js); i += NTHR) {
                            const int l2 = i / (je - js), j = js + i - l2 * (je - js);
                            const long long x0 = to_fixed(__ldg(gy + (2 * lp0 + l2) * N + k_lo + j), eg);
                            const int kappa = 2 * j + 1 - NY;
                            unsigned char *row = G + l2 * GROWS * GB + 7 + j;
                            long long xa = x0, xb = mul_nu<9>(x0, kappa);
#pragma unroll
                            for (int q = 0; q < NN; ++q) {
                                unsigned char *o = row + gplane(false, q) * GB;
                                if (gdigits(false, q) == 7) put_bytes<7>(o, xa);
                                else if (gdigits(false, q) == 6) put_bytes<6>(o, xa);
                                else if (gdigits(false, q) == 5) put_bytes<5>(o, xa);
                                else if (gdigits(false, q) == 4) put_bytes<4>(o, xa);
                                else put_bytes<3>(o, xa);
                                const long long nx = mul_nu<8>(xb, kappa) - xa;
                                xa = xb;
                                xb = nx;
                            }
                        }
                        __syncthreads();
                        const bool shared_pair = np < NGR;   // all warps on one pair, one item each
                        const int pr = shared_pair ? 0 : warp >> 3, lp = lp0 + pr;
                        const unsigned char *g_lane = G + pr * K3_PAIR + (lr4 >> 2) * GROWS * GB + 4 + 4 * kp;
                        for (int ps = 0; ps < npass; ++ps) {
                            const unsigned char *a_lane = reinterpret_cast<const unsigned char *>(planes) + 8 * (lr4 + 8 * ps) + 8 * kp;
                            for (int k = 0; k < (shared_pair ? 1 : 2); ++k) {
                                const int it = shared_pair ? warp : c_items[warp & 7][k];
                                const int s0 = (it & 1) ? mid : 0, s1 = (it & 1) ? steps : mid;
                                switch (it >> 1) {
                                    case 0: correlate_item<0>(C, LG, a_lane, g_lane, sh, s0, s1, 32 * ps, lane, 2 * lp); break;
                                    case 1: correlate_item<1>(C, LG, a_lane, g_lane, sh, s0, s1, 32 * ps, lane, 2 * lp); break;
                                    case 2: correlate_item<2>(C, LG, a_lane, g_lane, sh, s0, s1, 32 * ps, lane, 2 * lp); break;
                                    case 3: correlate_item<3>(C, LG, a_lane, g_lane, sh, s0, s1, 32 * ps, lane, 2 * lp); break;
                                    case 4: correlate_item<4>(C, LG, a_lane, g_lane, sh, s0, s1, 32 * ps, lane, 2 * lp); break;
                                    case 5: correlate_item<5>(C, LG, a_lane, g_lane, sh, s0, s1, 32 * ps, lane, 2 * lp); break;
                                    case 6: correlate_item<6>(C, LG, a_lane, g_lane, sh, s0, s1, 32 * ps, lane, 2 * lp); break;
                                    default: correlate_item<7>(C, LG, a_lane, g_lane, sh, s0, s1, 32 * ps, lane, 2 * lp); break;
                                }
                            }
                        }
                    }
                    __syncthreads();
                    // node weights and their derivatives (prefix and suffix products with the product rule, two
                    // threads per read), the reads on this segment's spline piece
                    const int *sm = S.segm[sg];
                    if (tid < 2) gscale[tid] = 0;
                    if (sm[9] != S.segm[sg ? sg - 1 : 0][9]) {
                        if (tid < NN * 3) node_reads(P, X, S, t_lo, u0, tid / 3, tid % 3, sm[9]);
                        __syncthreads();
                    }
                    const int id = tid < WNS ? tid : tid - WNS;
                    const bool low = tid < WNS, half = tid < 2 * WNS;
                    double e = 0.0, run = 1.0, drun = 0.0;
                    double *w = wn + id, *dw = dwn + id;
                    if (half) {
                        e = S.nodeu[id] - (double)sm[id % 9];
                        if (low) {
                            for (int a = 0; a < T / 2; ++a) {
                                w[a * WNS] = run;
                                dw[a * WNS] = drun;
                                const double f = fma(e, S.lc1[a], S.lc0[a]);
                                drun = fma(drun, f, run * S.lc1[a]);
                                run *= f;
                            }
                        } else {
                            for (int a = T - 1; a >= T / 2; --a) {
                                const double sg1 = ((T - 1 - a) & 1) ? -1.0 : 1.0;
                                w[a * WNS] = sg1 * run;
                                dw[a * WNS] = sg1 * drun;
                                const double f = fma(e, S.rc1[a], S.rc0[a]);
                                drun = fma(drun, f, run * S.rc1[a]);
                                run *= f;
                            }
                        }
                    }
                    __syncthreads();
                    if (half) {
                        if (low) {
                            for (int a = T / 2; a < T; ++a) {
                                const double r = w[a * WNS], dr = dw[a * WNS];
                                w[a * WNS] = run * r;
                                dw[a * WNS] = fma(drun, r, run * dr);
                                const double f = fma(e, S.lc1[a], S.lc0[a]);
                                drun = fma(drun, f, run * S.lc1[a]);
                                run *= f;
                            }
                        } else {
                            for (int a = T / 2 - 1; a >= 0; --a) {
                                const double sg1 = ((T - 1 - a) & 1) ? -1.0 : 1.0, r = w[a * WNS], dr = dw[a * WNS];
                                w[a * WNS] = sg1 * (run * r);
                                dw[a * WNS] = sg1 * fma(drun, r, run * dr);
                                const double f = fma(e, S.rc1[a], S.rc0[a]);
                                drun = fma(drun, f, run * S.rc1[a]);
                                run *= f;
                            }
                        }
                    }
                    // correlations at the nodes: sum over the orders (cheb of node NN - 1 - n is that of n with
                    // odd orders negated)
                    for (int i = tid; i < 12 * LG; i += blockDim.x) {
                        const int l = i / (2 * LG), r = i - l * 2 * LG;
                        double *c = C + l * NN * 2 * LG + r;
                        double v[NN];
#pragma unroll
                        for (int q = 0; q < NN; ++q) v[q] = c[q * 2 * LG];
#pragma unroll
                        for (int n = 0; n < NN / 2; ++n) {
                            double ev = 0.0, od = 0.0;
#pragma unroll
                            for (int q = 0; q < NN; q += 2) {
                                ev = fma(X.cheb[q][n], v[q], ev);
                                od = fma(X.cheb[q + 1][n], v[q + 1], od);
                            }
                            c[n * 2 * LG] = ev + od;
                            c[(NN - 1 - n) * 2 * LG] = ev - od;
                        }
                    }
                    __syncthreads();
                    if (tid < NN * 24) {
                        const int n = tid / 24, l = (tid % 24) >> 2, er = (tid >> 1) & 1, pol = tid & 1;
                        const int rd = er ? c_lr[l] : 3 + l;
                        const double *c = C + ((l * NN + n) * 2 + pol) * LG + sm[rd] - mmin;
                        const double *a = wn + n * 9 + rd, *b = dwn + n * 9 + rd;
                        double v = 0.0, d = 0.0;
                        for (int t = 0; t < T; ++t) {
                            v = fma(a[t * WNS], c[t], v);
                            d = fma(b[t * WNS], c[t], d);
                        }
                        dots[n][l][er][2 * pol] = v;
                        dots[n][l][er][2 * pol + 1] = d;
                    }
                    __syncthreads();
                    double *geo = wn;   // [node][link][6]: the weights are done with
                    if (tid < 128 && (tid & 63) < NN * 6) {   // an angle per thread: lambda, then beta and psi two warps on
                        double t[3] = {0.0, 0.0, 0.0};
                        const int th = tid >> 6, n = (tid & 63) / 6, l = (tid & 63) % 6;
                        double *q = geo + 6 * (tid & 63);
                        sky_terms(P, S.skc, S.npos[n], l, dots[n][l][0], dots[n][l][1], th, th + 1, t, q);
                        const double unit = pow2(eg) * pow2(ex);
                        for (int c = 0; c < 3; ++c) Gs[c] += t[c] * unit;
                        if (th == 0) atomicMax(&gscale[0], __float_as_int((float)fmax(fabs(q[0]), fabs(q[1]))) & 0x7fffffff);
                        atomicMax(&gscale[1], __float_as_int((float)fmax(fabs(q[2 + 2 * th]), fabs(q[3 + 2 * th]))) & 0x7fffffff);
                    }
                    __syncthreads();
                    bool fits = true;
                    if (tid < 36) {
                        const int l = tid / 6, i = tid % 6;
                        const double de = S.nodeu[3 + l] - S.nodeu[(NN - 1) * 9 + 3 + l];
                        const double dr = S.nodeu[c_lr[l]] - S.nodeu[(NN - 1) * 9 + c_lr[l]];
                        const float delta = 0.51f * (float)fmax(fabs(de), fabs(dr));   // half the drift; the nodes end at 0.98
                        fits = sky_series_fits(X, geo + 6 * l + i, 36, __int_as_float(gscale[i > 1]), delta);
                    }
                    if (__syncthreads_or(!fits)) {
                        bad = true;
                        break;
                    }
                }
                if (bad) Gs[0] = Gs[1] = Gs[2] = 0.0;
            }
            __syncthreads();
            if (bad)
                for (int j = tid; j < nb; j += blockDim.x) {
                    const int64_t k = k_lo + j;
                    double x[9], L[6], rr[3][4], sig[3];
                    orbit_all(P.po, P.t0 + (double)k * P.dt, x, L);
                    for (int i = 0; i < 3; ++i) {
                        sig[i] = (S.skc.k[0] * x[3 * i] + S.skc.k[1] * x[3 * i + 1] + S.skc.k[2] * x[3 * i + 2]) / C_LIGHT * P.inv_dt;
                        read_vd_scalar(S, T, ti.hp, ti.hc, ti.nh, k + f0, u0 - sig[i], rr[i]);
                    }
                    for (int l = 0; l < 6; ++l) {
                        const double gl = __ldg(gy + l * N + k);
                        if (gl == 0.0) continue;
                        double ee[4], t[3] = {0.0, 0.0, 0.0};
                        read_vd_scalar(S, T, ti.hp, ti.hc, ti.nh, k + f0, u0 - L[l] * P.inv_dt - sig[c_ls[l]], ee);
                        sky_terms(P, S.skc, x, l, ee, rr[c_lr[l]], 0, 2, t, nullptr);
                        for (int c = 0; c < 3; ++c) Gs[c] = fma(gl, t[c], Gs[c]);
                    }
                }
        }
        // fixed-order block reduction: warp tree, then warps in order
        for (int t = 0; t < 3; ++t) {
            double v = Gs[t];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
            if (lane == 0) red[t][warp] = v;
        }
        __syncthreads();
        if (tid < 3) {
            double s = 0.0;
            for (int w = 0; w < NTHR / 32; ++w) s += red[tid][w];
            B.partial[3 * g + tid] = s;
        }
        __syncthreads();
    }
}

}  // namespace

int launch_fx_bwd(int kind, int order, const FwdParams &P, const BwdParams &B, FxPlan *F, int sms, void *stream)
{
    if (P.src.tile_off && !P.src.skyc && kind != 0) return (int)cudaErrorInvalidValue;  // sky frames of a batch
    int T = order + 1;
    FxTab X;
    if (const int e = fx_table_for(F, stream, &X)) return e;
    const int64_t known = kind == 1 ? B.h_total_tiles : P.total_tiles;
    // 512 threads a block where the launch has at most a block per SM
    const int nthr = known >= 0 && known <= sms ? 512 : 256;
    void *k = nthr == 512 ? (kind == 0 ? (void *)k_fx_tdi_adj<512> : kind == 1 ? (void *)k_fx_proj_adj<512> : (void *)k_fx_sky_adj<512>)
                          : (kind == 0 ? (void *)k_fx_tdi_adj<256> : kind == 1 ? (void *)k_fx_proj_adj<256> : (void *)k_fx_sky_adj<256>);
    const size_t smem = kind == 0 ? k1_w(T) + FX_TDI_W
                        : kind == 1 ? K2_PLANES + nthr / 256 * K2_GROUP
                                    : k3_c(T, nthr) + sizeof(double) * 12 * NN * (size_t)X.lags;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return (int)e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, nthr, smem);
    if (e != cudaSuccess) return (int)e;
    if (per_sm < 1) return (int)cudaErrorLaunchOutOfResources;
    int64_t grid = (int64_t)per_sm * sms;
    if (known >= 0 && known < grid) grid = known;
    if (grid < 1) grid = 1;
    void *args[] = {(void *)&P, (void *)&X, (void *)&B, (void *)&T};
    return (int)cudaLaunchKernel(k, dim3((unsigned)grid), dim3(nthr), args, smem, (cudaStream_t)stream);
}

}  // namespace lr
