// FP64 forward kernel on the tensor cores: projection, TDI, or both fused, for a block of outputs.
//
// What bounds it.  GB300 issues 2 FP64 FMAs per SM and clock, so the per-sample form (lr_fwd64.cu: 60
// reads of T taps per output, five FP64 operations per tap) spends ~8000 FP64 operations per output and
// sits on that pipe.  Here an output costs ~100 FP64 operations; the taps are exact integer products on
// the tensor cores (half-precision operands, FP32 accumulators).
//
// How.  Over a block every read's weights are smooth functions of time: the fractional offset of read r,
// eps_r(t) = u_r(t) - m_r, drifts by at most ~1e-4 samples per sample (projection) or ~1e-7 (TDI).  So
//   1. the sums of all reads of one series are merged into one stencil per output: link l is
//        y_l[j] = sum_c W+_l(t_j)[c] h+[j + c] + Wx_l(t_j)[c] hx[j + c],
//      W+_l = c+_l (w_emission - w_reception) over the union of the two stencils; channel X is four links'
//      stencils, each the signed sum of that link's four delayed reads;
//   2. W(t) is expanded in Chebyshev polynomials of the block's normalised time nu, W = sum_q b_q T_q(nu),
//      from FP64 Lagrange weights and geometry at 8 (projection) or 4 (TDI) Chebyshev nodes: the
//      truncation is below 2^-54 of W for drifts of 1e-4 samples per sample (v/c of the orbit);
//   3. the b_q and the staged series are 56-bit fixed point in seven balanced base-256 digits, each digit
//      exact in half precision, and A_{q,L}[j] = sum_c sum_{i+k=L} digit_i(b_q)[c] digit_k(h)[j + c], L = 0..6,
//      is accumulated in FP32 (slices of an exact product on low-precision units, as in Ozaki's scheme):
//      products are at most 2^14, 5 taps x links of them meet at level 4, which is 290 in the projection,
//      1140 in TDI, 1254 and 1360 in the adjoint's K2 and K3.  Sums below 2^24 are exact integers; to pass it
//      three quarters of 1360 digit pairs would have to be at the end of their range with agreeing signs (digits
//      of either sign sum to less than 2^20).  Level 6 carries level 7 (each series digit extended by the
//      next one to 11 bits), which keeps the products left out below 2^-56;
//   4. sum_q A_q T_q(nu) is Clenshaw's recurrence in 64-bit integers: nu is a multiple of 2^-9, so each
//      step is a small integer product and a shift.
// The digits that a higher q cannot have (|b_q| falls by ~2^-7 per order) are left out: 121 of 224 digit
// products for the projection, 62 of 112 for TDI.
//
// A delayed read's stencil moves by one sample when floor(u_r) steps and the orbit splines change piece at
// a knot.  Both are found per block (grid of samples, every sample near a step) and split the block into
// segments; each has its own expansion (with the segment's stencils and spline piece continued over the
// whole block) and its own share of the rows.
//
// Layout of the contraction (mma.sync m16n8k16): row a of a block of 16 is samples 8a..8a+7, column b the
// sample within the row, so the left operand is the staged series itself, series[8a + c], and the right
// one the stencil shifted by b, W[c - b]; neither is expanded in memory.  The projection takes rows of 4
// samples and two links as the columns' other half: both links read the same strain, and 29 taps + 3 fit
// 32 steps of k where 29 + 7 need 48.  A lane's four k-values are taken
// as four consecutive c (the same permutation of k on both sides), so a lane reads its two left registers
// of a row with one 8-byte load and its right registers from four consecutive digit bytes, which become
// halves by placing them under the exponent of 1024 and subtracting 1152.
//
// Measured (fused, order 25, one year of 3 153 600 outputs): 44.45 ms sample by sample, 3.4 to 4.0 ms here (the
// source's position sets how many segments a block has), with 3.0e-12 relative error against 64 bits where
// the sample form has 3.5e-12; 65 536 outputs: 490 us and 108 us.  Two blocks share an SM; the tensor pipe
// and the FP64 pipe (weights, transforms) are each busy a quarter of the time, the rest is latency of the short
// FP64 phases.  Steps on the way, one year: 4.36 ms with 8-sample rows in the projection and the TDI stencils
// computed in every block; 65 536 outputs: 113 us with the weights and the links' patterns of the nodes on the
// same warps, the TDI stencils' scale found in the block, and a barrier more for each of the two scales.
//
// Where the expansion does not apply, the block is evaluated sample by sample in FP64 as in lr_fwd64.cu: a
// NaN or infinity in the series, outputs that read values far below the block's largest (the fixed point is
// relative to it: RANGE_PROJ, RANGE_TDI), coefficients above the digits reserved for their
// order (a source within ~1 degree of an arm direction, an orbit that moves faster), too many segments.
#include "lr_fx64.cuh"

namespace lr {
namespace {

// ---------------------------------------------------------------- the block's link series
// Fills ys[6][NY] with the link series of rows 0 .. ny - 1 (sample k_lo + row).
template <int NTHR>
__device__ void project_block(const FwdParams &P, const FxTab &X, Shared &S, int T, int64_t k_lo, int ny, double u, double *ys,
                              unsigned char *work)
{
    const int tid = threadIdx.x, h = (T - 2) / 2;
    const int64_t f0 = (int64_t)floor(u);
    const double u0 = u - floor(u);
    const double t_lo = P.t0 + (double)k_lo * P.dt;
    const TileInfo &ti = S.ti;
    uint16_t *planes = reinterpret_cast<uint16_t *>(work);
    unsigned char *W = work + FX_PROJ_PLANES;
    double *wn = reinterpret_cast<double *>(work + FX_PROJ_PLANES + FX_PROJ_W);

    projection_segments(P, X, S, t_lo, u0, ny);
    const int nseg = S.nseg;
    const int mmin = S.mmin, KW = S.mmax - mmin + T;   // taps of a merged stencil
    const int nks = (KW + 3 + 15) / 16;
    bool bad = S.bad || nks * 16 > 64;
    // strain window: row j reads samples w_lo + j .. w_lo + j + KW - 1
    const int64_t w_lo = k_lo + f0 + mmin - h;
    const int WL = ny + KW - 1;
    constexpr int NV = (DL + NTHR - 1) / NTHR;
    double vp[NV], vc[NV];
    if (!bad) {
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            const int p = tid + i * NTHR;
            vp[i] = vc[i] = 0.0;
            if (p < WL) {
                const int64_t idx = w_lo + p;
                if (P.gen_strain) {
                    gb_strain(ti.gb, P.t0, P.dt, idx, vp[i], vc[i]);
                } else if (idx >= 0 && idx < ti.nh) {
                    vp[i] = __ldg(ti.hp + idx);
                    vc[i] = __ldg(ti.hc + idx);
                }
            }
            const unsigned a = abs_hi(vp[i]), b = abs_hi(vc[i]);
            if (!P.gen_strain && (a > b ? a : b) >= 0x7ff00000u) atomicOr(P.err, ERR_NONFINITE);
            const unsigned w = warp_max(a > b ? a : b);
            if ((tid & 31) == 0 && p < DL) S.st[0][p >> 5] = w;
        }
    }
    __syncthreads();
    int ex = 0;
    unsigned vmax = 1;
    const bool in_range = !bad && range_ok<0>(S.st, 1, WL, KW, RANGE_PROJ, &vmax, &ex);
    if (!bad && vmax == 0) {  // a block of zeros (or of subnormal high words): the response is zero
        bool any = false;
#pragma unroll
        for (int i = 0; i < NV; ++i) any |= vp[i] != 0.0 || vc[i] != 0.0;
        if (!__syncthreads_or(any)) {
            for (int i = tid; i < 6 * NY; i += blockDim.x) ys[i] = 0.0;
            __syncthreads();
            return;
        }
        bad = true;
    }
    bad |= !in_range;
    if (!bad) {
        for (int i = 0; i < NV; ++i) {
            const int p = tid + i * NTHR;
            if (p < DL) {
                digits_to_planes(planes, p, vp[i], ex);
                digits_to_planes(planes + 7 * DL, p, vc[i], ex);
            }
        }
    }
    const uint32_t lane = tid & 31, warp = tid >> 5, lr4 = lane >> 2, kp = lane & 3;
    const uint32_t sh = 8 * ((7 - lr4) & 3);
    for (int sg = 0; sg < nseg && !bad; ++sg) {
        if (!projection_stencils<false>(P, X, S, T, t_lo, u0, sg, KW, W, wn)) {
            bad = true;
            break;
        }
        const int nq = S.nq;
        const bool last = S.last;
        const int js = S.segj[sg], je = S.segj[sg + 1];
        const int mb0 = js >> 6, nmb = ((je - 1) >> 6) - mb0 + 1;
        // item: 64 rows (16 groups of 4 samples) of two links; column = link, sample within the group
        for (int it = warp; it < nmb * 3; it += blockDim.x >> 5) {
            const int lp = it % 3, mb = mb0 + it / 3;
            const int lw = 2 * lp + (int)(lr4 >> 2);   // the link whose stencil this lane loads
            const int l = 2 * lp + (int)(kp >> 1);     // the link of this lane's sums
            const unsigned char *a_lane = reinterpret_cast<const unsigned char *>(planes) + 8 * (16 * mb + (int)lr4) + 8 * kp;
            const unsigned char *w_lane = W + 2 * lw * PD * WS + 4 + 4 * (kp + ((3 - (lr4 & 3)) >> 2));
            int kappa[4], jr[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                jr[r] = 64 * mb + 4 * (int)(lr4 + (r >> 1) * 8) + 2 * (int)(kp & 1) + (r & 1);
                kappa[r] = 2 * jr[r] + 1 - NY;
            }
            long long b1[4] = {0, 0, 0, 0}, b2[4] = {0, 0, 0, 0};
            if (nq > 4) {
                float acc[4][7][4];
                if (last) contract<4, 4, false, true>(acc, a_lane, w_lane, sh, nks, nullptr);
                else contract<4, 4, false>(acc, a_lane, w_lane, sh, nks, nullptr);
                clenshaw<4, 4, false>(acc, kappa, b1, b2);
            }
            if (nq > 2) {
                float acc[2][7][4];
                if (last) contract<2, 2, false, true>(acc, a_lane, w_lane, sh, nks, nullptr);
                else contract<2, 2, false>(acc, a_lane, w_lane, sh, nks, nullptr);
                clenshaw<2, 2, false>(acc, kappa, b1, b2);
            }
            if (nq > 1) {
                float acc[1][7][4];
                if (last) contract<1, 1, false, true>(acc, a_lane, w_lane, sh, nks, nullptr);
                else contract<1, 1, false>(acc, a_lane, w_lane, sh, nks, nullptr);
                clenshaw<1, 1, false>(acc, kappa, b1, b2);
            }
            float acc[1][7][4];
            contract<0, 1, false>(acc, a_lane, w_lane, sh, nks, nullptr);
            const int unit = ex + S.wexp[l] - 57;
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const long long v = levels<0>(acc[0], r) + mul_nu<9>(b1[r], kappa[r]) - b2[r];
                const int64_t k = k_lo + jr[r];
                if (jr[r] >= js && jr[r] < je) ys[l * NY + jr[r]] = k >= 0 && k < ti.N ? from_fixed(v, unit) : 0.0;
            }
        }
    }
    __syncthreads();
    if (!bad) return;
    // sample by sample, on the strain window of all reads that the plan's bounds allow
    double *hwp = reinterpret_cast<double *>(work), *hwc = hwp + FX_PROJ_PLANES / 16;
    const int64_t s_lo = k_lo + f0 - P.sig_b - P.lproj_b - h - 2;
    const int slen = ny + 2 * P.sig_b + P.lproj_b + T + 4;
    bool nonfinite = false;
    for (int j = tid; j < slen; j += blockDim.x) {
        const int64_t i = s_lo + j;
        double a = 0.0, b = 0.0;
        if (P.gen_strain) {
            gb_strain(ti.gb, P.t0, P.dt, i, a, b);
        } else if (i >= 0 && i < ti.nh) {
            a = __ldg(ti.hp + i);
            b = __ldg(ti.hc + i);
        }
        nonfinite |= !P.gen_strain && !(isfinite(a) && isfinite(b));
        hwp[j] = a;
        hwc[j] = b;
    }
    if (nonfinite) atomicOr(P.err, ERR_NONFINITE);
    __syncthreads();
    for (int j = tid; j < ny; j += blockDim.x) {
        const int64_t k = k_lo + j;
        double y[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
        if (k >= 0 && k < ti.N) {
            const SkyConst &K = S.skc;
            double x[9], L[6], sig[3], rp[3], rc[3];
            orbit_all(P.po, P.t0 + (double)k * P.dt, x, L);
            for (int i = 0; i < 3; ++i) {
                sig[i] = (K.k[0] * x[3 * i] + K.k[1] * x[3 * i + 1] + K.k[2] * x[3 * i + 2]) / C_LIGHT * P.inv_dt;
                rp[i] = read_scalar(S, T, hwp, k + f0, u0 - sig[i], s_lo, slen, P.err);
                rc[i] = read_scalar(S, T, hwc, k + f0, u0 - sig[i], s_lo, slen, P.err);
            }
            for (int a = 0; a < 3; ++a) {
                const int r = a, s = (a + 1) % 3, lf = a, lb = 5 - a;
                double d0 = x[3 * r] - x[3 * s], d1 = x[3 * r + 1] - x[3 * s + 1], d2 = x[3 * r + 2] - x[3 * s + 2];
                const double inv = 1.0 / sqrt(d0 * d0 + d1 * d1 + d2 * d2);
                d0 *= inv; d1 *= inv; d2 *= inv;
                const double un = K.u[0] * d0 + K.u[1] * d1 + K.u[2] * d2, vn = K.v[0] * d0 + K.v[1] * d1 + K.v[2] * d2;
                const double kn = K.k[0] * d0 + K.k[1] * d1 + K.k[2] * d2;
                const double xip = un * un - vn * vn, xic = 2.0 * un * vn;
                const double xp = K.c2p * xip + K.s2p * xic, xc = -K.s2p * xip + K.c2p * xic;
                const double uf = u0 - L[lf] * P.inv_dt - sig[s], ub = u0 - L[lb] * P.inv_dt - sig[r];
                double ep = read_scalar(S, T, hwp, k + f0, uf, s_lo, slen, P.err), ec = read_scalar(S, T, hwc, k + f0, uf, s_lo, slen, P.err);
                y[lf] = (xp * (ep - rp[r]) + xc * (ec - rc[r])) / (2.0 * (1.0 - kn));
                ep = read_scalar(S, T, hwp, k + f0, ub, s_lo, slen, P.err);
                ec = read_scalar(S, T, hwc, k + f0, ub, s_lo, slen, P.err);
                y[lb] = (xp * (ep - rp[s]) + xc * (ec - rc[s])) / (2.0 * (1.0 + kn));
            }
        }
        for (int l = 0; l < 6; ++l) ys[l * NY + j] = y[l];
    }
    __syncthreads();
}

// ---------------------------------------------------------------- the block's X, Y, Z
// Link rows ys[6][NY] (ny = nb + HL + HR of them, row = output + HL) to outputs; ys is overwritten.
// Each output is handed to `emit(i, X, Y, Z)` by one thread.
template <int NTHR, class Emit>
__device__ void tdi_block(const FwdParams &P, const FxTab &X, Shared &S, int T, int64_t n0, int nb, double *ys, unsigned char *work,
                          Emit emit)
{
    const int tid = threadIdx.x, h = (T - 2) / 2, ny = nb + P.HL + P.HR;
    const uint32_t lane = tid & 31, warp = tid >> 5, lr4 = lane >> 2, kp = lane & 3;
    const double t_lo = P.t0 + (double)n0 * P.dt;
    double *wt = reinterpret_cast<double *>(work);
    uint16_t *planes = reinterpret_cast<uint16_t *>(work);
    const int xb = T * WTS * 8;
    unsigned char *W = work + (xb > FX_TDI_PLANES ? xb : FX_TDI_PLANES);

    if (tid < NY / 32) S.brk[tid] = 0;
    if (tid == 32) {
        S.nlist = 0;
        S.bad = 0;
        S.mmin = 1 << 29;
        S.mmax = -(1 << 29);
    }
    if (tid == 64) S.fast = X.tab ? table_segments(P, X, S, t_lo, nb) : 0;
    __syncthreads();
    // the first and last link rows are spare: no stencil reaches them
#pragma unroll
    for (int i = 0; i < NY / NTHR; ++i) {
        const int j = tid + NTHR * i;
        unsigned w[6];
#pragma unroll
        for (int l = 0; l < 6; ++l) w[l] = warp_max(j >= 1 && j < ny - 1 ? abs_hi(ys[l * NY + j]) : 0u);
        constexpr SlotTab slots = make_slots();
#pragma unroll
        for (int ch = 0; ch < 3; ++ch)
            if (lane == 0)
                S.st[ch][j >> 5] = max(max(w[slots.link[ch][0]], w[slots.link[ch][1]]), max(w[slots.link[ch][2]], w[slots.link[ch][3]]));
    }
    const bool fast = S.fast != 0;
    if (!fast) find_tdi_segments(P, S, t_lo, nb);
    __syncthreads();
    const int nseg = S.nseg;
    bool bad = S.bad;
    int ey = 0;
    unsigned vmax;
    const bool in_range = range_ok<1>(S.st, 3, ny, T + P.HL - h - 2, RANGE_TDI, &vmax, &ey);
    if (vmax == 0) {
        bool any = false;
        for (int i = tid; i < 6 * NY; i += blockDim.x) any |= i % NY < ny && ys[i] != 0.0;
        if (!__syncthreads_or(any)) {
            for (int i = tid; i < nb; i += blockDim.x) emit(i, 0.0, 0.0, 0.0);
            __syncthreads();
            return;
        }
        bad = true;
    }
    bad |= !in_range;
    long long *part = reinterpret_cast<long long *>(ys);  // [2][3][NY], one segment: the planes hold the series
    int done = 0;                                          // outputs kept in ys[0..2][.] by earlier segments
    for (int sg = 0; sg < nseg && !bad; ++sg) {
        const int piece = S.segm[sg][NTERM];
        const int mmin = fast ? X.meta[FX_META * piece + 1] : S.mmin;
        const int KW = fast ? X.meta[FX_META * piece] : (S.mmax > 0 ? S.mmax : 0) - mmin + T;
        const int nks = (KW + 7 + 15) / 16;
        const int j0 = P.HL + mmin - h;                        // link row of the stencil's first tap for output 0
        if (!fast && (nks * 16 > 64 || j0 < 1 || S.mmax > 0)) {
            bad = true;
            break;
        }
        int ew;
        if (!(fast ? tdi_stencils<false, NTHR>(P, X, S, t_lo, sg, KW, W, &ew)
                   : tdi_stencils_nodes<false, NTHR>(P, X, S, T, t_lo, sg, KW, mmin, W, wt, &ew))) {
            bad = true;
            break;
        }
        const int js = S.segj[sg], je = S.segj[sg + 1];
        // link rows that only earlier outputs read are left out: their place holds those outputs now
        for (int i = tid; i < 6 * DL; i += blockDim.x) {
            const int l = i / DL, p = i - l * DL, j = p + j0;
            digits_to_planes(planes + l * 7 * DL, p, p >= js && j < ny - 1 ? ys[l * NY + j] : 0.0, ey);
        }
        __syncthreads();
        count_orders<NT>(S);
        const int mb0 = js >> 7, nmb = ((je - 1) >> 7) - mb0 + 1;
        const int unit = ey + ew - 57;
        const uint32_t sh = 8 * ((7 - lr4) & 3);
        const bool hi = S.nq > 1, last = S.last;
        const int per = nmb * 3;
        if (nseg == 1) {
            // order 0 and the higher orders are separate items (28 and 34 digit products)
            for (int it = warp; it < (hi ? 2 : 1) * per; it += blockDim.x >> 5) {
                const int half = it / per, ch = it % per % 3, mb = mb0 + it % per / 3;
                const unsigned char *a_lane = reinterpret_cast<const unsigned char *>(planes) + 16 * (16 * mb + (int)lr4) + 8 * kp;
                const unsigned char *w_lane = W + 4 * ch * TD * WS + 4 * (kp + ((7 - lr4) >> 2));
                if (half == 0) {
                    float acc[1][7][4];
                    contract<0, 1, true>(acc, a_lane, w_lane, sh, nks, c_slots.link[ch]);
#pragma unroll
                    for (int r = 0; r < 4; ++r)
                        part[ch * NY + 128 * mb + 8 * (lr4 + (r >> 1) * 8) + 2 * kp + (r & 1)] = levels<0>(acc[0], r);
                } else {
                    float acc[3][7][4];
                    if (last) contract<1, 3, true, true>(acc, a_lane, w_lane, sh, nks, c_slots.link[ch]);
                    else contract<1, 3, true>(acc, a_lane, w_lane, sh, nks, c_slots.link[ch]);
                    int kappa[4];
                    long long b1[4] = {0, 0, 0, 0}, b2[4] = {0, 0, 0, 0};
#pragma unroll
                    for (int r = 0; r < 4; ++r) kappa[r] = 2 * (128 * mb + 8 * (int)(lr4 + (r >> 1) * 8) + 2 * (int)kp + (r & 1)) + 1 - NY;
                    clenshaw<1, 3, true>(acc, kappa, b1, b2);
#pragma unroll
                    for (int r = 0; r < 4; ++r)
                        part[(3 + ch) * NY + ((kappa[r] + NY - 1) >> 1)] = mul_nu<9>(b1[r], kappa[r]) - b2[r];
                }
            }
            __syncthreads();
            for (int i = tid; i < nb; i += blockDim.x) {
                double o[3];
#pragma unroll
                for (int c = 0; c < 3; ++c) o[c] = from_fixed(part[c * NY + i] + (hi ? part[(3 + c) * NY + i] : 0), unit);
                emit(i, o[0], o[1], o[2]);
            }
            done = nb;
        } else {
            // a block with a step: one item per channel; the outputs are kept in ys[0..2], in rows that the
            // later segments do not read (their first link row is past output je)
            for (int it = warp; it < per; it += blockDim.x >> 5) {
                const int ch = it % 3, mb = mb0 + it / 3;
                const unsigned char *a_lane = reinterpret_cast<const unsigned char *>(planes) + 16 * (16 * mb + (int)lr4) + 8 * kp;
                const unsigned char *w_lane = W + 4 * ch * TD * WS + 4 * (kp + ((7 - lr4) >> 2));
                int kappa[4];
                long long b1[4] = {0, 0, 0, 0}, b2[4] = {0, 0, 0, 0};
#pragma unroll
                for (int r = 0; r < 4; ++r) kappa[r] = 2 * (128 * mb + 8 * (int)(lr4 + (r >> 1) * 8) + 2 * (int)kp + (r & 1)) + 1 - NY;
                if (hi) {
                    float acc[3][7][4];
                    if (last) contract<1, 3, true, true>(acc, a_lane, w_lane, sh, nks, c_slots.link[ch]);
                    else contract<1, 3, true>(acc, a_lane, w_lane, sh, nks, c_slots.link[ch]);
                    clenshaw<1, 3, true>(acc, kappa, b1, b2);
                }
                float acc[1][7][4];
                contract<0, 1, true>(acc, a_lane, w_lane, sh, nks, c_slots.link[ch]);
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const int i = (kappa[r] + NY - 1) >> 1;
                    if (i >= js && i < je) ys[ch * NY + i] = from_fixed(levels<0>(acc[0], r) + mul_nu<9>(b1[r], kappa[r]) - b2[r], unit);
                }
            }
            done = je;
        }
    }
    __syncthreads();
    if (nseg > 1 || bad)
        for (int i = tid; i < done; i += blockDim.x) emit(i, ys[i], ys[NY + i], ys[2 * NY + i]);
    if (!bad) {
        __syncthreads();
        return;
    }
    // the other outputs sample by sample
    for (int i = done + tid; i < nb; i += blockDim.x) {
        const int64_t n = n0 + i;
        double L[6], o[3];
        orbit_delays(P.to, P.t0 + (double)n * P.dt, L);
        for (int l = 0; l < 6; ++l) L[l] *= P.inv_dt;
        for (int ch = 0; ch < 3; ++ch) {
            double acc = 0.0;
            for (int c = 0; c < 2; ++c) {
                double sum = ys[c_tdifx.link[ch][c][0] * NY + i + P.HL], D = 0.0;
                for (int q = 1; q <= P.q_terms; ++q) {
                    D += L[c_tdifx.pair[ch][c][q]];
                    sum += read_scalar(S, T, ys + c_tdifx.link[ch][c][q] * NY, n, -D, n0 - P.HL, ny, P.err);
                }
                acc = c == 0 ? sum : acc - sum;
            }
            o[ch] = acc;
        }
        emit(i, o[0], o[1], o[2]);
    }
    __syncthreads();
}

// ---------------------------------------------------------------- kernel
// NTHR threads: 256 (two CTAs per SM), or 512 where a launch has at most a block per SM (65536 samples, order 25: 125 -> 113 us)
template <int KIND, int NTHR>
__global__ void __launch_bounds__(NTHR, NTHR == 256 ? 2 : 1) k_fx64(FwdParams P, FxTab X, int T)
{
    extern __shared__ __align__(16) unsigned char sm_raw[];
    double *ys = reinterpret_cast<double *>(sm_raw);
    unsigned char *work = sm_raw + 6 * NY * 8;
    __shared__ Shared S;
    const int tid = threadIdx.x;
    if (tid < T) {
        const int h = (T - 2) / 2;
        S.lc1[tid] = 1.0 / (double)(tid + 1);
        S.lc0[tid] = (double)(h - tid) / (double)(tid + 1);
        S.rc1[tid] = 1.0 / (double)(T - tid);
        S.rc0[tid] = (double)(h - tid) / (double)(T - tid);
    }
    const bool like = KIND == KIND_LIKE;
    const int64_t total = P.total_tiles >= 0 ? P.total_tiles : P.src.tile_off[P.src.S];
    for (int64_t g = blockIdx.x; g < total; g += gridDim.x) {
        int64_t src = 0;
        if (tid < 32 && P.src.tile_off) src = find_source(P, g);
        if (tid == 0) {
            S.ti = tile_info_of(P, g, src, KIND == KIND_PROJECT ? 6 : 3);
            if (KIND != KIND_TDI) S.skc = P.src.tile_off ? P.src.skyc[src] : P.src.skyc1;
            if (!S.ti.ok) atomicOr(P.err, ERR_OFFSETS);
            if (like && !(S.ti.ok && S.ti.nb > 0)) like_store(P, g, 0.0, 0.0);
        }
        __syncthreads();
        if (S.ti.ok && S.ti.nb > 0) {
            const TileInfo &ti = S.ti;
            const int nb = (int)ti.nb;
            if (KIND == KIND_PROJECT) {
                project_block<NTHR>(P, X, S, T, ti.n0, nb, (P.t0 - ti.t0h) / P.dt, ys, work);
                for (int i = tid; i < nb; i += blockDim.x)
#pragma unroll
                    for (int l = 0; l < 6; ++l) ti.out[l * ti.N + ti.n0 + i] = ys[l * NY + i];
            } else {
                const int ny = nb + P.HL + P.HR;
                const int64_t k_lo = ti.n0 - P.HL;
                if (KIND == KIND_TDI) {
                    for (int l = 0; l < 6; ++l)
                        for (int j = tid; j < ny; j += blockDim.x) {
                            const int64_t k = k_lo + j;
                            ys[l * NY + j] = k >= 0 && k < ti.N ? __ldg(ti.yin + l * ti.N + k) : 0.0;
                        }
                    __syncthreads();
                } else {
                    project_block<NTHR>(P, X, S, T, k_lo, ny, (P.t0 - ti.t0h) / P.dt, ys, work);
                }
                double dh = 0.0, hh = 0.0;
                tdi_block<NTHR>(P, X, S, T, ti.n0, nb, ys, work, [&](int i, double vx, double vy, double vz) {
                    const int64_t n = ti.n0 + i;
                    if (ti.out) {
                        ti.out[n] = vx;
                        ti.out[ti.N + n] = vy;
                        ti.out[2 * ti.N + n] = vz;
                    }
                    if (like && ti.dat) {
                        const double da = __ldg(ti.dat + n), de = __ldg(ti.dat + ti.N + n), dT = __ldg(ti.dat + 2 * ti.N + n);
                        if (!(isfinite(da) && isfinite(de) && isfinite(dT))) atomicOr(P.err, ERR_NONFINITE);
                        like_terms(P.like, vx, vy, vz, da, de, dT, dh, hh);
                    }
                });
                if (like) {
                    block_sum2(dh, hh, S.red);
                    if (tid == 0) like_store(P, g, ti.dat ? dh : nan_d(), ti.dat ? hh : nan_d());
                }
            }
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------- the plan's TDI table
// One CTA per spline piece of the TDI orbit: where no delayed read's stencil steps within the piece, the
// merged stencils of the 12 (channel, link) pairs as polynomials of degree 5 in the piece's coordinate on
// [-1, 1] (weights at six Chebyshev nodes; over a 1e5 s piece the delays move by ~1e-3 samples, so the next
// order is below 2^-54).  meta: taps (0: no entry), the first tap's position and the scale's exponent.  The stencils depend on the
// orbit alone; from the table a block's expansion is 20 FP64 operations per tap, against ~130 per read and
// node computed in the block.
__global__ void __launch_bounds__(256) k_fx_table(FwdParams P, FxTab X, int T, double *tab, int *meta, int tab_kw)
{
    extern __shared__ double wt[];  // [T][TQ * NTERM + 1]
    constexpr int TQ = FX_TAB_Q, WTT = TQ * NTERM + 1;
    __shared__ double pc[6][4], eps[TQ][NTERM];
    __shared__ double lc1[64], lc0[64], rc1[64], rc0[64];
    __shared__ int mm[NTERM], mmin, mmax, bad, wmax;
    const int tid = threadIdx.x, k = blockIdx.x, h = (T - 2) / 2, qn = P.q_terms;
    if (tid < T) {
        lc1[tid] = 1.0 / (double)(tid + 1);
        lc0[tid] = (double)(h - tid) / (double)(tid + 1);
        rc1[tid] = 1.0 / (double)(T - tid);
        rc0[tid] = (double)(h - tid) / (double)(T - tid);
    }
    if (tid >= 64 && tid < 70) {  // delays in samples as polynomials of X = 2 x - 1
        const Coef4 q = ldg4(piece_row(P.to, k) + 9 + tid - 64);
        double *o = pc[tid - 64];
        o[0] = (q.a + 0.5 * q.b + 0.25 * q.c + 0.125 * q.d) * P.inv_dt;
        o[1] = (0.5 * q.b + 0.5 * q.c + 0.375 * q.d) * P.inv_dt;
        o[2] = (0.25 * q.c + 0.375 * q.d) * P.inv_dt;
        o[3] = 0.125 * q.d * P.inv_dt;
    }
    if (tid == 70) {
        mmin = 1 << 29;
        mmax = -(1 << 29);
        bad = 0;
        wmax = 0;
    }
    __syncthreads();
    if (tid < NTERM && tid % 7 < qn) {
        const int cc = tid / 7, q = tid % 7 + 1;
        double D[4] = {0.0, 0.0, 0.0, 0.0};
        for (int i = 1; i <= q; ++i)
            for (int c = 0; c < 4; ++c) D[c] += pc[c_tdifx.pair[cc >> 1][cc & 1][i]][c];
        const double R = fabs(D[1]) + fabs(D[2]) + fabs(D[3]) + 1e-9;
        const double fl = floor(-D[0]);
        if (floor(-D[0] - R) != fl || floor(-D[0] + R) != fl || !(fl < 0.0) || !(fl > -1e6)) {
            bad = 1;
        } else {
            mm[tid] = (int)fl;
            atomicMin(&mmin, (int)fl);
            atomicMax(&mmax, (int)fl);
            for (int n = 0; n < TQ; ++n) {
                const double x = X.tab_node[n];
                eps[n][tid] = -fma(x, fma(x, fma(x, D[3], D[2]), D[1]), D[0]) - fl;
            }
        }
    }
    __syncthreads();
    const int KW = (mmax > 0 ? mmax : 0) - mmin + T;
    if (bad || KW > tab_kw || KW + 7 > 64 || P.HL + mmin - h < 1) {
        if (tid < FX_META) meta[FX_META * k + tid] = 0;
        return;
    }
    for (int i = tid; i < TQ * NTERM; i += blockDim.x)
        if (i % 7 < qn) {
            const double e = eps[i / NTERM][i % NTERM];
            double L = 1.0, R = 1.0;
            for (int a = 0; a < T; ++a) {
                wt[a * WTT + i] = L;
                L *= fma(e, lc1[a], lc0[a]);
            }
            for (int a = T - 1; a >= 0; --a) {
                wt[a * WTT + i] *= ((T - 1 - a) & 1) ? -R : R;
                R *= fma(e, rc1[a], rc0[a]);
            }
        }
    __syncthreads();
    bool ok = true;
    float most = 0.0f;   // bound of the stencils over the piece, the orders' magnitudes added
    for (int i = tid; i < 12 * KW; i += blockDim.x) {
        const int cs = i / KW, tap = i - cs * KW, ch = cs >> 2, sl = cs & 3;
        double V[TQ], b[TQ];
        for (int n = 0; n < TQ; ++n) V[n] = 0.0;
        for (int x = 0; x < 4; ++x) {
            const int tm = c_slots.term[ch][sl][x], c = tm >> 3, q = tm & 7;
            if (q > qn) continue;
            const int id = (ch * 2 + c) * 7 + q - 1, a = q ? tap - (mm[id] - mmin) : (tap == h - mmin ? 0 : -1);
            if (a < 0 || a >= T) continue;
            for (int n = 0; n < TQ; ++n) {
                const double w = q ? wt[a * WTT + n * NTERM + id] : 1.0;
                V[n] += c ? -w : w;
            }
        }
#pragma unroll
        for (int q = 0; q < TQ; ++q) {
            double v = 0.0;
#pragma unroll
            for (int n = 0; n < TQ; ++n) v = fma(V[n], X.tab_cheb[q][n], v);
            b[q] = v;
        }
        const double m[TQ] = {b[0] - b[2] + b[4], b[1] - 3.0 * b[3] + 5.0 * b[5], 2.0 * b[2] - 8.0 * b[4],
                              4.0 * b[3] - 20.0 * b[5], 8.0 * b[4], 16.0 * b[5]};
        ok &= fabs(m[TQ - 1]) < 9e-13;  // 2^-40: the order left out is then below 2^-54
        double sum = 0.0;
        for (int q = 0; q < TQ; ++q) {
            tab[((size_t)k * TQ + q) * 12 * tab_kw + cs * tab_kw + tap] = m[q];
            sum += fabs(m[q]);
        }
        most = fmaxf(most, (float)sum);
    }
    atomicMax(&wmax, (int)__float_as_uint(most));
    ok = !__syncthreads_or(!ok);
    if (tid == 0) {
        // 2 % for blocks that reach past the piece
        const float top = __int_as_float(wmax) * 1.02f;
        const bool in = top > 1e-30f && top < 1e30f;
        meta[FX_META * k] = ok && in ? KW : 0;
        meta[FX_META * k + 1] = mmin;
        meta[FX_META * k + 2] = in ? (int)(__float_as_uint(top) >> 23) - 126 : 0;   // exponent of the scale
        meta[FX_META * k + 3] = 0;
    }
}

template <int NTHR>
void *kernel_of(int kind)
{
    switch (kind) {
        case KIND_PROJECT: return (void *)k_fx64<KIND_PROJECT, NTHR>;
        case KIND_TDI: return (void *)k_fx64<KIND_TDI, NTHR>;
        case KIND_FUSED: return (void *)k_fx64<KIND_FUSED, NTHR>;
        default: return (void *)k_fx64<KIND_LIKE, NTHR>;
    }
}

size_t smem_of(int T)
{
    const size_t proj = FX_PROJ_PLANES + FX_PROJ_W + sizeof(double) * (size_t)T * WNS;
    size_t x = sizeof(double) * (size_t)T * WTS;
    if (x < FX_TDI_PLANES) x = FX_TDI_PLANES;
    const size_t tdi = x + FX_TDI_W;
    return 6 * NY * 8 + (proj > tdi ? proj : tdi);
}

}  // namespace

int fx_max_tile(const FwdParams &P, int order)
{
    const int T = order + 1;
    const int chain = P.HL - (T - 2) / 2 - 2;  // bound of a chained delay, samples
    // merged stencils within 64 taps with the 7 columns' shift; the sample-by-sample window in its place
    if (7 + T + chain + 1 > 64 || 3 + T + 2 * P.lproj_b + 2 > 57) return 0;
    if (NY + 2 * P.sig_b + P.lproj_b + T + 4 > FX_PROJ_PLANES / 16) return 0;
    // forward halos, and the adjoint's window of link samples around a tile of strain
    const int fwd = NY - P.HL - P.HR, adj = NY - T - 2 * P.lproj_b - 2;
    return fwd < adj ? fwd : adj;
}

void fx_tables(const FwdParams &P, int order, int precision, double max_delay, FxTab &X)
{
    X.range_adj = precision == LR_MIXED ? RANGE_ADJ_MIXED : RANGE_ADJ;
    const double pi = 3.14159265358979323846;
    X.icdt = P.inv_dt / C_LIGHT;
    // lags between a link sample and the strain it reads: the reads lie within two arms, one more while one steps
    X.lags = (order + 1 + (int)ceil(2.04 * max_delay * P.inv_dt) + 1 + 15) & ~15;
    if (X.lags > 64) X.lags = 64;
    for (int n = 0; n < NN; ++n) X.node_j[n] = 0.5 * (NY * (1.0 + cos(pi * (2 * n + 1) / (2 * NN))) - 1.0);
    for (int q = 0; q < NN; ++q)
        for (int n = 0; n < NN / 2; ++n)
            X.cheb[q][n] = (q ? 2.0 : 1.0) / NN * cos(pi * ((q * (2 * n + 1)) % (4 * NN)) / (2 * NN));
    for (int n = 0; n < NT; ++n) X.tnode_j[n] = 0.5 * (NY * (1.0 + cos(pi * (2 * n + 1) / (2 * NT))) - 1.0);
    for (int q = 0; q < NT; ++q)
        for (int n = 0; n < NT / 2; ++n)
            X.tcheb[q][n] = (q ? 2.0 : 1.0) / NT * cos(pi * ((q * (2 * n + 1)) % (4 * NT)) / (2 * NT));
    for (int n = 0; n < FX_TAB_Q; ++n) {
        X.tab_node[n] = cos(pi * (2 * n + 1) / (2 * FX_TAB_Q));
        for (int q = 0; q < FX_TAB_Q; ++q)
            X.tab_cheb[q][n] = (q ? 2.0 : 1.0) / FX_TAB_Q * cos(pi * ((q * (2 * n + 1)) % (4 * FX_TAB_Q)) / (2 * FX_TAB_Q));
    }
}

size_t fx_table_bytes(const FwdParams &P, int order)
{
    // plans with very many spline pieces work without the table
    const int T = order + 1, kw = T + (P.HL - (T - 2) / 2 - 2) + 1;
    const size_t per = sizeof(double) * FX_TAB_Q * 12 * (size_t)kw + FX_META * sizeof(int);
    return P.to.nint <= FX_TAB_PIECES ? per * (size_t)P.to.nint : 0;
}

int fx_table_build(const FwdParams &P, int order, FxPlan *F)
{
    const int T = order + 1, kw = T + (P.HL - (T - 2) / 2 - 2) + 1;
    double *tab = static_cast<double *>(F->mem);
    int *meta = reinterpret_cast<int *>(tab + (size_t)P.to.nint * FX_TAB_Q * 12 * kw);
    const size_t smem = sizeof(double) * (size_t)T * (FX_TAB_Q * NTERM + 1);
    cudaError_t e = cudaFuncSetAttribute((const void *)k_fx_table, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    cudaEvent_t ev = nullptr;
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
    if (e != cudaSuccess) return (int)e;
    k_fx_table<<<P.to.nint, 256, smem, 0>>>(P, F->tab, T, tab, meta, kw);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaEventRecord(ev, 0);
    if (e != cudaSuccess) {
        cudaEventDestroy(ev);
        return (int)e;
    }
    F->ready = ev;
    F->tab.tab = tab;
    F->tab.meta = meta;
    F->tab.tab_kw = kw;
    return 0;
}

void fx_plan_free(FxPlan *F)
{
    if (!F) return;
    if (F->ready) cudaEventDestroy((cudaEvent_t)F->ready);
    if (F->mem) cudaFree(F->mem);  // waits for the device
    delete F;
}

// The launch's parameters.  Until the table's kernel is known to be done the stream waits for it; a captured
// launch cannot (the event was recorded outside the capture), there the host waits.  While a stream is being
// captured in global mode, by this thread or another, event calls are refused and break that capture: the event
// belongs to no capture, so they are made in relaxed mode.
int fx_table_for(FxPlan *F, void *str, FxTab *X)
{
    const cudaStream_t stream = (cudaStream_t)str;
    *X = F->tab;
    if (!F->ready) return 0;
    const cudaEvent_t ev = (cudaEvent_t)F->ready;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    cudaError_t e = cudaStreamIsCapturing(stream, &cap);
    if (e != cudaSuccess) return (int)e;
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    e = cudaThreadExchangeStreamCaptureMode(&mode);
    if (e != cudaSuccess) return (int)e;
    if (cap != cudaStreamCaptureStatusNone) {
        e = cudaEventSynchronize(ev);
    } else {
        e = cudaEventQuery(ev);
        if (e == cudaErrorNotReady) {
            cudaGetLastError();
            e = cudaStreamWaitEvent(stream, ev);
        } else if (e == cudaSuccess) {
            F->ready = nullptr;
            e = cudaEventDestroy(ev);
        }
    }
    const cudaError_t e2 = cudaThreadExchangeStreamCaptureMode(&mode);
    return (int)(e != cudaSuccess ? e : e2);
}

int launch_fx64(int kind, int order, const FwdParams &P, int sms, void *stream)
{
    if (P.src.tile_off && !P.src.skyc && kind != KIND_TDI) return (int)cudaErrorInvalidValue;  // sky frames of a batch
    const int nthr = P.total_tiles >= 0 && P.total_tiles <= sms ? 512 : 256;
    void *k = nthr == 512 ? kernel_of<512>(kind) : kernel_of<256>(kind);
    int T = order + 1;
    const size_t smem = smem_of(T);
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return (int)e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, nthr, smem);
    if (e != cudaSuccess) return (int)e;
    if (per_sm < 1) return (int)cudaErrorLaunchOutOfResources;
    int64_t grid = (int64_t)per_sm * sms;
    if (P.total_tiles >= 0 && P.total_tiles < grid) grid = P.total_tiles;
    if (grid < 1) grid = 1;
    FxTab X;
    if (const int te = fx_table_for(P.fx, stream, &X)) return te;
    void *args[] = {(void *)&P, (void *)&X, (void *)&T};
    return (int)cudaLaunchKernel(k, dim3((unsigned)grid), dim3(nthr), args, smem, (cudaStream_t)stream);
}

}  // namespace lr
