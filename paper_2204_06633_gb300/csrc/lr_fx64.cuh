// Device code shared by the tensor-core FP64 kernels (lr_fx64.cu forward, lr_fxbwd.cu adjoint): fixed-point
// digits, the contraction, and the expansion of the projection's merged stencils over a block.  The method is
// described in lr_fx64.cu.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "lr_device.cuh"
#include "lr_fx64.h"
#include "lr_tdi_table.cuh"

namespace lr {
namespace {

constexpr int NY = FX_ROWS;       // rows (link samples or outputs) of a block
constexpr int DL = NY + 64;       // staged samples per digit plane
constexpr int WS = 72;            // bytes per digit row of a stencil: 7 zeros, the taps, zeros
constexpr int NN = FX_NODES, NT = FX_TDI_NODES;
constexpr int MAXSEG = 10;
constexpr int GP = 32;            // spacing of the projection's grid samples
constexpr int NG = NY / GP + 1;
constexpr int GT = 64;            // spacing of the TDI grid samples
constexpr int NGT = NY / GT + 1;
constexpr int NTERM = 42;
constexpr int WTS = 4 * NTERM + 1;   // row length of the TDI node weights (odd: no bank conflicts)
constexpr int WNS = NN * 9;
static_assert(2 * WNS <= 160 && NN * 6 == 48, "roles of node_weights");
// merged TDI taps per thread: at most 12 stencils of 57 taps
__host__ __device__ constexpr int tap_reps(int nthr) { return (12 * 57 + nthr - 1) / nthr; }
constexpr int NSTR = DL / 32;     // stretches of 32 samples of a staged series
// Most binary orders between a block's largest value and the largest of any window that an output reads.  The
// fixed point is relative to the block, so a quiet output beside a loud stretch loses those bits; beyond the
// limit the block is evaluated sample by sample.  Error of such outputs against binary128, digits over sample
// kernels (orders 11 to 41, a stretch 2^k of the rest): projection and TDI at 0.1 mHz 0.07 to 0.13 for k = 0, 0.5 to
// 0.8 for 3, 1.1 to 1.7 for 4, 17 to 26 for 8; TDI alone at 1 mHz 0.9 to 1.1, 1.0 to 1.3, 1.4 to 1.8, 2.4 to
// 3.4 for 5, 16 to 23; strain gradients 0.66 for k = 0, 0.89 for 6, 2.1 for 8.  Link series cross zero: a 0.1 mHz
// source's stretches of 32 samples reach 2^5, any two of them 2^4, and 1 % of its blocks (a fifth at an order less)
// would be evaluated sample by sample without TDI's extra order for single stretches.  The sky gradient is a sum over the block,
// in which the loud part has its own term.  Mixed plans' adjoints keep 43 bits of the quietest part, more than the
// float-float kernels that they would run on otherwise (5e-13 from FP64, the digits 7e-14 at k = 11), in a tenth of the
// time of the sample form.
constexpr int RANGE_PROJ = 3, RANGE_TDI = 4, RANGE_ADJ = 5, RANGE_ADJ_MIXED = 12, RANGE_SKY = 12;
// the last order's coefficient must be below 2^-45 of the stencil's scale: the next one is then below 2^-53
constexpr unsigned long long LAST_MAX = 1024;

// digits of order q that are left out at the top: |b_q| < 2^-8z of the stencil's scale
__host__ __device__ constexpr int zq(bool tdi, int q)
{
    return tdi ? (q == 0 ? 0 : 2 * q - 1) : (q == 0 ? 0 : q < 5 ? q - 1 : q - 2);
}
__host__ __device__ constexpr int digit_row(bool tdi, int q)  // first digit row of order q (closed form: folds at compile time)
{
    return tdi ? (q == 0 ? 0 : q == 1 ? 7 : q == 2 ? 13 : q == 3 ? 17 : 19)
               : (q <= 2 ? 7 * q : q == 3 ? 20 : q == 4 ? 25 : q == 5 ? 29 : q == 6 ? 33 : q == 7 ? 36 : 38);
}
constexpr int PD = digit_row(false, NN), TD = digit_row(true, NT);  // digit rows per stencil: 38, 19

__constant__ int c_lr[6] = {0, 1, 2, 0, 2, 1}, c_ls[6] = {1, 2, 0, 2, 1, 0};
__constant__ int c_by_emitter[3][2] = {{2, 5}, {0, 4}, {1, 3}};
__constant__ TdiTab c_tdifx = make_tdi_tab();

// per channel the four links it reads, and per (channel, link) its reads: (chain, q) pairs
struct SlotTab {
    signed char link[3][4];
    signed char term[3][4][4];  // 8 * chain + q
};
__host__ __device__ constexpr SlotTab make_slots()
{
    SlotTab s{};
    const TdiTab t = make_tdi_tab();
    for (int ch = 0; ch < 3; ++ch) {
        int used = 0, n[4] = {0, 0, 0, 0};
        for (int c = 0; c < 2; ++c)
            for (int q = 0; q < CHAIN_TERMS; ++q) {
                int k = 0;
                while (k < used && s.link[ch][k] != t.link[ch][c][q]) ++k;
                if (k == used) s.link[ch][used++] = t.link[ch][c][q];
                s.term[ch][k][n[k]++] = (signed char)(8 * c + q);
            }
    }
    return s;
}
__constant__ SlotTab c_slots = make_slots();

struct Shared {
    TileInfo ti;
    SkyConst skc;
    double lc1[64], lc0[64], rc1[64], rc0[64];  // Lagrange factors (prefix, suffix) of the nodes
    union {  // the projection's grid and nodes, then the TDI's
        struct {
            double npos[NN][9], nodeu[NN * 9], ncf[NN][12];
            float fg[NG][9];
            int mg[NG][10];
        };
        struct {
            double lg[NGT][6], lnode[NT][6];
            int mgt[NGT][NTERM + 1];
            float fgt[NGT][NTERM];
        };
    };
    int segm[MAXSEG][NTERM + 1];  // stencil positions (9 or 42) and the spline piece of each segment
    int segj[MAXSEG + 1];
    double xc, xs;
    int nseg, nlist, fast;
    unsigned brk[NY / 32];
    int list[NTERM * 8 + 8];
    int mmin, mmax;
    int cmax[6], wexp[6];
    unsigned st[3][NSTR];   // largest high word per stretch, of each set of series that one output reads
    unsigned long long qor[NN];  // OR of the coefficients' magnitudes per order
    int nq, last;                // orders in use; whether those above 0 have their last digit only
    int bad;
    double red[2 * 16];
};

__device__ __forceinline__ void mma_f16(float *c, const uint32_t *a, uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// two digit bytes (biased by 128) to two halves: 0x6400 | u is 1024 + u, minus 1152 is the digit
__device__ __forceinline__ uint32_t digits_h2(uint32_t bytes, uint32_t sel)
{
    uint32_t v, r;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(v) : "r"(bytes), "r"(0x64646464u), "r"(sel));
    asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(0x64806480u));
    return r;
}

// digit + next digit / 256, rounded to half (11 bits)
__device__ __forceinline__ uint32_t extend_h2(uint32_t d, uint32_t next)
{
    uint32_t r;
    asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(r) : "r"(next), "r"(0x1c001c00u), "r"(d));
    return r;
}

__device__ __forceinline__ double pow2(int e) { return __longlong_as_double((long long)(1023 + e) << 52); }

// balanced digits: bytes 1..6 of v + 0x808080808080 are the digits plus 128, the rest is digit 0
constexpr long long DIGIT_BIAS = 0x808080808080ll;

// ---------------------------------------------------------------- contraction
// acc[i][L][.] += the level sums of orders QF .. QF + NQ - 1 over `parts` series of `nks` steps of 16 taps
template <int QF, int NQ, bool TDI, bool LAST = false>
__device__ __forceinline__ void contract(float (&acc)[NQ][7][4], const unsigned char *a_lane,
                                         const unsigned char *w_lane, uint32_t sh, int nks, const signed char *links)
{
    constexpr int ZM = LAST ? 6 : zq(TDI, QF);  // the smallest z of the group
    constexpr int NA = ZM ? 8 - ZM : 7;  // digit planes of the series that it needs
    constexpr int PARTS = TDI ? 4 : 2, ROWS = TDI ? TD : PD;
    constexpr int RS = TDI ? 16 : 8;     // bytes between rows of the left operand: 8 or 4 samples
#pragma unroll
    for (int i = 0; i < NQ; ++i)
#pragma unroll
        for (int L = 0; L < 7; ++L)
#pragma unroll
            for (int r = 0; r < 4; ++r) acc[i][L][r] = 0.0f;
#pragma unroll 1
    for (int part = 0; part < PARTS; ++part) {
        const unsigned char *pa = a_lane + (TDI ? links[part] : part) * (7 * DL * 2);
        const unsigned char *pw = w_lane + part * ROWS * WS;
#pragma unroll 1
        for (int ks = 0; ks < nks; ++ks, pa += 32, pw += 16) {
            uint32_t a[NA][4];
#pragma unroll
            for (int k = 0; k < NA; ++k) {
                const uint2 lo = *reinterpret_cast<const uint2 *>(pa + k * DL * 2);
                const uint2 hi = *reinterpret_cast<const uint2 *>(pa + k * DL * 2 + 8 * RS);
                a[k][0] = lo.x; a[k][1] = hi.x; a[k][2] = lo.y; a[k][3] = hi.y;
            }
#pragma unroll
            for (int i = 0; i < NQ; ++i) {
                const int z = zq(TDI, QF + i), row = digit_row(TDI, QF + i);
#pragma unroll
                for (int d = LAST ? 6 : z; d < 7; ++d) {
                    const uint32_t *w = reinterpret_cast<const uint32_t *>(pw + (row + d - z) * WS);
                    const uint32_t u = __funnelshift_r(w[0], w[1], sh);
                    const uint32_t b0 = digits_h2(u, 0x4140u), b1 = digits_h2(u, 0x4342u);
#pragma unroll
                    for (int k = 0; k < 6 - d; ++k) mma_f16(acc[i][d + k], a[k], b0, b1);
                    // level 6 takes level 7 along: its series digit is extended by the next one
                    if (d == 0) {
                        mma_f16(acc[i][6], a[6], b0, b1);
                    } else {
                        uint32_t x[4];
#pragma unroll
                        for (int r = 0; r < 4; ++r) x[r] = extend_h2(a[6 - d][r], a[7 - d][r]);
                        mma_f16(acc[i][6], x, b0, b1);
                    }
                }
            }
        }
    }
}

// level sums of one order to fixed point (unit: an eighth of level 5)
template <int Z>
__device__ __forceinline__ long long levels(const float (&acc)[7][4], int r)
{
    long long v = 0;
#pragma unroll
    for (int L = Z; L < 6; ++L) v = v * 256 + (long long)__float2int_rn(acc[L][r]);
    return v * 8 + __float2int_rn(acc[6][r] * 0.03125f);
}

// (kappa * b) >> S with rounding, |kappa| <= 511
template <int S>
__device__ __forceinline__ long long mul_nu(long long b, int kappa)
{
    const unsigned k = (unsigned)(kappa < 0 ? -kappa : kappa);
    const long long hi = (long long)(int)(b >> 32) * (long long)(int)k;
    const long long lo = (long long)((unsigned long long)(unsigned)b * (unsigned long long)k);
    const long long r = (hi << (32 - S)) + ((lo + (1ll << (S - 1))) >> S);
    return kappa < 0 ? -r : r;
}

// one group's part of Clenshaw's recurrence (orders QF + NQ - 1 down to QF, q >= 1 steps only)
template <int QF, int NQ, bool TDI>
__device__ __forceinline__ void clenshaw(const float (&acc)[NQ][7][4], const int *kappa, long long *b1, long long *b2)
{
    static_assert(QF >= 1, "order 0 closes the recurrence");
#pragma unroll
    for (int r = 0; r < 4; ++r) {
#pragma unroll
        for (int i = NQ - 1; i >= 0; --i) {
            long long v;
            switch (zq(TDI, QF + i)) {
                case 0: v = levels<0>(acc[i], r); break;
                case 1: v = levels<1>(acc[i], r); break;
                case 2: v = levels<2>(acc[i], r); break;
                case 3: v = levels<3>(acc[i], r); break;
                case 4: v = levels<4>(acc[i], r); break;
                case 5: v = levels<5>(acc[i], r); break;
                default: v = levels<6>(acc[i], r); break;
            }
            const long long nb = v + mul_nu<8>(b1[r], kappa[r]) - b2[r];
            b2[r] = b1[r];
            b1[r] = nb;
        }
    }
}

// ---------------------------------------------------------------- Lagrange weights and scalar reads
// centered Lagrange weights at eps (prefix and suffix products), written with a stride
__device__ __forceinline__ void lagrange_to(const Shared &S, int T, double e, double *w, int stride)
{
    double L = 1.0;
    for (int a = 0; a < T; ++a) {
        w[a * stride] = L;
        L *= fma(e, S.lc1[a], S.lc0[a]);
    }
    double R = 1.0;
    for (int a = T - 1; a >= 0; --a) {
        const double v = w[a * stride] * R;
        w[a * stride] = ((T - 1 - a) & 1) ? -v : v;
        R *= fma(e, S.rc1[a], S.rc0[a]);
    }
}

// the Horner form of lr_device.cuh (horner1) with the factors from the tables
__device__ __forceinline__ double read_scalar(const Shared &S, int T, const double *s, int64_t base, double u,
                                              int64_t w_lo, int wlen, int *err)
{
    const int h = (T - 2) / 2;
    const double fl = floor(u), e = u - fl;
    const int64_t st = base + (int64_t)fl - h - w_lo;
    if (st < 0 || st + T > wlen) {
        atomicOr(err, ERR_WINDOW);
        return 0.0;
    }
    const double *p = s + st;
    double L = -1.0, acc = -p[0];
    for (int j = 1; j < T; ++j) {
        L = L * -fma(e, S.lc1[j - 1], S.lc0[j - 1]);
        acc = fma(acc, fma(e, S.rc1[j], S.rc0[j]), L * p[j]);
    }
    return acc;
}

// ---------------------------------------------------------------- positions of the reads
// whole part of a read's position, kept where differences of two fit an int: positions run away where an orbit's
// end pieces are continued far outside its knots, and the blocks there are sent to the sample form
constexpr int STENCIL_FAR = 1 << 28;
__device__ __forceinline__ int stencil_at(double u)
{
    const int m = (int)floor(u);
    return m < -STENCIL_FAR ? -STENCIL_FAR : m > STENCIL_FAR ? STENCIL_FAR : m;
}

__device__ __forceinline__ const Coef4 *piece_row(const OrbitDev &o, int k) { return reinterpret_cast<const Coef4 *>(o.coef) + (size_t)k * NSERIES; }

// spline piece of time t and the coordinate within it; forced >= 0: that piece, continued
__device__ __forceinline__ const Coef4 *row_at(const OrbitDev &o, double t, int forced, double *x, int *piece)
{
    const double u = (t - o.t_first) * o.inv_dk;
    int k = forced;
    if (forced < 0) {
        k = (int)floor(u);
        k = k < 0 ? 0 : (k > o.nint - 1 ? o.nint - 1 : k);
    }
    *piece = k;
    *x = u - (double)k;
    return piece_row(o, k);
}

// spacecraft s at time t: k.x/(c dt) and, when pos is not null, its position
__device__ __forceinline__ double sigma_at(const FwdParams &P, const FxTab &X, const SkyConst &S, const Coef4 *row, double x, int s,
                                           double *pos)
{
    double v[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) v[d] = cubic(ldg4(row + 3 * s + d), x);
    if (pos) {
#pragma unroll
        for (int d = 0; d < 3; ++d) pos[3 * s + d] = v[d];
    }
    return (S.k[0] * v[0] + S.k[1] * v[1] + S.k[2] * v[2]) * X.icdt;
}

// positions of the three reads of spacecraft s (its reception, the emissions to the two others)
__device__ __forceinline__ void reads_of(const FwdParams &P, const FxTab &X, const SkyConst &S, const Coef4 *row, double x, int s,
                                         double u0, double *u, double *pos)
{
    const double sig = sigma_at(P, X, S, row, x, s, pos);
    u[0] = u0 - sig;
#pragma unroll
    for (int i = 0; i < 2; ++i) u[1 + i] = u0 - cubic(ldg4(row + 9 + c_by_emitter[s][i]), x) * P.inv_dt - sig;
}

// the same at expansion node n, with the spacecraft's position, on a given spline piece
__device__ __forceinline__ void node_reads(const FwdParams &P, const FxTab &X, Shared &S, double t_lo, double u0, int n, int s, int piece)
{
    double x, u[3];
    int k;
    const Coef4 *row = row_at(P.po, t_lo + X.node_j[n] * P.dt, piece, &x, &k);
    reads_of(P, X, S.skc, row, x, s, u0, u, S.npos[n]);
#pragma unroll
    for (int i = 0; i < 3; ++i) S.nodeu[n * 9 + (i == 0 ? s : 3 + c_by_emitter[s][i - 1])] = u[i];
}

// position (samples, relative to the row) of read rd (0-2 receptions, 3 + l emissions) at time t
__device__ __forceinline__ double read_pos(const FwdParams &P, const FxTab &X, const SkyConst &S, double u0, double t, int rd, int *piece)
{
    double x;
    const Coef4 *row = row_at(P.po, t, -1, &x, piece);
    const int s = rd < 3 ? rd : c_ls[rd - 3];
    const double sig = sigma_at(P, X, S, row, x, s, nullptr);
    return rd < 3 ? u0 - sig : u0 - cubic(ldg4(row + 9 + rd - 3), x) * P.inv_dt - sig;
}

// chained delay (samples) of a term (channel, chain, q) at time t
__device__ __forceinline__ double chain_delay(const FwdParams &P, double t, int term, int *piece)
{
    double x;
    const Coef4 *row = row_at(P.to, t, -1, &x, piece);
    const int cc = term / 7, q = term % 7 + 1;
    double D = 0.0;
    for (int k = 1; k <= q; ++k) D += cubic(ldg4(row + 9 + c_tdifx.pair[cc >> 1][cc & 1][k]), x) * P.inv_dt;
    return D;
}

// bits of brk -> segment starts (thread 0); sets bad when there are too many
__device__ __forceinline__ void collect_segments(Shared &S, int rows)
{
    int n = 1;
    S.segj[0] = 0;
    for (int w = 0; w < NY / 32; ++w) {
        unsigned b = S.brk[w];
        while (b) {
            const int j = 32 * w + __ffs(b) - 1;
            b &= b - 1;
            if (j <= 0 || j >= rows) continue;
            if (n >= MAXSEG) {
                S.bad = 1;
                break;
            }
            S.segj[n++] = j;
        }
    }
    S.segj[n] = rows;
    S.nseg = n;
}

__device__ __forceinline__ unsigned abs_hi(double v) { return (unsigned)__double2hiint(v) & 0x7fffffffu; }

__device__ __forceinline__ unsigned warp_max(unsigned v) { return __reduce_max_sync(0xffffffffu, v); }

// From the stretches' maxima (of `sets` sets, over n samples): the block's largest high word, the exponent e with max
// < 2^e, and whether every window of taps samples that holds anything but zeros comes within `bits` orders of it
// (SLACK more where the window may lie in one stretch and the two around it come within `bits`).  Every warp for
// itself.
template <int SLACK>
__device__ __forceinline__ bool range_ok(const unsigned (*st)[NSTR], int sets, int n, int taps, int bits, unsigned *vmax, int *e)
{
    const int lane = threadIdx.x & 31, stretches = (n + 31) >> 5;
    const bool whole = n - 32 * lane >= (taps < 32 ? taps : 32);   // a window fits in the lane's stretch
    unsigned hi = 0, one = 0x7fffffffu, two = 0x7fffffffu;
    for (int c = 0; c < sets; ++c) {
        const unsigned m = lane < stretches ? st[c][lane] : 0u, next = __shfl_down_sync(0xffffffffu, m, 1), w = max(m, next);
        hi = max(hi, m);
        if (m && whole) one = min(one, m);
        if (w && lane < stretches - 1) two = min(two, w);
    }
    hi = warp_max(hi);
    one = __reduce_min_sync(0xffffffffu, one);
    two = __reduce_min_sync(0xffffffffu, two);
    *vmax = hi;
    const int eb = (int)(hi >> 20);
    *e = eb - 1022;
    // a window of more than 32 samples is in two stretches at least
    return eb >= 200 && eb <= 1900 && (taps > 32 || eb - (int)(one >> 20) <= bits + SLACK) && eb - (int)(two >> 20) <= bits;
}

// v * 2^(55 - e), |v| < 2^e, rounded to an integer: shifts of the significand (FP64 conversions issue at a
// 64th of the integer rate)
__device__ __forceinline__ long long to_fixed(double v, int e)
{
    const long long b = __double_as_longlong(v);
    const int E = (int)((b >> 52) & 0x7ff);
    const unsigned long long m = ((unsigned long long)b & 0xfffffffffffffull) | (E ? 1ull << 52 : 0ull);
    const int s = E - e - 1020;  // at most 2 for |v| < 2^e
    unsigned long long r;
    if (s >= 0) r = s < 9 ? m << s : 1ull << 61;   // beyond every digit's range
    else r = s > -60 ? ((m >> (-s - 1)) + 1) >> 1 : 0ull;
    return b < 0 ? -(long long)r : (long long)r;
}

// v * 2^e to FP64, rounded to nearest (ties away), for results in the normal range
__device__ __forceinline__ double from_fixed(long long v, int e)
{
    if (v == 0) return 0.0;
    const unsigned long long a = (unsigned long long)(v < 0 ? -v : v);
    const int z = __clzll((long long)a);
    // significand with its leading one at bit 52; the rounding carry moves into the exponent
    const unsigned long long m = (((a << z) >> 10) + 1) >> 1;
    const unsigned long long bits = m + ((unsigned long long)(1023 + 63 - z + e - 1) << 52);
    return __longlong_as_double((long long)(bits | (v < 0 ? 1ull << 63 : 0ull)));
}

// seven digit planes (halves) of v in units of 2^(e - 55) at index p
__device__ __forceinline__ void digits_to_planes(uint16_t *pl, int p, double v, int e)
{
    const long long X = to_fixed(v, e) + DIGIT_BIAS;
    const uint32_t top = (uint32_t)((int)(X >> 48) + 128);  // 0 .. 256
    const uint32_t lo = (uint32_t)X, hi = (uint32_t)(X >> 32);
    const uint32_t d[7] = {top, (hi >> 8) & 255u, hi & 255u, lo >> 24, (lo >> 16) & 255u, (lo >> 8) & 255u, lo & 255u};
#pragma unroll
    for (int i = 0; i < 7; ++i) {
        uint32_t r;
        asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(0x6400u + d[i]), "r"(0x6480u));
        pl[i * DL + p] = (uint16_t)r;
    }
}

// digit bytes of one stencil coefficient (integer units); false when it needs more than its digits
template <int Z>
__device__ __forceinline__ bool coef_digits(unsigned char *w, long long b)
{
    constexpr long long bias = DIGIT_BIAS & ((1ll << (8 * (6 - Z))) - 1);
    const long long X = b + bias;
    const long long top = X >> (8 * (6 - Z));
    w[0] = (unsigned char)((int)top + 128);
#pragma unroll
    for (int i = 1; i < 7 - Z; ++i) w[i * WS] = (unsigned char)(X >> (8 * (6 - Z - i)));
    return top >= -128 && top <= 127;
}

// coefficient b of a stencil of scale 2^e (integer work: conversions and scalings would be FP64 issue slots)
template <bool TDI, int Q>
__device__ __forceinline__ bool coef_store(unsigned char *w, double b, int e, unsigned long long *mag)
{
    const long long v = to_fixed(b, e);
    mag[Q] |= (unsigned long long)(v < 0 ? -v : v);
    return coef_digits<zq(TDI, Q)>(w + digit_row(TDI, Q) * WS, v);
}

// magnitudes of the block's coefficients per order, over all threads (then count_orders after a barrier)
template <int N>
__device__ __forceinline__ void orders_in_use(Shared &S, const unsigned long long *mag)
{
#pragma unroll
    for (int q = 0; q < N; ++q) {
        const unsigned hi = __reduce_or_sync(0xffffffffu, (unsigned)(mag[q] >> 32));
        const unsigned lo = __reduce_or_sync(0xffffffffu, (unsigned)mag[q]);
        if ((threadIdx.x & 31) == 0 && (hi | lo)) atomicOr(&S.qor[q], (unsigned long long)hi << 32 | lo);
    }
}

// the number of orders in use, and whether the orders above 0 (constant delays and positions: rounding of
// the transform) fit their last digit; ends with a barrier
template <int N>
__device__ __forceinline__ void count_orders(Shared &S)
{
    if (threadIdx.x < 32) {
        const unsigned long long m = threadIdx.x < N ? S.qor[threadIdx.x] : 0;
        const unsigned used = __ballot_sync(0xffffffffu, m != 0), big = __ballot_sync(0xffffffffu, threadIdx.x > 0 && m >= 64);
        if (threadIdx.x == 0) {
            S.nq = 32 - __clz((int)used);
            S.last = big == 0;
        }
    }
    __syncthreads();
}

// ---------------------------------------------------------------- projection stencils
// Positions of the reads are relative to row + floor((t0 - t0h) / dt); u0 is the fraction that is left of that
// offset.  The whole part goes into indices alone: a strain that begins 10^6 samples before the outputs would take
// 20 bits from the reads' fractions (6e-12 of the response, and no block's expansion would fit).
// Segments of rows 0 .. rows - 1 (row 0 at time t_lo) in which no read's stencil steps and the orbit's spline
// piece stays: fills segj, segm, nseg, mmin, mmax and the reads at the expansion nodes.
__device__ void projection_segments(const FwdParams &P, const FxTab &X, Shared &S, double t_lo, double u0, int rows)
{
    const int tid = threadIdx.x;
    // stencil positions on the grid samples, and the reads at the expansion nodes (on row 0's spline piece)
    if (tid < (NG + NN) * 3) {
        const int g = tid / 3, s = tid % 3;
        if (g < NG) {
            double x;
            int piece;
            const Coef4 *row = row_at(P.po, t_lo + (double)(g * GP) * P.dt, -1, &x, &piece);
            if (s == 0) S.mg[g][9] = piece;
            double u[3];
            reads_of(P, X, S.skc, row, x, s, u0, u, nullptr);
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const int rd = i == 0 ? s : 3 + c_by_emitter[s][i - 1];
                const double fl = floor(u[i]);
                S.mg[g][rd] = stencil_at(fl);
                S.fg[g][rd] = (float)(u[i] - fl);
            }
        } else {
            double x;
            int piece;
            row_at(P.po, t_lo, -1, &x, &piece);
            node_reads(P, X, S, t_lo, u0, g - NG, s, piece);
        }
    }
    if (tid < NY / 32) S.brk[tid] = 0;
    if (tid == 192) {
        S.nlist = 0;
        S.bad = 0;
        S.mmin = 1 << 29;
        S.mmax = -(1 << 29);
    }
    __syncthreads();
    // intervals in which a stencil may step or the spline piece changes
    for (int i = tid; i < (NG - 1) * 10; i += blockDim.x) {
        const int g = i / 10, rd = i % 10;
        bool look = S.mg[g][rd] != S.mg[g + 1][rd];
        if (rd < 9) {
            const float a = S.fg[g][rd], b = S.fg[g + 1][rd];
            const int gm = g > 0 ? g - 1 : 0;   // second difference of the position around the interval
            const float d2 = fabsf((float)(S.mg[gm][rd] + S.mg[gm + 2][rd] - 2 * S.mg[gm + 1][rd]) + S.fg[gm][rd] +
                                   S.fg[gm + 2][rd] - 2.0f * S.fg[gm + 1][rd]);
            const float thr = 2e-6f + 2.0f * d2;
            look |= fminf(fminf(a, 1.0f - a), fminf(b, 1.0f - b)) < thr;
        }
        if (look && g * GP < rows) S.list[atomicAdd(&S.nlist, 1)] = i;
    }
    __syncthreads();
    for (int i = tid >> 5; i < S.nlist; i += blockDim.x >> 5) {
        const int g = S.list[i] / 10, rd = S.list[i] % 10, lane = tid & 31;
        const int j = g * GP + lane + 1;   // rows g GP + 1 .. (g + 1) GP against the row before
        int piece;
        const double u = read_pos(P, X, S.skc, u0, t_lo + (double)j * P.dt, rd < 9 ? rd : 0, &piece);
        const int m = rd < 9 ? stencil_at(u) : piece;
        const int prev = __shfl_up_sync(0xffffffffu, m, 1);
        if (m != (lane ? prev : S.mg[g][rd]) && j < NY) atomicOr(&S.brk[j >> 5], 1u << (j & 31));
    }
    __syncthreads();
    if (tid == 0) collect_segments(S, rows);
    __syncthreads();
    const int nseg = S.nseg;
    if (tid < nseg * 10) {
        const int sg = tid / 10, rd = tid % 10;
        int m = S.mg[0][rd];
        if (sg) {
            int piece;
            const double u = read_pos(P, X, S.skc, u0, t_lo + (double)S.segj[sg] * P.dt, rd < 9 ? rd : 0, &piece);
            m = rd < 9 ? stencil_at(u) : piece;
        }
        S.segm[sg][rd] = m;
        if (rd < 9) {
            atomicMin(&S.mmin, m);
            atomicMax(&S.mmax, m);
            if (m <= -STENCIL_FAR || m >= STENCIL_FAR) S.bad = 1;
        }
    }
    __syncthreads();
}

// Lagrange weights wn[T][node, read] and pattern coefficients of segment sg at the expansion nodes.  Starts
// with a barrier in the caller; ends after the last write (a barrier is needed before reading).
__device__ __forceinline__ void node_weights(const FwdParams &P, const FxTab &X, Shared &S, int T, double t_lo, double u0,
                                             int sg, double *wn)
{
    const int tid = threadIdx.x;
    const int *sm = S.segm[sg];
    if (sm[9] != S.segm[sg ? sg - 1 : 0][9] && tid < NN * 3) node_reads(P, X, S, t_lo, u0, tid / 3, tid % 3, sm[9]);
    if (tid >= 192 && tid < 198) S.cmax[tid - 192] = 0;
    if (tid >= 200 && tid < 200 + NN) S.qor[tid - 200] = 0;
    __syncthreads();
    // Lagrange weights at the nodes, two threads per read: prefix products of the lower half and suffix
    // products of the upper half, then each carries on through the other's half.  They fill warps 0 to 4; the
    // links' patterns take 16 lanes of warps 5, 6 and 7 (an FP64 instruction holds its scheduler's pipe for 64
    // cycles however few lanes it has, so the four schedulers get 130 to 155 of them each).
    if (tid < 160) {
        const int id = tid < WNS ? tid : tid - WNS;
        const bool low = tid < WNS, half = tid < 2 * WNS;
        double e = 0.0, run = 1.0;
        double *w = wn + id;
        if (half) {
            e = S.nodeu[id] - (double)sm[id % 9];
            if (low) {
#pragma unroll 4
                for (int a = 0; a < T / 2; ++a) {
                    w[a * WNS] = run;
                    run *= fma(e, S.lc1[a], S.lc0[a]);
                }
            } else {
#pragma unroll 4
                for (int a = T - 1; a >= T / 2; --a) {
                    w[a * WNS] = ((T - 1 - a) & 1) ? -run : run;
                    run *= fma(e, S.rc1[a], S.rc0[a]);
                }
            }
        }
        asm volatile("bar.sync 1, 160;" ::: "memory");
        if (half) {
            if (low) {
#pragma unroll 4
                for (int a = T / 2; a < T; ++a) {
                    w[a * WNS] *= run;
                    run *= fma(e, S.lc1[a], S.lc0[a]);
                }
            } else {
#pragma unroll 4
                for (int a = T / 2 - 1; a >= 0; --a) {
                    w[a * WNS] *= ((T - 1 - a) & 1) ? -run : run;
                    run *= fma(e, S.rc1[a], S.rc0[a]);
                }
            }
        }
    } else if (tid < 256 && (tid & 31) < 16) {
        const int at = ((tid >> 5) - 5) * 16 + (tid & 31), n = at / 6, l = at % 6, r = c_lr[l], s = c_ls[l];
        const SkyConst &K = S.skc;
        const double *x = S.npos[n];
        double d0 = x[3 * r] - x[3 * s], d1 = x[3 * r + 1] - x[3 * s + 1], d2 = x[3 * r + 2] - x[3 * s + 2];
        const double inv = rsqrt(d0 * d0 + d1 * d1 + d2 * d2);
        d0 *= inv; d1 *= inv; d2 *= inv;
        const double un = K.u[0] * d0 + K.u[1] * d1 + K.u[2] * d2;
        const double vn = K.v[0] * d0 + K.v[1] * d1 + K.v[2] * d2;
        const double kn = K.k[0] * d0 + K.k[1] * d1 + K.k[2] * d2;
        const double xip = un * un - vn * vn, xic = 2.0 * un * vn;
        const double gf = 0.5 / (1.0 - kn);
        const double cp = (K.c2p * xip + K.s2p * xic) * gf, cc = (K.c2p * xic - K.s2p * xip) * gf;
        S.ncf[n][2 * l] = cp;
        S.ncf[n][2 * l + 1] = cc;
        // NaN and infinity give the largest keys
        atomicMax(&S.cmax[l], (int)(__float_as_uint((float)fmax(fabs(cp), fabs(cc))) & 0x7fffffffu));
        if (!isfinite(gf)) S.bad = 1;
    }
    __syncthreads();
}

// exponent of a stencil's scale, 2 max|c| with slack for offsets just outside [0, 1)
__device__ __forceinline__ int stencil_exp(int cmax)
{
    const float m = __int_as_float(cmax) * 2.4f;
    return m > 1e-30f && m < 1e30f ? (int)(__float_as_uint(m) >> 23) - 126 : -126;
}

// Digit rows W of segment sg's merged stencils (REV: taps in reverse, one scale for all links); false when the
// expansion does not fit.  Begins and ends with a barrier.
template <bool REV>
__device__ bool projection_stencils(const FwdParams &P, const FxTab &X, Shared &S, int T, double t_lo, double u0,
                                    int sg, int KW, unsigned char *W, double *wn)
{
    const int tid = threadIdx.x, mmin = S.mmin;
    const int *sm = S.segm[sg];
    __syncthreads();  // the previous segment's stencils and nodes are free
    for (int i = tid; i < FX_PROJ_W / 16; i += blockDim.x)
        reinterpret_cast<uint4 *>(W)[i] = make_uint4(0x80808080u, 0x80808080u, 0x80808080u, 0x80808080u);
    node_weights(P, X, S, T, t_lo, u0, sg, wn);
    int cm[6], call = 0;
#pragma unroll
    for (int l = 0; l < 6; ++l) {
        cm[l] = S.cmax[l];
        call = max(call, cm[l]);
    }
    if (tid == 0)
        for (int l = 0; l < 6; ++l) S.wexp[l] = stencil_exp(REV ? call : cm[l]);   // REV: one scale for the sum over the links
    bool fits = !S.bad;
    unsigned long long mag[NN] = {};
    if (fits)
        for (int i = tid; i < 12 * KW; i += blockDim.x) {
            const int lp = i / KW, tap = i - lp * KW, l = lp >> 1;
            const int ae = tap - (sm[3 + l] - mmin), ar = tap - (sm[c_lr[l]] - mmin);
            const bool ine = ae >= 0 && ae < T, inr = ar >= 0 && ar < T;
            const double *we = wn + ae * WNS + 3 + l, *wr = wn + ar * WNS + c_lr[l];
            double V[NN];
#pragma unroll
            for (int n = 0; n < NN; ++n)
                V[n] = S.ncf[n][lp] * ((ine ? we[9 * n] : 0.0) - (inr ? wr[9 * n] : 0.0));
            unsigned char *w = W + lp * PD * WS + 7 + (REV ? KW - 1 - tap : tap);
            // Chebyshev coefficients: nodes n and NN - 1 - n are opposite
            double e[NN / 2], o[NN / 2];
#pragma unroll
            for (int n = 0; n < NN / 2; ++n) {
                e[n] = V[n] + V[NN - 1 - n];
                o[n] = V[n] - V[NN - 1 - n];
            }
            double b[NN];
#pragma unroll
            for (int q = 0; q < NN; ++q) {
                double v = 0.0;
#pragma unroll
                for (int n = 0; n < NN / 2; ++n) v = fma((q & 1) ? o[n] : e[n], X.cheb[q][n], v);
                b[q] = v;
            }
            const int ew = stencil_exp(REV ? call : S.cmax[l]);
            fits &= coef_store<false, 0>(w, b[0], ew, mag);
            fits &= coef_store<false, 1>(w, b[1], ew, mag);
            fits &= coef_store<false, 2>(w, b[2], ew, mag);
            fits &= coef_store<false, 3>(w, b[3], ew, mag);
            fits &= coef_store<false, 4>(w, b[4], ew, mag);
            fits &= coef_store<false, 5>(w, b[5], ew, mag);
            fits &= coef_store<false, 6>(w, b[6], ew, mag);
            unsigned long long m7[NN] = {};
            fits &= coef_store<false, 7>(w, b[7], ew, m7) && m7[7] < LAST_MAX;
            mag[7] |= m7[7];
        }
    orders_in_use<NN>(S, mag);
    if (__syncthreads_or(!fits)) return false;
    count_orders<NN>(S);
    return true;
}

// ---------------------------------------------------------------- the plan's TDI table
// Chebyshev coefficients of one tap over the block, from the piece's polynomial p (degree 5 in its coordinate
// on [-1, 1]) moved to the block's centre xc and scaled by its half width xs
__device__ __forceinline__ void table_coefs(double *p, double xc, double xs, double *b)
{
#pragma unroll
    for (int k = 0; k < NT; ++k)
#pragma unroll
        for (int q = FX_TAB_Q - 2; q >= k; --q) p[q] = fma(xc, p[q + 1], p[q]);
    const double m1 = p[1] * xs, x2 = xs * xs, m2 = p[2] * x2, m3 = p[3] * (x2 * xs);
    b[0] = fma(0.5, m2, p[0]);
    b[1] = fma(0.75, m3, m1);
    b[2] = 0.5 * m2;
    b[3] = 0.25 * m3;
}

// Segments of a block on the plan's expansion table (one per spline piece, at most two): their starts and
// pieces, or 0 when a piece has no entry or the block leaves the orbit's knots: the end pieces are continued
// there, and the table's polynomials and their one stencil position hold within a piece only.  One thread.
__device__ int table_segments(const FwdParams &P, const FxTab &X, Shared &S, double t_lo, int nb)
{
    double x;
    int a, b;
    row_at(P.to, t_lo, -1, &x, &a);
    const double ua = x + (double)a;
    row_at(P.to, t_lo + (double)(nb - 1) * P.dt, -1, &x, &b);
    if (ua < 0.0 || x + (double)b > (double)P.to.nint) return 0;
    if (b > a + 1 || X.meta[FX_META * a] == 0 || X.meta[FX_META * b] == 0) return 0;
    S.nseg = 1 + (b > a);
    S.segj[0] = 0;
    S.segm[0][NTERM] = a;
    S.segj[S.nseg] = nb;
    if (b > a) {  // first output of the second piece
        int i = (int)(((double)b - ua) / (P.dt * P.to.inv_dk)), k;
        i = i < 2 ? 1 : i - 1;
        for (; i < nb - 1; ++i) {
            row_at(P.to, t_lo + (double)i * P.dt, -1, &x, &k);
            if (k >= b) break;
        }
        S.segj[1] = i;
        S.segm[1][NTERM] = b;
    }
    return 1;
}

// The TDI's segments where the plan has no table: stencil steps of all delayed reads on a grid of samples
// and every sample near one; fills segj, segm, nseg, mmin and mmax.
__device__ void find_tdi_segments(const FwdParams &P, Shared &S, double t_lo, int nb)
{
    const int tid = threadIdx.x, qn = P.q_terms;
    const uint32_t lane = tid & 31, warp = tid >> 5;
    if (tid < NGT * 6) {
        const int g = tid / 6, l = tid % 6;
        double x;
        int piece;
        const Coef4 *row = row_at(P.to, t_lo + (double)(g * GT) * P.dt, -1, &x, &piece);
        S.lg[g][l] = cubic(ldg4(row + 9 + l), x) * P.inv_dt;
        if (l == 0) S.mgt[g][NTERM] = piece;
    }
    __syncthreads();
    if (tid < NGT * 6) {
        const int g = tid / 6, cc = tid % 6;
        double D = 0.0;
        for (int q = 1; q <= qn; ++q) {
            D += S.lg[g][c_tdifx.pair[cc >> 1][cc & 1][q]];
            const double fl = floor(-D);
            S.mgt[g][cc * 7 + q - 1] = stencil_at(fl);
            S.fgt[g][cc * 7 + q - 1] = (float)(-D - fl);
        }
    }
    __syncthreads();
    for (int i = tid; i < (NGT - 1) * 7; i += blockDim.x) {  // interval, position in the chain (or the piece)
        const int g = i / 7, q = i % 7;
        if (g * GT >= nb) continue;
        for (int cc = 0; cc < 6; ++cc) {
            if (q >= qn) break;
            const int tm = cc * 7 + q;
            const float a = S.fgt[g][tm], b = S.fgt[g + 1][tm];
            const int gm = g > 0 ? g - 1 : 0;
            const float d2 = fabsf((float)(S.mgt[gm][tm] + S.mgt[gm + 2][tm] - 2 * S.mgt[gm + 1][tm]) + S.fgt[gm][tm] +
                                   S.fgt[gm + 2][tm] - 2.0f * S.fgt[gm + 1][tm]);
            const float thr = 1e-6f + 2.0f * d2;
            if (S.mgt[g][tm] != S.mgt[g + 1][tm] || fminf(fminf(a, 1.0f - a), fminf(b, 1.0f - b)) < thr)
                S.list[atomicAdd(&S.nlist, 1)] = g * (NTERM + 1) + tm;
        }
        if (q == 0 && S.mgt[g][NTERM] != S.mgt[g + 1][NTERM]) S.list[atomicAdd(&S.nlist, 1)] = g * (NTERM + 1) + NTERM;
    }
    __syncthreads();
    for (int i = warp; i < S.nlist; i += blockDim.x >> 5) {
        const int g = S.list[i] / (NTERM + 1), tm = S.list[i] % (NTERM + 1);
        int last = 0;
        for (int c = 0; c <= GT; c += 32) {
            const int j = g * GT + c + (int)lane;
            int piece;
            const double D = chain_delay(P, t_lo + (double)j * P.dt, tm < NTERM ? tm : 0, &piece);
            const int m = tm < NTERM ? stencil_at(-D) : piece;
            int prev = __shfl_up_sync(0xffffffffu, m, 1);
            if (lane == 0) prev = c ? last : m;
            last = __shfl_sync(0xffffffffu, m, 31);
            if (m != prev && c + (int)lane <= GT && j < NY) atomicOr(&S.brk[j >> 5], 1u << (j & 31));
        }
    }
    __syncthreads();
    if (tid == 0) collect_segments(S, nb);
    __syncthreads();
    const int nseg = S.nseg;
    for (int i = tid; i < nseg * (NTERM + 1); i += blockDim.x) {
        const int sg = i / (NTERM + 1), tm = i % (NTERM + 1);
        int piece;
        const double D = chain_delay(P, t_lo + (double)S.segj[sg] * P.dt, tm < NTERM ? tm : 0, &piece);
        const int m = tm < NTERM ? stencil_at(-D) : piece;
        S.segm[sg][tm] = m;
        if (tm < NTERM && tm % 7 < qn) {
            atomicMin(&S.mmin, m);
            atomicMax(&S.mmax, m);
        }
    }
}

// Digit rows W of segment sg's merged TDI stencils (REV: taps in reverse) from the plan's table, whose entries
// are on their way while the rows are filled; *ew_out: their scale.  False when the coefficients do not fit
// their digits.  Begins and ends with a barrier.
template <bool REV, int NTHR>
__device__ __forceinline__ bool tdi_stencils(const FwdParams &P, const FxTab &X, Shared &S, double t_lo, int sg, int KW,
                                             unsigned char *W, int *ew_out)
{
    const int tid = threadIdx.x, piece = S.segm[sg][NTERM];
    double p[tap_reps(NTHR)][FX_TAB_Q];
    const double *c = X.tab + (size_t)piece * FX_TAB_Q * 12 * X.tab_kw;
#pragma unroll
    for (int rep = 0; rep < tap_reps(NTHR); ++rep) {
        const int i = tid + NTHR * rep;
        if (i < 12 * KW) {
            const int at = (i / KW) * X.tab_kw + i % KW;
#pragma unroll
            for (int q = 0; q < FX_TAB_Q; ++q) p[rep][q] = __ldg(c + q * 12 * X.tab_kw + at);
        }
    }
    const int ew = X.meta[FX_META * piece + 2];
    *ew_out = ew;
    __syncthreads();
    for (int i = tid; i < FX_TDI_W / 16; i += NTHR)
        reinterpret_cast<uint4 *>(W)[i] = make_uint4(0x80808080u, 0x80808080u, 0x80808080u, 0x80808080u);
    if (tid < NT) S.qor[tid] = 0;
    if (tid == NTHR - 1) {
        S.xc = 2.0 * ((t_lo + 0.5 * (NY - 1) * P.dt - P.to.t_first) * P.to.inv_dk - (double)piece) - 1.0;
        S.xs = NY * P.dt * P.to.inv_dk;
    }
    __syncthreads();
    const double xc = S.xc, xs = S.xs;
    bool fits = true;
    unsigned long long mag[NT] = {};
#pragma unroll
    for (int rep = 0; rep < tap_reps(NTHR); ++rep) {
        const int i = tid + NTHR * rep;
        if (i < 12 * KW) {
            const int cs = i / KW, tap = i - cs * KW;
            unsigned char *w = W + cs * TD * WS + 7 + (REV ? KW - 1 - tap : tap);
            double b[NT];
            table_coefs(p[rep], xc, xs, b);
            fits &= coef_store<true, 0>(w, b[0], ew, mag);
            fits &= coef_store<true, 1>(w, b[1], ew, mag);
            fits &= coef_store<true, 2>(w, b[2], ew, mag);
            fits &= coef_store<true, 3>(w, b[3], ew, mag);
        }
    }
    orders_in_use<NT>(S, mag);
    return !__syncthreads_or(!fits);
}

// The same from the delayed reads' weights at four nodes (wt [T][WTS]), for blocks that the table does not cover.
template <bool REV, int NTHR>
__device__ __noinline__ bool tdi_stencils_nodes(const FwdParams &P, const FxTab &X, Shared &S, int T, double t_lo, int sg,
                                                   int KW, int mmin, unsigned char *W, double *wt, int *ew_out)
{
    const int tid = threadIdx.x, lane = tid & 31, h = (T - 2) / 2, qn = P.q_terms;
    const int *sm = S.segm[sg];
    const int piece = sm[NTERM];
    __syncthreads();
    for (int i = tid; i < FX_TDI_W / 16; i += blockDim.x)
        reinterpret_cast<uint4 *>(W)[i] = make_uint4(0x80808080u, 0x80808080u, 0x80808080u, 0x80808080u);
    if (tid < NT * 6) {
        const int n = tid / 6, l = tid % 6;
        double x;
        int k;
        const Coef4 *row = row_at(P.to, t_lo + X.tnode_j[n] * P.dt, piece, &x, &k);
        S.lnode[n][l] = cubic(ldg4(row + 9 + l), x) * P.inv_dt;
    }
    if (tid == 64) {
        S.cmax[0] = 0;
        for (int q = 0; q < NT; ++q) S.qor[q] = 0;
    }
    __syncthreads();
    // the node weights take the planes' place; with more than one segment the series is sliced again
    if (tid < NT * NTERM) {
        const int n = tid / NTERM, tm = tid % NTERM, cc = tm / 7, q = tm % 7 + 1;
        if (q <= qn) {
            double D = 0.0;
            for (int k = 1; k <= q; ++k) D += S.lnode[n][c_tdifx.pair[cc >> 1][cc & 1][k]];
            lagrange_to(S, T, -D - (double)sm[tm], wt + tid, WTS);
        }
    }
    __syncthreads();
    // merged stencils: the reads of one (channel, link) added tap by tap
    double b[tap_reps(NTHR)][NT];
    float bm = 0.0f;
#pragma unroll
    for (int rep = 0; rep < tap_reps(NTHR); ++rep) {
        const int i = tid + NTHR * rep;
        {
            double V[NT] = {0.0, 0.0, 0.0, 0.0};
            if (i < 12 * KW) {
                const int cs = i / KW, tap = i - cs * KW, ch = cs >> 2, sl = cs & 3;
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    const int tm = c_slots.term[ch][sl][x], c = tm >> 3, q = tm & 7;
                    if (q > qn) continue;
                    if (q == 0) {
                        if (tap == h - mmin) {
#pragma unroll
                            for (int n = 0; n < NT; ++n) V[n] += c ? -1.0 : 1.0;
                        }
                        continue;
                    }
                    const int id = (ch * 2 + c) * 7 + q - 1, a = tap - (sm[id] - mmin);
                    if (a < 0 || a >= T) continue;
                    const double *w = wt + a * WTS + id;
#pragma unroll
                    for (int n = 0; n < NT; ++n) V[n] += c ? -w[n * NTERM] : w[n * NTERM];
                }
            }
            const double e0 = V[0] + V[3], e1 = V[1] + V[2], o0 = V[0] - V[3], o1 = V[1] - V[2];
#pragma unroll
            for (int q = 0; q < NT; ++q)
                b[rep][q] = (q & 1) ? fma(o0, X.tcheb[q][0], o1 * X.tcheb[q][1]) : fma(e0, X.tcheb[q][0], e1 * X.tcheb[q][1]);
        }
        bm = fmaxf(bm, fabsf((float)b[rep][0]));
    }
    bm = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(bm)));
    if (lane == 0) atomicMax(&S.cmax[0], (int)__float_as_uint(bm));
    __syncthreads();
    const float sm_max = __int_as_float(S.cmax[0]) * 1.01f;
    *ew_out = sm_max > 1e-30f && sm_max < 1e30f ? (int)(__float_as_uint(sm_max) >> 23) - 126 : 0;
    bool fits = sm_max < 1e30f;
    unsigned long long mag[NT] = {};
#pragma unroll
    for (int rep = 0; rep < tap_reps(NTHR); ++rep) {
        const int i = tid + NTHR * rep;
        if (i < 12 * KW) {
            const int cs = i / KW, tap = i - cs * KW;
            unsigned char *w = W + cs * TD * WS + 7 + (REV ? KW - 1 - tap : tap);
            fits &= coef_store<true, 0>(w, b[rep][0], *ew_out, mag);
            fits &= coef_store<true, 1>(w, b[rep][1], *ew_out, mag);
            fits &= coef_store<true, 2>(w, b[rep][2], *ew_out, mag);
            fits &= coef_store<true, 3>(w, b[rep][3], *ew_out, mag);
        }
    }
    orders_in_use<NT>(S, mag);
    return !__syncthreads_or(!fits);
}

// the source of tile g, by one warp: 32 probes a round
__device__ __forceinline__ int64_t find_source(const FwdParams &P, int64_t g)
{
    const int64_t *to = P.src.tile_off;
    int64_t lo = 0, hi = P.src.S;  // to[lo] <= g < to[hi]
    while (hi - lo > 1) {
        const int64_t step = (hi - lo + 31) >> 5, at = lo + step * ((threadIdx.x & 31) + 1);
        const unsigned below = __ballot_sync(0xffffffffu, at < hi && __ldg(to + at) <= g);
        const int64_t n = __popc(below);
        const int64_t nlo = lo + step * n, nhi = nlo + step;
        lo = nlo;
        hi = nhi < hi ? nhi : hi;
    }
    return lo;
}

}  // namespace
}  // namespace lr
