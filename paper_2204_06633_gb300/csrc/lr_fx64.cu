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
//      is accumulated in FP32: products are at most 2^14 and fewer than 2^10 of them meet in the levels
//      below 5, so those sums are exact integers; level 6 carries level 7 (each series digit extended by
//      the next one to 11 bits), which keeps the products left out below 2^-56;
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
// Measured (fused, order 25, one year of 3 153 600 outputs): 44.45 ms sample by sample, 3.65 ms here, with
// 1.3e-13 relative error against 64 bits where the sample form has 1.4e-13.  Two blocks share an SM; the
// tensor pipe is busy a third of the time and the FP64 pipe (weights, transforms) a quarter, the rest is
// latency of the short FP64 phases.  With 8-sample rows in the projection and the TDI stencils computed in
// every block it was 4.36 ms.
//
// Where the expansion does not apply, the block is evaluated sample by sample in FP64 as in lr_fwd64.cu: a
// NaN or infinity in the series, values that span more than 12 bits between 32-sample stretches (the
// fixed point is relative to the block's largest value), coefficients above the digits reserved for their
// order (a source within ~1 degree of an arm direction, an orbit that moves faster), too many segments.
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
constexpr int REPS = (12 * 57 + 255) / 256;  // merged TDI taps per thread: at most 12 stencils of 57 taps
constexpr int RANGE_BITS = 12;
// the last order's coefficient must be below 2^-45 of the stencil's scale: the next one is then below 2^-53
constexpr double LAST_MAX = 1024.0;

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
    int nseg, nlist, fast;
    unsigned brk[NY / 32];
    int list[NTERM * 8 + 8];
    int mmin, mmax;
    int cmax[6], wexp[6];
    unsigned vmax, vmin;
    unsigned long long qor[NN];  // OR of the coefficients' magnitudes per order
    int nq, last;                // orders in use; whether those above 0 have their last digit only
    int bad;
    double red[2 * 8];
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

// largest and smallest non-zero of the 32-sample stretches' maxima (high words)
__device__ __forceinline__ void range_update(Shared &S, unsigned m)
{
    const unsigned w = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0 && w) {
        atomicMax(&S.vmax, w);
        atomicMin(&S.vmin, w);
    }
}

// the exponent e with max < 2^e when the values fit the fixed point; false otherwise
__device__ __forceinline__ bool range_ok(const Shared &S, int *e)
{
    const int eb = (int)(S.vmax >> 20), es = (int)(S.vmin >> 20);
    *e = eb - 1022;
    return eb >= 200 && eb <= 1900 && eb - es <= RANGE_BITS;
}

// v * 2^(55 - e), |v| < 2^e, rounded to an integer: shifts of the significand (FP64 conversions issue at a
// 64th of the integer rate)
__device__ __forceinline__ long long to_fixed(double v, int e)
{
    const long long b = __double_as_longlong(v);
    const int E = (int)((b >> 52) & 0x7ff);
    const unsigned long long m = ((unsigned long long)b & 0xfffffffffffffull) | (E ? 1ull << 52 : 0ull);
    const int s = E - e - 1020;  // at most 2
    unsigned long long r;
    if (s >= 0) r = m << s;
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

template <bool TDI, int Q>
__device__ __forceinline__ bool coef_store(unsigned char *w, double b, unsigned long long *mag)
{
    const long long v = __double2ll_rn(b);
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

// ---------------------------------------------------------------- the block's link series
// Fills ys[6][NY] with the link series of rows 0 .. ny - 1 (sample k_lo + row).
__device__ void project_block(const FwdParams &P, const FxTab &X, Shared &S, int T, int64_t k_lo, int ny, double u0, double *ys,
                              unsigned char *work)
{
    const int tid = threadIdx.x, h = (T - 2) / 2;
    const double fl0 = floor(u0);
    const double t_lo = P.t0 + (double)k_lo * P.dt;
    const TileInfo &ti = S.ti;
    uint16_t *planes = reinterpret_cast<uint16_t *>(work);
    unsigned char *W = work + FX_PROJ_PLANES;
    double *wn = reinterpret_cast<double *>(work + FX_PROJ_PLANES + FX_PROJ_W);

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
                S.mg[g][rd] = (int)(fl - fl0);
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
        S.vmax = 0;
        S.vmin = 0x7fffffffu;
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
        if (look && g * GP < ny) S.list[atomicAdd(&S.nlist, 1)] = i;
    }
    __syncthreads();
    for (int i = tid >> 5; i < S.nlist; i += blockDim.x >> 5) {
        const int g = S.list[i] / 10, rd = S.list[i] % 10, lane = tid & 31;
        const int j = g * GP + lane + 1;   // rows g GP + 1 .. (g + 1) GP against the row before
        int piece;
        const double u = read_pos(P, X, S.skc, u0, t_lo + (double)j * P.dt, rd < 9 ? rd : 0, &piece);
        const int m = rd < 9 ? (int)(floor(u) - fl0) : piece;
        const int prev = __shfl_up_sync(0xffffffffu, m, 1);
        if (m != (lane ? prev : S.mg[g][rd]) && j < NY) atomicOr(&S.brk[j >> 5], 1u << (j & 31));
    }
    __syncthreads();
    if (tid == 0) collect_segments(S, ny);
    __syncthreads();
    const int nseg = S.nseg;
    if (tid < nseg * 10) {
        const int sg = tid / 10, rd = tid % 10;
        int m = S.mg[0][rd];
        if (sg) {
            int piece;
            const double u = read_pos(P, X, S.skc, u0, t_lo + (double)S.segj[sg] * P.dt, rd < 9 ? rd : 0, &piece);
            m = rd < 9 ? (int)(floor(u) - fl0) : piece;
        }
        S.segm[sg][rd] = m;
        if (rd < 9) {
            atomicMin(&S.mmin, m);
            atomicMax(&S.mmax, m);
        }
    }
    __syncthreads();
    const int mmin = S.mmin, KW = S.mmax - mmin + T;   // taps of a merged stencil
    const int nks = (KW + 3 + 15) / 16;
    bool bad = S.bad || nks * 16 > 64;
    // strain window: row j reads samples w_lo + j .. w_lo + j + KW - 1
    const int64_t w_lo = k_lo + (int64_t)fl0 + mmin - h;
    const int WL = ny + KW - 1;
    double vp[3], vc[3];
    if (!bad) {
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const int p = tid + i * 256;
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
            if ((a > b ? a : b) >= 0x7ff00000u) atomicOr(P.err, ERR_NONFINITE);
            range_update(S, a > b ? a : b);
        }
    }
    __syncthreads();
    int ex = 0;
    const unsigned vmax = S.vmax;
    if (!bad && vmax == 0) {  // a block of zeros (or of subnormal high words): the response is zero
        bool any = false;
#pragma unroll
        for (int i = 0; i < 3; ++i) any |= vp[i] != 0.0 || vc[i] != 0.0;
        if (!__syncthreads_or(any)) {
            for (int i = tid; i < 6 * NY; i += blockDim.x) ys[i] = 0.0;
            __syncthreads();
            return;
        }
        bad = true;
    }
    if (!bad) bad = !range_ok(S, &ex);
    if (!bad) {
        for (int i = 0; i < 3; ++i) {
            const int p = tid + i * 256;
            if (p < DL) {
                digits_to_planes(planes, p, vp[i], ex);
                digits_to_planes(planes + 7 * DL, p, vc[i], ex);
            }
        }
    }
    const uint32_t lane = tid & 31, warp = tid >> 5, lr4 = lane >> 2, kp = lane & 3;
    const uint32_t sh = 8 * ((7 - lr4) & 3);
    for (int sg = 0; sg < nseg && !bad; ++sg) {
        const int *sm = S.segm[sg];
        __syncthreads();  // the previous segment's stencils and nodes are free
        for (int i = tid; i < FX_PROJ_W / 16; i += blockDim.x)
            reinterpret_cast<uint4 *>(W)[i] = make_uint4(0x80808080u, 0x80808080u, 0x80808080u, 0x80808080u);
        if (sm[9] != S.segm[sg ? sg - 1 : 0][9] && tid < NN * 3) node_reads(P, X, S, t_lo, u0, tid / 3, tid % 3, sm[9]);
        if (tid >= 192 && tid < 198) S.cmax[tid - 192] = 0;
        if (tid >= 200 && tid < 200 + NN) S.qor[tid - 200] = 0;
        __syncthreads();
        // Lagrange weights at the nodes, two threads per read: prefix products of the lower half and suffix
        // products of the upper half, then each carries on through the other's half
        const int id = tid < WNS ? tid : tid - WNS;
        const bool low = tid < WNS, half = tid < 2 * WNS;
        double e = 0.0, run = 1.0;
        if (half) {
            e = S.nodeu[id] - (fl0 + (double)sm[id % 9]);
            double *w = wn + id;
            if (low) {
                for (int a = 0; a < T / 2; ++a) {
                    w[a * WNS] = run;
                    run *= fma(e, S.lc1[a], S.lc0[a]);
                }
            } else {
                for (int a = T - 1; a >= T / 2; --a) {
                    w[a * WNS] = ((T - 1 - a) & 1) ? -run : run;
                    run *= fma(e, S.rc1[a], S.rc0[a]);
                }
            }
        } else if (tid >= 160 && tid < 160 + NN * 6) {
            const int n = (tid - 160) / 6, l = (tid - 160) % 6, r = c_lr[l], s = c_ls[l];
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
        if (half) {
            double *w = wn + id;
            if (low) {
                for (int a = T / 2; a < T; ++a) {
                    w[a * WNS] *= run;
                    run *= fma(e, S.lc1[a], S.lc0[a]);
                }
            } else {
                for (int a = T / 2 - 1; a >= 0; --a) {
                    w[a * WNS] *= ((T - 1 - a) & 1) ? -run : run;
                    run *= fma(e, S.rc1[a], S.rc0[a]);
                }
            }
        }
        __syncthreads();
        if (tid < 6) {  // the stencil's scale: 2 max|c| with slack for offsets just outside [0, 1)
            const float m = __int_as_float(S.cmax[tid]) * 2.4f;
            S.wexp[tid] = m > 1e-30f && m < 1e30f ? (int)(__float_as_uint(m) >> 23) - 126 : -126;
        }
        __syncthreads();
        if (tid < NN * 12) S.ncf[tid / 12][tid % 12] *= pow2(55 - S.wexp[(tid % 12) >> 1]);
        __syncthreads();
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
                unsigned char *w = W + lp * PD * WS + 7 + tap;
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
                fits &= coef_store<false, 0>(w, b[0], mag);
                fits &= coef_store<false, 1>(w, b[1], mag);
                fits &= coef_store<false, 2>(w, b[2], mag);
                fits &= coef_store<false, 3>(w, b[3], mag);
                fits &= coef_store<false, 4>(w, b[4], mag);
                fits &= coef_store<false, 5>(w, b[5], mag);
                fits &= coef_store<false, 6>(w, b[6], mag);
                fits &= coef_store<false, 7>(w, b[7], mag) && fabs(b[7]) < LAST_MAX;
            }
        orders_in_use<NN>(S, mag);
        if (__syncthreads_or(!fits)) {
            bad = true;
            break;
        }
        count_orders<NN>(S);
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
    const int64_t s_lo = k_lo + (int64_t)fl0 - P.sig_b - P.lproj_b - h - 2;
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
                rp[i] = read_scalar(S, T, hwp, k, u0 - sig[i], s_lo, slen, P.err);
                rc[i] = read_scalar(S, T, hwc, k, u0 - sig[i], s_lo, slen, P.err);
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
                double ep = read_scalar(S, T, hwp, k, uf, s_lo, slen, P.err), ec = read_scalar(S, T, hwc, k, uf, s_lo, slen, P.err);
                y[lf] = (xp * (ep - rp[r]) + xc * (ec - rc[r])) / (2.0 * (1.0 - kn));
                ep = read_scalar(S, T, hwp, k, ub, s_lo, slen, P.err);
                ec = read_scalar(S, T, hwc, k, ub, s_lo, slen, P.err);
                y[lb] = (xp * (ep - rp[s]) + xc * (ec - rc[s])) / (2.0 * (1.0 + kn));
            }
        }
        for (int l = 0; l < 6; ++l) ys[l * NY + j] = y[l];
    }
    __syncthreads();
}

// Chebyshev coefficients of one tap over the block, from the piece's polynomial (degree 5 in its coordinate
// on [-1, 1]) moved to the block's centre xc and scaled by its half width xs
__device__ __forceinline__ void table_coefs(const FwdParams &P, const FxTab &X, int piece, int at, double xc, double xs, double *b)
{
    const double *c = X.tab + (size_t)piece * FX_TAB_Q * 12 * X.tab_kw + at;
    const int st = 12 * X.tab_kw;
    double p[FX_TAB_Q];
#pragma unroll
    for (int q = 0; q < FX_TAB_Q; ++q) p[q] = __ldg(c + q * st);
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
// pieces, or 0 when a piece has no entry.  One thread.
__device__ int table_segments(const FwdParams &P, const FxTab &X, Shared &S, double t_lo, int nb)
{
    double x;
    int a, b;
    row_at(P.to, t_lo, -1, &x, &a);
    const double ua = x + (double)a;
    row_at(P.to, t_lo + (double)(nb - 1) * P.dt, -1, &x, &b);
    if (b > a + 1 || X.meta[2 * a] == 0 || X.meta[2 * b] == 0) return 0;
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
            S.mgt[g][cc * 7 + q - 1] = (int)fl;
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
            const int m = tm < NTERM ? (int)floor(-D) : piece;
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
        const int m = tm < NTERM ? (int)floor(-D) : piece;
        S.segm[sg][tm] = m;
        if (tm < NTERM && tm % 7 < qn) {
            atomicMin(&S.mmin, m);
            atomicMax(&S.mmax, m);
        }
    }
}

// ---------------------------------------------------------------- the block's X, Y, Z
// Link rows ys[6][NY] (ny = nb + HL + HR of them, row = output + HL) to outputs; ys is overwritten.
// Each output is handed to `emit(i, X, Y, Z)` by one thread.
template <class Emit>
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
    const int qn = P.q_terms;

    if (tid < NY / 32) S.brk[tid] = 0;
    if (tid == 32) {
        S.nlist = 0;
        S.bad = 0;
        S.vmax = 0;
        S.vmin = 0x7fffffffu;
        S.mmin = 1 << 29;
        S.mmax = -(1 << 29);
    }
    if (tid == 64) S.fast = X.tab ? table_segments(P, X, S, t_lo, nb) : 0;
    __syncthreads();
    // the first and last link rows are spare: no stencil reaches them
    for (int l = 0; l < 6; ++l)
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int j = tid + 256 * i;
            range_update(S, j >= 1 && j < ny - 1 ? abs_hi(ys[l * NY + j]) : 0u);
        }
    const bool fast = S.fast != 0;
    if (!fast) find_tdi_segments(P, S, t_lo, nb);
    __syncthreads();
    const int nseg = S.nseg;
    bool bad = S.bad;
    int ey = 0;
    const bool zero = S.vmax == 0;
    if (zero) {
        bool any = false;
        for (int i = tid; i < 6 * NY; i += blockDim.x) any |= i % NY < ny && ys[i] != 0.0;
        if (!__syncthreads_or(any)) {
            for (int i = tid; i < nb; i += blockDim.x) emit(i, 0.0, 0.0, 0.0);
            __syncthreads();
            return;
        }
        bad = true;
    }
    if (!bad) bad = !range_ok(S, &ey);
    long long *part = reinterpret_cast<long long *>(ys);  // [2][3][NY], one segment: the planes hold the series
    int done = 0;                                          // outputs kept in ys[0..2][.] by earlier segments
    for (int sg = 0; sg < nseg && !bad; ++sg) {
        const int *sm = S.segm[sg];
        const int piece = sm[NTERM];
        const int mmin = fast ? X.meta[2 * piece + 1] : S.mmin;
        const int KW = fast ? X.meta[2 * piece] : (S.mmax > 0 ? S.mmax : 0) - mmin + T;
        const int nks = (KW + 7 + 15) / 16;
        const int j0 = P.HL + mmin - h;                        // link row of the stencil's first tap for output 0
        if (!fast && (nks * 16 > 64 || j0 < 1 || S.mmax > 0)) {
            bad = true;
            break;
        }
        __syncthreads();
        for (int i = tid; i < FX_TDI_W / 16; i += blockDim.x)
            reinterpret_cast<uint4 *>(W)[i] = make_uint4(0x80808080u, 0x80808080u, 0x80808080u, 0x80808080u);
        if (!fast && tid < NT * 6) {
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
        if (!fast && tid < NT * NTERM) {
            const int n = tid / NTERM, tm = tid % NTERM, cc = tm / 7, q = tm % 7 + 1;
            if (q <= qn) {
                double D = 0.0;
                for (int k = 1; k <= q; ++k) D += S.lnode[n][c_tdifx.pair[cc >> 1][cc & 1][k]];
                lagrange_to(S, T, -D - (double)sm[tm], wt + tid, WTS);
            }
        }
        __syncthreads();
        // merged stencils: the reads of one (channel, link) added tap by tap at the four nodes, or the plan's
        // table around the block's centre
        const double xc = 2.0 * ((t_lo + 0.5 * (NY - 1) * P.dt - P.to.t_first) * P.to.inv_dk - (double)piece) - 1.0;
        const double xs = NY * P.dt * P.to.inv_dk;
        double b[REPS][NT];
        float bm = 0.0f;
#pragma unroll
        for (int rep = 0; rep < REPS; ++rep) {
            const int i = tid + 256 * rep;
            if (i < 12 * KW && fast) {
                table_coefs(P, X, piece, (i / KW) * X.tab_kw + i % KW, xc, xs, b[rep]);
            } else {
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
        const int ew = sm_max > 1e-30f && sm_max < 1e30f ? (int)(__float_as_uint(sm_max) >> 23) - 126 : 0;
        const double ws = pow2(55 - ew);
        bool fits = sm_max < 1e30f;
        unsigned long long mag[NT] = {};
#pragma unroll
        for (int rep = 0; rep < REPS; ++rep) {
            const int i = tid + 256 * rep;
            if (i < 12 * KW) {
                const int cs = i / KW, tap = i - cs * KW;
                unsigned char *w = W + cs * TD * WS + 7 + tap;
                fits &= coef_store<true, 0>(w, b[rep][0] * ws, mag);
                fits &= coef_store<true, 1>(w, b[rep][1] * ws, mag);
                fits &= coef_store<true, 2>(w, b[rep][2] * ws, mag);
                fits &= coef_store<true, 3>(w, b[rep][3] * ws, mag);
            }
        }
        orders_in_use<NT>(S, mag);
        if (__syncthreads_or(!fits)) {
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
                for (int q = 1; q <= qn; ++q) {
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

// ---------------------------------------------------------------- kernel
template <int KIND>
__global__ void __launch_bounds__(256, 2) k_fx64(FwdParams P, FxTab X, int T)
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
                project_block(P, X, S, T, ti.n0, nb, (P.t0 - ti.t0h) / P.dt, ys, work);
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
                    project_block(P, X, S, T, k_lo, ny, (P.t0 - ti.t0h) / P.dt, ys, work);
                }
                double dh = 0.0, hh = 0.0;
                tdi_block(P, X, S, T, ti.n0, nb, ys, work, [&](int i, double vx, double vy, double vz) {
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
// order is below 2^-54).  meta: taps (0: no entry) and the first tap's position.  The stencils depend on the
// orbit alone; from the table a block's expansion is 20 FP64 operations per tap, against ~130 per read and
// node computed in the block.
__global__ void __launch_bounds__(256) k_fx_table(FwdParams P, FxTab X, int T, double *tab, int *meta, int tab_kw)
{
    extern __shared__ double wt[];  // [T][TQ * NTERM + 1]
    constexpr int TQ = FX_TAB_Q, WTT = TQ * NTERM + 1;
    __shared__ double pc[6][4], eps[TQ][NTERM];
    __shared__ double lc1[64], lc0[64], rc1[64], rc0[64];
    __shared__ int mm[NTERM], mmin, mmax, bad;
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
        if (tid == 0) meta[2 * k] = meta[2 * k + 1] = 0;
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
        for (int q = 0; q < TQ; ++q) tab[((size_t)k * TQ + q) * 12 * tab_kw + cs * tab_kw + tap] = m[q];
    }
    ok = !__syncthreads_or(!ok);
    if (tid == 0) {
        meta[2 * k] = ok ? KW : 0;
        meta[2 * k + 1] = mmin;
    }
}

void *kernel_of(int kind)
{
    switch (kind) {
        case KIND_PROJECT: return (void *)k_fx64<KIND_PROJECT>;
        case KIND_TDI: return (void *)k_fx64<KIND_TDI>;
        case KIND_FUSED: return (void *)k_fx64<KIND_FUSED>;
        default: return (void *)k_fx64<KIND_LIKE>;
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
    return NY - P.HL - P.HR;
}

void fx_tables(const FwdParams &P, FxTab &X)
{
    const double pi = 3.14159265358979323846;
    X.icdt = P.inv_dt / C_LIGHT;
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
    const size_t per = sizeof(double) * FX_TAB_Q * 12 * (size_t)kw + 2 * sizeof(int);
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
// launch cannot (the event was recorded outside the capture), there the host waits.
static int table_for(FxPlan *F, cudaStream_t stream, FxTab *X)
{
    *X = F->tab;
    if (!F->ready) return 0;
    const cudaEvent_t ev = (cudaEvent_t)F->ready;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    cudaError_t e = cudaStreamIsCapturing(stream, &cap);
    if (e != cudaSuccess) return (int)e;
    if (cap != cudaStreamCaptureStatusNone) {
        cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;  // event calls are refused in the other modes
        e = cudaThreadExchangeStreamCaptureMode(&mode);
        if (e != cudaSuccess) return (int)e;
        e = cudaEventSynchronize(ev);
        const cudaError_t e2 = cudaThreadExchangeStreamCaptureMode(&mode);
        if (e == cudaSuccess) e = e2;
        return (int)e;
    }
    e = cudaEventQuery(ev);
    if (e == cudaErrorNotReady) {
        cudaGetLastError();
        return (int)cudaStreamWaitEvent(stream, ev);
    }
    if (e != cudaSuccess) return (int)e;
    F->ready = nullptr;
    return (int)cudaEventDestroy(ev);
}

int launch_fx64(int kind, int order, const FwdParams &P, int sms, void *stream)
{
    void *k = kernel_of(kind);
    int T = order + 1;
    const size_t smem = smem_of(T);
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return (int)e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, 256, smem);
    if (e != cudaSuccess) return (int)e;
    if (per_sm < 1) return (int)cudaErrorLaunchOutOfResources;
    int64_t grid = (int64_t)per_sm * sms;
    if (P.total_tiles >= 0 && P.total_tiles < grid) grid = P.total_tiles;
    if (grid < 1) grid = 1;
    FxTab X;
    if (const int te = table_for(P.fx, (cudaStream_t)stream, &X)) return te;
    void *args[] = {(void *)&P, (void *)&X, (void *)&T};
    return (int)cudaLaunchKernel(k, dim3((unsigned)grid), dim3(256), args, smem, (cudaStream_t)stream);
}

}  // namespace lr
