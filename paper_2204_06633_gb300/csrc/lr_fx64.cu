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
// one the stencil shifted by b, W[c - b]; neither is expanded in memory.  A lane's four k-values are taken
// as four consecutive c (the same permutation of k on both sides), so a lane reads its two left registers
// of a row with one 8-byte load and its right registers from four consecutive digit bytes, which become
// halves by placing them under the exponent of 1024 and subtracting 1152.
//
// Measured (fused, order 25, one year of 3 153 600 outputs): 44.45 ms sample by sample, 4.36 ms here, with
// 1.3e-13 relative error against 64 bits where the sample form has 1.4e-13.
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
constexpr int GP = 16;            // spacing of the projection's grid samples
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
            double npos[NN][9], neps[NN * 9], ncf[NN][12];
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
    int nseg, nlist;
    unsigned brk[NY / 32];
    int list[NTERM * 8 + 8];
    int mmin, mmax;
    int cmax[6], wexp[6];
    unsigned vmax, vmin;
    unsigned qmask;
    int bad;
    double red[2 * 8];
};

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint2 lds64(uint32_t a)
{
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a));
    return v;
}
__device__ __forceinline__ uint32_t lds32(uint32_t a)
{
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ void mma_f16(float *c, const uint32_t *a, uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
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
template <int QF, int NQ, bool TDI>
__device__ __forceinline__ void contract(float (&acc)[NQ][7][4], uint32_t a_lane, uint32_t w_lane, uint32_t sh, int nks,
                                         const signed char *links)
{
    constexpr int ZM = zq(TDI, QF);      // the smallest z of the group
    constexpr int NA = ZM ? 8 - ZM : 7;  // digit planes of the series that it needs
    constexpr int PARTS = TDI ? 4 : 2, ROWS = TDI ? TD : PD;
#pragma unroll
    for (int i = 0; i < NQ; ++i)
#pragma unroll
        for (int L = 0; L < 7; ++L)
#pragma unroll
            for (int r = 0; r < 4; ++r) acc[i][L][r] = 0.0f;
#pragma unroll 1
    for (int part = 0; part < PARTS; ++part) {
        uint32_t pa = a_lane + (uint32_t)((TDI ? links[part] : part) * 7 * DL * 2);
        uint32_t pw = w_lane + (uint32_t)(part * ROWS * WS);
#pragma unroll 1
        for (int ks = 0; ks < nks; ++ks, pa += 32, pw += 16) {
            uint32_t a[NA][4];
#pragma unroll
            for (int k = 0; k < NA; ++k) {
                const uint2 lo = lds64(pa + k * DL * 2), hi = lds64(pa + k * DL * 2 + 128);
                a[k][0] = lo.x; a[k][1] = hi.x; a[k][2] = lo.y; a[k][3] = hi.y;
            }
#pragma unroll
            for (int i = 0; i < NQ; ++i) {
                const int z = zq(TDI, QF + i), row = digit_row(TDI, QF + i);
#pragma unroll
                for (int d = z; d < 7; ++d) {
                    const uint32_t w0 = lds32(pw + (row + d - z) * WS), w1 = lds32(pw + (row + d - z) * WS + 4);
                    const uint32_t u = __funnelshift_r(w0, w1, sh);
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
__device__ __forceinline__ double sigma_at(const FwdParams &P, const SkyConst &S, const Coef4 *row, double x, int s,
                                           double *pos)
{
    double v[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) v[d] = cubic(ldg4(row + 3 * s + d), x);
    if (pos) {
#pragma unroll
        for (int d = 0; d < 3; ++d) pos[3 * s + d] = v[d];
    }
    return (S.k[0] * v[0] + S.k[1] * v[1] + S.k[2] * v[2]) * P.fx.icdt;
}

// position (samples, relative to the row) of read rd (0-2 receptions, 3 + l emissions) at time t
__device__ __forceinline__ double read_pos(const FwdParams &P, const SkyConst &S, double u0, double t, int rd, int *piece)
{
    double x;
    const Coef4 *row = row_at(P.po, t, -1, &x, piece);
    const int s = rd < 3 ? rd : c_ls[rd - 3];
    const double sig = sigma_at(P, S, row, x, s, nullptr);
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

// seven digit planes (halves) of v * scale at index p
__device__ __forceinline__ void digits_to_planes(uint16_t *pl, int p, double v, double scale)
{
    const long long X = __double2ll_rn(v * scale) + DIGIT_BIAS;
    const uint32_t top = (uint32_t)((int)(X >> 48) + 128);  // 0 .. 256
    const uint32_t lo = (uint32_t)X, hi = (uint32_t)(X >> 32);
    const uint32_t d[7] = {top, (hi >> 8) & 255u, hi & 255u, lo >> 24, (lo >> 16) & 255u, (lo >> 8) & 255u, lo & 255u};
#pragma unroll
    for (int i = 0; i < 7; i += 1) {
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
__device__ __forceinline__ bool coef_store(unsigned char *w, double b, unsigned &mask)
{
    const long long v = __double2ll_rn(b);
    if (v) mask |= 1u << Q;
    return coef_digits<zq(TDI, Q)>(w + digit_row(TDI, Q) * WS, v);
}

// ---------------------------------------------------------------- the block's link series
// Fills ys[6][NY] with the link series of rows 0 .. ny - 1 (sample k_lo + row).
__device__ void project_block(const FwdParams &P, Shared &S, int T, int64_t k_lo, int ny, double u0, double *ys,
                              unsigned char *work)
{
    const int tid = threadIdx.x, h = (T - 2) / 2;
    const double fl0 = floor(u0);
    const double t_lo = P.t0 + (double)k_lo * P.dt;
    const TileInfo &ti = S.ti;
    uint16_t *planes = reinterpret_cast<uint16_t *>(work);
    unsigned char *W = work + FX_PROJ_PLANES;
    double *wn = reinterpret_cast<double *>(work + FX_PROJ_PLANES + FX_PROJ_W);

    // stencil positions on the grid samples
    if (tid < NG * 3) {
        const int g = tid / 3, s = tid % 3;
        const double t = t_lo + (double)(g * GP) * P.dt;
        double x;
        int piece;
        const Coef4 *row = row_at(P.po, t, -1, &x, &piece);
        const double sig = sigma_at(P, S.skc, row, x, s, nullptr);
        if (s == 0) S.mg[g][9] = piece;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const int rd = i == 0 ? s : 3 + c_by_emitter[s][i - 1];
            const double u = i == 0 ? u0 - sig : u0 - cubic(ldg4(row + 9 + rd - 3), x) * P.inv_dt - sig;
            const double fl = floor(u);
            S.mg[g][rd] = (int)(fl - fl0);
            S.fg[g][rd] = (float)(u - fl);
        }
    }
    if (tid < NY / 32) S.brk[tid] = 0;
    if (tid == 32) {
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
        const int j = g * GP + (lane < GP ? lane : GP);
        int piece;
        const double u = read_pos(P, S.skc, u0, t_lo + (double)j * P.dt, rd < 9 ? rd : 0, &piece);
        const int m = rd < 9 ? (int)(floor(u) - fl0) : piece;
        const int prev = __shfl_up_sync(0xffffffffu, m, 1);
        if (lane >= 1 && lane <= GP && m != prev && j < NY) atomicOr(&S.brk[j >> 5], 1u << (j & 31));
    }
    __syncthreads();
    if (tid == 0) collect_segments(S, ny);
    __syncthreads();
    const int nseg = S.nseg;
    if (tid < nseg * 10) {
        const int sg = tid / 10, rd = tid % 10;
        int piece;
        const double u = read_pos(P, S.skc, u0, t_lo + (double)S.segj[sg] * P.dt, rd < 9 ? rd : 0, &piece);
        const int m = rd < 9 ? (int)(floor(u) - fl0) : piece;
        S.segm[sg][rd] = m;
        if (rd < 9) {
            atomicMin(&S.mmin, m);
            atomicMax(&S.mmax, m);
        }
    }
    __syncthreads();
    const int mmin = S.mmin, KW = S.mmax - mmin + T;   // taps of a merged stencil
    const int nks = (KW + 7 + 15) / 16;
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
        const double scale = pow2(55 - ex);
        for (int i = 0; i < 3; ++i) {
            const int p = tid + i * 256;
            if (p < DL) {
                digits_to_planes(planes, p, vp[i], scale);
                digits_to_planes(planes + 7 * DL, p, vc[i], scale);
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
        if (tid < NN * 3) {
            const int n = tid / 3, s = tid % 3;
            const double t = t_lo + P.fx.node_j[n] * P.dt;
            double x;
            int piece;
            const Coef4 *row = row_at(P.po, t, sm[9], &x, &piece);
            const double sig = sigma_at(P, S.skc, row, x, s, S.npos[n]);
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const int rd = i == 0 ? s : 3 + c_by_emitter[s][i - 1];
                const double u = i == 0 ? u0 - sig : u0 - cubic(ldg4(row + 9 + rd - 3), x) * P.inv_dt - sig;
                S.neps[n * 9 + rd] = u - (fl0 + (double)sm[rd]);
            }
        }
        if (tid >= 64 && tid < 70) S.cmax[tid - 64] = 0;
        if (tid == 70) S.qmask = 0;
        __syncthreads();
        if (tid < NN * 9) {
            lagrange_to(S, T, S.neps[tid], wn + tid, WNS);
        } else if (tid >= 96 && tid < 96 + NN * 3) {
            const int n = (tid - 96) / 3, r = (tid - 96) % 3, s = (r + 1) % 3;
            const SkyConst &K = S.skc;
            const double *x = S.npos[n];
            double d0 = x[3 * r] - x[3 * s], d1 = x[3 * r + 1] - x[3 * s + 1], d2 = x[3 * r + 2] - x[3 * s + 2];
            const double inv = 1.0 / sqrt(d0 * d0 + d1 * d1 + d2 * d2);
            d0 *= inv; d1 *= inv; d2 *= inv;
            const double un = K.u[0] * d0 + K.u[1] * d1 + K.u[2] * d2;
            const double vn = K.v[0] * d0 + K.v[1] * d1 + K.v[2] * d2;
            const double kn = K.k[0] * d0 + K.k[1] * d1 + K.k[2] * d2;
            const double xip = un * un - vn * vn, xic = 2.0 * un * vn;
            const double xp = K.c2p * xip + K.s2p * xic, xc = -K.s2p * xip + K.c2p * xic;
            const double gf = 1.0 / (2.0 * (1.0 - kn)), gr = 1.0 / (2.0 * (1.0 + kn));
            const double c4[4] = {xp * gf, xc * gf, xp * gr, xc * gr};
            double *o = S.ncf[n];
            o[2 * r] = c4[0];
            o[2 * r + 1] = c4[1];
            o[2 * (5 - r)] = c4[2];
            o[2 * (5 - r) + 1] = c4[3];
            // NaN and infinity give the largest keys
            atomicMax(&S.cmax[r], (int)(__float_as_uint((float)fmax(fabs(c4[0]), fabs(c4[1]))) & 0x7fffffffu));
            atomicMax(&S.cmax[5 - r], (int)(__float_as_uint((float)fmax(fabs(c4[2]), fabs(c4[3]))) & 0x7fffffffu));
            if (!(isfinite(gf) && isfinite(gr))) S.bad = 1;
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
        unsigned mask = 0;
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
                    for (int n = 0; n < NN / 2; ++n) v = fma((q & 1) ? o[n] : e[n], P.fx.cheb[q][n], v);
                    b[q] = v;
                }
                fits &= coef_store<false, 0>(w, b[0], mask);
                fits &= coef_store<false, 1>(w, b[1], mask);
                fits &= coef_store<false, 2>(w, b[2], mask);
                fits &= coef_store<false, 3>(w, b[3], mask);
                fits &= coef_store<false, 4>(w, b[4], mask);
                fits &= coef_store<false, 5>(w, b[5], mask);
                fits &= coef_store<false, 6>(w, b[6], mask);
                fits &= coef_store<false, 7>(w, b[7], mask) && fabs(b[7]) < LAST_MAX;
            }
        mask = __reduce_or_sync(0xffffffffu, mask);
        if (lane == 0 && mask) atomicOr(&S.qmask, mask);
        if (__syncthreads_or(!fits)) {
            bad = true;
            break;
        }
        const unsigned qm = S.qmask;
        const int js = S.segj[sg], je = S.segj[sg + 1];
        const int mb0 = js >> 7, nmb = ((je - 1) >> 7) - mb0 + 1;
        for (int it = warp; it < nmb * 6; it += blockDim.x >> 5) {
            const int l = it % 6, mb = mb0 + it / 6;
            const uint32_t a_lane = smem_u32(planes) + 16u * (16u * mb + lr4) + 8u * kp;
            const uint32_t w_lane = smem_u32(W) + (uint32_t)(2 * l * PD * WS) + 4u * (kp + ((7u - lr4) >> 2));
            int kappa[4], jr[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                jr[r] = 128 * mb + 8 * (int)(lr4 + (r >> 1) * 8) + 2 * (int)kp + (r & 1);
                kappa[r] = 2 * jr[r] + 1 - NY;
            }
            long long b1[4] = {0, 0, 0, 0}, b2[4] = {0, 0, 0, 0};
            if (qm & 0xf0u) {
                float acc[4][7][4];
                contract<4, 4, false>(acc, a_lane, w_lane, sh, nks, nullptr);
                clenshaw<4, 4, false>(acc, kappa, b1, b2);
            }
            if (qm & 0xfcu) {
                float acc[2][7][4];
                contract<2, 2, false>(acc, a_lane, w_lane, sh, nks, nullptr);
                clenshaw<2, 2, false>(acc, kappa, b1, b2);
            }
            if (qm & 0xfeu) {
                float acc[1][7][4];
                contract<1, 1, false>(acc, a_lane, w_lane, sh, nks, nullptr);
                clenshaw<1, 1, false>(acc, kappa, b1, b2);
            }
            float acc[1][7][4];
            contract<0, 1, false>(acc, a_lane, w_lane, sh, nks, nullptr);
            const double unit = pow2(ex + S.wexp[l] - 57);
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const long long v = levels<0>(acc[0], r) + mul_nu<9>(b1[r], kappa[r]) - b2[r];
                const int64_t k = k_lo + jr[r];
                if (jr[r] >= js && jr[r] < je) ys[l * NY + jr[r]] = k >= 0 && k < ti.N ? (double)v * unit : 0.0;
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

// ---------------------------------------------------------------- the block's X, Y, Z
// Link rows ys[6][NY] (ny = nb + HL + HR of them, row = output + HL) to outputs; ys is overwritten.
// Each output is handed to `emit(i, X, Y, Z)` by one thread.
template <class Emit>
__device__ void tdi_block(const FwdParams &P, Shared &S, int T, int64_t n0, int nb, double *ys, unsigned char *work,
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
    if (tid >= 64 && tid < 64 + NGT * 6) {
        const int g = (tid - 64) / 6, l = (tid - 64) % 6;
        double x;
        int piece;
        const Coef4 *row = row_at(P.to, t_lo + (double)(g * GT) * P.dt, -1, &x, &piece);
        S.lg[g][l] = cubic(ldg4(row + 9 + l), x) * P.inv_dt;
        if (l == 0) S.mgt[g][NTERM] = piece;
    }
    __syncthreads();
    // the first and last link rows are spare: no stencil reaches them
    for (int l = 0; l < 6; ++l)
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int j = tid + 256 * i;
            range_update(S, j >= 1 && j < ny - 1 ? abs_hi(ys[l * NY + j]) : 0u);
        }
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
    __syncthreads();
    const int mmin = S.mmin, mmax = S.mmax > 0 ? S.mmax : 0;  // the undelayed read sits at 0
    const int KW = mmax - mmin + T, nks = (KW + 7 + 15) / 16;
    const int j0 = P.HL + mmin - h;                            // link row of the stencil's first tap for output 0
    bool bad = S.bad || nks * 16 > 64 || j0 < 1 || mmax > 0;
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
        __syncthreads();
        for (int i = tid; i < FX_TDI_W / 16; i += blockDim.x)
            reinterpret_cast<uint4 *>(W)[i] = make_uint4(0x80808080u, 0x80808080u, 0x80808080u, 0x80808080u);
        if (tid < NT * 6) {
            const int n = tid / 6, l = tid % 6;
            double x;
            int piece;
            const Coef4 *row = row_at(P.to, t_lo + P.fx.tnode_j[n] * P.dt, sm[NTERM], &x, &piece);
            S.lnode[n][l] = cubic(ldg4(row + 9 + l), x) * P.inv_dt;
        }
        if (tid == 64) {
            S.qmask = 0;
            S.cmax[0] = 0;
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
        // merged stencils: the reads of one (channel, link) added tap by tap at the four nodes
        double b[REPS][NT];
        float bm = 0.0f;
#pragma unroll
        for (int rep = 0; rep < REPS; ++rep) {
            const int i = tid + 256 * rep;
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
                b[rep][q] = (q & 1) ? fma(o0, P.fx.tcheb[q][0], o1 * P.fx.tcheb[q][1]) : fma(e0, P.fx.tcheb[q][0], e1 * P.fx.tcheb[q][1]);
            bm = fmaxf(bm, fabsf((float)b[rep][0]));
        }
        bm = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(bm)));
        if (lane == 0) atomicMax(&S.cmax[0], (int)__float_as_uint(bm));
        __syncthreads();
        const float sm_max = __int_as_float(S.cmax[0]) * 1.01f;
        const int ew = sm_max > 1e-30f && sm_max < 1e30f ? (int)(__float_as_uint(sm_max) >> 23) - 126 : 0;
        const double ws = pow2(55 - ew);
        bool fits = sm_max < 1e30f;
        unsigned mask = 0;
#pragma unroll
        for (int rep = 0; rep < REPS; ++rep) {
            const int i = tid + 256 * rep;
            if (i < 12 * KW) {
                const int cs = i / KW, tap = i - cs * KW;
                unsigned char *w = W + cs * TD * WS + 7 + tap;
                fits &= coef_store<true, 0>(w, b[rep][0] * ws, mask);
                fits &= coef_store<true, 1>(w, b[rep][1] * ws, mask);
                fits &= coef_store<true, 2>(w, b[rep][2] * ws, mask);
                fits &= coef_store<true, 3>(w, b[rep][3] * ws, mask);
            }
        }
        mask = __reduce_or_sync(0xffffffffu, mask);
        if (lane == 0 && mask) atomicOr(&S.qmask, mask);
        if (__syncthreads_or(!fits)) {
            bad = true;
            break;
        }
        const int js = S.segj[sg], je = S.segj[sg + 1];
        const double scale = pow2(55 - ey);
        // link rows that only earlier outputs read are left out: their place holds those outputs now
        for (int i = tid; i < 6 * DL; i += blockDim.x) {
            const int l = i / DL, p = i - l * DL, j = p + j0;
            digits_to_planes(planes + l * 7 * DL, p, p >= js && j < ny - 1 ? ys[l * NY + j] : 0.0, scale);
        }
        __syncthreads();
        const unsigned qm = S.qmask;
        const int mb0 = js >> 7, nmb = ((je - 1) >> 7) - mb0 + 1;
        const double unit = pow2(ey + ew - 57);
        const uint32_t sh = 8 * ((7 - lr4) & 3);
        const bool hi = (qm & 14u) != 0;
        const int per = nmb * 3;
        if (nseg == 1) {
            // order 0 and the higher orders are separate items (28 and 34 digit products)
            for (int it = warp; it < (hi ? 2 : 1) * per; it += blockDim.x >> 5) {
                const int half = it / per, ch = it % per % 3, mb = mb0 + it % per / 3;
                const uint32_t a_lane = smem_u32(planes) + 16u * (16u * mb + lr4) + 8u * kp;
                const uint32_t w_lane = smem_u32(W) + (uint32_t)(4 * ch * TD * WS) + 4u * (kp + ((7u - lr4) >> 2));
                if (half == 0) {
                    float acc[1][7][4];
                    contract<0, 1, true>(acc, a_lane, w_lane, sh, nks, c_slots.link[ch]);
#pragma unroll
                    for (int r = 0; r < 4; ++r)
                        part[ch * NY + 128 * mb + 8 * (lr4 + (r >> 1) * 8) + 2 * kp + (r & 1)] = levels<0>(acc[0], r);
                } else {
                    float acc[3][7][4];
                    contract<1, 3, true>(acc, a_lane, w_lane, sh, nks, c_slots.link[ch]);
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
                for (int c = 0; c < 3; ++c) o[c] = (double)(part[c * NY + i] + (hi ? part[(3 + c) * NY + i] : 0)) * unit;
                emit(i, o[0], o[1], o[2]);
            }
            done = nb;
        } else {
            // a block with a step: one item per channel; the outputs are kept in ys[0..2], in rows that the
            // later segments do not read (their first link row is past output je)
            for (int it = warp; it < per; it += blockDim.x >> 5) {
                const int ch = it % 3, mb = mb0 + it / 3;
                const uint32_t a_lane = smem_u32(planes) + 16u * (16u * mb + lr4) + 8u * kp;
                const uint32_t w_lane = smem_u32(W) + (uint32_t)(4 * ch * TD * WS) + 4u * (kp + ((7u - lr4) >> 2));
                int kappa[4];
                long long b1[4] = {0, 0, 0, 0}, b2[4] = {0, 0, 0, 0};
#pragma unroll
                for (int r = 0; r < 4; ++r) kappa[r] = 2 * (128 * mb + 8 * (int)(lr4 + (r >> 1) * 8) + 2 * (int)kp + (r & 1)) + 1 - NY;
                if (hi) {
                    float acc[3][7][4];
                    contract<1, 3, true>(acc, a_lane, w_lane, sh, nks, c_slots.link[ch]);
                    clenshaw<1, 3, true>(acc, kappa, b1, b2);
                }
                float acc[1][7][4];
                contract<0, 1, true>(acc, a_lane, w_lane, sh, nks, c_slots.link[ch]);
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const int i = (kappa[r] + NY - 1) >> 1;
                    if (i >= js && i < je) ys[ch * NY + i] = (double)(levels<0>(acc[0], r) + mul_nu<9>(b1[r], kappa[r]) - b2[r]) * unit;
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

// ---------------------------------------------------------------- kernel
template <int KIND>
__global__ void __launch_bounds__(256, 2) k_fx64(FwdParams P, int T)
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
        if (tid == 0) {
            S.ti = tile_info(P, g, KIND == KIND_PROJECT ? 6 : 3);
            if (KIND != KIND_TDI) S.skc = make_sky(S.ti.sky);
            if (!S.ti.ok) atomicOr(P.err, ERR_OFFSETS);
            if (like && !(S.ti.ok && S.ti.nb > 0)) like_store(P, g, 0.0, 0.0);
        }
        __syncthreads();
        if (S.ti.ok && S.ti.nb > 0) {
            const TileInfo &ti = S.ti;
            const int nb = (int)ti.nb;
            if (KIND == KIND_PROJECT) {
                project_block(P, S, T, ti.n0, nb, (P.t0 - ti.t0h) / P.dt, ys, work);
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
                    project_block(P, S, T, k_lo, ny, (P.t0 - ti.t0h) / P.dt, ys, work);
                }
                double dh = 0.0, hh = 0.0;
                tdi_block(P, S, T, ti.n0, nb, ys, work, [&](int i, double X, double Y, double Z) {
                    const int64_t n = ti.n0 + i;
                    if (ti.out) {
                        ti.out[n] = X;
                        ti.out[ti.N + n] = Y;
                        ti.out[2 * ti.N + n] = Z;
                    }
                    if (like && ti.dat) {
                        const double da = __ldg(ti.dat + n), de = __ldg(ti.dat + ti.N + n), dT = __ldg(ti.dat + 2 * ti.N + n);
                        if (!(isfinite(da) && isfinite(de) && isfinite(dT))) atomicOr(P.err, ERR_NONFINITE);
                        like_terms(P.like, X, Y, Z, da, de, dT, dh, hh);
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
    if (7 + T + chain + 1 > 64 || 7 + T + 2 * P.lproj_b + 2 > 64) return 0;
    if (NY + 2 * P.sig_b + P.lproj_b + T + 4 > FX_PROJ_PLANES / 16) return 0;
    return NY - P.HL - P.HR;
}

void fx_tables(FwdParams &P)
{
    const double pi = 3.14159265358979323846;
    P.fx.icdt = P.inv_dt / C_LIGHT;
    for (int n = 0; n < NN; ++n) P.fx.node_j[n] = 0.5 * (NY * (1.0 + cos(pi * (2 * n + 1) / (2 * NN))) - 1.0);
    for (int q = 0; q < NN; ++q)
        for (int n = 0; n < NN / 2; ++n)
            P.fx.cheb[q][n] = (q ? 2.0 : 1.0) / NN * cos(pi * ((q * (2 * n + 1)) % (4 * NN)) / (2 * NN));
    for (int n = 0; n < NT; ++n) P.fx.tnode_j[n] = 0.5 * (NY * (1.0 + cos(pi * (2 * n + 1) / (2 * NT))) - 1.0);
    for (int q = 0; q < NT; ++q)
        for (int n = 0; n < NT / 2; ++n)
            P.fx.tcheb[q][n] = (q ? 2.0 : 1.0) / NT * cos(pi * ((q * (2 * n + 1)) % (4 * NT)) / (2 * NT));
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
    void *args[] = {(void *)&P, (void *)&T};
    return (int)cudaLaunchKernel(k, dim3((unsigned)grid), dim3(256), args, smem, (cudaStream_t)stream);
}

}  // namespace lr
