// mp_fp64_tc.cu -- three of the float64 path's four contractions on the tensor cores, by exact
// integer slices.
//
// GB300 does about 0.6 T float64 operations a second, 1/1700 of its 16-bit tensor rate, so
// contractions of GenASiS II Sec. 2.2 (the azimuthal factor of Eq. (AngularMomentsDiscrete) and both
// of Eq. (Solution)) run here as sums of exact 16-bit products: every float64 operand row
// is scaled by a power of two of its own to a 55-bit fixed-point magnitude, cut into seven
// 8-bit balanced digits (integers of magnitude <= 128, exact in float16), and the products
// of digit pairs are added by tcgen05 MMAs.  (Slicing operands so that the low-precision
// products add without error is the scheme of Ozaki, Ogita, Oishi and Rump, Numer.
// Algorithms 59 (2012) 95.)  Digit pairs (a, b) with the same a + b share a weight
// 2^-8(a+b) and one float32 accumulator; a chain of K <= 146 terms stays below
// 7 * 146 * 2^14 < 2^24, so every partial sum is an integer that float32 holds exactly and
// the tensor core's truncating addition never truncates.  Pairs with a + b >= 7 are left
// out: they weigh at most 2^-56 of (row maximum x column maximum) each.  The seven
// accumulators are put together as a 64-bit integer and leave as float64 by integer
// instructions (ldexp, on the float64 pipe, for results outside the normal range).
//
// Accuracy.  The operands are fixed-point: a value 2^k below its row's (or table column's) maximum
// keeps 55 - k bits.  A result of K terms is off by at most K 2^-51 x (row maximum) x (column
// maximum), and since roundings and left-out digits have either sign by about sqrt(K) 2^-55 of it (K
// 2^-56 where all small cells of a row are equal), whether or not the two maxima meet at one index.
// A float64 sum is off by a multiple of 2^-53 of the sum of its terms' magnitudes.  The steps below can afford that: the
// azimuthal tables are of one size along a row of cells (a factor of two in their widths is let in)
// and themselves off by the rounding of m phi, 2^-53 m phi of their maximum; and the synthesis delivers Phi alone, whose sum over the
// orders is of the size of the row maxima (errors stay at 2^-53 of the largest |Phi| of the
// shell; G of an order m near the poles, a small part of it there, is less accurate by itself).
// The theta part of the moments cannot (sin^m theta against a clump near the pole): it is summed
// in float64, k64_theta_rows in mp_fp64.cu.
//
// Two kernels.  A is always the data (split on the fly), B a table (split once per mesh),
// D = A B^T:
//   k64_contract_tc  long K, few columns (K streamed):
//       (a1) F[i][p][j] = sum_k rho[i][j][k] Iph[p][k]      rows (i, j), K = n_phi
//   k64_expand_tc    short K, many columns (A kept, columns streamed):
//       (d1) G[i][p][j] = sum_l C[q][i] Ith[t][j] / dmu_j    rows (i, cos | sin) of one order m,
//                                                            columns j, K = L + 1 - m
//       (d2) Phi[i][j][k] = sum_p G[i][p][j] Iph[p][k]/dphi_k  rows (i, j), columns k, K = 2 L (the
//            column m = 0 of the table is 1: G[i][0][j] joins the sums as an integer)
// The seven digit matrices of B are stacked along N: digit a of A times the first 7 - a
// digits of B is one MMA of N = (7 - a) Nt columns whose result lands Nt a columns to the
// right, so a K step of 16 takes seven MMAs for its 28 products and reads A seven times
// instead of 28 (with one MMA per pair the shared-memory reads of A would bound it).
//
// What bounds them: not the tensor core (33 % of the time in the long contraction, 49 % in the
// long expansion at 1024 x 256 x 512 cells, l_max = 32) nor HBM (22 and 34 %), but the integer
// instructions that split and rejoin the operands (half the rate of float32's: their pipe is 53 and
// 58 % busy) and the hand-offs between the warps that issue them.  Measured there against float64
// on CUDA cores: (a1) 29.5 ms -> 691 us, (d1) 2143 -> 66 us, (d2) 13.9 ms -> 427 us; at 512 x 128 x
// 256, l_max = 16: 1918 -> 91, 200 -> 16, 891 -> 69 us.  (Rounding the operands instead of
// truncating them is 38 and 3 us of (a1).)
#include <algorithm>
#include <cmath>

#include <cuda_fp16.h>

#include "mp_fp64_join.h"
#include "mp_internal.h"
#include "ptx.cuh"

namespace mp {

namespace {

constexpr int kDig = 7;              // digits per operand
constexpr int kChunkSteps = 8;       // contract: K steps (of 16) that share a row exponent and a chain
constexpr int kDrainAt = 2;          // contract: steps of an item split before the one before it is drained
constexpr int kExpandKMax = 146;     // expand: longest chain (7 * 146 * 2^14 < 2^24)
constexpr int kWorkWarps = 16;
constexpr int kThreadsX = (kWorkWarps + 4) * 32;  // expand: two MMA issuers, a table producer for each
// contract: a fifth warpgroup (three MMA issuers, the table producer) gives registers to the four
// that split: 640 x 96 = 512 x 112 + 128 x 32
constexpr int kIssuersC = 3;
constexpr int kThreadsC = (kWorkWarps + kIssuersC + 1) * 32;
constexpr int kRegsWork = 112, kRegsRest = 32;
constexpr int kExpNan = 2047;        // row exponent of a row with an infinity or a NaN
constexpr int kNtX = 32;             // expand: columns per block
constexpr int kRowsX = kDig * kNtX;  // expand: stacked table rows of a block
constexpr int kKeepX = 2;             // expand: octets of k a thread keeps between its two looks at them
constexpr int kBoxX = 32 * 64;       // expand: a warp's output box, 32 rows of 8 float64

// A slot of one K step: [digit][octet of k][128 rows][8 k]
constexpr int kLboA1 = 128 * 16;
constexpr int kDigA1 = 2 * kLboA1;
constexpr int kSlotA1 = kDig * kDigA1;
constexpr int kLboA2 = 128 * 16;
constexpr int kDigA2 = 2 * kLboA2;
constexpr int kStepA2 = kDig * kDigA2;

__host__ __device__ inline int ceil16(int x) { return (x + 15) & ~15; }

// Contract: the columns of a set (a pass over the density), 64 at
// most, in halves of up to 32, each padded to a multiple of 16 (accumulator blocks start on such
// columns) and stacked by itself: 7 * 32 of the half's 256 columns of tensor memory.  A
// projection of P = 2 L + 1 columns with L a multiple of 8 would pay a block of 16 for its one
// column m = 0 seven times over and, at l_max = 32, no longer fit one pass; its column m = 0 takes
// one block of 16 behind the first half instead, with the seven weights as its columns: for
// digit a of A the table rows of that block are the column's digits a places further down.
constexpr int kHalf = 32;
constexpr int kNtMax = 64;
constexpr int kEtLd = kNtMax + 4;   // column exponents of a set (the own block's at kNtMax)
constexpr int kRows0 = kDig * 16;   // table rows of the column m = 0: [digit of A][16]

// Padded columns of half h of a set of N columns.
__host__ __device__ inline int half_cols(int N, int h)
{
    const int n = N - h * kHalf;
    return n <= 0 ? 0 : ceil16(n < kHalf ? n : kHalf);
}

// ---------------------------------------------------------------------------- digits
// |x| as a 55-bit integer relative to the row exponent (x = +- V 2^(E - 1077), V <= 2^55, rounded
// to nearest: truncation takes up to one unit off every cell of a ring in the same direction), with
// 0x80 added to its six low bytes: byte b of the sum less 128 is then a balanced digit, and the
// seventh byte the leading one (0 .. 128).  e8 = E + 8.  The integer is formed with one bit more, so
// that its rounding rides on the addition and costs the two shifts behind it.
__device__ __forceinline__ void fix55(uint32_t lo, uint32_t hi, int e8, uint32_t &wl, uint32_t &wh)
{
    const int n = e8 - (int)((hi >> 20) & 0x7FFu);
    const uint32_t th = __funnelshift_l(lo, hi, 11) | 0x80000000u, tl = lo << 11;
    uint32_t vl = __funnelshift_rc(tl, th, n), vh;
    asm("shr.u32 %0, %1, %2;" : "=r"(vh) : "r"(th), "r"(n));
    const int n2 = max(n - 32, 0);
    asm("shr.u32 %0, %1, %2;" : "=r"(vl) : "r"(vl), "r"(n2));
    asm("add.cc.u32 %0, %2, 0x01010101;\n\taddc.u32 %1, %3, 0x00010101;" : "=r"(wl), "=r"(wh) : "r"(vl), "r"(vh));
    wl = __funnelshift_r(wl, wh, 1);
    wh >>= 1;
}

// The digits of two neighbouring values as float16 pairs, d[0] the leading one: byte b becomes
// the float16 1024 + b (bits 0x6400 | b), and one packed multiply-add takes 1024 + 128 off and
// applies the sign.
__device__ __forceinline__ void digits2(uint32_t wl0, uint32_t wh0, uint32_t hi0, uint32_t wl1, uint32_t wh1,
                                        uint32_t hi1, uint32_t (&d)[kDig])
{
    const uint32_t sg = __byte_perm(hi0, hi1, 0x7632);
    const uint32_t one = (sg & 0x80008000u) | 0x3C003C00u;         // +-1
    const uint32_t off = (sg & 0x80008000u) ^ 0xE480E480u;         // -+1152
    const uint32_t off_top = (sg & 0x80008000u) ^ 0xE400E400u;     // -+1024
    const uint32_t k64 = 0x64646464u;
    const uint32_t g01 = __byte_perm(wl0, wl1, 0x5140), g23 = __byte_perm(wl0, wl1, 0x7362);
    const uint32_t g45 = __byte_perm(wh0, wh1, 0x5140), g6 = __byte_perm(wh0, wh1, 0x7362);
    const uint32_t h[kDig] = {__byte_perm(g6, k64, 0x4140),  __byte_perm(g45, k64, 0x4342),
                              __byte_perm(g45, k64, 0x4140), __byte_perm(g23, k64, 0x4342),
                              __byte_perm(g23, k64, 0x4140), __byte_perm(g01, k64, 0x4342),
                              __byte_perm(g01, k64, 0x4140)};
#pragma unroll
    for (int i = 0; i < kDig; ++i)
        asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(d[i]) : "r"(h[i]), "r"(one), "r"(i == 0 ? off_top : off));
}

__device__ __forceinline__ uint32_t abs_hi(double x) { return (uint32_t)__double2hiint(x) & 0x7FFFFFFFu; }

// Rows next to the bottom of the float64 range (denormals among them): their values times
// 2^300, which is exact, and the exponent of the largest.  Out of line: inlined, the multiplies
// were predicated instead of branched around and kept the float64 pipe 29 % busy.
template <int N>
__device__ __noinline__ void scale_up_n(double *x)
{
#pragma unroll
    for (int e = 0; e < N; ++e) x[e] *= 0x1p300;
}
template <int N>
__device__ __forceinline__ void scale_up(double (&x)[N])
{
    double y[N];
#pragma unroll
    for (int e = 0; e < N; ++e) y[e] = x[e];
    scale_up_n<N>(y);
#pragma unroll
    for (int e = 0; e < N; ++e) x[e] = y[e];
}
__device__ __noinline__ int scaled_up_exponent(uint32_t max_hi)
{
    return (int)(abs_hi(__hiloint2double((int)max_hi, -1) * 0x1p300) >> 20);
}

// hi:lo 2^e2 (a signed 64-bit integer below 2^62 in magnitude) as float64 by integer
// instructions, rounded to nearest; sets `odd` when the result is outside the normal range
// (the caller then takes ldexp).
__device__ __forceinline__ double scaled_i64(uint32_t lo, uint32_t hi, int e2, bool &odd)
{
    const uint32_t sg = (uint32_t)((int)hi >> 31);
    uint32_t ul, uh, l, h;
    asm("sub.cc.u32 %0, %2, %4;\n\tsubc.u32 %1, %3, %4;" : "=r"(ul), "=r"(uh) : "r"(lo ^ sg), "r"(hi ^ sg), "r"(sg));
    // leading one to bit 62: shift left by n, in two steps past 32
    const uint32_t top = uh ? uh : ul;
    const int n = (uh ? -1 : 31) + __clz((int)top);
    const int n2 = max(n - 32, 0);
    asm("shl.b32 %0, %1, %2;" : "=r"(h) : "r"(__funnelshift_lc(ul, uh, n)), "r"(n2));
    asm("shl.b32 %0, %1, %2;" : "=r"(l) : "r"(ul), "r"(n));
    asm("add.cc.u32 %0, %0, 0x200;\n\taddc.u32 %1, %1, 0;" : "+r"(l), "+r"(h));
    const int be = 1023 + 62 - 1 + e2 - n;             // exponent field less one: the leading one adds it
    odd |= (unsigned)be > 2044u && top != 0;
    const uint32_t rl = __funnelshift_r(l, h, 10);
    const uint32_t rh = (h >> 10) + (top ? (uint32_t)be << 20 : 0u);
    return __hiloint2double((int)(rh | (hi & 0x80000000u)), (int)rl);
}

// The same through ldexp, for results outside the normal range; NaN for a row that holds one.
__device__ __noinline__ double scaled_i64_slow(uint32_t lo, uint32_t hi, int e2, int row_exponent)
{
    if (row_exponent >= kExpNan) return __longlong_as_double(0x7FF8000000000000ll);
    return ldexp((double)(long long)(((unsigned long long)hi << 32) | lo), e2);
}

// An integer held in a float32: below 2^22 in magnitude by one addition (the integer appears
// in the low mantissa bits of 1.5 2^23 + x), otherwise by a conversion (a quarter of the rate).
template <bool SMALL>
__device__ __forceinline__ int acc_int(float x)
{
    return SMALL ? __float_as_int(x + 12582912.0f) - 0x4B400000 : __float2int_rn(x);
}

// The seven accumulators of one result as a 64-bit integer in units of 2^(56 + DS) (of 2^110 =
// the product of the operands' scales): the two lightest are added in float32 (a rounding of
// 2^-(54 - DS) of the row and column maxima at most), the others exactly.  NM: how many of the
// leading ones are below 2^22.
template <int NM, int DS>
__device__ __forceinline__ void acc_sum(const float (&t)[kDig], uint32_t &lo, uint32_t &hi)
{
    constexpr float w5 = 1.0f / (1 << DS), w6 = w5 / 256.0f;
    const float t56 = fmaf(t[6], w6, DS ? t[5] * w5 : t[5]);
    const int a0 = acc_int<(NM > 0)>(t[0]), a1 = acc_int<(NM > 1)>(t[1]), a2 = acc_int<(NM > 2)>(t[2]);
    const int a3 = acc_int<(NM > 3)>(t[3]), a4 = acc_int<(NM > 4)>(t[4]);
    // (a chain of 128 terms: 6 pairs, 6 * 128 * 2^14 2^-DS < 2^22 from DS = 2 on)
    const int a5 = acc_int<(NM > 5 || DS >= 2)>(t56);
    const long long l = (long long)(a2 * 256 + a3) * (65536 >> DS) +
                        (NM > 4 ? (long long)(a4 * (256 >> DS) + a5) : (long long)a4 * (256 >> DS) + a5);
    if (DS == 0) {
        lo = (uint32_t)l;
        hi = (uint32_t)(l >> 32) + (uint32_t)(a0 * 256 + a1);
    } else {
        const long long v = l + (long long)(a0 * 256 + a1) * (long long)((1ull << 32) >> DS);
        lo = (uint32_t)v;
        hi = (uint32_t)(v >> 32);
    }
}

// The sum for chains short enough that all but the lightest accumulators, or all of them
// (NM >= 5), stay below 2^22: the integers keep the offset 0x4B400000 of their float bits
// through the multiplies (no pair overflows 32 unsigned bits) and one 64-bit constant takes
// all of them off, so that the sum needs two integer-pipe instructions (the rest is on the FMA
// pipe; integer logic runs at half its rate and bounds the kernel).
__device__ __forceinline__ void acc_sum_small(const float (&t)[kDig], uint32_t &lo, uint32_t &hi)
{
    uint32_t a[6];
#pragma unroll
    for (int i = 0; i < 5; ++i) a[i] = (uint32_t)__float_as_int(t[i] + 12582912.0f);
    a[5] = (uint32_t)__float_as_int(fmaf(t[6], 0.00390625f, t[5]) + 12582912.0f);
    constexpr uint32_t kPair = 0x4B400000u * 257u;  // modulo 2^32
    constexpr unsigned long long kOff =
        (unsigned long long)kPair * 65536u + kPair + ((unsigned long long)kPair << 32);
    const unsigned long long v = (unsigned long long)(a[2] * 256u + a[3]) * 65536u + (a[4] * 256u + a[5]) +
                                 ((unsigned long long)(a[0] * 256u + a[1]) << 32) - kOff;
    lo = (uint32_t)v;
    hi = (uint32_t)(v >> 32);
}

// One chain of several (DS >= 2) whose first three accumulators stay below 2^22 (the next two may
// not, and are converted): the integers keep their offsets as in acc_sum_small, ChainJoin's in all.
template <int DS>
__device__ __forceinline__ unsigned long long acc_sum_chain(const float (&t)[kDig])
{
    constexpr float w5 = 1.0f / (1 << DS), w6 = w5 / 256.0f;
    uint32_t a[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) a[i] = (uint32_t)__float_as_int(t[i] + 12582912.0f);
    const uint32_t a5 = (uint32_t)__float_as_int(fmaf(t[6], w6, t[5] * w5) + 12582912.0f);
    // (the offset of a3 is exact: the sum is an integer up to 2^24)
    const uint32_t a3 = (uint32_t)__float2int_rn(t[3] + 8388608.0f), a4 = (uint32_t)__float2int_rn(t[4]);
    return ChainJoin<DS>::sum(a[0], a[1], a[2], a3, a4, a5);
}

// Eight results of one row at once: hi:lo 2^(e0 + et) as in scaled_i64, for integers of 33 bits or
// more (the common case); false when one is smaller.
template <int N>
__device__ __forceinline__ bool scaled_row(const uint32_t (&lo)[N], const uint32_t (&hi)[N], const int (&be0)[N],
                                           double (&out)[N])
{
    uint32_t least = 0xFFFFFFFFu;
#pragma unroll
    for (int e = 0; e < N; ++e) {
        const uint32_t sg = (uint32_t)((int)hi[e] >> 31);
        uint32_t ul, uh, h, l;
        asm("sub.cc.u32 %0, %2, %4;\n\tsubc.u32 %1, %3, %4;" : "=r"(ul), "=r"(uh) : "r"(lo[e] ^ sg), "r"(hi[e] ^ sg), "r"(sg));
        least = min(least, uh);
        const int n = __clz((int)uh) - 1;  // leading one to bit 62
        h = __funnelshift_l(ul, uh, n);
        l = ul << (n & 31);
        asm("add.cc.u32 %0, %0, 0x200;\n\taddc.u32 %1, %1, 0;" : "+r"(l), "+r"(h));
        const uint32_t rh = (h >> 10) + ((uint32_t)(be0[e] - n) << 20);
        out[e] = __hiloint2double((int)(rh | (hi[e] & 0x80000000u)), (int)__funnelshift_r(l, h, 10));
    }
    return least != 0;
}

// x 2^-n (n <= 62), rounded to nearest.
__device__ __forceinline__ long long shift_round(long long x, int n) { return (x + ((1ll << n) >> 1)) >> n; }

// ---------------------------------------------------------------------------- tables
enum { TAB_PROJECT = 0, TAB_EXPAND_TH = 1, TAB_EXPAND_PH = 2 };

struct TabParams {
    const double *Ith, *Iph, *Iphc, *dmu;
    uint8_t *tab;
    const unsigned long long *off;  // byte offset per set (pass, or order m)
    int *et;                        // column exponents, [set][et_ld]
    int kind, n_t, n_p, L, P, pass_cols, m0, et_ld;
    int *bound;  // largest sum an accumulator can reach: expand, the sixth; contract, the third
};

// First column of a projection pass; m0: the column m = 0 rides on pass 0 in a block of its own.
__host__ __device__ inline int pass_col0(int s, int pass_cols, int m0) { return s * pass_cols + m0; }
__host__ __device__ inline int pass_ncols(int s, int pass_cols, int m0, int P)
{
    const int n = P - pass_col0(s, pass_cols, m0);
    return n < pass_cols ? n : pass_cols;
}

__device__ __forceinline__ double tab_value(const TabParams &t, int set, int n, int k)
{
    switch (t.kind) {
    case TAB_PROJECT:  // n = -1: the column m = 0 in its own block
        return t.Iph[(size_t)(n < 0 ? 0 : pass_col0(set, t.pass_cols, t.m0) + n) * t.n_p + k];
    case TAB_EXPAND_TH: return t.Ith[(size_t)tri(set + k, set) * t.n_t + n] / t.dmu[n];
    default: return t.Iphc[(size_t)(k + 1) * t.n_p + n];  // m >= 1: the column m = 0 is 1 everywhere
    }
}

// One warp per table column n of one set: its exponent, then its digits.  The contract table is
// [K step]{per half [octet][7 Nt rows][8], row = digit Nt + n; for a column m = 0 of its own
// then [digit of A][octet][16 rows][8]}; expand tables are blocks of 32
// columns, [block][K step][octet][7 x 32][8].  Cells past K are never written (the tables
// start as zeros).
__global__ void __launch_bounds__(128) k64_digit_tables(const TabParams t)
{
    const int set = blockIdx.y, lane = threadIdx.x & 31;
    const bool own0 = t.kind == TAB_PROJECT && t.m0 && set == 0;
    const int n = blockIdx.x * 4 + (threadIdx.x >> 5) - (own0 ? 1 : 0);
    int N, K;
    switch (t.kind) {
    case TAB_PROJECT: N = pass_ncols(set, t.pass_cols, t.m0, t.P), K = t.n_p; break;
    case TAB_EXPAND_TH: N = t.n_t, K = t.L + 1 - set; break;
    default: N = t.n_p, K = t.P - 1; break;
    }
    if (n >= N) return;
    uint32_t mx = 0;
    for (int k = lane; k < K; k += 32) mx = max(mx, abs_hi(tab_value(t, set, n, k)));
    mx = __reduce_max_sync(0xFFFFFFFFu, mx);
    // (phi expansion: every column at the scale of the m = 0 column, which is 1 and not in the table)
    const int E = t.kind == TAB_EXPAND_PH ? 1023 : (int)(mx >> 20);
    if (lane == 0) t.et[(size_t)set * t.et_ld + (n < 0 ? kNtMax : n)] = E;
    if (E == 0) return;  // zeros
    const bool stacked = t.kind == TAB_PROJECT;
    const int hf = stacked && n >= kHalf, h0 = half_cols(N, 0), h1 = half_cols(N, 1);
    const int nd = !stacked ? kNtX : hf ? h1 : h0, rows = kDig * nd;
    const int main_rows = stacked ? kDig * (h0 + h1) : rows;
    const size_t step = (size_t)(main_rows + (own0 ? kRows0 : 0)) * 32;
    const int steps = max(1, (K + 15) / 16);
    uint8_t *base = t.tab + t.off[set] + (stacked ? 0 : (size_t)(n / kNtX) * steps * step);
    const int nr = stacked ? n - hf * kHalf : n % kNtX;
    if (hf) base += (size_t)kDig * h0 * 32;
    int s5 = 0, s6 = 0, s3 = 0, s3max = 0;
    for (int k0 = 0; k0 < K; k0 += 32) {
        const int k = k0 + lane;
        if (k < K) {
            const double x = tab_value(t, set, n, k);
            const uint32_t hi = (uint32_t)__double2hiint(x);
            uint32_t wl, wh, d[kDig];
            fix55((uint32_t)__double2loint(x), hi, E + 8, wl, wh);
            if ((hi & 0x7FF00000u) == 0) wl = 0x80808080u, wh = 0x00008080u;  // zeros stay zeros
            digits2(wl, wh, hi, wl, wh, hi, d);
#pragma unroll
            for (int i = 0; i < kDig; ++i) {
                const int v = abs(__half2int_rn(__ushort_as_half((unsigned short)(d[i] & 0xFFFFu))));
                (i < 6 ? s5 : s6) += v;
                if (i < 3) s3 += v;
            }
            uint8_t *dst = base + (size_t)(k >> 4) * step + (k & 7) * 2;
            const int oct = (k >> 3) & 1;
            if (n >= 0) {
#pragma unroll
                for (int i = 0; i < kDig; ++i)
                    *reinterpret_cast<uint16_t *>(dst + (size_t)(oct * rows + i * nd + nr) * 16) =
                        (uint16_t)(d[i] & 0xFFFFu);
            } else {
#pragma unroll
                for (int a = 0; a < kDig; ++a)
#pragma unroll
                    for (int i = 0; i + a < kDig; ++i)
                        *reinterpret_cast<uint16_t *>(dst + (size_t)main_rows * 32 +
                                                      (size_t)(a * 32 + oct * 16 + a + i) * 16) =
                            (uint16_t)(d[i] & 0xFFFFu);
            }
        }
        if ((k0 + 32) % (16 * kChunkSteps) == 0 || k0 + 32 >= K) {  // the end of one of A's chains
            s3max = max(s3max, __reduce_add_sync(0xFFFFFFFFu, s3));
            s3 = 0;
        }
    }
    // digits of A are at most 128
    if (!stacked) {
        // the sixth accumulator takes pairs with the first six digits of B, the seventh joins it
        // divided by 256
        s5 = __reduce_add_sync(0xFFFFFFFFu, s5);
        s6 = __reduce_add_sync(0xFFFFFFFFu, s6);
        if (lane == 0) atomicMax(t.bound, 128 * s5 + (s5 + s6) / 2 + 2);
    } else if (lane == 0) {
        atomicMax(t.bound, 128 * s3max);
    }
}

// ---------------------------------------------------------------------------- contract
struct ContractParams {
    const double *src;
    double *dst;
    const uint8_t *tab;
    const unsigned long long *off;
    const int *et;
    int *err;
    long long R;
    int n_t, n_p, P, ldJ;
    int n_steps, n_chunks, ds;  // ds: low bits of a chain's 62-bit sum dropped, so that n_chunks of them fit
                                   // (the template's DS, or where that is negative at run time)
    int n_units, npass, pass_cols, m0;
    int ns_a, ns_b, nacc, slot_b, cols_max;
};

struct ContractUnit {
    int set, col0;         // pass and its first column
    int N, Nt[2], own0;    // columns, those of its halves padded; the column m = 0 in a block of its own
    long long row0;
    __device__ __forceinline__ uint32_t step_bytes() const
    {
        return (uint32_t)(kDig * (Nt[0] + Nt[1]) + (own0 ? kRows0 : 0)) * 32;
    }
};

__device__ __forceinline__ ContractUnit contract_unit(const ContractParams &p, int u)
{
    ContractUnit r;
    const int tile = u / p.npass;
    r.set = u - tile * p.npass;
    r.row0 = (long long)tile * 128;
    r.col0 = pass_col0(r.set, p.pass_cols, p.m0);
    r.N = pass_ncols(r.set, p.pass_cols, p.m0, p.P);
    r.own0 = p.m0 && r.set == 0;
    r.Nt[0] = half_cols(r.N, 0);
    r.Nt[1] = half_cols(r.N, 1);
    return r;
}

// Start of row `r` of a unit in the source (n_phi contiguous values), or nullptr past the last row.
__device__ __forceinline__ const double *contract_row(const ContractParams &p, const ContractUnit &u, int r)
{
    const long long row = u.row0 + r;
    return row < p.R ? p.src + row * p.n_p : nullptr;
}

// Roles: warps 0-15 split A (each thread four neighbouring k of one row per K step, the whole
// chunk of 128 k in registers: its row maxima come from a shuffle over the row's four threads,
// and a step's registers take the next chunk's loads as soon as it is split, so 128 KB are in
// flight a CTA) and drain the accumulators between their steps; warp 16 owns tensor memory;
// warps 16-18 issue the MMAs, warp 19 copies the table.  (The parameters stay in constant memory:
// copied to registers, as the compiler does with up to 128 bytes of them, they cost 20 bytes of
// spills and 89 -> 118 us at 512 x 128 x 256 cells, l_max = 16.)
template <bool VEC, int DS, int NM>
__global__ void __launch_bounds__(kThreadsC, 1) k64_contract_tc(const __grid_constant__ ContractParams prm)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127));
    uint8_t *sA = smem;
    uint8_t *sB = sA + (size_t)prm.ns_a * kSlotA1;
    long long *sAcc = reinterpret_cast<long long *>(sB + (size_t)prm.ns_b * prm.slot_b);  // [columns][128], several chunks
    int *sE = reinterpret_cast<int *>(sAcc + (prm.n_chunks > 1 ? (size_t)prm.cols_max * 128 : 0));  // [4][128]
    uint64_t *bars = reinterpret_cast<uint64_t *>(sE + 4 * 128);
    uint64_t *a_full = bars, *a_empty = a_full + prm.ns_a, *b_full = a_empty + prm.ns_a, *b_empty = b_full + prm.ns_b;
    uint64_t *acc_full = b_empty + prm.ns_b, *acc_empty = acc_full + 2, *e_full = acc_empty + 2, *drain_bar = e_full + 4;
    uint32_t *tmem_holder = reinterpret_cast<uint32_t *>(drain_bar + 1);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_holder + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < prm.ns_a; ++s) {
            mbar_init(smem_u32(&a_full[s]), kWorkWarps);
            mbar_init(smem_u32(&a_empty[s]), kIssuersC);
        }
        for (int s = 0; s < prm.ns_b; ++s) {
            mbar_init(smem_u32(&b_full[s]), 1);
            mbar_init(smem_u32(&b_empty[s]), kIssuersC);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&acc_full[b]), kIssuersC);
            mbar_init(smem_u32(&acc_empty[b]), kWorkWarps);
        }
        for (int b = 0; b < 4; ++b) mbar_init(smem_u32(&e_full[b]), kWorkWarps);
        mbar_init(smem_u32(drain_bar), kIssuersC);
        *abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == kWorkWarps) {
        tmem_alloc(smem_u32(tmem_holder), 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_holder;
    const uint32_t acc_stride = prm.nacc == 2 ? 256 : 0;
    pdl_wait();  // the source comes from the previous kernels
    const long long budget = wait_budget(prm.err);

    if (warp >= kWorkWarps) {
        setmaxnreg_dec<kRegsRest>();
        if (warp == kWorkWarps + kIssuersC) {
            // ---------------- table producer
            if (lane == 0) {
                Ring rb;
                int issued = 0;
                bool ok = true;
                for (int u = blockIdx.x; u < prm.n_units && ok; u += gridDim.x) {
                    const ContractUnit un = contract_unit(prm, u);
                    const uint8_t *src = prm.tab + prm.off[un.set];
                    const uint32_t bytes = un.step_bytes();
                    for (int s = 0; s < prm.n_steps; ++s, rb.next(prm.ns_b)) {
                        ok = mbar_wait(smem_u32(&b_empty[rb.idx]), rb.phase ^ 1, abort_flag, prm.err, budget);
                        if (!ok) break;
                        const uint32_t bar = smem_u32(&b_full[rb.idx]);
                        mbar_arrive_expect_tx(bar, bytes);
                        bulk_load(smem_u32(sB + (size_t)rb.idx * prm.slot_b), src + (size_t)s * bytes, bytes, bar);
                        ++issued;
                    }
                }
                drain_ring(b_full, rb, prm.ns_b, issued);
            }
        } else {
            // ---------------- MMA issuers (the whole warp waits, one lane issues): one for each half of
            // the columns and one for the column m = 0 of its own block; each commits every step,
            // with or without MMAs.  One warp alone issuing all of a step's MMAs took 2000 cycles
            // for 1200 cycles of tensor time.
            const uint32_t leader = elect_one();
            const int mine = warp - kWorkWarps;
            const uint64_t ad0 = sdesc_noswizzle(smem_u32(sA), kLboA1, 128);
            const uint32_t a_lo0 = (uint32_t)ad0, a_hi = (uint32_t)(ad0 >> 32);
            Ring ra, rb;
            int it = 0;
            bool ok = true;
            for (int u = blockIdx.x; u < prm.n_units && ok; u += gridDim.x) {
                const ContractUnit un = contract_unit(prm, u);
                const int n = mine < 2 ? un.Nt[mine] : 0;          // this issuer's columns
                const bool own = mine == 2 && un.own0;
                // its table rows and accumulators
                const uint32_t b_off = mine == 0 ? 0u : (uint32_t)(kDig * (un.Nt[0] + (own ? un.Nt[1] : 0))) * 32;
                const uint64_t bd0 = sdesc_noswizzle(smem_u32(sB) + b_off, own ? 256u : (uint32_t)n * kDig * 16, 128);
                const uint32_t b_lo0 = (uint32_t)bd0, b_hi = (uint32_t)(bd0 >> 32);
                const uint32_t d_off = mine == 1 ? 256u : own ? (uint32_t)(kDig * un.Nt[0]) : 0u;
                for (int c = 0; c < prm.n_chunks && ok; ++c, ++it) {
                    const int b = prm.nacc == 2 ? it & 1 : 0, nth = prm.nacc == 2 ? it >> 1 : it;
                    ok = warp_all(mbar_wait(smem_u32(&acc_empty[b]), (nth & 1) ^ 1, abort_flag, prm.err, budget));
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t d0 = tmem_base + (uint32_t)b * acc_stride + d_off;
                    const int steps = min(kChunkSteps, prm.n_steps - c * kChunkSteps);
                    for (int s = 0; s < steps; ++s, ra.next(prm.ns_a), rb.next(prm.ns_b)) {
                        ok = warp_all(mbar_wait(smem_u32(&b_full[rb.idx]), rb.phase, abort_flag, prm.err, budget) &&
                                      mbar_wait(smem_u32(&a_full[ra.idx]), ra.phase, abort_flag, prm.err, budget));
                        if (!ok) break;
                        const uint32_t a_lo = a_lo0 + (uint32_t)ra.idx * (kSlotA1 / 16);
                        const uint32_t b_lo = b_lo0 + (uint32_t)(rb.idx * (prm.slot_b / 16));
                        if (n == kHalf) {
#pragma unroll
                            for (int i = 0; i < kDig; ++i)
                                umma_warp(d0 + (uint32_t)(i * kHalf), a_lo + i * (kDigA1 / 16), a_hi, b_lo, b_hi,
                                              idesc_f16_f32(128, (kDig - i) * kHalf), (s | i) != 0, leader);
                        } else if (n == 16) {
#pragma unroll
                            for (int i = 0; i < kDig; ++i)
                                umma_warp(d0 + (uint32_t)(i * 16), a_lo + i * (kDigA1 / 16), a_hi, b_lo, b_hi,
                                              idesc_f16_f32(128, (kDig - i) * 16), (s | i) != 0, leader);
                        } else if (own) {
#pragma unroll
                            for (int i = 0; i < kDig; ++i)
                                umma_warp(d0, a_lo + i * (kDigA1 / 16), a_hi, b_lo + i * 32, b_hi,
                                              idesc_f16_f32(128, 16), (s | i) != 0, leader);
                        }
                        umma_commit_warp(smem_u32(&a_empty[ra.idx]), leader);
                        umma_commit_warp(smem_u32(&b_empty[rb.idx]), leader);
                    }
                    if (ok) umma_commit_warp(smem_u32(&acc_full[b]), leader);
                }
            }
            umma_commit_warp(smem_u32(drain_bar), leader);
            const long long t0 = clock64();
            while (!mbar_try_wait(smem_u32(drain_bar), 0) && clock64() - t0 < MP_WAIT_BUDGET_CYCLES) {
            }
            __syncwarp();
        }
    } else {
        // ---------------- split + drain
        setmaxnreg_inc<kRegsWork>();
        // split: row, k = 16 step + 4 quad + 0..3; the quads of a row sit in lanes l, l ^ 1, l ^ 16,
        // so that a half warp's 8-byte stores are 128 consecutive bytes (8 rows of one octet)
        const int crow = 8 * warp + ((lane >> 1) & 7), quad = (lane & 1) | ((lane >> 4) << 1);
        const int q4 = warp & 3, grp = warp >> 2;                  // drain: lane quarter, column group
        const uint32_t a_off = (uint32_t)((quad >> 1) * kLboA1 + crow * 16 + (quad & 1) * 8);
        double v[kChunkSteps][4];
        bool ok = true, bad = false;

        // K step s of a chunk: `p` at the thread's first k of the chunk, `lim` terms left from it
        // (none or fewer past the last row)
        bool whole = false;  // a whole chunk of a whole warp's rows: no bounds to look at
        auto load_step = [&](const double *p, int lim, int s, double (&x)[4]) {
            if (VEC && whole) {
                ldg_f64x4(p + 16 * s, x);
            } else if (VEC) {  // (lim is a multiple of four)
#pragma unroll
                for (int e = 0; e < 4; ++e) x[e] = 0.0;
                if (lim > 16 * s) ldg_f64x4(p + 16 * s, x);
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e) x[e] = lim > 16 * s + e ? __ldg(p + 16 * s + e) : 0.0;
            }
        };
        // the thread's place in the first chunk of unit u
        auto unit_at = [&](int u, const double *&p, int &lim) {
            p = u < prm.n_units ? contract_row(prm, contract_unit(prm, u), crow) : nullptr;
            lim = p ? prm.n_p - 4 * quad : 0;
            p += 4 * quad;
        };

        Ring ra;
        int it = 0, Er = 0;  // Er: running exponent of this thread's drain row
        int u = blockIdx.x, c = 0, pu = -1, pc = 0;  // this item, the one before (not yet drained)
        const double *src;
        int lim;
        unit_at(u, src, lim);
#pragma unroll
        for (int s = 0; s < kChunkSteps; ++s) load_step(src, lim, s, v[s]);
        while (ok && (u < prm.n_units || pu >= 0)) {
            const int steps = u < prm.n_units ? min(kChunkSteps, prm.n_steps - c * kChunkSteps) : 0;
            const int u2 = c + 1 == prm.n_chunks ? u + (int)gridDim.x : u, c2 = c + 1 == prm.n_chunks ? 0 : c + 1;
            uint32_t mx = 0;
#pragma unroll
            for (int s = 0; s < kChunkSteps; ++s)
#pragma unroll
                for (int e = 0; e < 4; ++e) mx = max(mx, abs_hi(v[s][e]));
            mx = max(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, 1));
            mx = max(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, 16));
            int E = (int)(mx >> 20);
            const bool tiny = E < 128;
            bad |= E >= kExpNan;
            // next to the bottom of the float64 range (denormals among it): scaled up exactly
            if (tiny) E = max(128, scaled_up_exponent(mx));
            // four exponent buffers: a warp splits at most two items ahead of another one's drain
            if (quad == 0 && steps) sE[(it & 3) * 128 + crow] = tiny ? E - 300 : E;
            __syncwarp();
            if (lane == 0 && steps) mbar_arrive(smem_u32(&e_full[it & 3]));
            const int e8 = E + 8;
            if (c2) {
                src += 16 * kChunkSteps;
                lim -= 16 * kChunkSteps;
            } else {
                unit_at(u2, src, lim);
            }
            whole = VEC && warp_all(lim > 16 * (kChunkSteps - 1) + 3);
            // the last step's loads of the next item are needed as soon as they are issued: they
            // come from L2 then, where this has brought the item by that time
            if (lim > 0) {
                const double *pf = src + 28 * quad;
                if (lim > 28 * quad) prefetch_l2(pf);
                if (lim > 28 * quad + 16) prefetch_l2(pf + 16);
            }
#pragma unroll
            for (int s = 0; s < kChunkSteps; ++s) {
                if (s == kDrainAt) {
                    // ---- the accumulators of the item before this one into the row's running
                    // sums, after its last chunk to memory (two steps of this item are split by
                    // now, so the MMAs have work as soon as the accumulators are free)
                    if (pu >= 0 && ok) {
                        const ContractUnit un = contract_unit(prm, pu);
                        const int b = prm.nacc == 2 ? (it - 1) & 1 : 0, nth = prm.nacc == 2 ? (it - 1) >> 1 : it - 1;
                        ok = warp_all(mbar_wait(smem_u32(&e_full[(it - 1) & 3]), ((it - 1) >> 2) & 1, abort_flag, prm.err, budget) &&
                                      mbar_wait(smem_u32(&acc_full[b]), nth & 1, abort_flag, prm.err, budget));
                        if (!ok) break;
                        tc_fence_after();
                        const int row = 32 * q4 + lane;
                        const bool last = pc == prm.n_chunks - 1;
                        const int Ec = sE[((it - 1) & 3) * 128 + row];
                        // running sums are kept at the largest exponent of the row's chunks so far
                        const int dsr = DS < 0 ? prm.ds : 0;  // run-time part of the dropped bits
                        int sh_old = 0, sh_new = dsr;
                        if (pc == 0) {
                            Er = Ec;
                        } else {
                            const int En = max(Er, Ec);
                            sh_old = min(62, En - Er);
                            sh_new = min(62, En - Ec + dsr);
                            Er = En;
                        }
                        const bool shifts = DS != 0 && !warp_all((sh_old | sh_new) == 0);
                        double *dst = nullptr;  // column n of the unit: dst + n ldJ
                        const long long r = un.row0 + row;
                        if (last && r < prm.R) {
                            const int i = (int)((unsigned)r / (unsigned)prm.n_t), j = (int)r - i * prm.n_t;
                            dst = prm.dst + ((size_t)i * prm.P + un.col0) * prm.ldJ + j;
                        }
                        const uint32_t col = tmem_base + (uint32_t)b * acc_stride + ((uint32_t)(q4 * 32) << 16);
                        const int e_base = 56 + (DS < 0 ? prm.ds : DS) + Er - 2154;
                        // one result: its seven accumulators into the running sum at `pa` or, after
                        // the last chunk, to `out`
                        auto result = [&](const float (&a)[kDig], long long *pa, int et, double *out, bool in) {
                            uint32_t lo, hi;
                            if (DS != 0) {
                                long long x, o = 0;
                                if (pc > 0) {
                                    o = *pa;
                                    if (shifts) o = shift_round(o, sh_old);
                                }
                                if (DS > 0 && NM >= 3) {
                                    x = (long long)acc_sum_chain<(DS > 0 ? DS : 2)>(a);
                                    if (shifts)
                                        x = shift_round(x - (long long)ChainJoin<(DS > 0 ? DS : 2)>::offset, sh_new) + o;
                                    else
                                        x = x + o - (long long)ChainJoin<(DS > 0 ? DS : 2)>::offset;
                                } else {
                                    acc_sum<NM, (DS > 0 ? DS : 0)>(a, lo, hi);
                                    x = (long long)(((unsigned long long)hi << 32) | lo);
                                    if (shifts) x = shift_round(x, sh_new);
                                    x += o;
                                }
                                if (!last) {
                                    *pa = x;
                                    return;
                                }
                                lo = (uint32_t)x;
                                hi = (uint32_t)(x >> 32);
                            } else {
                                acc_sum<NM, 0>(a, lo, hi);
                            }
                            bool odd = Er >= kExpNan;
                            double x = scaled_i64(lo, hi, e_base + et, odd);
                            if (odd) x = scaled_i64_slow(lo, hi, e_base + et, Er);
                            if (in) *out = x;
                        };
                        const int *et = prm.et + (size_t)un.set * kEtLd;
                        // groups of four columns, dealt to the four warps of a lane quarter (the
                        // padding up to Nt holds zeros); the column m = 0 of its own block, with its
                        // weights side by side, goes to the last of them
                        const int n_first = 4 * grp;
                        if (DS > 0 && NM >= 3 && !last && !shifts) {
                            // the usual chain before the last, rows whose exponents agree: read all
                            // seven sums and the integer so far at once, no result to look at
                            for (int n = n_first; n < un.N; n += 16) {
                                uint32_t t[kDig][4];
                                const int hf = n >> 5, nt = un.Nt[hf];
                                const uint32_t c0 = col + (uint32_t)(hf * 256 + (n & 31));
#pragma unroll
                                for (int i = 0; i < kDig; ++i) tmem_ld4(c0 + (uint32_t)(i * nt), t[i]);
                                unsigned long long *pa = reinterpret_cast<unsigned long long *>(sAcc) + (size_t)n * 128 + row;
                                unsigned long long o[4] = {0, 0, 0, 0};
                                if (pc > 0) {
#pragma unroll
                                    for (int e = 0; e < 4; ++e) o[e] = pa[e * 128];
                                }
                                tmem_ld_wait();
#pragma unroll
                                for (int e = 0; e < 4; ++e) {
                                    float a[kDig];
#pragma unroll
                                    for (int i = 0; i < kDig; ++i) a[i] = __uint_as_float(t[i][e]);
                                    pa[e * 128] = acc_sum_chain<(DS > 0 ? DS : 2)>(a) + o[e] - ChainJoin<(DS > 0 ? DS : 2)>::offset;
                                }
                            }
                        } else
                        for (int n = n_first; n < un.N; n += 16) {
                            uint32_t t[kDig][4];
                            const int hf = n >> 5, nt = un.Nt[hf];
                            const uint32_t c0 = col + (uint32_t)(hf * 256 + (n & 31));
#pragma unroll
                            for (int i = 0; i < kDig; ++i) tmem_ld4(c0 + (uint32_t)(i * nt), t[i]);
                            int4 e4 = make_int4(0, 0, 0, 0);
                            if (last) e4 = __ldg(reinterpret_cast<const int4 *>(et + n));
                            const int ee[4] = {e4.x, e4.y, e4.z, e4.w};
                            tmem_ld_wait();
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                float a[kDig];
#pragma unroll
                                for (int i = 0; i < kDig; ++i) a[i] = __uint_as_float(t[i][e]);
                                result(a, sAcc + (size_t)(n + e) * 128 + row, ee[e], dst + (size_t)(n + e) * prm.ldJ,
                                       dst && n + e < un.N);
                            }
                        }
                        if (un.own0 && grp == 3) {
                            uint32_t w[8];
                            tmem_ld8(col + (uint32_t)(kDig * un.Nt[0]), w);
                            tmem_ld_wait();
                            float a[kDig];
#pragma unroll
                            for (int i = 0; i < kDig; ++i) a[i] = __uint_as_float(w[i]);
                            result(a, sAcc + (size_t)(un.Nt[0] + un.Nt[1]) * 128 + row, __ldg(et + kNtMax), dst - (size_t)un.col0 * prm.ldJ,
                                   dst != nullptr);
                        }
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(smem_u32(&acc_empty[b]));
                    }
#pragma unroll
                    for (int s0 = 0; s0 < kDrainAt; ++s0) load_step(src, lim, s0, v[s0]);
                }
                if (s < steps) {
                    ok = ok && warp_all(mbar_wait(smem_u32(&a_empty[ra.idx]), ra.phase ^ 1, abort_flag, prm.err, budget));
                    if (!ok) break;
                    uint8_t *dst = sA + (size_t)ra.idx * kSlotA1 + a_off;
                    uint32_t wl[4], wh[4], d0[kDig], d1[kDig];
                    if (tiny) scale_up(v[s]);
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        fix55((uint32_t)__double2loint(v[s][e]), (uint32_t)__double2hiint(v[s][e]), e8, wl[e], wh[e]);
                    digits2(wl[0], wh[0], (uint32_t)__double2hiint(v[s][0]), wl[1], wh[1],
                            (uint32_t)__double2hiint(v[s][1]), d0);
                    digits2(wl[2], wh[2], (uint32_t)__double2hiint(v[s][2]), wl[3], wh[3],
                            (uint32_t)__double2hiint(v[s][3]), d1);
#pragma unroll
                    for (int i = 0; i < kDig; ++i)
                        *reinterpret_cast<uint2 *>(dst + i * kDigA1) = make_uint2(d0[i], d1[i]);
                    fence_proxy_async_smem();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&a_full[ra.idx]));
                    ra.next(prm.ns_a);
                }
                if (s >= kDrainAt) load_step(src, lim, s, v[s]);
            }
            pu = steps ? u : -1;
            pc = c;
            u = u2;
            c = c2;
            ++it;
        }
        if (bad) atomicOr(prm.err, DEV_ERR_NONFINITE);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == kWorkWarps) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 512);
    }
}

// ---------------------------------------------------------------------------- expand
struct ExpandParams {
    const double *src;
    double *dst;
    const uint8_t *tab;
    const unsigned long long *off;
    const int *et;
    int *err;
    long long R;
    int n_r, n_t, n_p, L, P, ldJ, ldI;
    int N, n_blk, n_units, n_split, n_groups, n_groups0, et_ld;
    int a_steps, ns_b, tma;       // a_steps: K steps of A held at once; ns_b: table slots per issuer; tma: Phi leaves by TMA stores
};

struct ExpandUnit {
    int set, K, steps, n_chunks, chunk_steps, blk0, blk1, pairs, rot;
    long long row0;
    // first block of the unit's gi-th pair: each CTA starts at another pair, so that the CTAs do
    // not all read the same table blocks at the same time
    __device__ __forceinline__ int pair(int gi) const
    {
        const int v = gi + rot;
        return blk0 + 2 * (v < pairs ? v : v - pairs);
    }
};

template <bool THETA>
__device__ __forceinline__ ExpandUnit expand_unit(const ExpandParams &p, int u)
{
    ExpandUnit r;
    if (!THETA) {
        const int tile = u / p.n_split, part = u - tile * p.n_split;
        r.set = 0;
        r.K = p.P - 1;
        r.row0 = (long long)tile * 128;
        // whole pairs of blocks per part
        const int pairs = (p.n_blk + 1) / 2;
        r.blk0 = 2 * (int)((long long)pairs * part / p.n_split);
        r.blk1 = min(p.n_blk, 2 * (int)((long long)pairs * (part + 1) / p.n_split));
    } else {
        if (u < p.n_groups0) {
            r.set = 0;
            r.row0 = (long long)u * 128;
        } else {
            const int v = u - p.n_groups0;
            r.set = 1 + v / p.n_groups;
            r.row0 = (long long)(v - (r.set - 1) * p.n_groups) * 64;
        }
        r.K = p.L + 1 - r.set;
        r.blk0 = 0;
        r.blk1 = p.n_blk;
    }
    r.steps = max(1, (r.K + 15) / 16);  // (l_max = 0 leaves no term: one step of zeros)
    r.n_chunks = r.steps <= p.a_steps ? 1 : 2;
    r.chunk_steps = (r.steps + r.n_chunks - 1) / r.n_chunks;
    r.pairs = (r.blk1 - r.blk0 + 1) / 2;
    r.rot = (int)(blockIdx.x % (unsigned)max(1, r.pairs));
    return r;
}

// Roles: warps 0-15 split the unit's A (128 rows, the whole K or, past a_steps, half of it at a
// time) and turn finished blocks of 32 columns into float64; the even and the odd blocks have an
// accumulator, an MMA issuer (warps 16, 17) and a table producer (warps 18, 19) each.  With K
// in one piece A is split once per unit; in two it is split again for every pair of blocks.
template <bool THETA, int NM>
__global__ void __launch_bounds__(kThreadsX, 1) k64_expand_tc(const __grid_constant__ CUtensorMap tm_out, const ExpandParams prm)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    constexpr uint32_t kSlotB = kRowsX * 32;
    uint8_t *sOut = smem;                                   // [16 warps][32 rows][8] float64, 64-byte swizzle
    uint8_t *sA = sOut + kWorkWarps * kBoxX;
    uint8_t *sB = sA + (size_t)prm.a_steps * kStepA2;
    uint32_t *sMax = reinterpret_cast<uint32_t *>(sB + (size_t)2 * prm.ns_b * kSlotB);  // [2 units][4][128]
    uint64_t *bars = reinterpret_cast<uint64_t *>(sMax + 8 * 128);
    uint64_t *b_full = bars, *b_empty = b_full + 2 * prm.ns_b;
    uint64_t *a_full = b_empty + 2 * prm.ns_b, *a_free = a_full + 1;
    uint64_t *acc_full = a_free + 1, *acc_empty = acc_full + 2, *m_full = acc_empty + 2, *drain_bar = m_full + 1;
    uint32_t *tmem_holder = reinterpret_cast<uint32_t *>(drain_bar + 2);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_holder + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < 2 * prm.ns_b; ++s) {
            mbar_init(smem_u32(&b_full[s]), 1);
            mbar_init(smem_u32(&b_empty[s]), 1);
        }
        mbar_init(smem_u32(a_full), kWorkWarps);
        mbar_init(smem_u32(a_free), 2);
        mbar_init(smem_u32(m_full), kWorkWarps);
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&acc_full[b]), 1);
            mbar_init(smem_u32(&acc_empty[b]), kWorkWarps);
        }
        mbar_init(smem_u32(&drain_bar[0]), 1);
        mbar_init(smem_u32(&drain_bar[1]), 1);
        *abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == kWorkWarps) {
        tmem_alloc(smem_u32(tmem_holder), 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_holder;
    pdl_wait();  // the source comes from the previous kernels
    const long long budget = wait_budget(prm.err);

    if (warp >= kWorkWarps + 2) {
        // ---------------- table producers, one for each issuer's half of the ring
        if (lane == 0) {
            const int mine = warp - kWorkWarps - 2;
            uint64_t *my_full = b_full + mine * prm.ns_b, *my_empty = b_empty + mine * prm.ns_b;
            uint8_t *ring = sB + (size_t)mine * prm.ns_b * kSlotB;
            Ring rb;
            int issued = 0, blk = 0;
            bool ok = true;
            for (int u = blockIdx.x; u < prm.n_units && ok; u += gridDim.x) {
                const ExpandUnit un = expand_unit<THETA>(prm, u);
                const uint8_t *src = prm.tab + prm.off[un.set];
                for (int gi = 0; gi < un.pairs && ok; ++gi) {
                    const int g = un.pair(gi);
                    const int nbs = min(2, un.blk1 - g);
                    const int nb = (blk & 1) ^ mine;  // this producer's block of the pair
                    blk += nbs;
                    if (nb >= nbs) continue;
                    const uint8_t *from = src + (size_t)(g + nb) * un.steps * kSlotB;
                    for (int s = 0; s < un.steps; ++s, rb.next(prm.ns_b)) {
                        ok = mbar_wait(smem_u32(&my_empty[rb.idx]), rb.phase ^ 1, abort_flag, prm.err, budget);
                        if (!ok) break;
                        const uint32_t bar = smem_u32(&my_full[rb.idx]);
                        mbar_arrive_expect_tx(bar, kSlotB);
                        bulk_load(smem_u32(ring + (size_t)rb.idx * kSlotB), from + (size_t)s * kSlotB, kSlotB, bar);
                        ++issued;
                    }
                }
            }
            drain_ring(my_full, rb, prm.ns_b, issued);
        }
    } else if (warp >= kWorkWarps) {
        // ---------------- MMA issuers (the whole warp waits, one lane issues): one for the even
        // blocks, one for the odd ones, each with an accumulator of its own.  One issuer alone took
        // 500 to 800 cycles a K step of seven MMAs (448 cycles of tensor time).
        const uint32_t leader = elect_one();
        const int mine = warp - kWorkWarps;
        const uint32_t d0 = tmem_base + (uint32_t)mine * 256;
        const uint32_t a_lo0 = (uint32_t)sdesc_noswizzle(smem_u32(sA), kLboA2, 128);
        const uint32_t a_hi = (uint32_t)(sdesc_noswizzle(smem_u32(sA), kLboA2, 128) >> 32);
        uint8_t *ring = sB + (size_t)mine * prm.ns_b * kSlotB;  // this issuer's half of the table ring
        uint64_t *my_full = b_full + mine * prm.ns_b, *my_empty = b_empty + mine * prm.ns_b;
        const uint32_t b_lo0 = (uint32_t)sdesc_noswizzle(smem_u32(ring), kRowsX * 16, 128);
        const uint32_t b_hi = (uint32_t)(sdesc_noswizzle(smem_u32(ring), kRowsX * 16, 128) >> 32);
        Ring rb;
        int blk = 0, conv = 0;  // blocks and splits of A so far
        bool ok = true;
        for (int u = blockIdx.x; u < prm.n_units && ok; u += gridDim.x) {
            const ExpandUnit un = expand_unit<THETA>(prm, u);
            for (int gi = 0; gi < un.pairs && ok; ++gi) {
                const int nbs = min(2, un.blk1 - un.pair(gi));
                for (int ch = 0; ch < un.n_chunks && ok; ++ch) {
                    if (un.n_chunks > 1 || gi == 0) {
                        ok = warp_all(mbar_wait(smem_u32(a_full), conv & 1, abort_flag, prm.err, budget));
                        if (!ok) break;
                        ++conv;
                    }
                    const int s0 = ch * un.chunk_steps, s1 = min(un.steps, s0 + un.chunk_steps);
                    for (int nb = 0; nb < nbs && ok; ++nb) {
                        if (((blk + nb) & 1) != mine) continue;
                        if (ch == 0) {
                            ok = warp_all(mbar_wait(smem_u32(&acc_empty[mine]), (((blk + nb) >> 1) & 1) ^ 1, abort_flag,
                                                           prm.err, budget));
                            if (!ok) break;
                            tc_fence_after();
                        }
                        uint32_t a_lo = a_lo0;
                        for (int s = s0; s < s1; ++s, rb.next(prm.ns_b), a_lo += kStepA2 / 16) {
                            ok = warp_all(mbar_wait(smem_u32(&my_full[rb.idx]), rb.phase, abort_flag, prm.err, budget));
                            if (!ok) break;
                            const uint32_t b_lo = b_lo0 + (uint32_t)rb.idx * (kSlotB / 16);
#pragma unroll
                            for (int i = 0; i < kDig; ++i)
                                umma_warp(d0 + (uint32_t)(i * kNtX), a_lo + i * (kDigA2 / 16), a_hi, b_lo, b_hi,
                                              idesc_f16_f32(128, (kDig - i) * kNtX), (s | i) != 0, leader);
                            umma_commit_warp(smem_u32(&my_empty[rb.idx]), leader);
                        }
                        if (ok && ch == un.n_chunks - 1) umma_commit_warp(smem_u32(&acc_full[mine]), leader);
                    }
                    // this piece of A has been read
                    if (ok && (un.n_chunks > 1 || gi == un.pairs - 1)) umma_commit_warp(smem_u32(a_free), leader);
                }
                blk += nbs;
            }
        }
        // both issuers' MMAs are complete before the block gives its memory back
        umma_commit_warp(smem_u32(&drain_bar[mine]), leader);
        const long long t0 = clock64();
        while (!mbar_try_wait(smem_u32(&drain_bar[mine]), 0) && clock64() - t0 < MP_WAIT_BUDGET_CYCLES) {
        }
        __syncwarp();
    } else {
        // ---------------- split + drain
        const int crow = threadIdx.x & 127, cg = threadIdx.x >> 7;  // split: row, octets cg, cg + 4, ...
        const int q4 = warp & 3, grp = warp >> 2;  // drain: lane quarter (row 32 q4 + lane = crow), 8 columns
        bool ok = true;
        int blk = 0, splits = 0, lu = 0;
        const uint64_t policy = l2_evict_first_policy();  // Phi is not read again here

        for (int u = blockIdx.x; u < prm.n_units && ok; u += gridDim.x, ++lu) {
            const ExpandUnit un = expand_unit<THETA>(prm, u);
            // element k of this thread's row: src + base + (PH: k ldJ; TH: ((m + k)^2 + p) ldI)
            const double *base = nullptr;
            if (!THETA) {
                const long long r = un.row0 + crow;
                if (r < prm.R) {
                    const int i = (int)(r / prm.n_t), j = (int)(r - (long long)i * prm.n_t);
                    base = prm.src + (size_t)i * prm.P * prm.ldJ + j;
                }
            } else {
                const int a = un.set ? crow >> 6 : 0, i = (int)un.row0 + (un.set ? crow & 63 : crow);
                if (i < prm.n_r) base = prm.src + (size_t)(un.set ? 2 * un.set - 1 + a : 0) * prm.ldI + i;
            }
            // start of this thread's drain row (32 q4 + lane = crow) in the output, where it is not
            // stored by TMA
            double *out_row = nullptr;
            if (!THETA && !prm.tma && un.row0 + crow < prm.R) out_row = prm.dst + (un.row0 + crow) * prm.n_p;
            auto element = [&](int k) -> double {
                if (!base || k >= un.K) return 0.0;
                return !THETA ? __ldg(base + (size_t)(k + 1) * prm.ldJ)
                              : __ldg(base + (size_t)(un.set + k) * (un.set + k) * prm.ldI);
            };
            // phi: the column m = 0, each thread its own row's (the drain row is the split row)
            double g0 = 0.0;
            if (!THETA && base) g0 = __ldg(base);
            uint32_t mx = abs_hi(g0);
            // the first octets stay in registers for the split, further ones are read again
            double x0[kKeepX][8];
#pragma unroll
            for (int c = 0; c < kKeepX; ++c)
#pragma unroll
                for (int e = 0; e < 8; ++e) x0[c][e] = element(8 * (cg + 4 * c) + e);
            for (int o = cg + 4 * kKeepX; o < 2 * un.steps; o += 4) {
                double x[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) x[e] = element(8 * o + e);
#pragma unroll
                for (int e = 0; e < 8; ++e) mx = max(mx, abs_hi(x[e]));
            }
#pragma unroll
            for (int c = 0; c < kKeepX; ++c)
#pragma unroll
                for (int e = 0; e < 8; ++e) mx = max(mx, abs_hi(x0[c][e]));
            uint32_t *row_max = sMax + (lu & 1) * 512 + crow;
            row_max[cg * 128] = mx;
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(m_full));
            ok = warp_all(mbar_wait(smem_u32(m_full), lu & 1, abort_flag, prm.err, budget));
            if (!ok) break;
            mx = max(max(row_max[0], row_max[128]), max(row_max[256], row_max[384]));
            int E = (int)(mx >> 20), E0 = 0;
            if (E < 128) {  // next to the bottom of the float64 range: scaled up exactly
                E = max(128, scaled_up_exponent(mx));
                E0 = -300;
            }
            const int Erow = E + E0;
            const int e8 = E + 8;
            // in units of 2^56: 1.0 in the table would be 2^54, so a quarter of its 55-bit integer
            uint32_t g0_lo = 0, g0_hi = 0;
            if (!THETA) {
                if (E0) {
                    double t[1] = {g0};
                    scale_up(t);
                    g0 = t[0];
                }
                uint32_t wl, wh;
                fix55((uint32_t)__double2loint(g0), (uint32_t)__double2hiint(g0), e8, wl, wh);
                long long q = (long long)((((unsigned long long)wh << 32 | wl) - 0x0000808080808080ull + 2) >> 2);
                if (g0 < 0.0) q = -q;
                g0_lo = (uint32_t)q;
                g0_hi = (uint32_t)(q >> 32);
            }

            auto split_octet = [&](double (&x)[8], int o, int s0) {
                if (E0) scale_up(x);
                uint32_t d[4][kDig];
#pragma unroll
                for (int e = 0; e < 8; e += 2) {
                    uint32_t wl0, wh0, wl1, wh1;
                    const uint32_t h0 = (uint32_t)__double2hiint(x[e]), h1 = (uint32_t)__double2hiint(x[e + 1]);
                    fix55((uint32_t)__double2loint(x[e]), h0, e8, wl0, wh0);
                    fix55((uint32_t)__double2loint(x[e + 1]), h1, e8, wl1, wh1);
                    digits2(wl0, wh0, h0, wl1, wh1, h1, d[e >> 1]);
                }
                uint8_t *dst = sA + (size_t)((o >> 1) - s0) * kStepA2 + (o & 1) * kLboA2 + crow * 16;
#pragma unroll
                for (int i = 0; i < kDig; ++i)
                    *reinterpret_cast<uint4 *>(dst + i * kDigA2) = make_uint4(d[0][i], d[1][i], d[2][i], d[3][i]);
            };
            // A for the K steps of piece ch, once the MMAs of the piece before have read theirs
            auto split = [&](int ch) -> bool {
                if (splits > 0 &&
                    !warp_all(mbar_wait(smem_u32(a_free), (splits - 1) & 1, abort_flag, prm.err, budget)))
                    return false;
                ++splits;
                const int s0 = ch * un.chunk_steps, s1 = min(un.steps, s0 + un.chunk_steps);
                int o = 2 * s0 + cg;
                if (un.n_chunks == 1) {
#pragma unroll
                    for (int c = 0; c < kKeepX; ++c, o += 4)
                        if (o < 2 * s1) split_octet(x0[c], o, s0);
                }
                for (; o < 2 * s1; o += 4) {
                    double x[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) x[e] = element(8 * o + e);
                    split_octet(x, o, s0);
                }
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(a_full));
                return true;
            };

            if (un.n_chunks == 1) ok = split(0);
            for (int gi = 0; gi < un.pairs && ok; ++gi) {
                const int g = un.pair(gi);
                const int nbs = min(2, un.blk1 - g);
                if (un.n_chunks > 1)
                    for (int ch = 0; ch < un.n_chunks && ok; ++ch) ok = split(ch);
                for (int nb = 0; nb < nbs && ok; ++nb, ++blk) {
                    const int b = blk & 1;
                    ok = warp_all(mbar_wait(smem_u32(&acc_full[b]), (blk >> 1) & 1, abort_flag, prm.err, budget));
                    if (!ok) break;
                    tc_fence_after();
                    uint32_t t[kDig][8];
                    const uint32_t col = tmem_base + (uint32_t)b * 256 + ((uint32_t)(q4 * 32) << 16) + grp * 8;
#pragma unroll
                    for (int i = 0; i < kDig; ++i) tmem_ld8(col + (uint32_t)(i * kNtX), t[i]);
                    const int n0 = (g + nb) * kNtX + grp * 8;
                    // column exponents (padded to whole blocks); the phi table, cell means of cos
                    // and sin, has one scale
                    int Et[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) Et[e] = 1023;
                    if (THETA) {
                        const int4 *pe = reinterpret_cast<const int4 *>(prm.et + (size_t)un.set * prm.et_ld + n0);
                        const int4 e0 = __ldg(pe), e1 = __ldg(pe + 1);
                        Et[0] = e0.x, Et[1] = e0.y, Et[2] = e0.z, Et[3] = e0.w;
                        Et[4] = e1.x, Et[5] = e1.y, Et[6] = e1.z, Et[7] = e1.w;
                    }
                    tmem_ld_wait();
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&acc_empty[b]));
                    double out[8];
                    uint32_t lo[8], hi[8];
                    int be0[8];
                    const int e_base = 56 + Erow - 2154;
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        float a[kDig];
#pragma unroll
                        for (int i = 0; i < kDig; ++i) a[i] = __uint_as_float(t[i][e]);
                        if (NM >= 6)
                            acc_sum_small(a, lo[e], hi[e]);
                        else
                            acc_sum<NM, 0>(a, lo[e], hi[e]);
                        if (!THETA)
                            asm("add.cc.u32 %0, %0, %2;\n\taddc.u32 %1, %1, %3;" : "+r"(lo[e]), "+r"(hi[e]) : "r"(g0_lo), "r"(g0_hi));
                        be0[e] = e_base + Et[e] + 1084;
                    }
                    // exponents in the middle of the range keep every result normal
                    bool odd = !THETA ? (unsigned)(Erow - 200) > 1600u : Erow >= kExpNan;
                    if (THETA) {
#pragma unroll
                        for (int e = 0; e < 8; ++e) odd |= (unsigned)(be0[e] - 64) > 1900u;
                    }
                    if ((!scaled_row<8>(lo, hi, be0, out) || odd) && base) {
                        // small integers (zeros among them), rows near the ends of the range or with a NaN
#pragma unroll
                        for (int e = 0; e < 8; ++e) out[e] = scaled_i64_slow(lo[e], hi[e], be0[e] - 1084, Erow);
                    }
                    if (THETA || prm.tma) {
                        // the warp's box of 32 rows x 8 columns: 64-byte rows, 16-byte pieces permuted
                        // by the TMA's 64-byte swizzle
                        uint8_t *box = sOut + warp * kBoxX;
                        if (lane == 0) bulk_wait_read_all();  // the box before has left
                        __syncwarp();
#pragma unroll
                        for (int c = 0; c < 4; ++c)
                            *reinterpret_cast<double2 *>(box + lane * 64 + ((c ^ ((lane >> 1) & 3)) << 4)) =
                                make_double2(out[2 * c], out[2 * c + 1]);
                        fence_proxy_async_smem();
                        __syncwarp();
                        if (lane == 0) {
                            if (THETA) {
                                const int r0 = 32 * q4, a = un.set ? r0 >> 6 : 0;
                                const int i = (int)un.row0 + (un.set ? r0 & 63 : r0);
                                if (i < prm.n_r && n0 < prm.N)
                                    tma_store_3d(&tm_out, smem_u32(box), n0, un.set ? 2 * un.set - 1 + a : 0, i);
                            } else if (n0 < prm.N && un.row0 + 32 * q4 < prm.R) {
                                tma_store_2d_hint(&tm_out, smem_u32(box), n0, (int)(un.row0 + 32 * q4), policy);
                            }
                            bulk_commit();
                        }
                    } else if (out_row) {
#pragma unroll
                        for (int e = 0; e < 8; ++e)
                            if (n0 + e < prm.N) out_row[n0 + e] = out[e];
                    }
                }
            }
        }
        if (lane == 0) bulk_wait_all();
    }
    tc_fence_before();
    __syncthreads();
    if (warp == kWorkWarps) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 512);
    }
}

}  // namespace

// ---------------------------------------------------------------------------- host side

namespace {

constexpr int kSmemMax = 227 * 1024;

int ceil_log2(int x)
{
    int b = 0;
    while ((1 << b) < x) ++b;
    return b;
}

// Ring depths and shared memory of a contraction of K terms whose widest set has N columns (and
// a column m = 0 of its own).
bool plan_contract(int K, int N, int own0, Fp64Contract &c)
{
    const int Nt = half_cols(N, 0) + half_cols(N, 1);
    c.n_steps = (K + 15) / 16;
    c.n_chunks = (c.n_steps + kChunkSteps - 1) / kChunkSteps;
    c.ds = c.n_chunks == 1 ? 0 : c.n_chunks <= 4 ? 2 : c.n_chunks <= 16 ? 4 : ceil_log2(c.n_chunks);
    c.cols_max = Nt + own0;
    c.nacc = N <= kHalf ? 2 : 1;
    c.slot_b = (kDig * Nt + (own0 ? kRows0 : 0)) * 32;
    if (N > kNtMax || c.ds > 31) return false;
    const int fixed = (c.n_chunks > 1 ? c.cols_max * 1024 : 0) + 4 * 128 * 4 + 512;
    for (auto d : {std::pair<int, int>{4, 4}, {4, 3}, {3, 3}, {3, 2}, {2, 2}}) {
        c.ns_a = d.first;
        c.ns_b = d.second;
        c.smem = fixed + c.ns_a * kSlotA1 + c.ns_b * c.slot_b;
        if (c.smem <= kSmemMax) return true;
    }
    return false;
}

bool plan_expand(int K, Fp64Expand &x)
{
    if (K > kExpandKMax) return false;
    const int steps = std::max(1, (K + 15) / 16);
    x.a_steps = steps <= 5 ? steps : (steps + 1) / 2;
    const int fixed = x.a_steps * kStepA2 + kWorkWarps * kBoxX + 8 * 128 * 4 + 1024 + 256;
    for (x.ns_b = 8; x.ns_b >= 2; --x.ns_b) {
        x.smem = fixed + 2 * x.ns_b * kRowsX * 32;
        if (x.smem <= kSmemMax) return true;
    }
    return false;
}

size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

}  // namespace

void plan_fp64_tc(mp_mesh *m, bool far_moments)
{
    Fp64Plan &f = m->fp;
    f = Fp64Plan();
    f.ldJ = round_up(m->n_t, 4);
    // columns per pass over the density; the column m = 0 gets a block of its own where the
    // others fill blocks of 16 without it
    f.m0 = m->L > 0 && m->L % 8 == 0;
    const int cols = m->P - f.m0;
    f.npass = (cols + kNtMax - 1) / kNtMax;
    f.pass_cols = (cols + f.npass - 1) / f.npass;
    if (f.npass > 1) f.pass_cols = std::min(kNtMax, ceil16(f.pass_cols));
    // 2 l_max terms in the chains of the phi synthesis, row indices in 32 bits
    if (m->L > 71 || m->R >= (1LL << 31)) return;
    // below 16 azimuthal cells (axisymmetric meshes have one) a 16-wide K step is mostly padding
    // and the sums are short: CUDA cores
    const bool few = m->n_p < 16;

    // Moments whose radial weights reach 1e150 (l_max = 48 over five decades of r): their squares
    // leave the float64 range, so neither they nor the differences of two solutions have a norm,
    // and equality is the one way to compare them.  They stay sums in the order of the CUDA-core
    // kernels, those of mp_moments_noalloc, to the last bit.  It costs their speed: 260 x 130 x 150
    // cells, l_max = 64: 346 -> 1860 us a solve (3594 with the synthesis on CUDA cores as well).
    //
    // Azimuthal cells of widths more than a factor of two apart leave the projection there too: its
    // fixed point is that of the widest cell, so the others of a ring whose largest cell is narrow
    // are off by up to K 2^-56 x (widest / narrowest) of what the largest adds, K 2^-53 in a float64
    // sum with two bits less for where the values lie between powers of two.  (One of 64 cells 1e-6
    // as wide, and hot: 3e-11 of the moments' terms.)
    double widest = 0.0, narrowest = HUGE_VAL;
    for (int k = 0; k < m->n_p; ++k) {
        widest = std::max(widest, m->h_ph[k + 1] - m->h_ph[k]);
        narrowest = std::min(narrowest, m->h_ph[k + 1] - m->h_ph[k]);
    }
    // Small meshes: a tensor-core kernel of this file takes 11 to 15 us for a single tile, where the
    // CUDA-core ones take 6 and more by their products.  The two cross (both sides' times in
    // us): projection with the theta contraction behind it at 0.6 M products (40 x 24 x 17 cells, l_max =
    // 8: 21.5 against 19.6; 64 x 32 x 64, 2: 21.7 against 22.6), later where F's rows of polar cells
    // are short (512 x 1 x 64, 16: 24.6 against 19.3); synthesis where the phi products and three
    // times the theta products (uncoalesced) reach 6 M (64 x 32 x 64, 8: 24.1 against 20.1; 16: 26.6
    // against 27.2); theta synthesis alone at 0.6 M (128 x 64 x 1, 2: 12.5 against 7.3; 8: 12.5
    // against 15.8).
    const double phi_products = (double)m->R * m->n_p * m->P, theta_products = (double)m->R * m->KL;
    f.proj_on = !few && !far_moments && widest <= 2.0 * narrowest && phi_products >= (m->n_t >= 8 ? 0.6e6 : 4.8e6) &&
                plan_contract(m->n_p, f.pass_cols, f.m0, f.ph_c);
    f.rows = f.proj_on || (few && !far_moments);
    f.on = (few ? theta_products >= 0.6e6 : phi_products + 3.0 * theta_products >= 6e6) && plan_expand(m->L + 1, f.th_x);
    f.phi_on = f.on && !few && plan_expand(m->P - 1, f.ph_x);
    if (f.on) f.ldI = round_up(m->n_r, 4);
}

size_t fp64_tc_arena(mp_mesh *m)
{
    Fp64Plan &f = m->fp;
    const int L = m->L;
    size_t at = 0;
    auto take = [&](size_t bytes) {
        const size_t o = at;
        at = align256(at + bytes);
        return o;
    };
    f.off_ld = std::max(L + 1, f.npass);
    f.h_off.assign((size_t)3 * f.off_ld, 0);
    unsigned long long *ox = f.h_off.data(), *op = ox + f.off_ld;
    unsigned long long x = 0;
    const int n_blk = (m->n_t + kNtX - 1) / kNtX;
    for (int mm = 0; mm <= L && f.on; ++mm) {
        ox[mm] = x;
        x += (unsigned long long)n_blk * ((L + 1 - mm + 15) / 16) * kRowsX * 32;
    }
    const unsigned long long pstep = (unsigned long long)f.ph_c.n_steps * f.ph_c.slot_b;
    for (int s = 0; s < f.npass; ++s) op[s] = s * pstep;
    f.o_tab_x = take(x);
    f.o_tab_pc = take(f.proj_on ? f.npass * pstep : 0);
    f.o_tab_px = take(f.phi_on ? (size_t)((m->n_p + kNtX - 1) / kNtX) * std::max(1, (m->P - 1 + 15) / 16) * kRowsX * 32 : 0);
    f.o_off = take(f.h_off.size() * sizeof(unsigned long long));
    f.o_et_x = take((size_t)(L + 1) * round_up(m->n_t, kNtX) * 4);
    f.o_et_pc = take((size_t)f.npass * kEtLd * 4);
    f.o_bound = take(4 * sizeof(int));
    f.o_et_px = take((size_t)round_up(m->n_p, kNtX) * 4);
    return at;
}

static const unsigned long long *fp64_off(const mp_mesh *m, int which)
{
    return reinterpret_cast<const unsigned long long *>(m->fp.arena + m->fp.o_off) + (size_t)which * m->fp.off_ld;
}

// The contraction's variants: 32-byte loads, the bits dropped from a chain's sum
// (none for one chain; 2 for up to 4, 4 for up to 16, the number of bits at run time beyond) and,
// for several chains, whether the table keeps the first three accumulators below 2^22.
template <int NM>
static void (*contract_kernel_nm(int vec, int ds, int n_chunks))(ContractParams)
{
    auto pick = [&](auto k0, auto k2, auto k4, auto kr) {
        return n_chunks == 1 ? k0 : ds == 2 ? k2 : ds == 4 ? k4 : kr;
    };
    return vec ? pick(k64_contract_tc<true, 0, 2>, k64_contract_tc<true, 2, NM>, k64_contract_tc<true, 4, NM>,
                      k64_contract_tc<true, -1, 2>)
               : pick(k64_contract_tc<false, 0, 2>, k64_contract_tc<false, 2, NM>, k64_contract_tc<false, 4, NM>,
                      k64_contract_tc<false, -1, 2>);
}
static void (*contract_kernel(int vec, int ds, int n_chunks, int small))(ContractParams)
{
    return small ? contract_kernel_nm<3>(vec, ds, n_chunks) : contract_kernel_nm<2>(vec, ds, n_chunks);
}

static void (*expand_kernel(int theta, int nm))(const CUtensorMap, ExpandParams)
{
    if (theta) return nm == 6 ? k64_expand_tc<true, 6> : nm == 3 ? k64_expand_tc<true, 3> : k64_expand_tc<true, 1>;
    return nm == 6 ? k64_expand_tc<false, 6> : nm == 3 ? k64_expand_tc<false, 3> : k64_expand_tc<false, 1>;
}

cudaError_t launch_fp64_tc_tables(mp_mesh *m)
{
    Fp64Plan &f = m->fp;
    const int L = m->L;
    cudaError_t e = cudaMemsetAsync(f.arena, 0, f.arena_bytes, m->stream);
    if (e != cudaSuccess) return e;
    e = cudaMemcpyAsync(f.arena + f.o_off, f.h_off.data(), f.h_off.size() * sizeof(unsigned long long),
                        cudaMemcpyHostToDevice, m->stream);
    if (e != cudaSuccess) return e;
    auto build = [&](int kind, size_t tab, int off, size_t et, int et_ld, int n_max, int n_sets) {
        TabParams t{m->d_Ith, m->d_Iph, m->d_Iphc, m->d_dmu, f.arena + tab, fp64_off(m, off),
                    reinterpret_cast<int *>(f.arena + et), kind, m->n_t, m->n_p, L, m->P, f.pass_cols, f.m0, et_ld,
                    reinterpret_cast<int *>(f.arena + f.o_bound) + kind};
        k64_digit_tables<<<dim3((n_max + 3) / 4, n_sets), 128, 0, m->stream>>>(t);
    };
    if (f.on) build(TAB_EXPAND_TH, f.o_tab_x, 0, f.o_et_x, round_up(m->n_t, kNtX), m->n_t, L + 1);
    if (f.proj_on) build(TAB_PROJECT, f.o_tab_pc, 1, f.o_et_pc, kEtLd, f.pass_cols + f.m0, f.npass);
    if (f.phi_on) build(TAB_EXPAND_PH, f.o_tab_px, 2, f.o_et_px, round_up(m->n_p, kNtX), m->n_p, 1);
    // 227 KB of dynamic shared memory for the kernels of this file (per device)
    for (int vec = 0; vec < 2; ++vec)
        for (int v = 0; v < 8; ++v) {
            const int ds = v < 6 ? (v >> 1) * 2 : 5;
            e = cudaFuncSetAttribute((const void *)contract_kernel(vec, ds, ds ? 2 : 1, v & 1),
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax);
            if (e != cudaSuccess) return e;
        }
    for (int theta = 0; theta < 2; ++theta) {
        for (int nm : {1, 3, 6}) {
            e = cudaFuncSetAttribute((const void *)expand_kernel(theta, nm), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     kSmemMax);
            if (e != cudaSuccess) return e;
        }
    }
    return cudaGetLastError();
}

cudaError_t fp64_tc_bounds(mp_mesh *m)
{
    int b[3] = {0, 0, 0};
    cudaError_t e = cudaMemcpy(b, m->fp.arena + m->fp.o_bound, sizeof(b), cudaMemcpyDeviceToHost);
    m->fp.ph_c.small = b[TAB_PROJECT] < (1 << 22);
    m->fp.th_x.small = b[TAB_EXPAND_TH] < (1 << 22);
    m->fp.ph_x.small = b[TAB_EXPAND_PH] < (1 << 22);
    return e;
}

static cudaError_t launch_expand(mp_mesh *m, int theta, const double *src, double *dst, const char *name)
{
    const Fp64Plan &f = m->fp;
    const Fp64Expand &x = theta ? f.th_x : f.ph_x;
    ExpandParams p{};
    p.src = src;
    p.dst = dst;
    p.tab = f.arena + (theta ? f.o_tab_x : f.o_tab_px);
    p.off = fp64_off(m, theta ? 0 : 2);
    p.et = reinterpret_cast<const int *>(f.arena + (theta ? f.o_et_x : f.o_et_px));
    p.err = m->d_err;
    p.R = m->R;
    p.n_r = m->n_r, p.n_t = m->n_t, p.n_p = m->n_p, p.L = m->L, p.P = m->P, p.ldJ = f.ldJ, p.ldI = f.ldI;
    p.N = theta ? m->n_t : m->n_p;
    p.n_blk = (p.N + kNtX - 1) / kNtX;
    p.n_groups = (m->n_r + 63) / 64, p.n_groups0 = (m->n_r + 127) / 128;
    p.et_ld = round_up(p.N, kNtX);
    p.a_steps = x.a_steps, p.ns_b = x.ns_b;
    const int tiles = (int)((m->R + 127) / 128), pairs = (p.n_blk + 1) / 2;
    // fewer tiles than SMs: a tile's columns go to several CTAs (each splits the tile's A)
    p.n_split = theta ? 1 : std::max(1, std::min(pairs, m->num_sms / std::max(1, tiles)));
    p.n_units = theta ? p.n_groups0 + m->L * p.n_groups : tiles * p.n_split;
    // TMA stores where the rows' starts are multiples of 16 bytes
    p.tma = theta || (m->n_p % 2 == 0 && (reinterpret_cast<uintptr_t>(dst) & 15) == 0);
    CUtensorMap map = theta ? m->tm_G64 : m->tm_phi;
    if (!theta && p.tma && m->tm_phi_ptr != dst) {
        if (make_map_f64_rows(&m->tm_phi, dst, m->R, m->n_p, 32, 8) != MP_OK) return cudaErrorInvalidValue;
        m->tm_phi_ptr = dst;
        map = m->tm_phi;
    }
    cudaEvent_t ev;
    prof_begin(m, name, &ev);
    // leading accumulators below 2^22: all where the table's digits keep them there (l_max up to
    // about 35), else by the length of the chains (one more pair of digits each)
    const int K = theta ? m->L + 1 : m->P - 1;
    const int nm = x.small ? 6 : 3 * K < 256 ? 3 : 1;
    auto kern = expand_kernel(theta, nm);
    cudaError_t e = launch_pdl(kern, dim3(std::min(p.n_units, m->num_sms)), dim3(kThreadsX), x.smem,
                               m->stream, map, p);
    prof_end(m, name, ev);
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_fp64_tc_project(mp_mesh *m, const double *rho)
{
    const Fp64Plan &f = m->fp;
    const Fp64Contract &c = f.ph_c;
    ContractParams p{};
    p.src = rho;
    p.dst = m->d_F64;
    p.tab = f.arena + f.o_tab_pc;
    p.off = fp64_off(m, 1);
    p.et = reinterpret_cast<const int *>(f.arena + f.o_et_pc);
    p.err = m->d_err;
    p.R = m->R;
    p.n_t = m->n_t, p.n_p = m->n_p, p.P = m->P, p.ldJ = f.ldJ;
    p.n_steps = c.n_steps, p.n_chunks = c.n_chunks, p.ds = c.ds;
    p.npass = f.npass, p.pass_cols = f.pass_cols, p.m0 = f.m0;
    p.n_units = (int)((m->R + 127) / 128) * f.npass;
    p.ns_a = c.ns_a, p.ns_b = c.ns_b, p.nacc = c.nacc, p.slot_b = c.slot_b, p.cols_max = c.cols_max;
    // 32-byte loads where every row starts on a 32-byte boundary
    const bool vec = m->n_p % 4 == 0 && (reinterpret_cast<uintptr_t>(rho) & 31) == 0;
    auto kern = contract_kernel(vec, c.ds, c.n_chunks, c.small);
    cudaEvent_t ev;
    prof_begin(m, "fp64_phi_project", &ev);
    cudaError_t e = launch_pdl(kern, dim3(std::min(p.n_units, m->num_sms)), dim3(kThreadsC), c.smem,
                               m->stream, p);
    prof_end(m, "fp64_phi_project", ev);
    return e != cudaSuccess ? e : cudaGetLastError();
}
cudaError_t launch_fp64_tc_synth_theta(mp_mesh *m)
{
    return launch_expand(m, 1, m->d_C, m->d_G64, "fp64_theta_synth");
}
cudaError_t launch_fp64_tc_synth_phi(mp_mesh *m, double *phi)
{
    return launch_expand(m, 0, m->d_G64, phi, "fp64_phi_synth");
}

}  // namespace mp
