// mp_fp64_tc.cu -- the float64 path's four contractions on the tensor cores, to float64
// accuracy, by exact integer slices.
//
// GB300 does about 0.5 T float64 operations a second, 1/1700 of its 16-bit tensor rate, so
// the contractions of GenASiS II Sec. 2.2 (both factors of Eq. (AngularMomentsDiscrete) and
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
// instructions; no step uses the float64 pipe.  A value 2^k below its row's maximum keeps
// 55 - k bits; float64 sums of such rows carry a rounding error of that size as well.
//
// Two kernels serve the four steps.  A is always the data (split on the fly), B a table
// (split once per mesh), D = A B^T:
//   k64_contract_tc  long K, few columns (K streamed):
//       (a1) F[i][p][j] = sum_k rho[i][j][k] Iph[p][k]      rows (i, j), K = n_phi
//       (a2) A[i][q]    = 4 pi G sum_j F[i][p][j] Ith[t][j]  rows (i, cos | sin) of one order m,
//                                                            columns l = m .. L, K = n_theta
//   k64_expand_tc    short K, many columns (A kept, columns streamed):
//       (d1) G[i][p][j] = sum_l C[q][i] Ith[t][j] / dmu_j    rows (i, cos | sin) of one order m,
//                                                            columns j, K = L + 1 - m
//       (d2) Phi[i][j][k] = sum_p G[i][p][j] Iph[p][k]/dphi_k  rows (i, j), columns k, K = 2 L + 1
// The seven digit matrices of B are stacked along N: digit a of A times the first 7 - a
// digits of B is one MMA of N = (7 - a) Nt columns whose result lands Nt a columns to the
// right, so a K step of 16 takes seven MMAs for its 28 products and reads A seven times
// instead of 28 (with one MMA per pair the shared-memory reads of A would bound it).
#include <algorithm>

#include <cuda_fp16.h>

#include "mp_internal.h"
#include "ptx.cuh"

namespace mp {

namespace {

constexpr int kDig = 7;              // digits per operand
constexpr int kChunkSteps = 8;       // contract: K steps (of 16) that share a row exponent and a chain
constexpr int kExpandKMax = 146;     // expand: longest chain (7 * 146 * 2^14 < 2^24)
constexpr int kWorkWarps = 16;
constexpr int kThreads = (kWorkWarps + 2) * 32;
constexpr int kExpNan = 2047;        // row exponent of a row with an infinity or a NaN
constexpr int kNtX = 32;             // expand: columns per block
constexpr int kRowsX = kDig * kNtX;  // expand: stacked table rows of a block

// contract: A slot of one K step: [digit][octet of k][128 rows][8 k]; the octets are 64 bytes
// further apart than their size, so that a half warp's 8-byte stores (4 rows x 2 octets x 2)
// fall on different banks
constexpr int kLboA1 = 128 * 16 + 64;
constexpr int kDigA1 = 2 * kLboA1;
constexpr int kSlotA1 = kDig * kDigA1;
// expand: the same without the pad (a warp stores 32 consecutive rows)
constexpr int kLboA2 = 128 * 16;
constexpr int kDigA2 = 2 * kLboA2;
constexpr int kStepA2 = kDig * kDigA2;

__host__ __device__ inline int ceil16(int x) { return (x + 15) & ~15; }

// Contract: the columns of a set in tensor memory. Accumulator blocks start on multiples of 16
// columns, so a set of N columns takes Nt = N rounded up to 16 for each of the seven weights
// (64 at most: 7 * 64 = 448 of 512).  A projection of P = 2 L + 1 columns with L a multiple of 8
// would pay a block of 16 for its one column m = 0 seven times over and, at l_max = 32, no longer
// fit one pass; its column m = 0 takes one block of 16 instead, with the seven weights as its
// columns: for digit a of A the table rows of that block are the column's digits a places
// further down.
constexpr int kNtMax = 64;
constexpr int kRows0 = kDig * 16;   // table rows of the column m = 0: [digit of A][16]

// ---------------------------------------------------------------------------- digits
// |x| as a 55-bit integer relative to the row exponent (x = +- V 2^(E - 1077), V < 2^55,
// truncated), with 0x80 added to its six low bytes: byte b of the sum less 128 is then a
// balanced digit, and the seventh byte the leading one (0 .. 128).  e9 = E + 9.
__device__ __forceinline__ void fix55(uint32_t lo, uint32_t hi, int e9, uint32_t &wl, uint32_t &wh)
{
    const int n = e9 - (int)((hi >> 20) & 0x7FFu);
    const uint32_t th = __funnelshift_l(lo, hi, 11) | 0x80000000u, tl = lo << 11;
    uint32_t vl = __funnelshift_rc(tl, th, n), vh;
    asm("shr.u32 %0, %1, %2;" : "=r"(vh) : "r"(th), "r"(n));
    const int n2 = max(n - 32, 0);
    asm("shr.u32 %0, %1, %2;" : "=r"(vl) : "r"(vl), "r"(n2));
    asm("add.cc.u32 %0, %2, 0x80808080;\n\taddc.u32 %1, %3, 0x00008080;" : "=r"(wl), "=r"(wh) : "r"(vl), "r"(vh));
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

// acc 2^e2 as float64 by integer instructions (round to nearest); results outside the normal
// range go through ldexp.
__device__ __forceinline__ double scaled_i64(long long acc, int e2)
{
    const unsigned long long u0 = acc < 0 ? 0ull - (unsigned long long)acc : (unsigned long long)acc;
    if (u0 == 0) return 0.0;
    const int lz = __clzll((long long)u0);
    const unsigned long long u = u0 << lz;
    const int be = 1023 + 63 - lz + e2;
    if (be < 1 || be > 2045) return ldexp((double)acc, e2);
    const unsigned long long r = (u >> 11) + ((u >> 10) & 1ull);
    const unsigned long long b = ((unsigned long long)(be - 1) << 52) + r + (acc < 0 ? 1ull << 63 : 0ull);
    return __longlong_as_double((long long)b);
}

// D (float32, tensor memory) (+)= A B^T for one digit of A: N may pass the 256 columns of one
// MMA instruction.
__device__ __forceinline__ void mma_digit(uint32_t d, uint32_t a, uint32_t lbo_a, uint32_t b, uint32_t lbo_b, int N,
                                          uint32_t acc)
{
    const uint64_t ad = sdesc_noswizzle(a, lbo_a, 128);
    const int n0 = N > 256 ? 256 : N;
    umma_bf16(d, ad, sdesc_noswizzle(b, lbo_b, 128), idesc_f16_f32(128, n0), acc);
    if (N > 256) umma_bf16(d + 256, ad, sdesc_noswizzle(b + 256 * 16, lbo_b, 128), idesc_f16_f32(128, N - 256), acc);
}

// ---------------------------------------------------------------------------- tables
enum { TAB_PROJECT = 0, TAB_CONTRACT = 1, TAB_EXPAND_TH = 2, TAB_EXPAND_PH = 3 };

struct TabParams {
    const double *Ith, *Iph, *Iphc, *dmu;
    uint8_t *tab;
    const unsigned long long *off;  // byte offset per set (pass, or order m)
    int *et;                        // column exponents, [set][et_ld]
    int kind, n_t, n_p, L, P, pass_cols, m0, et_ld;
};

// Sets of the theta contraction: order m = s, columns l = m .. m + 63, for s = 0 .. L; the
// columns past 64 of the orders that have them as sets L + 1 + m.
__host__ __device__ inline int set_order(int s, int L) { return s <= L ? s : s - L - 1; }
__host__ __device__ inline int set_col0(int s, int L) { return s <= L ? 0 : kNtMax; }
__host__ __device__ inline int set_cols(int s, int L)
{
    const int n = L + 1 - set_order(s, L) - set_col0(s, L);
    return n < kNtMax ? n : kNtMax;
}
__host__ __device__ inline int set_extra(int L) { return L + 1 > kNtMax ? L + 1 - kNtMax : 0; }

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
    case TAB_CONTRACT: {
        const int m = set_order(set, t.L);
        return t.Ith[(size_t)tri(m + set_col0(set, t.L) + n, m) * t.n_t + k];
    }
    case TAB_EXPAND_TH: return t.Ith[(size_t)tri(set + k, set) * t.n_t + n] / t.dmu[n];
    default: return t.Iphc[(size_t)k * t.n_p + n];
    }
}

// One warp per table column n of one set: its exponent, then its digits.  Contract tables are
// [K step]{[octet][7 Nt rows][8], row = digit Nt + n; for a column m = 0 of its own then
// [digit of A][octet][16 rows][8]}; expand tables are blocks of 32
// columns, [block][K step][octet][7 x 32][8].  Cells past K are never written (the tables
// start as zeros).
__global__ void __launch_bounds__(128) k64_digit_tables(const TabParams t, int n_sets)
{
    const int set = blockIdx.y, lane = threadIdx.x & 31;
    const bool own0 = t.kind == TAB_PROJECT && t.m0 && set == 0;
    const int n = blockIdx.x * 4 + (threadIdx.x >> 5) - (own0 ? 1 : 0);
    int N, K;
    switch (t.kind) {
    case TAB_PROJECT: N = pass_ncols(set, t.pass_cols, t.m0, t.P), K = t.n_p; break;
    case TAB_CONTRACT: N = set_cols(set, t.L), K = t.n_t; break;
    case TAB_EXPAND_TH: N = t.n_t, K = t.L + 1 - set; break;
    default: N = t.n_p, K = t.P; break;
    }
    if (n >= N) return;
    uint32_t mx = 0;
    for (int k = lane; k < K; k += 32) mx = max(mx, abs_hi(tab_value(t, set, n, k)));
    mx = __reduce_max_sync(0xFFFFFFFFu, mx);
    const int E = (int)(mx >> 20);
    if (lane == 0) t.et[(size_t)set * t.et_ld + (n < 0 ? kNtMax : n)] = E;
    if (E == 0) return;  // zeros
    const bool stacked = t.kind == TAB_PROJECT || t.kind == TAB_CONTRACT;
    const int nd = stacked ? ceil16(N) : kNtX, rows = kDig * nd;
    const size_t step = (size_t)(rows + (own0 ? kRows0 : 0)) * 32;
    const int steps = (K + 15) / 16;
    uint8_t *base = t.tab + t.off[set] + (stacked ? 0 : (size_t)(n / kNtX) * steps * step);
    const int nr = stacked ? n : n % kNtX;
    for (int k = lane; k < K; k += 32) {
        const double x = tab_value(t, set, n, k);
        const uint32_t hi = (uint32_t)__double2hiint(x);
        uint32_t wl, wh, d[kDig];
        fix55((uint32_t)__double2loint(x), hi, E + 9, wl, wh);
        if ((hi & 0x7FF00000u) == 0) wl = 0x80808080u, wh = 0x00008080u;  // zeros stay zeros
        digits2(wl, wh, hi, wl, wh, hi, d);
        uint8_t *dst = base + (size_t)(k >> 4) * step + (k & 7) * 2;
        const int oct = (k >> 3) & 1;
        if (n >= 0) {
#pragma unroll
            for (int i = 0; i < kDig; ++i)
                *reinterpret_cast<uint16_t *>(dst + (size_t)(oct * rows + i * nd + nr) * 16) = (uint16_t)(d[i] & 0xFFFFu);
        } else {
#pragma unroll
            for (int a = 0; a < kDig; ++a)
#pragma unroll
                for (int i = 0; i + a < kDig; ++i)
                    *reinterpret_cast<uint16_t *>(dst + (size_t)rows * 32 + (size_t)(a * 32 + oct * 16 + a + i) * 16) =
                        (uint16_t)(d[i] & 0xFFFFu);
        }
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
    int theta;                     // 0: (a1), 1: (a2)
    int n_r, n_t, n_p, L, KL, P, ldJ;
    int K, n_steps, n_chunks, ds;  // ds: low bits of the 72-bit sum dropped, so that K terms fit 63 bits
    int n_units, npass, pass_cols, m0, n_groups, n_groups0, et_ld;
    int ns_a, ns_b, nacc, slot_b, cols_max, vec;
    double scale;                  // (a2) 4 pi G
};

struct ContractUnit {
    int set, order, col0;  // pass or theta set; its order (theta) and first column
    int N, Nt, own0;       // columns, rounded up to 16; the column m = 0 in a block of its own
    long long row0;        // (a1) first row; (a2) first shell
    __device__ __forceinline__ uint32_t step_bytes() const { return (uint32_t)(kDig * Nt + (own0 ? kRows0 : 0)) * 32; }
};

__device__ __forceinline__ ContractUnit contract_unit(const ContractParams &p, int u)
{
    ContractUnit r;
    if (!p.theta) {
        const int tile = u / p.npass;
        r.set = u - tile * p.npass;
        r.order = 0;
        r.row0 = (long long)tile * 128;
        r.col0 = pass_col0(r.set, p.pass_cols, p.m0);
        r.N = pass_ncols(r.set, p.pass_cols, p.m0, p.P);
        r.own0 = p.m0 && r.set == 0;
    } else {
        // order 0 (rows are 128 shells), then the orders with cos and sin rows of 64 shells
        const int extra = set_extra(p.L), v0 = p.n_groups0 * (extra ? 2 : 1);
        if (u < v0) {
            r.set = u < p.n_groups0 ? 0 : p.L + 1;
            r.row0 = (long long)(u < p.n_groups0 ? u : u - p.n_groups0) * 128;
        } else {
            const int v = (u - v0) / p.n_groups;
            r.set = v < p.L ? 1 + v : p.L + 2 + (v - p.L);
            r.row0 = (long long)(u - v0 - v * p.n_groups) * 64;
        }
        r.order = set_order(r.set, p.L);
        r.col0 = r.order + set_col0(r.set, p.L);
        r.N = set_cols(r.set, p.L);
        r.own0 = 0;
    }
    r.Nt = ceil16(r.N);
    return r;
}

// Start of row `r` of a unit in the source (K contiguous values), or nullptr past the last row.
__device__ __forceinline__ const double *contract_row(const ContractParams &p, const ContractUnit &u, int r)
{
    if (!p.theta) {
        const long long row = u.row0 + r;
        return row < p.R ? p.src + row * p.n_p : nullptr;
    }
    const int i = (int)u.row0 + (u.order ? r >> 1 : r);
    const int col = u.order ? 2 * u.order - 1 + (r & 1) : 0;
    return i < p.n_r ? p.src + ((size_t)i * p.P + col) * p.ldJ : nullptr;
}

// Roles: warps 0-15 split A (each thread four neighbouring k of one row per K step, the whole
// chunk of 128 k in registers: its row maxima come from a shuffle over the row's four threads,
// and a step's registers take the next chunk's loads as soon as it is split, so 128 KB are in
// flight a CTA) and drain the accumulators between their steps; warp 16 owns tensor memory
// and issues the MMAs; warp 17 copies the table.
__global__ void __launch_bounds__(kThreads, 1) k64_contract_tc(const ContractParams prm)
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
            mbar_init(smem_u32(&a_empty[s]), 1);
        }
        for (int s = 0; s < prm.ns_b; ++s) {
            mbar_init(smem_u32(&b_full[s]), 1);
            mbar_init(smem_u32(&b_empty[s]), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&acc_full[b]), 1);
            mbar_init(smem_u32(&acc_empty[b]), kWorkWarps);
        }
        for (int b = 0; b < 4; ++b) mbar_init(smem_u32(&e_full[b]), kWorkWarps);
        mbar_init(smem_u32(drain_bar), 1);
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
    pdl_trigger();
    pdl_wait();  // the source comes from the previous kernels

    if (warp == kWorkWarps + 1) {
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
                    ok = mbar_wait(smem_u32(&b_empty[rb.idx]), rb.phase ^ 1, abort_flag, prm.err);
                    if (!ok) break;
                    const uint32_t bar = smem_u32(&b_full[rb.idx]);
                    mbar_arrive_expect_tx(bar, bytes);
                    bulk_load(smem_u32(sB + (size_t)rb.idx * prm.slot_b), src + (size_t)s * bytes, bytes, bar);
                    ++issued;
                }
            }
            drain_ring(b_full, rb, prm.ns_b, issued);
        }
    } else if (warp == kWorkWarps) {
        // ---------------- MMA issuer
        if (lane == 0) {
            Ring ra, rb;
            int it = 0;
            bool ok = true;
            for (int u = blockIdx.x; u < prm.n_units && ok; u += gridDim.x) {
                const ContractUnit un = contract_unit(prm, u);
                for (int c = 0; c < prm.n_chunks && ok; ++c, ++it) {
                    const int b = prm.nacc == 2 ? it & 1 : 0, nth = prm.nacc == 2 ? it >> 1 : it;
                    ok = mbar_wait(smem_u32(&acc_empty[b]), (nth & 1) ^ 1, abort_flag, prm.err);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t d0 = tmem_base + (uint32_t)b * acc_stride;
                    const int steps = min(kChunkSteps, prm.n_steps - c * kChunkSteps);
                    for (int s = 0; s < steps; ++s, ra.next(prm.ns_a), rb.next(prm.ns_b)) {
                        ok = mbar_wait(smem_u32(&b_full[rb.idx]), rb.phase, abort_flag, prm.err) &&
                             mbar_wait(smem_u32(&a_full[ra.idx]), ra.phase, abort_flag, prm.err);
                        if (!ok) break;
                        tc_fence_after();
                        const uint32_t a0 = smem_u32(sA + (size_t)ra.idx * kSlotA1);
                        const uint32_t b0 = smem_u32(sB + (size_t)rb.idx * prm.slot_b);
#pragma unroll
                        for (int i = 0; i < kDig; ++i)
                            mma_digit(d0 + (uint32_t)(i * un.Nt), a0 + i * kDigA1, kLboA1, b0, (uint32_t)un.Nt * kDig * 16,
                                      (kDig - i) * un.Nt, (s | i) != 0);
                        if (un.own0) {
#pragma unroll
                            for (int i = 0; i < kDig; ++i)
                                mma_digit(d0 + (uint32_t)(kDig * un.Nt), a0 + i * kDigA1, kLboA1,
                                          b0 + (uint32_t)un.Nt * kDig * 32 + i * 512, 256, 16, (s | i) != 0);
                        }
                        umma_commit(smem_u32(&a_empty[ra.idx]));
                        umma_commit(smem_u32(&b_empty[rb.idx]));
                    }
                    if (ok) umma_commit(smem_u32(&acc_full[b]));
                }
            }
            umma_commit(smem_u32(drain_bar));
            const long long t0 = clock64();
            while (!mbar_try_wait(smem_u32(drain_bar), 0) && clock64() - t0 < MP_WAIT_BUDGET_CYCLES) {
            }
        }
    } else {
        // ---------------- split + drain
        const int crow = 8 * warp + (lane >> 2), quad = lane & 3;  // split: row, k = 16 step + 4 quad + 0..3
        const int q4 = warp & 3, grp = warp >> 2;                  // drain: lane quarter, column group
        const uint32_t a_off = (uint32_t)((quad >> 1) * kLboA1 + crow * 16 + (quad & 1) * 8);
        double v[kChunkSteps][4];
        bool ok = true, bad = false;

        auto load_step = [&](const double *row, int step, double (&x)[4]) {
            const int k = 16 * step + 4 * quad;
#pragma unroll
            for (int e = 0; e < 4; ++e) x[e] = 0.0;
            if (row) {
                if (prm.vec) {
                    if (k < prm.K) {
                        const double2 t = __ldg(reinterpret_cast<const double2 *>(row + k));
                        x[0] = t.x, x[1] = t.y;
                    }
                    if (k + 2 < prm.K) {
                        const double2 t = __ldg(reinterpret_cast<const double2 *>(row + k + 2));
                        x[2] = t.x, x[3] = t.y;
                    }
                } else {
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if (k + e < prm.K) x[e] = __ldg(row + k + e);
                }
            }
        };

        // the accumulators of item `it` (unit un, chunk c) into the row's running sums, after
        // the last chunk to memory; Er: the running exponent of this thread's row
        int Er = 0;
        auto drain = [&](const ContractUnit &un, int c, int it) -> bool {
            const int b = prm.nacc == 2 ? it & 1 : 0, nth = prm.nacc == 2 ? it >> 1 : it;
            // the row exponents of this item are written, its MMAs complete
            if (!warp_all(mbar_wait(smem_u32(&e_full[it & 3]), (it >> 2) & 1, abort_flag, prm.err) &&
                          mbar_wait(smem_u32(&acc_full[b]), nth & 1, abort_flag, prm.err)))
                return false;
            tc_fence_after();
            const int row = 32 * q4 + lane;
            const bool last = c == prm.n_chunks - 1;
            const int Ec = sE[(it & 3) * 128 + row];
            // running sums are kept at the largest exponent of the row's chunks so far
            int sh_old = 0, sh_new = 0;
            if (c == 0) {
                Er = Ec;
            } else {
                const int En = max(Er, Ec);
                sh_old = min(63, En - Er);
                sh_new = min(63, En - Ec);
                Er = En;
            }
            double *dst = nullptr;  // column n of the unit: dst + n ldJ, or dst + (col0 + n)^2
            if (!prm.theta) {
                const long long r = un.row0 + row;
                if (r < prm.R) {
                    const int i = (int)(r / prm.n_t), j = (int)(r - (long long)i * prm.n_t);
                    dst = prm.dst + ((size_t)i * prm.P + un.col0) * prm.ldJ + j;
                }
            } else {
                const int i = (int)un.row0 + (un.order ? row >> 1 : row);
                if (i < prm.n_r) dst = prm.dst + (size_t)i * prm.KL + (un.order ? 2 * un.order - 1 + (row & 1) : 0);
            }
            const uint32_t col = tmem_base + (uint32_t)b * acc_stride + ((uint32_t)(q4 * 32) << 16);
            // groups of four columns, dealt to the four warps of a lane quarter; the column m = 0
            // of its own block (its seven weights side by side) comes last, as column N
            const int n_cols = un.N + un.own0;
            for (int n = 4 * grp; n < n_cols; n += 16) {
                uint32_t t[kDig][4];
                const bool own = n + 3 >= un.N && un.own0;  // N is a multiple of 16 then: n = N
                if (!own) {
#pragma unroll
                    for (int i = 0; i < kDig; ++i) tmem_ld4(col + (uint32_t)(i * un.Nt + n), t[i]);
                } else {
                    uint32_t w[4];
                    tmem_ld4(col + (uint32_t)(kDig * un.Nt), w);
                    tmem_ld4(col + (uint32_t)(kDig * un.Nt + 4), t[4]);
                    tmem_ld_wait();
                    t[6][0] = t[4][2];
                    t[5][0] = t[4][1];
                    t[0][0] = w[0];
                    t[1][0] = w[1];
                    t[2][0] = w[2];
                    t[3][0] = w[3];
                }
                tmem_ld_wait();
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    if (n + e >= n_cols) break;
                    int a[kDig];
#pragma unroll
                    for (int i = 0; i < kDig; ++i) a[i] = __float2int_rn(__uint_as_float(t[i][e]));
                    const long long hi = (long long)a[0] * 65536 + ((long long)a[1] * 256 + a[2]);
                    const long long lo = (long long)a[3] * 16777216 + (long long)a[4] * 65536 +
                                         ((long long)a[5] * 256 + a[6]);
                    long long s = (hi << (32 - prm.ds)) + ((lo + (1ll << (prm.ds - 1))) >> prm.ds);
                    if (prm.n_chunks > 1) {
                        long long *pa = sAcc + (size_t)(n + e) * 128 + row;
                        s >>= sh_new;
                        if (c > 0) s += *pa >> sh_old;
                        if (!last) *pa = s;
                    }
                    if (last && dst) {
                        const int Et = __ldg(prm.et + (size_t)un.set * prm.et_ld + (own ? kNtMax : n + e));
                        const double x = Er >= kExpNan ? __longlong_as_double(0x7FF8000000000000ll)
                                                       : scaled_i64(s, 48 + prm.ds + Er + Et - 2154);
                        if (prm.theta)
                            dst[(size_t)(un.col0 + n + e) * (un.col0 + n + e)] = prm.scale * x;
                        else
                            dst[own ? -(long long)un.col0 * prm.ldJ : (long long)(n + e) * prm.ldJ] = x;
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&acc_empty[b]));
            return true;
        };

        Ring ra;
        int it = 0, pend_c = 0;
        bool pend = false;
        ContractUnit un{}, pend_u{};
        const double *row = nullptr;
        int u = blockIdx.x;
        if (u < prm.n_units) {
            un = contract_unit(prm, u);
            row = contract_row(prm, un, crow);
#pragma unroll
            for (int s = 0; s < kChunkSteps; ++s) load_step(row, s, v[s]);
        }
        int c = 0;
        while (u < prm.n_units && ok) {
            const int steps = min(kChunkSteps, prm.n_steps - c * kChunkSteps);
            // the item after this one, whose loads follow the splitting of this one's registers
            int u2 = u, c2 = c + 1;
            ContractUnit un2 = un;
            const double *row2 = row;
            if (c2 == prm.n_chunks) {
                c2 = 0;
                u2 = u + (int)gridDim.x;
                row2 = nullptr;
                if (u2 < prm.n_units) {
                    un2 = contract_unit(prm, u2);
                    row2 = contract_row(prm, un2, crow);
                }
            }
            uint32_t mx = 0;
#pragma unroll
            for (int s = 0; s < kChunkSteps; ++s)
#pragma unroll
                for (int e = 0; e < 4; ++e) mx = max(mx, abs_hi(v[s][e]));
            mx = max(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, 1));
            mx = max(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, 2));
            int E = (int)(mx >> 20), E0 = 0;
            bad |= E >= kExpNan;
            if (E < 128) {  // next to the bottom of the float64 range: scaled up exactly
                E = max(128, (int)(abs_hi(__hiloint2double((int)mx, -1) * 0x1p300) >> 20));
                E0 = -300;
            }
            // four exponent buffers: a warp splits at most two items ahead of another one's drain
            if (quad == 0) sE[(it & 3) * 128 + crow] = E + E0;
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&e_full[it & 3]));
            const int e9 = E + 9;
#pragma unroll
            for (int s = 0; s < kChunkSteps; ++s) {
                if (s < steps && ok) {
                    if (s == 2 && pend) {
                        ok = drain(pend_u, pend_c, it - 1);
                        pend = false;
                    }
                    if (ok) ok = warp_all(mbar_wait(smem_u32(&a_empty[ra.idx]), ra.phase ^ 1, abort_flag, prm.err));
                    if (ok) {
                        uint8_t *dst = sA + (size_t)ra.idx * kSlotA1 + a_off;
                        uint32_t wl[4], wh[4], d0[kDig], d1[kDig];
                        if (E0) {
#pragma unroll
                            for (int e = 0; e < 4; ++e) v[s][e] *= 0x1p300;
                        }
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            fix55((uint32_t)__double2loint(v[s][e]), (uint32_t)__double2hiint(v[s][e]), e9, wl[e],
                                  wh[e]);
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
                }
                load_step(row2, c2 * kChunkSteps + s, v[s]);
            }
            if (!ok) break;
            if (pend) ok = drain(pend_u, pend_c, it - 1);
            pend = true;
            pend_u = un;
            pend_c = c;
            ++it;
            u = u2;
            c = c2;
            un = un2;
            row = row2;
        }
        if (ok && pend) drain(pend_u, pend_c, it - 1);
        if (bad && !prm.theta) atomicOr(prm.err, DEV_ERR_NONFINITE);
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
    int theta;                    // 1: (d1), 0: (d2)
    int n_r, n_t, n_p, L, P, ldJ, ldI;
    int N, n_blk, n_units, n_split, n_groups, n_groups0, et_ld;
    int a_steps, ns_b, vec;       // a_steps: K steps of A held at once
};

struct ExpandUnit {
    int set, K, steps, n_chunks, chunk_steps, blk0, blk1;
    long long row0;
};

__device__ __forceinline__ ExpandUnit expand_unit(const ExpandParams &p, int u)
{
    ExpandUnit r;
    if (!p.theta) {
        const int tile = u / p.n_split, part = u - tile * p.n_split;
        r.set = 0;
        r.K = p.P;
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
    r.steps = (r.K + 15) / 16;
    r.n_chunks = r.steps <= p.a_steps ? 1 : 2;
    r.chunk_steps = (r.steps + r.n_chunks - 1) / r.n_chunks;
    return r;
}

// Roles: warps 0-15 split the unit's A (128 rows, the whole K or, past a_steps, half of it at a
// time) and turn finished blocks into float64; warp 16 owns tensor memory and issues the MMAs of
// one block of 32 columns while the other block's accumulators are drained; warp 17 copies the
// table.  With K in one piece A is split once per unit; in two it is split again for every pair
// of blocks.
__global__ void __launch_bounds__(kThreads, 1) k64_expand_tc(const ExpandParams prm)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127));
    constexpr uint32_t kSlotB = kRowsX * 32;
    uint8_t *sA = smem;
    uint8_t *sB = sA + (size_t)prm.a_steps * kStepA2;
    uint8_t *sOut = sB + (size_t)prm.ns_b * kSlotB;                   // [16 warps][32 rows][8] float64
    uint32_t *sMax = reinterpret_cast<uint32_t *>(sOut + kWorkWarps * 2048);  // [2 units][4][128]
    uint64_t *bars = reinterpret_cast<uint64_t *>(sMax + 8 * 128);
    uint64_t *b_full = bars, *b_empty = b_full + prm.ns_b;
    uint64_t *a_full = b_empty + prm.ns_b, *a_free = a_full + 1;
    uint64_t *acc_full = a_free + 1, *acc_empty = acc_full + 2, *m_full = acc_empty + 2, *drain_bar = m_full + 1;
    uint32_t *tmem_holder = reinterpret_cast<uint32_t *>(drain_bar + 1);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_holder + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < prm.ns_b; ++s) {
            mbar_init(smem_u32(&b_full[s]), 1);
            mbar_init(smem_u32(&b_empty[s]), 1);
        }
        mbar_init(smem_u32(a_full), kWorkWarps);
        mbar_init(smem_u32(a_free), 1);
        mbar_init(smem_u32(m_full), kWorkWarps);
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&acc_full[b]), 1);
            mbar_init(smem_u32(&acc_empty[b]), kWorkWarps);
        }
        mbar_init(smem_u32(drain_bar), 1);
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
    pdl_trigger();
    pdl_wait();  // the source comes from the previous kernels

    if (warp == kWorkWarps + 1) {
        // ---------------- table producer
        if (lane == 0) {
            Ring rb;
            int issued = 0;
            bool ok = true;
            for (int u = blockIdx.x; u < prm.n_units && ok; u += gridDim.x) {
                const ExpandUnit un = expand_unit(prm, u);
                const uint8_t *src = prm.tab + prm.off[un.set];
                for (int g = un.blk0; g < un.blk1 && ok; g += 2)
                    for (int ch = 0; ch < un.n_chunks && ok; ++ch)
                        for (int nb = g; nb < min(g + 2, un.blk1) && ok; ++nb)
                            for (int s = ch * un.chunk_steps; s < min(un.steps, (ch + 1) * un.chunk_steps);
                                 ++s, rb.next(prm.ns_b)) {
                                ok = mbar_wait(smem_u32(&b_empty[rb.idx]), rb.phase ^ 1, abort_flag, prm.err);
                                if (!ok) break;
                                const uint32_t bar = smem_u32(&b_full[rb.idx]);
                                mbar_arrive_expect_tx(bar, kSlotB);
                                bulk_load(smem_u32(sB + (size_t)rb.idx * kSlotB),
                                          src + ((size_t)nb * un.steps + s) * kSlotB, kSlotB, bar);
                                ++issued;
                            }
            }
            drain_ring(b_full, rb, prm.ns_b, issued);
        }
    } else if (warp == kWorkWarps) {
        // ---------------- MMA issuer
        if (lane == 0) {
            Ring rb;
            int blk = 0, conv = 0;  // blocks and splits of A so far
            bool ok = true;
            for (int u = blockIdx.x; u < prm.n_units && ok; u += gridDim.x) {
                const ExpandUnit un = expand_unit(prm, u);
                for (int g = un.blk0; g < un.blk1 && ok; g += 2) {
                    const int nbs = min(2, un.blk1 - g);
                    for (int ch = 0; ch < un.n_chunks && ok; ++ch) {
                        if (un.n_chunks > 1 || g == un.blk0) {
                            ok = mbar_wait(smem_u32(a_full), conv & 1, abort_flag, prm.err);
                            if (!ok) break;
                            ++conv;
                        }
                        const int s0 = ch * un.chunk_steps, s1 = min(un.steps, s0 + un.chunk_steps);
                        for (int nb = 0; nb < nbs && ok; ++nb) {
                            const int b = (blk + nb) & 1;
                            if (ch == 0) ok = mbar_wait(smem_u32(&acc_empty[b]), (((blk + nb) >> 1) & 1) ^ 1, abort_flag, prm.err);
                            if (!ok) break;
                            tc_fence_after();
                            const uint32_t d0 = tmem_base + (uint32_t)b * 256;
                            for (int s = s0; s < s1; ++s, rb.next(prm.ns_b)) {
                                ok = mbar_wait(smem_u32(&b_full[rb.idx]), rb.phase, abort_flag, prm.err);
                                if (!ok) break;
                                tc_fence_after();
                                const uint32_t a0 = smem_u32(sA + (size_t)(s - s0) * kStepA2);
                                const uint32_t b0 = smem_u32(sB + (size_t)rb.idx * kSlotB);
#pragma unroll
                                for (int i = 0; i < kDig; ++i)
                                    umma_bf16(d0 + (uint32_t)(i * kNtX), sdesc_noswizzle(a0 + i * kDigA2, kLboA2, 128),
                                              sdesc_noswizzle(b0, kRowsX * 16, 128),
                                              idesc_f16_f32(128, (kDig - i) * kNtX), (s | i) != 0);
                                umma_commit(smem_u32(&b_empty[rb.idx]));
                            }
                            if (ok && ch == un.n_chunks - 1) umma_commit(smem_u32(&acc_full[b]));
                        }
                        if (ok && un.n_chunks > 1) umma_commit(smem_u32(a_free));
                    }
                    blk += nbs;
                }
            }
            umma_commit(smem_u32(drain_bar));
            const long long t0 = clock64();
            while (!mbar_try_wait(smem_u32(drain_bar), 0) && clock64() - t0 < MP_WAIT_BUDGET_CYCLES) {
            }
        }
    } else {
        // ---------------- split + drain
        const int crow = threadIdx.x & 127, cg = threadIdx.x >> 7;  // split: row, octets cg, cg + 4, ...
        const int q4 = warp & 3, grp = warp >> 2;                   // drain: lane quarter, 8-column group
        uint8_t *stage = sOut + warp * 2048;
        bool ok = true;
        int blk = 0, freed = 0, lu = 0;
        int Erow = 0;  // exponent of drain row 32 q4 + lane (= crow's when cg = grp: the same thread)

        for (int u = blockIdx.x; u < prm.n_units && ok; u += gridDim.x, ++lu) {
            const ExpandUnit un = expand_unit(prm, u);
            // element k of this thread's row: src + base + (PH: k ldJ; TH: ((m + k)^2 + p) ldI)
            const double *base = nullptr;
            if (!prm.theta) {
                const long long r = un.row0 + crow;
                if (r < prm.R) {
                    const int i = (int)(r / prm.n_t), j = (int)(r - (long long)i * prm.n_t);
                    base = prm.src + (size_t)i * prm.P * prm.ldJ + j;
                }
            } else {
                const int a = un.set ? crow >> 6 : 0, i = (int)un.row0 + (un.set ? crow & 63 : crow);
                if (i < prm.n_r) base = prm.src + (size_t)(un.set ? 2 * un.set - 1 + a : 0) * prm.ldI + i;
            }
            auto element = [&](int k) -> double {
                if (!base || k >= un.K) return 0.0;
                return !prm.theta ? __ldg(base + (size_t)k * prm.ldJ)
                                  : __ldg(base + (size_t)(un.set + k) * (un.set + k) * prm.ldI);
            };
            uint32_t mx = 0;
            for (int o = cg; o < 2 * un.steps; o += 4) {
                double x[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) x[e] = element(8 * o + e);
#pragma unroll
                for (int e = 0; e < 8; ++e) mx = max(mx, abs_hi(x[e]));
            }
            uint32_t *row_max = sMax + (lu & 1) * 512 + crow;
            row_max[cg * 128] = mx;
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(m_full));
            ok = warp_all(mbar_wait(smem_u32(m_full), lu & 1, abort_flag, prm.err));
            if (!ok) break;
            mx = max(max(row_max[0], row_max[128]), max(row_max[256], row_max[384]));
            int E = (int)(mx >> 20), E0 = 0;
            double up = 1.0;
            if (E < 128) {  // next to the bottom of the float64 range: scaled up exactly
                up = 0x1p300;
                E = max(128, (int)(abs_hi(__hiloint2double((int)mx, -1) * up) >> 20));
                E0 = -300;
            }
            Erow = E + E0;
            const int e9 = E + 9;

            auto split = [&](int ch) {
                const int s0 = ch * un.chunk_steps, s1 = min(un.steps, s0 + un.chunk_steps);
                for (int o = 2 * s0 + cg; o < 2 * s1; o += 4) {
                    double x[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) x[e] = element(8 * o + e);
                    if (E0) {
#pragma unroll
                        for (int e = 0; e < 8; ++e) x[e] *= up;
                    }
                    uint32_t d[4][kDig];
#pragma unroll
                    for (int e = 0; e < 8; e += 2) {
                        uint32_t wl0, wh0, wl1, wh1;
                        const uint32_t h0 = (uint32_t)__double2hiint(x[e]), h1 = (uint32_t)__double2hiint(x[e + 1]);
                        fix55((uint32_t)__double2loint(x[e]), h0, e9, wl0, wh0);
                        fix55((uint32_t)__double2loint(x[e + 1]), h1, e9, wl1, wh1);
                        digits2(wl0, wh0, h0, wl1, wh1, h1, d[e >> 1]);
                    }
                    uint8_t *dst = sA + (size_t)((o >> 1) - s0) * kStepA2 + (o & 1) * kLboA2 + crow * 16;
#pragma unroll
                    for (int i = 0; i < kDig; ++i)
                        *reinterpret_cast<uint4 *>(dst + i * kDigA2) = make_uint4(d[0][i], d[1][i], d[2][i], d[3][i]);
                }
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(a_full));
            };

            // with K in one piece A is free here: every block of the last unit has been drained
            if (un.n_chunks == 1) split(0);
            for (int g = un.blk0; g < un.blk1 && ok; g += 2) {
                const int nbs = min(2, un.blk1 - g);
                if (un.n_chunks > 1)
                    for (int ch = 0; ch < un.n_chunks && ok; ++ch) {
                        if (ch > 0) {
                            ok = warp_all(mbar_wait(smem_u32(a_free), freed & 1, abort_flag, prm.err));
                            ++freed;
                        }
                        if (ok) split(ch);
                    }
                for (int nb = 0; nb < nbs && ok; ++nb, ++blk) {
                    const int b = blk & 1;
                    ok = warp_all(mbar_wait(smem_u32(&acc_full[b]), (blk >> 1) & 1, abort_flag, prm.err));
                    if (!ok) break;
                    tc_fence_after();
                    uint32_t t[kDig][8];
                    const uint32_t col = tmem_base + (uint32_t)b * 256 + ((uint32_t)(q4 * 32) << 16) + grp * 8;
#pragma unroll
                    for (int i = 0; i < kDig; ++i) tmem_ld8(col + (uint32_t)(i * kNtX), t[i]);
                    tmem_ld_wait();
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&acc_empty[b]));
                    const int n0 = (g + nb) * kNtX + grp * 8;
                    // rows of 64 bytes in 16-byte pieces, the pieces permuted so that neither the
                    // stores (one row a lane) nor the loads (four lanes a row) share a bank
                    double out[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        // the two lightest accumulators as one number (2^-56 of the row and column
                        // maxima below the rounding); the others are exact integers
                        const float t56 = fmaf(__uint_as_float(t[6][e]), 0.00390625f, __uint_as_float(t[5][e]));
                        int a[6];
#pragma unroll
                        for (int i = 0; i < 5; ++i) a[i] = __float2int_rn(__uint_as_float(t[i][e]));
                        a[5] = __float2int_rn(t56);
                        const long long hi = (long long)(a[0] * 256 + a[1]) << 32;
                        const long long lo = ((long long)a[2] * 256 + a[3]) * 65536 + ((long long)a[4] * 256 + a[5]);
                        const int n = n0 + e;
                        const int Et = n < prm.N ? __ldg(prm.et + (size_t)un.set * prm.et_ld + n) : 0;
                        out[e] = Erow >= kExpNan ? __longlong_as_double(0x7FF8000000000000ll)
                                                 : scaled_i64(hi + lo, 56 + Erow + Et - 2154);
                    }
#pragma unroll
                    for (int cpc = 0; cpc < 4; ++cpc)
                        *reinterpret_cast<double2 *>(stage + lane * 64 + ((cpc ^ ((lane >> 1) & 3)) << 4)) =
                            make_double2(out[2 * cpc], out[2 * cpc + 1]);
                    __syncwarp();
#pragma unroll
                    for (int r8 = 0; r8 < 4; ++r8) {
                        const int rr = 8 * r8 + (lane >> 2), cpc = lane & 3, n = n0 + 2 * cpc;
                        const double2 x =
                            *reinterpret_cast<const double2 *>(stage + rr * 64 + ((cpc ^ ((rr >> 1) & 3)) << 4));
                        const int row = 32 * q4 + rr;
                        double *dst = nullptr;
                        if (!prm.theta) {
                            if (un.row0 + row < prm.R) dst = prm.dst + (un.row0 + row) * prm.n_p;
                        } else {
                            const int a = un.set ? row >> 6 : 0, i = (int)un.row0 + (un.set ? row & 63 : row);
                            if (i < prm.n_r)
                                dst = prm.dst + ((size_t)i * prm.P + (un.set ? 2 * un.set - 1 + a : 0)) * prm.ldJ;
                        }
                        if (dst) {
                            if (prm.vec && n + 1 < prm.N) {
                                if (prm.theta)
                                    *reinterpret_cast<double2 *>(dst + n) = x;  // read again by the next step
                                else
                                    __stcs(reinterpret_cast<double2 *>(dst + n), x);
                            } else {
                                if (n < prm.N) dst[n] = x.x;
                                if (n + 1 < prm.N) dst[n + 1] = x.y;
                            }
                        }
                    }
                    __syncwarp();
                }
                // the pair's accumulators have been read, so both splits' MMAs are complete
                if (un.n_chunks > 1 && ok) {
                    ok = warp_all(mbar_wait(smem_u32(a_free), freed & 1, abort_flag, prm.err));
                    ++freed;
                }
            }
        }
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
    const int Nt = ceil16(N);
    c.n_steps = (K + 15) / 16;
    c.n_chunks = (c.n_steps + kChunkSteps - 1) / kChunkSteps;
    c.ds = std::max(1, ceil_log2(K));
    c.cols_max = N + own0;
    c.nacc = kDig * Nt + (own0 ? 16 : 0) <= 256 ? 2 : 1;
    c.slot_b = (kDig * Nt + (own0 ? kRows0 : 0)) * 32;
    if (Nt > kNtMax || c.ds > 31) return false;
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
    const int steps = (K + 15) / 16;
    x.a_steps = steps <= 6 ? steps : (steps + 1) / 2;
    const int fixed = x.a_steps * kStepA2 + kWorkWarps * 2048 + 8 * 128 * 4 + 512;
    for (x.ns_b = 6; x.ns_b >= 2; --x.ns_b) {
        x.smem = fixed + x.ns_b * kRowsX * 32;
        if (x.smem <= kSmemMax) return true;
    }
    return false;
}

size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

}  // namespace

bool plan_fp64_tc(mp_mesh *m)
{
    Fp64Plan &f = m->fp;
    f = Fp64Plan();
    f.ldJ = round_up(m->n_t, 4);
    f.ldI = round_up(m->n_r, 4);
    // columns per pass over the density; the column m = 0 gets a block of its own where the
    // others fill blocks of 16 without it
    f.m0 = m->L > 0 && m->L % 8 == 0;
    const int cols = m->P - f.m0;
    f.npass = (cols + kNtMax - 1) / kNtMax;
    f.pass_cols = (cols + f.npass - 1) / f.npass;
    if (f.npass > 1) f.pass_cols = std::min(kNtMax, ceil16(f.pass_cols));
    if (m->L > 71 || !plan_contract(m->n_t, std::min(m->L + 1, kNtMax), 0, f.th_c) || !plan_expand(m->L + 1, f.th_x)) {
        f = Fp64Plan();  // the CUDA-core path and its layouts
        return false;
    }
    // below 16 azimuthal cells (axisymmetric meshes have one) a 16-wide K step is mostly padding
    // and the sums are short: CUDA cores
    f.phi_on = m->n_p >= 16 && plan_contract(m->n_p, f.pass_cols, f.m0, f.ph_c) && plan_expand(m->P, f.ph_x);
    f.on = 1;
    return true;
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
    const int n_sets = L + 1 + set_extra(L);
    f.off_ld = n_sets + 1;
    f.h_off.assign((size_t)4 * f.off_ld, 0);
    unsigned long long *oc = f.h_off.data(), *ox = oc + f.off_ld, *op = ox + f.off_ld;
    unsigned long long c = 0, x = 0;
    const int n_blk = (m->n_t + kNtX - 1) / kNtX;
    for (int s = 0; s < n_sets; ++s) {
        oc[s] = c;
        c += (unsigned long long)f.th_c.n_steps * kDig * ceil16(set_cols(s, L)) * 32;
    }
    for (int mm = 0; mm <= L; ++mm) {
        ox[mm] = x;
        x += (unsigned long long)n_blk * ((L + 1 - mm + 15) / 16) * kRowsX * 32;
    }
    const unsigned long long pstep = (unsigned long long)f.ph_c.n_steps * f.ph_c.slot_b;
    for (int s = 0; s < f.npass; ++s) op[s] = s * pstep;
    f.o_tab_c = take(c);
    f.o_tab_x = take(x);
    f.o_tab_pc = take(f.phi_on ? f.npass * pstep : 0);
    f.o_tab_px = take(f.phi_on ? (size_t)((m->n_p + kNtX - 1) / kNtX) * ((m->P + 15) / 16) * kRowsX * 32 : 0);
    f.o_off = take(f.h_off.size() * sizeof(unsigned long long));
    f.o_et_c = take((size_t)n_sets * (kNtMax + 1) * 4);
    f.o_et_x = take((size_t)(L + 1) * m->n_t * 4);
    f.o_et_pc = take((size_t)f.npass * (kNtMax + 1) * 4);
    f.o_et_px = take((size_t)m->n_p * 4);
    return at;
}

static const unsigned long long *fp64_off(const mp_mesh *m, int which)
{
    return reinterpret_cast<const unsigned long long *>(m->fp.arena + m->fp.o_off) + (size_t)which * m->fp.off_ld;
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
                    reinterpret_cast<int *>(f.arena + et), kind, m->n_t, m->n_p, L, m->P, f.pass_cols, f.m0, et_ld};
        k64_digit_tables<<<dim3((n_max + 3) / 4, n_sets), 128, 0, m->stream>>>(t, n_sets);
    };
    build(TAB_CONTRACT, f.o_tab_c, 0, f.o_et_c, kNtMax + 1, std::min(L + 1, kNtMax), L + 1 + set_extra(L));
    build(TAB_EXPAND_TH, f.o_tab_x, 1, f.o_et_x, m->n_t, m->n_t, L + 1);
    if (f.phi_on) {
        build(TAB_PROJECT, f.o_tab_pc, 2, f.o_et_pc, kNtMax + 1, f.pass_cols + f.m0, f.npass);
        build(TAB_EXPAND_PH, f.o_tab_px, 3, f.o_et_px, m->n_p, m->n_p, 1);
    }
    // 227 KB of dynamic shared memory for the kernels of this file (per device)
    e = cudaFuncSetAttribute(k64_contract_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k64_expand_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

static cudaError_t launch_contract(mp_mesh *m, int theta, const double *src, double *dst, const char *name)
{
    const Fp64Plan &f = m->fp;
    const Fp64Contract &c = theta ? f.th_c : f.ph_c;
    ContractParams p{};
    p.src = src;
    p.dst = dst;
    p.tab = f.arena + (theta ? f.o_tab_c : f.o_tab_pc);
    p.off = fp64_off(m, theta ? 0 : 2);
    p.et = reinterpret_cast<const int *>(f.arena + (theta ? f.o_et_c : f.o_et_pc));
    p.err = m->d_err;
    p.R = m->R;
    p.theta = theta;
    p.n_r = m->n_r, p.n_t = m->n_t, p.n_p = m->n_p, p.L = m->L, p.KL = m->KL, p.P = m->P, p.ldJ = f.ldJ;
    p.K = theta ? m->n_t : m->n_p;
    p.n_steps = c.n_steps, p.n_chunks = c.n_chunks, p.ds = c.ds;
    p.npass = f.npass, p.pass_cols = f.pass_cols, p.m0 = f.m0;
    p.n_groups = (m->n_r + 63) / 64, p.n_groups0 = (m->n_r + 127) / 128;
    const int extra = set_extra(m->L);
    p.n_units = theta ? p.n_groups0 * (extra ? 2 : 1) + (m->L + std::max(0, extra - 1)) * p.n_groups : (int)((m->R + 127) / 128) * f.npass;
    p.et_ld = kNtMax + 1;
    p.ns_a = c.ns_a, p.ns_b = c.ns_b, p.nacc = c.nacc, p.slot_b = c.slot_b, p.cols_max = c.cols_max;
    p.scale = 12.566370614359172954 * m->G;
    // 16-byte loads where every row starts on a 16-byte boundary (and K is even)
    p.vec = theta ? (m->n_t % 2 == 0) : (m->n_p % 2 == 0 && (reinterpret_cast<uintptr_t>(src) & 15) == 0);
    cudaEvent_t ev;
    prof_begin(m, name, &ev);
    cudaError_t e = launch_pdl(k64_contract_tc, dim3(std::min(p.n_units, m->num_sms)), dim3(kThreads), c.smem,
                               m->stream, p);
    prof_end(m, name, ev);
    return e != cudaSuccess ? e : cudaGetLastError();
}

static cudaError_t launch_expand(mp_mesh *m, int theta, const double *src, double *dst, const char *name)
{
    const Fp64Plan &f = m->fp;
    const Fp64Expand &x = theta ? f.th_x : f.ph_x;
    ExpandParams p{};
    p.src = src;
    p.dst = dst;
    p.tab = f.arena + (theta ? f.o_tab_x : f.o_tab_px);
    p.off = fp64_off(m, theta ? 1 : 3);
    p.et = reinterpret_cast<const int *>(f.arena + (theta ? f.o_et_x : f.o_et_px));
    p.err = m->d_err;
    p.R = m->R;
    p.theta = theta;
    p.n_r = m->n_r, p.n_t = m->n_t, p.n_p = m->n_p, p.L = m->L, p.P = m->P, p.ldJ = f.ldJ, p.ldI = f.ldI;
    p.N = theta ? m->n_t : m->n_p;
    p.n_blk = (p.N + kNtX - 1) / kNtX;
    p.n_groups = (m->n_r + 63) / 64, p.n_groups0 = (m->n_r + 127) / 128;
    p.et_ld = theta ? m->n_t : m->n_p;
    p.a_steps = x.a_steps, p.ns_b = x.ns_b;
    const int tiles = (int)((m->R + 127) / 128), pairs = (p.n_blk + 1) / 2;
    // fewer tiles than SMs: a tile's columns go to several CTAs (each splits the tile's A)
    p.n_split = theta ? 1 : std::max(1, std::min(pairs, m->num_sms / std::max(1, tiles)));
    p.n_units = theta ? p.n_groups0 + m->L * p.n_groups : tiles * p.n_split;
    p.vec = theta || (m->n_p % 2 == 0 && (reinterpret_cast<uintptr_t>(dst) & 15) == 0);
    cudaEvent_t ev;
    prof_begin(m, name, &ev);
    cudaError_t e = launch_pdl(k64_expand_tc, dim3(std::min(p.n_units, m->num_sms)), dim3(kThreads), x.smem,
                               m->stream, p);
    prof_end(m, name, ev);
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_fp64_tc_project(mp_mesh *m, const double *rho)
{
    return launch_contract(m, 0, rho, m->d_F64, "fp64_phi_project");
}
cudaError_t launch_fp64_tc_theta(mp_mesh *m)
{
    return launch_contract(m, 1, m->d_F64, m->d_A, "fp64_theta_contract");
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
