// mp_gravity.cu -- gravitational source terms of the fluid balance equations
// (GenASiS II, Sec. 3, Eq. (BalancedVariablesGravitational)) from a potential
// on the solver's mesh:
//
//   grad[a] = d(Phi)/dx^a   (x = r, theta, phi; coordinate derivatives)
//   S[a]    = -rho grad[a]  (momentum source, covariant components)
//   E       = -rho v^a grad[a]  (energy source; v contravariant)
//
// Each derivative is the simplest centred difference, over the two nearest
// cells along the coordinate (the rule the paper states with the sources):
// (Phi[hi] - Phi[lo]) / (x_c[hi] - x_c[lo]) with cell centres at coordinate
// midpoints.  phi wraps around when the azimuthal edges span 2 pi; at the ends
// of r, theta (and of a shorter azimuthal range) the two nearest cells are the
// cell itself and its one neighbour.  A single cell along a coordinate, or two
// azimuthal cells on a full circle, give a zero derivative.
//
// One block per (shell, polar cell) row, threads along phi (rows of fewer than 32 cells:
// one thread per cell over the flattened mesh).  The potential is
// read through the cache (each value serves the six neighbouring differences:
// rows j +- 1 and shells i +- 1 are read by nearby blocks while they are still
// in L2); density, velocity and the outputs stream once (evict-first).  All
// arithmetic is to float64 accuracy: the differences and their scalings in integers where that is
// exact work (scaled_difference), the rest on the float64 pipe.
#include <cmath>
#include <cstring>

#include "mp_internal.h"
#include "ptx.cuh"

namespace mp {

namespace {

// (a - b) w in integer instructions where that is exact work: a and b of one sign and within 2^9
// of each other, as neighbouring cells of a potential are, subtract exactly as 62-bit integers;
// the difference is normalised, multiplied by w's significand (64 x 64 -> the upper 64 bits) and
// rounded once, to nearest, ties away from zero (the float64 expression rounds the difference and
// the product: the two agree within one unit in the last place).  No difference at all, everywhere
// on an axis of symmetry, gives +0.  False for anything else (zero operands, denormals,
// infinities, NaN, a sign change, results near the ends of the range), which takes the float64
// pipe.  That pipe issues one warp's instruction every 64 cycles a scheduler here and bounded the
// kernel with 12 a cell; three differences and their scalings on the integer pipe leave it 6.
__device__ __forceinline__ bool scaled_difference(double a, double b, const GradStencil &s, double &g)
{
    const uint32_t la = (uint32_t)__double2loint(a), ha = (uint32_t)__double2hiint(a);
    const uint32_t lb = (uint32_t)__double2loint(b), hb = (uint32_t)__double2hiint(b);
    // sign and exponent together: of values of different sign the fields are far apart
    const int ea = (int)(ha >> 20), eb = (int)(hb >> 20), em = max(ea, eb);
    const int sa = 9 + ea - em, sb = 9 + eb - em;
    const uint32_t mah = (ha & 0xFFFFFu) | 0x100000u, mbh = (hb & 0xFFFFFu) | 0x100000u;
    uint32_t dl, dh;
    asm("sub.cc.u32 %0, %2, %4;\n\tsubc.u32 %1, %3, %5;"
        : "=r"(dl), "=r"(dh)
        : "r"(la << (sa & 31)), "r"(__funnelshift_l(la, mah, sa)), "r"(lb << (sb & 31)), "r"(__funnelshift_l(lb, mbh, sb)));
    const uint32_t sg = (uint32_t)((int)dh >> 31);
    uint32_t ul, uh;
    asm("sub.cc.u32 %0, %2, %4;\n\tsubc.u32 %1, %3, %4;" : "=r"(ul), "=r"(uh) : "r"(dl ^ sg), "r"(dh ^ sg), "r"(sg));
    // leading one to bit 63, from the lower word where the upper one is empty
    const bool low = uh == 0;
    uh = low ? ul : uh;
    const int n5 = __clz((int)uh), n = low ? n5 + 32 : n5;
    const uint32_t n1 = __funnelshift_l(low ? 0u : ul, uh, n5), n0 = low ? 0u : ul << (n5 & 31);
    const unsigned long long t = (unsigned long long)n1 * s.w0 + __umulhi(n0, s.w0);
    const unsigned long long v = (unsigned long long)n0 * s.w1 + (uint32_t)t;
    const unsigned long long p = (unsigned long long)n1 * s.w1 + (uint32_t)(t >> 32) + (uint32_t)(v >> 32);
    uint32_t pl = (uint32_t)p, ph = (uint32_t)(p >> 32);
    // leading one to bit 62, then to bit 52 of the significand
    const int top = (int)(ph >> 31);
    pl = __funnelshift_r(pl, ph, top);
    ph >>= top;
    asm("add.cc.u32 %0, %0, 0x200;\n\taddc.u32 %1, %1, 0;" : "+r"(pl), "+r"(ph));
    const int be = (em & 0x7FF) + s.we - 1022 - n + top;  // exponent field less one
    const uint32_t rl = __funnelshift_r(pl, ph, 10), rh = (ph >> 10) + ((uint32_t)be << 20);
    const bool none = uh == 0;  // (rl is 0 then)
    g = __hiloint2double(none ? 0 : (int)(rh | ((ha ^ sg) & 0x80000000u)), (int)rl);
    return (sa | sb) >= 0 && (unsigned)((em & 0x7FF) - 64) < 1983u && (none || (unsigned)be < 2045u);
}

// The float64 form, out of line (inlined, its instructions were issued for every cell and selected
// afterwards) and with loads of its own, so that nothing is kept for it.
__device__ __noinline__ double scaled_difference_f64(const double *hi, const double *lo, const GradStencil *s)
{
    return (__ldg(hi) - __ldg(lo)) * s->w;
}

template <int V>
__device__ __forceinline__ void load_cells(const double *p, double (&x)[V], bool stream)
{
    if (V == 2) {
        const double2 t = stream ? __ldcs(reinterpret_cast<const double2 *>(p)) : __ldg(reinterpret_cast<const double2 *>(p));
        x[0] = t.x;
        x[V - 1] = t.y;
    } else {
        x[0] = stream ? __ldcs(p) : __ldg(p);
    }
}

template <int V>
__device__ __forceinline__ void store_cells(double *p, const double (&x)[V])
{
    if (V == 2)
        __stcs(reinterpret_cast<double2 *>(p), make_double2(x[0], x[V - 1]));
    else
        __stcs(p, x[0]);
}

// V neighbouring azimuthal cells a thread: 2 where every row starts on a 16-byte boundary (half
// the memory instructions, twice the loads in flight), in blocks of 64 threads (260 against 251 us in
// blocks of 128, in the form of that time; rows in a loop 296).  An axis on which a cell of the warp
// does not fit goes the float64 way by itself and loads its values again: kept for it, they cost
// spills at the 64 registers that four blocks of 256 threads leave.  At 512 x 128 x 256, S and E: 381
// us with every operation on the float64 pipe, 240 so, on any potential of one sign (with one test
// for all three axes and differences below 33 bits left to the float64 form: 249, and 388 on
// symmetric or flat ones, 310 on Phi of a split solve); 381 -> 287 with an odd number of azimuthal
// cells (410 there).  Noise of both signs takes 388.  The float64 pipe's floor is 163 us, HBM's 178.
// INT false: every difference on the float64 pipe, for gradients alone with one cell a thread (six
// float64 operations a cell in all: 53 us against 58 at 512 x 128 x 40; two cells a thread are faster in
// integers there too, 205 -> 191 at 512 x 128 x 256).
template <int V, bool INT>
__global__ void __launch_bounds__(256, V == 2 ? 4 : 6) k_gravity(const double *__restrict__ phi, const double *__restrict__ rho,
                                                 const double *__restrict__ v, double *__restrict__ grad,
                                                 double *__restrict__ S, double *__restrict__ E,
                                                 const GradStencil *__restrict__ st, int n_r, int n_t, int n_p,
                                                 long long N)
{
    const long long row = blockIdx.x;  // i n_t + j
    const int i = (int)(row / n_t), j = (int)(row - (long long)i * n_t);
    const GradStencil gr = st[i], gt = st[n_r + j];
    const GradStencil *sp = st + n_r + n_t;
    const double *p_row = phi + row * n_p;
    const double *p_rlo = phi + ((long long)gr.lo * n_t + j) * n_p, *p_rhi = phi + ((long long)gr.hi * n_t + j) * n_p;
    const double *p_tlo = phi + ((long long)i * n_t + gt.lo) * n_p, *p_thi = phi + ((long long)i * n_t + gt.hi) * n_p;
    for (int k = V * threadIdx.x; k < n_p; k += V * blockDim.x) {
        const long long c = row * n_p + k;
        // every load of the cells first
        double hi[3][V], lo[3][V], nr[V], v0[V], v1[V], v2[V];
        GradStencil gp[V];
        load_cells<V>(p_rhi + k, hi[0], false);
        load_cells<V>(p_rlo + k, lo[0], false);
        load_cells<V>(p_thi + k, hi[1], false);
        load_cells<V>(p_tlo + k, lo[1], false);
#pragma unroll
        for (int e = 0; e < V; ++e) {
            gp[e] = sp[k + e];
            hi[2][e] = __ldg(p_row + gp[e].hi);
            lo[2][e] = __ldg(p_row + gp[e].lo);
        }
        load_cells<V>(rho + c, nr, true);
        if (E) {
            load_cells<V>(v + c, v0, true);
            load_cells<V>(v + N + c, v1, true);
            load_cells<V>(v + 2 * N + c, v2, true);
        }
        double g[3][V];
        bool fits[3] = {true, true, true};
#pragma unroll
        for (int e = 0; e < V; ++e) {
            nr[e] = -nr[e];
            if constexpr (!INT) {
                g[0][e] = (hi[0][e] - lo[0][e]) * gr.w;
                g[1][e] = (hi[1][e] - lo[1][e]) * gt.w;
                g[2][e] = (hi[2][e] - lo[2][e]) * gp[e].w;
                continue;
            }
            fits[0] &= scaled_difference(hi[0][e], lo[0][e], gr, g[0][e]);
            fits[1] &= scaled_difference(hi[1][e], lo[1][e], gt, g[1][e]);
            fits[2] &= scaled_difference(hi[2][e], lo[2][e], gp[e], g[2][e]);
        }
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            if (fits[a]) continue;
#pragma unroll
            for (int e = 0; e < V; ++e)
                g[a][e] = a == 0 ? scaled_difference_f64(p_rhi + k + e, p_rlo + k + e, st + i)
                          : a == 1 ? scaled_difference_f64(p_thi + k + e, p_tlo + k + e, st + n_r + j)
                                   : scaled_difference_f64(p_row + sp[k + e].hi, p_row + sp[k + e].lo, sp + k + e);
        }
        if (grad) {
#pragma unroll
            for (int a = 0; a < 3; ++a) store_cells<V>(grad + a * N + c, g[a]);
        }
        if (S) {
#pragma unroll
            for (int a = 0; a < 3; ++a) {
#pragma unroll
                for (int e = 0; e < V; ++e) g[a][e] *= nr[e];
                store_cells<V>(S + a * N + c, g[a]);
            }
            if (E) {
                // E = v^a S_a: the products are already there
#pragma unroll
                for (int e = 0; e < V; ++e) v0[e] = fma(v2[e], g[2][e], fma(v1[e], g[1][e], v0[e] * g[0][e]));
                store_cells<V>(E + c, v0);
            }
        } else if (E) {
#pragma unroll
            for (int e = 0; e < V; ++e) v0[e] = nr[e] * fma(v2[e], g[2][e], fma(v1[e], g[1][e], v0[e] * g[0][e]));
            store_cells<V>(E + c, v0);
        }
    }
}

// The same sources with one thread per cell over the flattened mesh, for rows shorter than
// a warp (2-D meshes have one azimuthal cell: a block per row would hold one busy thread).
__global__ void __launch_bounds__(256) k_gravity_flat(const double *__restrict__ phi, const double *__restrict__ rho,
                                                      const double *__restrict__ v, double *__restrict__ grad,
                                                      double *__restrict__ S, double *__restrict__ E,
                                                      const GradStencil *__restrict__ st, int n_r, int n_t,
                                                      int n_p, long long N)
{
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= N) return;
    const long long row = c / n_p;
    const int k = (int)(c - row * n_p);
    const int i = (int)(row / n_t), j = (int)(row - (long long)i * n_t);
    const GradStencil gr = st[i], gt = st[n_r + j], gp = st[n_r + n_t + k];
    const double *p_r = phi + (long long)j * n_p + k, *p_t = phi + (long long)i * n_t * n_p + k;
    const double g0 = (__ldg(p_r + (long long)gr.hi * n_t * n_p) - __ldg(p_r + (long long)gr.lo * n_t * n_p)) * gr.w;
    const double g1 = (__ldg(p_t + (long long)gt.hi * n_p) - __ldg(p_t + (long long)gt.lo * n_p)) * gt.w;
    const double g2 = (__ldg(phi + row * n_p + gp.hi) - __ldg(phi + row * n_p + gp.lo)) * gp.w;
    if (grad) {
        grad[c] = g0;
        grad[N + c] = g1;
        grad[2 * N + c] = g2;
    }
    const double nr = -rho[c];
    if (S) {
        const double s0 = nr * g0, s1 = nr * g1, s2 = nr * g2;
        S[c] = s0;
        S[N + c] = s1;
        S[2 * N + c] = s2;
        if (E) E[c] = fma(v[2 * N + c], s2, fma(v[N + c], s1, v[c] * s0));
    } else if (E) {
        E[c] = nr * fma(v[2 * N + c], g2, fma(v[N + c], g1, v[c] * g0));
    }
}

// lo, hi, 1/dx per cell along one axis (the rule of the file header)
void axis_stencil(const std::vector<double> &e, bool periodic, GradStencil *out)
{
    const int n = (int)e.size() - 1;
    std::vector<double> xc(n);
    for (int i = 0; i < n; ++i) xc[i] = 0.5 * (e[i] + e[i + 1]);
    const double period = e[n] - e[0];
    for (int i = 0; i < n; ++i) {
        int lo, hi;
        double dx;
        if (n == 1) {
            lo = hi = 0;
            dx = 0.0;
        } else if (periodic) {
            lo = (i + n - 1) % n;
            hi = (i + 1) % n;
            const double x_lo = xc[lo] - (i == 0 ? period : 0.0);
            const double x_hi = xc[hi] + (i == n - 1 ? period : 0.0);
            dx = (lo == hi) ? 0.0 : x_hi - x_lo;
        } else {
            lo = i > 0 ? i - 1 : 0;
            hi = i < n - 1 ? i + 1 : n - 1;
            dx = xc[hi] - xc[lo];
        }
        out[i].lo = lo;
        out[i].hi = hi;
        out[i].w = dx != 0.0 ? 1.0 / dx : 0.0;
        unsigned long long b;
        std::memcpy(&b, &out[i].w, sizeof(b));
        const int e = (int)(b >> 52) & 0x7FF;
        const unsigned long long m = (b << 11) | (1ull << 63);
        const bool normal = out[i].w > 0.0 && e > 0 && e < 0x7FF;
        out[i].w0 = normal ? (uint32_t)m : 0u;
        out[i].w1 = normal ? (uint32_t)(m >> 32) : 0u;
        out[i].we = normal ? e : -100000;
        out[i].unused = 0;
    }
}

}  // namespace

cudaError_t gravity_prepare(mp_mesh *m)
{
    constexpr double kTwoPi = 6.283185307179586477;
    std::vector<GradStencil> h((size_t)m->n_r + m->n_t + m->n_p);
    axis_stencil(m->h_r, false, h.data());
    axis_stencil(m->h_th, false, h.data() + m->n_r);
    const double span = m->h_ph.back() - m->h_ph.front();
    const bool full_circle = std::fabs(span - kTwoPi) <= 1e-12 * kTwoPi;
    axis_stencil(m->h_ph, full_circle, h.data() + m->n_r + m->n_t);
    cudaError_t e = cudaMalloc(reinterpret_cast<void **>(&m->d_gst), h.size() * sizeof(GradStencil));
    if (e != cudaSuccess) return e;
    m->device_bytes += h.size() * sizeof(GradStencil);
    return cudaMemcpy(m->d_gst, h.data(), h.size() * sizeof(GradStencil), cudaMemcpyHostToDevice);
}

cudaError_t launch_gravity(mp_mesh *m, const double *phi, const double *rho, const double *v, double *grad, double *S,
                           double *E)
{
    cudaEvent_t ev;
    prof_begin(m, "gravity_sources", &ev);
    if (m->n_p < 32) {
        k_gravity_flat<<<(unsigned)((m->N + 255) / 256), 256, 0, m->stream>>>(phi, rho, v, grad, S, E, m->d_gst, m->n_r,
                                                                              m->n_t, m->n_p, m->N);
    } else {
        const auto bits = [](const void *p) { return reinterpret_cast<uintptr_t>(p); };
        // two cells a thread where every row of every array starts on a 16-byte boundary (the arrays of
        // three components are N cells apart) and a row still fills a warp
        const bool pairs = m->n_p % 2 == 0 && m->n_p >= 64 &&
                           ((bits(phi) | bits(rho) | bits(v) | bits(grad) | bits(S) | bits(E)) & 15) == 0;
        const int cells = pairs ? m->n_p / 2 : m->n_p;
        const int threads = std::min(pairs ? 64 : 256, 32 * ((cells + 31) / 32));
        auto kern = pairs ? k_gravity<2, true> : S || E ? k_gravity<1, true> : k_gravity<1, false>;
        kern<<<(unsigned)m->R, threads, 0, m->stream>>>(phi, rho, v, grad, S, E, m->d_gst, m->n_r, m->n_t, m->n_p, m->N);
    }
    prof_end(m, "gravity_sources", ev);
    return cudaGetLastError();
}

}  // namespace mp
