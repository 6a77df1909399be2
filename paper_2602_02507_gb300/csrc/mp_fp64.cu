// mp_fp64.cu -- the float64 path: its contractions on CUDA cores in float64 (GB300's float64
// rate bounds them) and the dispatch to their tensor-core form (mp_fp64_tc.cu).  The theta
// contraction always runs here; the other steps do beyond the range of the tensor-core form (l_max >
// 71), for small meshes and few azimuthal cells, for moments whose squares overflow, and in
// mp_moments_noalloc, whose scratch is fixed.  A solve with the tensor-core steps against one without: 46.3 -> 1.63 ms at
// 1024 x 256 x 512 cells, l_max = 32; 3.10 -> 0.22 ms at 512 x 128 x 256, 16; 1.53 -> 0.15 ms at 353 x
// 96 x 192, 20; 340 -> 117 us at 471 x 128 x 1, 20.
// Steps of GenASiS II Sec. 2.2:
//   (a1) F[row][p]  = sum_k Iph[p][k] rho[row][k]                 (phi part of Eq. AngularMomentsDiscrete)
//   (a2) A[i][q]    = 4 pi G sum_j Ith[t][j] F[i n_t + j][p]      (theta part)
//   (d1) G[row][p]  = sum_{l>=m} (Ith[t][j] / dmu_j) C[i][q]       (theta part of Eq. Solution)
//   (d2) Phi[row][k]= sum_p G[row][p] Iph[p][k] / dphi_k           (phi part)
// with row = i n_t + j, q = l^2 + p, t = t(l, m(p)).
#include "mp_internal.h"
#include "ptx.cuh"

namespace mp {

namespace {

constexpr double kFourPi = 12.566370614359172954;

// (a1): one block per group of rows; rho rows staged in shared memory.
constexpr int kRowsPerBlock = 4;

__global__ void __launch_bounds__(256) k64_project(const double *__restrict__ rho, const double *__restrict__ Iph,
                                                   double *__restrict__ F, long long R, int n_p, int P, int *err)
{
    extern __shared__ double srow[];  // [kRowsPerBlock][n_p]
    const long long row0 = (long long)blockIdx.x * kRowsPerBlock;
    const int nrows = (int)min((long long)kRowsPerBlock, R - row0);
    bool bad = false;
    for (int e = threadIdx.x; e < nrows * n_p; e += blockDim.x) {
        const double v = rho[row0 * n_p + e];
        bad |= !isfinite(v);
        srow[e] = v;
    }
    if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(err, DEV_ERR_NONFINITE);
    for (int o = threadIdx.x; o < nrows * P; o += blockDim.x) {
        const int rr = o / P, p = o % P;
        const double *s = srow + (size_t)rr * n_p;
        const double *w = Iph + (size_t)p * n_p;
        double acc = 0.0;
        for (int k = 0; k < n_p; ++k) acc = fma(w[k], s[k], acc);
        F[(row0 + rr) * P + p] = acc;
    }
}

// (a2): one block per shell, one thread per moment.
__global__ void __launch_bounds__(256) k64_theta(const double *__restrict__ F, const double *__restrict__ Ith,
                                                 double *__restrict__ A, int n_t, int L, int KL, int P, double scale)
{
    const int i = blockIdx.x;
    for (int q = threadIdx.x; q < KL; q += blockDim.x) {
        int l = 0;
        while ((l + 1) * (l + 1) <= q) ++l;
        const int p = q - l * l;
        const int t = tri(l, pcol_m(p));
        const double *f = F + (size_t)i * n_t * P + p;
        const double *w = Ith + (size_t)t * n_t;
        double acc = 0.0;
        for (int j = 0; j < n_t; ++j) acc = fma(w[j], f[(size_t)j * P], acc);
        A[(size_t)i * KL + q] = scale * acc;
    }
}

// (a2) with F as [n_r][P][ldJ]: in float64 whatever the other steps do.  The table (sin^m theta
// near the poles) and a row of F may be large at different cells, and a product of fixed-point
// operands, scaled by the maxima of both, then loses what a float64 sum keeps: a clump near the pole
// left moments of order 16 with errors of 1e-5 of their own terms.  A block takes 32 rows (shells,
// or cos and sin of 16 shells) of one order and 32 of its degrees; chunks of 32 polar cells of both
// operands pass through shared memory, a lane sums its row for up to four degrees, in the
// order of k64_theta.  The float64 pipe bounds it, so lanes are rows (always full) and not degrees,
// and the degrees are dealt to the warps one by one (to the SM's four quarters evenly).
// 512 x 128 x 256 cells, l_max = 16: 76 us as k64_theta, 53 so; 1024 x 256 x 512, 32: 688 -> 479 (0.6 T
// products a second, all the pipe does); fixed-point slices on the tensor cores took 20 and 92.
constexpr int kThRows = 32, kThDeg = 32, kThCells = 32, kThWarps = 8, kThWarpDeg = kThDeg / kThWarps;

// One chunk: ND degrees (rows kThWarps apart of sT) of the lane's row.
template <int ND>
__device__ __forceinline__ void theta_chunk(const double (*sF)[kThRows + 1], const double (*sT)[kThCells], int lane,
                                            int cells, double (&acc)[kThWarpDeg])
{
    if (cells == kThCells) {
#pragma unroll 4
        for (int j = 0; j < kThCells; j += 2) {
            const double f0 = sF[j][lane], f1 = sF[j + 1][lane];
#pragma unroll
            for (int c = 0; c < ND; ++c) {
                const double2 w = *reinterpret_cast<const double2 *>(&sT[kThWarps * c][j]);
                acc[c] = fma(w.y, f1, fma(w.x, f0, acc[c]));
            }
        }
    } else {
        for (int j = 0; j < cells; ++j)
#pragma unroll
            for (int c = 0; c < ND; ++c) acc[c] = fma(sT[kThWarps * c][j], sF[j][lane], acc[c]);
    }
}

__global__ void __launch_bounds__(32 * kThWarps) k64_theta_rows(const double *__restrict__ F, const double *__restrict__ Ith,
                                                      double *__restrict__ A, int n_r, int n_t, int L, int KL, int P,
                                                      int ldJ, double scale)
{
    __shared__ double sF[kThCells][kThRows + 1];
    __shared__ __align__(16) double sT[kThDeg][kThCells];
    const int n_dg = (L + kThDeg) / kThDeg, m = blockIdx.y / n_dg, d0 = (blockIdx.y - m * n_dg) * kThDeg;
    const int N = min(kThDeg, L + 1 - m - d0);  // degrees m + d0 ... of this block
    const int i0 = blockIdx.x * (m ? kThRows / 2 : kThRows);
    if (N <= 0 || i0 >= n_r) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // loads: cell `lane` of rows (and degrees) warp, warp + kThWarps, ...
    double f[kThWarpDeg], t[kThWarpDeg];
    auto load = [&](int j0) {
        const int j = j0 + lane;
#pragma unroll
        for (int k = 0; k < kThWarpDeg; ++k) {
            const int r = warp + kThWarps * k, i = i0 + (m ? r >> 1 : r), p = m ? 2 * m - 1 + (r & 1) : 0;
            f[k] = j < n_t && i < n_r ? __ldg(F + ((size_t)i * P + p) * ldJ + j) : 0.0;
            t[k] = j < n_t && r < N ? __ldg(Ith + (size_t)tri(m + d0 + r, m) * n_t + j) : 0.0;
        }
    };
    double acc[kThWarpDeg] = {};
    const int nd = (N - warp + kThWarps - 1) / kThWarps;  // degrees of this warp
    load(0);
    for (int j0 = 0; j0 < n_t; j0 += kThCells) {
        __syncthreads();  // the chunk before has been read
#pragma unroll
        for (int k = 0; k < kThWarpDeg; ++k) {
            sF[lane][warp + kThWarps * k] = f[k];
            sT[warp + kThWarps * k][lane] = t[k];
        }
        __syncthreads();
        if (j0 + kThCells < n_t) load(j0 + kThCells);
        const int cells = min(kThCells, n_t - j0);
        switch (nd) {
        case 4: theta_chunk<4>(sF, sT + warp, lane, cells, acc); break;
        case 3: theta_chunk<3>(sF, sT + warp, lane, cells, acc); break;
        case 2: theta_chunk<2>(sF, sT + warp, lane, cells, acc); break;
        case 1: theta_chunk<1>(sF, sT + warp, lane, cells, acc); break;
        }
    }
    const int i = i0 + (m ? lane >> 1 : lane), p = m ? 2 * m - 1 + (lane & 1) : 0;
    if (i >= n_r) return;
#pragma unroll
    for (int c = 0; c < kThWarpDeg; ++c) {
        const int d = warp + kThWarps * c, l = m + d0 + d;
        if (d < N) A[(size_t)i * KL + l * l + p] = scale * acc[c];
    }
}

// (d1): one thread per (row, p).
__global__ void __launch_bounds__(256) k64_synth_theta(const double *__restrict__ C, const double *__restrict__ Ith,
                                                       const double *__restrict__ dmu, double *__restrict__ Gm,
                                                       long long R, int n_t, int L, int KL, int P)
{
    const long long o = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (o >= R * P) return;
    const long long row = o / P;
    const int p = (int)(o % P);
    const int i = (int)(row / n_t), j = (int)(row % n_t);
    const int m = pcol_m(p);
    const double inv = 1.0 / dmu[j];
    double acc = 0.0;
    for (int l = m; l <= L; ++l) acc = fma(Ith[(size_t)tri(l, m) * n_t + j] * inv, C[(size_t)i * KL + l * l + p], acc);
    Gm[o] = acc;
}

// (d2): one thread per cell.
__global__ void __launch_bounds__(256) k64_synth_phi(const double *__restrict__ Gm, const double *__restrict__ Iphc,
                                                     double *__restrict__ phi, long long N, int n_p, int P)
{
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= N) return;
    const long long row = c / n_p;
    const int k = (int)(c % n_p);
    const double *g = Gm + row * P;
    double acc = 0.0;
    for (int p = 0; p < P; ++p) acc = fma(g[p], Iphc[(size_t)p * n_p + k], acc);
    phi[c] = acc;
}

// (a1) and (d2) for a few azimuthal cells, beside the tensor-core theta stages: F and G as
// [n_r][P][ldJ], neighbouring threads on neighbouring polar cells.  Each thread of the projection
// takes kFewCols columns of its cell row (a block for each column made 19,000 blocks of one product
// a thread at 471 x 128 x 1 cells, l_max = 20), and the synthesis sums in four chains: latency
// bounds both (the projection 16.5 -> 12.7 us there).
constexpr int kFewCols = 8;

__global__ void __launch_bounds__(128) k64_project_few(const double *__restrict__ rho, const double *__restrict__ Iph,
                                                       double *__restrict__ F, int n_t, int n_p, int P, int ldJ,
                                                       int *err)
{
    const int i = blockIdx.x, p0 = blockIdx.y * kFewCols, np = min(kFewCols, P - p0);
    for (int j = threadIdx.x + blockIdx.z * blockDim.x; j < n_t; j += blockDim.x * gridDim.z) {
        const double *s = rho + ((size_t)i * n_t + j) * n_p;
        double acc[kFewCols] = {};
        bool bad = false;
        for (int k = 0; k < n_p; ++k) {
            const double v = __ldg(s + k);
            bad |= !isfinite(v);
#pragma unroll
            for (int q = 0; q < kFewCols; ++q)
                if (q < np) acc[q] = fma(__ldg(Iph + (size_t)(p0 + q) * n_p + k), v, acc[q]);
        }
        if (bad && p0 == 0) atomicOr(err, DEV_ERR_NONFINITE);
#pragma unroll
        for (int q = 0; q < kFewCols; ++q)
            if (q < np) F[((size_t)i * P + p0 + q) * ldJ + j] = acc[q];
    }
}

__global__ void __launch_bounds__(128) k64_synth_phi_few(const double *__restrict__ Gm, const double *__restrict__ Iphc,
                                                         double *__restrict__ phi, int n_t, int n_p, int P, int ldJ)
{
    const int i = blockIdx.x;
    for (int c = threadIdx.x + blockIdx.y * blockDim.x; c < n_t * n_p; c += blockDim.x * gridDim.y) {
        const int k = c / n_t, j = c - k * n_t;
        const double *g = Gm + (size_t)i * P * ldJ + j;
        double acc[4] = {};
        int p = 0;
        for (; p + 4 <= P; p += 4)
#pragma unroll
            for (int q = 0; q < 4; ++q)
                acc[q] = fma(__ldg(g + (size_t)(p + q) * ldJ), __ldg(Iphc + (size_t)(p + q) * n_p + k), acc[q]);
        for (; p < P; ++p) acc[0] = fma(__ldg(g + (size_t)p * ldJ), __ldg(Iphc + (size_t)p * n_p + k), acc[0]);
        phi[((size_t)i * n_t + j) * n_p + k] = (acc[0] + acc[1]) + (acc[2] + acc[3]);
    }
}

}  // namespace

cudaError_t launch_fp64_project(mp_mesh *m, const double *rho)
{
    if (m->fp.proj_on) return launch_fp64_tc_project(m, rho);
    if (m->fp.rows) {
        cudaEvent_t ev;
        prof_begin(m, "fp64_phi_project", &ev);
        const int threads = std::min(128, round_up(m->n_t, 32));
        k64_project_few<<<dim3(m->n_r, (m->P + kFewCols - 1) / kFewCols, (m->n_t + threads - 1) / threads), threads, 0,
                          m->stream>>>(rho, m->d_Iph, m->d_F64, m->n_t, m->n_p, m->P, m->fp.ldJ, m->d_err);
        prof_end(m, "fp64_phi_project", ev);
        return cudaGetLastError();
    }
    const long long blocks = (m->R + kRowsPerBlock - 1) / kRowsPerBlock;
    const size_t smem = (size_t)kRowsPerBlock * m->n_p * sizeof(double);
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(k64_project, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    cudaEvent_t ev;
    prof_begin(m, "fp64_phi_project", &ev);
    k64_project<<<(unsigned)blocks, 256, smem, m->stream>>>(rho, m->d_Iph, m->d_F64, m->R, m->n_p, m->P, m->d_err);
    prof_end(m, "fp64_phi_project", ev);
    return cudaGetLastError();
}

cudaError_t launch_fp64_moments_into(const mp_mesh *m, const double *rho, double *F, double *A)
{
    const long long blocks = (m->R + kRowsPerBlock - 1) / kRowsPerBlock;
    const size_t smem = (size_t)kRowsPerBlock * m->n_p * sizeof(double);
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(k64_project, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    k64_project<<<(unsigned)blocks, 256, smem, m->stream>>>(rho, m->d_Iph, F, m->R, m->n_p, m->P, m->d_err);
    k64_theta<<<m->n_r, 256, 0, m->stream>>>(F, m->d_Ith, A, m->n_t, m->L, m->KL, m->P, kFourPi * m->G);
    return cudaGetLastError();
}

cudaError_t launch_fp64_theta(mp_mesh *m)
{
    cudaEvent_t ev;
    prof_begin(m, "fp64_theta_contract", &ev);
    if (m->fp.rows)
        k64_theta_rows<<<dim3((m->n_r + kThRows / 2 - 1) / (kThRows / 2), (m->L + 1) * ((m->L + kThDeg) / kThDeg)), 32 * kThWarps, 0,
                         m->stream>>>(m->d_F64, m->d_Ith, m->d_A, m->n_r, m->n_t, m->L, m->KL, m->P, m->fp.ldJ,
                                      kFourPi * m->G);
    else
        k64_theta<<<m->n_r, 256, 0, m->stream>>>(m->d_F64, m->d_Ith, m->d_A, m->n_t, m->L, m->KL, m->P,
                                                kFourPi * m->G);
    prof_end(m, "fp64_theta_contract", ev);
    return cudaGetLastError();
}

cudaError_t launch_fp64_synth(mp_mesh *m, double *phi)
{
    cudaEvent_t ev;
    if (m->fp.on) {
        cudaError_t e = launch_fp64_tc_synth_theta(m);
        if (e != cudaSuccess) return e;
        if (m->fp.phi_on) return launch_fp64_tc_synth_phi(m, phi);
        prof_begin(m, "fp64_phi_synth", &ev);
        const int cells = m->n_t * m->n_p;
        const int threads = std::min(128, round_up(cells, 32));
        k64_synth_phi_few<<<dim3(m->n_r, (cells + threads - 1) / threads), threads, 0, m->stream>>>(
            m->d_G64, m->d_Iphc, phi, m->n_t, m->n_p, m->P, m->fp.ldJ);
        prof_end(m, "fp64_phi_synth", ev);
        return cudaGetLastError();
    }
    prof_begin(m, "fp64_theta_synth", &ev);
    {
        const long long n = m->R * m->P;
        k64_synth_theta<<<(unsigned)((n + 255) / 256), 256, 0, m->stream>>>(m->d_C, m->d_Ith, m->d_dmu, m->d_G64,
                                                                            m->R, m->n_t, m->L, m->KL, m->P);
    }
    prof_end(m, "fp64_theta_synth", ev);
    prof_begin(m, "fp64_phi_synth", &ev);
    k64_synth_phi<<<(unsigned)((m->N + 255) / 256), 256, 0, m->stream>>>(m->d_G64, m->d_Iphc, phi, m->N, m->n_p,
                                                                         m->P);
    prof_end(m, "fp64_phi_synth", ev);
    return cudaGetLastError();
}

}  // namespace mp
