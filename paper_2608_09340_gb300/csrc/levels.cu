// Statistical equilibrium of a multi-level molecule (Sec. 2.1.3, Eq.
// boltzmann generalised to n levels) and the pieces of the Lambda iteration
// that run per cell: one thread per cell, FP64.
//
// Rates for each pair u > l: collisions C_ul = k_ul n_coll and, by detailed
// balance, C_lu = (g_u/g_l) C_ul exp(-(E_u - E_l)/T); radiation l -> u at the
// Monte Carlo absorption rate Gamma_lu, u -> l at A_ul + (g_l/g_u) Gamma_lu
// (spontaneous plus stimulated emission). The steady state sum_j n_j R_ji =
// n_i sum_j R_ij, with the last equation replaced by sum_i n_i = n_mol, is
// solved by Gaussian elimination with partial pivoting.
#include <math.h>

#include "krl_internal.cuh"

namespace krl {

namespace {

// The Boltzmann weights are the same in every cell: one thread per level forms
// them once per block (FP64 issues a warp instruction in 16 cycles, and an
// exponential is some forty of them): 128^3 cells, 5 levels, 0.74 -> 0.19 ms.
__global__ void __launch_bounds__(256) k_lte(LevelConst L, const float* n_mol, int ncell, double* pops)
{
    __shared__ double w[kMaxLevels];
    if ((int)threadIdx.x < L.n) w[threadIdx.x] = L.g[threadIdx.x] * exp(-(L.E[threadIdx.x] - L.E[0]) / L.T);
    __syncthreads();
    double z = 0.0;
    for (int i = 0; i < L.n; ++i) z += w[i];
    for (unsigned c = blockIdx.x * blockDim.x + threadIdx.x; c < (unsigned)ncell; c += gridDim.x * blockDim.x) {
        const double nm = (double)n_mol[c];
        for (int i = 0; i < L.n; ++i) pops[(size_t)c * L.n + i] = nm * w[i] / z;
    }
}

__global__ void k_level_field(const double* pops, int ncell, int n_lev, int lev, double scale, float* out)
{
    int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= ncell) return;
    out[c] = (float)(scale * pops[(size_t)c * n_lev + lev]);
}

// FP64 sum of n_u A over cells into *total, in a fixed order (so the result
// does not depend on scheduling): kSumBlocks blocks each sum a grid-strided
// share into partials[block], then one block sums the partials.
constexpr int kSumBlocks = 512;

__device__ __forceinline__ double block_sum256(double v, double* sh)
{
    sh[threadIdx.x] = v;
    __syncthreads();
    for (int off = 128; off > 0; off >>= 1) {
        if (threadIdx.x < off) sh[threadIdx.x] += sh[threadIdx.x + off];
        __syncthreads();
    }
    return sh[0];
}

__global__ void k_sum_rate_part(const double* pops, int ncell, int n_lev, int u, double A, double* partials)
{
    __shared__ double sh[256];
    double s = 0.0;
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < ncell; c += gridDim.x * blockDim.x)
        s += pops[(size_t)c * n_lev + u] * A;
    const double b = block_sum256(s, sh);
    if (threadIdx.x == 0) partials[blockIdx.x] = b;
}

__global__ void k_sum_rate_final(const double* partials, int n, double* total)
{
    __shared__ double sh[256];
    double s = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) s += partials[i];
    const double b = block_sum256(s, sh);
    if (threadIdx.x == 0) *total = b;
}

// Gamma_c = (L / N) sigma0 exc_c / dx^2 with L = total * dx^3 photons/s.
__global__ void k_gamma(const double* exc, int ncell, const double* total, double dx, double sigma0, double n_packets,
                        double* gamma)
{
    int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= ncell) return;
    const double Lum = (*total) * dx * dx * dx;
    gamma[c] = Lum / n_packets * sigma0 * exc[c] / (dx * dx);
}

// Gaussian elimination with partial pivoting from column COL on. One
// instantiation per column: every index is a constant, also where the
// compiler would not unroll a loop nest of this size.
template <int N, int COL = 0>
__device__ __forceinline__ void eliminate(double (&M)[N][N + 1])
{
    if constexpr (COL < N) {
        int piv = COL;
        double best = fabs(M[COL][COL]);
#pragma unroll
        for (int r = COL + 1; r < N; ++r)
            if (fabs(M[r][COL]) > best) { best = fabs(M[r][COL]); piv = r; }
#pragma unroll
        for (int r = COL + 1; r < N; ++r) {
            const bool sw = piv == r;
#pragma unroll
            for (int j = COL; j <= N; ++j) {
                const double a = M[COL][j], b = M[r][j];
                M[COL][j] = sw ? b : a;
                M[r][j] = sw ? a : b;
            }
        }
        const double d = M[COL][COL];
        if (d != 0.0) {                     // (singular, an n_mol = 0 cell: leaves zeros)
#pragma unroll
            for (int r = COL + 1; r < N; ++r) {
                const double f = M[r][COL] / d;
                if (f != 0.0) {
#pragma unroll
                    for (int j = COL; j <= N; ++j) M[r][j] -= f * M[COL][j];
                }
            }
        }
        eliminate<N, COL + 1>(M);
    }
}

// One thread per cell, N levels. What the cells share, the detailed-balance
// factors and the ratios of degeneracies of each pair, is formed once per
// block; the matrices are unrolled over N, so that they live in registers (with
// 3 levels 8 bytes of spills, with 8 levels 112) and the pivoting
// is selects. Bound by the FP64 pipe (2 lanes per clock and SM): 16 divisions
// and about 200 other operations per cell at 5 levels. 128^3 cells, 5 levels:
// 2.8 -> 1.34 ms; before, each cell formed the exponentials and ratios (20 of
// each) itself, and the matrices lived in local memory. Whole calls with 2, 3,
// 4, 5, 6, 7 and 8 levels: 1.39, 1.47, 2.06, 3.10, 4.39, 5.94 and 7.74 ms
// before, 0.30, 0.53, 0.87, 1.43, 1.86, 2.51 and 3.30 now.
template <int N>
__global__ void __launch_bounds__(128) k_solve(LevelConst L, const double* gamma, int ncell, const float* n_coll,
                                               const float* n_mol, double* pops, unsigned long long* max_change)
{
    __shared__ double s_up[N][N], s_ex[N][N], s_dn[N][N];      // [u][l]: g_u / g_l, exp(-(E_u - E_l) / T), g_l / g_u
    __shared__ int s_t[N][N];                                  // transition of the pair, or -1
    for (int q = threadIdx.x; q < N * N; q += blockDim.x) {
        const int u = q / N, l = q % N;
        if (u > l) {
            s_up[u][l] = L.g[u] / L.g[l];
            s_ex[u][l] = exp(-(L.E[u] - L.E[l]) / L.T);
            s_dn[u][l] = L.g[l] / L.g[u];
            int t = -1;
            for (int k = 0; k < L.n_trans; ++k)
                if (L.tu[k] == u && L.tl[k] == l) t = k;
            s_t[u][l] = t;
        }
    }
    __syncthreads();
    for (unsigned c = blockIdx.x * blockDim.x + threadIdx.x; c < (unsigned)ncell; c += gridDim.x * blockDim.x) {
        double R[N][N];
        const double nc = n_coll ? (double)n_coll[c] : 0.0;
#pragma unroll
        for (int u = 1; u < N; ++u)
#pragma unroll
            for (int l = 0; l < u; ++l) {
                const double Cul = L.k[u][l] * nc;
                R[l][u] = s_up[u][l] * Cul * s_ex[u][l];
                R[u][l] = L.A[u][l] + Cul;
                const int t = s_t[u][l];
                if (t >= 0) {
                    const double G = gamma[(size_t)t * ncell + c];
                    R[l][u] += G;
                    R[u][l] += s_dn[u][l] * G;
                }
            }
        // M[i][j] = R[j][i] (i != j), M[i][i] = -sum_j R[i][j]; last row: conservation
        double M[N][N + 1];
#pragma unroll
        for (int i = 0; i < N; ++i) {
            double out = 0.0;
#pragma unroll
            for (int j = 0; j < N; ++j) {
                if (j != i) {
                    M[i][j] = R[j][i];
                    out += R[i][j];
                }
            }
            M[i][i] = -out;
            M[i][N] = 0.0;
        }
        const double nm = (double)n_mol[c];
#pragma unroll
        for (int j = 0; j < N; ++j) M[N - 1][j] = 1.0;
        M[N - 1][N] = nm;
        eliminate<N>(M);
        double x[N];
#pragma unroll
        for (int i = N - 1; i >= 0; --i) {
            double s = M[i][N];
#pragma unroll
            for (int j = i + 1; j < N; ++j) s -= M[i][j] * x[j];
            x[i] = M[i][i] != 0.0 ? s / M[i][i] : 0.0;
        }
        double change = 0.0;
#pragma unroll
        for (int i = 0; i < N; ++i) {
            double* p = pops + (size_t)c * N + i;
            const double old = *p;
            const double v = x[i] > 0.0 ? x[i] : 0.0;     // round-off below zero
            change = fmax(change, fabs(v - old));
            *p = v;
        }
        // (rounding is monotonic: the largest of the quotients; an infinite
        // density has none)
        change = nm > 0.0 && nm < (double)INFINITY ? change / nm : 0.0;
        // (most cells change less than some other has: no atomic for them)
        const unsigned long long bits = (unsigned long long)__double_as_longlong(change);
        if (max_change && bits > *(volatile unsigned long long*)max_change) atomicMax(max_change, bits);
    }
}

// Blocks of a grid-stride kernel that shares set-up per block: 16 per SM.
int stride_blocks(int ncell, int threads, int sm_count)
{
    const int full = (int)(((unsigned)ncell + threads - 1) / threads);
    return full < sm_count * 16 ? full : sm_count * 16;
}

template <int N>
void launch_solve(const LevelConst& L, const double* gamma, int ncell, const float* n_coll, const float* n_mol, double* pops,
                  unsigned long long* max_change, int sm_count, cudaStream_t s)
{
    k_solve<N><<<stride_blocks(ncell, 128, sm_count), 128, 0, s>>>(L, gamma, ncell, n_coll, n_mol, pops, max_change);
}

}  // namespace

cudaError_t levels_lte(const LevelConst& L, const float* n_mol, int ncell, double* pops, int sm_count, cudaStream_t s)
{
    k_lte<<<stride_blocks(ncell, 256, sm_count), 256, 0, s>>>(L, n_mol, ncell, pops);
    return cudaGetLastError();
}

cudaError_t levels_field(const double* pops, int ncell, int n_lev, int lev, double scale, float* out, cudaStream_t s)
{
    k_level_field<<<(ncell + 255) / 256, 256, 0, s>>>(pops, ncell, n_lev, lev, scale, out);
    return cudaGetLastError();
}

size_t levels_sum_scratch_doubles() { return 1 + (size_t)kSumBlocks; }

cudaError_t levels_sum_rate(const double* pops, int ncell, int n_lev, int u, double A, double* total, cudaStream_t s)
{
    k_sum_rate_part<<<kSumBlocks, 256, 0, s>>>(pops, ncell, n_lev, u, A, total + 1);
    k_sum_rate_final<<<1, 256, 0, s>>>(total + 1, kSumBlocks, total);
    return cudaGetLastError();
}

cudaError_t levels_gamma(const double* exc, int ncell, const double* total, double dx, double sigma0, double n_packets,
                         double* gamma, cudaStream_t s)
{
    k_gamma<<<(ncell + 255) / 256, 256, 0, s>>>(exc, ncell, total, dx, sigma0, n_packets, gamma);
    return cudaGetLastError();
}

cudaError_t levels_solve(const LevelConst& L, const double* gamma, int ncell, const float* n_coll, const float* n_mol,
                         double* pops, unsigned long long* max_change, int sm_count, cudaStream_t s)
{
    switch (L.n) {
    case 2: launch_solve<2>(L, gamma, ncell, n_coll, n_mol, pops, max_change, sm_count, s); break;
    case 3: launch_solve<3>(L, gamma, ncell, n_coll, n_mol, pops, max_change, sm_count, s); break;
    case 4: launch_solve<4>(L, gamma, ncell, n_coll, n_mol, pops, max_change, sm_count, s); break;
    case 5: launch_solve<5>(L, gamma, ncell, n_coll, n_mol, pops, max_change, sm_count, s); break;
    case 6: launch_solve<6>(L, gamma, ncell, n_coll, n_mol, pops, max_change, sm_count, s); break;
    case 7: launch_solve<7>(L, gamma, ncell, n_coll, n_mol, pops, max_change, sm_count, s); break;
    case 8: launch_solve<8>(L, gamma, ncell, n_coll, n_mol, pops, max_change, sm_count, s); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace krl
