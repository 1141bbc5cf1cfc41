// Per-line setup on the device, all arithmetic in FP64, results stored as
// float32 (the method builds its tables in double precision and keeps them
// in single precision, Sec. 2.3):
//
//  * the ph_mode 2 Voigt slice H(a, |x|) at 5000 nodes uniform in log10|x|
//    on [-4, 3], stored as ln H (Sec. 2.2.1, 2.3.1);
//  * the velocity sampler (Sec. 2.1.1): 40 incoming-frequency rows (18
//    uniform below |x| = 8, 22 log-spaced to 300) of ln CDF of
//    p(u | x) ~ exp(-u^2) / (a^2 + (x-u)^2) at 251 u-nodes on [-6, 6];
//  * the R_IIA kernel table (Eq. riia-table) on 201 Delta x 200 |x| x 40 g
//    nodes, built from the same discrete sampler masses;
//  * per-cell records {line-centre tau per cell width, V/b} (Eq. sigma0),
//    destruction probabilities (Eq. eps) and the emission CDF over cells.
#include <math.h>

#include "krl_internal.cuh"
#include "voigt.cuh"

namespace krl {

namespace {

constexpr double kPi = 3.14159265358979323846;

// FP64 issues one warp instruction in 16 cycles on this part (2 lanes per
// clock and SM), so the builds below are bound by the FP64 pipes they keep
// busy: each spreads its transcendental work over all SMs in small blocks and
// leaves only the sums, whose order fixes the tables' last bits, to one
// thread: 0.09 ms without the R table, 1.6 ms before.

// Fourier coefficients of Weideman's expansion: one block per coefficient,
// the trapezoidal terms in parallel, added in index order by one thread.
// 520 us as one 48-thread block that evaluated the terms serially.
constexpr int kWeidemanTerms = 4 * kWeidemanN - 1;
constexpr int kCoefBlock = 64;

__device__ void weideman_block(double* c, int N, double L, int n)
{
    __shared__ double f[kWeidemanTerms], cs[kWeidemanTerms];
    const int M = 2 * N;
    for (int q = threadIdx.x; q < kWeidemanTerms; q += blockDim.x) {
        const int k = q - M + 1;
        double th = k * kPi / M;
        double t = L * tan(0.5 * th);
        f[q] = (L * L + t * t) * exp(-t * t);
        cs[q] = cos(n * th);
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    double s = 0.0;
    for (int q = 0; q < kWeidemanTerms; ++q) s += f[q] * cs[q];
    c[n - 1] = s / (2.0 * M);
}

__global__ void k_weideman(double* c, int N, double L) { weideman_block(c, N, L, (int)blockIdx.x + 1); }

// One-warp blocks: the slice's 5000 nodes then reach every SM's FP64 pipe
// (493 us as 20 blocks of 256).
constexpr int kVoigtBlock = 32;

__global__ void k_voigt(double a, const double* c, int N, double L, float* lnH, float* H0)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < kVoigtN) {
        double l = kVoigtL0 + (kVoigtL1 - kVoigtL0) * i / (kVoigtN - 1);
        double x = pow(10.0, l);
        lnH[i] = (float)log(voigt_H(a, x, c, N, L));
    }
    if (i == 0) *H0 = (float)voigt_H(a, 0.0, c, N, L);
}

// Line-profile mode 1 table: ln H(a_j, x_i) with log10 a_j uniform on
// [kV2LaMin, kV2LaMax] (kV2Na nodes) and log10 x_i uniform on [kVoigtL0,
// kVoigtL1] (kV2Nx nodes); one thread per entry.
__global__ void k_voigt2d(const double* c, int N, double L, float* out)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= kV2Na * kV2Nx) return;
    const int j = k / kV2Nx, i = k % kV2Nx;
    const double a = pow(10.0, kV2LaMin + (kV2LaMax - kV2LaMin) * j / (kV2Na - 1));
    const double x = pow(10.0, kVoigtL0 + (kVoigtL1 - kVoigtL0) * i / (kV2Nx - 1));
    out[k] = (float)log(voigt_H(a, x, c, N, L));
}

// Mass of p(u | x) in the u-cell [lo, hi]: the Lorentz factor L(u) times
// the second-order expansion of exp(-u^2) about the midpoint m, integrated
// exactly: exp(-m^2) [I0 - 2 m I1 + (2 m^2 - 1) I2], Ik = int (u-m)^k L du.
// u-node j = -6 + 0.048 j, rounded after the product and after the sum (no
// fused multiply-add): the node at u = 0 must be exactly 0, because for a
// tiny damping parameter a shift of 1e-16 moves the Lorentz spike of width a
// across a cell edge.
__device__ __forceinline__ double unode(int j) { return __dadd_rn(kUsU0, __dmul_rn(kUsDu, (double)j)); }

__device__ double cell_mass(double x, double a, int j)
{
    double lo = unode(j);
    double hi = unode(j + 1);
    double m = 0.5 * (lo + hi);
    double dl = lo - x, dh = hi - x;
    // Lorentz integral (atan(dh/a) - atan(dl/a)) / a; when the cell lies on
    // one side of x the two angles nearly cancel for small a, so use
    // atan(A) - atan(B) = atan((A - B) / (1 + A B)) there
    double I0 = (dl * dh > 0.0) ? atan((hi - lo) * a / (a * a + dl * dh)) / a
                                : (atan(dh / a) - atan(dl / a)) / a;
    double Jx = 0.5 * log((a * a + dh * dh) / (a * a + dl * dl));
    double xm = x - m;
    double I1 = Jx + xm * I0;
    double I2 = (hi - lo) - a * a * I0 + 2.0 * xm * Jx + xm * xm * I0;
    return exp(-m * m) * (I0 - 2.0 * m * I1 + (2.0 * m * m - 1.0) * I2);
}

__device__ double us_xnode(int i)
{
    return i < 18 ? 8.0 * i / 18.0 : 8.0 * pow(37.5, (i - 18) / 21.0);
}

// First stage of a line's tables, all independent of one another: blocks
// [0, N) one Weideman coefficient each; then the sampler rows' cell masses,
// the ln sigmoid of the guide bins' left edges, and (with_r) the cell masses
// at the R table's |x| nodes, one value per thread.
constexpr int kUsMasses = kUsNx * (kUsNu - 1);
constexpr int kRMasses = kRnX * (kUsNu - 1);

__global__ void __launch_bounds__(kCoefBlock) k_line_stage1(double a, double* coef, int N, double L, double* us_mass,
                                                            double* guide_lt, double* r_mass)
{
    if ((int)blockIdx.x < N) {
        weideman_block(coef, N, L, (int)blockIdx.x + 1);
        return;
    }
    int e = ((int)blockIdx.x - N) * kCoefBlock + (int)threadIdx.x;
    if (e < kUsMasses) {
        us_mass[e] = cell_mass(us_xnode(e / (kUsNu - 1)), a, e % (kUsNu - 1));
        return;
    }
    e -= kUsMasses;
    if (e < kGuideN) {
        const double w = -kGuideW + 2.0 * kGuideW * e / kGuideN;
        guide_lt[e] = -log1p(exp(-w));          // ln sigmoid(w)
        return;
    }
    e -= kGuideN;
    if (r_mass && e < kRMasses) {
        double x = kRxMax * (e / (kUsNu - 1)) / (kRnX - 1);
        r_mass[e] = cell_mass(x, a, e % (kUsNu - 1));
    }
}

// One block per sampler row: the running sums of the cell masses by one
// thread in index order (the last one is the row's total), then the
// normalised CDF's logs and the guide in parallel. The masses are positive
// (the expansion of exp(-u^2) over a cell is), so the row does not decrease
// and a guide entry, the largest node j <= kUsNu - 2 with row[j] <= lt, is
// found by bisection. 545 us when one thread also divided and built the
// guide.
__global__ void __launch_bounds__(256) k_usampler(const double* us_mass, const double* guide_lt, float* xs,
                                                  float* lncdf, unsigned char* guide)
{
    __shared__ double run[kUsNu];
    __shared__ float row[kUsNu];
    const int i = blockIdx.x;
    for (int j = threadIdx.x; j < kUsNu - 1; j += blockDim.x) run[j + 1] = us_mass[i * (kUsNu - 1) + j];
    __syncthreads();
    if (threadIdx.x == 0) {
        xs[i] = (float)us_xnode(i);
        double s = 0.0;
        run[0] = 0.0;
        for (int j = 1; j < kUsNu; ++j) {
            s += run[j];
            run[j] = s;
        }
    }
    __syncthreads();
    const double tot = run[kUsNu - 1];
    for (int j = threadIdx.x; j < kUsNu; j += blockDim.x) {
        const double C = run[j] / tot;
        const float v = (float)log(j > 0 && C > kUsFloor ? C : kUsFloor);
        row[j] = v;
        lncdf[(size_t)i * kUsNu + j] = v;
    }
    __syncthreads();
    for (int m = threadIdx.x; m < kGuideN; m += blockDim.x) {
        const double lt = guide_lt[m];
        int lo = 0, hi = kUsNu - 2;             // row[lo] <= lt or lo = 0; row[hi + 1] > lt or hi = kUsNu - 2
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if ((double)row[mid] <= lt) lo = mid;
            else hi = mid - 1;
        }
        guide[(size_t)i * kGuideN + m] = (unsigned char)lo;
    }
}

// Normalises the masses at one R-table |x| node in place (one block per
// node; the total in index order by one thread).
__global__ void __launch_bounds__(256) k_rnorm(double* p)
{
    __shared__ double m[kUsNu - 1];
    __shared__ double tot;
    double* row = p + (size_t)blockIdx.x * (kUsNu - 1);
    for (int k = threadIdx.x; k < kUsNu - 1; k += blockDim.x) m[k] = row[k];
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int k = 0; k < kUsNu - 1; ++k) s += m[k];
        tot = s;
    }
    __syncthreads();
    for (int k = threadIdx.x; k < kUsNu - 1; k += blockDim.x) row[k] = m[k] / tot;
}

// rquad(k, j, i) = the R table's four (g, x) corners of cell (k, j) at Delta_i.
__global__ void k_rquad(const float* rtab, float4* rquad)
{
    const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= kRquadElems) return;
    const int i = (int)(e % kRnD);
    const int j = (int)((e / kRnD) % (kRnX - 1));
    const int k = (int)(e / ((size_t)kRnD * (kRnX - 1)));
    const float* r00 = rtab + ((size_t)k * kRnX + j) * kRnD + i;
    rquad[e] = make_float4(r00[0], r00[kRnD], r00[(size_t)kRnX * kRnD], r00[(size_t)kRnX * kRnD + kRnD]);
}

// R(D_i; x_j, g_k) = sum_c p_c(x_j) G(D_i - m_c (g_k - 1); s_k). The Gaussian
// depends on (k, c, i) only, so it is tabulated first (2.0e6 exponentials
// instead of 4.0e8, one per table entry and sampler cell) and the table is a
// product of [x_j][c] with [c][D_i] for each g_k: 4.0e8 FP64 multiply-adds,
// 0.64 ms at the FP64 pipes' rate. Measured 0.15 ms (kernel) + 0.79 ms
// (product); 19.9 ms with the exponential in the sum. The sum runs over c in
// index order, as a serial sum would.
struct RNode {
    double gm1, inv2s2, norm;
};

__device__ __forceinline__ RNode r_node(int kg)
{
    double g = -1.0 + 2.0 * kg / (kRnG - 1);
    double sg = sqrt(fmax(0.0, 1.0 - g * g)) / sqrt(2.0);
    double s = sg > kRsMin ? sg : kRsMin;
    return RNode{g - 1.0, 0.5 / (s * s), 1.0 / (sqrt(2.0 * kPi) * s)};
}

constexpr size_t kRkernElems = (size_t)kRnG * (kUsNu - 1) * kRnD;

// kern[k][c][i] = exp(-y^2 / (2 s_k^2)); one block per (c, k).
__global__ void __launch_bounds__(224) k_rkernel(double* kern)
{
    const int c = blockIdx.x, kg = blockIdx.y, i = threadIdx.x;
    __shared__ RNode sn;
    if (threadIdx.x == 0) sn = r_node(kg);
    __syncthreads();
    if (i >= kRnD) return;
    const RNode nd = sn;
    double D = -kRdMax + kRdStep * i;
    double lo = unode(c);
    double hi = unode(c + 1);
    double m = 0.5 * (lo + hi);
    double y = D - m * nd.gm1;
    kern[((size_t)kg * (kUsNu - 1) + c) * kRnD + i] = exp(-y * y * nd.inv2s2);
}

// One block per (kRtJ nodes x_j, g_k), one thread per D_i: each kernel value
// is read once for kRtJ sums. 40 x 25 blocks of 7 warps, all resident.
constexpr int kRtJ = 8;

__global__ void __launch_bounds__(224) k_rtable(const double* p, const double* kern, float* rtab)
{
    const int j0 = blockIdx.x * kRtJ, kg = blockIdx.y, i = threadIdx.x;
    __shared__ double sp[kRtJ][kUsNu - 1];
    __shared__ double norm;
    for (int q = threadIdx.x; q < kRtJ * (kUsNu - 1); q += blockDim.x)
        sp[q / (kUsNu - 1)][q % (kUsNu - 1)] = p[(size_t)j0 * (kUsNu - 1) + q];
    if (threadIdx.x == 0) norm = r_node(kg).norm;
    __syncthreads();
    if (i >= kRnD) return;
    const double* e = kern + (size_t)kg * (kUsNu - 1) * kRnD + i;
    double acc[kRtJ];
#pragma unroll
    for (int j = 0; j < kRtJ; ++j) acc[j] = 0.0;
    for (int c = 0; c < kUsNu - 1; ++c) {
        const double v = e[(size_t)c * kRnD];
#pragma unroll
        for (int j = 0; j < kRtJ; ++j) acc[j] += sp[j][c] * v;
    }
#pragma unroll
    for (int j = 0; j < kRtJ; ++j) rtab[((size_t)kg * kRnX + j0 + j) * kRnD + i] = (float)(acc[j] * norm);
}
static_assert(kRnX % kRtJ == 0 && kRnD <= 224, "R table tiling");
static_assert(kRkernElems * sizeof(double) <= kRquadElems * sizeof(float4), "the kernel table fits rquad's buffer");

__global__ void k_fields(FieldArgs F)
{
    int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= F.ncell) return;
    double tau = (double)F.opacity[c] * F.tau_scale;
    float4 r;
    r.x = (float)tau;
    r.y = F.vx ? (float)((double)F.vx[c] * F.inv_b) : 0.0f;
    r.z = F.vy ? (float)((double)F.vy[c] * F.inv_b) : 0.0f;
    r.w = F.vz ? (float)((double)F.vz[c] * F.inv_b) : 0.0f;
    F.cells[c] = r;
    if (F.eps) {
        double q = F.n_coll ? F.k_ul * (double)F.n_coll[c] : 0.0;
        F.eps[c] = (float)(q / (F.A_ul + q));
    }
}

__global__ void k_validate(const float* f, int n, int allow_negative, int* bad)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float v = f[i];
    if (!isfinite(v) || (!allow_negative && v < 0.0f)) atomicOr(bad, 1);
}

// Block-level inclusive scan in FP64, 256 threads x 8 elements per block.
constexpr int kScanT = 256;
constexpr int kScanE = 8;
constexpr int kScanChunk = kScanT * kScanE;

__device__ double block_inclusive_scan(double v, double* sh)
{
    int t = threadIdx.x;
    sh[t] = v;
    __syncthreads();
    for (int off = 1; off < kScanT; off <<= 1) {
        double add = t >= off ? sh[t - off] : 0.0;
        __syncthreads();
        sh[t] += add;
        __syncthreads();
    }
    double r = sh[t];
    __syncthreads();
    return r;
}

__global__ void k_scan_local(const float* rate, int n, double* out, double* block_tot, int* bad)
{
    __shared__ double sh[kScanT];
    size_t base = (size_t)blockIdx.x * kScanChunk + (size_t)threadIdx.x * kScanE;
    double v[kScanE];
    double run = 0.0;
    for (int e = 0; e < kScanE; ++e) {
        size_t i = base + e;
        double r = 0.0;
        if (i < (size_t)n) {
            float f = rate[i];
            if (!isfinite(f) || f < 0.0f) atomicOr(bad, 1);
            r = (double)f;
        }
        run += r;
        v[e] = run;
    }
    double incl = block_inclusive_scan(run, sh);
    double excl = incl - run;
    for (int e = 0; e < kScanE; ++e) {
        size_t i = base + e;
        if (i < (size_t)n) out[i] = v[e] + excl;
    }
    if (threadIdx.x == kScanT - 1) block_tot[blockIdx.x] = incl;
}

// Single block: exclusive offsets of the block totals (sequential per thread chunk).
__global__ void k_scan_totals(double* tot, int nb)
{
    __shared__ double sh[kScanT];
    int per = (nb + kScanT - 1) / kScanT;
    int b0 = threadIdx.x * per;
    double run = 0.0;
    for (int b = b0; b < b0 + per && b < nb; ++b) run += tot[b];
    double incl = block_inclusive_scan(run, sh);
    double off = incl - run;
    for (int b = b0; b < b0 + per && b < nb; ++b) {
        double t = tot[b];
        tot[b] = off;
        off += t;
    }
}

__global__ void k_scan_total(const double* out, int n, double* offs, int nb, int* bad)
{
    double total = out[n - 1] + offs[(n - 1) / kScanChunk];
    offs[nb] = total;
    if (!(total > 0.0)) atomicOr(bad, 2);
}

__global__ void k_scan_finish(double* out, int n, const double* offs, int nb)
{
    size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (size_t)n) return;
    double total = offs[nb];
    if (!(total > 0.0)) return;
    out[i] = (out[i] + offs[i / kScanChunk]) / total;
}

__global__ void k_cdf_guide(const double* cdf, int n, int* guide)
{
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b > (1 << kCdfGuideBits)) return;
    const double edge = (double)b / (1 << kCdfGuideBits);
    int l = 0, h = n - 1;
    while (l < h) {
        const int m = (int)(((unsigned)l + (unsigned)h) >> 1);
        if (cdf[m] > edge) h = m;
        else l = m + 1;
    }
    guide[b] = l;
}

__global__ void k_add_counters(unsigned long long* out, const unsigned long long* in, int n)
{
    int i = threadIdx.x;
    if (i < n && in[i]) atomicAdd(out + i, in[i]);   // runs on other streams may add too
}

__global__ void k_add_counters_batch(unsigned long long* const* dst, const unsigned long long* src, int n_models)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_models * ST_N) return;
    const unsigned long long v = src[i];
    if (v) atomicAdd(dst[i / ST_N] + (i % ST_N), v);
}

}  // namespace

cudaError_t add_counters_batch(unsigned long long* const* dst, const unsigned long long* src, int n_models,
                               cudaStream_t s)
{
    const int n = n_models * ST_N;
    k_add_counters_batch<<<(n + 127) / 128, 128, 0, s>>>(dst, src, n_models);
    return cudaGetLastError();
}

// Scratch of the table builds: coefficients, sampler masses, guide edges, R masses.
constexpr size_t kWorkMass = 64, kWorkLt = kWorkMass + kUsMasses, kWorkR = kWorkLt + kGuideN;
size_t line_tables_work_doubles() { return kWorkR + kRMasses; }

cudaError_t build_line_tables(double a, const LineTables& T, bool with_r, cudaStream_t s)
{
    const int N = kWeidemanN;
    const double L = weideman_L(N);
    double* coef = T.work;
    double* us_mass = T.work + kWorkMass;
    double* lt = T.work + kWorkLt;
    double* p = T.work + kWorkR;
    const int values = kUsMasses + kGuideN + (with_r ? kRMasses : 0);
    k_line_stage1<<<N + (values + kCoefBlock - 1) / kCoefBlock, kCoefBlock, 0, s>>>(a, coef, N, L, us_mass, lt,
                                                                                  with_r ? p : nullptr);
    k_voigt<<<(kVoigtN + kVoigtBlock - 1) / kVoigtBlock, kVoigtBlock, 0, s>>>(a, coef, N, L, T.voigt_lnH, T.H0);
    k_usampler<<<kUsNx, 256, 0, s>>>(us_mass, lt, T.us_x, T.us_lncdf, T.us_guide);
    if (with_r) {
        // the kernel table lives in rquad's buffer until k_rquad fills that
        double* kern = reinterpret_cast<double*>(T.rquad);
        k_rkernel<<<dim3(kUsNu - 1, kRnG), 224, 0, s>>>(kern);
        k_rnorm<<<kRnX, 256, 0, s>>>(p);
        k_rtable<<<dim3(kRnX / kRtJ, kRnG), 224, 0, s>>>(p, kern, T.rtab);
        k_rquad<<<(unsigned)((kRquadElems + 255) / 256), 256, 0, s>>>(T.rtab, T.rquad);
    }
    return cudaGetLastError();
}

cudaError_t build_voigt2d(float* out, double* work, cudaStream_t s)
{
    const int N = kWeidemanN;
    const double L = weideman_L(N);
    k_weideman<<<N, kCoefBlock, 0, s>>>(work, N, L);
    k_voigt2d<<<(kV2Na * kV2Nx + 255) / 256, 256, 0, s>>>(work, N, L, out);
    return cudaGetLastError();
}

cudaError_t derive_fields(const FieldArgs& F, cudaStream_t s)
{
    k_fields<<<(F.ncell + 255) / 256, 256, 0, s>>>(F);
    return cudaGetLastError();
}

cudaError_t validate_field(const float* f, int n, bool allow_negative, int* bad, cudaStream_t s)
{
    if (!f || n <= 0) return cudaSuccess;
    k_validate<<<(n + 255) / 256, 256, 0, s>>>(f, n, allow_negative ? 1 : 0, bad);
    return cudaGetLastError();
}

size_t emission_cdf_work_doubles(int n) { return (size_t)(n + kScanChunk - 1) / kScanChunk + 1; }

cudaError_t emission_cdf(const float* rate, int n, double* cdf, double* work, size_t work_doubles,
                         int* bad, cudaStream_t s)
{
    int nb = (n + kScanChunk - 1) / kScanChunk;
    if ((size_t)nb + 1 > work_doubles) return cudaErrorInvalidValue;
    k_scan_local<<<nb, kScanT, 0, s>>>(rate, n, cdf, work, bad);
    k_scan_totals<<<1, kScanT, 0, s>>>(work, nb);
    k_scan_total<<<1, 1, 0, s>>>(cdf, n, work, nb, bad);
    k_scan_finish<<<(n + 255) / 256, 256, 0, s>>>(cdf, n, work, nb);
    return cudaGetLastError();
}

cudaError_t emission_guide(const double* cdf, int n, int* guide, cudaStream_t s)
{
    k_cdf_guide<<<((1 << kCdfGuideBits) + 128) / 128, 128, 0, s>>>(cdf, n, guide);
    return cudaGetLastError();
}

cudaError_t add_counters(unsigned long long* out, const unsigned long long* in, int n, cudaStream_t s)
{
    k_add_counters<<<1, 32, 0, s>>>(out, in, n);
    return cudaGetLastError();
}

}  // namespace krl
