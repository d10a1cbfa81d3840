// The banded FTCG coefficient matrix C for band r > 1 (Sec. III-C, Eq. ftcg, Eq. cr; in 2-D C_2
// of Eq. twodftcg), reading (i): C minimises || T C - I ||_F over matrices that are zero outside
// the band |j - k| <= r - 1 of the acquisition order (the minimisation of Eq. difopt with its
// diagonal constraint widened to 2r - 1 diagonals). T = Psi Omega is taken as the data-frame Gram
// matrix on the N x N pixel lattice, T_jk = Dx(lambda_k - lambda_j) Dy(lambda_k - lambda_j) with
// the Dirichlet kernel D(d) = N^-1 sum_p exp(2 pi i d p / N) = exp(-i pi d / N) sin(pi d) /
// (N sin(pi d / N)), p in {-N/2 .. N/2 - 1}.
//
// The problem separates over the columns of C: column k solves the least-squares problem
// T[:, S_k] c = e_k over its band rows S_k, whose normal equations are
// (T^2)[S_k, S_k] c = T[S_k, k] (T is Hermitian). At r = 1 this is alpha_k = 1 / S_k (the
// diagonal weights); with the whole index range as band it is C = T^+ (Eq. dif3), whose image is
// the frame approximation (Eq. insert).
//
// Everything runs in FP64 on the device, on real matrices: exp(-i pi d / N) is a product of one
// phase per sample, so T = Phi^H rho Phi with Phi = diag(exp(-i pi (lambda_jx + lambda_jy) / N))
// and rho_jk = prod sin(pi d) / (N sin(pi d / N)) real and symmetric, T^2 = Phi^H rho^2 Phi, and
// column k is c_i = conj(phi_i) c'_i phi_k with (rho^2)[S_k, S_k] c' = rho[S_k, k]. Steps: rho (a
// tile and its transpose per CTA), the band of rho^2 ((rho^2)_{a,a+o}, o = 0..2r-2), and one
// Cholesky solve of the (2r-1) x (2r-1) system per column. The cost is O(M^2 r) and
// the memory 8 M^2 bytes, so the path accepts M <= 8192 (the size of the paper's rasters and of
// the tiny configuration). ftcg_adjoint then forms tau = C v (2r - 1 terms per sample) and
// spreads tau with unit weights (Eq. ftcg: tau = C f^).
//
// The FP64 pipe (2 multiply-adds per SM and clock) bounds all of it, so the design counts FP64
// instructions. Tiny configuration (M = 4096, r = 5), us: rho 4680 as a complex matrix with two
// sinpi and a sincospi per axis and entry, here 928; the band of its square 1684 (one warp per
// complex entry, every row read 18 times), here 398 (151 M multiply-adds take 240 at the pipe's
// rate); solve 90, here 43.

#include <cmath>

#include "ftcg_internal.cuh"

namespace ftcg {

namespace {

constexpr int kBandMaxR = 12;                 // 2r - 1 <= 23 unknowns per column (the paper's
                                              // largest band, 23 for the asterisk raster)
constexpr int kBandMaxM = 8192;

struct cd {
    double x, y;
};

// Per sample: {x, y, sin pi x, cos pi x}, {sin pi y, cos pi y, phi}; phi = exp(-i pi (x + y) / N)
// has period 2 N in either coordinate, which is taken out first.
struct BandSample {
    double x, y, sx, cx, sy, cy;
    cd phi;
};

__global__ void k_band_prep(const double* __restrict__ lam, int M, int N,
                            BandSample* __restrict__ out) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= M) return;
    BandSample b;
    b.x = lam[2 * j];
    b.y = lam[2 * j + 1];
    sincospi(b.x, &b.sx, &b.cx);
    sincospi(b.y, &b.sy, &b.cy);
    const double n2 = 2.0 * N;
    const double q = fma(-n2, rint(b.x / n2), b.x) + fma(-n2, rint(b.y / n2), b.y);
    double s, c;
    sincospi(q / N, &s, &c);
    b.phi = {c, -s};
    out[j] = b;
}

// sin(pi z) for |z| <= 1/2: the Taylor series in z^2 up to z^21 (the next term is below 1e-18)
__device__ __forceinline__ double sin_pi(double z) {
    const double t = z * z;
    double p = 5.392664662608129e-10;                // (-1)^k pi^(2k+1) / (2k+1)!, k = 10..0
    p = fma(p, t, -2.2948428997269873e-08);
    p = fma(p, t, 7.952054001475513e-07);
    p = fma(p, t, -2.1915353447830217e-05);
    p = fma(p, t, 0.00046630280576761255);
    p = fma(p, t, -0.0073704309457143504);
    p = fma(p, t, 0.08214588661112823);
    p = fma(p, t, -0.5992645293207921);
    p = fma(p, t, 2.5501640398773455);
    p = fma(p, t, -5.16771278004997);
    p = fma(p, t, 3.141592653589793);
    return p * z;
}

// rho of one axis as numerator and denominator, for the lag d of two samples with the sines and
// cosines given: d = N m + d', |d'| <= N / 2; sin(pi d) = sin(pi d') by the angle difference (its
// absolute error 2e-16 is divided by N sin(pi d' / N) >= 1.5), for |d'| < 1/2 by the series (no
// cancellation); sin(pi d / N) = (-1)^m sin(pi d' / N).
__device__ __forceinline__ void rho_axis(double xj, double sj, double cj, double xa, double sa,
                                         double ca, double N, double invN, double* num,
                                         double* den) {
    const double d = xj - xa;
    const double magic = 6755399441055744.0;       // 1.5 * 2^52: rounds to an integer
    const double t = fma(d, invN, magic), dr = fma(-(t - magic), N, d);
    double n = fma(sj, ca, -(cj * sa));
    double e = N * sin_pi(dr * invN);
    // compared by the exponent bits, off the FP64 pipe
    const unsigned hi = (unsigned)__double2hiint(dr) & 0x7fffffffu;
    // lag 0, and below 2^-332 (rho differs from 1 by 1e-199 there), so that the product of the two
    // axes' factors stays a normal number
    const bool zero = hi < (1023u - 332u) << 20;
    if (hi < (1023u - 1u) << 20) n = zero ? 1.0 : sin_pi(dr);        // |dr| < 1/2
    if (zero) e = 1.0;
    *num = n;
    *den = __double2loint(t) & 1 ? -e : e;
}

// rho over the upper tile pairs: CTA (tile row, tile column >= tile row) of 32 x 32 entries,
// written as they are and transposed. While the tiles leave SMs idle, Z = 4 CTAs take 8 rows of a
// tile each: an entry is about 60 FP64 instructions, so that a whole tile is 15 us of one SM's pipe.
// Whole call at M = 100, r = 1, us: one thread per entry 101, tiles by one CTA 117, by four 97.
constexpr int kGramTile = 32;
template <int Z>
__global__ void __launch_bounds__(256)
    k_gram(const BandSample* __restrict__ smp, int M, int N, double* __restrict__ rho) {
    if (blockIdx.x < blockIdx.y) return;
    __shared__ double sa[kGramTile][7], sj[kGramTile][7], out[kGramTile][kGramTile + 1];
    const int a0 = blockIdx.y * kGramTile, j0 = blockIdx.x * kGramTile;
    if (threadIdx.x < 2 * kGramTile) {
        const int i = threadIdx.x & (kGramTile - 1);
        const int g = min(M - 1, (threadIdx.x < kGramTile ? a0 : j0) + i);
        double* o = threadIdx.x < kGramTile ? sa[i] : sj[i];
        const BandSample b = smp[g];
        o[0] = b.x; o[1] = b.sx; o[2] = b.cx; o[3] = b.y; o[4] = b.sy; o[5] = b.cy;
    }
    __syncthreads();
    const double Nd = (double)N, invN = 1.0 / N;
    const int jj = threadIdx.x & 31, ar = threadIdx.x >> 5;
    const double* q = sj[jj];
    for (int ai = ar + (Z > 1 ? 8 * blockIdx.z : 0); ai < kGramTile; ai += 8 * Z) {
        const double* p = sa[ai];
        double nx, dx, ny, dy;
        rho_axis(q[0], q[1], q[2], p[0], p[1], p[2], Nd, invN, &nx, &dx);
        rho_axis(q[3], q[4], q[5], p[3], p[4], p[5], Nd, invN, &ny, &dy);
        const double v = nx * ny / (dx * dy);
        out[ai][jj] = v;
        if (a0 + ai < M && j0 + jj < M) rho[(int64_t)(a0 + ai) * M + j0 + jj] = v;
    }
    if (blockIdx.x == blockIdx.y) return;
    __syncthreads();
    if (Z > 1 && (jj >> 3) % Z != blockIdx.z) return;      // the rows of this CTA
    for (int ji = ar; ji < kGramTile; ji += 8)
        if (j0 + ji < M && a0 + jj < M) rho[(int64_t)(j0 + ji) * M + a0 + jj] = out[jj][ji];
}

// G2[a * nb + o] = (rho^2)_{a, a+o} = sum_j rho_aj rho_{a+o,j}, o = 0..nb-1 (0 past the last
// sample). A CTA takes the ar nb <= 256 entries of ar rows, one per thread; the ar + nb - 1 rows
// are staged 64 columns at a time, so that each is read about twice instead of 2 nb times, and a
// thread adds the sums of 64 terms (blocked summation). The rows per CTA are such that a small M
// occupies the GPU too: with as many as fit, M = 100, r = 1 ran on two SMs (whole call 120 us; one warp
// per entry 103).
constexpr int kG2Cols = 64, kG2MaxRows = 64;
__global__ void __launch_bounds__(256)
    k_gram2_band(const double* __restrict__ rho, int M, int nb, int ar, double* __restrict__ G2) {
    extern __shared__ double sm_g2[];              // (ar + nb - 1) rows of kG2Cols + 1
    const int a0 = blockIdx.x * ar, rows = ar + nb - 1, ld = kG2Cols + 1;
    const int ia = threadIdx.x / nb, o = threadIdx.x - ia * nb;
    const bool on = ia < ar && a0 + ia < M;
    double sum = 0.0;
    for (int j0 = 0; j0 < M; j0 += kG2Cols) {
        __syncthreads();
        for (int i = threadIdx.x; i < rows * kG2Cols; i += 256) {
            const int r = i / kG2Cols, c = i - r * kG2Cols;
            sm_g2[r * ld + c] = a0 + r < M && j0 + c < M ? rho[(int64_t)(a0 + r) * M + j0 + c] : 0.0;
        }
        __syncthreads();
        if (on) {
            const double *p = sm_g2 + ia * ld, *q = p + o * ld;
            double part[4] = {0.0, 0.0, 0.0, 0.0};     // four chains in flight
#pragma unroll 4
            for (int c = 0; c < kG2Cols; c += 4)
#pragma unroll
                for (int k = 0; k < 4; ++k) part[k] = fma(p[c + k], q[c + k], part[k]);
            sum += (part[0] + part[1]) + (part[2] + part[3]);
        }
    }
    if (on) G2[(int64_t)(a0 + ia) * nb + o] = sum;
}

// Column k: A c' = rhs with A_il = (rho^2)_{S_i, S_l}, rhs_i = rho_{S_i, k}, S = k0..k1; Cholesky
// A = L L^T in FP64, forward and back substitution. Coefficients C[k * nc + (i - k + r - 1)] =
// conj(phi_i) c'_i phi_k for the band rows i = S; rows outside [0, M) stay zero. A status bit
// records a non-positive pivot (a column whose band is rank deficient; its coefficients stay zero).
// kSolveCols columns per block, each thread with its packed lower triangle (row i from
// i (i + 1) / 2) and right-hand side in shared memory.
constexpr int kSolveCols = 8;

__host__ __device__ constexpr int packed_len(int nc) { return nc * (nc + 1) / 2 + nc; }

__global__ void k_band_solve(const double* __restrict__ rho, const double* __restrict__ G2,
                             const BandSample* __restrict__ smp, int M, int r, int nb,
                             cd* __restrict__ C, unsigned* __restrict__ status) {
    extern __shared__ double sm_band[];
    const int k = blockIdx.x * kSolveCols + threadIdx.x;
    if (k >= M) return;
    const int nc = 2 * r - 1;
    double* L = sm_band + threadIdx.x * packed_len(nc);
    double* y = L + nc * (nc + 1) / 2;
    auto at = [&](int i, int l) -> double& { return L[i * (i + 1) / 2 + l]; };
    const int k0 = max(0, k - r + 1), k1 = min(M - 1, k + r - 1);
    const int n = k1 - k0 + 1;
    for (int i = 0; i < n; ++i)
        for (int l = 0; l <= i; ++l) at(i, l) = G2[(int64_t)(k0 + l) * nb + (i - l)];
    bool ok = true;
    for (int l = 0; l < n && ok; ++l) {
        double d = at(l, l);
        for (int m = 0; m < l; ++m) d -= at(l, m) * at(l, m);
        if (!(d > 0.0)) {
            ok = false;
            break;
        }
        const double dl = sqrt(d);
        at(l, l) = dl;
        for (int i = l + 1; i < n; ++i) {
            double v = at(i, l);
            for (int m = 0; m < l; ++m) v -= at(i, m) * at(l, m);
            at(i, l) = v / dl;
        }
    }
    cd* out = C + (int64_t)k * nc;
    for (int i = 0; i < nc; ++i) out[i] = {0.0, 0.0};
    if (!ok) {
        atomicOr(status, STATUS_BAD_WEIGHT_SUM);
        return;
    }
    for (int i = 0; i < n; ++i) {                          // L y = rhs
        double v = rho[(int64_t)(k0 + i) * M + k];         // rho_{S_i, k}
        for (int m = 0; m < i; ++m) v -= at(i, m) * y[m];
        y[i] = v / at(i, i);
    }
    for (int i = n - 1; i >= 0; --i) {                     // L^T c' = y
        double v = y[i];
        for (int m = i + 1; m < n; ++m) v -= y[m] * at(m, i);
        y[i] = v / at(i, i);
    }
    const cd pk = smp[k].phi;
    for (int i = 0; i < n; ++i) {
        const cd pi = smp[k0 + i].phi;
        out[k0 + i - k + r - 1] = {y[i] * (pk.x * pi.x + pk.y * pi.y),
                                   y[i] * (pk.y * pi.x - pk.x * pi.y)};
    }
}

}  // namespace

// tau_j = sum_k C_jk v_k over the band: column k's coefficient of row j = k + o sits at
// C[k * nc + o + r - 1]
__global__ void k_band_apply(const cd* __restrict__ C, const float2* __restrict__ v, int64_t M,
                             int r, float2* __restrict__ tau) {
    const int nc = 2 * r - 1;
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < M;
         j += (int64_t)gridDim.x * blockDim.x) {
        double sx = 0.0, sy = 0.0;
        for (int o = -(r - 1); o <= r - 1; ++o) {
            const int64_t k = j - o;
            if (k < 0 || k >= M) continue;
            const cd c = C[k * nc + o + r - 1];
            const float2 vk = v[k];
            sx += c.x * vk.x - c.y * vk.y;
            sy += c.x * vk.y + c.y * vk.x;
        }
        tau[j] = make_float2((float)sx, (float)sy);
    }
}

ftcg_status_t band_apply(const Plan& p, const void* vals, cudaStream_t s) {
    int64_t b = (p.M + 255) / 256;
    if (b > 152 * 8) b = 152 * 8;
    if (b < 1) b = 1;
    k_band_apply<<<(unsigned)b, 256, 0, s>>>(reinterpret_cast<const cd*>(p.band_c),
                                             reinterpret_cast<const float2*>(vals), p.M,
                                             p.band_r, reinterpret_cast<float2*>(p.band_tau));
    FTCG_CK(cudaGetLastError());
    return FTCG_SUCCESS;
}

void release_band(Plan* p) {
    if (p->band_c) cudaFree(p->band_c);
    if (p->band_tau) cudaFree(p->band_tau);
    p->band_c = nullptr;
    p->band_tau = nullptr;
    p->band_r = 0;
}

}  // namespace ftcg

using namespace ftcg;

extern "C" ftcg_status_t ftcg_band(ftcg_plan_t plan, int32_t r, void* d_coef_out,
                                   ftcg_stream_t stream) {
    FTCG_API_BEGIN
    clear_error();
    if (!plan) {
        set_error("ftcg_band: plan is NULL");
        return FTCG_ERR_INVALID_VALUE;
    }
    Plan* p = reinterpret_cast<Plan*>(plan);
    if (r < 1 || r > kBandMaxR) {
        set_error("ftcg_band: r must be in 1..%d", kBandMaxR);
        return FTCG_ERR_INVALID_VALUE;
    }
    if (p->M > kBandMaxM) {
        set_error("ftcg_band: M = %lld > %d: the exact band costs O(M^2 r) and 8 M^2 bytes",
                  (long long)p->M, kBandMaxM);
        return FTCG_ERR_NOT_SUPPORTED;
    }
    if (p->opts.precision != FTCG_PREC_FP32) {
        set_error("ftcg_band: needs an FP32 plan");
        return FTCG_ERR_NOT_SUPPORTED;
    }
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    p->last_stream = s;
    const int M = (int)p->M;
    release_band(p);
    if (M == 0) return FTCG_SUCCESS;
    const int nc = 2 * r - 1, nb = 2 * r - 1;      // unknowns per column, offsets of T^2
    BandSample* smp = nullptr;                     // then rho and G2: one allocation
    cd* C = nullptr;
    FTCG_CK(pool_malloc(&smp, (size_t)M * sizeof(BandSample) +
                                  ((size_t)M * M + (size_t)M * nb) * sizeof(double), s));
    double* rho = reinterpret_cast<double*>(smp + M);
    double* G2 = rho + (size_t)M * M;
    FTCG_CK(pool_malloc(&C, (size_t)M * nc * sizeof(cd), s));
    p->band_c = C;
    FTCG_CK(pool_malloc(&p->band_tau, (size_t)M * sizeof(float2), s));
    p->band_r = r;
    k_band_prep<<<(M + 127) / 128, 128, 0, s>>>(p->lambda, M, p->N, smp);
    const int nt = (M + kGramTile - 1) / kGramTile;
    int dev = 0, sms = 0;
    FTCG_CK(cudaGetDevice(&dev));
    FTCG_CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    if (nt * (nt + 1) / 2 < sms)
        k_gram<4><<<dim3(nt, nt, 4), 256, 0, s>>>(smp, M, p->N, rho);
    else
        k_gram<1><<<dim3(nt, nt), 256, 0, s>>>(smp, M, p->N, rho);
    const int ar = std::min(std::min(kG2MaxRows, 256 / nb), std::max(4, (M + sms - 1) / sms));
    k_gram2_band<<<(M + ar - 1) / ar, 256, (size_t)(ar + nb - 1) * (kG2Cols + 1) * sizeof(double),
                   s>>>(rho, M, nb, ar, G2);
    const size_t sm = (size_t)kSolveCols * packed_len(nc) * sizeof(double);
    k_band_solve<<<(M + kSolveCols - 1) / kSolveCols, kSolveCols, sm, s>>>(rho, G2, smp, M, r, nb, C,
                                                                           p->status);
    FTCG_CK(cudaGetLastError());
    if (d_coef_out)
        FTCG_CK(cudaMemcpyAsync(d_coef_out, C, (size_t)M * nc * sizeof(cd),
                                cudaMemcpyDeviceToDevice, s));
    FTCG_CK(pool_free(smp, s));
    // C replaces the diagonal weights: spread tau = C v with unit weights
    FTCG_TRY(launch_set_alpha(*p, nullptr, FTCG_WEIGHTS_F64, s));
    p->band_r = r;
    unsigned st = 0;
    FTCG_CK(cudaMemcpyAsync(&st, p->status, sizeof(unsigned), cudaMemcpyDeviceToHost, s));
    FTCG_CK(cudaStreamSynchronize(s));
    if (st & STATUS_BAD_WEIGHT_SUM) {
        FTCG_CK(cudaMemsetAsync(p->status, 0, sizeof(unsigned), s));
        set_error("ftcg_band: a column's band normal matrix is not positive definite (its "
                  "coefficients are set to zero)");
        return FTCG_ERR_NUMERIC;
    }
    return FTCG_SUCCESS;
    FTCG_API_END
}
