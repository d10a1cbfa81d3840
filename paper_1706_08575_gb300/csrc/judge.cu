// The exact judge of predicted weights (spec extension (4): the exact construction stays as
// fallback and judge). For K samples spread over the acquisition order the exact weight sum
// S_k = sum_j F_N(lambda_jx - lambda_kx) F_N(lambda_jy - lambda_ky) (Eq. difopt at r = 1; F_N the
// normalised Fejer kernel sin^2(pi d) / (N^2 sin^2(pi d / N))) is summed directly over all M
// samples. The ratios alpha_pred S_k estimate the predicted weights' error: their median is a
// per-ping calibration factor (a global density factor that local features cannot see), and the
// spread of the calibrated ratios around 1 estimates the remaining relative weight error, which
// the image error follows. Within the caller's bound the calibrated predictions are installed;
// otherwise the exact FP64 weights (ftcg_weights) are computed and installed instead.
//
// The sums are the judge's whole cost (K M terms), so they avoid FP64 arithmetic, which runs at a
// small fraction of the FP32 rate here. Each coordinate is first reduced once, in FP64, modulo N
// (F_N has period N) and split into an integer n and a fraction f in [-1/2, 1/2], rounded to FP32.
// A lag d = lambda_j - lambda_k is then the exact integer n_j - n_k, wrapped into [-N/2, N/2], plus
// the FP32 difference f_j - f_k: its absolute error is a few 1e-8 at any distance, and F_N is
// smooth on that scale (near d = 0 both sines of the quotient carry the same relative error).
// sin(pi d) = +-sin(pi (f_j - f_k)) since the integer part only flips the sign; a term is then
// the square of sin(pi df_x) sin(pi df_y) / (N^2 sin(pi d_x / N) sin(pi d_y / N)) in FP32, a few
// ulps, with the sines as polynomials on [-1/2, 1/2]. Each thread sums its terms in FP32 with
// Kahan compensation; the threads' sums are combined in FP64. Samples with a non-finite or huge
// coordinate are left out of the sums (as the gridding leaves them out), and a judged sample of
// that kind gets S = NaN, which the verdict skips.

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <vector>

#include "ftcg_internal.cuh"

namespace ftcg {

namespace {

constexpr int kJudgeThreads = 256;
constexpr float kJudgeSkip = 1e30f;        // n of a sample left out of the sums
constexpr int kJudgeCols = 4;              // judged samples per block

// Per sample {n_x, n_y, f_x, f_y}: lambda mod N = n + f, n an integer (|n| <= N / 2, exact in FP32).
__global__ void k_judge_prep(const double* __restrict__ lam, int64_t M, int N,
                             float4* __restrict__ pts) {
    const double invN = 1.0 / N;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < M;
         i += (int64_t)gridDim.x * blockDim.x) {
        float n[2], f[2];
        bool ok = true;
        for (int a = 0; a < 2; ++a) {
            const double x = lam[2 * i + a];
            ok = ok && isfinite(x) && fabs(x) < 1099511627776.0;     // 2^40
            const double r = ok ? x - N * rint(x * invN) : 0.0;      // |r| <= N/2 (+ rounding)
            const double q = rint(r);
            n[a] = (float)q;
            f[a] = (float)(r - q);
        }
        pts[i] = ok ? make_float4(n[0], n[1], f[0], f[1])
                    : make_float4(kJudgeSkip, kJudgeSkip, 0.f, 0.f);
    }
}

// sin(pi x) for |x| <= 1/2: x P(x^2), P interpolating sin(pi x) / x at the five Chebyshev points of
// x^2 in [0, 1/4] (4e-9 relative); the leading coefficient split so that its rounding drops out
__device__ __forceinline__ float sin_pi32(float x) {
    const float t = x * x;
    float q = fmaf(t, 0.07765591227601387f, -0.5982904112834275f);
    q = fmaf(t, q, 2.550077386528912f);
    q = fmaf(t, q, -5.167710076668315f);
    q = fmaf(t, q, 0.0009676400772034f);           // 3.1415926400772034 - 3.140625
    return fmaf(x, 3.140625f, x * q);
}

// One axis of F_N^(1/2) for the lag dn + df (dn an integer, |dn| <= N, |df| <= 1), up to sign:
// numerator sin(pi df), denominator sin(pi d / N); (1, 1 / N) at lag 0 and below 1e-12 (F_N differs
// from 1 by 3e-24 there), so that no product of the two axes' factors leaves the normal FP32 range.
__device__ __forceinline__ void fejer_axis(float dn, float df, float N, float invN, float* num,
                                           float* den) {
    if (fabsf(dn) > 0.5f * N) dn -= copysignf(N, dn);
    float dr = dn + df;
    if (fabsf(dr) > 0.5f * N) dr -= copysignf(N, dr);    // exact (Sterbenz); now |dr| <= N/2
    const float magic = 12582912.0f;                     // 1.5 * 2^23: rounds to an integer
    const float fr = df - ((df + magic) - magic);        // sin(pi df) up to sign, |fr| <= 1/2
    const bool zero = fabsf(dr) < 1e-12f;
    *num = zero ? 1.0f : sin_pi32(fr);
    *den = zero ? invN : sin_pi32(dr * invN);
}

// Block (b, p): the sums over part p of the samples of judged samples 4 b .. 4 b + 3, so that a
// sample's record is loaded once per four terms and the launch fills the GPU whatever K is. Bound:
// instruction issue (FP32). One block per judged sample with sinpif and two divisions a term took
// 625 us for K = 256, M = 211,250 (54 M terms); this 153.
__global__ void __launch_bounds__(kJudgeThreads)
    k_fejer_sums(const float4* __restrict__ pts, int64_t M, int N, int K, int64_t per,
                 double* __restrict__ part) {
    float4 pk[kJudgeCols];
    float s[kJudgeCols], c[kJudgeCols];                  // Kahan sums and their compensations
#pragma unroll
    for (int i = 0; i < kJudgeCols; ++i) {
        const int64_t k = min(K - 1, (int)blockIdx.x * kJudgeCols + i);
        pk[i] = pts[(k * 2 + 1) * M / (2 * (int64_t)K)];
        s[i] = c[i] = 0.0f;
    }
    const float Nf = (float)N, invN = 1.0f / Nf, invN2 = invN * invN;
    const int64_t j1 = min(M, (blockIdx.y + 1) * per);
    for (int64_t j = blockIdx.y * per + threadIdx.x; j < j1; j += kJudgeThreads) {
        const float4 q = pts[j];
        if (q.x == kJudgeSkip) continue;
#pragma unroll
        for (int i = 0; i < kJudgeCols; ++i) {
            float nx, dx, ny, dy;
            fejer_axis(q.x - pk[i].x, q.z - pk[i].z, Nf, invN, &nx, &dx);
            fejer_axis(q.y - pk[i].y, q.w - pk[i].w, Nf, invN, &ny, &dy);
            const float r = (nx * ny) * invN2 / (dx * dy);
            const float y = fmaf(r, r, -c[i]);
            const float u = s[i] + y;
            c[i] = (u - s[i]) - y;
            s[i] = u;
        }
    }
    __shared__ double sum[kJudgeCols][kJudgeThreads / 32];
#pragma unroll
    for (int i = 0; i < kJudgeCols; ++i) {
        double acc = (double)s[i] - (double)c[i];
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if ((threadIdx.x & 31) == 0) sum[i][threadIdx.x >> 5] = acc;
    }
    __syncthreads();
    const int i = threadIdx.x, k = blockIdx.x * kJudgeCols + i;
    if (i < kJudgeCols && k < K) {
        double t = 0.0;
        for (int w = 0; w < kJudgeThreads / 32; ++w) t += sum[i][w];
        part[(int64_t)blockIdx.y * K + k] = t;
    }
}

// S_k from its parts, in order (NaN for a judged sample that is left out), and alpha_pred there
__global__ void k_judge_finish(const double* __restrict__ part, int parts,
                               const float4* __restrict__ pts, const double* __restrict__ alpha,
                               int64_t M, int K, double* __restrict__ S, double* __restrict__ a) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= K) return;
    const int64_t j = ((int64_t)i * 2 + 1) * M / (2 * (int64_t)K);
    double t = 0.0;
    for (int p = 0; p < parts; ++p) t += part[(int64_t)p * K + i];
    S[i] = pts[j].x == kJudgeSkip ? __longlong_as_double(0x7ff8000000000000LL) : t;
    a[i] = alpha[j];
}

__global__ void k_scale_alpha(const double* __restrict__ a, int64_t M, double s,
                              double* __restrict__ out) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < M;
         i += (int64_t)gridDim.x * blockDim.x)
        out[i] = a[i] * s;
}

}  // namespace

// Launch the judge's sums for one plan (asynchronous): d_S (K) and d_a (K) the predicted weights
// at the same samples.
ftcg_status_t judge_launch(const Plan& p, const double* d_alpha, int K, double* d_S,
                           double* d_a, cudaStream_t s) {
    // parts: about eight blocks per SM, at least 1024 samples each (and a whole number of strides)
    const int kb = (K + kJudgeCols - 1) / kJudgeCols;
    int dev = 0, sms = 0;
    FTCG_CK(cudaGetDevice(&dev));
    FTCG_CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const int64_t want = std::max<int64_t>(1, (8 * (int64_t)sms + kb - 1) / kb);
    int64_t per = std::max<int64_t>(1024, (p.M + want - 1) / want);
    per = (per + kJudgeThreads - 1) / kJudgeThreads * kJudgeThreads;
    const int parts = (int)((p.M + per - 1) / per);
    float4* pts = nullptr;
    double* part = nullptr;
    FTCG_CK(pool_malloc(&pts, (size_t)p.M * sizeof(float4), s));
    const cudaError_t got = pool_malloc(&part, (size_t)parts * K * sizeof(double), s);
    if (got != cudaSuccess) {
        pool_free(pts, s);
        FTCG_CK(got);
    }
    const int64_t b = std::min<int64_t>((p.M + 255) / 256, 152 * 8);
    k_judge_prep<<<(unsigned)std::max<int64_t>(1, b), 256, 0, s>>>(p.lambda, p.M, p.N, pts);
    k_fejer_sums<<<dim3(kb, parts), kJudgeThreads, 0, s>>>(pts, p.M, p.N, K, per, part);
    k_judge_finish<<<(K + 127) / 128, 128, 0, s>>>(part, parts, pts, d_alpha, p.M, K, d_S, d_a);
    const cudaError_t launched = cudaGetLastError();
    pool_free(part, s);
    FTCG_CK(pool_free(pts, s));
    FTCG_CK(launched);
    return FTCG_SUCCESS;
}

// Decide from the host copies of S and alpha_pred: stats = {median ratio, rms and max of the
// calibrated relative errors}; true when the rms is within max_rel_err.
bool judge_decide(const double* S, const double* a, int K, double max_rel_err, double* stats) {
    std::vector<double> r;
    r.reserve(K);
    for (int i = 0; i < K; ++i) {
        const double q = a[i] * S[i];                         // alpha_pred / alpha_exact
        if (std::isfinite(q)) r.push_back(q);                 // samples left out: S = NaN
    }
    if (r.empty()) {
        stats[0] = stats[1] = stats[2] = std::nan("");
        return false;
    }
    const size_t n = r.size();
    std::vector<double> sorted(r);
    std::sort(sorted.begin(), sorted.end());
    const double med = n % 2 ? sorted[n / 2] : 0.5 * (sorted[n / 2 - 1] + sorted[n / 2]);
    double ss = 0.0, mx = 0.0;
    for (double q : r) {
        const double e = q / med - 1.0;
        ss += e * e;
        mx = std::max(mx, std::fabs(e));
    }
    const double rms = std::sqrt(ss / n);
    stats[0] = med;
    stats[1] = rms;
    stats[2] = mx;
    return std::isfinite(med) && med > 0.0 && rms <= max_rel_err;
}

// Install the verdict: the calibrated predictions (alpha_pred / median) or the exact weights.
ftcg_status_t judge_install(Plan& p, const double* d_alpha, bool accept, double med,
                            cudaStream_t s) {
    release_band(&p);
    if (!accept) return compute_weights(p, nullptr, s);
    double* tmp = nullptr;
    FTCG_CK(pool_malloc(&tmp, (size_t)p.M * sizeof(double), s));
    int64_t b = std::min<int64_t>((p.M + 255) / 256, 152 * 8);
    k_scale_alpha<<<(unsigned)std::max<int64_t>(1, b), 256, 0, s>>>(d_alpha, p.M, 1.0 / med,
                                                                    tmp);
    FTCG_CK(cudaGetLastError());
    ftcg_status_t st = launch_set_alpha(p, tmp, FTCG_WEIGHTS_F64, s);
    FTCG_CK(pool_free(tmp, s));
    return st;
}

}  // namespace ftcg

using namespace ftcg;

extern "C" ftcg_status_t ftcg_weights_judge(ftcg_plan_t plan, const double* d_alpha, int32_t K,
                                            double max_rel_err, int32_t* h_accepted,
                                            double* h_stats, ftcg_stream_t stream) {
    FTCG_API_BEGIN
    clear_error();
    if (!plan || !d_alpha) {
        set_error("ftcg_weights_judge: plan or weights NULL");
        return FTCG_ERR_INVALID_VALUE;
    }
    Plan* p = reinterpret_cast<Plan*>(plan);
    if (K < 1 || K > 65536 || K > p->M || !(max_rel_err >= 0.0)) {
        set_error("ftcg_weights_judge: K must be in 1..min(M, 65536) and max_rel_err >= 0");
        return FTCG_ERR_INVALID_VALUE;
    }
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    p->last_stream = s;
    double *dS = nullptr, *da = nullptr;
    FTCG_CK(pool_malloc(&dS, (size_t)2 * K * sizeof(double), s));
    da = dS + K;
    const ftcg_status_t launched = judge_launch(*p, d_alpha, K, dS, da, s);
    if (launched != FTCG_SUCCESS) {
        pool_free(dS, s);
        return launched;
    }
    std::vector<double> h(2 * (size_t)K);
    FTCG_CK(cudaMemcpyAsync(h.data(), dS, 2 * (size_t)K * sizeof(double), cudaMemcpyDeviceToHost,
                            s));
    FTCG_CK(cudaStreamSynchronize(s));
    FTCG_CK(pool_free(dS, s));
    double stats[3];
    const bool ok = judge_decide(h.data(), h.data() + K, K, max_rel_err, stats);
    if (h_stats)
        for (int i = 0; i < 3; ++i) h_stats[i] = stats[i];
    if (h_accepted) *h_accepted = ok ? 1 : 0;
    return judge_install(*p, d_alpha, ok, stats[0], s);
    FTCG_API_END
}
