// The frame approximation on the device (Sec. III-B, Eq. afr / afrm; 2-D: Eq. twodframe,
// twodframeB): the minimum-norm least-squares image x = E^+ v of the data frame
// E_jp = exp(-2 pi i lambda_j . p / N), computed by CGLS (conjugate gradients on the normal
// equations, Hestenes-Stiefel form) with the plan's gridded operators standing in for E
// (ftcg_forward) and E^H (ftcg_adjoint). Optional row weights w_j (for example the FTCG weights)
// turn the problem into min || W^(1/2) (E x - v) ||: started from zero, the first iterate is a
// multiple of E^H W v, the FTCG image, and the FTCG weights act as a preconditioner (Sec. V-C's
// condition numbers of Psi and C_2).
//
// Vectors are FP32 complex (the operators' precision); the scalars of the recursion (the squared
// norms gamma_k = ||E^H W r||^2 and ||W^(1/2) E p||^2) are FP64 device reductions into one slot per
// iteration, so that nothing is reset or rotated between iterations, and the step
// lengths are formed on the device from them, so an iteration queues its kernels without any
// host synchronisation; the host reads the residual history once at the end. Small problems are
// bound by the number of kernels in the chain (four of this file's per iteration, overlapped by
// programmatic dependent launch; with six, a pass to scale q and scalars reset in between, ten
// iterations at N = 256, 80 k samples took 892 us, now 715). An iteration whose
// gamma has fallen to tol^2 gamma_0 (or whose search direction vanished) freezes the iterate.

#include <cmath>
#include <vector>

#include "ftcg_internal.cuh"

namespace ftcg {

namespace {

constexpr int kThreads = 256;

// device scalars of the recursion, iters + 1 of each: gamma after iteration k, the new squared
// residual that iteration k found, and ||W^(1/2) E p||^2 of iteration k
struct Scalars {
    double *gamma, *fresh, *qq;
    double tol2;
    // iteration k leaves x and p as they are: converged before it, or its direction vanished
    __device__ __forceinline__ bool frozen(int k) const {
        return !(gamma[k - 1] > tol2 * gamma[0]) || !(qq[k] > 0.0);
    }
};

int blocks_for(int64_t n) {
    int64_t b = (n + kThreads - 1) / kThreads;
    if (b < 1) b = 1;
    if (b > 152 * 8) b = 152 * 8;
    return (int)b;
}

__device__ __forceinline__ double block_sum(double v) {
    __shared__ double part[kThreads / 32];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x < 32) {
        s = threadIdx.x < kThreads / 32 ? part[threadIdx.x] : 0.0;
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    }
    return s;                                   // valid in thread 0
}

// sw_j = sqrt(w_j) (1 without weights); r = sw v
__global__ void k_init(const float2* __restrict__ v, const double* __restrict__ w, int64_t M,
                       float* __restrict__ sw, float2* __restrict__ r) {
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < M;
         j += (int64_t)gridDim.x * blockDim.x) {
        const float s = w ? (float)sqrt(w[j]) : 1.0f;
        sw[j] = s;
        r[j] = make_float2(s * v[j].x, s * v[j].y);
    }
}

// out += sum |sw x|^2 (sw may be null)
__global__ void k_norm2(const float2* __restrict__ x, const float* __restrict__ sw, int64_t n,
                        double* __restrict__ out) {
    pdl_wait();
    pdl_allow_next();
    double acc = 0.0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        float2 a = x[i];
        if (sw) {
            a.x *= sw[i];
            a.y *= sw[i];
        }
        acc += (double)a.x * a.x + (double)a.y * a.y;
    }
    acc = block_sum(acc);
    if (threadIdx.x == 0) atomicAdd(out, acc);
}

// x += a p over the image, r -= a sw q over the samples, a = gamma / qq (0 once frozen)
__global__ void k_step(float2* __restrict__ x, const float2* __restrict__ p, int64_t nimg,
                       float2* __restrict__ r, const float2* __restrict__ q,
                       const float* __restrict__ sw, int64_t M, const Scalars sc, int k) {
    pdl_wait();
    pdl_allow_next();
    const float a = sc.frozen(k) ? 0.0f : (float)(sc.gamma[k - 1] / sc.qq[k]);
    const int64_t n = nimg > M ? nimg : M;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        if (i < nimg) {
            const float2 pi = p[i];
            float2 xi = x[i];
            xi.x = fmaf(a, pi.x, xi.x);
            xi.y = fmaf(a, pi.y, xi.y);
            x[i] = xi;
        }
        if (i < M) {
            const float2 qi = q[i];
            const float s = sw[i];
            float2 ri = r[i];
            ri.x = fmaf(-a, __fmul_rn(s, qi.x), ri.x);
            ri.y = fmaf(-a, __fmul_rn(s, qi.y), ri.y);
            r[i] = ri;
        }
    }
}

// p = s + (gamma_new / gamma) p (p unchanged once frozen); gamma after iteration k
__global__ void k_direction(const float2* __restrict__ s, float2* __restrict__ p, int64_t n,
                            const Scalars sc, int k) {
    pdl_wait();
    pdl_allow_next();
    const bool fz = sc.frozen(k);
    if (blockIdx.x == 0 && threadIdx.x == 0) sc.gamma[k] = fz ? sc.gamma[k - 1] : sc.fresh[k];
    if (fz) return;
    const float beta = (float)(sc.fresh[k] / sc.gamma[k - 1]);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const float2 si = s[i];
        float2 pi = p[i];
        pi.x = fmaf(beta, pi.x, si.x);
        pi.y = fmaf(beta, pi.y, si.y);
        p[i] = pi;
    }
}

}  // namespace

}  // namespace ftcg

using namespace ftcg;

extern "C" ftcg_status_t ftcg_cgls(ftcg_plan_t plan, const void* d_values,
                                   const double* d_row_weights, int32_t iters, double tol,
                                   void* d_image, double* h_resnorms, int32_t* h_iters,
                                   ftcg_stream_t stream) {
    FTCG_API_BEGIN
    clear_error();
    if (!plan || !d_image) {
        set_error("ftcg_cgls: plan or image is NULL");
        return FTCG_ERR_INVALID_VALUE;
    }
    Plan* p = reinterpret_cast<Plan*>(plan);
    if (p->M > 0 && !d_values) {
        set_error("ftcg_cgls: values pointer is NULL");
        return FTCG_ERR_INVALID_VALUE;
    }
    if (iters < 0 || iters > 100000 || !(tol >= 0.0) || !std::isfinite(tol)) {
        set_error("ftcg_cgls: iters must be in 0..100000 and tol >= 0");
        return FTCG_ERR_INVALID_VALUE;
    }
    if (p->opts.precision != FTCG_PREC_FP32) {
        set_error("ftcg_cgls: needs an FP32 plan (the row weights are applied in FP32)");
        return FTCG_ERR_NOT_SUPPORTED;
    }
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    p->last_stream = s;
    const int64_t M = p->M, nimg = (int64_t)p->N * p->N;
    float2* x = reinterpret_cast<float2*>(d_image);
    FTCG_CK(cudaMemsetAsync(x, 0, nimg * sizeof(float2), s));
    if (M == 0) {
        if (h_resnorms)
            for (int k = 0; k <= iters; ++k) h_resnorms[k] = 0.0;
        if (h_iters) *h_iters = 0;
        return FTCG_SUCCESS;
    }
    float *sw = nullptr;
    float2 *r = nullptr, *q = nullptr, *sv = nullptr, *pv = nullptr;
    double* slots = nullptr;                       // three of iters + 1
    FTCG_CK(pool_malloc(&sw, M * sizeof(float), s));
    FTCG_CK(pool_malloc(&r, M * sizeof(float2), s));
    FTCG_CK(pool_malloc(&q, M * sizeof(float2), s));
    FTCG_CK(pool_malloc(&sv, nimg * sizeof(float2), s));
    FTCG_CK(pool_malloc(&pv, nimg * sizeof(float2), s));
    const size_t ns = (size_t)iters + 1;
    FTCG_CK(pool_malloc(&slots, 3 * ns * sizeof(double), s));
    FTCG_CK(cudaMemsetAsync(slots, 0, 3 * ns * sizeof(double), s));
    const Scalars sc{slots, slots + ns, slots + 2 * ns, tol * tol};
    ftcg_status_t st = FTCG_SUCCESS;
    auto norm2 = [&](const float2* v, const float* w, int64_t n, double* out) {
        return launch_pdl(k_norm2, dim3(blocks_for(n)), dim3(kThreads), 0, s, v, w, n, out);
    };
    auto run = [&]() -> ftcg_status_t {
        k_init<<<blocks_for(M), kThreads, 0, s>>>(reinterpret_cast<const float2*>(d_values),
                                                 d_row_weights, M, sw, r);
        FTCG_CK(cudaGetLastError());
        // the plan's adjoint spreads with its installed weights: sw for the iteration, so that
        // adjoint(r) = E^H (sw r)
        FTCG_TRY(install_alpha(*p, sw, FTCG_WEIGHTS_F32, s));
        FTCG_TRY(adjoint_device(p, r, FTCG_VALUES_C64, pv, s, false));   // p = E^H W v
        FTCG_CK(norm2(pv, nullptr, nimg, sc.gamma));
        for (int k = 1; k <= iters; ++k) {
            FTCG_TRY(forward_device(p, pv, q, s));                       // q = E p
            FTCG_CK(norm2(q, sw, M, sc.qq + k));
            FTCG_CK(launch_pdl(k_step, dim3(blocks_for(nimg > M ? nimg : M)), dim3(kThreads), 0, s,
                               x, (const float2*)pv, nimg, r, (const float2*)q, (const float*)sw, M,
                               sc, k));
            FTCG_TRY(adjoint_device(p, r, FTCG_VALUES_C64, sv, s, false));   // s = E^H (sw r)
            FTCG_CK(norm2(sv, nullptr, nimg, sc.fresh + k));
            FTCG_CK(launch_pdl(k_direction, dim3(blocks_for(nimg)), dim3(kThreads), 0, s,
                               (const float2*)sv, pv, nimg, sc, k));
        }
        return FTCG_SUCCESS;
    };
    st = run();
    // restore the plan's own weights whatever happened above
    ftcg_status_t rs = install_alpha(*p, p->alpha_cur, FTCG_WEIGHTS_F32, s);
    if (st == FTCG_SUCCESS) st = rs;
    std::vector<double> h(iters + 1, 0.0);
    if (st == FTCG_SUCCESS) {
        cudaError_t ce = cudaMemcpyAsync(h.data(), sc.gamma, (iters + 1) * sizeof(double),
                                         cudaMemcpyDeviceToHost, s);
        if (ce == cudaSuccess) ce = cudaStreamSynchronize(s);
        if (ce != cudaSuccess) {
            set_error("ftcg_cgls: reading the residual history: %s", cudaGetErrorString(ce));
            st = FTCG_ERR_CUDA;
        }
        for (double& g : h) g = std::sqrt(g);
    }
    pool_free(sw, s);
    pool_free(r, s);
    pool_free(q, s);
    pool_free(sv, s);
    pool_free(pv, s);
    pool_free(slots, s);
    if (st != FTCG_SUCCESS) return st;
    int done = iters;
    for (int k = 0; k <= iters; ++k)
        if (!(h[k] > tol * h[0])) {
            done = k;
            break;
        }
    if (h_resnorms)
        for (int k = 0; k <= iters; ++k) h_resnorms[k] = h[k];
    if (h_iters) *h_iters = done;
    return FTCG_SUCCESS;
    FTCG_API_END
}
