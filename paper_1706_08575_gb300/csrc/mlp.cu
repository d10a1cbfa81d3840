// Learned FTCG weights: a small MLP predicts each sample's diagonal weight (Eq. difopt at r = 1)
// from its local k-space neighbourhood, so that the expensive exact construction is not needed
// per ping. The exact weights stay available (ftcg_weights) as the training labels and the judge.
//
// Features of sample k: the offsets lambda_j - lambda_k of its 16 nearest other samples (ordered
// by distance, ties by index; 32 values) and one caller-supplied scalar (the normalised range
// wavenumber), stored as 48 bfloat16 (zero padded to three k-steps of 16).
// Network: 33 -> 64 -> 64 -> 64 -> 1 with the tanh form of GELU; output y = log alpha.
//
// kNN: the samples are hashed into square cells of side h (about two samples per cell) by a
// counting sort; the query searches rings of cells around its own, keeping the best 16 (distance,
// index) pairs, and stops after ring r once the 16th distance is below r h (no unvisited sample can
// be closer), so the neighbour sets are exact.
// MLP: BF16 tensor-core mma.sync m16n8k16 with FP32 accumulation; one warp owns 16 rows, and the
// FP32 accumulator fragment of one layer is repacked in registers as the A fragment of the next.
// Training: one kernel per step runs forward, backward and the weight gradients of 64 rows at a time
// without leaving shared memory, and writes per-CTA partial gradients; a second one sums them in a
// fixed order and applies Adam to an FP32 master copy.

#include <cmath>
#include <cstring>
#include <map>
#include <mutex>
#include <new>
#include <vector>

#include "ftcg_internal.cuh"

namespace ftcg {
namespace {

constexpr int kNb = 16;                 // neighbours
constexpr int kIn = 2 * kNb + 1;        // 33 inputs
constexpr int kInPad = 48;              // three k-steps of 16
constexpr int kHid = 64;
constexpr int kLd1 = kInPad + 8;        // shared-memory row strides (bank-conflict padding)
constexpr int kLdH = kHid + 8;
// packed FP32 parameters: W1 [33][64], b1, W2 [64][64], b2, W3 [64][64], b3, w4 [64], b4
constexpr int oW1 = 0, ob1 = oW1 + kIn * kHid, oW2 = ob1 + kHid, ob2 = oW2 + kHid * kHid;
constexpr int oW3 = ob2 + kHid, ob3 = oW3 + kHid * kHid, ow4 = ob3 + kHid, ob4 = ow4 + kHid;
constexpr int kParams = ob4 + 1;        // 10561

// ---------------------------------------------------------------------------------------------
// kNN features
// ---------------------------------------------------------------------------------------------
__global__ void k_bbox(const double* __restrict__ lam, int64_t M, double* __restrict__ out) {
    __shared__ double s[4][256];
    double mnx = 1e300, mny = 1e300, mxx = -1e300, mxy = -1e300;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < M;
         i += (int64_t)gridDim.x * blockDim.x) {
        const double x = lam[2 * i], y = lam[2 * i + 1];
        mnx = fmin(mnx, x); mny = fmin(mny, y); mxx = fmax(mxx, x); mxy = fmax(mxy, y);
        if (isnan(x) || isnan(y)) mxx = INFINITY;   // fmin / fmax skip NaN: make it visible
    }
    s[0][threadIdx.x] = mnx; s[1][threadIdx.x] = mny; s[2][threadIdx.x] = mxx; s[3][threadIdx.x] = mxy;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) {
            s[0][threadIdx.x] = fmin(s[0][threadIdx.x], s[0][threadIdx.x + o]);
            s[1][threadIdx.x] = fmin(s[1][threadIdx.x], s[1][threadIdx.x + o]);
            s[2][threadIdx.x] = fmax(s[2][threadIdx.x], s[2][threadIdx.x + o]);
            s[3][threadIdx.x] = fmax(s[3][threadIdx.x], s[3][threadIdx.x + o]);
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        out[4 * blockIdx.x + 0] = s[0][0];
        out[4 * blockIdx.x + 1] = s[1][0];
        out[4 * blockIdx.x + 2] = s[2][0];
        out[4 * blockIdx.x + 3] = s[3][0];
    }
}

struct Hash {
    double x0, y0, h, inv_h;
    int nx, ny;
};

__device__ __forceinline__ int cell_of(double v, double v0, double inv_h, int n) {
    int c = (int)floor((v - v0) * inv_h);
    return c < 0 ? 0 : (c >= n ? n - 1 : c);
}

__global__ void k_cell_count(const double* __restrict__ lam, int64_t M, Hash hs,
                             int* __restrict__ cnt, int* __restrict__ cell) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < M;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int cx = cell_of(lam[2 * i], hs.x0, hs.inv_h, hs.nx);
        const int cy = cell_of(lam[2 * i + 1], hs.y0, hs.inv_h, hs.ny);
        const int c = cy * hs.nx + cx;
        cell[i] = c;
        atomicAdd(cnt + c, 1);
    }
}

__global__ void k_cell_scatter(int64_t M, const int* __restrict__ cell, int* __restrict__ cursor,
                               int* __restrict__ sorted) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < M;
         i += (int64_t)gridDim.x * blockDim.x)
        sorted[atomicAdd(cursor + cell[i], 1)] = (int)i;
}

// Sorted copies of the coordinates: pts[s] = lambda_{sorted[s]} (FP64) and pts32[s] = the same
// relative to the bounding-box corner, rounded to FP32 (for the candidate filter).
__global__ void k_gather_pts(const double* __restrict__ lam, int64_t M, const int* __restrict__ sorted,
                             double x0, double y0, double2* __restrict__ pts,
                             float2* __restrict__ pts32) {
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < M;
         s += (int64_t)gridDim.x * blockDim.x) {
        const int j = sorted[s];
        const double x = lam[2 * j], y = lam[2 * j + 1];
        pts[s] = make_double2(x, y);
        pts32[s] = make_float2((float)(x - x0), (float)(y - y0));
    }
}

// Exact 16 nearest neighbours, one thread per query, queries in cell order (a warp's queries are
// neighbours). The ring search visits cells at Chebyshev distance r = 0, 1, ... and stops once the
// 16th best squared distance is below (r h)^2. A candidate is first tested in FP32 against the
// current 16th distance d16 with the slack T(d16) = 2^-16 d16 + 4 e sqrt(d16) + 4 e^2, where
// e bounds the FP32 offset error (2^-24 of twice the bounding-box extent): a candidate whose FP32
// distance exceeds d16 + T cannot beat d16 exactly. The others get the FP64 distance
// (dx dx + dy dy, rounded like the brute force) and enter the list, ordered by (distance, index);
// distances are compared as the integer images of their non-negative FP64 bit patterns.
__global__ void __launch_bounds__(128)
    k_knn(const double* __restrict__ lam, const double* __restrict__ aux, int64_t M, Hash hs,
          const int* __restrict__ start, const int* __restrict__ sorted,
          const double2* __restrict__ pts, const float2* __restrict__ pts32, float err,
          __nv_bfloat16* __restrict__ feat, int* __restrict__ nbr, bool vec) {
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < M;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int i = sorted[t];
        const double2 pi = pts[t];
        const float2 qi = pts32[t];
        const int cx = cell_of(pi.x, hs.x0, hs.inv_h, hs.nx);
        const int cy = cell_of(pi.y, hs.y0, hs.inv_h, hs.ny);
        unsigned long long bk[kNb];
        int bj[kNb];
#pragma unroll
        for (int k = 0; k < kNb; ++k) {
            bk[k] = ~0ull;
            bj[k] = 0x7fffffff;
        }
        float thr = INFINITY;
        const int rmax = max(hs.nx, hs.ny);
        for (int r = 0; r <= rmax; ++r) {
            for (int dy = -r; dy <= r; ++dy) {
                const int yy = cy + dy;
                if (yy < 0 || yy >= hs.ny) continue;
                const int step = (dy == -r || dy == r) ? 1 : 2 * r;
                for (int dx = -r; dx <= r; dx += (step > 0 ? step : 1)) {
                    const int xx = cx + dx;
                    if (xx < 0 || xx >= hs.nx) continue;
                    const int c = yy * hs.nx + xx;
                    const int s1 = start[c + 1];
                    for (int s = start[c]; s < s1; ++s) {
                        if (s == (int)t) continue;
                        const float2 q = pts32[s];
                        const float fx = q.x - qi.x, fy = q.y - qi.y;
                        if (fmaf(fx, fx, fy * fy) > thr) continue;
                        const double2 pj = pts[s];
                        const double ddx = __dsub_rn(pj.x, pi.x);
                        const double ddy = __dsub_rn(pj.y, pi.y);
                        const double d2 = __dadd_rn(__dmul_rn(ddx, ddx), __dmul_rn(ddy, ddy));
                        const unsigned long long key = (unsigned long long)__double_as_longlong(d2);
                        const int j = sorted[s];
                        if (key > bk[kNb - 1] || (key == bk[kNb - 1] && j > bj[kNb - 1])) continue;
                        bk[kNb - 1] = key;
                        bj[kNb - 1] = j;
#pragma unroll
                        for (int k = kNb - 1; k > 0; --k) {
                            const bool sw = bk[k] < bk[k - 1] || (bk[k] == bk[k - 1] && bj[k] < bj[k - 1]);
                            if (sw) {
                                const unsigned long long tk = bk[k]; bk[k] = bk[k - 1]; bk[k - 1] = tk;
                                const int tj = bj[k]; bj[k] = bj[k - 1]; bj[k - 1] = tj;
                            }
                        }
                        if (bj[kNb - 1] != 0x7fffffff) {
                            const float d16 = (float)__longlong_as_double((long long)bk[kNb - 1]);
                            thr = d16 + (d16 * 1.52587890625e-5f + 4.0f * err * sqrtf(d16) +
                                         4.0f * err * err);
                        }
                    }
                }
            }
            // unvisited samples lie at least r h away (less a rounding margin of the cell index)
            const double reach = r * hs.h * (1.0 - 1e-9);
            if (bj[kNb - 1] != 0x7fffffff &&
                __longlong_as_double((long long)bk[kNb - 1]) < reach * reach)
                break;
        }
        // the feature row (offsets of the 16 neighbours, aux, zero padding) as 24 bf16 pairs,
        // stored as six 16-byte vectors (vec) or pair by pair
        uint32_t row[kInPad / 2];
#pragma unroll
        for (int k = 0; k < kNb; ++k) {
            const int j = bj[k] == 0x7fffffff ? i : bj[k];   // fewer than 16 samples in all
            const uint32_t lo = __bfloat16_as_ushort(__double2bfloat16(__dsub_rn(lam[2 * j], pi.x)));
            const uint32_t hi =
                __bfloat16_as_ushort(__double2bfloat16(__dsub_rn(lam[2 * j + 1], pi.y)));
            row[k] = lo | (hi << 16);
        }
        row[kNb] = __bfloat16_as_ushort(__double2bfloat16(aux ? aux[i] : 0.0));
#pragma unroll
        for (int k = kNb + 1; k < kInPad / 2; ++k) row[k] = 0u;
        if (vec) {
            uint4* f4 = reinterpret_cast<uint4*>(feat + (int64_t)i * kInPad);
#pragma unroll
            for (int q = 0; q < kInPad / 8; ++q)
                f4[q] = make_uint4(row[4 * q], row[4 * q + 1], row[4 * q + 2], row[4 * q + 3]);
            if (nbr) {
                int4* n4 = reinterpret_cast<int4*>(nbr + (int64_t)i * kNb);
#pragma unroll
                for (int q = 0; q < kNb / 4; ++q) {
                    int v[4];
#pragma unroll
                    for (int r = 0; r < 4; ++r)
                        v[r] = bj[4 * q + r] == 0x7fffffff ? -1 : bj[4 * q + r];
                    n4[q] = make_int4(v[0], v[1], v[2], v[3]);
                }
            }
        } else {
            uint32_t* f2 = reinterpret_cast<uint32_t*>(feat + (int64_t)i * kInPad);
#pragma unroll
            for (int k = 0; k < kInPad / 2; ++k) f2[k] = row[k];
            if (nbr) {
#pragma unroll
                for (int k = 0; k < kNb; ++k)
                    nbr[(int64_t)i * kNb + k] = bj[k] == 0x7fffffff ? -1 : bj[k];
            }
        }
    }
}

// ---------------------------------------------------------------------------------------------
// MLP on BF16 tensor cores
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ void mma16816(float* d, const uint32_t* a, uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
        "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    const uint32_t l = __bfloat16_as_ushort(__float2bfloat16_rn(lo));
    const uint32_t h = __bfloat16_as_ushort(__float2bfloat16_rn(hi));
    return l | (h << 16);
}

__device__ __forceinline__ float bf16r(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

__device__ __forceinline__ float gelu(float z) {
    const float c = 0.7978845608028654f;
    return 0.5f * z * (1.0f + tanhf(c * (z + 0.044715f * z * z * z)));
}

// gelu(z) and its derivative, sharing the tanh
__device__ __forceinline__ float gelu_with_grad(float z, float* grad) {
    const float c = 0.7978845608028654f;
    const float t = tanhf(c * (z + 0.044715f * z * z * z));
    *grad = 0.5f * (1.0f + t) + 0.5f * z * (1.0f - t * t) * c * (1.0f + 3.0f * 0.044715f * z * z);
    return 0.5f * z * (1.0f + t);
}

// BF16 weights in shared memory, Wt[out][in] (B fragment pairs along in); biases and w4 in FP32.
struct MlpSmem {
    __nv_bfloat16 w1t[kHid * kLd1];
    __nv_bfloat16 w2t[kHid * kLdH], w3t[kHid * kLdH];
    float b1[kHid], b2[kHid], b3[kHid], w4[kHid], b4;
};

// Coalesced reads of P, transposed stores: the other way round a warp's load touched 32 sectors, and
// staging was a third of the forward pass (211,250 rows 108 us, now 69; 20,200 rows 32, now 18).
__device__ void load_smem(MlpSmem& s, const float* __restrict__ P) {
    for (int i = threadIdx.x; i < kHid * kLd1; i += blockDim.x) {
        const int k = i / kHid, o = i - k * kHid;
        s.w1t[o * kLd1 + k] = __float2bfloat16_rn(k < kIn ? P[oW1 + k * kHid + o] : 0.f);
    }
    for (int i = threadIdx.x; i < kHid * kHid; i += blockDim.x) {
        const int k = i / kHid, o = i - k * kHid;
        s.w2t[o * kLdH + k] = __float2bfloat16_rn(P[oW2 + i]);
        s.w3t[o * kLdH + k] = __float2bfloat16_rn(P[oW3 + i]);
    }
    for (int i = threadIdx.x; i < kHid; i += blockDim.x) {
        s.b1[i] = P[ob1 + i];
        s.b2[i] = P[ob2 + i];
        s.b3[i] = P[ob3 + i];
        s.w4[i] = bf16r(P[ow4 + i]);
    }
    if (threadIdx.x == 0) s.b4 = P[ob4];
}

__device__ __forceinline__ uint32_t ld32(const __nv_bfloat16* p) {
    return *reinterpret_cast<const uint32_t*>(p);
}

// acc[8][4] = A(16 x 16 ksteps) * W, B fragments from Wt (row = output, ld = stride)
template <int KSTEPS>
__device__ __forceinline__ void gemm_rows(float (*acc)[4], const uint32_t (*a)[4],
                                          const __nv_bfloat16* wt, int ld, int g, int t) {
#pragma unroll
    for (int kk = 0; kk < KSTEPS; ++kk)
#pragma unroll
        for (int nt = 0; nt < 8; ++nt) {
            const __nv_bfloat16* p = wt + (8 * nt + g) * ld + 16 * kk + 2 * t;
            mma16816(acc[nt], a[kk], ld32(p), ld32(p + 8));
        }
}

// GELU on the accumulators; A fragments of the next layer
__device__ __forceinline__ void act_layer(float (*acc)[4], uint32_t (*anext)[4]) {
    float h[8][4];
#pragma unroll
    for (int nt = 0; nt < 8; ++nt)
#pragma unroll
        for (int q = 0; q < 4; ++q) h[nt][q] = bf16r(gelu(acc[nt][q]));
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
        anext[kk][0] = pack_bf16(h[2 * kk][0], h[2 * kk][1]);
        anext[kk][1] = pack_bf16(h[2 * kk][2], h[2 * kk][3]);
        anext[kk][2] = pack_bf16(h[2 * kk + 1][0], h[2 * kk + 1][1]);
        anext[kk][3] = pack_bf16(h[2 * kk + 1][2], h[2 * kk + 1][3]);
    }
}

__device__ __forceinline__ void init_bias(float (*acc)[4], const float* b, int t) {
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
        acc[nt][0] = acc[nt][2] = b[8 * nt + 2 * t];
        acc[nt][1] = acc[nt][3] = b[8 * nt + 2 * t + 1];
    }
}

// alpha = exp(y) of every feature row.
__global__ void __launch_bounds__(128)
    k_mlp_forward(const __nv_bfloat16* __restrict__ X, int64_t M, const float* __restrict__ P,
                  double* __restrict__ alpha) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    MlpSmem& s = *reinterpret_cast<MlpSmem*>(smem_raw);
    load_smem(s, P);
    __syncthreads();
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t tile = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5);
         tile * 16 < M; tile += nwarps) {
        const int64_t r0 = tile * 16;
        uint32_t a1[3][4];
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
            const int64_t row = r0 + g + 8 * hh;
            const bool ok = row < M;
            const __nv_bfloat16* xr = X + (ok ? row : 0) * kInPad;
#pragma unroll
            for (int kk = 0; kk < 3; ++kk) {
                a1[kk][hh] = ok ? ld32(xr + 16 * kk + 2 * t) : 0u;
                a1[kk][2 + hh] = ok ? ld32(xr + 16 * kk + 8 + 2 * t) : 0u;
            }
        }
        float acc[8][4];
        uint32_t an[4][4];
        init_bias(acc, s.b1, t);
        gemm_rows<3>(acc, a1, s.w1t, kLd1, g, t);
        act_layer(acc, an);
        init_bias(acc, s.b2, t);
        gemm_rows<4>(acc, an, s.w2t, kLdH, g, t);
        act_layer(acc, an);
        init_bias(acc, s.b3, t);
        gemm_rows<4>(acc, an, s.w3t, kLdH, g, t);
        act_layer(acc, an);
        // output layer in FP32 on the BF16-rounded h3 (the A fragments hold exactly those values)
        float part[2] = {0.f, 0.f};
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) {
                const uint32_t lo = an[kk][hh], hi = an[kk][2 + hh];
                const int c0 = 16 * kk + 2 * t;
                part[hh] += __uint_as_float(lo << 16) * s.w4[c0] +
                            __uint_as_float(lo & 0xffff0000u) * s.w4[c0 + 1] +
                            __uint_as_float(hi << 16) * s.w4[c0 + 8] +
                            __uint_as_float(hi & 0xffff0000u) * s.w4[c0 + 9];
            }
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
            part[hh] += __shfl_xor_sync(0xffffffffu, part[hh], 1);
            part[hh] += __shfl_xor_sync(0xffffffffu, part[hh], 2);
        }
        if (t == 0)
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) {
                const int64_t row = r0 + g + 8 * hh;
                if (row < M) alpha[row] = exp((double)(part[hh] + s.b4));
            }
    }
}

// ---------------------------------------------------------------------------------------------
// Training: forward, backward and weight gradients of 64 rows by one CTA of 8 warps.
//
// Warp (rg, hf) = (warp & 3, warp >> 2) owns rows 16 rg .. 16 rg + 15 and half hf of the 64 columns of
// every layer, so that a layer costs a thread 16 activations. The BF16 rows of X, h1..h3 and
// dz3..dz1 stay in shared memory, where ldmatrix reads them as A operands of the next product
// (straight) and as both operands of act^T dz (transposed); one copy Wt[out][in] of each weight
// serves the forward product (straight) and dh = dz W^T (transposed). gelu'(z) is kept in registers
// from the forward pass. The weight gradients accumulate in the MMA fragments over all tiles of the
// CTA. Bound: the chain of 13 dependent phases of one tile, not bytes (about 1 MB of X per step at
// B = 8192) or tensor rate; hence small tiles (128 CTAs at B = 8192) and everything in one launch.
// Measured at B = 8192, us per step: separate forward, backward, per-layer weight-gradient kernels
// of 8 CTAs each and serial reductions 571; this kernel and k_mlp_update 18.2 (B = 200,000: 1231
// and 144).
constexpr int kTrainRows = 64, kTrainThreads = 256;
constexpr int kPartStride = (kParams + 1 + 31) / 32 * 32;   // packed gradients, then the loss

struct TrainSmem {
    __nv_bfloat16 x[kTrainRows * kLd1];
    __nv_bfloat16 h[3][kTrainRows * kLdH];     // h1..h3
    __nv_bfloat16 dz[3][kTrainRows * kLdH];    // dz1..dz3
    __nv_bfloat16 w1t[kHid * kLd1];
    __nv_bfloat16 w2t[kHid * kLdH], w3t[kHid * kLdH];
    float bias[3][kHid], w4[kHid];
    float ypart[2][kTrainRows], target[kTrainRows], dy[kTrainRows];
    float small[4][5][kHid];
    float b4;
};

__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], const __nv_bfloat16* p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"((uint32_t)__cvta_generic_to_shared(p)) : "memory");
}
__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], const __nv_bfloat16* p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"((uint32_t)__cvta_generic_to_shared(p)) : "memory");
}

// acc[4][4] += A(rows 16 rg .., KSTEPS k-steps, row stride LDA) * W(columns 32 hf ..), W from
// wt[out][in] (forward, LDW) or, TRANS, from wt[out][in] as W^T (backward: k = out, n = in).
template <int KSTEPS, int LDA, int LDW, bool TRANS>
__device__ __forceinline__ void train_gemm(float (&acc)[4][4], const __nv_bfloat16* a,
                                           const __nv_bfloat16* wt, int rg, int hf, int lane) {
    const int r8 = lane & 7, q = lane >> 3;
#pragma unroll
    for (int kk = 0; kk < KSTEPS; ++kk) {
        uint32_t af[4];
        ldsm4(af, a + (16 * rg + (q & 1) * 8 + r8) * LDA + 16 * kk + (q >> 1) * 8);
#pragma unroll
        for (int np = 0; np < 2; ++np) {               // two 8-column tiles per load
            const int n0 = 32 * hf + 16 * np;
            uint32_t b[4];
            if constexpr (TRANS)
                ldsm4t(b, wt + (16 * kk + (q & 1) * 8 + r8) * LDW + n0 + (q >> 1) * 8);
            else
                ldsm4(b, wt + (n0 + (q >> 1) * 8 + r8) * LDW + 16 * kk + (q & 1) * 8);
            mma16816(acc[2 * np], af, b[0], b[1]);
            mma16816(acc[2 * np + 1], af, b[2], b[3]);
        }
    }
}

// acc[4][4] += act^T dz over the tile's rows: features 16 mt .., columns 32 hf ..
template <int LDA>
__device__ __forceinline__ void train_wgrad(float (&acc)[4][4], const __nv_bfloat16* act,
                                            const __nv_bfloat16* dz, int mt, int hf, int lane) {
    const int r8 = lane & 7, q = lane >> 3;
#pragma unroll
    for (int kk = 0; kk < kTrainRows / 16; ++kk) {
        uint32_t af[4];
        ldsm4t(af, act + (16 * kk + (q >> 1) * 8 + r8) * LDA + 16 * mt + (q & 1) * 8);
#pragma unroll
        for (int np = 0; np < 2; ++np) {
            uint32_t b[4];
            ldsm4t(b, dz + (16 * kk + (q & 1) * 8 + r8) * kLdH + 32 * hf + 16 * np + (q >> 1) * 8);
            mma16816(acc[2 * np], af, b[0], b[1]);
            mma16816(acc[2 * np + 1], af, b[2], b[3]);
        }
    }
}

// Partial gradients and loss of the mean squared error over the CTA's tiles of 64 batch rows, in
// part[blockIdx.x * kPartStride ..] (packed as the parameters, then the loss). Batch row r is
// row idx[r] (or r) of X and target. vec: X is 16-byte aligned (else 4-byte loads).
__global__ void __launch_bounds__(kTrainThreads)
    k_mlp_train(const __nv_bfloat16* __restrict__ X, const double* __restrict__ target,
                const int* __restrict__ idx, int64_t B, const float* __restrict__ P,
                float* __restrict__ part, bool vec) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    TrainSmem& s = *reinterpret_cast<TrainSmem*>(smem_raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int g = lane >> 2, t = lane & 3, rg = warp & 3, hf = warp >> 2;
    pdl_wait();                                        // the last step's update of P
    pdl_allow_next();
    for (int i = tid; i < kHid * kLd1; i += kTrainThreads) {
        const int k = i / kHid, o = i - k * kHid;      // coalesced reads, transposed stores
        s.w1t[o * kLd1 + k] = __float2bfloat16_rn(k < kIn ? P[oW1 + k * kHid + o] : 0.f);
    }
    for (int i = tid; i < kHid * kHid; i += kTrainThreads) {
        const int k = i / kHid, o = i - k * kHid;
        s.w2t[o * kLdH + k] = __float2bfloat16_rn(P[oW2 + i]);
        s.w3t[o * kLdH + k] = __float2bfloat16_rn(P[oW3 + i]);
    }
    if (tid < kHid) {
        s.bias[0][tid] = P[ob1 + tid];
        s.bias[1][tid] = P[ob2 + tid];
        s.bias[2][tid] = P[ob3 + tid];
        s.w4[tid] = bf16r(P[ow4 + tid]);
    }
    if (tid == 0) s.b4 = P[ob4];
    float wg[3][4][4] = {};                            // weight gradients of W1, W2, W3
    float sb[3] = {0.f, 0.f, 0.f}, sw4 = 0.f, sdy = 0.f, lsum = 0.f;
    const float Bf = (float)B;
    for (int64_t r0 = (int64_t)blockIdx.x * kTrainRows; r0 < B;
         r0 += (int64_t)gridDim.x * kTrainRows) {
        __syncthreads();                               // weights staged; the last tile consumed
        for (int i = tid; i < kTrainRows * (kInPad / 8); i += kTrainThreads) {
            const int r = i / (kInPad / 8), c = i - r * (kInPad / 8);
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            if (r0 + r < B) {
                const int64_t src = idx ? (int64_t)idx[r0 + r] : r0 + r;
                const __nv_bfloat16* p = X + src * kInPad + 8 * c;
                if (vec) v = *reinterpret_cast<const uint4*>(p);
                else v = make_uint4(ld32(p), ld32(p + 2), ld32(p + 4), ld32(p + 6));
            }
            *reinterpret_cast<uint4*>(s.x + r * kLd1 + 8 * c) = v;
        }
        if (tid < kTrainRows && r0 + tid < B)
            s.target[tid] = (float)target[idx ? (int64_t)idx[r0 + tid] : r0 + tid];
        __syncthreads();
        float gg[3][4][4];                             // gelu'(z) of the thread's cells
        float acc[4][4];
#pragma unroll
        for (int l = 0; l < 3; ++l) {
#pragma unroll
            for (int nt = 0; nt < 4; ++nt) {
                const int c = 32 * hf + 8 * nt + 2 * t;
                acc[nt][0] = acc[nt][2] = s.bias[l][c];
                acc[nt][1] = acc[nt][3] = s.bias[l][c + 1];
            }
            if (l == 0) train_gemm<3, kLd1, kLd1, false>(acc, s.x, s.w1t, rg, hf, lane);
            else train_gemm<4, kLdH, kLdH, false>(acc, s.h[l - 1], l == 1 ? s.w2t : s.w3t, rg, hf,
                                                  lane);
            float yp[2] = {0.f, 0.f};
#pragma unroll
            for (int nt = 0; nt < 4; ++nt) {
                const int c = 32 * hf + 8 * nt + 2 * t;
#pragma unroll
                for (int hh = 0; hh < 2; ++hh) {
                    const float h0 = bf16r(gelu_with_grad(acc[nt][2 * hh], &gg[l][nt][2 * hh]));
                    const float h1 = bf16r(gelu_with_grad(acc[nt][2 * hh + 1],
                                                          &gg[l][nt][2 * hh + 1]));
                    *reinterpret_cast<uint32_t*>(s.h[l] + (16 * rg + g + 8 * hh) * kLdH + c) =
                        pack_bf16(h0, h1);
                    if (l == 2) yp[hh] += h0 * s.w4[c] + h1 * s.w4[c + 1];
                }
            }
            if (l == 2) {
#pragma unroll
                for (int hh = 0; hh < 2; ++hh) {
                    yp[hh] += __shfl_xor_sync(0xffffffffu, yp[hh], 1);
                    yp[hh] += __shfl_xor_sync(0xffffffffu, yp[hh], 2);
                    if (t == 0) s.ypart[hf][16 * rg + g + 8 * hh] = yp[hh];
                }
            }
            __syncthreads();
        }
        if (tid < kTrainRows) {
            float d = 0.f;
            if (r0 + tid < B) {
                const float e = (s.ypart[0][tid] + s.ypart[1][tid]) + s.b4 - s.target[tid];
                d = 2.0f * e / Bf;
                lsum += e * e / Bf;
            }
            s.dy[tid] = d;                             // rows past B: zero gradients throughout
        }
        __syncthreads();
#pragma unroll
        for (int l = 2; l >= 0; --l) {                 // dz of layer l, then dh of the one below
#pragma unroll
            for (int nt = 0; nt < 4; ++nt) {
                const int c = 32 * hf + 8 * nt + 2 * t;
#pragma unroll
                for (int hh = 0; hh < 2; ++hh) {
                    const int row = 16 * rg + g + 8 * hh;
                    float d0, d1;
                    if (l == 2) {
                        d0 = s.dy[row] * s.w4[c] * gg[l][nt][2 * hh];
                        d1 = s.dy[row] * s.w4[c + 1] * gg[l][nt][2 * hh + 1];
                    } else {
                        d0 = acc[nt][2 * hh] * gg[l][nt][2 * hh];
                        d1 = acc[nt][2 * hh + 1] * gg[l][nt][2 * hh + 1];
                    }
                    *reinterpret_cast<uint32_t*>(s.dz[l] + row * kLdH + c) = pack_bf16(d0, d1);
                }
            }
            __syncthreads();
            if (l > 0) {
#pragma unroll
                for (int nt = 0; nt < 4; ++nt)
                    acc[nt][0] = acc[nt][1] = acc[nt][2] = acc[nt][3] = 0.f;
                train_gemm<4, kLdH, kLdH, true>(acc, s.dz[l], l == 2 ? s.w3t : s.w2t, rg, hf, lane);
                train_wgrad<kLdH>(wg[l], s.h[l - 1], s.dz[l], rg, hf, lane);
            } else if (rg < kInPad / 16) {
                train_wgrad<kLd1>(wg[0], s.x, s.dz[0], rg, hf, lane);
            }
        }
        const int col = tid & 63, ph = tid >> 6;       // biases and the output layer
        for (int r = 16 * ph; r < 16 * ph + 16; ++r) {
#pragma unroll
            for (int l = 0; l < 3; ++l) sb[l] += __bfloat162float(s.dz[l][r * kLdH + col]);
            sw4 += __bfloat162float(s.h[2][r * kLdH + col]) * s.dy[r];
            if (col == 0) sdy += s.dy[r];
        }
    }
    float* out = part + (int64_t)blockIdx.x * kPartStride;
    const int offs[3] = {oW1, oW2, oW3};
#pragma unroll
    for (int l = 0; l < 3; ++l)
#pragma unroll
        for (int nt = 0; nt < 4; ++nt)
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) {
                const int m = 16 * rg + g + 8 * hh;
                if (m < (l == 0 ? kIn : kHid))
                    *reinterpret_cast<float2*>(out + offs[l] + m * kHid + 32 * hf + 8 * nt + 2 * t) =
                        make_float2(wg[l][nt][2 * hh], wg[l][nt][2 * hh + 1]);
            }
    {
        const int col = tid & 63, ph = tid >> 6;
        for (int l = 0; l < 3; ++l) s.small[ph][l][col] = sb[l];
        s.small[ph][3][col] = sw4;
        if (col == 0) s.small[ph][4][0] = sdy;
        // rows of the loss live in warps 0 and 1
        for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
        if (lane == 0 && warp < 2) s.small[0][4][1 + warp] = lsum;
        __syncthreads();
        const int goff[4] = {ob1, ob2, ob3, ow4};
        if (ph == 0)
            for (int q = 0; q < 4; ++q)
                out[goff[q] + col] = ((s.small[0][q][col] + s.small[1][q][col]) +
                                      s.small[2][q][col]) + s.small[3][q][col];
        if (tid == 0) {
            out[ob4] = ((s.small[0][4][0] + s.small[1][4][0]) + s.small[2][4][0]) + s.small[3][4][0];
            out[kParams] = s.small[0][4][1] + s.small[0][4][2];
        }
    }
}

// Gradients (and the loss) as the sums of the CTAs' partials, in a fixed order (so bitwise
// reproducible): slice k of 8 adds partials k, k + 8, ..., then the slices are added in order. With
// apply set, one Adam step on the FP32 master parameters follows.
struct AdamStep {
    int apply = 0;
    float lr = 0.f, b1 = 0.f, b2 = 0.f, ob1 = 0.f, ob2 = 0.f, eps = 0.f, c1 = 1.f, c2 = 1.f;
};
constexpr int kUpdSlices = 8;
__global__ void __launch_bounds__(32 * kUpdSlices)
    k_mlp_update(const float* __restrict__ part, int nparts, float* __restrict__ grad,
                 float* __restrict__ loss, float* __restrict__ P, float* __restrict__ m,
                 float* __restrict__ v, const AdamStep ad) {
    __shared__ float sum[kUpdSlices][32];
    const int lane = threadIdx.x & 31, k = threadIdx.x >> 5;
    const int i = blockIdx.x * 32 + lane;              // < kPartStride
    pdl_wait();                                        // the partials
    pdl_allow_next();
    float acc = 0.f;
#pragma unroll 8
    for (int b = k; b < nparts; b += kUpdSlices) acc += part[(int64_t)b * kPartStride + i];
    sum[k][lane] = acc;
    __syncthreads();
    if (k != 0 || i > kParams) return;
    float g = sum[0][lane];
#pragma unroll
    for (int q = 1; q < kUpdSlices; ++q) g += sum[q][lane];
    if (i == kParams) {
        *loss = g;
        return;
    }
    grad[i] = g;
    if (!ad.apply) return;
    const float mi = ad.b1 * m[i] + ad.ob1 * g;
    const float vi = ad.b2 * v[i] + ad.ob2 * (g * g);
    m[i] = mi;
    v[i] = vi;
    P[i] -= ad.lr * (mi / ad.c1) / (sqrtf(vi / ad.c2) + ad.eps);
}

int nb(int64_t n, int t, int cap = 152 * 16) {
    int64_t b = (n + t - 1) / t;
    return (int)std::max<int64_t>(1, std::min<int64_t>(b, cap));
}

}  // namespace

struct Mlp {
    float* P = nullptr;      // FP32 master parameters (kParams)
    float* m = nullptr;      // Adam moments
    float* v = nullptr;
    float* grad = nullptr;
    float* loss = nullptr;
    int64_t step = 0;
    float* part = nullptr;       // per-CTA partial gradients of a training step (first use)
    int parts = 0;               // CTAs it has room for
};

namespace {

// CTAs of a training step on this device: two per SM, at most one per 64 rows
ftcg_status_t train_ctas(int64_t B, int* out) {
    int dev = 0, sms = 0;
    FTCG_CK(cudaGetDevice(&dev));
    FTCG_CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    *out = (int)std::min<int64_t>((B + kTrainRows - 1) / kTrainRows, 2 * (int64_t)sms);
    return FTCG_SUCCESS;
}

ftcg_status_t ensure_parts(Mlp* q, int ctas) {
    if (ctas <= q->parts) return FTCG_SUCCESS;
    if (q->part) FTCG_CK(cudaFree(q->part));
    q->part = nullptr;
    q->parts = 0;
    FTCG_CK(cudaMalloc(&q->part, (size_t)ctas * kPartStride * sizeof(float)));
    q->parts = ctas;
    return FTCG_SUCCESS;
}

ftcg_status_t mlp_fail(const char* m) {
    set_error("%s", m);
    return FTCG_ERR_INVALID_VALUE;
}

ftcg_status_t launch_forward(Mlp* q, const __nv_bfloat16* X, int64_t M, double* alpha,
                             cudaStream_t s) {
    const size_t sm = sizeof(MlpSmem);
    // one wave of resident CTAs (shared memory: six per SM), each staging the weights once
    const int blocks = nb((M + 63) / 64, 1, 152 * 6);
    FTCG_CK(cudaFuncSetAttribute(k_mlp_forward, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)sm));
    k_mlp_forward<<<blocks, 128, sm, s>>>(X, M, q->P, alpha);
    FTCG_CK(cudaGetLastError());
    return FTCG_SUCCESS;
}

// gradients of one batch into q->grad and its loss into q->loss, then (ad.apply) an Adam step
ftcg_status_t train_batch(Mlp* q, const __nv_bfloat16* X, const double* target, const int* idx,
                          int64_t B, const AdamStep& ad, cudaStream_t s) {
    int ctas = 0;
    FTCG_TRY(train_ctas(B, &ctas));
    FTCG_TRY(ensure_parts(q, ctas));
    const size_t sm = sizeof(TrainSmem);
    FTCG_CK(cudaFuncSetAttribute(k_mlp_train, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    FTCG_CK(launch_pdl(k_mlp_train, dim3(ctas), dim3(kTrainThreads), sm, s, X, target, idx, B,
                       (const float*)q->P, q->part, (reinterpret_cast<uintptr_t>(X) & 15) == 0));
    FTCG_CK(launch_pdl(k_mlp_update, dim3(kPartStride / 32), dim3(32 * kUpdSlices), 0, s,
                       (const float*)q->part, ctas, q->grad, q->loss, q->P, q->m, q->v, ad));
    return FTCG_SUCCESS;
}

// ---------------------------------------------------------------------------------------------
// kNN feature requests (one or many rasters)
// ---------------------------------------------------------------------------------------------
struct FeatJob {
    const double* lam;
    const double* aux;
    int64_t M;
    __nv_bfloat16* out;
    int32_t* nbr;
};

// The spatial hash of a raster from the per-block partials of its bounding box: square cells of
// about one sample each (at most 4096 per axis, also when the samples lie on a line), and the
// bound on the FP32 offset error (2^-24 of twice the extent, with a 1% margin). False when a
// coordinate is not finite.
bool hash_from_box(const double* part, int nblk, int64_t M, Hash* hs, float* err) {
    double x0 = 1e300, y0 = 1e300, x1 = -1e300, y1 = -1e300;
    for (int i = 0; i < nblk; ++i) {
        x0 = std::min(x0, part[4 * i]);
        y0 = std::min(y0, part[4 * i + 1]);
        x1 = std::max(x1, part[4 * i + 2]);
        y1 = std::max(y1, part[4 * i + 3]);
    }
    if (!std::isfinite(x0) || !std::isfinite(y0) || !std::isfinite(x1) || !std::isfinite(y1))
        return false;
    const double area = std::max((x1 - x0) * (y1 - y0), 1e-300);
    double h = std::sqrt(area / (double)M);
    if (!(h > 0)) h = 1.0;
    h = std::max(h, std::max(x1 - x0, y1 - y0) / 4096.0);
    if (!(h > 0)) h = 1.0;
    hs->x0 = x0;
    hs->y0 = y0;
    hs->h = h;
    hs->inv_h = 1.0 / h;
    hs->nx = std::max(1, (int)std::ceil((x1 - x0) / h + 1e-9));
    hs->ny = std::max(1, (int)std::ceil((y1 - y0) / h + 1e-9));
    *err = (float)(2.0 * std::max(x1 - x0, y1 - y0) * 5.9604644775390625e-8 * 1.01);
    return true;
}

// The counting sort of one raster into its hash cells and the kNN search, enqueued on s
// (asynchronous; the temporaries come from the pool and are released on s).
ftcg_status_t launch_knn(const FeatJob& j, const Hash& hs, float err, cudaStream_t s) {
    const int64_t M = j.M;
    const int64_t ncell = (int64_t)hs.nx * hs.ny;
    int *cnt = nullptr, *start = nullptr, *cell = nullptr, *sorted = nullptr;
    double2* pts = nullptr;
    float2* pts32 = nullptr;
    FTCG_CK(pool_malloc(&cnt, (ncell + 1) * sizeof(int), s));
    FTCG_CK(pool_malloc(&start, (ncell + 1) * sizeof(int), s));
    FTCG_CK(pool_malloc(&cell, M * sizeof(int), s));
    FTCG_CK(pool_malloc(&sorted, M * sizeof(int), s));
    FTCG_CK(pool_malloc(&pts, M * sizeof(double2), s));
    FTCG_CK(pool_malloc(&pts32, M * sizeof(float2), s));
    FTCG_CK(cudaMemsetAsync(cnt, 0, (ncell + 1) * sizeof(int), s));
    k_cell_count<<<nb(M, 256), 256, 0, s>>>(j.lam, M, hs, cnt, cell);
    FTCG_TRY(exclusive_scan_i32(cnt, start, ncell + 1, s));
    FTCG_CK(cudaMemcpyAsync(cnt, start, (ncell + 1) * sizeof(int), cudaMemcpyDeviceToDevice, s));
    k_cell_scatter<<<nb(M, 256), 256, 0, s>>>(M, cell, cnt, sorted);
    k_gather_pts<<<nb(M, 256), 256, 0, s>>>(j.lam, M, sorted, hs.x0, hs.y0, pts, pts32);
    // 16-byte row stores need 16-byte aligned outputs (rows are 96 and 64 bytes)
    const bool vec = (reinterpret_cast<uintptr_t>(j.out) & 15) == 0 &&
                     (reinterpret_cast<uintptr_t>(j.nbr) & 15) == 0;
    k_knn<<<nb(M, 128, 152 * 32), 128, 0, s>>>(j.lam, j.aux, M, hs, start, sorted, pts, pts32, err,
                                                  j.out, j.nbr, vec);
    const cudaError_t e = cudaGetLastError();
    pool_free(cnt, s);
    pool_free(start, s);
    pool_free(cell, s);
    pool_free(sorted, s);
    pool_free(pts, s);
    pool_free(pts32, s);
    FTCG_CK(e);
    return FTCG_SUCCESS;
}

// Side streams over which the searches of a multi-raster request are spread (created once per
// device, non-blocking; ordered after and before the caller's stream by events).
constexpr int kFeatStreams = 4;

ftcg_status_t feat_streams(cudaStream_t* out) {
    static std::mutex mu;
    static std::map<int, std::vector<cudaStream_t>> by_dev;
    int dev = 0;
    FTCG_CK(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lk(mu);
    auto& v = by_dev[dev];
    while ((int)v.size() < kFeatStreams) {
        cudaStream_t st = nullptr;
        FTCG_CK(cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking));
        v.push_back(st);
    }
    for (int k = 0; k < kFeatStreams; ++k) out[k] = v[k];
    return FTCG_SUCCESS;
}

// Features of n rasters: the bounding boxes of all of them with one synchronisation, then the
// rasters' sorts and searches back to back (spread over the side streams when n > 1), then one
// synchronisation. A raster with a non-finite coordinate fails the request before any search.
ftcg_status_t features_impl(const FeatJob* jobs, int n, cudaStream_t s, const char* what) {
    std::vector<int> nblk(n, 0), boff(n + 1, 0);
    for (int i = 0; i < n; ++i) {
        nblk[i] = jobs[i].M > 0 ? nb(jobs[i].M, 256, 1024) : 0;
        boff[i + 1] = boff[i] + nblk[i];
    }
    if (boff[n] == 0) return FTCG_SUCCESS;
    double* bb = nullptr;
    FTCG_CK(pool_malloc(&bb, (size_t)boff[n] * 4 * sizeof(double), s));
    for (int i = 0; i < n; ++i)
        if (nblk[i]) k_bbox<<<nblk[i], 256, 0, s>>>(jobs[i].lam, jobs[i].M, bb + 4 * boff[i]);
    std::vector<double> hb((size_t)boff[n] * 4);
    FTCG_CK(cudaGetLastError());
    FTCG_CK(cudaMemcpyAsync(hb.data(), bb, hb.size() * sizeof(double), cudaMemcpyDeviceToHost, s));
    FTCG_CK(cudaStreamSynchronize(s));
    pool_free(bb, s);
    std::vector<Hash> hs(n);
    std::vector<float> err(n, 0.f);
    for (int i = 0; i < n; ++i) {
        if (!nblk[i]) continue;
        if (!hash_from_box(hb.data() + 4 * boff[i], nblk[i], jobs[i].M, &hs[i], &err[i])) {
            if (n == 1)
                set_error("%s: non-finite coordinates", what);
            else
                set_error("%s: raster %d has non-finite coordinates", what, i);
            return FTCG_ERR_NUMERIC;
        }
    }
    int active = 0;
    for (int i = 0; i < n; ++i) active += nblk[i] ? 1 : 0;
    if (active == 1) {
        for (int i = 0; i < n; ++i)
            if (nblk[i]) FTCG_TRY(launch_knn(jobs[i], hs[i], err[i], s));
        FTCG_CK(cudaStreamSynchronize(s));
        return FTCG_SUCCESS;
    }
    cudaStream_t side[kFeatStreams];
    FTCG_TRY(feat_streams(side));
    cudaEvent_t ev[kFeatStreams + 1];
    for (auto& e : ev) FTCG_CK(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
    ftcg_status_t st = FTCG_SUCCESS;
    cudaError_t ce = cudaEventRecord(ev[kFeatStreams], s);
    for (int k = 0; k < kFeatStreams && ce == cudaSuccess; ++k)
        ce = cudaStreamWaitEvent(side[k], ev[kFeatStreams], 0);
    for (int i = 0, k = 0; i < n && ce == cudaSuccess && st == FTCG_SUCCESS; ++i) {
        if (!nblk[i]) continue;
        st = launch_knn(jobs[i], hs[i], err[i], side[k]);
        k = (k + 1) % kFeatStreams;
    }
    // the caller's stream waits for every side stream, also after a failed launch
    for (int k = 0; k < kFeatStreams; ++k) {
        cudaEventRecord(ev[k], side[k]);
        cudaStreamWaitEvent(s, ev[k], 0);
    }
    const cudaError_t se = cudaStreamSynchronize(s);
    for (auto& e : ev) cudaEventDestroy(e);
    if (st != FTCG_SUCCESS) return st;
    FTCG_CK(ce);
    FTCG_CK(se);
    return FTCG_SUCCESS;
}

}  // namespace
}  // namespace ftcg

using namespace ftcg;

extern "C" {

ftcg_status_t ftcg_features(const double* d_lambda, const double* d_aux, int64_t M,
                            void* d_features, int32_t* d_neighbors, ftcg_stream_t stream) {
    FTCG_API_BEGIN
    clear_error();
    if (M < 0 || (M > 0 && (!d_lambda || !d_features)))
        return mlp_fail("ftcg_features: bad arguments");
    if (M > (int64_t)INT32_MAX / kNb) return mlp_fail("ftcg_features: M too large");
    const FeatJob job{d_lambda, d_aux, M, reinterpret_cast<__nv_bfloat16*>(d_features), d_neighbors};
    return features_impl(&job, 1, reinterpret_cast<cudaStream_t>(stream), "ftcg_features");
    FTCG_API_END
}

ftcg_status_t ftcg_features_batch(int32_t n, const double* const* d_lambda,
                                  const double* const* d_aux, const int64_t* M,
                                  void* const* d_features, int32_t* const* d_neighbors,
                                  ftcg_stream_t stream) {
    FTCG_API_BEGIN
    clear_error();
    if (n < 0 || (n > 0 && (!d_lambda || !M || !d_features)))
        return mlp_fail("ftcg_features_batch: bad arguments");
    std::vector<FeatJob> jobs(n);
    for (int i = 0; i < n; ++i) {
        if (M[i] < 0 || (M[i] > 0 && (!d_lambda[i] || !d_features[i]))) {
            set_error("ftcg_features_batch: bad arguments for raster %d", i);
            return FTCG_ERR_INVALID_VALUE;
        }
        if (M[i] > (int64_t)INT32_MAX / kNb) {
            set_error("ftcg_features_batch: raster %d: M too large", i);
            return FTCG_ERR_INVALID_VALUE;
        }
        jobs[i] = FeatJob{d_lambda[i], d_aux ? d_aux[i] : nullptr, M[i],
                          reinterpret_cast<__nv_bfloat16*>(d_features[i]),
                          d_neighbors ? d_neighbors[i] : nullptr};
    }
    return features_impl(jobs.data(), n, reinterpret_cast<cudaStream_t>(stream),
                         "ftcg_features_batch");
    FTCG_API_END
}

ftcg_status_t ftcg_mlp_create(ftcg_mlp_t* out, const float* h_params) {
    FTCG_API_BEGIN
    clear_error();
    if (!out || !h_params) return mlp_fail("ftcg_mlp_create: NULL argument");
    *out = nullptr;
    Mlp* q = new (std::nothrow) Mlp();
    if (!q) return mlp_fail("ftcg_mlp_create: host allocation failed");
    const size_t bytes = kParams * sizeof(float);
    if (cudaMalloc(&q->P, bytes) != cudaSuccess || cudaMalloc(&q->m, bytes) != cudaSuccess ||
        cudaMalloc(&q->v, bytes) != cudaSuccess || cudaMalloc(&q->grad, bytes) != cudaSuccess ||
        cudaMalloc(&q->loss, sizeof(float)) != cudaSuccess) {
        cudaFree(q->P); cudaFree(q->m); cudaFree(q->v); cudaFree(q->grad); cudaFree(q->loss);
        delete q;
        set_error("ftcg_mlp_create: device allocation failed");
        return FTCG_ERR_OUT_OF_MEMORY;
    }
    cudaMemcpy(q->P, h_params, bytes, cudaMemcpyHostToDevice);
    cudaMemset(q->m, 0, bytes);
    cudaMemset(q->v, 0, bytes);
    *out = reinterpret_cast<ftcg_mlp_t>(q);
    return FTCG_SUCCESS;
    FTCG_API_END
}

ftcg_status_t ftcg_mlp_state(ftcg_mlp_t mlp, float* h_params, float* h_m, float* h_v,
                             int64_t* step, int32_t set) {
    FTCG_API_BEGIN
    clear_error();
    if (!mlp) return mlp_fail("ftcg_mlp_state: NULL model");
    Mlp* q = reinterpret_cast<Mlp*>(mlp);
    const size_t bytes = kParams * sizeof(float);
    const cudaMemcpyKind k = set ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToHost;
    FTCG_CK(cudaDeviceSynchronize());
    if (h_params) FTCG_CK(set ? cudaMemcpy(q->P, h_params, bytes, k) : cudaMemcpy(h_params, q->P, bytes, k));
    if (h_m) FTCG_CK(set ? cudaMemcpy(q->m, h_m, bytes, k) : cudaMemcpy(h_m, q->m, bytes, k));
    if (h_v) FTCG_CK(set ? cudaMemcpy(q->v, h_v, bytes, k) : cudaMemcpy(h_v, q->v, bytes, k));
    if (step) {
        if (set) q->step = *step;
        else *step = q->step;
    }
    return FTCG_SUCCESS;
    FTCG_API_END
}

ftcg_status_t ftcg_mlp_predict(ftcg_mlp_t mlp, const void* d_features, int64_t M,
                               double* d_alpha_out, ftcg_stream_t stream) {
    FTCG_API_BEGIN
    clear_error();
    if (!mlp || M < 0 || (M > 0 && (!d_features || !d_alpha_out)))
        return mlp_fail("ftcg_mlp_predict: bad arguments");
    if (M == 0) return FTCG_SUCCESS;
    Mlp* q = reinterpret_cast<Mlp*>(mlp);
    return launch_forward(q, reinterpret_cast<const __nv_bfloat16*>(d_features), M, d_alpha_out,
                          reinterpret_cast<cudaStream_t>(stream));
    FTCG_API_END
}

ftcg_status_t ftcg_mlp_grads(ftcg_mlp_t mlp, const void* d_features, const double* d_target,
                             const int32_t* d_index, int64_t B, float* h_grads, float* h_loss,
                             ftcg_stream_t stream) {
    FTCG_API_BEGIN
    clear_error();
    if (!mlp || B <= 0 || !d_features || !d_target) return mlp_fail("ftcg_mlp_grads: bad arguments");
    Mlp* q = reinterpret_cast<Mlp*>(mlp);
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    FTCG_TRY(train_batch(q, reinterpret_cast<const __nv_bfloat16*>(d_features), d_target, d_index,
                         B, AdamStep{}, s));
    if (h_grads)
        FTCG_CK(cudaMemcpyAsync(h_grads, q->grad, kParams * sizeof(float), cudaMemcpyDeviceToHost, s));
    if (h_loss) FTCG_CK(cudaMemcpyAsync(h_loss, q->loss, sizeof(float), cudaMemcpyDeviceToHost, s));
    FTCG_CK(cudaStreamSynchronize(s));
    return FTCG_SUCCESS;
    FTCG_API_END
}

ftcg_status_t ftcg_mlp_train_step(ftcg_mlp_t mlp, const void* d_features, const double* d_target,
                                  const int32_t* d_index, int64_t B, float lr, float* h_loss,
                                  ftcg_stream_t stream) {
    FTCG_API_BEGIN
    clear_error();
    if (!mlp || B <= 0 || !d_features || !d_target || !(lr > 0))
        return mlp_fail("ftcg_mlp_train_step: bad arguments");
    Mlp* q = reinterpret_cast<Mlp*>(mlp);
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    // 1 - beta is formed in FP64: 1.f - 0.999f in FP32 is 1.3e-5 away from 0.001
    const double b1 = 0.9, b2 = 0.999, n = (double)(q->step + 1);
    const AdamStep ad{1, lr, (float)b1, (float)b2, (float)(1.0 - b1), (float)(1.0 - b2), 1e-8f,
                      (float)(1.0 - std::pow(b1, n)), (float)(1.0 - std::pow(b2, n))};
    FTCG_TRY(train_batch(q, reinterpret_cast<const __nv_bfloat16*>(d_features), d_target, d_index,
                         B, ad, s));
    q->step += 1;
    if (h_loss) {
        FTCG_CK(cudaMemcpyAsync(h_loss, q->loss, sizeof(float), cudaMemcpyDeviceToHost, s));
        FTCG_CK(cudaStreamSynchronize(s));
    }
    return FTCG_SUCCESS;
    FTCG_API_END
}

ftcg_status_t ftcg_mlp_destroy(ftcg_mlp_t mlp) {
    FTCG_API_BEGIN
    clear_error();
    if (!mlp) return FTCG_SUCCESS;
    Mlp* q = reinterpret_cast<Mlp*>(mlp);
    cudaDeviceSynchronize();
    cudaFree(q->part);
    cudaFree(q->P);
    cudaFree(q->m);
    cudaFree(q->v);
    cudaFree(q->grad);
    cudaFree(q->loss);
    delete q;
    return FTCG_SUCCESS;
    FTCG_API_END
}

}  // extern "C"
