// The exact weights' lag route (weights.cu has the method) without the FP64 pipe: two-float (FP32
// pair) and 64-bit fixed-point arithmetic on a power-of-two lag grid of side L = 256..8192.
//
// FP64 runs at 1/64 of the FP32 rate on this GPU and was 85-87 % busy in every step of the FP64
// route, so its time was its count of FP64 instructions. Here positions are 46-bit fixed point, the
// window is a two-float polynomial per (tap, 1/128 of a cell), window products are summed as 64-bit
// integers (exactly, so the sums of a tile do not depend on their order) in shared memory, and the
// transforms and the interpolation carry FP32 pairs (about 2^-46 relative to the largest term). The
// window's own truncation exp(-beta) is larger than all of that, which is the condition on which
// compute_weights takes this route (split_lag_side, kUneven). Rms error against pair-by-pair FP64 sums on
// 60 polar rasters (N = 64..1024, M = 1 k..2 M, sigma = 2, w = 12): 1.00 to 1.02 times the FP64 route's at
// N a power of two (large ping 2.3e-12), 0.01 to 0.9 times elsewhere, where this lag grid is finer.
//
// Steps (lag grid transposed, [x][y]: a tile's cells and a transform's line are contiguous in y):
//   k_lag_origin   window polynomials, lag weights times window divisions (first blocks); 46-bit
//                  positions; samples counted per 64 x 64 tile of first taps
//   k_lag_scan     tile offsets, work items, occupied column pairs;  k_lag_scatter  the sort
//   k_lag_spread   W1: tiles in shared memory, then FP64 atomics into the grid
//   k_lag_fft_y    along y, two real columns per complex line, first N frequencies kept
//   k_lag_fft_x    along x and back, with the lag weights between (one pass over memory)
//   k_lag_fft_y    back along y;  k_lag_interp  W3 and the reciprocal

#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <map>
#include <mutex>
#include <vector>

#include "fft_smem.cuh"
#include "ftcg_internal.cuh"

namespace ftcg {

namespace {

// ---- two-float arithmetic ------------------------------------------------------------------
// A value is the unevaluated sum h + l. Sums keep l unnormalised (|l| stays within a few ulp of
// the largest h that entered): 8 operations; products 4. The _rn forms keep the compiler from
// contracting the error terms away.
struct ff {
    float h, l;
};
struct cff {
    ff x, y;
};

__device__ __forceinline__ ff two_sum(float a, float b) {
    const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
    return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}
__device__ __forceinline__ ff operator+(ff a, ff b) {
    const ff s = two_sum(a.h, b.h);
    return {s.h, __fadd_rn(__fadd_rn(a.l, b.l), s.l)};
}
__device__ __forceinline__ ff operator-(ff a) { return {-a.h, -a.l}; }
__device__ __forceinline__ ff operator-(ff a, ff b) { return a + (-b); }
__device__ __forceinline__ ff operator*(ff a, ff b) {
    const float p = __fmul_rn(a.h, b.h);
    return {p, fmaf(a.l, b.h, fmaf(a.h, b.l, fmaf(a.h, b.h, -p)))};
}
__device__ __forceinline__ ff norm(ff a) {           // |a.l| <= |a.h|
    const float s = __fadd_rn(a.h, a.l);
    return {s, __fadd_rn(__fsub_rn(a.h, s), a.l)};
}
__device__ __forceinline__ cff operator+(cff a, cff b) { return {a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ cff operator-(cff a, cff b) { return {a.x - b.x, a.y - b.y}; }
__device__ __forceinline__ cff operator*(cff a, cff b) {
    return {a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x};
}
__device__ __forceinline__ cff conj(cff a) { return {a.x, -a.y}; }
__device__ __forceinline__ cff from4(float4 v) { return {{v.x, v.y}, {v.z, v.w}}; }
__device__ __forceinline__ float4 to4(cff v) { return make_float4(v.x.h, v.x.l, v.y.h, v.y.l); }

// ---- positions, window, tables ---------------------------------------------------------------
constexpr int kFrac = 46;                          // position bits below one lag cell
constexpr unsigned long long kFracMask = (1ull << kFrac) - 1;
constexpr int kPieceBits = 7, kPieces = 1 << kPieceBits;
constexpr int kSplitMaxW = 12;
constexpr int kLagTile = 64;                       // first-tap tile side
constexpr int kLagLd = 76;                         // tile cells with the taps' reach, row pitch
constexpr int kLagCells = kLagLd * kLagLd;
constexpr int kProdBits = 44;                      // window products in units of 2^-44
constexpr int kMaxChunk = 1023;                    // samples of one work item (see k_lag_spread)
constexpr int kLagThreads = 512, kLagWarps = kLagThreads / 32;

// Window polynomials: with f = (first tap) - (u - w/2) in [0, 1), piece i = floor(128 f) and
// y = 128 f - i - 1/2, phi of tap l is c0 + y (c1 + y (c2 + y (c3 + y c4))), interpolating
// phi(w/2 - l - f) at five Chebyshev points; c0, c1, c2 as pairs. ta = {c0, c1}, tb = {c2, c3, c4},
// indexed [i * w + l]. Lag weights: fac[m + N] = r(m)^2 (N - |m|) / N^2, m = -N..N-1, r the
// reciprocal window transform (applied twice: on the way in and on the way out).
// Eight lanes per polynomial: lane n < 5 evaluates the window at node n, lane k < 5 sums
// coefficient k.
// Done by the first blocks of k_lag_origin: in a launch of its own 10 us of FP64 latency on a small
// grid (weights of a 211 k-sample raster 291 us, now 283; of 20 k 166, 163).
struct TableArgs {
    int W, N, blocks;
    double beta;
    float4 *ta, *tb;
    const double* r;
    float2* fac;
};
__device__ __forceinline__ void lag_tables(const TableArgs& t, int block) {
    const int W = t.W, N = t.N;
    const double beta = t.beta, *r = t.r;
    float4 *ta = t.ta, *tb = t.tb;
    float2* fac = t.fac;
    const int tid = block * 256 + threadIdx.x, id = tid >> 3, n = tid & 7;
    if (id < kPieces * W) {                        // uniform within the eight lanes
        const unsigned mask = 0xffu << (threadIdx.x & 24);
        const int i = id / W, l = id - i * W;
        auto co = [](int m) {                      // cos(pi m / 10)
            const double c[11] = {1.0, 0.95105651629515357, 0.80901699437494745,
                                  0.58778525229247314, 0.30901699437494745, 0.0,
                                  -0.30901699437494745, -0.58778525229247314,
                                  -0.80901699437494745, -0.95105651629515357, -1.0};
            m %= 20;
            return c[m <= 10 ? m : 20 - m];
        };
        const double z = (0.5 * W - l - (i + 0.5 + 0.5 * co(2 * n + 1)) / kPieces) * (2.0 / W);
        const double q = 1.0 - z * z;
        const double f = q >= 0.0 ? exp(beta * (sqrt(q) - 1.0)) : 0.0;
        double ak = 0.0;                           // Chebyshev coefficient n
        for (int m = 0; m < 5; ++m)
            ak += (n == 0 ? 0.2 : 0.4) * __shfl_sync(mask, f, m, 8) * co((2 * m + 1) * n);
        double a[5];
        for (int k = 0; k < 5; ++k) a[k] = __shfl_sync(mask, ak, k, 8);
        // powers of Y = 2 y, then of y
        const double c[3] = {a[0] - a[2] + a[4], 2.0 * (a[1] - 3.0 * a[3]),
                             4.0 * (2.0 * a[2] - 8.0 * a[4])};
        float h[3], lo[3];
        for (int k = 0; k < 3; ++k) {
            h[k] = (float)c[k];
            lo[k] = (float)(c[k] - (double)h[k]);
        }
        if (n == 0) ta[id] = make_float4(h[0], lo[0], h[1], lo[1]);
        if (n == 1) tb[id] = make_float4(h[2], lo[2], (float)(32.0 * a[3]), (float)(128.0 * a[4]));
    }
    if (tid < 2 * N) {
        const int m = tid - N;
        const double v = r[tid] * r[tid] * (double)(N - (m < 0 ? -m : m)) / ((double)N * N);
        const float h = (float)v;
        fac[tid] = make_float2(h, (float)(v - (double)h));
    }
}

__device__ __forceinline__ ff window_eval(const float4& a, const float4& b, float yh, float yl) {
    const float p2 = __fmul_rn(yh, fmaf(b.w, yh, b.z));
    const float bh = __fadd_rn(b.x, p2);
    const float bl = __fadd_rn(__fadd_rn(__fsub_rn(b.x, bh), p2), b.y);
    const float p1 = __fmul_rn(yh, bh);
    const float e1 = fmaf(yl, bh, fmaf(yh, bl, fmaf(yh, bh, -p1)));
    const ff s1 = two_sum(a.z, p1);
    const float al = __fadd_rn(s1.l, __fadd_rn(e1, a.w));
    const float p0 = __fmul_rn(yh, s1.h);
    const float e0 = fmaf(yl, s1.h, fmaf(yh, al, fmaf(yh, s1.h, -p0)));
    const float h = __fadd_rn(a.x, p0);
    return {h, __fadd_rn(__fadd_rn(__fsub_rn(a.x, h), p0), __fadd_rn(e0, a.y))};
}

// piece and y = (yh, yl) of a position word (46 fraction bits)
__device__ __forceinline__ void piece_of(unsigned long long pos, unsigned* i, float* yh, float* yl) {
    constexpr int rb = kFrac - kPieceBits;         // 39 bits within a piece
    const unsigned long long f = pos & kFracMask;
    *i = (unsigned)(f >> rb);
    const long long v = (long long)(f & ((1ull << rb) - 1)) - (1ll << (rb - 1));
    *yh = (float)(int)(v >> 15) * 5.9604644775390625e-08f;                   // 2^-24
    *yl = (float)(int)(v & 32767) * 1.8189894035458565e-12f;                 // 2^-39
}

// A sorted sample: y of the x and of the y axis as pairs (float4), and in one word the first tap
// within the tile (6 + 6 bits: x << 6 | y), then the pieces (7 + 7 bits, x above y).
__device__ __forceinline__ int cell_of(unsigned w) {
    return (int)((w >> 6) & 63u) * kLagLd + (int)(w & 63u);
}

// Coordinates to positions: X = lambda 2^(46 + e) as an integer and u 2^46 = X mul / 2^64 with
// mul = 2^64 L / (N 2^e), e such that 2^62 <= mul < 2^63.
struct PosScale {
    double to_x, ok, N, invN;                      // 2^(46 + e); 2 sigma (the FP64 route's scale)
    long long mul;
};
inline PosScale pos_scale(int N, int L, double sigma) {
    int extra = 0;
    while (((long long)N << extra) <= 2ll * L) ++extra;      // mul < 2^63
    const unsigned __int128 num = (unsigned __int128)L << 64;
    const unsigned __int128 den = (unsigned __int128)N << extra;
    return {std::ldexp(1.0, kFrac + extra), 2.0 * sigma, (double)N, 1.0 / N,
            (long long)((num + den / 2) / den)};
}

// One axis: (first tap mod L) << 46 | f, or ~0 for a coordinate that is not finite or too large
// (the same test as the FP64 route's). In integers, so that u is right to a unit at every N: the
// FP64 product with L / N, off by half an ulp of u, put the weights off by 6e-10 at N = 300 and 65536
// periods from the origin. Far out (|lambda| >= 2^12 at L = 4 N) the whole periods are taken out
// first, which is exact.
__device__ __forceinline__ unsigned long long position(double lam, const PosScale& ps, int W, int L) {
    double t = __dmul_rn(lam, ps.to_x);            // exact
    if (((unsigned)__double2hiint(t) & 0x7fffffffu) >= (1023u + 62u) << 20) {
        const double q = __dmul_rn(lam, ps.ok);
        if (!isfinite(q) || !(fabs(q) < 1125899906842624.0)) return ~0ull;
        t = __dmul_rn(fma(-ps.N, rint(__dmul_rn(lam, ps.invN)), lam), ps.to_x);
    }
    const long long X = __double2ll_rn(t);
    const long long u = __mul64hi(X, ps.mul) +
                        (long long)(((unsigned long long)X * (unsigned long long)ps.mul) >> 63);
    const long long a = u - ((long long)W << (kFrac - 1));
    const long long c = (a + (long long)kFracMask) >> kFrac;
    return ((unsigned long long)(c & (L - 1)) << kFrac) |
           (unsigned long long)((c << kFrac) - a);
}

// Per sample: the two position words and its rank among the samples of its tile (in arrival
// order, one atomic per warp and tile); the columns where taps start. Dropped samples get weight 0.
__global__ void __launch_bounds__(256)
    k_lag_origin(const double* __restrict__ lam, int M, const PosScale ps, int W,
                 int L, ulonglong2* __restrict__ pos, int* __restrict__ rank,
                 int* __restrict__ cnt, unsigned char* __restrict__ first,
                 double* __restrict__ alpha, const TableArgs tables) {
    const int nt = L / kLagTile, lane = threadIdx.x & 31;
    const int block = (int)blockIdx.x - tables.blocks, nblocks = (int)gridDim.x - tables.blocks;
    if (block < 0) {
        lag_tables(tables, (int)blockIdx.x);
        return;
    }
    for (int64_t base = (int64_t)block * blockDim.x + (threadIdx.x & ~31); base < M;
         base += (int64_t)nblocks * blockDim.x) {
        const int64_t j = base + lane;
        int tile = -1;
        if (j < M) {
            const unsigned long long px = position(lam[2 * j], ps, W, L);
            const unsigned long long py = position(lam[2 * j + 1], ps, W, L);
            if (px == ~0ull || py == ~0ull) {
                alpha[j] = 0.0;
                pos[j] = make_ulonglong2(~0ull, ~0ull);
            } else {
                const int cx = (int)(px >> kFrac), cy = (int)(py >> kFrac);
                tile = (cx / kLagTile) * nt + cy / kLagTile;
                first[cx] = 1;
                pos[j] = make_ulonglong2(px, py);
            }
        }
        const unsigned same = __match_any_sync(0xffffffffu, tile);
        const int leader = __ffs(same) - 1;
        int r0 = 0;
        if (lane == leader && tile >= 0) r0 = atomicAdd(cnt + tile, __popc(same));
        r0 = __shfl_sync(0xffffffffu, r0, leader);
        if (tile >= 0) rank[j] = r0 + __popc(same & ((1u << lane) - 1u));
    }
}

// One block: start[t] = samples before tile t, items {tile, begin, end} of at most chunk samples
// each, and occ[p] = some tap reaches column 2 p or 2 p + 1.
constexpr int kScanThreads = 1024;
__global__ void __launch_bounds__(kScanThreads)
    k_lag_scan(const int* __restrict__ cnt, int ntiles, int chunk, int* __restrict__ start,
               int4* __restrict__ items, int* __restrict__ nitems,
               const unsigned char* __restrict__ first, int W, int L,
               unsigned char* __restrict__ occ) {
    __shared__ int s_a[kScanThreads / 32], s_b[kScanThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int per = (ntiles + kScanThreads - 1) / kScanThreads;
    const int t0 = min(ntiles, tid * per), t1 = min(ntiles, t0 + per);
    int a = 0, b = 0;
    for (int t = t0; t < t1; ++t) {
        a += cnt[t];
        b += (cnt[t] + chunk - 1) / chunk;
    }
    int xa = a, xb = b;
    for (int o = 1; o < 32; o <<= 1) {
        const int ya = __shfl_up_sync(0xffffffffu, xa, o), yb = __shfl_up_sync(0xffffffffu, xb, o);
        if (lane >= o) {
            xa += ya;
            xb += yb;
        }
    }
    if (lane == 31) {
        s_a[warp] = xa;
        s_b[warp] = xb;
    }
    __syncthreads();
    if (warp == 0) {
        int va = s_a[lane], vb = s_b[lane];
        for (int o = 1; o < 32; o <<= 1) {
            const int ya = __shfl_up_sync(0xffffffffu, va, o);
            const int yb = __shfl_up_sync(0xffffffffu, vb, o);
            if (lane >= o) {
                va += ya;
                vb += yb;
            }
        }
        s_a[lane] = va;
        s_b[lane] = vb;
    }
    __syncthreads();
    a = xa - a + (warp ? s_a[warp - 1] : 0);
    b = xb - b + (warp ? s_b[warp - 1] : 0);
    for (int t = t0; t < t1; ++t) {
        const int n = cnt[t];
        start[t] = a;
        for (int k = 0; k < n; k += chunk) items[b++] = make_int4(t, a + k, a + min(n, k + chunk), 0);
        a += n;
    }
    if (tid == kScanThreads - 1) *nitems = s_b[kScanThreads / 32 - 1];
    for (int p = tid; p < L / 2; p += kScanThreads) {
        unsigned char any = 0;
        for (int q = 0; q <= W; ++q) any |= first[(2 * p + 1 - q) & (L - 1)];
        occ[p] = any;
    }
}

__global__ void __launch_bounds__(256)
    k_lag_scatter(const ulonglong2* __restrict__ pos, const int* __restrict__ rank, int M, int L,
                  const int* __restrict__ start, float4* __restrict__ sy,
                  uint2* __restrict__ sw) {
    const int nt = L / kLagTile;
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < M;
         j += (int64_t)gridDim.x * blockDim.x) {
        const ulonglong2 p = pos[j];
        if (p.x == ~0ull) continue;
        const unsigned cx = (unsigned)(p.x >> kFrac), cy = (unsigned)(p.y >> kFrac);
        const int at = start[cx / kLagTile * nt + cy / kLagTile] + rank[j];
        unsigned ix, iy;
        float4 y;
        piece_of(p.x, &ix, &y.x, &y.y);
        piece_of(p.y, &iy, &y.z, &y.w);
        sy[at] = y;
        sw[at] = make_uint2((cx % kLagTile) << 6 | cy % kLagTile | iy << 12 | ix << 19, (unsigned)j);
    }
}

// zero the occupied column pairs of the grid (2 L doubles each)
__global__ void __launch_bounds__(256)
    k_lag_zero(double* __restrict__ grid, const unsigned char* __restrict__ occ, int L) {
    if (!occ[blockIdx.x]) return;
    double2* g = reinterpret_cast<double2*>(grid + (int64_t)blockIdx.x * 2 * L);
    for (int i = threadIdx.x; i < L; i += 256) g[i] = make_double2(0.0, 0.0);
}

// ---- W1 ----------------------------------------------------------------------------------------
// One item = up to kMaxChunk samples of one tile, accumulated in shared memory. A warp takes one
// sample at a time: lanes 0..w-1 evaluate its y taps, lanes 16..16+w-1 its x taps; then lane (h, l)
// adds the products of x taps h, h + 2, ... with y tap l, 24 of 32 lanes on two rows of distinct
// banks. A window value is a 22-bit integer plus a remainder below 2^-22 kept in FP32 (units 2^-44),
// so a product is one 32 x 32 -> 64 bit multiply plus two FP32 multiply-adds that round the cross
// terms to an integer. The 64-bit sum T of a cell is kept by two native 32-bit shared-memory
// atomics that need nothing back: T mod 2^32, and A = the sum of the products >> 22. With fewer than
// 1024 products, each at most 2^44, A does not overflow and A 2^22 <= T < A 2^22 + 2^32, which
// determines T. The grid receives the sums as integers in FP64.
// Two 32-bit shared atomics per tap are the cheapest sum on this GPU (large ping, 302 M taps,
// probe without arithmetic): 111 us, against 293 for 64-bit shared atomics, 483 for 64-bit and
// 585 for FP64 global ones. Bound: instruction issue. Large ping: 1657 us in FP64 with global
// atomics; here 367 us (223 instructions per sample with 64-bit products and a carry, 579 us).
struct SpreadSmem {
    float4 ta[kPieces * kSplitMaxW], tb[kPieces * kSplitMaxW];
    unsigned lo[kLagCells], hi[kLagCells];
    float4 xv[kLagWarps][16];
    int item;
};

// WT: the window width at compile time (0: the argument)
template <int WT>
__global__ void __launch_bounds__(kLagThreads, 2)
    k_lag_spread(const float4* __restrict__ sy, const uint2* __restrict__ sw,
                 const int4* __restrict__ items, const int* __restrict__ nitems,
                 int* __restrict__ next, const float4* __restrict__ ta,
                 const float4* __restrict__ tb, int w_arg, int L, double* __restrict__ grid) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SpreadSmem& s = *reinterpret_cast<SpreadSmem*>(smem_raw);
    const int W = WT ? WT : w_arg;
    for (int i = threadIdx.x; i < kPieces * W; i += kLagThreads) {
        s.ta[i] = ta[i];
        s.tb[i] = tb[i];
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, h = lane >> 4, l = lane & 15;
    const int tap = min(l, W - 1), nt = L / kLagTile, ni = *nitems, shift = h ? 19 : 12;
    const bool on = l < W;
    for (;;) {
        __syncthreads();                           // tables staged; the last item flushed
        if (threadIdx.x == 0) s.item = atomicAdd(next, 1);
        for (int i = threadIdx.x; i < kLagCells; i += kLagThreads) s.lo[i] = s.hi[i] = 0u;
        __syncthreads();
        if (s.item >= ni) return;
        const int4 item = items[s.item];
        int j = item.y + warp;
        float4 py = make_float4(0.f, 0.f, 0.f, 0.f);
        unsigned pw = 0u;
        if (j < item.z) {
            py = sy[j];
            pw = sw[j].x;
        }
        while (j < item.z) {
            const float4 cy = py;
            const unsigned cw = pw;
            j += kLagWarps;
            if (j < item.z) {
                py = sy[j];
                pw = sw[j].x;
            }
            const int e = (int)((cw >> shift) & (kPieces - 1)) * W + tap;
            const ff v = window_eval(s.ta[e], s.tb[e], h ? cy.x : cy.z, h ? cy.y : cy.w);
            // v = v1 + v2 with v1 a multiple of 2^-22, v2 in [0, 2^-22); 0 <= v <= 1
            const float vh = fmaxf(0.f, v.h), t = __fadd_rd(2.0f, vh);
            unsigned i1 = __float_as_uint(t) - 0x40000000u;
            float v1 = __fsub_rn(t, 2.0f), v2 = __fadd_rn(__fsub_rn(vh, v1), v.l);
            if (v2 < 0.f && i1 > 0u) {             // borrow
                --i1;
                v1 -= 2.384185791015625e-07f;      // 2^-22
                v2 += 2.384185791015625e-07f;
            }
            v2 = fmaxf(0.f, v2) * 17592186044416.0f;
            if (h) s.xv[warp][l] = make_float4(__uint_as_float(i1), vh, v2, 0.f);
            const unsigned y1 = __shfl_sync(0xffffffffu, i1, l);
            const float y1f = __shfl_sync(0xffffffffu, v1, l);
            const float y2f = __shfl_sync(0xffffffffu, v2, l);
            __syncwarp();
            const int base = cell_of(cw) + h * kLagLd + l;
            if (on) {
#pragma unroll
                for (int k = 0; k < kSplitMaxW / 2; ++k) {
                    if (2 * k + h >= W) break;
                    const float4 x = s.xv[warp][2 * k + h];
                    // (x1 + x2) y2 + x2 y1, rounded to an integer in the low mantissa bits
                    const float c = fmaf(x.z, y1f, fmaf(x.y, y2f, 8388608.0f));
                    const unsigned long long prod = (unsigned long long)__float_as_uint(x.x) * y1 +
                                                    (__float_as_uint(c) - 0x4b000000u);
                    const int at = base + 2 * k * kLagLd;
                    atomicAdd(&s.lo[at], (unsigned)prod);
                    atomicAdd(&s.hi[at], (unsigned)(prod >> 22));
                }
            }
            __syncwarp();                          // the x taps are read before the next sample's
        }
        __syncthreads();
        const int X0 = item.x / nt * kLagTile, Y0 = item.x % nt * kLagTile;
        for (int r = warp; r < kLagTile + W - 1; r += kLagWarps) {
            double* g = grid + (int64_t)((X0 + r) & (L - 1)) * L;
            for (int c = lane; c < kLagTile + W - 1; c += 32) {
                const unsigned lo = s.lo[r * kLagLd + c];
                const unsigned long long a = (unsigned long long)s.hi[r * kLagLd + c] << 22;
                const unsigned long long v = a + (lo - (unsigned)a);
                if (v != 0ull) atomicAdd(g + ((Y0 + c) & (L - 1)), __ull2double_rn(v));
            }
        }
    }
}

// ---- transforms --------------------------------------------------------------------------------
// Stockham stages of radix 16 (then the rest) as in fft_smem.cuh, 16 values per thread in FP32
// pairs; exponent sign + throughout (a forward transform conjugates before and after). A CTA holds
// one line (two of 256, for a full warp): with 4096 values per CTA the x pass of a 20 k-sample ping
// (L = 1024, N = 256) was 64 CTAs and the forward y pass 128, 27.6 and 19.0 us (ncu); now 26.0 and
// 12.2.
// Twiddles from a table of pairs, [stage][(r - 1) NS + k] = exp(2 pi i r k / (NS R)).
__host__ __device__ constexpr int lag_lines(int L) { return L < 512 ? 512 / L : 1; }
__host__ __device__ constexpr int lag_threads(int L) { return L / 16 * lag_lines(L); }
__host__ __device__ constexpr size_t lag_smem(int L) {
    return (size_t)lag_lines(L) * sfft::padded_len(L) * sizeof(float4);
}
__host__ __device__ constexpr int lag_tw_offset(int L, int S) {
    int off = 0;
    for (int i = 1; i < S; ++i) off += (sfft::stage_radix(L, i) - 1) * sfft::stage_ns(L, i);
    return off;
}
constexpr int lag_tw_total(int L) { return lag_tw_offset(L, sfft::num_stages(L)); }

__device__ __forceinline__ constexpr ff pair_of(double v) {
    return {(float)v, (float)(v - (double)(float)v)};
}

// a exp(2 pi i m / 16), compile-time m in 0..7
template <int m>
__device__ __forceinline__ cff rot16(cff a) {
    constexpr double C = 0.92387953251128675613, S = 0.38268343236508977173,
                     R = 0.70710678118654752440;
    if constexpr (m == 0) {
        return a;
    } else if constexpr (m == 4) {
        return {-a.y, a.x};
    } else if constexpr (m == 2) {
        return {(a.x - a.y) * pair_of(R), (a.x + a.y) * pair_of(R)};
    } else if constexpr (m == 6) {
        return {(a.x + a.y) * pair_of(-R), (a.x - a.y) * pair_of(R)};
    } else {
        constexpr double c = m == 1 ? C : m == 3 ? S : m == 5 ? -S : -C;
        constexpr double s = m == 1 || m == 7 ? S : C;
        return a * cff{pair_of(c), pair_of(s)};
    }
}

template <int R, int LEN, int K = 0>
__device__ __forceinline__ void lag_butterflies(cff (&v)[R]) {
    if constexpr (K < LEN / 2) {
#pragma unroll
        for (int i = 0; i < R; i += LEN) {
            const cff a = v[i + K], b = rot16<K * (16 / LEN)>(v[i + K + LEN / 2]);
            v[i + K] = a + b;
            v[i + K + LEN / 2] = a - b;
        }
        lag_butterflies<R, LEN, K + 1>(v);
    }
}
template <int R, int LEN = 2>
__device__ __forceinline__ void lag_levels(cff (&v)[R]) {
    if constexpr (LEN <= R) {
        lag_butterflies<R, LEN>(v);
        lag_levels<R, LEN * 2>(v);
    }
}
template <int R>
__device__ __forceinline__ void lag_dft(cff (&v)[R]) {
    cff t[R];
#pragma unroll
    for (int i = 0; i < R; ++i) t[i] = v[sfft::bitrev(i, R)];
#pragma unroll
    for (int i = 0; i < R; ++i) v[i] = t[i];
    lag_levels<R>(v);
}

// In place: u[r] = x[t + r L / 16] in, u[r] = X[t + r L / 16] out, by the L / 16 threads of a line
// (t: index in the line, sm: the line's buffer, free on entry). The radix-16 stages are one loop at
// run time, not unrolled: unrolled, two transforms are more code than the instruction cache holds
// (x pass of the large ping 178 us with 3 of 5 stall cycles waiting for instructions, here 127).
template <int L>
__device__ __forceinline__ void lag_transform(cff (&u)[16], float4* sm,
                                              const float4* __restrict__ tw, int t) {
    constexpr int NSTAGE = sfft::num_stages(L), RL = sfft::stage_radix(L, NSTAGE - 1);
    constexpr int N16 = RL == 16 ? NSTAGE : NSTAGE - 1;      // stages of radix 16
#pragma unroll 1
    for (int S = 0, lg = 0; S < N16; ++S, lg += 4) {         // NS = 2^lg
        const int k = t & ((1 << lg) - 1);
        if (S > 0) {
#pragma unroll
            for (int r = 0; r < 16; ++r) u[r] = from4(sm[sfft::padded(t) + r * sfft::padded(L / 16)]);
            const float4* w = tw + k;
#pragma unroll
            for (int r = 1; r < 16; ++r) u[r] = u[r] * from4(__ldg(w + ((r - 1) << lg)));
            tw += 15 << lg;
            __syncthreads();                       // every read before any write
        }
        lag_dft<16>(u);
        if (RL != 16 || S + 1 < N16) {
            const int at = (t - k) * 16 + k;
#pragma unroll
            for (int q = 0; q < 16; ++q) sm[sfft::padded(at + (q << lg))] = to4(u[q]);
            __syncthreads();
        }
    }
    if constexpr (RL != 16) {                      // the rest: 16 / RL butterflies per thread
        constexpr int NS = L / RL, NB = 16 / RL;
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            const int j = t + b * (L / 16);        // < NS: the twiddle index too
            cff v[RL];
#pragma unroll
            for (int r = 0; r < RL; ++r) v[r] = from4(sm[sfft::padded(j + r * NS)]);
#pragma unroll
            for (int r = 1; r < RL; ++r) v[r] = v[r] * from4(__ldg(tw + (r - 1) * NS + j));
            lag_dft<RL>(v);
#pragma unroll
            for (int q = 0; q < RL; ++q) u[b + q * NB] = v[q];
        }
    }
    __syncthreads();                               // the buffer is free again
}

// a non-negative FP64 integer below 2^63, times 2^-kProdBits, as an FP32 pair (integer work only)
__device__ __forceinline__ ff pair_from_bits(double d) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(d);
    if (b == 0ull) return {0.f, 0.f};
    const int e = (int)(b >> 52) - 1023 - kProdBits;
    const float h = __uint_as_float(((unsigned)(e + 127) << 23) | ((unsigned)(b >> 29) & 0x7fffffu));
    const float u = __uint_as_float((unsigned)(e - 52 + 127) << 23);
    return {h, (float)((unsigned)b & 0x1fffffffu) * u};
}

// Along y: pair p of columns (2 p, 2 p + 1) as one complex line a + i b. INV = false: forward,
// the first N frequencies of each column into spec[m][x]; INV = true: from spec back to the two
// real columns, as FP32 pairs over the grid.
template <int L, bool INV>
__global__ void __launch_bounds__(lag_threads(L), 65536 / 128 / lag_threads(L))
    k_lag_fft_y(double* __restrict__ grid, float4* __restrict__ spec, int N,
                const unsigned char* __restrict__ occ, const float4* __restrict__ tw) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int LINES = lag_lines(L), TL = L / 16;
    const int line = threadIdx.x / TL, t = threadIdx.x - line * TL;
    const int p = blockIdx.x * LINES + line;
    float4* sm = reinterpret_cast<float4*>(smem_raw) + line * sfft::padded_len(L);
    const bool on = occ[p] != 0;
    if constexpr (LINES == 1) {
        if (!on) return;
    } else {
        if (!__syncthreads_or(on)) return;
    }
    cff u[16];
    if constexpr (!INV) {
        const double* a = grid + (int64_t)p * 2 * L;
#pragma unroll
        for (int r = 0; r < 16; ++r) {             // conjugated: a - i b
            const int y = t + r * TL;
            u[r] = {{0.f, 0.f}, {0.f, 0.f}};
            if (on) u[r] = {pair_from_bits(a[y]), -pair_from_bits(a[L + y])};
        }
        lag_transform<L>(u, sm, tw, t);
#pragma unroll
        for (int r = 0; r < 16; ++r) sm[sfft::padded(t + r * TL)] = to4(u[r]);
        __syncthreads();
        if (!on) return;
        // z(m) = conj(u(m)); A = (z(m) + conj z(L - m)) / 2, B = (z(m) - conj z(L - m)) / 2i
        for (int m = t; m < N; m += TL) {
            const cff z = conj(from4(sm[sfft::padded(m)]));
            const cff w = from4(sm[sfft::padded((L - m) & (L - 1))]);
            const cff A = z + w, B = z - w;
            auto half = [](ff x) -> ff { x = norm(x); return {0.5f * x.h, 0.5f * x.l}; };
            float4* o = spec + (int64_t)m * L + 2 * p;
            o[0] = to4({half(A.x), half(A.y)});
            o[1] = to4({half(B.y), half(-B.x)});
        }
    } else {
#pragma unroll
        for (int r = 0; r < 16; ++r) {             // A + i B, and its mirror image
            const int m = t + r * TL;
            const bool low = m < N, high = m > L - N;
            u[r] = {{0.f, 0.f}, {0.f, 0.f}};
            if (on && (low || high)) {
                const float4* s = spec + (int64_t)(low ? m : L - m) * L + 2 * p;
                const cff A = from4(s[0]), B = from4(s[1]);
                if (m == 0) u[r] = {A.x, B.x};
                else if (low) u[r] = {A.x - B.y, A.y + B.x};
                else u[r] = {A.x + B.y, B.x - A.y};
            }
        }
        lag_transform<L>(u, sm, tw, t);
        if (!on) return;
        float2* o = reinterpret_cast<float2*>(grid) + (int64_t)p * 2 * L;
#pragma unroll
        for (int r = 0; r < 16; ++r) {
            const ff re = norm(u[r].x), im = norm(u[r].y);
            o[t + r * TL] = make_float2(re.h, re.l);
            o[L + t + r * TL] = make_float2(im.h, im.l);
        }
    }
}

// Along x, rows m = 0..N-1 of spec: forward, times the lag weights, back (one loop, for the
// instruction cache); only occupied columns are read (the others are zero) and written. energy: the
// kEnergy partial sums of |coefficient|^2 over all frequencies, which is the mean square of the S grid.
constexpr int kEnergy = 32;
template <int L>
__global__ void __launch_bounds__(lag_threads(L), 65536 / 128 / lag_threads(L))
    k_lag_fft_x(float4* __restrict__ spec, int N, const unsigned char* __restrict__ occ,
                const float4* __restrict__ tw, const float2* __restrict__ fac,
                double* __restrict__ energy) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int LINES = lag_lines(L), TL = L / 16;
    const int line = threadIdx.x / TL, t = threadIdx.x - line * TL;
    const int m = blockIdx.x * LINES + line;
    float4* sm = reinterpret_cast<float4*>(smem_raw) + line * sfft::padded_len(L);
    const bool on = m < N;
    float4* row = spec + (int64_t)m * L;
    cff u[16];
#pragma unroll
    for (int r = 0; r < 16; ++r) {
        const int x = t + r * TL;
        u[r] = {{0.f, 0.f}, {0.f, 0.f}};
        if (on && occ[x >> 1]) u[r] = conj(from4(row[x]));
    }
    const float2 f2 = on ? fac[m + N] : make_float2(0.f, 0.f);
    const ff fy{f2.x, f2.y};
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {
        lag_transform<L>(u, sm, tw, t);
        if (pass == 0) {
            float sq = 0.f;
#pragma unroll
            for (int r = 0; r < 16; ++r) {
                const int q = t + r * TL;
                const int i = q < N ? q + N : q - (L - N);           // m_x + N
                if (q < N || q >= L - N) {
                    const float2 g = fac[i];
                    const ff f = fy * ff{g.x, g.y};
                    u[r] = {u[r].x * f, -(u[r].y * f)};
                    sq = fmaf(u[r].x.h, u[r].x.h, fmaf(u[r].y.h, u[r].y.h, sq));
                } else {
                    u[r] = {{0.f, 0.f}, {0.f, 0.f}};
                }
            }
            if (m > 0) sq += sq;                   // row -m
            for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
            if ((threadIdx.x & 31) == 0) atomicAdd(energy + blockIdx.x % kEnergy, (double)sq);
        }
    }
    if (!on) return;
#pragma unroll
    for (int r = 0; r < 16; ++r) {
        const int x = t + r * TL;
        if (occ[x >> 1]) row[x] = to4({norm(u[r].x), norm(u[r].y)});
    }
}

// ---- W3 and W4 ---------------------------------------------------------------------------------
// One item at a time: the tile's cells of the S grid (pairs) in shared memory, four lanes per
// sample; lane q holds taps q, q + 4, q + 8 of both axes, sums its columns over the x taps (shuffled)
// and weights them; alpha = 1 / S by one Newton step on the FP32 reciprocal. Bound: instruction issue
// (12 FP32 operations per tap). Large ping: 888 us in FP64 from global memory, here 306 us.
//
// The transforms' rounding is relative to the whole raster: it puts an S_k off by 1.1e-14 (rms) of the
// S grid's root mean square. A sample alone next to a dense cluster sees that as a larger relative error
// than the window's truncation once rms / S_k is above some 100 (N = 512: 1.2 times the error of the FP64
// route at 128..256, 1.9 at 256..1024; with 4 M samples in one spot 13 times). From kUneven on the raster is
// left to the FP64 route, whose rounding does not show. A polar raster reaches 11 (2 M samples, N = 256).
constexpr float kUneven = 64.0f;
constexpr unsigned kBadSum = 1u, kTooUneven = 2u;
struct InterpSmem {
    float4 ta[kPieces * kSplitMaxW], tb[kPieces * kSplitMaxW];
    float2 g[kLagCells];
    int item;
};

template <int WT>
__global__ void __launch_bounds__(kLagThreads, 2)
    k_lag_interp(const float4* __restrict__ sy, const uint2* __restrict__ sw,
                 const int4* __restrict__ items, const int* __restrict__ nitems,
                 int* __restrict__ next, const float4* __restrict__ ta,
                 const float4* __restrict__ tb, int w_arg, int L, const float2* __restrict__ grid,
                 const double* __restrict__ energy, const float2* __restrict__ fac, int N,
                 double* __restrict__ alpha, unsigned* __restrict__ bad,
                 unsigned* __restrict__ status) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    InterpSmem& s = *reinterpret_cast<InterpSmem*>(smem_raw);
    const int W = WT ? WT : w_arg;
    for (int i = threadIdx.x; i < kPieces * W; i += kLagThreads) {
        s.ta[i] = ta[i];
        s.tb[i] = tb[i];
    }
    const int q = threadIdx.x & 3, nt = L / kLagTile, ni = *nitems;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    static_assert(kEnergy == 32, "one lane per partial sum");
    double ms = energy[lane];
    for (int o = 16; o > 0; o >>= 1) ms += __shfl_xor_sync(0xffffffffu, ms, o);
    // S_k is a window's sum over the grid: 1 / r(0)^2 = 1 / (N fac[m = 0]) times its cells
    const float least = sqrtf((float)ms) / ((float)N * fac[N].x * kUneven);
    bool uneven = false;
    for (;;) {
        __syncthreads();                           // tables staged; the last tile consumed
        if (threadIdx.x == 0) s.item = atomicAdd(next, 1);
        __syncthreads();
        if (s.item >= ni) break;
        const int4 item = items[s.item];
        const int X0 = item.x / nt * kLagTile, Y0 = item.x % nt * kLagTile;
        for (int r = warp; r < kLagTile + W - 1; r += kLagWarps) {   // every y of those columns
            const float2* g = grid + (int64_t)((X0 + r) & (L - 1)) * L;
            for (int c = lane; c < kLagLd; c += 32) s.g[r * kLagLd + c] = g[(Y0 + c) & (L - 1)];
        }
        __syncthreads();
        for (int j0 = item.y; j0 < item.z; j0 += kLagThreads / 4) {
            const int j = j0 + threadIdx.x / 4;
            const bool on = j < item.z;
            const float4 y = sy[on ? j : item.y];
            const uint2 w = sw[on ? j : item.y];
            const int px = (int)(w.x >> 19) * W, py = (int)((w.x >> 12) & (kPieces - 1)) * W;
            ff fx[3], fy[3], acc[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const int l = q + 4 * c;
                fx[c] = fy[c] = acc[c] = {0.f, 0.f};
                if (l < W) {
                    fx[c] = window_eval(s.ta[px + l], s.tb[px + l], y.x, y.y);
                    fy[c] = window_eval(s.ta[py + l], s.tb[py + l], y.z, y.w);
                }
            }
            const float2* g = s.g + cell_of(w.x) + q;
#pragma unroll
            for (int r = 0; r < kSplitMaxW; ++r) {
                if (r >= W) break;
                const ff f{__shfl_sync(0xffffffffu, fx[r >> 2].h, r & 3, 4),
                           __shfl_sync(0xffffffffu, fx[r >> 2].l, r & 3, 4)};
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    const float2 v = g[r * kLagLd + 4 * c];
                    acc[c] = acc[c] + f * ff{v.x, v.y};
                }
            }
            ff sum = fy[0] * acc[0] + fy[1] * acc[1] + fy[2] * acc[2];
#pragma unroll
            for (int o = 1; o < 4; o <<= 1)
                sum = sum + ff{__shfl_xor_sync(0xffffffffu, sum.h, o),
                               __shfl_xor_sync(0xffffffffu, sum.l, o)};
            if (q == 0 && on) {
                sum = norm(sum);
                double a = 0.0;
                if (sum.h < least) {
                    uneven = true;
                } else if (sum.h > 0.0f && isfinite(sum.h)) {
                    const float r0 = __frcp_rn(sum.h);
                    const float e = fmaf(-sum.l, r0, fmaf(-sum.h, r0, 1.0f));
                    a = (double)r0 + (double)__fmul_rn(r0, e);
                } else if (!(atomicOr(status, STATUS_BAD_WEIGHT_SUM) & STATUS_BAD_WEIGHT_SUM)) {
                    atomicOr(bad, kBadSum);        // reported once per ftcg_check
                }
                alpha[w.y] = a;
            }
        }
    }
    if (uneven) atomicOr(bad, kTooUneven);
}

// ---- host ------------------------------------------------------------------------------------
// Twiddle tables of the six line lengths, per device, made on first use and kept (at most 0.4 MB).
std::mutex g_tw_mu;
std::map<std::pair<int, int>, float4*> g_tw;

ftcg_status_t lag_twiddles(int L, cudaStream_t s, const float4** out) {
    int dev = 0;
    FTCG_CK(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lk(g_tw_mu);
    auto it = g_tw.find({dev, L});
    if (it == g_tw.end()) {
        std::vector<float4> t((size_t)lag_tw_total(L));
        const long double tau = 6.283185307179586476925286766559L;
        for (int S = 1; S < sfft::num_stages(L); ++S) {
            const int R = sfft::stage_radix(L, S), NS = sfft::stage_ns(L, S);
            for (int r = 1; r < R; ++r)
                for (int k = 0; k < NS; ++k) {
                    const long double a = tau * ((long long)r * k) / ((long long)NS * R);
                    const double c = (double)std::cos(a), d = (double)std::sin(a);
                    const float ch = (float)c, dh = (float)d;
                    t[lag_tw_offset(L, S) + (r - 1) * NS + k] =
                        make_float4(ch, (float)(c - ch), dh, (float)(d - dh));
                }
        }
        float4* d = nullptr;
        FTCG_CK(cudaMalloc(&d, t.size() * sizeof(float4)));
        cudaError_t e = cudaMemcpyAsync(d, t.data(), t.size() * sizeof(float4),
                                        cudaMemcpyHostToDevice, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);   // complete before another stream's use
        if (e != cudaSuccess) cudaFree(d);
        FTCG_CK(e);
        it = g_tw.emplace(std::make_pair(dev, L), d).first;
    }
    *out = it->second;
    return FTCG_SUCCESS;
}

template <int L>
ftcg_status_t lag_transforms(double* grid, float4* spec, int N, const unsigned char* occ,
                             const float2* fac, const float4* tw, double* energy, cudaStream_t s) {
    constexpr int NT = lag_threads(L), LINES = lag_lines(L);
    const int sm = (int)lag_smem(L);
    FTCG_CK(cudaFuncSetAttribute(k_lag_fft_y<L, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm));
    FTCG_CK(cudaFuncSetAttribute(k_lag_fft_y<L, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm));
    FTCG_CK(cudaFuncSetAttribute(k_lag_fft_x<L>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm));
    k_lag_fft_y<L, false><<<L / 2 / LINES, NT, sm, s>>>(grid, spec, N, occ, tw);
    k_lag_fft_x<L><<<(N + LINES - 1) / LINES, NT, sm, s>>>(spec, N, occ, tw, fac, energy);
    k_lag_fft_y<L, true><<<L / 2 / LINES, NT, sm, s>>>(grid, spec, N, occ, tw);
    FTCG_CK(cudaGetLastError());
    return FTCG_SUCCESS;
}

// pool memory released on every path
struct Arena {
    char* p = nullptr;
    cudaStream_t s = nullptr;
    size_t used = 0;
    ~Arena() {
        if (p) pool_free(p, s);
    }
    template <typename T>
    T* take(size_t n) {                            // without memory: counts the bytes only
        T* q = p ? reinterpret_cast<T*>(p + used) : nullptr;
        used += (n * sizeof(T) + 255) & ~(size_t)255;
        return q;
    }
};

}  // namespace

// The lag grid side of this route: the power of two (256..8192) from 2 sigma N up; 0 where it is not
// taken: without such a side, with a window so wide (weight_width > 12, or exp(-beta) < 1e-13 at the
// plan's own oversampling) that its truncation no longer covers the pairs' rounding of about 1e-14,
// and where the truncation could be larger than on the FP64 route's grid of side 2 sigma N. It is the
// same on the same grid. On a finer one it is smaller on average, but varies from raster to raster by
// more than narrow windows or a grid a few per cent finer gain (rms error against that route, polar
// rasters: w = 4, sigma = 3 up to 5.0 times, w = 12 at sigma = 2.25, 1008 to 1024 cells, 2.7 times). The
// default window gains for certain from a tenth more cells on (0.01 to 0.6), and at the default
// sigma = 2 at every side measured (N = 64..1030: 0.01 to 1.03).
int split_lag_side(const Plan& p) {
    const int W = p.opts.weight_width > 0 ? p.opts.weight_width : 12;
    if (W > kSplitMaxW || es_beta(W, p.sigma) > 29.9) return 0;
    int L = 256;
    while (L < 2 * p.G) L <<= 1;
    if (L > 8192) return 0;
    const bool same = L == 2 * p.G && p.sigma >= 2.0;
    const bool finer = W == 12 && p.sigma >= 1.25 && p.sigma <= 2.0 &&
                       (p.sigma == 2.0 || L >= 2.2 * p.G);
    return same || finer ? L : 0;
}

// *uneven: the raster is left to the FP64 route (see kUneven); its weights here don't count.
ftcg_status_t compute_weights_split(Plan& p, double* d_alpha_out, cudaStream_t s, bool* uneven) {
    *uneven = false;
    const int W = p.opts.weight_width > 0 ? p.opts.weight_width : 12;
    const int L = split_lag_side(p), N = p.N, M = (int)p.M;
    const Window wa{W, es_beta(W, (double)L / (2.0 * N))};
    const float4* tw = nullptr;
    FTCG_TRY(lag_twiddles(L, s, &tw));
    int dev = 0, sms = 0;
    FTCG_CK(cudaGetDevice(&dev));
    FTCG_CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const int ntiles = (L / kLagTile) * (L / kLagTile);
    // items small enough that every SM gets some, large enough to amortise a tile's flush
    const int chunk = std::min(kMaxChunk, std::max(64, M / (4 * sms)));
    const int max_items = std::min(ntiles, M) + M / chunk;
    Arena ar;
    ar.s = s;
    double *r2, *grid, *alpha, *energy;
    float4 *ta, *tb, *spec;
    float2* fac;
    ulonglong2* pos;
    float4* sy;
    uint2* sw;
    int *rank, *start, *cnt, *nitems, *next;
    int4* items;
    unsigned char *first, *occ;
    unsigned* bad;
    size_t zero_bytes = 0;
    auto lay_out = [&]() {
        ar.used = 0;
        cnt = ar.take<int>(ntiles);                // cleared together, up to energy
        first = ar.take<unsigned char>(L);
        bad = ar.take<unsigned>(1);
        next = ar.take<int>(2);                    // item counters of W1 and W3
        energy = ar.take<double>(kEnergy);
        zero_bytes = ar.used;
        r2 = ar.take<double>(2 * (size_t)N);
        fac = ar.take<float2>(2 * (size_t)N);
        ta = ar.take<float4>(kPieces * W);
        tb = ar.take<float4>(kPieces * W);
        occ = ar.take<unsigned char>(L / 2);
        start = ar.take<int>(ntiles);
        items = ar.take<int4>(max_items);
        nitems = ar.take<int>(1);
        pos = ar.take<ulonglong2>(M);
        sy = ar.take<float4>(M);
        sw = ar.take<uint2>(M);
        rank = ar.take<int>(M);
        spec = ar.take<float4>((size_t)N * L);
        grid = ar.take<double>((size_t)L * L);
        alpha = d_alpha_out ? d_alpha_out : ar.take<double>(M);
    };
    lay_out();
    if (pool_malloc(&ar.p, ar.used, s) != cudaSuccess) {
        cudaGetLastError();
        ar.p = nullptr;
        set_error("ftcg_weights: cannot allocate the lag grid, its spectrum and the sorted samples "
                  "(%zu bytes)", ar.used);
        return FTCG_ERR_OUT_OF_MEMORY;
    }
    lay_out();
    FTCG_CK(cudaMemsetAsync(ar.p, 0, zero_bytes, s));
    FTCG_TRY(window_factors(r2, 2 * N, L, wa, s));
    const int tab = std::max(8 * kPieces * W, 2 * N);
    const TableArgs tables{W, N, (tab + 255) / 256, wa.beta, ta, tb, r2, fac};
    const int mb = std::min((M + 255) / 256, sms * 8);
    k_lag_origin<<<tables.blocks + mb, 256, 0, s>>>(p.lambda, M, pos_scale(N, L, p.sigma), W, L, pos,
                                                    rank, cnt, first, alpha, tables);
    k_lag_scan<<<1, kScanThreads, 0, s>>>(cnt, ntiles, chunk, start, items, nitems, first, W, L, occ);
    k_lag_scatter<<<mb, 256, 0, s>>>(pos, rank, M, L, start, sy, sw);
    k_lag_zero<<<L / 2, 256, 0, s>>>(grid, occ, L);
    const int ctas = std::min(max_items, 2 * sms);
    auto spread = W == 12 ? k_lag_spread<12> : k_lag_spread<0>;
    auto interp = W == 12 ? k_lag_interp<12> : k_lag_interp<0>;
    FTCG_CK(cudaFuncSetAttribute(spread, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)sizeof(SpreadSmem)));
    FTCG_CK(cudaFuncSetAttribute(interp, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)sizeof(InterpSmem)));
    spread<<<ctas, kLagThreads, sizeof(SpreadSmem), s>>>(sy, sw, items, nitems, next, ta, tb, W, L,
                                                         grid);
    FTCG_CK(cudaGetLastError());
    switch (L) {
        case 256: FTCG_TRY(lag_transforms<256>(grid, spec, N, occ, fac, tw, energy, s)); break;
        case 512: FTCG_TRY(lag_transforms<512>(grid, spec, N, occ, fac, tw, energy, s)); break;
        case 1024: FTCG_TRY(lag_transforms<1024>(grid, spec, N, occ, fac, tw, energy, s)); break;
        case 2048: FTCG_TRY(lag_transforms<2048>(grid, spec, N, occ, fac, tw, energy, s)); break;
        case 4096: FTCG_TRY(lag_transforms<4096>(grid, spec, N, occ, fac, tw, energy, s)); break;
        default: FTCG_TRY(lag_transforms<8192>(grid, spec, N, occ, fac, tw, energy, s)); break;
    }
    interp<<<ctas, kLagThreads, sizeof(InterpSmem), s>>>(
        sy, sw, items, nitems, next + 1, ta, tb, W, L, reinterpret_cast<const float2*>(grid), energy,
        fac, N, alpha, bad, p.status);
    FTCG_CK(cudaGetLastError());
    FTCG_TRY(launch_set_alpha(p, alpha, FTCG_WEIGHTS_F64, s));
    unsigned seen = 0;
    FTCG_CK(cudaMemcpyAsync(&seen, bad, sizeof(unsigned), cudaMemcpyDeviceToHost, s));
    FTCG_CK(cudaStreamSynchronize(s));
    *uneven = (seen & kTooUneven) != 0;
    if (seen & kBadSum) {
        set_error("ftcg_weights: a weight sum S_k was <= 0 or not finite (weight set to 0)");
        return FTCG_ERR_NUMERIC;
    }
    return FTCG_SUCCESS;
}

}  // namespace ftcg
