// The inverse FFT of the adjoint for power-of-two grid sides, as two passes of shared-memory
// transforms, the second fused with the window division and crop (Eq. twodcg's sum over l, then
// Eq. newadm):
//   pass A  one CTA per block of kColBlock adjacent grid columns that some tap reaches: the
//           columns are loaded into shared memory, transformed along y (length G) and stored back;
//           columns no tap reaches are zero and stay zero, so they are skipped;
//   pass B  one CTA per image row: grid row (p_y mod G) is loaded, transformed along x, and only
//           the N kept frequencies p_x are written, each divided by the window transforms
//           (I_p = h_p / (phi^(p_x / G) phi^(p_y / G))), straight into the image.
// Each 1-D transform is a self-sorting (Stockham) sequence of radix-16/8/4/2 stages: with
// Ns the size of the transforms already done, a stage takes the R values
// x[j + r L / R] (r = 0..R-1), multiplies value r by w^(r k L / (Ns R)), k = j mod Ns,
// w = exp(+2 pi i / L), takes their R-point DFT V_q (sign +) and writes V_q to
// y[(j - k) R + k + q Ns]; after the last stage (Ns = L) the output is in natural order.
// Twiddles come from per-stage tables of w^m computed in FP64 and rounded to FP32; shared-memory
// indices are padded by one element per 16 to spread strided accesses over the banks.

#include "fft_smem.cuh"

#include <algorithm>
#include <cmath>
#include <map>
#include <mutex>
#include <utility>
#include <vector>

namespace ftcg {

namespace {

using namespace sfft;

template <int L>
__global__ void __launch_bounds__(kColThreads, kColMinBlocks)
    k_fft_cols(float2* __restrict__ grid, const int* __restrict__ blocks,
               const float2* __restrict__ tw) {
    extern __shared__ float2 sm[];
    pdl_wait();                                // the grid is complete
    pdl_allow_next();
    cols_body<L>(grid, blocks[blockIdx.x] * kColBlock, tw, sm);
}

template <int L>
__global__ void __launch_bounds__(row_threads(L))
    k_fft_rows_crop(const float2* __restrict__ grid, const unsigned* __restrict__ mask,
                    const float2* __restrict__ tw, const float2* __restrict__ r2, int N,
                    float2* __restrict__ img) {
    extern __shared__ float2 sm[];
    pdl_wait();                                // the column pass is complete
    rows_body<L>(grid, mask, tw, r2, N, img, blockIdx.x, sm);
}

template <int L>
ftcg_status_t run_smem_fft(const Plan& p, float2* img, cudaStream_t s, cudaEvent_t mid) {
    const size_t smA = (size_t)kColBlock * col_stride(L) * sizeof(float2);
    const size_t smB = (size_t)padded_len(L) * sizeof(float2);
    FTCG_CK(cudaFuncSetAttribute(k_fft_cols<L>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)smA));
    FTCG_CK(cudaFuncSetAttribute(k_fft_rows_crop<L>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)smB));
    if (p.n_col_blocks > 0) {
        FTCG_CK(launch_pdl(k_fft_cols<L>, dim3(p.n_col_blocks), dim3(kColThreads), smA, s,
                           p.grid, (const int*)p.col_blocks, p.tw));
    }
    if (mid) FTCG_CK(cudaEventRecord(mid, s));
    FTCG_CK(launch_pdl(k_fft_rows_crop<L>, dim3(p.N), dim3(row_threads(L)), smB, s,
                       (const float2*)p.grid, (const unsigned*)p.col_mask, p.tw,
                       (const float2*)p.deapod2, p.N, img));
    return FTCG_SUCCESS;
}

template <int L>
__global__ void __launch_bounds__(row_threads(L))
    k_fft_fwd_rows(const float2* __restrict__ img, const unsigned* __restrict__ mask,
                   const float2* __restrict__ tw, const float2* __restrict__ r2, int N,
                   float2* __restrict__ grid) {
    extern __shared__ float2 sm[];
    pdl_wait();                                // the image, and the last use of the grid
    pdl_allow_next();
    fwd_rows_body<L>(img, mask, tw, r2, N, grid, blockIdx.x, sm);
}

template <int L>
__global__ void __launch_bounds__(kColThreads, kColMinBlocks)
    k_fft_fwd_cols(float2* __restrict__ grid, int N, const int* __restrict__ blocks,
                   const float2* __restrict__ tw) {
    extern __shared__ float2 sm[];
    pdl_wait();                                // the row pass is complete
    pdl_allow_next();
    fwd_cols_body<L>(grid, N, blocks[blockIdx.x] * kColBlock, tw, sm);
}

// Large ping (G = 2048, half of the columns occupied), us: zero fill, padding in FP64 and the full
// cuFFT transform 64; these two passes 24.
template <int L>
ftcg_status_t run_smem_fft_forward(const Plan& p, const float2* img, cudaStream_t s) {
    if (p.n_col_blocks == 0) return FTCG_SUCCESS;
    const size_t smA = (size_t)kColBlock * col_stride(L) * sizeof(float2);
    const size_t smB = (size_t)padded_len(L) * sizeof(float2);
    FTCG_CK(cudaFuncSetAttribute(k_fft_fwd_cols<L>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)smA));
    FTCG_CK(cudaFuncSetAttribute(k_fft_fwd_rows<L>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)smB));
    FTCG_CK(launch_pdl(k_fft_fwd_rows<L>, dim3(p.N), dim3(row_threads(L)), smB, s, img,
                       (const unsigned*)p.col_mask, p.tw, (const float2*)p.deapod2,
                       p.N, p.grid));
    FTCG_CK(launch_pdl(k_fft_fwd_cols<L>, dim3(p.n_col_blocks), dim3(kColThreads), smA, s, p.grid,
                       p.N, (const int*)p.col_blocks, p.tw));
    return FTCG_SUCCESS;
}

}  // namespace

ftcg_status_t exec_smem_fft_forward(Plan* p, const float2* img, cudaStream_t s) {
    switch (p->G) {
        case 64: return run_smem_fft_forward<64>(*p, img, s);
        case 128: return run_smem_fft_forward<128>(*p, img, s);
        case 256: return run_smem_fft_forward<256>(*p, img, s);
        case 512: return run_smem_fft_forward<512>(*p, img, s);
        case 1024: return run_smem_fft_forward<1024>(*p, img, s);
        case 2048: return run_smem_fft_forward<2048>(*p, img, s);
        case 4096: return run_smem_fft_forward<4096>(*p, img, s);
        default:
            set_error("internal: no shared-memory FFT for G = %d", p->G);
            return FTCG_ERR_NOT_SUPPORTED;
    }
}

bool smem_fft_supported(int G) {
    // From 64 on: the tiny raster's adjoint (G = 128) took three cuFFT launches and the window
    // division, 29.7 us in all; with the two passes 22.1.
    return G >= 64 && G <= 4096 && (G & (G - 1)) == 0;
}

namespace {

// Stage tables of the seven sides, per device, made on first use and kept (60 KB in all): a plan
// that computes its own spends 30 us in the host's sines and a transfer.
std::mutex g_tw_mu;
std::map<std::pair<int, int>, float2*> g_tw;

ftcg_status_t side_twiddles(int G, cudaStream_t s, const float2** out) {
    int dev = 0;
    FTCG_CK(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lk(g_tw_mu);
    auto it = g_tw.find({dev, G});
    if (it == g_tw.end()) {
        std::vector<float2> tw;
        switch (G) {
            case 64: tw = stage_twiddles<64>(); break;
            case 128: tw = stage_twiddles<128>(); break;
            case 256: tw = stage_twiddles<256>(); break;
            case 512: tw = stage_twiddles<512>(); break;
            case 1024: tw = stage_twiddles<1024>(); break;
            case 2048: tw = stage_twiddles<2048>(); break;
            default: tw = stage_twiddles<4096>(); break;
        }
        float2* d = nullptr;
        FTCG_CK(cudaMalloc(&d, tw.size() * sizeof(float2)));
        cudaError_t e = cudaMemcpyAsync(d, tw.data(), tw.size() * sizeof(float2),
                                        cudaMemcpyHostToDevice, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);   // complete before another stream's use
        if (e != cudaSuccess) cudaFree(d);
        FTCG_CK(e);
        it = g_tw.emplace(std::make_pair(dev, G), d).first;
    }
    *out = it->second;
    return FTCG_SUCCESS;
}

}  // namespace

ftcg_status_t build_smem_fft(Plan* p, const std::vector<unsigned char>& occ, cudaStream_t s,
                             int64_t* bytes) {
    const int G = p->G;
    std::vector<int> blocks;
    for (int b = 0; b < G / kColBlock; ++b) {
        bool any = false;
        for (int c = 0; c < kColBlock; ++c) any = any || occ[b * kColBlock + c];
        if (any) blocks.push_back(b);
    }
    p->n_col_blocks = (int)blocks.size();
    const size_t nmask = (G / kColBlock + 31) / 32, nblk = blocks.size();
    std::vector<int> up(nblk + nmask, 0);               // the blocks, then the mask
    std::copy(blocks.begin(), blocks.end(), up.begin());
    for (int b : blocks) up[nblk + (b >> 5)] |= (int)(1u << (b & 31));
    FTCG_CK(pool_malloc(&p->col_blocks, up.size() * sizeof(int), s));
    *bytes += up.size() * sizeof(int);
    p->col_mask = reinterpret_cast<unsigned*>(p->col_blocks + nblk);
    FTCG_CK(cudaMemcpyAsync(p->col_blocks, up.data(), up.size() * sizeof(int),
                            cudaMemcpyHostToDevice, s));
    FTCG_TRY(side_twiddles(G, s, &p->tw));
    FTCG_CK(cudaStreamSynchronize(s));          // the host vector goes out of scope
    p->smem_fft = true;
    return FTCG_SUCCESS;
}

ftcg_status_t exec_smem_fft(Plan* p, float2* img, cudaStream_t s, cudaEvent_t mid) {
    switch (p->G) {
        case 64: return run_smem_fft<64>(*p, img, s, mid);
        case 128: return run_smem_fft<128>(*p, img, s, mid);
        case 256: return run_smem_fft<256>(*p, img, s, mid);
        case 512: return run_smem_fft<512>(*p, img, s, mid);
        case 1024: return run_smem_fft<1024>(*p, img, s, mid);
        case 2048: return run_smem_fft<2048>(*p, img, s, mid);
        case 4096: return run_smem_fft<4096>(*p, img, s, mid);
        default:
            set_error("internal: no shared-memory FFT for G = %d", p->G);
            return FTCG_ERR_NOT_SUPPORTED;
    }
}

void release_smem_fft(Plan* p) {
    pool_free(p->col_blocks, nullptr);
    p->col_mask = nullptr;
    p->tw = nullptr;
    p->col_blocks = nullptr;
    p->n_col_blocks = 0;
    p->smem_fft = false;
}

}  // namespace ftcg
