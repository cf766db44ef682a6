// Max pooling over NHWC fp32 activations: the one layer between the stem and the first residual
// block of the ResNets measured in Sec. 4.5, so that a whole convolution backbone can be chained
// through this library.  Pure streaming work with 16-byte loads and stores, window positions outside the image ignored.
// k_maxpool: any window, one thread per (output pixel, 4 channels), a load per window position.
// k_maxpool_3x3s2: the 3x3 / 2 window; a thread walks down ROWS output rows of its column and four channels, so that an input
// row is loaded once for the two output rows that share it and the loads of a whole column are in flight together.  Bound
// by HBM: 112 x 112 x 64 at batch 64 / 128 / 1 takes 45 / 85 / 2.0 us (78 / 151 / 3.8 with k_maxpool; copy rate: 39 / 78 / 0.6).
#include <cfloat>

#include "nm_internal.h"
#include "nm_ptx.cuh"

namespace {

__global__ void k_maxpool(const float4* __restrict__ x, int h, int w, int c4, int kh, int kw, int stride_h,
                          int stride_w, int pad_h, int pad_w, int ho, int wo, size_t total, float4* __restrict__ y)
{
    nmk::pdl_wait();   // x is usually the output of the kernel launched just before
    for (size_t i = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; i < total;
         i += static_cast<size_t>(gridDim.x) * blockDim.x) {
        const int cq = static_cast<int>(i % c4);
        size_t pix = i / c4;
        const int ow = static_cast<int>(pix % wo);
        pix /= wo;
        const int oh = static_cast<int>(pix % ho);
        const size_t n = pix / ho;
        float4 m = make_float4(-FLT_MAX, -FLT_MAX, -FLT_MAX, -FLT_MAX);
        for (int i_h = 0; i_h < kh; ++i_h) {
            const int ih = oh * stride_h - pad_h + i_h;
            if (ih < 0 || ih >= h) continue;
            for (int i_w = 0; i_w < kw; ++i_w) {
                const int iw = ow * stride_w - pad_w + i_w;
                if (iw < 0 || iw >= w) continue;
                const float4 v = __ldg(x + ((n * h + ih) * w + iw) * c4 + cq);
                m.x = fmaxf(m.x, v.x); m.y = fmaxf(m.y, v.y); m.z = fmaxf(m.z, v.z); m.w = fmaxf(m.w, v.w);
            }
        }
        y[i] = m;
    }
}

template <int ROWS>
__global__ void __launch_bounds__(256) k_maxpool_3x3s2(const float4* __restrict__ x, int h, int w, int c4, int pad_h, int pad_w, int ho, int wo,
                                                       int row_blocks, unsigned total, float4* __restrict__ y)
{
    // from the end: of an input that does not fit the L2, the part the kernel before wrote last is still there (7x7 / 2 stem and this at batch 64
    // 116.9 -> 109.2 us, at batch 128 216.4 -> 208.6)
    const unsigned id = (gridDim.x - 1u - blockIdx.x) * 256u + threadIdx.x;
    nmk::pdl_wait();
    if (id >= total) return;
    unsigned t = id / static_cast<unsigned>(c4);
    const int cq = static_cast<int>(id - t * static_cast<unsigned>(c4));
    unsigned u = t / static_cast<unsigned>(wo);
    const int ow = static_cast<int>(t - u * static_cast<unsigned>(wo));
    const unsigned n = u / static_cast<unsigned>(row_blocks);
    const int oh0 = static_cast<int>(u - n * static_cast<unsigned>(row_blocks)) * ROWS;
    // A position outside the image is replaced by the nearest one inside, which is in the window too (no window is empty).
    const int iw0 = ow * 2 - pad_w, ih0 = oh0 * 2 - pad_h;
    const int l = max(iw0, 0), m = min(max(iw0 + 1, 0), w - 1), r = min(iw0 + 2, w - 1);
    const float4* image = x + static_cast<size_t>(n) * h * w * c4 + cq;
    float4 row[2 * ROWS + 1];   // maximum over the three columns
#pragma unroll
    for (int i = 0; i < 2 * ROWS + 1; ++i) {
        const int ih = min(max(ih0 + i, 0), h - 1);
        const float4* src = image + static_cast<size_t>(ih) * w * c4;
        const float4 a = __ldg(src + static_cast<size_t>(l) * c4), b = __ldg(src + static_cast<size_t>(m) * c4),
                     c = __ldg(src + static_cast<size_t>(r) * c4);
        row[i] = make_float4(fmaxf(fmaxf(a.x, b.x), c.x), fmaxf(fmaxf(a.y, b.y), c.y), fmaxf(fmaxf(a.z, b.z), c.z),
                             fmaxf(fmaxf(a.w, b.w), c.w));
    }
    float4* dst = y + ((static_cast<size_t>(n) * ho + oh0) * wo + ow) * c4 + cq;
#pragma unroll
    for (int i = 0; i < ROWS; ++i) {
        if (oh0 + i >= ho) break;
        const float4 a = row[2 * i], b = row[2 * i + 1], c = row[2 * i + 2];
        // the lowest finite value stands for "no value", as in k_maxpool
        dst[static_cast<size_t>(i) * wo * c4] =
            make_float4(fmaxf(fmaxf(fmaxf(a.x, b.x), c.x), -FLT_MAX), fmaxf(fmaxf(fmaxf(a.y, b.y), c.y), -FLT_MAX),
                        fmaxf(fmaxf(fmaxf(a.z, b.z), c.z), -FLT_MAX), fmaxf(fmaxf(fmaxf(a.w, b.w), c.w), -FLT_MAX));
    }
}

// Self-test of the failure path the convolution kernels share: a wait on a barrier that nobody will
// ever complete runs out of its poll budget, the block reports through the status word exactly as
// the kernels do, and returns normally.
__global__ void k_wait_expiry(int* status, uint32_t polls)
{
    __shared__ uint64_t bar;
    const uint32_t b = nmk::smem_u32(&bar);
    if (threadIdx.x == 0) {
        nmk::mbar_init(b, 1);
        nmk::mbar_fence_init();
    }
    __syncthreads();
    const bool ok = nmk::mbar_wait_polls(b, 0, polls);
    if (!__syncthreads_and(ok ? 1 : 0) && threadIdx.x == 0) {
        atomicExch(status + 0, static_cast<int>(NM_ERR_TIMEOUT));
        atomicExch(status + 1, 99);   // where: the self-test
        atomicExch(status + 2, static_cast<int>(blockIdx.x));
    }
}

}  // namespace

extern "C" nm_status_t nm_selftest_wait_expiry(const nm_weights_t* w, void* cuda_stream)
{
    if (!w || w->magic != NM_MAGIC) return nmhost::fail(NM_ERR_INVALID_ARG, "nm_selftest_wait_expiry: bad weights handle");
    k_wait_expiry<<<1, 32, 0, static_cast<cudaStream_t>(cuda_stream)>>>(w->status, 2000u);
    nmhost::count_launch(1);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return nmhost::fail(NM_ERR_CUDA, "nm_selftest_wait_expiry launch: %s", cudaGetErrorString(e));
    return NM_OK;
}

extern "C" nm_status_t nm_maxpool2d(const float* x, int batch, int h, int w, int c, int kh, int kw, int stride_h,
                                    int stride_w, int pad_h, int pad_w, float* y, void* cuda_stream)
{
    if (!x || !y) return nmhost::fail(NM_ERR_INVALID_ARG, "nm_maxpool2d: x or y is NULL");
    if (batch < 1 || h < 1 || w < 1 || c < 1 || kh < 1 || kw < 1 || stride_h < 1 || stride_w < 1 || pad_h < 0 || pad_w < 0)
        return nmhost::fail(NM_ERR_INVALID_ARG, "nm_maxpool2d: sizes must be positive, padding >= 0");
    if (pad_h >= kh || pad_w >= kw)
        return nmhost::fail(NM_ERR_INVALID_ARG, "nm_maxpool2d: padding must be smaller than the window (no empty windows)");
    if (c % 4 != 0) return nmhost::fail(NM_ERR_UNSUPPORTED, "nm_maxpool2d: c must be a multiple of 4");
    if ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(y)) & 15u)
        return nmhost::fail(NM_ERR_INVALID_ARG, "nm_maxpool2d: x and y must be 16-byte aligned");
    const long long eh = static_cast<long long>(h) + 2ll * pad_h - kh, ew = static_cast<long long>(w) + 2ll * pad_w - kw;
    if (eh < 0 || ew < 0) return nmhost::fail(NM_ERR_INVALID_ARG, "nm_maxpool2d: the window does not fit the padded image");
    const int ho = static_cast<int>(eh / stride_h) + 1, wo = static_cast<int>(ew / stride_w) + 1;
    const cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    // Four rows per thread where that still makes two full rounds of threads (2048 per SM), one row below (fewer threads
    // than that leave the loads of too few columns in flight).
    const long long columns = static_cast<long long>(batch) * wo * (c / 4);
    const bool tall = columns * ((ho + 3) / 4) >= 148ll * 2048 * 2;
    const int row_blocks = tall ? (ho + 3) / 4 : ho;
    if (kh == 3 && kw == 3 && stride_h == 2 && stride_w == 2 && columns * row_blocks < (1ll << 31)) {
        const unsigned n = static_cast<unsigned>(columns * row_blocks);
        cudaError_t e = nmhost::launch_pdl(tall ? k_maxpool_3x3s2<4> : k_maxpool_3x3s2<1>, (n + 255u) / 256u, 256u, 0, st,
                                           reinterpret_cast<const float4*>(x), h, w, c / 4, pad_h, pad_w, ho, wo, row_blocks, n,
                                           reinterpret_cast<float4*>(y));
        nmhost::count_launch(1);
        if (e == cudaSuccess) e = cudaGetLastError();
        if (e != cudaSuccess) return nmhost::fail(NM_ERR_CUDA, "nm_maxpool2d launch: %s", cudaGetErrorString(e));
        return NM_OK;
    }
    const size_t total = static_cast<size_t>(batch) * ho * wo * (c / 4);
    size_t blocks = (total + 255) / 256;
    if (blocks > 148 * 16) blocks = 148 * 16;
    cudaError_t e = nmhost::launch_pdl(k_maxpool, static_cast<unsigned>(blocks), 256u, 0, st,
                                       reinterpret_cast<const float4*>(x), h, w, c / 4, kh, kw, stride_h, stride_w, pad_h,
                                       pad_w, ho, wo, total, reinterpret_cast<float4*>(y));
    nmhost::count_launch(1);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) return nmhost::fail(NM_ERR_CUDA, "nm_maxpool2d launch: %s", cudaGetErrorString(e));
    return NM_OK;
}
