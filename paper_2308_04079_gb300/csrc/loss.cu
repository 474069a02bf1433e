// loss.cu -- the training loss of Sec. 5.1: L = (1 - lambda) L1 + lambda (1 - SSIM), and its
// gradient with respect to the rendered image.
//
// SSIM (Wang et al. 2004) per channel with an 11x11 Gaussian window (sigma 1.5, normalised),
// C1 = 0.01^2, C2 = 0.03^2, zero padding outside the image ("same" size), averaged over all
// pixels and channels; L1 is the mean absolute difference.  With the window moments at pixel p
//   mx = w*x, my = w*y, Exx = w*x^2, Eyy = w*y^2, Exy = w*(x y)   (w* = windowed sum)
//   A1 = 2 mx my + C1, A2 = 2 (Exy - mx my) + C2, B1 = mx^2 + my^2 + C1,
//   B2 = Exx - mx^2 + Eyy - my^2 + C2, S = A1 A2 / (B1 B2),
// the derivative of S(p) with respect to the image x at q is
//   w(p - q) [dS/dmx(p) + 2 x(q) dS/dExx(p) + y(q) dS/dExy(p)],
//   dS/dmx = 2 my (A2 - A1) / (B1 B2) - 2 mx S (B2 - B1) / (B1 B2),
//   dS/dExx = -S / B2,  dS/dExy = 2 A1 / (B1 B2),
// so dSSIM/dx = (w * a) + 2 x (w * b) + y (w * c) with the coefficient maps a, b, c of
// dS/dmx, dS/dExx, dS/dExy (w is symmetric).  Pass 1 computes the moments, S, L1 and the
// coefficient maps; pass 2 windows the coefficient maps and forms dL/dx.  Both passes are
// separable 11-tap convolutions on 32x32 output tiles (the three channels in turn), staged with
// their halo in shared memory.  Bound by the instructions of the windows: a thread computes four
// consecutive outputs of a row, then eight of a column, from registers, reading each input once for
// all of them, and the pairs (x, y), (x^2, y^2) and (a, b) go through packed arithmetic.  The window
// weights come with the arguments: computing them in fp64 in every block cost more than a third of
// both passes.  1080p: 111 + 92 us with scalar maps, two and four outputs per thread and in-kernel
// weights (210 us a call), now 131 us a call against 11 us for its 75 MB of images.
#include <cmath>
#include <cstring>

#include "gs_device.cuh"
#include "gs_kernels.h"

namespace gs {
namespace {

constexpr int kWin = 11, kHalf = 5;
constexpr int kTile = 32;
constexpr int kIn = kTile + 2 * kHalf;   // 42
constexpr int kLossThreads = 128;
constexpr int kRowsPer = 8;              // output rows per thread in the vertical passes
constexpr int kColsPer = 4;              // output columns per thread in the horizontal passes
static_assert(kTile * kTile == kLossThreads * kRowsPer, "one row group per thread");
constexpr int kItems = kIn * (kTile / kColsPer);   // (row, column group) items of a horizontal pass
// Row strides in elements: odd, so that lanes on consecutive rows hit different banks.
constexpr int kInStride = kIn + 1, kRowStride = kTile + 1;

struct LossArgs {
    const float* img;     // [3, H, W]
    const float* target;  // [3, H, W]
    int W, H;
    float lambda;
    float2* coef_ab;      // [3 channels][H * W]: dS/dmx, dS/dExx
    float* coef_c;        // [3 channels][H * W]: dS/dExy
    // normalised 1-D Gaussian window, sigma 1.5 (the 2-D one is its outer product), once and in pairs
    float win[kWin];
    f32x2 win2[kWin];
    double* partial;      // [blocks][2]: sums of S and |x - y| of every tile
    unsigned int* done;   // block counter of pass 1 (zeroed)
    float* out_loss;      // [3]: L, L1, mean SSIM
    float* dL_dimg;       // [3, H, W]
};

// The part of a tile's staged inputs one thread moves: column `col` of rows row, row + 3, ... (42
// columns x 3 rows = 126 of the 128 threads).  Pass 1 fetches the next channel's while this one is
// windowed (load latency was most of its stalls); pass 2 gains more from a sixth block per SM.
constexpr int kFetch = kIn / 3;
static_assert(kIn % 3 == 0 && 3 * kIn <= kLossThreads, "three rows per trip");
struct Fetch {
    int col, row, y0;
    bool on;
    const size_t at;      // of the first row's element in the image (valid where `on` and in range)
    __device__ __forceinline__ Fetch(const LossArgs& a, int bx, int by)
        : col(threadIdx.x % kIn), row(threadIdx.x / kIn), y0(by + (int)threadIdx.x / kIn - kHalf),
          on((int)threadIdx.x < 3 * kIn && bx + col - kHalf >= 0 && bx + col - kHalf < a.W),
          at((size_t)((long long)y0 * a.W + bx + col - kHalf)) {}
    __device__ __forceinline__ bool in(const LossArgs& a, int i) const {
        return on && (unsigned)(y0 + 3 * i) < (unsigned)a.H;
    }
    __device__ __forceinline__ size_t of(const LossArgs& a, int i) const { return at + (size_t)(3 * i) * a.W; }
    __device__ __forceinline__ bool stages() const { return (int)threadIdx.x < 3 * kIn; }
    __device__ __forceinline__ int slot(int i) const { return (row + 3 * i) * kInStride + col; }
};

// Pass 1: window moments, SSIM, L1 and the coefficient maps of one 32x32 tile, all channels.
__global__ void __launch_bounds__(kLossThreads, 5) k_ssim_forward(const __grid_constant__ LossArgs a) {
    __shared__ float2 s_in[kIn * kInStride];                                   // (x, y)
    __shared__ float2 s_m[kIn * kRowStride], s_q[kIn * kRowStride];            // windowed (x, y), (x^2, y^2)
    __shared__ float s_p[kIn * kRowStride];                                    // windowed x y
    __shared__ double s_red[2][8];
    const int tid = threadIdx.x;
    const int bx = blockIdx.x * kTile, by = blockIdx.y * kTile;
    const size_t P = (size_t)a.W * a.H;
    // per-thread sums of at most 3 x 8 terms in [-1, 1] and [0, 1] stay in fp32; blocks and the
    // grid sum in fp64
    float sum_s = 0.f, sum_l1 = 0.f;
    const Fetch f(a, bx, by);
    float fx[kFetch], fy[kFetch];
    auto fetch = [&](int ch) {
#pragma unroll
        for (int i = 0; i < kFetch; ++i) {
            fx[i] = f.in(a, i) ? a.img[ch * P + f.of(a, i)] : 0.f;
            fy[i] = f.in(a, i) ? a.target[ch * P + f.of(a, i)] : 0.f;
        }
    };
    fetch(0);
    for (int ch = 0; ch < 3; ++ch) {
        __syncthreads();   // the previous channel's reads of the staged maps are done
        if (f.stages())
#pragma unroll
            for (int i = 0; i < kFetch; ++i) s_in[f.slot(i)] = make_float2(fx[i], fy[i]);
        __syncthreads();
        // horizontal windows: lanes take consecutive rows of one column group
        for (int k = tid; k < kItems; k += kLossThreads) {
            const int c0 = (k / kIn) * kColsPer, r = k % kIn;
            f32x2 m[kColsPer], q[kColsPer];
            float p[kColsPer];
#pragma unroll
            for (int j = 0; j < kColsPer; ++j) {
                m[j] = q[j] = 0;
                p[j] = 0.f;
            }
#pragma unroll
            for (int cc = 0; cc < kColsPer + kWin - 1; ++cc) {
                const float2 v = s_in[r * kInStride + c0 + cc];
                const f32x2 v2 = pack2(v.x, v.y), vv = mul2(v2, v2);
                const float xy = v.x * v.y;
#pragma unroll
                for (int j = 0; j < kColsPer; ++j)
                    if (cc - j >= 0 && cc - j < kWin) {
                        const float w = a.win[cc - j];
                        const f32x2 w2 = a.win2[cc - j];
                        m[j] = fma2(w2, v2, m[j]);
                        q[j] = fma2(w2, vv, q[j]);
                        p[j] = fmaf(w, xy, p[j]);
                    }
            }
#pragma unroll
            for (int j = 0; j < kColsPer; ++j) {
                float2 o;
                unpack2(m[j], o.x, o.y);
                s_m[r * kRowStride + c0 + j] = o;
                unpack2(q[j], o.x, o.y);
                s_q[r * kRowStride + c0 + j] = o;
                s_p[r * kRowStride + c0 + j] = p[j];
            }
        }
        if (ch < 2) fetch(ch + 1);
        __syncthreads();
        const float C1 = 0.01f * 0.01f, C2 = 0.03f * 0.03f;
        // vertical windows: a thread takes kRowsPer consecutive rows of one column
        const int cc = tid % kTile, r0 = (tid / kTile) * kRowsPer;
        f32x2 mm[kRowsPer], qq[kRowsPer];
        float pp[kRowsPer];
#pragma unroll
        for (int j = 0; j < kRowsPer; ++j) {
            mm[j] = qq[j] = 0;
            pp[j] = 0.f;
        }
#pragma unroll
        for (int rr = 0; rr < kRowsPer + kWin - 1; ++rr) {
            const float2 m = s_m[(r0 + rr) * kRowStride + cc], q = s_q[(r0 + rr) * kRowStride + cc];
            const float p = s_p[(r0 + rr) * kRowStride + cc];
            const f32x2 m2 = pack2(m.x, m.y), q2 = pack2(q.x, q.y);
#pragma unroll
            for (int j = 0; j < kRowsPer; ++j)
                if (rr - j >= 0 && rr - j < kWin) {
                    const float w = a.win[rr - j];
                    const f32x2 w2 = a.win2[rr - j];
                    mm[j] = fma2(w2, m2, mm[j]);
                    qq[j] = fma2(w2, q2, qq[j]);
                    pp[j] = fmaf(w, p, pp[j]);
                }
        }
        float2* const ab = a.coef_ab + ch * P;
        float* const cm = a.coef_c + ch * P;
#pragma unroll
        for (int j = 0; j < kRowsPer; ++j) {
            const int r = r0 + j;
            const int px = bx + cc, py = by + r;
            if (px >= a.W || py >= a.H) continue;
            float mx, my, exx, eyy;
            unpack2(mm[j], mx, my);
            unpack2(qq[j], exx, eyy);
            const float exy = pp[j];
            const float A1 = 2.f * mx * my + C1, A2 = 2.f * (exy - mx * my) + C2;
            const float B1 = mx * mx + my * my + C1, B2 = (exx - mx * mx) + (eyy - my * my) + C2;
            const float inv = 1.f / (B1 * B2);
            const float S = A1 * A2 * inv;
            const size_t at = (size_t)py * a.W + px;
            ab[at] = make_float2(2.f * my * (A2 - A1) * inv - 2.f * mx * S * (B2 - B1) * inv, -S / B2);
            cm[at] = 2.f * A1 * inv;
            sum_s += S;
            const float2 v = s_in[(r + kHalf) * kInStride + cc + kHalf];
            sum_l1 += fabsf(v.x - v.y);
        }
    }
    // block sums (fixed order), then the last block adds the tiles in index order
    double d_s = sum_s, d_l1 = sum_l1;
    for (int o = 16; o > 0; o >>= 1) {
        d_s += __shfl_xor_sync(0xffffffffu, d_s, o);
        d_l1 += __shfl_xor_sync(0xffffffffu, d_l1, o);
    }
    if ((tid & 31) == 0) {
        s_red[0][tid >> 5] = d_s;
        s_red[1][tid >> 5] = d_l1;
    }
    __syncthreads();
    const int blocks = gridDim.x * gridDim.y, bid = blockIdx.y * gridDim.x + blockIdx.x;
    __shared__ bool s_last;
    if (tid == 0) {
        double s0 = 0.0, s1 = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) { s0 += s_red[0][w]; s1 += s_red[1][w]; }
        a.partial[2 * bid] = s0;
        a.partial[2 * bid + 1] = s1;
        __threadfence();
        s_last = atomicAdd(a.done, 1u) == (unsigned)(blocks - 1);
    }
    __syncthreads();
    if (s_last) {   // the last block: its threads sum the tiles' partials in a fixed order
        __threadfence();
        double p0 = 0.0, p1 = 0.0;
        for (int b = tid; b < blocks; b += blockDim.x) {
            p0 += __ldcg(a.partial + 2 * b);
            p1 += __ldcg(a.partial + 2 * b + 1);
        }
        for (int o = 16; o > 0; o >>= 1) {
            p0 += __shfl_xor_sync(0xffffffffu, p0, o);
            p1 += __shfl_xor_sync(0xffffffffu, p1, o);
        }
        __syncthreads();
        if ((tid & 31) == 0) {
            s_red[0][tid >> 5] = p0;
            s_red[1][tid >> 5] = p1;
        }
        __syncthreads();
    }
    if (s_last && tid == 0) {
        double s0 = 0.0, s1 = 0.0;
        for (int k = 0; k < (int)(blockDim.x >> 5); ++k) {
            s0 += s_red[0][k];
            s1 += s_red[1][k];
        }
        const double n = 3.0 * (double)P;
        const double ssim = s0 / n, l1 = s1 / n;
        a.out_loss[0] = (float)((1.0 - a.lambda) * l1 + a.lambda * (1.0 - ssim));
        a.out_loss[1] = (float)l1;
        a.out_loss[2] = (float)ssim;
    }
}

// Pass 2: dL/dx = (1 - lambda) sign(x - y) / N - lambda / N [(w * a) + 2 x (w * b) + y (w * c)].
__global__ void __launch_bounds__(kLossThreads, 6) k_ssim_backward(const __grid_constant__ LossArgs a) {
    __shared__ float2 s_ab[kIn * kInStride], s_hab[kIn * kRowStride];   // (a, b), staged and windowed by rows
    __shared__ float s_c[kIn * kInStride], s_hc[kIn * kRowStride];      // c
    const int tid = threadIdx.x;
    const int bx = blockIdx.x * kTile, by = blockIdx.y * kTile;
    const size_t P = (size_t)a.W * a.H;
    const float invN = 1.0f / (3.0f * (float)P);
    const Fetch f(a, bx, by);
    float2 fab[kFetch];
    float fc[kFetch];
    auto fetch = [&](int ch) {
#pragma unroll
        for (int i = 0; i < kFetch; ++i) {
            fab[i] = f.in(a, i) ? a.coef_ab[ch * P + f.of(a, i)] : make_float2(0.f, 0.f);
            fc[i] = f.in(a, i) ? a.coef_c[ch * P + f.of(a, i)] : 0.f;
        }
    };
    for (int ch = 0; ch < 3; ++ch) {
        fetch(ch);
        __syncthreads();   // the previous channel's reads of the staged maps are done
        if (f.stages())
#pragma unroll
            for (int i = 0; i < kFetch; ++i) {
                s_ab[f.slot(i)] = fab[i];
                s_c[f.slot(i)] = fc[i];
            }
        __syncthreads();
        for (int k = tid; k < kItems; k += kLossThreads) {
            const int c0 = (k / kIn) * kColsPer, r = k % kIn;
            f32x2 h[kColsPer];
            float hc[kColsPer];
#pragma unroll
            for (int j = 0; j < kColsPer; ++j) {
                h[j] = 0;
                hc[j] = 0.f;
            }
#pragma unroll
            for (int cc = 0; cc < kColsPer + kWin - 1; ++cc) {
                const float2 v = s_ab[r * kInStride + c0 + cc];
                const float c = s_c[r * kInStride + c0 + cc];
                const f32x2 v2 = pack2(v.x, v.y);
#pragma unroll
                for (int j = 0; j < kColsPer; ++j)
                    if (cc - j >= 0 && cc - j < kWin) {
                        const float w = a.win[cc - j];
                        const f32x2 w2 = a.win2[cc - j];
                        h[j] = fma2(w2, v2, h[j]);
                        hc[j] = fmaf(w, c, hc[j]);
                    }
            }
#pragma unroll
            for (int j = 0; j < kColsPer; ++j) {
                float2 o;
                unpack2(h[j], o.x, o.y);
                s_hab[r * kRowStride + c0 + j] = o;
                s_hc[r * kRowStride + c0 + j] = hc[j];
            }
        }
        __syncthreads();
        const int cc = tid % kTile, r0 = (tid / kTile) * kRowsPer;
        const int px = bx + cc;
        // the pixels of this thread, in flight during the vertical windows
        float xv[kRowsPer], yv[kRowsPer];
#pragma unroll
        for (int j = 0; j < kRowsPer; ++j) {
            const bool in = px < a.W && by + r0 + j < a.H;
            const size_t at = ch * P + (size_t)(by + r0 + j) * a.W + px;
            xv[j] = in ? a.img[at] : 0.f;
            yv[j] = in ? a.target[at] : 0.f;
        }
        f32x2 acc[kRowsPer];
        float accc[kRowsPer];
#pragma unroll
        for (int j = 0; j < kRowsPer; ++j) {
            acc[j] = 0;
            accc[j] = 0.f;
        }
#pragma unroll
        for (int rr = 0; rr < kRowsPer + kWin - 1; ++rr) {
            const float2 v = s_hab[(r0 + rr) * kRowStride + cc];
            const float c = s_hc[(r0 + rr) * kRowStride + cc];
            const f32x2 v2 = pack2(v.x, v.y);
#pragma unroll
            for (int j = 0; j < kRowsPer; ++j)
                if (rr - j >= 0 && rr - j < kWin) {
                    const float w = a.win[rr - j];
                    const f32x2 w2 = a.win2[rr - j];
                    acc[j] = fma2(w2, v2, acc[j]);
                    accc[j] = fmaf(w, c, accc[j]);
                }
        }
#pragma unroll
        for (int j = 0; j < kRowsPer; ++j) {
            const int py = by + r0 + j;
            if (px >= a.W || py >= a.H) continue;
            const float d = xv[j] - yv[j];
            const float sgn = d > 0.f ? 1.f : (d < 0.f ? -1.f : 0.f);
            float wa, wb;
            unpack2(acc[j], wa, wb);
            const float dssim = wa + 2.f * xv[j] * wb + yv[j] * accc[j];
            a.dL_dimg[ch * P + (size_t)py * a.W + px] = (1.f - a.lambda) * invN * sgn - a.lambda * invN * dssim;
        }
    }
}

}  // namespace
}  // namespace gs

using namespace gs;

extern "C" size_t gs_loss_workspace_size(int width, int height) {
    if (width <= 0 || height <= 0 || width > 32768 || height > 32768) return 0;
    const size_t P = (size_t)width * height;
    const size_t blocks = (size_t)((width + kTile - 1) / kTile) * ((height + kTile - 1) / kTile);
    return 256 + ((9 * P * sizeof(float) + 255) / 256) * 256 + blocks * 2 * sizeof(double);
}

extern "C" gs_status gs_loss_l1_dssim(const float* img, const float* target, int width, int height, float lambda,
                                     void* ws, size_t ws_bytes, float* out_loss, float* dL_dimg, cudaStream_t s) {
    const size_t need = gs_loss_workspace_size(width, height);
    if (!need || !img || !target || !ws || !out_loss || !dL_dimg || ws_bytes < need) return GS_ERR_INVALID_ARG;
    if (!(lambda >= 0.f && lambda <= 1.f)) return GS_ERR_INVALID_ARG;
    if (reinterpret_cast<uintptr_t>(ws) % 256) return GS_ERR_INVALID_ARG;
    const size_t P = (size_t)width * height;
    char* base = static_cast<char*>(ws);
    LossArgs a;
    a.img = img;
    a.target = target;
    a.W = width;
    a.H = height;
    a.lambda = lambda;
    a.done = reinterpret_cast<unsigned int*>(base);
    a.coef_ab = reinterpret_cast<float2*>(base + 256);
    a.coef_c = reinterpret_cast<float*>(base + 256) + 6 * P;
    double win[kWin], sum = 0.0;
    for (int k = 0; k < kWin; ++k) sum += win[k] = std::exp(-(double)((k - kHalf) * (k - kHalf)) / (2.0 * 1.5 * 1.5));
    for (int k = 0; k < kWin; ++k) {
        a.win[k] = (float)(win[k] / sum);
        const float pair[2] = {a.win[k], a.win[k]};
        std::memcpy(&a.win2[k], pair, sizeof(pair));
    }
    a.partial = reinterpret_cast<double*>(base + 256 + ((9 * P * sizeof(float) + 255) / 256) * 256);
    a.out_loss = out_loss;
    a.dL_dimg = dL_dimg;
    if (cudaMemsetAsync(a.done, 0, sizeof(unsigned int), s) != cudaSuccess) return GS_ERR_CUDA;
    const dim3 grid((width + kTile - 1) / kTile, (height + kTile - 1) / kTile);
    k_ssim_forward<<<grid, kLossThreads, 0, s>>>(a);
    k_ssim_backward<<<grid, kLossThreads, 0, s>>>(a);
    return cudaGetLastError() == cudaSuccess ? GS_OK : GS_ERR_CUDA;
}
