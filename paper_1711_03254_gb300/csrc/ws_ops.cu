// Elementwise pieces of the warm-start surrogate: pooling, upsampling and
// their adjoints, ReLU adjoint, masked MSE loss, Adam, FP32 -> BF16 copies.
// Channels-last tensors with row strides.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

#include "../../include/ws.h"

namespace ws {

using bf16 = __nv_bfloat16;

// The kernels from here to k_to_bf16 move data and do little else, so a thread
// handles V = 8 channels with 16-byte accesses where every row starts on a
// 16-byte boundary and C is a multiple of 8, and V = 1 otherwise; indices are
// 32-bit (I) where the element count allows, because a 64-bit division costs more
// than the element.  One thread per element with 64-bit divisions took, at 64^3
// positions: ReLU adjoint of 4 x 32 channels 103 us, upsampling to 64 channels
// 108, pooling of 32 channels 15.2, the cast of 16 channels 14.2.
template <int V, class T = bf16> struct Vec {
    // aligned for the 16-byte accesses below, wherever the compiler keeps it
    alignas(V * sizeof(T) % 16 == 0 ? 16 : alignof(T)) T v[V];
    __device__ __forceinline__ void load(const T *p) {
        if constexpr (V * sizeof(T) % 16 == 0) {
#pragma unroll
            for (int j = 0; j < (int)(V * sizeof(T) / 16); ++j)
                reinterpret_cast<uint4 *>(v)[j] = reinterpret_cast<const uint4 *>(p)[j];
        } else {
#pragma unroll
            for (int j = 0; j < V; ++j) v[j] = p[j];
        }
    }
    __device__ __forceinline__ void store(T *p) const {
        if constexpr (V * sizeof(T) % 16 == 0) {
#pragma unroll
            for (int j = 0; j < (int)(V * sizeof(T) / 16); ++j)
                reinterpret_cast<uint4 *>(p)[j] = reinterpret_cast<const uint4 *>(v)[j];
        } else {
#pragma unroll
            for (int j = 0; j < V; ++j) p[j] = v[j];
        }
    }
};

// vector i of a C-channel tensor of size (n, D, H, W): first channel and position
template <int V, class I>
__device__ __forceinline__ void decode(I i, int C, int W, int H, int D, int &c, int &x, int &y, int &z, int &n) {
    const I cv = (I)(C / V);
    I q = i / cv;
    c = (int)(i - q * cv) * V;
    I r = q / (I)W;
    x = (int)(q - r * (I)W);
    q = r / (I)H;
    y = (int)(r - q * (I)H);
    n = (int)(q / (I)D);
    z = (int)(q - (I)n * (I)D);
}

__device__ __forceinline__ long long at(int n, int z, int y, int x, int D, int H, int W, int ld) {
    return ((((long long)n * D + z) * H + y) * W + x) * ld;
}

template <class I> __device__ __forceinline__ I thread_index() { return (I)blockIdx.x * (I)blockDim.x + threadIdx.x; }

// y (D x H x W) = mean of the 2x2x2 children of x (2D x 2H x 2W)
template <int V, class I>
__global__ void k_pool(const bf16 *__restrict__ x, int ldx, bf16 *__restrict__ y, int ldy, I total, int D, int H,
                       int W, int C) {
    const I i = thread_index<I>();
    if (i >= total) return;
    int c, xo, yo, zo, n;
    decode<V, I>(i, C, W, H, D, c, xo, yo, zo, n);
    Vec<V> v[8], o;
#pragma unroll
    for (int j = 0; j < 8; ++j)
        v[j].load(x + at(n, 2 * zo + (j >> 2), 2 * yo + ((j >> 1) & 1), 2 * xo + (j & 1), 2 * D, 2 * H, 2 * W, ldx) + c);
#pragma unroll
    for (int e = 0; e < V; ++e) {
        float s = 0.f;
#pragma unroll
        for (int j = 0; j < 8; ++j) s += __bfloat162float(v[j].v[e]);
        o.v[e] = __float2bfloat16_rn(s * 0.125f);
    }
    o.store(y + at(n, zo, yo, xo, D, H, W, ldy) + c);
}

// the 8 children in dx (2D x 2H x 2W) (+)= dy(parent) / 8
template <int V, class I>
__global__ void k_pool_bwd(const bf16 *__restrict__ dy, int ldy, bf16 *__restrict__ dx, int ldx, I total, int D, int H,
                           int W, int C, int accumulate) {
    const I i = thread_index<I>();
    if (i >= total) return;
    int c, x, y, z, n;
    decode<V, I>(i, C, W, H, D, c, x, y, z, n);
    Vec<V> g, o;
    g.load(dy + at(n, z, y, x, D, H, W, ldy) + c);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        bf16 *p = dx + at(n, 2 * z + (j >> 2), 2 * y + ((j >> 1) & 1), 2 * x + (j & 1), 2 * D, 2 * H, 2 * W, ldx) + c;
        if (accumulate) o.load(p);
#pragma unroll
        for (int e = 0; e < V; ++e) {
            float s = __bfloat162float(g.v[e]) * 0.125f;
            if (accumulate) s += __bfloat162float(o.v[e]);
            o.v[e] = __float2bfloat16_rn(s);
        }
        o.store(p);
    }
}

// the 8 children in y (2D x 2H x 2W) = x(parent)
template <int V, class I>
__global__ void k_up(const bf16 *__restrict__ x, int ldx, bf16 *__restrict__ y, int ldy, I total, int D, int H, int W,
                     int C) {
    const I i = thread_index<I>();
    if (i >= total) return;
    int c, xi, yi, zi, n;
    decode<V, I>(i, C, W, H, D, c, xi, yi, zi, n);
    Vec<V> v;
    v.load(x + at(n, zi, yi, xi, D, H, W, ldx) + c);
#pragma unroll
    for (int j = 0; j < 8; ++j)
        v.store(y + at(n, 2 * zi + (j >> 2), 2 * yi + ((j >> 1) & 1), 2 * xi + (j & 1), 2 * D, 2 * H, 2 * W, ldy) + c);
}

// dx (D x H x W) (+)= sum of the 8 children of dy (2D x 2H x 2W)
template <int V, class I>
__global__ void k_up_bwd(const bf16 *__restrict__ dy, int ldy, bf16 *__restrict__ dx, int ldx, I total, int D, int H,
                         int W, int C, int accumulate) {
    const I i = thread_index<I>();
    if (i >= total) return;
    int c, x, y, z, n;
    decode<V, I>(i, C, W, H, D, c, x, y, z, n);
    Vec<V> v[8], o;
#pragma unroll
    for (int j = 0; j < 8; ++j)
        v[j].load(dy + at(n, 2 * z + (j >> 2), 2 * y + ((j >> 1) & 1), 2 * x + (j & 1), 2 * D, 2 * H, 2 * W, ldy) + c);
    bf16 *p = dx + at(n, z, y, x, D, H, W, ldx) + c;
    if (accumulate) o.load(p);
#pragma unroll
    for (int e = 0; e < V; ++e) {
        float s = 0.f;
#pragma unroll
        for (int j = 0; j < 8; ++j) s += __bfloat162float(v[j].v[e]);
        if (accumulate) s += __bfloat162float(o.v[e]);
        o.v[e] = __float2bfloat16_rn(s);
    }
    o.store(p);
}

template <int V, class I>
__global__ void k_relu_bwd(const bf16 *__restrict__ y, int ldy, bf16 *__restrict__ dy, int lddy, I total, int C) {
    const I i = thread_index<I>();
    if (i >= total) return;
    const I cv = (I)(C / V), p = i / cv;
    const int c = (int)(i - p * cv) * V;
    bf16 *d = dy + (long long)p * lddy + c;
    Vec<V> a, g;
    a.load(y + (long long)p * ldy + c);
    g.load(d);
#pragma unroll
    for (int e = 0; e < V; ++e)
        if (!(__bfloat162float(a.v[e]) > 0.f)) g.v[e] = __float2bfloat16_rn(0.f);
    g.store(d);
}

__global__ void k_mse(const float *__restrict__ pred, int ldp, const float *__restrict__ target,
                      const uint8_t *__restrict__ mask, const float *__restrict__ wch, bf16 *__restrict__ dpred,
                      int lddp, float *__restrict__ loss, long long P, int C, float inv_count) {
    const long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    float l = 0.f;
    if (p < P) {
        const bool m = mask[p] != 0;
        for (int c = 0; c < lddp; ++c) {
            float g = 0.f;
            if (m && c < C) {
                const float d = pred[p * ldp + c] - target[p * C + c];
                l += wch[c] * d * d * inv_count;
                g = 2.f * wch[c] * d * inv_count;
            }
            dpred[p * lddp + c] = __float2bfloat16_rn(g);
        }
    }
    // block reduction of the loss
    __shared__ float sh[256];
    sh[threadIdx.x] = l;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0) atomicAdd(loss, sh[0]);
}

__global__ void k_adam(float *__restrict__ w, float *__restrict__ m, float *__restrict__ v, float *__restrict__ g,
                       bf16 *__restrict__ wb, long long n, float lr_t, float b1, float b2, float eps, float wd) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i] + wd * w[i];
    g[i] = 0.f;  // the gradient buffer is ready for the next accumulation
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float wi = w[i] - lr_t * mi / (sqrtf(vi) + eps);
    w[i] = wi;
    if (wb) wb[i] = __float2bfloat16_rn(wi);
}

template <int V, class I>
__global__ void k_to_bf16(const float *__restrict__ x, int ldx, bf16 *__restrict__ y, int ldy, I total, int C) {
    const I i = thread_index<I>();
    if (i >= total) return;
    const I cv = (I)(C / V), p = i / cv;
    const int c = (int)(i - p * cv) * V;
    Vec<V, float> f;
    f.load(x + (long long)p * ldx + c);
    Vec<V> o;
#pragma unroll
    for (int e = 0; e < V; ++e) o.v[e] = __float2bfloat16_rn(f.v[e]);
    o.store(y + (long long)p * ldy + c);
}

// whether rows of `ld` elements of `size` bytes from p start on 16-byte boundaries
static bool rows16(const void *p, int ld, int size) {
    return (reinterpret_cast<uintptr_t>(p) & 15) == 0 && ((long long)ld * size) % 16 == 0;
}
// f(vector width, total) with the width as a std::integral_constant and the
// vector count as the index type: 8 channels per thread where `vec` holds and C
// is a multiple of 8, 32-bit indices where the threads of the launch fit
template <class F> static void with_width(bool vec, long long positions, int C, F &&f) {
    const bool v8 = vec && C % 8 == 0;
    const long long total = positions * (v8 ? C / 8 : C);
    const bool small = total <= 0x7FFFFFFFLL - 256;
    if (v8 && small) f(std::integral_constant<int, 8>{}, (uint32_t)total);
    else if (v8) f(std::integral_constant<int, 8>{}, total);
    else if (small) f(std::integral_constant<int, 1>{}, (uint32_t)total);
    else f(std::integral_constant<int, 1>{}, total);
}

static unsigned blocks_for(long long total) { return (unsigned)((total + 255) / 256); }
static bool dims_ok(int N, int D, int H, int W, int C) { return N > 0 && D > 0 && H > 0 && W > 0 && C > 0; }

}  // namespace ws

using namespace ws;

extern "C" {

int ws_avgpool2(const void *x, int ldx, void *y, int ldy, int N, int D, int H, int W, int C, void *stream) {
    if (!x || !y || !dims_ok(N, D, H, W, C) || (D | H | W) & 1 || ldx < C || ldy < C) return 1;
    const long long positions = (long long)N * (D / 2) * (H / 2) * (W / 2);
    with_width(rows16(x, ldx, 2) && rows16(y, ldy, 2), positions, C, [&](auto v, auto total) {
        k_pool<decltype(v)::value><<<blocks_for(total), 256, 0, (cudaStream_t)stream>>>(
            (const bf16 *)x, ldx, (bf16 *)y, ldy, total, D / 2, H / 2, W / 2, C);
    });
    return cudaGetLastError() == cudaSuccess ? 0 : 2;
}

int ws_avgpool2_bwd(const void *dy, int ldy, void *dx, int ldx, int N, int D, int H, int W, int C, int accumulate,
                    void *stream) {
    if (!dy || !dx || !dims_ok(N, D, H, W, C) || (D | H | W) & 1 || ldx < C || ldy < C) return 1;
    const long long positions = (long long)N * (D / 2) * (H / 2) * (W / 2);
    with_width(rows16(dy, ldy, 2) && rows16(dx, ldx, 2), positions, C, [&](auto v, auto total) {
        k_pool_bwd<decltype(v)::value><<<blocks_for(total), 256, 0, (cudaStream_t)stream>>>(
            (const bf16 *)dy, ldy, (bf16 *)dx, ldx, total, D / 2, H / 2, W / 2, C, accumulate);
    });
    return cudaGetLastError() == cudaSuccess ? 0 : 2;
}

int ws_upsample2(const void *x, int ldx, void *y, int ldy, int N, int D, int H, int W, int C, void *stream) {
    if (!x || !y || !dims_ok(N, D, H, W, C) || ldx < C || ldy < C) return 1;
    with_width(rows16(x, ldx, 2) && rows16(y, ldy, 2), (long long)N * D * H * W, C, [&](auto v, auto total) {
        k_up<decltype(v)::value><<<blocks_for(total), 256, 0, (cudaStream_t)stream>>>(
            (const bf16 *)x, ldx, (bf16 *)y, ldy, total, D, H, W, C);
    });
    return cudaGetLastError() == cudaSuccess ? 0 : 2;
}

int ws_upsample2_bwd(const void *dy, int ldy, void *dx, int ldx, int N, int D, int H, int W, int C, int accumulate,
                     void *stream) {
    if (!dy || !dx || !dims_ok(N, D, H, W, C) || ldx < C || ldy < C) return 1;
    with_width(rows16(dy, ldy, 2) && rows16(dx, ldx, 2), (long long)N * D * H * W, C, [&](auto v, auto total) {
        k_up_bwd<decltype(v)::value><<<blocks_for(total), 256, 0, (cudaStream_t)stream>>>(
            (const bf16 *)dy, ldy, (bf16 *)dx, ldx, total, D, H, W, C, accumulate);
    });
    return cudaGetLastError() == cudaSuccess ? 0 : 2;
}

int ws_relu_bwd(const void *y, int ldy, void *dy, int lddy, long long P, int C, void *stream) {
    if (!y || !dy || P < 1 || C < 1 || ldy < C || lddy < C) return 1;
    with_width(rows16(y, ldy, 2) && rows16(dy, lddy, 2), P, C, [&](auto v, auto total) {
        k_relu_bwd<decltype(v)::value><<<blocks_for(total), 256, 0, (cudaStream_t)stream>>>(
            (const bf16 *)y, ldy, (bf16 *)dy, lddy, total, C);
    });
    return cudaGetLastError() == cudaSuccess ? 0 : 2;
}

int ws_mse_loss(const float *pred, int ldp, const float *target, const uint8_t *mask, const float *wch, void *dpred,
                int lddp, float *loss, long long P, int C, void *stream) {
    if (!pred || !target || !mask || !wch || !dpred || !loss || P < 1 || C < 1 || ldp < C || lddp < C) return 1;
    k_mse<<<blocks_for(P), 256, 0, (cudaStream_t)stream>>>(pred, ldp, target, mask, wch, (bf16 *)dpred, lddp, loss,
                                                           P, C, 1.0f / (float)(P * C));
    return cudaGetLastError() == cudaSuccess ? 0 : 2;
}

int ws_adam(float *w, float *m, float *v, float *g, void *wb, long long n, float lr_t, float beta1, float beta2,
            float eps, float weight_decay, void *stream) {
    if (!w || !m || !v || !g || n < 1) return 1;
    k_adam<<<blocks_for(n), 256, 0, (cudaStream_t)stream>>>(w, m, v, g, (bf16 *)wb, n, lr_t, beta1, beta2, eps,
                                                            weight_decay);
    return cudaGetLastError() == cudaSuccess ? 0 : 2;
}

int ws_to_bf16(const float *x, int ldx, void *y, int ldy, long long P, int C, void *stream) {
    if (!x || !y || P < 1 || C < 1 || ldx < C || ldy < C) return 1;
    with_width(rows16(x, ldx, 4) && rows16(y, ldy, 2), P, C, [&](auto v, auto total) {
        k_to_bf16<decltype(v)::value><<<blocks_for(total), 256, 0, (cudaStream_t)stream>>>(x, ldx, (bf16 *)y, ldy,
                                                                                           total, C);
    });
    return cudaGetLastError() == cudaSuccess ? 0 : 2;
}

}  // extern "C"
