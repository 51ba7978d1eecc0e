// cwo_holo.cu -- the steps of phase-only hologram optimisation around a propagation and its adjoint:
// phase -> field on the canvas, |u|^2 on the window, the mean squared residual against a target,
// the seed of the adjoint, and the gradient of the phase.
//
// All five are elementwise over the canvas or the window and bound by memory: each reads what it needs
// once and writes its result once, two complex values a thread.  As separate tensor operators a
// loss and its gradient at 1080 x 1920 in a 2048^2 canvas were about 60 launches and 960 us of host
// time around 250 us of propagation.  The window may start at any column and have any width: the
// canvas is walked in 16-byte pairs and each of the pair's pixels is tested.
#include <cuda_runtime.h>

#include <algorithm>

#include "cwo.h"
#include "cwo_fft.cuh"
#include "cwo_internal.h"

namespace cwo {
namespace {

struct Window { int h, w, nx, ny, ox, oy; };

// canvas value of pixel (x, y): f(index into the window) inside it, zero outside
template <class F>
__device__ __forceinline__ void canvas_pairs(const Window& W, float4* __restrict__ out, F&& f) {
    const int half = W.nx / 2;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < (long long)half * W.ny;
         i += (long long)gridDim.x * blockDim.x) {
        const int wy = (int)(i / half) - W.oy, wx = 2 * (int)(i % half) - W.ox;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (wy >= 0 && wy < W.h) {
            const long long k = (long long)wy * W.w + wx;
            if (wx >= 0 && wx < W.w) { const float2 a = f(k, 2 * i); v.x = a.x; v.y = a.y; }
            if (wx + 1 >= 0 && wx + 1 < W.w) { const float2 b = f(k + 1, 2 * i + 1); v.z = b.x; v.w = b.y; }
        }
        out[i] = v;
    }
}

__global__ void __launch_bounds__(256) k_field(const Window W, const float* __restrict__ phase, float4* __restrict__ out) {
    canvas_pairs(W, out, [&](long long k, long long) {
        float s, c;
        sincosf(__ldg(phase + k), &s, &c);
        return make_float2(c, s);
    });
}

// 2 u g s on the window, s = 1, or 2 gloss / (h w): the derivative of the mean of g^2 times the
// incoming gradient
__global__ void __launch_bounds__(256)
k_seed(const Window W, const float2* __restrict__ u, const float* __restrict__ gw, const float* __restrict__ gloss,
       float4* __restrict__ out) {
    const float s = gloss ? 2.0f * __ldg(gloss) / ((float)W.h * (float)W.w) : 1.0f;
    canvas_pairs(W, out, [&](long long k, long long c) {
        const float2 v = __ldg(u + c);
        const float g = 2.0f * (s * __ldg(gw + k));
        return make_float2(v.x * g, v.y * g);
    });
}

// pixel k of the window -> canvas index
__device__ __forceinline__ long long canvas_index(const Window& W, long long k) {
    const int y = (int)(k / W.w), x = (int)(k - (long long)y * W.w);
    return (long long)(W.oy + y) * W.nx + W.ox + x;
}

__global__ void __launch_bounds__(256) k_intensity(const Window W, const float2* __restrict__ u, float* __restrict__ out) {
    const long long n = (long long)W.h * W.w;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x) {
        const float2 v = __ldg(u + canvas_index(W, k));
        out[k] = fmaf(v.x, v.x, v.y * v.y);
    }
}

// d/dphi of a real loss through x = exp(i phi): Re(conj(g) i x)
__global__ void __launch_bounds__(256)
k_phase_grad(const Window W, const float2* __restrict__ g, const float* __restrict__ phase, float* __restrict__ out) {
    const long long n = (long long)W.h * W.w;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x) {
        const float2 v = __ldg(g + canvas_index(W, k));
        float s, c;
        sincosf(__ldg(phase + k), &s, &c);
        out[k] = fmaf(v.y, c, -v.x * s);
    }
}

// sums over a block in FP64, in a fixed order
__device__ __forceinline__ double block_sum(double v) {
    __shared__ double part[8];
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) v += __shfl_down_sync(0xffffffffu, v, d);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x == 0)
        for (int i = 0; i < 8; ++i) s += part[i];
    return s;
}

__global__ void __launch_bounds__(256)
k_residual(const Window W, const float2* __restrict__ u, const float* __restrict__ target, float* __restrict__ residual,
           double* __restrict__ partial) {
    const long long n = (long long)W.h * W.w;
    double s = 0.0;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x) {
        const float2 v = __ldg(u + canvas_index(W, k));
        const float d = fmaf(v.x, v.x, v.y * v.y) - __ldg(target + k);
        residual[k] = d;
        s += (double)d * (double)d;
    }
    s = block_sum(s);
    if (threadIdx.x == 0) partial[blockIdx.x] = s;
}
__global__ void __launch_bounds__(256) k_residual_mean(const double* __restrict__ partial, int n, double count, float* __restrict__ loss) {
    double s = 0.0;
    for (int i = threadIdx.x; i < n; i += 256) s += partial[i];
    s = block_sum(s);
    if (threadIdx.x == 0) *loss = (float)(s / count);
}

cwo_status fail(const char* msg) {
    set_last_error(msg);
    return CWO_ERR_INVALID_ARG;
}

cwo_status check_window(const Window& W, int* dev) {
    if (W.nx < 2 || W.ny < 1 || W.nx > CWO_MAX_SIDE || W.ny > CWO_MAX_SIDE || W.nx % 2) return fail("bad canvas size");
    if (W.h < 1 || W.w < 1 || W.ox < 0 || W.oy < 0 || W.h > W.ny - W.oy || W.w > W.nx - W.ox)
        return fail("the window does not lie inside the canvas");
    if (cudaGetDevice(dev) != cudaSuccess) {
        set_last_error("cudaGetDevice failed");
        return CWO_ERR_CUDA;
    }
    return CWO_OK;
}

cwo_status launched(cudaError_t e) {
    if (e == cudaSuccess) return CWO_OK;
    set_last_error(cudaGetErrorString(e));
    return CWO_ERR_CUDA;
}

unsigned blocks_for(long long n) { return (unsigned)std::min<long long>((n + 255) / 256, 152 * 8); }

}  // namespace
}  // namespace cwo

using namespace cwo;

extern "C" {

cwo_status cwo_hologram_field(const float* phase, int h, int w, int nx, int ny, int ox, int oy, void* field_c64, void* stream) {
    const Window W{h, w, nx, ny, ox, oy};
    int dev = 0;
    cwo_status st = check_window(W, &dev);
    const size_t nw = (size_t)h * w, nc = (size_t)nx * ny;
    if (st || (st = (cwo_status)check_device_buffer(phase, nw * 4, dev, "phase", 4)) ||
        (st = (cwo_status)check_device_buffer(field_c64, nc * 8, dev, "field", 16)))
        return st;
    k_field<<<blocks_for(nc / 2), 256, 0, (cudaStream_t)stream>>>(W, phase, (float4*)field_c64);
    return launched(cudaGetLastError());
}

cwo_status cwo_hologram_intensity(const void* u_c64, int h, int w, int nx, int ny, int ox, int oy, float* intensity, void* stream) {
    const Window W{h, w, nx, ny, ox, oy};
    int dev = 0;
    cwo_status st = check_window(W, &dev);
    const size_t nw = (size_t)h * w, nc = (size_t)nx * ny;
    if (st || (st = (cwo_status)check_device_buffer(u_c64, nc * 8, dev, "u", 8)) ||
        (st = (cwo_status)check_device_buffer(intensity, nw * 4, dev, "intensity", 4)))
        return st;
    k_intensity<<<blocks_for(nw), 256, 0, (cudaStream_t)stream>>>(W, (const float2*)u_c64, intensity);
    return launched(cudaGetLastError());
}

cwo_status cwo_hologram_loss(const void* u_c64, const float* target, int h, int w, int nx, int ny, int ox, int oy,
                             float* residual, float* loss, double* partial, void* stream) {
    const Window W{h, w, nx, ny, ox, oy};
    int dev = 0;
    cwo_status st = check_window(W, &dev);
    const size_t nw = (size_t)h * w, nc = (size_t)nx * ny;
    if (st || (st = (cwo_status)check_device_buffer(u_c64, nc * 8, dev, "u", 8)) ||
        (st = (cwo_status)check_device_buffer(target, nw * 4, dev, "target", 4)) ||
        (st = (cwo_status)check_device_buffer(residual, nw * 4, dev, "residual", 4)) ||
        (st = (cwo_status)check_device_buffer(loss, 4, dev, "loss", 4)) ||
        (st = (cwo_status)check_device_buffer(partial, CWO_HOLOGRAM_PARTIALS * 8, dev, "partial", 8)))
        return st;
    const unsigned nb = std::min<unsigned>(blocks_for(nw), CWO_HOLOGRAM_PARTIALS);
    k_residual<<<nb, 256, 0, (cudaStream_t)stream>>>(W, (const float2*)u_c64, target, residual, partial);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) {
        k_residual_mean<<<1, 256, 0, (cudaStream_t)stream>>>(partial, (int)nb, (double)nw, loss);
        e = cudaGetLastError();
    }
    return launched(e);
}

cwo_status cwo_hologram_seed(const void* u_c64, const float* g, const float* gloss, int h, int w, int nx, int ny, int ox,
                             int oy, void* out_c64, void* stream) {
    const Window W{h, w, nx, ny, ox, oy};
    int dev = 0;
    cwo_status st = check_window(W, &dev);
    const size_t nw = (size_t)h * w, nc = (size_t)nx * ny;
    if (st || (st = (cwo_status)check_device_buffer(u_c64, nc * 8, dev, "u", 8)) ||
        (st = (cwo_status)check_device_buffer(g, nw * 4, dev, "g", 4)) ||
        (gloss && (st = (cwo_status)check_device_buffer(gloss, 4, dev, "gloss", 4))) ||
        (st = (cwo_status)check_device_buffer(out_c64, nc * 8, dev, "out", 16)))
        return st;
    k_seed<<<blocks_for(nc / 2), 256, 0, (cudaStream_t)stream>>>(W, (const float2*)u_c64, g, gloss, (float4*)out_c64);
    return launched(cudaGetLastError());
}

cwo_status cwo_hologram_phase_grad(const void* g_c64, const float* phase, int h, int w, int nx, int ny, int ox, int oy,
                                   float* gphase, void* stream) {
    const Window W{h, w, nx, ny, ox, oy};
    int dev = 0;
    cwo_status st = check_window(W, &dev);
    const size_t nw = (size_t)h * w, nc = (size_t)nx * ny;
    if (st || (st = (cwo_status)check_device_buffer(g_c64, nc * 8, dev, "g", 8)) ||
        (st = (cwo_status)check_device_buffer(phase, nw * 4, dev, "phase", 4)) ||
        (st = (cwo_status)check_device_buffer(gphase, nw * 4, dev, "gphase", 4)))
        return st;
    k_phase_grad<<<blocks_for(nw), 256, 0, (cudaStream_t)stream>>>(W, (const float2*)g_c64, phase, gphase);
    return launched(cudaGetLastError());
}

}  // extern "C"
