// cwo_holo.cu -- the steps of phase-only hologram optimisation around a propagation and its adjoint:
// phase -> field on the canvas, |u|^2 on the window, the mean squared residual against a target,
// the seed of the adjoint, and the gradient of the phase.
//
// All five are elementwise over the canvas or the window and bound by memory: each reads what it needs
// once and writes its result once, two complex values a thread.  As separate tensor operators a
// loss and its gradient at 1080 x 1920 in a 2048^2 canvas were about 60 launches and 960 us of host
// time around 250 us of propagation; now 11 launches from two calls, and the propagations leave out the
// canvas rows outside the window (125 -> 99 us each): 260 us in all.  The window may start at any column and have any width: the
// canvas is walked in 16-byte pairs and each of the pair's pixels is tested.
#include <cuda_runtime.h>

#include <algorithm>

#include "cwo.h"
#include "cwo_fft.cuh"
#include "cwo_internal.h"

namespace cwo {
namespace {

struct Window { int h, w, nx, ny, ox, oy; };

// canvas rows [y0, y1) that k_field and k_seed write: whole groups of the rows that the plan propagates
struct Rows { int y0, y1; };
Rows rows_of(const Window& W, int group) {
    if (group <= 0) return {0, W.ny};
    return {W.oy / group * group, std::min(W.ny, (W.oy + W.h + group - 1) / group * group)};
}

// Rows are walked by the grid's second dimension, so that no thread divides (1080 x 1920: the forward half
// of a step 136 -> 132 us against rows and columns from 64-bit divisions of a flat index).
// canvas value of pixel (x, y): f(index into the window) inside it, zero outside
template <class F>
__device__ __forceinline__ void canvas_pairs(const Window& W, const Rows& rows, float4* __restrict__ out, F&& f) {
    const int half = W.nx / 2, i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= half) return;
    for (int y = rows.y0 + (int)blockIdx.y; y < rows.y1; y += gridDim.y) {
        const int wy = y - W.oy, wx = 2 * i - W.ox;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (wy >= 0 && wy < W.h) {
            const int k = wy * W.w + wx, c = y * W.nx + 2 * i;
            if (wx >= 0 && wx < W.w) { const float2 a = f(k, c); v.x = a.x; v.y = a.y; }
            if (wx + 1 >= 0 && wx + 1 < W.w) { const float2 b = f(k + 1, c + 1); v.z = b.x; v.w = b.y; }
        }
        out[(size_t)y * half + i] = v;
    }
}
// f(window index, canvas index) of the thread's pixels
template <class F>
__device__ __forceinline__ void window_pixels(const Window& W, F&& f) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= W.w) return;
    for (int y = blockIdx.y; y < W.h; y += gridDim.y) f(y * W.w + x, (W.oy + y) * W.nx + W.ox + x);
}

__global__ void __launch_bounds__(256) k_field(const Window W, const Rows rows, const float* __restrict__ phase, float4* __restrict__ out) {
    canvas_pairs(W, rows, out, [&](int k, int) {
        float s, c;
        sincosf(__ldg(phase + k), &s, &c);
        return make_float2(c, s);
    });
}

// 2 u g s on the window, s = 1, or 2 gloss / (h w): the derivative of the mean of g^2 times the
// incoming gradient
__global__ void __launch_bounds__(256)
k_seed(const Window W, const Rows rows, const float2* __restrict__ u, const float* __restrict__ gw, const float* __restrict__ gloss,
       float4* __restrict__ out) {
    const float s = gloss ? 2.0f * __ldg(gloss) / ((float)W.h * (float)W.w) : 1.0f;
    canvas_pairs(W, rows, out, [&](int k, int c) {
        const float2 v = __ldg(u + c);
        const float g = 2.0f * (s * __ldg(gw + k));
        return make_float2(v.x * g, v.y * g);
    });
}

__global__ void __launch_bounds__(256) k_intensity(const Window W, const float2* __restrict__ u, float* __restrict__ out) {
    window_pixels(W, [&](int k, int c) {
        const float2 v = __ldg(u + c);
        out[k] = fmaf(v.x, v.x, v.y * v.y);
    });
}

// d/dphi of a real loss through x = exp(i phi): Re(conj(g) i x)
__global__ void __launch_bounds__(256)
k_phase_grad(const Window W, const float2* __restrict__ g, const float* __restrict__ phase, float* __restrict__ out) {
    window_pixels(W, [&](int k, int c) {
        const float2 v = __ldg(g + c);
        float sn, cs;
        sincosf(__ldg(phase + k), &sn, &cs);
        out[k] = fmaf(v.y, cs, -v.x * sn);
    });
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
    float s = 0.f;   // of the few pixels of a thread; the sums over threads are in FP64
    window_pixels(W, [&](int k, int c) {
        const float2 v = __ldg(u + c);
        const float d = fmaf(v.x, v.x, v.y * v.y) - __ldg(target + k);
        residual[k] = d;
        s = fmaf(d, d, s);
    });
    const double sum = block_sum((double)s);
    if (threadIdx.x == 0) partial[blockIdx.y * gridDim.x + blockIdx.x] = sum;
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

// 256 threads across, about 8 blocks per SM in all (never more than CWO_HOLOGRAM_PARTIALS)
dim3 grid_for(int across, int rows) {
    const unsigned gx = (unsigned)(across + 255) / 256;
    return dim3(gx, std::max(1u, std::min((unsigned)rows, (unsigned)CWO_HOLOGRAM_PARTIALS / gx)));
}

}  // namespace
}  // namespace cwo

using namespace cwo;

namespace {

// u <- A u (or A^H u) in place; where the plan can, only the canvas rows of the window
cwo_status propagate(cwo_plan* plan, const Window& W, void* u, int adjoint, void* stream) {
    if (cwo_propagate_rows_group(plan) > 0)
        return cwo_propagate_rows(plan, u, u, W.oy, W.oy + W.h, W.oy, W.oy + W.h, adjoint, stream);
    return adjoint ? cwo_propagate_adjoint(plan, u, u, stream) : cwo_propagate(plan, u, u, stream);
}

}  // namespace

extern "C" {

cwo_status cwo_hologram_forward(cwo_plan* plan, const float* phase, const float* target, int h, int w, int ox, int oy,
                                void* u_c64, float* image, float* loss, double* partial, void* stream) {
    Window W{h, w, 0, 0, ox, oy};
    if (!plan_size(plan, &W.nx, &W.ny)) return fail("plan is NULL");
    int dev = 0;
    cwo_status st = check_window(W, &dev);
    const size_t nw = (size_t)h * w, nc = (size_t)W.nx * W.ny;
    if (st || (st = (cwo_status)check_device_buffer(phase, nw * 4, dev, "phase", 4)) ||
        (st = (cwo_status)check_device_buffer(u_c64, nc * 8, dev, "u", 16)) ||
        (st = (cwo_status)check_device_buffer(image, nw * 4, dev, "image", 4)))
        return st;
    if (target && ((st = (cwo_status)check_device_buffer(target, nw * 4, dev, "target", 4)) ||
                   (st = (cwo_status)check_device_buffer(loss, 4, dev, "loss", 4)) ||
                   (st = (cwo_status)check_device_buffer(partial, CWO_HOLOGRAM_PARTIALS * 8, dev, "partial", 8))))
        return st;
    const cudaStream_t s = (cudaStream_t)stream;
    const Rows rows = rows_of(W, cwo_propagate_rows_group(plan));
    k_field<<<grid_for(W.nx / 2, rows.y1 - rows.y0), 256, 0, s>>>(W, rows, phase, (float4*)u_c64);
    if ((st = launched(cudaGetLastError())) || (st = propagate(plan, W, u_c64, 0, stream))) return st;
    if (!target) {
        k_intensity<<<grid_for(W.w, W.h), 256, 0, s>>>(W, (const float2*)u_c64, image);
        return launched(cudaGetLastError());
    }
    const dim3 nb = grid_for(W.w, W.h);
    k_residual<<<nb, 256, 0, s>>>(W, (const float2*)u_c64, target, image, partial);
    if ((st = launched(cudaGetLastError()))) return st;
    k_residual_mean<<<1, 256, 0, s>>>(partial, (int)(nb.x * nb.y), (double)nw, loss);
    return launched(cudaGetLastError());
}

cwo_status cwo_hologram_backward(cwo_plan* plan, const float* phase, const void* u_c64, const float* g, const float* gloss, int h,
                                 int w, int ox, int oy, void* work_c64, float* gphase, void* stream) {
    Window W{h, w, 0, 0, ox, oy};
    if (!plan_size(plan, &W.nx, &W.ny)) return fail("plan is NULL");
    int dev = 0;
    cwo_status st = check_window(W, &dev);
    const size_t nw = (size_t)h * w, nc = (size_t)W.nx * W.ny;
    if (st || (st = (cwo_status)check_device_buffer(phase, nw * 4, dev, "phase", 4)) ||
        (st = (cwo_status)check_device_buffer(u_c64, nc * 8, dev, "u", 8)) ||
        (st = (cwo_status)check_device_buffer(g, nw * 4, dev, "g", 4)) ||
        (gloss && (st = (cwo_status)check_device_buffer(gloss, 4, dev, "gloss", 4))) ||
        (st = (cwo_status)check_device_buffer(work_c64, nc * 8, dev, "work", 16)) ||
        (st = (cwo_status)check_device_buffer(gphase, nw * 4, dev, "gphase", 4)))
        return st;
    const cudaStream_t s = (cudaStream_t)stream;
    const Rows rows = rows_of(W, cwo_propagate_rows_group(plan));
    k_seed<<<grid_for(W.nx / 2, rows.y1 - rows.y0), 256, 0, s>>>(W, rows, (const float2*)u_c64, g, gloss,
                                                                               (float4*)work_c64);
    if ((st = launched(cudaGetLastError())) || (st = propagate(plan, W, work_c64, 1, stream))) return st;
    k_phase_grad<<<grid_for(W.w, W.h), 256, 0, s>>>(W, (const float2*)work_c64, phase, gphase);
    return launched(cudaGetLastError());
}

}  // extern "C"
