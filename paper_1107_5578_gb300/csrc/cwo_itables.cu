// cwo_itables.cu -- per-item angular-spectrum axis tables (mixed batches, per-item distances) on the
// device.
//
// Every entry is the closed form of cwo_tables.h (asm_axis_entry), about twenty FP64 operations.  On
// the host they cost 20 to 60 us an item (256^2 to 4096^2) on threads spawned for the call, and an
// upload of 16 bytes an entry; here each entry is one thread, and the parameters of up to
// kAsmItems items travel in the launch: a batch of 12 512^2 items (4 of them Fresnel) took 132 us of
// host time before.  The unit is compiled without contraction of multiplies and adds (as is
// cwo_asm_tables.cpp), so that the entries are the host's bit for bit.
#include "cwo_internal.h"
#include "cwo_launch.cuh"
#include "cwo_tables.h"

namespace cwo {

__global__ void __launch_bounds__(256)
k_asm_tables(const __grid_constant__ AsmItemList d, const int* __restrict__ kbx, const int* __restrict__ kby, int px, int py,
             float4* __restrict__ tx, float4* __restrict__ ty, ItemParams* __restrict__ prm, float* __restrict__ kf) {
    pdl_wait();   // the tables may still be read by the previous call's passes
    const int i = blockIdx.x * blockDim.x + threadIdx.x, item = blockIdx.y;
    const AsmItem& a = d.item[item];
    if (i == 0) {
        if (prm) prm[item] = a.prm;
        if (kf) kf[item] = a.prm.kf;
    }
    if (!a.tables || i >= px + py) return;
    const bool x = i < px;
    const host::AsmAxis& ax = x ? a.x : a.y;
    const double kt = (double)(x ? __ldg(kbx + i) : __ldg(kby + (i - px)));
    const float4 v = host::asm_axis_entry(ax, kt * kt);
    if (x) tx[(size_t)item * px + i] = v;
    else ty[(size_t)item * py + (i - px)] = v;
}

cudaError_t launch_asm_tables(const AsmItemList& list, int items, const int* kbx, const int* kby, int px, int py, float4* tx,
                              float4* ty, ItemParams* prm, float* kf, cudaStream_t st) {
    if (items < 1 || items > kAsmItems) return cudaErrorInvalidValue;
    return pdl_launch(k_asm_tables, dim3((unsigned)((px + py + 255) / 256), (unsigned)items), dim3(256), 0, st, list, kbx,
                      kby, px, py, tx, ty, prm, kf);
}

}  // namespace cwo
