// cwo_asm_tables.cpp -- host tables of the angular-spectrum phase.
//
// A unit of its own because it is compiled without contraction of multiplies and adds, as is the device's
// k_asm_tables (cwo_itables.cu), so that a plan's own tables and the tables of a mixed batch are the same bit for
// bit.  The FP64 transforms of cwo_tables.cpp keep the compiler's contraction: without it the transform of a
// Fresnel axis takes 7.6 instead of 7.3 us at 1024 points and 34.9 instead of 32.7 at 4096 (Grace cores).
#include "cwo_tables.h"

namespace cwo {
namespace host {

void asm_axis_table(const AxisGeo& g, double pitch, double lambda, double z, bool is_x, float4* out) {
    const AsmAxis A = asm_axis(g.P, pitch, lambda, z, is_x);
    // every entry depends on kt^2 only: evaluate |kt| = 0 .. P/2 once, store at both indices
    const MirrorIndices m = mirror_indices(g);
    for (int k = 0; k <= g.P / 2; ++k) {
        const float4 v = asm_axis_entry(A, (double)k * (double)k);
        out[m.first[k]] = v;
        if (m.second[k] >= 0) out[m.second[k]] = v;
    }
}

}  // namespace host
}  // namespace cwo
