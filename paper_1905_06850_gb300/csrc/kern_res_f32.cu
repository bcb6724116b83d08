// kern_res_f32.cu -- instantiations of the register-resident solver of small
// stencil systems for T = float.
#include "resident.cuh"
#include "plcg_kernels.h"

namespace plcg {

template <int L>
static const void *res_rows(int rows)
{
    switch (rows) {
    case 1: return reinterpret_cast<const void *>(&resident_kernel<float, L, 1>);
    case 2: return reinterpret_cast<const void *>(&resident_kernel<float, L, 2>);
    case 4: return reinterpret_cast<const void *>(&resident_kernel<float, L, 4>);
    default: return nullptr;
    }
}

const void *kptr_resident_f32(int l, int rows)
{
    return l == 1 ? res_rows<1>(rows) : l == 2 ? res_rows<2>(rows) : l == 3 ? res_rows<3>(rows) : nullptr;
}

}  // namespace plcg
