// kern_res_f64.cu -- instantiations of the register-resident solver of small
// stencil systems for T = double.
#include "resident.cuh"
#include "plcg_kernels.h"

namespace plcg {

template <int L>
static const void *res_rows(int rows)
{
    switch (rows) {
    case 1: return reinterpret_cast<const void *>(&resident_kernel<double, L, 1>);
    case 2: return reinterpret_cast<const void *>(&resident_kernel<double, L, 2>);
    case 4: return reinterpret_cast<const void *>(&resident_kernel<double, L, 4>);
    default: return nullptr;
    }
}

const void *kptr_resident_f64(int l, int rows)
{
    return l == 1 ? res_rows<1>(rows) : l == 2 ? res_rows<2>(rows) : l == 3 ? res_rows<3>(rows) : nullptr;
}

}  // namespace plcg
