// kern_st_ahead.cu -- instantiations of the persistent solvers for large
// stencil systems: sweeps whose operands are copied a unit ahead, and systems
// whose lines are not whole 16-byte vectors, held at a padded pitch (FP64 with
// scaled bases).
#include "solver.cuh"
#include "plcg_kernels.h"

namespace plcg {

const void *kptr_st_ahead(bool f32, int l)
{
    if (f32) {
        switch (l) {
        case 1: return reinterpret_cast<const void *>(&plcg_kernel<float, 1, 4, kOpStencil, false, float, true>);
        case 2: return reinterpret_cast<const void *>(&plcg_kernel<float, 2, 4, kOpStencil, false, float, true>);
        default: return nullptr;
        }
    }
    switch (l) {
    case 1: return reinterpret_cast<const void *>(&plcg_kernel<double, 1, 2, kOpStencil, true, double, true>);
    case 2: return reinterpret_cast<const void *>(&plcg_kernel<double, 2, 2, kOpStencil, true, double, true>);
    default: return nullptr;
    }
}

const void *kptr_st_pad(bool f32, int l)   // l = 0: classic CG
{
    if (f32) {
        switch (l) {
        case 0: return reinterpret_cast<const void *>(&cg_kernel<float, 4, kOpStencil, float, true>);
        case 1: return reinterpret_cast<const void *>(&plcg_kernel<float, 1, 4, kOpStencil, false, float, true, true>);
        case 2: return reinterpret_cast<const void *>(&plcg_kernel<float, 2, 4, kOpStencil, false, float, true, true>);
        case 3: return reinterpret_cast<const void *>(&plcg_kernel<float, 3, 4, kOpStencil, false, float, false, true>);
        default: return nullptr;
        }
    }
    switch (l) {
    case 0: return reinterpret_cast<const void *>(&cg_kernel<double, 2, kOpStencil, double, true>);
    case 1: return reinterpret_cast<const void *>(&plcg_kernel<double, 1, 2, kOpStencil, true, double, true, true>);
    case 2: return reinterpret_cast<const void *>(&plcg_kernel<double, 2, 2, kOpStencil, true, double, true, true>);
    case 3: return reinterpret_cast<const void *>(&plcg_kernel<double, 3, 2, kOpStencil, true, double, false, true>);
    default: return nullptr;
    }
}

}  // namespace plcg
