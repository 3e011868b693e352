// Instantiations of the persistent multi-step kernel (FP32C): the compiled
// observable layouts with the potential signatures of the workloads.
#include "m2m_steps.cuh"

namespace m2m {

template <int L, int PK>
static void *either(bool solo) { return solo ? (void *)k_steps<L, PK, true> : (void *)k_steps<L, PK, false>; }

void *steps_kernel_f32(int layout, int pk, bool solo) {
    // the solo residual: the layouts with few observables
    if (layout == 2 && pk == PK_HERNQUIST) return either<2, PK_HERNQUIST>(solo);
    if (layout == 2 && pk == PK_HERNQUIST_NFW) return either<2, PK_HERNQUIST_NFW>(solo);
    if (layout == 3 && pk == PK_HERNQUIST) return either<3, PK_HERNQUIST>(solo);
    if (solo) return nullptr;
    if (layout == 1 && pk == PK_LOG) return (void *)k_steps<1, PK_LOG, false>;
    if (layout == 4 && pk == PK_LOG) return (void *)k_steps<4, PK_LOG, false>;
    return nullptr;
}

}  // namespace m2m
