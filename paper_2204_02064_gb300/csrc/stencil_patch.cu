// Instantiations of the patch kernel (small 2-D domains, K steps per exchange).
#include "stencil_registry.h"
#include "stencil_patch.cuh"

namespace perks {

void register_patch_kernels(std::vector<PatchEntry> &out) {
    patch_entries<double>(out, PERKS_F64);
    patch_entries<float>(out, PERKS_F32);
    patch_entries<__nv_bfloat16>(out, PERKS_BF16);
}

}  // namespace perks
