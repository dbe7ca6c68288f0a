// Instantiations of the slab-streaming stencil kernel, bf16 storage.
#include "stencil_registry.h"
#include "stencil_slab.cuh"

namespace perks {

void register_slab_bf16(std::vector<SlabEntry> &out) { slab_entries<__nv_bfloat16>(out, PERKS_BF16); }

}  // namespace perks
