// Instantiations of the slab-streaming stencil kernel, f32 storage.
#include "stencil_registry.h"
#include "stencil_slab.cuh"

namespace perks {

void register_slab_f32(std::vector<SlabEntry> &out) { slab_entries<float>(out, PERKS_F32); }

}  // namespace perks
