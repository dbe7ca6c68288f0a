// Instantiations of the slab-streaming stencil kernel, f64 storage.
#include "stencil_registry.h"
#include "stencil_slab.cuh"

namespace perks {

void register_slab_f64(std::vector<SlabEntry> &out) { slab_entries<double>(out, PERKS_F64); }

}  // namespace perks
