// Instantiations of the column-strip stencil kernel, f64 storage.
#include "stencil_registry.h"
#include "stencil_strip.cuh"

namespace perks {

void register_strip_f64(std::vector<StripKEntry> &out) {
    strip_entries<double, S2d5, 1>(out, PERKS_F64, SH_2D5);
    strip_entries<double, S2d5, 2>(out, PERKS_F64, SH_2D5);
    strip_entries<double, S2d9, 1>(out, PERKS_F64, SH_2D9);
    strip_entries<double, S2d9, 2>(out, PERKS_F64, SH_2D9);
    strip_entries<double, S2ds9, 1>(out, PERKS_F64, SH_2DS9);
    strip_entries<double, S2ds9, 2, 192>(out, PERKS_F64, SH_2DS9);
    strip_entries<double, S2d25, 1>(out, PERKS_F64, SH_2D25);
}

}  // namespace perks
