// Instantiations of the column-strip stencil kernel, bf16 storage.
#include "stencil_registry.h"
#include "stencil_strip.cuh"

namespace perks {

void register_strip_bf16(std::vector<StripKEntry> &out) {
    strip_entries<__nv_bfloat16, S2d5, 4>(out, PERKS_BF16, SH_2D5);
    strip_entries<__nv_bfloat16, S2d9, 4>(out, PERKS_BF16, SH_2D9);
    strip_entries<__nv_bfloat16, S2ds9, 2>(out, PERKS_BF16, SH_2DS9);
    strip_entries<__nv_bfloat16, S2ds9, 4, 192>(out, PERKS_BF16, SH_2DS9);
    strip_entries<__nv_bfloat16, S2d25, 2, 192>(out, PERKS_BF16, SH_2D25);
    // steps left over from whole sweeps
    strip_entries<__nv_bfloat16, S2d5, 1>(out, PERKS_BF16, SH_2D5, true);
    strip_entries<__nv_bfloat16, S2d9, 1>(out, PERKS_BF16, SH_2D9, true);
    strip_entries<__nv_bfloat16, S2ds9, 1>(out, PERKS_BF16, SH_2DS9, true);
    strip_entries<__nv_bfloat16, S2d25, 1, 192>(out, PERKS_BF16, SH_2D25, true);
}

}  // namespace perks
