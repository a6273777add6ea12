// Fused primal-dual kernel instances for 64 x 64 slices.
#include "pd_launch.cuh"

namespace pcs {
using Aux = Geo<64, 64, 1>;
static const KernelEntry k_entries[] = {
    // four elements per lane, us per iteration (isotropic weighted): 4-CTA clusters 4.4 (6.4) for 8 slices,
    // 5.4 (7.4) for 37 and 6.5 (8.2) for 76 (two CTAs per SM), 2-CTA 5.4 (7.5) for up to 76 and 7.9 (9.6)
    // for 152, one CTA 6.7 (8.0) for up to 152.  Eight per lane (the last of these, other bits, by option
    // only) 6.0 (8.6): 300 slices 11.9 against 13.2
    make_pair_entry<GeoPair<64, 4, 128, false, 4>, Aux, 1>(5.4f, 6.5f),
    make_pair_entry<GeoPair<64, 2, 256, false, 4>, Aux, 1>(5.45f, 7.9f),
    make_pair_entry<GeoPair<64, 1, 512, false, 4>, Aux, 1>(6.7f),
    make_pair_entry<GeoPair<64, 4, 128, false, 4>, Aux>(5.4f, 6.5f),
    make_pair_entry<GeoPair<64, 2, 256, false, 4>, Aux>(5.45f, 7.9f),
    make_pair_entry<GeoPair<64, 1, 512, false, 4>, Aux>(6.7f),
    make_pair_entry<GeoPair<64, 1, 256, false>, Aux>(0.f),
    make_resident_entry<GeoRes<64, 64, 1>>(),
};
const KernelEntry* entries_64(int* n) {
    *n = (int)(sizeof(k_entries) / sizeof(k_entries[0]));
    return k_entries;
}
}  // namespace pcs
