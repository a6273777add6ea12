// Fused primal-dual kernel instances for 64 x 64 slices.
#include "pd_launch.cuh"

namespace pcs {
using Aux = Geo<64, 64, 1>;
static const KernelEntry k_entries[] = {
    // four elements per lane, us per iteration (isotropic weighted): 4-CTA clusters 4.4 (6.4) for up to
    // 37 slices, 2-CTA 5.4 (7.5) for up to 76, one CTA 6.7 (8.0) for up to 152.  Eight per lane (the last
    // of these, other bits, by option only) 6.0 (8.6), and two per SM: 300 slices 11.9 against 13.2
    make_pair_entry<GeoPair<64, 4, 128, false, 4>, Aux, 1>(4.4f),
    make_pair_entry<GeoPair<64, 2, 256, false, 4>, Aux, 1>(5.4f),
    make_pair_entry<GeoPair<64, 1, 512, false, 4>, Aux, 1>(6.7f),
    make_pair_entry<GeoPair<64, 4, 128, false, 4>, Aux>(4.4f),
    make_pair_entry<GeoPair<64, 2, 256, false, 4>, Aux>(5.4f),
    make_pair_entry<GeoPair<64, 1, 512, false, 4>, Aux>(6.7f),
    make_pair_entry<GeoPair<64, 1, 256, false>, Aux>(0.f),
    make_resident_entry<GeoRes<64, 64, 1>>(),
};
const KernelEntry* entries_64(int* n) {
    *n = (int)(sizeof(k_entries) / sizeof(k_entries[0]));
    return k_entries;
}
}  // namespace pcs
