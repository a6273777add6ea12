// Fused primal-dual kernel instances for 64 x 64 slices.
#include "pd_launch.cuh"

namespace pcs {
using Aux = Geo<64, 64, 1>;
static const KernelEntry k_entries[] = {
    // four elements per lane: 4.3 us per iteration of one slice in 4-CTA clusters, against 5.7-6.2 with
    // eight and 6.6 for the resident kernel below (300 slices, 100 iterations: 1.34, 1.21, 1.34 ms)
    make_pair_entry<GeoPair<64, 4, 128, false, 4>, Aux, 1>(4.3f),
    make_pair_entry<GeoPair<64, 2, 256, false, 4>, Aux, 1>(5.3f),
    make_pair_entry<GeoPair<64, 1, 512, false, 4>, Aux, 1>(6.6f),
    make_pair_entry<GeoPair<64, 4, 128, false, 4>, Aux>(4.3f),
    make_pair_entry<GeoPair<64, 2, 256, false, 4>, Aux>(5.3f),
    make_pair_entry<GeoPair<64, 1, 512, false, 4>, Aux>(6.6f),
    make_pair_entry<GeoPair<64, 1, 256, false>, Aux>(0.f),
    make_resident_entry<GeoRes<64, 64, 1>>(),
};
const KernelEntry* entries_64(int* n) {
    *n = (int)(sizeof(k_entries) / sizeof(k_entries[0]));
    return k_entries;
}
}  // namespace pcs
