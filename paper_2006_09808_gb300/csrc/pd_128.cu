// Fused primal-dual kernel instances for 128 x 128 slices.
#include "pd_launch.cuh"

namespace pcs {
using Aux = Geo<128, 128, 4>;
static const KernelEntry k_entries[] = {
    // eight elements per lane: 7.5 / 9.3 / 12.6 us per iteration of up to 19 / 36 / 76 slices, against
    // 9.8 us (up to 36) for the resident kernel below; sixteen per lane (the last of these) takes
    // 19.0 us for up to 152
    make_pair_entry<GeoPair<128, 8, 128, false, 8>, Aux, 1>(7.5f),
    make_pair_entry<GeoPair<128, 4, 256, false, 8>, Aux, 1>(9.3f),
    make_pair_entry<GeoPair<128, 2, 512, true, 8>, Aux, 1>(12.6f),
    make_pair_entry<GeoPair<128, 8, 128, false, 8>, Aux>(7.5f),
    make_pair_entry<GeoPair<128, 4, 256, false, 8>, Aux>(9.3f),
    make_pair_entry<GeoPair<128, 2, 512, true, 8>, Aux>(12.6f),
    make_pair_entry<GeoPair<128, 1, 512, true>, Aux>(0.f),
    make_resident_entry<GeoRes<128, 128, 4>>(),
    make_entry<Geo<128, 128, 1, 2>>(),
    make_entry<Geo<128, 128, 2, 2>>(),
};
const KernelEntry* entries_128(int* n) {
    *n = (int)(sizeof(k_entries) / sizeof(k_entries[0]));
    return k_entries;
}
}  // namespace pcs
