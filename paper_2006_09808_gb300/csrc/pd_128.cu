// Fused primal-dual kernel instances for 128 x 128 slices.
#include "pd_launch.cuh"

namespace pcs {
using Aux = Geo<128, 128, 4>;
static const KernelEntry k_entries[] = {
    // eight elements per lane, us per iteration (isotropic weighted): 8-CTA clusters 7.7 (10.6) for up to
    // 8 slices, 9.3 (11.8) for 19, 11.2 for 37 (two CTAs per SM); 4-CTA 9.3-9.6 (12.3) for up to 36; 2-CTA 12.6 (16.1) for up to 76, against
    // 9.8 (up to 36) for the resident kernel below.  Sixteen per lane (the last of these) takes 19.3
    // (25.6) for up to 152 slices, where the 2-CTA shape takes 25.2 (32.3); its bits differ from the
    // others', so it is by option only
    make_pair_entry<GeoPair<128, 8, 128, false, 8>, Aux, 1>(9.3f, 11.2f),
    make_pair_entry<GeoPair<128, 4, 256, false, 8>, Aux, 1>(9.4f),
    make_pair_entry<GeoPair<128, 2, 512, true, 8>, Aux, 1>(12.6f),
    make_pair_entry<GeoPair<128, 8, 128, false, 8>, Aux>(9.3f, 11.2f),
    make_pair_entry<GeoPair<128, 4, 256, false, 8>, Aux>(9.4f),
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
