// Fused primal-dual kernel instances for 512 x 512 slices.
#include "pd_launch.cuh"

namespace pcs {
using Aux = Geo<512, 512, 8, 1>;
static const KernelEntry k_entries[] = {
    // 16-CTA clusters of one CTA per SM (7 or 8 resident, by device), us per iteration (isotropic weighted):
    // 32.5 (39.4) for up to 7 slices, 72 (87) for 15, 115 (139) for 24; 85-99 (94-133) up to 15 and 153-161
    // for 24 for the half-spectrum kernels below
    make_pair_entry<GeoPair<512, 16, 512, true>, Aux>(32.5f),
    make_entry<Geo<512, 512, 8, 1>>(),
    make_entry<Geo<512, 512, 8, 1, 512>>(),   // 16 warps per SM
    make_entry<Geo<512, 512, 16, 2>>(),       // 16-CTA clusters, two CTAs per SM
};
const KernelEntry* entries_512(int* n) {
    *n = (int)(sizeof(k_entries) / sizeof(k_entries[0]));
    return k_entries;
}
}  // namespace pcs
