// Fused primal-dual kernel instances for 512 x 512 slices.
#include "pd_launch.cuh"

namespace pcs {
using Aux = Geo<512, 512, 8, 1>;
static const KernelEntry k_entries[] = {
    // 16-CTA clusters of one CTA per SM (8 resident): 32.6 us per iteration of up to 8 slices, 85 us
    // (up to 15) for the half-spectrum kernels below
    make_pair_entry<GeoPair<512, 16, 512, true>, Aux>(32.6f),
    make_entry<Geo<512, 512, 8, 1>>(),
    make_entry<Geo<512, 512, 8, 1, 512>>(),   // 16 warps per SM
    make_entry<Geo<512, 512, 16, 2>>(),       // 16-CTA clusters, two CTAs per SM
};
const KernelEntry* entries_512(int* n) {
    *n = (int)(sizeof(k_entries) / sizeof(k_entries[0]));
    return k_entries;
}
}  // namespace pcs
