// Fused primal-dual kernel instances for 192 x 192 slices (radix-3 stages).
#include "pd_launch.cuh"

namespace pcs {
using Aux = Geo<192, 192, 2, 2>;
static const KernelEntry k_entries[] = {
    // 3-CTA clusters: 22.4 us per iteration of up to 48 slices, 47 for the half-spectrum kernel below;
    // larger clusters for fewer slices: 15.1 us (up to 20) and 12.0 us (up to 8)
    make_pair_entry<GeoPair<192, 3, 512, true>, Aux>(22.4f),
    make_pair_entry<GeoPair<192, 6, 256, false>, Aux>(15.1f),
    make_pair_entry<GeoPair<192, 12, 128, false>, Aux>(12.0f),
    make_entry<Geo<192, 192, 2, 2>>(),
};
const KernelEntry* entries_192(int* n) {
    *n = (int)(sizeof(k_entries) / sizeof(k_entries[0]));
    return k_entries;
}
}  // namespace pcs
