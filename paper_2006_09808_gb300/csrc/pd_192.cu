// Fused primal-dual kernel instances for 192 x 192 slices (radix-3 stages).
#include "pd_launch.cuh"

namespace pcs {
using Aux = Geo<192, 192, 2, 2>;
static const KernelEntry k_entries[] = {
    // us per iteration (isotropic weighted): 12-CTA clusters 12.4 (16.5) for up to 8 slices, 15.05 (19.3) for
    // 9 to 16 and 16.5 for 20 (two CTAs per SM from the ninth on), 6-CTA 15.4-15.7 (19.3) for up to 21 and,
    // on the balanced schedule, 16.8 (21.1) for 24, 3-CTA 22.8 (27.6) for up to 40; 47 (57) for the
    // half-spectrum kernel below
    make_pair_entry<GeoPair<192, 3, 512, true>, Aux>(22.8f),
    make_pair_entry<GeoPair<192, 6, 256, false>, Aux>(15.4f),
    make_pair_entry<GeoPair<192, 12, 128, false>, Aux>(15.05f, 16.8f),
    make_entry<Geo<192, 192, 2, 2>>(),
};
const KernelEntry* entries_192(int* n) {
    *n = (int)(sizeof(k_entries) / sizeof(k_entries[0]));
    return k_entries;
}
}  // namespace pcs
