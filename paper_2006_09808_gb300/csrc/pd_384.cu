// Fused primal-dual kernel instances for 384 x 384 slices (radix-3 stages).
#include "pd_launch.cuh"

namespace pcs {
using Aux = Geo<384, 384, 4, 1>;
static const KernelEntry k_entries[] = {
    // 8-CTA clusters (15 resident), p in global memory: 48.5 us per iteration of up to 15 slices, 107 of
    // 32, 117 of 36, against 96 (up to 30), 111 and 116 for the half-spectrum kernels below
    make_pair_entry<GeoPair<384, 8, 384, true>, Aux>(48.5f),
    make_entry<Geo<384, 384, 4, 1>>(),
    make_entry<Geo<384, 384, 4, 1, 384>>(),   // 12 warps per SM
};
const KernelEntry* entries_384(int* n) {
    *n = (int)(sizeof(k_entries) / sizeof(k_entries[0]));
    return k_entries;
}
}  // namespace pcs
