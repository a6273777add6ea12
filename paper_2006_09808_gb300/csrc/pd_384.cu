// Fused primal-dual kernel instances for 384 x 384 slices (radix-3 stages).
#include "pd_launch.cuh"

namespace pcs {
using Aux = Geo<384, 384, 4, 1>;
static const KernelEntry k_entries[] = {
    // 8-CTA clusters (15 resident), p in global memory, us per iteration (isotropic weighted): 47.3 (54)
    // for one slice, 50 (57) for 15, 78 (90) for 24, 105 (120) for 32, 118 (134) for 36, 156 (178) for 48,
    // against 96-99 (109-117) up to 16, 104-109, 113-120, 116-125 and 156-166 for the half-spectrum
    // kernels below
    make_pair_entry<GeoPair<384, 8, 384, true>, Aux>(50.f),
    make_entry<Geo<384, 384, 4, 1>>(),
    make_entry<Geo<384, 384, 4, 1, 384>>(),   // 12 warps per SM
};
const KernelEntry* entries_384(int* n) {
    *n = (int)(sizeof(k_entries) / sizeof(k_entries[0]));
    return k_entries;
}
}  // namespace pcs
