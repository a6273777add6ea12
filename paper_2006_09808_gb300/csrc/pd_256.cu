// Fused primal-dual kernel instances for 256 x 256 slices (spectrum spread over a cluster).
#include "pd_launch.cuh"

namespace pcs {
using Aux = Geo<256, 256, 4, 1, 512>;
static const KernelEntry k_entries[] = {
    // us per iteration (isotropic weighted): 4-CTA clusters 22.7 (29.6) for up to 36 slices (35 for the
    // half-spectrum kernel in the same geometry, Geo<256, 256, 4, 1, 512>); larger clusters for fewer
    // slices: 8-CTA 16.5 (23.2) for up to 15 and on the balanced schedule 22.5 (31.1) for 20, which 17.05
    // stands for (20 slices in 4-CTA clusters: 22.6 and 29.6), 16-CTA 14.2 (20.9) for up to 7 or 8 (by
    // device)
    make_pair_entry<GeoPair<256, 4, 512, true>, Aux>(22.7f),
    make_pair_entry<GeoPair<256, 8, 256, false>, Aux>(17.05f),
    make_pair_entry<GeoPair<256, 16, 128, false>, Aux>(14.2f),
    make_entry<Geo<256, 256, 4, 2>>(),
    make_resident_entry<GeoRes<256, 256, 8>>(),
    make_entry<Geo<256, 256, 2, 1>>(),
    // eight elements per lane, 512-thread CTAs (more warps per SM)
    make_resident_entry<GeoRes<256, 256, 8, 512, 8, 8>>(),
    // other FFT tile shapes: rows with 8 elements per lane (16 lanes per row, two row passes), or
    // columns with 8 (32 lanes per column)
    make_entry<Geo<256, 256, 4, 1, 512, 8, 16>>(),
    make_entry<Geo<256, 256, 4, 1, 512, 16, 8>>(),
};
const KernelEntry* entries_256(int* n) {
    *n = (int)(sizeof(k_entries) / sizeof(k_entries[0]));
    return k_entries;
}
}  // namespace pcs
