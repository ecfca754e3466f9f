// The list-mode pair kernels with the random flux (Eq. 7) for one and two species:
// k_pair's own lists and order of summation, so that a replica without the flux gives
// the same bits beside one with it as alone.
#include "k_pair_impl.cuh"

namespace tdpd {

void launch_pair_flux_lane(const PairArgs &a, cudaStream_t st, int part)
{
    if (a.ns == 1) launch_ns<1, true, false, true>(a, st, part);
    else launch_ns<2, true, false, true>(a, st, part);
}

}  // namespace tdpd
