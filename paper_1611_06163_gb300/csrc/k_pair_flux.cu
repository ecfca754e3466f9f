// The list-mode pair kernels with the random flux (Eq. 7) for more than two species.
#include "k_pair_multi.cuh"

namespace tdpd {

void launch_pair_flux(const PairArgs &a, cudaStream_t st)
{
    if (a.ns == 10) launch_multi_ns<10, false, true>(a, st);
    else if (a.ns <= 4) launch_multi_ns<4, true, true>(a, st);
    else launch_multi_ns<16, true, true>(a, st);
}

}  // namespace tdpd
