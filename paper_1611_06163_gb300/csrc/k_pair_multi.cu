// The list-mode pair kernels for more than two species: the paper's ten, and up
// to four or sixteen with the count at run time.
#include "k_pair_multi.cuh"

namespace tdpd {

void launch_pair_multi(const PairArgs &a, cudaStream_t st)
{
    if (a.ns == 10) launch_multi_ns<10, false, false>(a, st);
    else if (a.ns <= 4) launch_multi_ns<4, true, false>(a, st);
    else launch_multi_ns<16, true, false>(a, st);
}

}  // namespace tdpd
