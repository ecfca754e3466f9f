// The list-mode pair kernels for more than two species: the paper's ten, three, and
// up to four, eight or sixteen with the count at run time. A form reads and sums rows
// of its own length whatever the count, so the next longer one costs (fluids at a
// density of 3, us per step; k_pair's layout with a list per lane in brackets): five
// species, 286k particles, 315 in the form of eight, 408 in that of sixteen (365),
// six 324, 446 (430), eight 367, 458 (551); three species, 786k particles, 665 in their
// own form, 673-679 in that of four (665).
#include "k_pair_multi.cuh"

namespace tdpd {

void launch_pair_multi(const PairArgs &a, cudaStream_t st)
{
    if (a.ns == 10) launch_multi_ns<10, false, false>(a, st);
    else if (a.ns == 3) launch_multi_ns<3, false, false>(a, st);
    else if (a.ns <= 4) launch_multi_ns<4, true, false>(a, st);
    else if (a.ns <= 8) launch_multi_ns<8, true, false>(a, st);
    else launch_multi_ns<16, true, false>(a, st);
}

}  // namespace tdpd
