// Grouped level-0/1 convolution, T = double, block sizes 22 24 26.
#include "group_impl.cuh"

namespace lgf {
template struct GroupSize<double, 22>;
template struct GroupSize<double, 24>;
template struct GroupSize<double, 26>;
}  // namespace lgf
