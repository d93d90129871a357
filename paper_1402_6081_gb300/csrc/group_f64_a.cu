// Grouped level-0/1 convolution, T = double, block sizes 4 6 8 10 12.
#include "group_impl.cuh"

namespace lgf {
template struct GroupSize<double, 4>;
template struct GroupSize<double, 6>;
template struct GroupSize<double, 8>;
template struct GroupSize<double, 10>;
template struct GroupSize<double, 12>;
}  // namespace lgf
