// Grouped level-0/1 convolution, T = double, block sizes 28 30 32.
#include "group_impl.cuh"

namespace lgf {
template struct GroupSize<double, 28>;
template struct GroupSize<double, 30>;
template struct GroupSize<double, 32>;
}  // namespace lgf
