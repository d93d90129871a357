// Grouped level-0/1 convolution, T = float, block sizes 28 30 32.
#include "group_impl.cuh"

namespace lgf {
template struct GroupSize<float, 28>;
template struct GroupSize<float, 30>;
template struct GroupSize<float, 32>;
}  // namespace lgf
