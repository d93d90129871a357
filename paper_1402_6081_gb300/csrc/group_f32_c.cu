// Grouped level-0/1 convolution, T = float, block sizes 22 24 26.
#include "group_impl.cuh"

namespace lgf {
template struct GroupSize<float, 22>;
template struct GroupSize<float, 24>;
template struct GroupSize<float, 26>;
}  // namespace lgf
