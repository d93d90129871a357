// Grouped level-0/1 convolution, T = float, block sizes 14 16 18 20.
#include "group_impl.cuh"

namespace lgf {
template struct GroupSize<float, 14>;
template struct GroupSize<float, 16>;
template struct GroupSize<float, 18>;
template struct GroupSize<float, 20>;
}  // namespace lgf
