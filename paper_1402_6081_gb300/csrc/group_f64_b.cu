// Grouped level-0/1 convolution, T = double, block sizes 14 16 18 20.
#include "group_impl.cuh"

namespace lgf {
template struct GroupSize<double, 14>;
template struct GroupSize<double, 16>;
template struct GroupSize<double, 18>;
template struct GroupSize<double, 20>;
}  // namespace lgf
