// Grouped level-0/1 convolution, T = float, block sizes 4 6 8 10 12.
#include "group_impl.cuh"

namespace lgf {
template struct GroupSize<float, 4>;
template struct GroupSize<float, 6>;
template struct GroupSize<float, 8>;
template struct GroupSize<float, 10>;
template struct GroupSize<float, 12>;

#define LGF_GROUP_SWITCH(expr)                                                                                       \
    switch (n_b) {                                                                                                 \
        LGF_X(4, expr) LGF_X(6, expr) LGF_X(8, expr) LGF_X(10, expr) LGF_X(12, expr) LGF_X(14, expr) LGF_X(16, expr) \
        LGF_X(18, expr) LGF_X(20, expr) LGF_X(22, expr) LGF_X(24, expr) LGF_X(26, expr) LGF_X(28, expr)             \
        LGF_X(30, expr) LGF_X(32, expr)                                                                            \
    }
#define LGF_X(n, expr) \
    case n: { using C = grp::ColDim<n>; return expr; }

GroupShape group_shape(int n_b) {
    LGF_GROUP_SWITCH((GroupShape{C::IMG, C::COLS, C::RB, C::U}))
    return {};
}
}  // namespace lgf
