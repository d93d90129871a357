// Dispatch of the grouped level-0/1 convolution on the block size (group.h).
#include "group.h"

namespace lgf {

bool group_supported(int n_b) { return n_b >= 4 && n_b <= 32 && n_b % 2 == 0; }

#define LGF_GROUP_SIZES(X) X(4) X(6) X(8) X(10) X(12) X(14) X(16) X(18) X(20) X(22) X(24) X(26) X(28) X(30) X(32)

template <typename T>
cudaError_t Group<T>::forward(int n_b, const GroupTables& g, const T* f, void* xy, void* spec, int early,
                              cudaStream_t st) {
    switch (n_b) {
#define LGF_X(n) \
    case n: return GroupSize<T, n>::forward(g, f, xy, spec, early, st);
        LGF_GROUP_SIZES(LGF_X)
#undef LGF_X
        default: return cudaErrorInvalidValue;
    }
}
template <typename T>
cudaError_t Group<T>::products(int n_b, const GroupTables& g, const void* in, const void* kern, void* out,
                               int early, cudaStream_t st) {
    switch (n_b) {
#define LGF_X(n) \
    case n: return GroupSize<T, n>::products(g, in, kern, out, early, st);
        LGF_GROUP_SIZES(LGF_X)
#undef LGF_X
        default: return cudaErrorInvalidValue;
    }
}
template <typename T>
cudaError_t Group<T>::inverse(int n_b, const GroupTables& g, const void* xy, T* u, const T* add, int add_n,
                              int64_t add_stride, int early, cudaStream_t st) {
    switch (n_b) {
#define LGF_X(n) \
    case n: return GroupSize<T, n>::inverse(g, xy, u, add, add_n, add_stride, early, st);
        LGF_GROUP_SIZES(LGF_X)
#undef LGF_X
        default: return cudaErrorInvalidValue;
    }
}

template struct Group<float>;
template struct Group<double>;

}  // namespace lgf
