// Grouped level-0/1 convolution: declarations shared by the plan builder and
// the kernels (group_impl.cuh).
//
// Merged levels 0 and 1 (Sec. 4: level-1 nodes are the grid points) sum, for a
// target block, over every block of the 27 sibling groups around its own
// group: near field and level-1 interaction list together.  For a whole group
// that is the near field of one cube of N = 2 n_b points per edge, so the
// group itself is transformed, zero-padded to S = 4 n_b, and takes 27 complex
// products per frequency with the spectra of the offsets e N, |e_a| <= 1.  The
// group's spectrum has as many values as those of its eight blocks padded
// to 2 n_b, whose products are 8 x 27: the same sums, an eighth of the
// products.
#pragma once

#include <cstdint>

#include <cuda_runtime_api.h>

namespace lgf {

// Columns kx S + ky of a group's spectrum; a column is one z line.
inline int64_t group_columns(int n_b) { return int64_t(4 * n_b) * (2 * n_b + 1); }
// Stored rows of the kernel table: offsets id 13 .. 26 of 27 (x fastest), row
// id - 13; offset 26 - id is the conjugate.  FP64 [row][column][kz]; FP32
// [column][row][pair of frequencies] (re, re, im, im), a line's pairs in the
// order of its image.
constexpr int kGroupRows = 14;

// FP32 transforms the z lines a band of columns at a time, as part of the
// products, into images sized to stay in L2; FP64 keeps all spectra in device
// memory: there the arithmetic, not the traffic, is the bound.
template <typename T>
constexpr bool group_banded() { return sizeof(T) == 4; }

// A set of 2^3 target groups is a record of kSetInts ints: the 4^3 groups
// around it, x fastest from the set's lower corner minus 1, an absent one
// n_groups (FP32: a line of zeros) or -1 (FP64); its 8 groups, -1 absent; a
// mask of the 16 x rows that hold a source.
constexpr int kSetInts = 76;   // 16-byte multiple

struct GroupTables {
    int n_groups = 0, n_super = 0;
    const int* blk = nullptr;   // n_groups x 8: block of each child (-1: absent)
    const int* aux = nullptr;   // n_groups x 8: level-1 field slot added to its output (-1: none)
    const void* tw = nullptr;   // exp(2 pi i j / S), j < S, in the plan precision
    const int4* sets = nullptr; // n_super records
    // FP32: columns of a band, and its images (band_cols x (n_groups + 1) lines,
    // the last line of a column zero)
    int band_cols = 0;
    void* images = nullptr;
};
// FP32: values of a line's image, columns taken together, and a column's
// frequencies: 8 rows of rb, stored as 8 x pairs (re, re, im, im)
struct GroupShape { int image = 0, cols = 1, rb = 0, pairs = 0; };
GroupShape group_shape(int n_b);

// early: the kernel that precedes on st (the previous phase) may still be
// draining when this phase's first kernel starts (programmatic serialization;
// the kernels wait for it themselves).  The forward phase waits for all prior
// work; early there is for its own second kernel.
//
// One block size.  xy: n_groups * columns * N complex values (z lines of the
// x, y transforms); FP64: spec: columns * n_groups * S.
//   FP32: forward -> xy; products: xy -> out (as xy); inverse: out
//   FP64: forward -> xy, then spec; products: spec -> xy; inverse: xy
template <typename T, int NB>
struct GroupSize {
    static cudaError_t forward(const GroupTables& g, const T* f, void* xy, void* spec, int early, cudaStream_t st);
    static cudaError_t products(const GroupTables& g, const void* in, const void* kern, void* out, int early,
                                cudaStream_t st);
    // inverse xy transforms into the blocks of u, plus the level-1 field add
    // (slots of add_n^3 values, add_stride apart) when given
    static cudaError_t inverse(const GroupTables& g, const void* xy, T* u, const T* add, int add_n,
                               int64_t add_stride, int early, cudaStream_t st);
};

bool group_supported(int n_b);
template <typename T>
struct Group {
    static cudaError_t forward(int n_b, const GroupTables& g, const T* f, void* xy, void* spec, int early, cudaStream_t st);
    static cudaError_t products(int n_b, const GroupTables& g, const void* in, const void* kern, void* out,
                                int early, cudaStream_t st);
    static cudaError_t inverse(int n_b, const GroupTables& g, const void* xy, T* u, const T* add, int add_n,
                               int64_t add_stride, int early, cudaStream_t st);
};

}  // namespace lgf
