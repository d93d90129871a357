// Solve kernels for the block sizes that the per-block, in-shared-memory
// kernels cannot hold (even n_b of [18, 32]): the same steps of Sec. 3.1 with
// every size a run-time argument.
//
//  * Transforms (Eqs. alg_upfft, alg_dwfft): one axis per launch, between the
//    level's spectrum buffer and a scratch indexed by item that holds only
//    the planes a zero-padded line can reach, each output value of a line the
//    plain DFT sum over its non-zero inputs (at most n of the S samples are
//    non-zero along an axis: zero padding), with the twiddles of a table
//    filled from FP64 host values.  Consecutive threads take consecutive kx,
//    so every pass reads and writes whole 32-value runs.
//  * Products (Eq. alg_mult): a CTA per chunk of 32 frequencies and range of
//    target sibling groups, the chunk's 343 coefficient rows staged once in
//    shared memory from the half table, a warp per group at a time with the
//    sibling products of each neighbour group's present sources in registers.
//  * Reg and Interp (Eqs. alg_reg, alg_interp): the x and y passes by slabs of
//    an item's planes, the z passes (Reg: of a parent's eight children) by
//    bundles of columns; each sum over its row's band of the stencil matrix,
//    compensated FP32 sums where asked.
#include <algorithm>

#include "kernels_impl.cuh"

namespace lgf {
namespace gen {

using dev::cx;
using dev::czero;
using dev::ldg_cx;

constexpr int kThreads = 256;
constexpr int kLineThreads = 128;   // lines per CTA of the y / z passes

// (cos, sign sin)(2 pi m / S), m < S, into shared memory
template <typename T>
__device__ __forceinline__ void load_twiddles(cx<T>* tw_s, const cx<T>* __restrict__ twt, int S, int sign) {
    for (int m = threadIdx.x; m < S; m += blockDim.x) {
        const cx<T> w = ldg_cx(twt + m);
        tw_s[m] = {w.x, T(sign) * w.y};
    }
}
__device__ __forceinline__ int wrap(int i, int S) { return i >= S ? i - S : i; }

// ---- forward transform, x: real rows of the input to the first NX values.
// The N^2 NX outputs (row, k) of an item, k fastest, are cut into `tiles`
// tiles of tile_len; a CTA stages its tile's rows in shared memory and then
// computes kXTile / kThreads outputs per thread, the twiddle index (x k mod S)
// advanced by k per term.
constexpr int kXTile = 4 * kThreads;

template <typename T>
__global__ void __launch_bounds__(kThreads) g_r2c_x(const T* __restrict__ src, int64_t stride,
                                                    const R2CItem* __restrict__ items, int tiles, int tile_len,
                                                    cx<T>* __restrict__ A, int64_t nws, int S, int N,
                                                    const cx<T>* __restrict__ twt) {
    extern __shared__ __align__(16) unsigned char g_smem[];
    cx<T>* tw_s = reinterpret_cast<cx<T>*>(g_smem);
    T* rows = reinterpret_cast<T*>(tw_s + S);   // [rows of this tile][N]
    const int NX = S / 2 + 1, per_item = N * N * NX;
    const int it = blockIdx.x / tiles, j0 = (blockIdx.x % tiles) * tile_len;
    const int j1 = min(j0 + tile_len, per_item);
    const int row0 = j0 / NX, row1 = (j1 - 1) / NX + 1;
    const R2CItem item = items[it];
    const T* in = src + int64_t(item.src) * stride + int64_t(row0) * N;
    load_twiddles(tw_s, twt, S, -1);
    for (int q = threadIdx.x; q < (row1 - row0) * N; q += blockDim.x) rows[q] = __ldg(in + q);
    __syncthreads();
    cx<T>* out = A + int64_t(item.dst) * nws;
    for (int j = j0 + threadIdx.x; j < j1; j += blockDim.x) {
        const int k = j % NX, row = j / NX;
        const T* v = rows + (row - row0) * N;
        cx<T> acc = czero<T>();
        int idx = 0;
        for (int x = 0; x < N; ++x) {
            const cx<T> w = tw_s[idx];
            acc.x = fma(v[x], w.x, acc.x);
            acc.y = fma(v[x], w.y, acc.y);
            idx = wrap(idx + k, S);
        }
        const int y = row % N, z = row / N;
        out[(z * S + y) * NX + k] = acc;
    }
}

// ---- one complex axis (y: stride NX, planes z < N; z: stride S NX, all y)
// out[j] = sum_{m < nin} in[m] exp(sign i 2 pi j m / S), j < nout.  A side
// with slots addresses item it at slots[it * slot_stride] * its stride (the
// level's spectrum buffer), one without at it * its stride (the transform
// scratch, whose items hold only the planes the other passes use).  Thread
// per line (item, other, kx), kx fastest so the loads and stores of a warp are
// contiguous; the line's inputs are staged in shared memory (column per
// thread) and every output sums them against warp-uniform twiddles, two
// outputs per trip.
template <typename T>
__global__ void __launch_bounds__(kLineThreads) g_axis(const cx<T>* __restrict__ in,
                                                       const int* __restrict__ in_slots, int64_t in_ws,
                                                       cx<T>* __restrict__ out, const int* __restrict__ out_slots,
                                                       int64_t out_ws, int slot_stride, int n_items, int S, int nin,
                                                       int nout, int n_other, int64_t axis_stride,
                                                       int64_t other_stride, int sign,
                                                       const cx<T>* __restrict__ twt) {
    extern __shared__ __align__(16) unsigned char g_smem[];
    cx<T>* tw_s = reinterpret_cast<cx<T>*>(g_smem);
    cx<T>* col = tw_s + S + threadIdx.x;        // [nin][blockDim.x], this thread's column
    load_twiddles(tw_s, twt, S, sign);
    __syncthreads();
    const int NX = S / 2 + 1;
    const int64_t lines = int64_t(n_items) * n_other * NX;
    const int64_t L = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (L >= lines) return;
    const int kx = int(L % NX);
    const int64_t t = L / NX;
    const int o = int(t % n_other), it = int(t / n_other);
    const int64_t line = int64_t(o) * other_stride + kx;
    const int64_t ib = (in_slots ? int64_t(in_slots[int64_t(it) * slot_stride]) : int64_t(it)) * in_ws + line;
    const int64_t ob = (out_slots ? int64_t(out_slots[int64_t(it) * slot_stride]) : int64_t(it)) * out_ws + line;
    for (int m = 0; m < nin; ++m) col[m * blockDim.x] = ldg_cx(in + ib + int64_t(m) * axis_stride);
    for (int j = 0; j < nout; j += 2) {
        const int j1 = j + 1 < S ? j + 1 : 0;
        cx<T> a0 = czero<T>(), a1 = czero<T>();
        int i0 = 0, i1 = 0;
        for (int m = 0; m < nin; ++m) {
            const cx<T> v = col[m * blockDim.x];
            const cx<T> w0 = tw_s[i0], w1 = tw_s[i1];
            a0.x = fma(v.x, w0.x, fma(-v.y, w0.y, a0.x));
            a0.y = fma(v.x, w0.y, fma(v.y, w0.x, a0.y));
            a1.x = fma(v.x, w1.x, fma(-v.y, w1.y, a1.x));
            a1.y = fma(v.x, w1.y, fma(v.y, w1.x, a1.y));
            i0 = wrap(i0 + j, S);
            i1 = wrap(i1 + j1, S);
        }
        out[ob + int64_t(j) * axis_stride] = a0;
        if (j + 1 < nout) out[ob + int64_t(j + 1) * axis_stride] = a1;
    }
}

// ---- inverse transform, x: Hermitian rows to the first N real samples (+ add).
// The N^3 outputs (row, x) of an item, x fastest, cut into tiles as above; a
// CTA stages its tile's rows of NX values in shared memory.
template <typename T>
__global__ void __launch_bounds__(kThreads) g_c2r_x(const cx<T>* __restrict__ U, const C2RItem* __restrict__ items,
                                                    int tiles, int tile_len, T* __restrict__ dst, int64_t dst_stride,
                                                    const T* __restrict__ add, int add_n, int64_t add_stride,
                                                    int64_t nws, int S, int N, const cx<T>* __restrict__ twt) {
    extern __shared__ __align__(16) unsigned char g_smem[];
    cx<T>* tw_s = reinterpret_cast<cx<T>*>(g_smem);
    const int NX = S / 2 + 1, per_item = N * N * N;
    cx<T>* rows = tw_s + S;                     // [rows of this tile][NX]
    const int it = blockIdx.x / tiles, j0 = (blockIdx.x % tiles) * tile_len;
    const int j1 = min(j0 + tile_len, per_item);
    const int row0 = j0 / N, row1 = (j1 - 1) / N + 1;
    const C2RItem item = items[it];
    const cx<T>* in = U + int64_t(item.src) * nws;
    load_twiddles(tw_s, twt, S, +1);
    for (int q = threadIdx.x; q < (row1 - row0) * NX; q += blockDim.x) {
        const int row = row0 + q / NX, k = q % NX;
        rows[q] = ldg_cx(in + ((row / N) * S + row % N) * NX + k);
    }
    __syncthreads();
    T* out = dst + int64_t(item.dst) * dst_stride;
    const T* ad = (add != nullptr && item.aux >= 0) ? add + int64_t(item.aux) * add_stride : nullptr;
    for (int j = j0 + threadIdx.x; j < j1; j += blockDim.x) {
        const int x = j % N, row = j / N;
        const cx<T>* X = rows + (row - row0) * NX;
        // x[n] = X[0] + 2 sum_{0 < k < S/2} Re(X[k] e^{+i 2 pi n k / S}) + X[S/2] (-1)^n (S even)
        T acc = X[0].x;
        const int kmax = (S % 2 == 0) ? S / 2 : NX;
        int idx = wrap(x, S);
        for (int k = 1; k < kmax; ++k) {
            const cx<T> w = tw_s[idx];
            acc += T(2) * (X[k].x * w.x - X[k].y * w.y);
            idx = wrap(idx + x, S);
        }
        if (S % 2 == 0) acc += ((x & 1) ? T(-1) : T(1)) * X[S / 2].x;
        const int y = row % N, z = row / N;
        if (ad) acc += __ldg(ad + (z * add_n + y) * add_n + x);
        out[row * N + x] = acc;
    }
}

// ---- products: a CTA per (group range, chunk of 32 frequencies).  The table
// is stored chunk by chunk ([chunk][172][32], get_spectra), so a chunk's rows
// are one run; the 343 coefficient rows are staged from it once, then the
// CTA's 8 warps take the range's groups in turn (warp w: groups g0 + w, g0 +
// w + 8, ...).  Sources without a block (mask[q], bit c: child c of group q
// has a spectrum; the others' are zero) are skipped, which is most of the
// work where the level's groups are sparse.  27 intervals in 8 groups,
// 65 000 frequencies (n_b = 24, 144^3, FP32): 89 us; 181 with the table row by
// row (172 rows 520 KB apart) and all sources.
template <typename T>
__global__ void __launch_bounds__(256) g_mac(const cx<T>* __restrict__ fh, const cx<T>* __restrict__ kh,
                                             cx<T>* __restrict__ uh, const int* __restrict__ gnbr,
                                             const int* __restrict__ mask, int n_groups, int groups_per_cta,
                                             int include_self, int64_t nw, int64_t nws) {
    extern __shared__ __align__(16) unsigned char g_smem[];
    cx<T>* sk = reinterpret_cast<cx<T>*>(g_smem);   // [343][32]
    const int64_t w0 = int64_t(blockIdx.y) * 32;
    const int tid = threadIdx.y * 32 + threadIdx.x;
    {
        // stored row r: offset 171 + r, and conjugated offset 171 - r
        constexpr int kPer = 16 / int(sizeof(cx<T>)), kTotal = 172 * 32 / kPer, kBatch = 8;
        struct alignas(16) Vec { cx<T> v[kPer]; };
        const Vec* src = reinterpret_cast<const Vec*>(kh + int64_t(blockIdx.y) * 172 * 32);
        for (int base = tid; base < kTotal; base += kBatch * 256) {
            Vec v[kBatch];
#pragma unroll
            for (int j = 0; j < kBatch; ++j)
                if (base + j * 256 < kTotal) v[j] = src[base + j * 256];
#pragma unroll
            for (int j = 0; j < kBatch; ++j) {
                const int i = (base + j * 256) * kPer, r = i / 32;
                if (i >= 172 * 32) break;
                *reinterpret_cast<Vec*>(sk + (171 + r) * 32 + i % 32) = v[j];
                if (r == 0) continue;
#pragma unroll
                for (int k = 0; k < kPer; ++k) v[j].v[k] = dev::conjx(v[j].v[k]);
                *reinterpret_cast<Vec*>(sk + (171 - r) * 32 + i % 32) = v[j];
            }
        }
    }
    __syncthreads();
    const int64_t w = w0 + threadIdx.x;
    const int64_t wc = w < nw ? w : nw - 1;
    const int g0 = blockIdx.x * groups_per_cta, g1 = min(g0 + groups_per_cta, n_groups);
    for (int g = g0 + int(threadIdx.y); g < g1; g += 8) {
        cx<T> acc[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) acc[c] = czero<T>();
        for (int e = 0; e < 27; ++e) {
            if (e == 13 && !include_self) continue;
            const int q = __ldg(gnbr + int64_t(g) * 27 + e);
            const int m = q < 0 ? 0 : __ldg(mask + q);
            if (m == 0) continue;
            cx<T> F[8];
#pragma unroll
            for (int c = 0; c < 8; ++c)
                if (m >> c & 1) F[c] = ldg_cx(fh + (int64_t(q) * 8 + c) * nws + wc);
            // centre offset d = 2e of this neighbour in the 7^3 coefficient rows
            const cx<T>* kb = sk + ((2 * (e % 3) + 1) + 7 * (2 * (e / 3 % 3) + 1) + 49 * (2 * (e / 9) + 1)) * 32 +
                              threadIdx.x;
#pragma unroll
            for (int s = 0; s < 8; ++s) {
                if (!(m >> s & 1)) continue;
#pragma unroll
                for (int t = 0; t < 8; ++t) {
                    const int d = ((s & 1) - (t & 1)) + 7 * ((s >> 1 & 1) - (t >> 1 & 1)) + 49 * ((s >> 2) - (t >> 2));
                    acc[t] = dev::cmac(acc[t], F[s], kb[d * 32]);
                }
            }
        }
        if (w < nw) {
#pragma unroll
            for (int c = 0; c < 8; ++c) uh[(int64_t(g) * 8 + c) * nws + w] = acc[c];
        }
    }
}

// ---- Reg and Interp: 1D passes, value (o along the axis) = sum_k M(o, k)
// in[k along the axis], M(o, k) = W[c][o][k] (interpolation) or W[c][k][o]
// (its adjoint).  Every row of M is non-zero on one contiguous band of k (the
// n_max nearest nodes of a point, or for the adjoint the points whose stencils
// hold a node), found once per CTA (band[c][o] = lo | hi << 16).
//
// The x and y passes of an item need one plane at a time, the z pass a bundle
// of columns, so an item is cut into slabs of planes and then into bundles of
// columns, with the planes between the two launches in a slices buffer (one
// cube per item, L2-resident for the domains that leave SMs idle).  A CTA per
// item, all three passes on its cubes, left half the warps out (125 KB of
// cubes at n_I = 25: one CTA per SM) and ran 216 items in two waves.  Bound by
// the instructions of the sums (8 per compensated term) and their setup: 144^3,
// n_b = 24, compensated FP32, Reg 206 -> 88 us, Interp 167 -> 73 us.
//
// A warp takes one output index o for many lines: the weight is one broadcast
// read for kLines terms per lane and the band is the same for all lanes.

constexpr int kRiThreads = 256;
constexpr int kLines = 4;   // lines per lane

template <typename T, bool COMP>
struct Sum {
    T s = T(0), e = T(0);   // COMP: sum and its error; else two partial sums (two chains in flight)
    __device__ __forceinline__ void add(T w, T x, int k) {
        if constexpr (COMP) {
            dev::acc_comp(s, e, w, x);
        } else {
            T& a = k & 1 ? e : s;
            a = fma(w, x, a);
        }
    }
    __device__ __forceinline__ T get() const { return s + e; }
};

// one output of LINES lines of a lane: line j's value k at in[at[j] + k * st]
template <typename T, bool COMP, int LINES>
__device__ __forceinline__ void lines(Sum<T, COMP> (&acc)[LINES], const T* in, const int (&at)[LINES], int st,
                                      const T* w, int wstep, int lo, int hi) {
    int k = lo;
    for (; k + 1 < hi; k += 2) {
        const T w0 = w[k * wstep], w1 = w[(k + 1) * wstep];
#pragma unroll
        for (int j = 0; j < LINES; ++j) {
            acc[j].add(w0, in[at[j] + k * st], 0);
            acc[j].add(w1, in[at[j] + (k + 1) * st], 1);
        }
    }
    if (k < hi) {
#pragma unroll
        for (int j = 0; j < LINES; ++j) acc[j].add(w[k * wstep], in[at[j] + k * st], 0);
    }
}

// W (2 x n x n) and the bands of M for both children into shared memory
template <typename T, bool ADJ>
__device__ void load_stencil(T* W_s, int* band, const T* __restrict__ W, int n) {
    for (int i = threadIdx.x; i < 2 * n * n; i += kRiThreads) W_s[i] = __ldg(W + i);
    __syncthreads();
    const int lane = threadIdx.x & 31;
    for (int q = threadIdx.x / 32; q < 2 * n; q += kRiThreads / 32) {
        const int c = q / n, o = q % n;
        const T* Wc = W_s + c * n * n;
        auto live = [&](int k) { return k < n && (ADJ ? Wc[k * n + o] : Wc[o * n + k]) != T(0); };
        const unsigned long long m = uint64_t(__ballot_sync(~0u, live(lane))) |
                                     uint64_t(__ballot_sync(~0u, live(lane + 32))) << 32;
        if (lane == 0) band[q] = m == 0 ? 0 : (__ffsll(int64_t(m)) - 1) | ((64 - __clzll(int64_t(m))) << 16);
    }
    __syncthreads();
}

// bytes of W and the bands, and the planes of a slab (its lines: kLines per lane)
template <typename T>
__host__ __device__ size_t stencil_bytes(int n) {
    return (sizeof(T) * 2 * n * n + sizeof(int) * 2 * n + 15) / 16 * 16;
}
__host__ __device__ constexpr int slab_planes(int n) { return 32 * kLines / n; }

// x and y passes of a slab of planes of item q: child c = q & 7 (Reg: 8 items
// per parent) or slot[q] & 7 (Interp), the cube source[q] of src (edge in_n =
// NI, or NI - 1 and zero beyond), none where that is < 0.  Planes of NI (odd)
// rows of NI values: no bank conflicts along either axis.
template <typename T, bool ADJ, bool COMP>
__global__ void __launch_bounds__(kRiThreads) g_planes(const T* __restrict__ src, int in_n,
                                                       const int* __restrict__ source, const int* __restrict__ slot,
                                                       int slabs, const T* __restrict__ W, int NI,
                                                       T* __restrict__ slices) {
    extern __shared__ __align__(16) unsigned char g_smem[];
    const int N2 = NI * NI, P = slab_planes(NI);
    T* W_s = reinterpret_cast<T*>(g_smem);
    int* band = reinterpret_cast<int*>(W_s + 2 * N2);
    T* t1 = reinterpret_cast<T*>(g_smem + stencil_bytes<T>(NI));
    T* t2 = t1 + P * N2;
    const int q = blockIdx.x / slabs, z0 = (blockIdx.x % slabs) * P, np = min(P, in_n - z0);
    const int s = source[q];
    if (s < 0) return;   // uniform over the CTA
    const int c = slot ? slot[q] & 7 : q & 7;
    const T* in = src + (int64_t(s) * in_n + z0) * in_n * in_n;
    for (int i = threadIdx.x; i < np * N2; i += kRiThreads) {
        const int x = i % NI, r = i / NI, y = r % NI, z = r / NI;
        t1[i] = x < in_n && y < in_n ? __ldg(in + (z * in_n + y) * in_n + x) : T(0);
    }
    load_stencil<T, ADJ>(W_s, band, W, NI);
    const int lane = threadIdx.x & 31, warp = threadIdx.x / 32, rows = np * NI;
    int at[kLines];
#pragma unroll
    for (int j = 0; j < kLines; ++j) at[j] = min(lane + 32 * j, rows - 1) * NI;
    const int cx_ = c & 1, cy_ = (c >> 1) & 1, wstep = ADJ ? NI : 1;
    for (int o = warp; o < NI; o += kRiThreads / 32) {   // x: rows
        Sum<T, COMP> acc[kLines];
        const int b = band[cx_ * NI + o];
        lines<T, COMP, kLines>(acc, t1, at, 1, W_s + cx_ * N2 + (ADJ ? o : o * NI), wstep, b & 0xffff, b >> 16);
#pragma unroll
        for (int j = 0; j < kLines; ++j)
            if (lane + 32 * j < rows) t2[at[j] + o] = acc[j].get();
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kLines; ++j) {
        const int l = min(lane + 32 * j, rows - 1);
        at[j] = l / NI * N2 + l % NI;
    }
    T* out = slices + (int64_t(q) * NI + z0) * N2;
    for (int o = warp; o < NI; o += kRiThreads / 32) {   // y: columns of a plane
        Sum<T, COMP> acc[kLines];
        const int b = band[cy_ * NI + o];
        lines<T, COMP, kLines>(acc, t2, at, NI, W_s + cy_ * N2 + (ADJ ? o : o * NI), wstep, b & 0xffff, b >> 16);
#pragma unroll
        for (int j = 0; j < kLines; ++j)
            if (lane + 32 * j < rows) out[at[j] + o * NI] = acc[j].get();
    }
}

// Reg's z pass: a CTA per parent and 32 columns sums the present children's
// slices (planes below in_n), children in order.
template <typename T, bool COMP>
__global__ void __launch_bounds__(kRiThreads) g_reg_z(const int* __restrict__ child_index,
                                                      const int* __restrict__ parent_slot, int in_n, int bundles,
                                                      T* __restrict__ dst, const T* __restrict__ W, int NI,
                                                      const T* __restrict__ slices) {
    extern __shared__ __align__(16) unsigned char g_smem[];
    const int N2 = NI * NI, N3 = N2 * NI;
    T* W_s = reinterpret_cast<T*>(g_smem);
    int* band = reinterpret_cast<int*>(W_s + 2 * N2);
    T* t = reinterpret_cast<T*>(g_smem + stencil_bytes<T>(NI));   // [child][k][32]
    const int p = blockIdx.x / bundles, lane = threadIdx.x & 31, warp = threadIdx.x / 32;
    const int col = (blockIdx.x % bundles) * 32 + lane, colc = min(col, N2 - 1);
    for (int c = 0; c < 8; ++c) {
        if (child_index[p * 8 + c] < 0) continue;
        const T* in = slices + (int64_t(p) * 8 + c) * N3 + colc;
#pragma unroll 4
        for (int k = warp; k < in_n; k += kRiThreads / 32) t[(c * NI + k) * 32 + lane] = in[k * N2];
    }
    load_stencil<T, true>(W_s, band, W, NI);
    T* out = dst + int64_t(parent_slot[p]) * N3 + col;
    for (int o = warp; o < NI; o += kRiThreads / 32) {
        Sum<T, COMP> acc[1];
        for (int c = 0; c < 8; ++c) {
            if (child_index[p * 8 + c] < 0) continue;
            const int cz_ = c >> 2, b = band[cz_ * NI + o];
            const int at[1] = {c * NI * 32 + lane};
            lines<T, COMP, 1>(acc, t, at, 32, W_s + cz_ * N2 + o, NI, b & 0xffff, min(b >> 16, in_n));
        }
        if (col < N2) out[o * N2] = acc[0].get();
    }
}

// Interp's z pass: a CTA per item and 32 kLines columns, into the child's cube
// of u or (block != nullptr) added to its first NI - 1 nodes per axis in u's
// block.
template <typename T, bool COMP>
__global__ void __launch_bounds__(kRiThreads) g_interp_z(const int* __restrict__ slot, int bundles,
                                                         T* __restrict__ u, const T* __restrict__ W, int NI,
                                                         int accumulate, const int* __restrict__ block,
                                                         const T* __restrict__ slices) {
    extern __shared__ __align__(16) unsigned char g_smem[];
    constexpr int kCols = 32 * kLines;
    const int NB = NI - 1, N2 = NI * NI, N3 = N2 * NI;
    T* W_s = reinterpret_cast<T*>(g_smem);
    int* band = reinterpret_cast<int*>(W_s + 2 * N2);
    T* t = reinterpret_cast<T*>(g_smem + stencil_bytes<T>(NI));   // [k][kCols]
    const int it = blockIdx.x / bundles, col0 = (blockIdx.x % bundles) * kCols;
    const int lane = threadIdx.x & 31, warp = threadIdx.x / 32;
    const T* in = slices + int64_t(it) * N3;
#pragma unroll 4
    for (int i = threadIdx.x; i < NI * kCols; i += kRiThreads)
        t[i] = in[(i / kCols) * N2 + min(col0 + i % kCols, N2 - 1)];
    load_stencil<T, false>(W_s, band, W, NI);
    const int s = slot[it], cz_ = (s >> 2) & 1;
    int at[kLines], to[kLines];   // to: the column's place in the output, < 0: none
#pragma unroll
    for (int j = 0; j < kLines; ++j) {
        at[j] = lane + 32 * j;
        const int col = col0 + at[j], x = col % NI, y = col / NI;
        to[j] = block ? (x < NB && y < NB ? y * NB + x : -1) : (col < N2 ? col : -1);
    }
    const int nz = block ? NB : NI, step = block ? NB * NB : N2;
    T* out = block ? u + int64_t(block[it]) * NB * NB * NB : u + int64_t(s) * N3;
    const bool add = block || accumulate;
    for (int o = warp; o < nz; o += kRiThreads / 32) {
        Sum<T, COMP> acc[kLines];
        const int b = band[cz_ * NI + o];
        lines<T, COMP, kLines>(acc, t, at, kCols, W_s + cz_ * N2 + o * NI, 1, b & 0xffff, b >> 16);
#pragma unroll
        for (int j = 0; j < kLines; ++j) {
            if (to[j] < 0) continue;
            T* v = out + to[j] + o * step;
            *v = add ? *v + acc[j].get() : acc[j].get();
        }
    }
}

// an item's x-pass outputs in about equal tiles of at most kXTile
inline void x_tiles(int per_item, int* tiles, int* tile_len) {
    *tiles = (per_item + kXTile - 1) / kXTile;
    *tile_len = (per_item + *tiles - 1) / *tiles;
}

inline unsigned grid_for(int64_t total, int threads = kThreads) {
    return unsigned(std::max<int64_t>(1, (total + threads - 1) / threads));
}

// one complex-axis pass (see g_axis); FP64 lines use half the threads per CTA
// so that a CTA's staged columns stay near 64 KB
template <typename T>
cudaError_t axis_pass(const dev::cx<T>* in, const int* in_slots, int64_t in_ws, dev::cx<T>* out,
                      const int* out_slots, int64_t out_ws, int slot_stride, int n, int S, int nin, int nout,
                      int n_other, int64_t axis_stride, int64_t other_stride, int sign, const dev::cx<T>* tw,
                      cudaStream_t st) {
    const int threads = sizeof(T) == 8 ? kLineThreads / 2 : kLineThreads;
    const size_t smem = sizeof(dev::cx<T>) * (size_t(S) + size_t(nin) * threads);
    cudaError_t e = cudaFuncSetAttribute(g_axis<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
    if (e != cudaSuccess) return e;
    const int64_t lines = int64_t(n) * n_other * (S / 2 + 1);
    g_axis<T><<<grid_for(lines, threads), threads, smem, st>>>(in, in_slots, in_ws, out, out_slots, out_ws,
                                                              slot_stride, n, S, nin, nout, n_other, axis_stride,
                                                              other_stride, sign, tw);
    return launched();
}

}  // namespace gen

template <typename T>
cudaError_t Generic<T>::r2c(int S, int n_in, const T* src, int64_t stride, const R2CItem* items, int n, void* spec,
                            void* scratch, const void* twt, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    const int* slots = reinterpret_cast<const int*>(items) + 1;   // R2CItem::dst, 2 ints apart
    using C = dev::cx<T>;
    const int NX = S / 2 + 1;
    const int64_t nws = nws_of(S);
    auto* A = static_cast<C*>(spec);
    auto* B = static_cast<C*>(scratch);
    const auto* tw = static_cast<const C*>(twt);
    // x: rows (z, y < n_in) into A; y: A -> B (planes z < n_in); z: B -> A
    const int64_t bws = int64_t(n_in) * S * NX;
    int tiles = 0, tile_len = 0;
    gen::x_tiles(n_in * n_in * NX, &tiles, &tile_len);
    const size_t smem_x = sizeof(C) * S + sizeof(T) * size_t((tile_len - 1) / NX + 2) * n_in;
    gen::g_r2c_x<T><<<unsigned(int64_t(n) * tiles), gen::kThreads, smem_x, st>>>(src, stride, items, tiles, tile_len,
                                                                                 A, nws, S, n_in, tw);
    cudaError_t e = launched();
    if (e == cudaSuccess)
        e = gen::axis_pass<T>(A, slots, nws, B, nullptr, bws, 2, n, S, n_in, S, n_in, NX, int64_t(S) * NX, -1, tw, st);
    if (e == cudaSuccess)
        e = gen::axis_pass<T>(B, nullptr, bws, A, slots, nws, 2, n, S, n_in, S, S, int64_t(S) * NX, NX, -1, tw, st);
    return e;
}

template <typename T>
cudaError_t Generic<T>::c2r(int S, int n_out, const void* spec, const C2RItem* items, int n, void* scratch, T* dst,
                            int64_t ds, const T* add, int add_n, int64_t as, const void* twt, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    const int* slots = reinterpret_cast<const int*>(items);       // C2RItem::src, 3 ints apart
    using C = dev::cx<T>;
    const int NX = S / 2 + 1;
    const int64_t nws = nws_of(S);
    auto* U = const_cast<C*>(static_cast<const C*>(spec));
    auto* V = static_cast<C*>(scratch);
    const auto* tw = static_cast<const C*>(twt);
    // z: U -> V (planes z < n_out); y: V -> U keeping y < n_out; x: U -> reals
    const int64_t vws = int64_t(n_out) * S * NX;
    cudaError_t e = gen::axis_pass<T>(U, slots, nws, V, nullptr, vws, 3, n, S, S, n_out, S, int64_t(S) * NX, NX, +1,
                                      tw, st);
    if (e == cudaSuccess)
        e = gen::axis_pass<T>(V, nullptr, vws, U, slots, nws, 3, n, S, S, n_out, n_out, NX, int64_t(S) * NX, +1, tw,
                              st);
    if (e != cudaSuccess) return e;
    int tiles = 0, tile_len = 0;
    gen::x_tiles(n_out * n_out * n_out, &tiles, &tile_len);
    const size_t smem_x = sizeof(C) * (S + size_t((tile_len - 1) / n_out + 2) * NX);
    gen::g_c2r_x<T><<<unsigned(int64_t(n) * tiles), gen::kThreads, smem_x, st>>>(U, items, tiles, tile_len, dst, ds,
                                                                                 add, add_n, as, nws, S, n_out, tw);
    return launched();
}

template <typename T>
cudaError_t Generic<T>::mac(const void* fh, const void* kh, void* uh, const int* gnbr, const int* mask, int n_groups,
                            int S, int include_self, cudaStream_t st) {
    if (n_groups == 0) return cudaSuccess;
    const int64_t nw = nw_of(S), nws = nws_of(S);
    const int64_t chunks = (nw + 31) / 32;
    // groups per CTA: all of them when the chunks alone give four CTAs per SM
    // (two resident at a time), else fewer so that the grid keeps that size;
    // a multiple of the 8 warps
    const int64_t want = 4 * 152;
    int gpc = n_groups;
    if (chunks < want) gpc = int(std::max<int64_t>(8, int64_t(n_groups) * chunks / want));
    gpc = (gpc + 7) / 8 * 8;
    dim3 block(32, 8), grid(unsigned((n_groups + gpc - 1) / gpc), unsigned(chunks));
    const size_t smem = sizeof(dev::cx<T>) * 343 * 32;
    cudaError_t e = cudaFuncSetAttribute(gen::g_mac<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
    if (e != cudaSuccess) return e;
    gen::g_mac<T><<<grid, block, smem, st>>>(static_cast<const dev::cx<T>*>(fh), static_cast<const dev::cx<T>*>(kh),
                                             static_cast<dev::cx<T>*>(uh), gnbr, mask, n_groups, gpc, include_self, nw,
                                             nws);
    return launched();
}

template <typename T, bool ADJ, bool COMP>
static cudaError_t launch_planes(const T* src, int in_n, const int* source, const int* slot, int n_items, const T* W,
                                 int NI, T* slices, cudaStream_t st) {
    const int P = gen::slab_planes(NI), slabs = (in_n + P - 1) / P;
    const size_t smem = gen::stencil_bytes<T>(NI) + sizeof(T) * 2 * P * NI * NI;
    auto k = gen::g_planes<T, ADJ, COMP>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
    if (e != cudaSuccess) return e;
    k<<<unsigned(int64_t(n_items) * slabs), gen::kRiThreads, smem, st>>>(src, in_n, source, slot, slabs, W, NI, slices);
    return launched();
}

template <typename T, bool COMP>
static cudaError_t launch_reg(int NI, const T* src, int in_n, const int* child_index, const int* parent_slot,
                              int n_parents, T* dst, const T* W, T* slices, cudaStream_t st) {
    cudaError_t e = launch_planes<T, true, COMP>(src, in_n, child_index, nullptr, 8 * n_parents, W, NI, slices, st);
    if (e != cudaSuccess) return e;
    const int bundles = (NI * NI + 31) / 32;
    const size_t smem = gen::stencil_bytes<T>(NI) + sizeof(T) * 8 * NI * 32;
    auto k = gen::g_reg_z<T, COMP>;
    if ((e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem))) != cudaSuccess) return e;
    k<<<unsigned(int64_t(n_parents) * bundles), gen::kRiThreads, smem, st>>>(child_index, parent_slot, in_n, bundles,
                                                                            dst, W, NI, slices);
    return launched();
}

template <typename T, bool COMP>
static cudaError_t launch_interp(int NI, const int* slot, const int* parent, int n_items, T* u, const T* up,
                                 const T* W, int accumulate, const int* block, T* slices, cudaStream_t st) {
    cudaError_t e = launch_planes<T, false, COMP>(up, NI, parent, slot, n_items, W, NI, slices, st);
    if (e != cudaSuccess) return e;
    const int cols = 32 * gen::kLines, bundles = (NI * NI + cols - 1) / cols;
    const size_t smem = gen::stencil_bytes<T>(NI) + sizeof(T) * NI * cols;
    auto k = gen::g_interp_z<T, COMP>;
    if ((e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem))) != cudaSuccess) return e;
    k<<<unsigned(int64_t(n_items) * bundles), gen::kRiThreads, smem, st>>>(slot, bundles, u, W, NI, accumulate, block,
                                                                          slices);
    return launched();
}

template <typename T>
cudaError_t Generic<T>::reg(int n_b, const T* child_src, int child_is_block, const int* child_index,
                            const int* parent_slot, int n_parents, T* dst, const T* W_dev, int comp, T* slices,
                            cudaStream_t st) {
    if (n_parents == 0) return cudaSuccess;
    const int NI = n_b + 1, in_n = child_is_block ? n_b : NI;
    if constexpr (sizeof(T) == 4)
        if (comp)
            return launch_reg<T, true>(NI, child_src, in_n, child_index, parent_slot, n_parents, dst, W_dev, slices,
                                       st);
    return launch_reg<T, false>(NI, child_src, in_n, child_index, parent_slot, n_parents, dst, W_dev, slices, st);
}

template <typename T>
cudaError_t Generic<T>::interp(int n_b, const int* slot, const int* parent, int n_items, T* u, const T* up,
                               const T* W_dev, int accumulate, const int* block, int comp, T* slices,
                               cudaStream_t st) {
    if (n_items == 0) return cudaSuccess;
    const int NI = n_b + 1;
    if constexpr (sizeof(T) == 4)
        if (comp)
            return launch_interp<T, true>(NI, slot, parent, n_items, u, up, W_dev, accumulate, block, slices, st);
    return launch_interp<T, false>(NI, slot, parent, n_items, u, up, W_dev, accumulate, block, slices, st);
}

template struct Generic<float>;
template struct Generic<double>;

}  // namespace lgf
