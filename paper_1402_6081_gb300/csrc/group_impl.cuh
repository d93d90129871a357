// Kernels of the grouped level-0/1 convolution (group.h), templated on the
// arithmetic type and the block size; instantiated by group_f32_*.cu and
// group_f64_*.cu.
//
// A line of length S = 8 RB (RB = n_b / 2) is transformed by two register
// stages with one exchange through shared memory: with n = RB a + b and
// k = c + 8 d,
//   X[c + 8 d] = sum_b w_RB^{b d} ( w_S^{b c} sum_a w_8^{a c} x[RB a + b] ),
// a length-8 DFT over a by the thread of b (a >= 4 is padding), the twiddle,
// and a length-RB DFT over b by the thread of c.  The inverse runs the stages
// backwards and keeps a < 4.  At most 16 values per thread leave room for many
// warps, where one line per thread (64 complex values at n_b = 16) would not.
//
// Real rows y and y + n_b of a plane share one complex x transform; the y
// stage reads both spectra from the pair as it loads, so separating them
// costs no pass.
//
// Layouts.  A column is kx * S + ky.  xy[group][z / PZ][column][z % PZ]: what a
// plane kernel's CTA writes or reads is contiguous, whole cache lines per warp
// access (with a line's z values side by side it moved 32 bytes per request,
// and the requests in flight, not the bytes, bounded it: 128^3 inverse 37 us);
// a z kernel takes tens of consecutive columns of a group.  Spectra are
// [column][group][..]: the sources of a set lie near one another.
#pragma once

#include <algorithm>
#include <type_traits>

#include "lgf_internal.h"

#include "group.h"
#include "group_dft.cuh"

namespace lgf {
namespace grp {

template <typename T, int NB>
struct Dim {
    static constexpr int N = 2 * NB, S = 4 * NB, NX = S / 2 + 1, RB = NB / 2;
    static constexpr int LP = RB | 1;                  // pitch of an 8 x RB exchange: odd
    static constexpr int64_t NC = int64_t(S) * NX;     // columns
    // Plane kernels: PZ planes per CTA of 8 warps (16 for the long lines, whose
    // shared memory leaves room for one CTA per SM).  A team of 8 lanes per
    // plane takes LN lines through both stages, exchanging them in the warp's
    // own buffer (XB values).
    static constexpr int TH = RB <= 8 ? 256 : 512;
    static constexpr int LN = RB <= 8 ? 8 / RB : 1, R1 = (LN * RB + 7) / 8, R2 = LN;
    static constexpr int TEAMS(int pz) { return 4 / pz; }   // teams of a warp for the same plane
    static constexpr int XB(int pz) { return TEAMS(pz) * LN * 8 * RB * pz; }
    static constexpr size_t smem(int pz) {
        return sizeof(cx<T>) * (size_t(4 * RB) * NX * pz + size_t(TH / 32) * XB(pz) + S);
    }
    static constexpr int PZ = smem(4) <= 200 * 1024 ? 4 : smem(2) <= 200 * 1024 ? 2 : 1;
    // xy index of z 0 of a column of a group; z adds zoff(z)
    __host__ __device__ static constexpr int64_t xy(int g, int col) { return (int64_t(g) * (N / PZ) * NC + col) * PZ; }
    __host__ __device__ static constexpr int64_t zoff(int z) { return int64_t(z / PZ) * NC * PZ + z % PZ; }
    // a line's value (c, b) in the exchange buffer: the low bits of b exchanged
    // by c where RB is a power of two, so that both stages' accesses (four
    // planes times four consecutive b or c) fall into different banks
    __host__ __device__ static constexpr int at(int c, int b) {
        return c * RB + (RB == 2 ? b ^ ((c >> 1) & 1) : (RB & (RB - 1)) == 0 ? b ^ (c & 3) : b);
    }
    // products: whole columns per CTA, about 128 frequencies
    static constexpr int COLS = S >= 128 ? 1 : 128 / S;
    static constexpr int MT = (COLS * S + 31) / 32 * 32;
    // one line of the products' exchange: 8 x LP values, 8 mod 16 apart
    static constexpr int LINE = ((8 * LP + 7) / 16) * 16 + 8;
};

// The kernels of a solve follow one another with programmatic serialization: a
// kernel may start while its predecessor drains, reads its tables, and waits
// here before it touches what the predecessor writes or reads (nothing to wait
// for in a kernel launched the ordinary way).  Two rules keep that sound:
//  * What an earlier kernel of the chain writes (xy, spec, images) is read by
//    ordinary loads (ld_prev) through pointers without __restrict__: the
//    non-coherent loads that __ldg and const __restrict__ stand for need data
//    that nobody writes while the kernel lives, and this kernel lives before
//    its predecessor is done.  Tables of the plan are constant: ld, __ldg.
//  * A kernel lets its successor start only after its own wait, so at most two
//    of the chain live at once: none starts beside the last but one, which may
//    still read a buffer that the one between them rewrites (the images from
//    band to band, xy in k_gmac).
// Four launches of 4 us each: the 32^3 box of 8^3 blocks takes 14.3 us with it,
// 20.5 without (before this file's loads were ordinary ones and the signal
// stood before the wait: 13.7; larger domains measure the same either way).
__device__ __forceinline__ void let_next_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <typename T>
__device__ __forceinline__ cx<T> cmulw(cx<T> a, cx<T> w) {
    return {fma(a.x, w.x, -a.y * w.y), fma(a.x, w.y, a.y * w.x)};
}
template <typename T>
__device__ __forceinline__ cx<T> cmulc(cx<T> a, cx<T> w) {   // times the conjugate
    return {fma(a.x, w.x, a.y * w.y), fma(a.y, w.x, -a.x * w.y)};
}
template <typename T>
__device__ __forceinline__ cx<T> ld(const cx<T>* p) {
    if constexpr (sizeof(T) == 4) {
        const float2 v = __ldg(reinterpret_cast<const float2*>(p));
        return {v.x, v.y};
    } else {
        const double2 v = __ldg(reinterpret_cast<const double2*>(p));
        return {v.x, v.y};
    }
}

// ---------------------------------------------------------------------------
// Plane kernels.  Between the x and the y pass the PZ planes are in shared
// memory as Z[q RB + b][kx][plane]: the complex line of the rows y = l and
// l + n_b (l = b for q < 2, b + RB above) at kx (q even) or S - kx (q odd), so
// the y pass of one kx reads column kx of it alone and both passes exchange
// their stages within a warp; the one CTA barrier is between the passes.  Bound
// by latency at 128^3 (17 us forward, 22 us inverse; bytes alone 6.4), near the
// memory in large domains: 512^3 tori, forward 1.37 GB in 0.28 ms, inverse with
// the level-1 field 1.75 GB in 0.40 ms (5 TB/s).
template <typename T, int NB>
struct Plane {
    using D = Dim<T, NB>;
    static constexpr int RB = D::RB, S = D::S, NX = D::NX, PZ = D::PZ, TEAMS = D::TEAMS(PZ);
    static constexpr int LINES = TEAMS * D::LN;   // lines of a warp's step
    cx<T>* Z;
    cx<T>* X;          // this warp's exchange buffer
    const cx<T>* tw;
    int pz, team, lane8;
    __device__ __forceinline__ Plane(unsigned char* smem, const cx<T>* tw_dev) {
        Z = reinterpret_cast<cx<T>*>(smem);
        cx<T>* tws = Z + 4 * RB * NX * PZ;
        const int lane = int(threadIdx.x % 32);
        X = tws + S + int(threadIdx.x / 32) * D::XB(PZ);
        tw = tws;
        pz = lane % PZ;
        lane8 = (lane / PZ) % 8;
        team = lane / (PZ * 8);
        for (int i = threadIdx.x; i < S; i += D::TH) tws[i] = ld(tw_dev + i);
    }
    // round r of a stage of PER tasks per line: line within the step, task
    template <int PER>
    __device__ __forceinline__ bool task(int r, int& line, int& pos) const {
        const int i = r * 8 + lane8;
        line = team * D::LN + i / PER;
        pos = i % PER;
        return i < D::LN * PER;
    }
    __device__ __forceinline__ cx<T>& x(int line, int c, int b) { return X[(line * 8 * RB + D::at(c, b)) * PZ + pz]; }
    __device__ __forceinline__ cx<T>& z(int q, int b, int kx) { return Z[((q * RB + b) * NX + kx) * PZ + pz]; }
    // Z of the complex line l at frequency k
    __device__ __forceinline__ cx<T> line_at(int l, int k) {
        const int q = l < RB ? 0 : 2, b = l < RB ? l : l - RB;
        return 2 * k <= S ? z(q, b, k) : z(q + 1, b, S - k);
    }
    __device__ __forceinline__ void put_line(int l, int k, cx<T> v) {
        const int q = l < RB ? 0 : 2, b = l < RB ? l : l - RB;
        if (2 * k <= S) z(q, b, k) = v;
        if (2 * k >= S || k == 0) z(q + 1, b, k == 0 ? 0 : S - k) = v;
    }
};

// Forward x and y transforms of PZ planes of a group.
template <typename T, int NB>
__global__ void __launch_bounds__(Dim<T, NB>::TH, sizeof(T) == 4 && NB <= 16 ? 4 : 1)
    k_gxy_fwd(const T* __restrict__ f, const int* __restrict__ blk, const cx<T>* __restrict__ tw,
              cx<T>* __restrict__ xy) {
    using D = Dim<T, NB>;
    using P = Plane<T, NB>;
    constexpr int N = D::N, S = D::S, NX = D::NX, RB = D::RB, PZ = D::PZ, WARPS = D::TH / 32;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    P p(smem_raw, tw);
    const int g = blockIdx.x / (N / PZ), z = int(blockIdx.x % (N / PZ)) * PZ + p.pz, cz = z >= NB ? 4 : 0;
    const int warp = int(threadIdx.x / 32);
    // the plane's four blocks: x half, then y half
    int blocks[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) blocks[i] = __ldg(blk + int64_t(g) * 8 + i + cz);
    let_next_start();
    const int64_t zrow = int64_t(z - (cz ? NB : 0)) * NB * NB;
    __syncthreads();
    for (int l0 = warp * P::LINES; l0 < NB; l0 += WARPS * P::LINES) {
#pragma unroll
        for (int r = 0; r < D::R1; ++r) {
            int line, b;
            if (!p.template task<RB>(r, line, b) || l0 + line >= NB) continue;
            cx<T> x[8];
#pragma unroll
            for (int a = 0; a < 4; ++a) {   // RB a + b < n_b for a < 2
                const int64_t at = zrow + (l0 + line) * NB + (RB * (a & 1) + b);
                const int b0 = blocks[a >> 1], b1 = blocks[(a >> 1) + 2];
                x[a].x = b0 >= 0 ? __ldg(f + int64_t(b0) * (NB * NB * NB) + at) : T(0);
                x[a].y = b1 >= 0 ? __ldg(f + int64_t(b1) * (NB * NB * NB) + at) : T(0);
            }
#pragma unroll
            for (int a = 4; a < 8; ++a) x[a] = czero<T>();
            dft<8, -1, 4>(x);
#pragma unroll
            for (int c = 0; c < 8; ++c) p.x(line, c, b) = cmulc(x[c], p.tw[b * c]);
        }
        __syncwarp();
#pragma unroll
        for (int r = 0; r < D::R2; ++r) {
            int line, c;
            p.template task<8>(r, line, c);
            if (l0 + line >= NB) continue;
            cx<T> x[RB];
#pragma unroll
            for (int b = 0; b < RB; ++b) x[b] = p.x(line, c, b);
            dft<RB, -1, RB>(x);
#pragma unroll
            for (int d = 0; d < RB; ++d) p.put_line(l0 + line, c + 8 * d, x[d]);
        }
        __syncwarp();
    }
    __syncthreads();
    // y: rows y = RB a + b, from the lines b (a = 0, 2) and b + RB (a = 1, 3)
    cx<T>* out = xy + D::xy(g, 0) + D::zoff(z);
    for (int k0 = warp * P::LINES; k0 < NX; k0 += WARPS * P::LINES) {
#pragma unroll
        for (int r = 0; r < D::R1; ++r) {
            int line, b;
            if (!p.template task<RB>(r, line, b) || k0 + line >= NX) continue;
            cx<T> x[8];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const cx<T> u = p.z(2 * h, b, k0 + line), v = p.z(2 * h + 1, b, k0 + line);
                x[h] = {T(0.5) * (u.x + v.x), T(0.5) * (u.y - v.y)};
                x[h + 2] = {T(0.5) * (u.y + v.y), T(0.5) * (v.x - u.x)};
            }
#pragma unroll
            for (int a = 4; a < 8; ++a) x[a] = czero<T>();
            dft<8, -1, 4>(x);
#pragma unroll
            for (int c = 0; c < 8; ++c) p.x(line, c, b) = cmulc(x[c], p.tw[b * c]);
        }
        __syncwarp();
#pragma unroll
        for (int r = 0; r < D::R2; ++r) {
            int line, c;
            p.template task<8>(r, line, c);
            if (k0 + line >= NX) continue;
            cx<T> x[RB];
#pragma unroll
            for (int b = 0; b < RB; ++b) x[b] = p.x(line, c, b);
            dft<RB, -1, RB>(x);
            cx<T>* o = out + ((k0 + line) * S + c) * PZ;
#pragma unroll
            for (int d = 0; d < RB; ++d) o[8 * d * PZ] = x[d];
        }
        __syncwarp();
    }
}

// ---------------------------------------------------------------------------
// Forward z lines, FP64: N values in, S out; 32 consecutive columns of a group
// per CTA (16 where 32 would exceed the 48 KB of static shared memory).
template <int NB>
__host__ __device__ constexpr int z_lines() {
    return sizeof(cx<double>) * (32 * size_t(Dim<double, NB>::LINE) + Dim<double, NB>::S) <= 48 * 1024 ? 32 : 16;
}
template <int NB>
__global__ void __launch_bounds__(256) k_gz_fwd(const cx<double>* xy, const cx<double>* __restrict__ tw,
                                                cx<double>* __restrict__ spec, int n_groups) {
    using T = double;
    using D = Dim<T, NB>;
    constexpr int S = D::S, RB = D::RB, LP = D::LP, LINE = D::LINE, L = z_lines<NB>(), PER = (int(D::NC) + L - 1) / L;
    __shared__ cx<T> e[L * LINE];
    __shared__ cx<T> tws[S];
    for (int i = threadIdx.x; i < S; i += 256) tws[i] = ld(tw + i);
    wait_previous();
    let_next_start();
    __syncthreads();
    const int g = blockIdx.x / PER, c0 = blockIdx.x % PER * L, n = min(L, int(D::NC) - c0);
    for (int t = threadIdx.x; t < n * RB; t += 256) {
        const int b = t % RB, l = t / RB;
        const cx<T>* in = xy + D::xy(g, c0 + l);
        cx<T> x[8];
#pragma unroll
        for (int a = 0; a < 4; ++a) x[a] = ld_prev(in + D::zoff(RB * a + b));
#pragma unroll
        for (int a = 4; a < 8; ++a) x[a] = czero<T>();
        dft<8, -1, 4>(x);
#pragma unroll
        for (int c = 0; c < 8; ++c) e[l * LINE + c * LP + b] = cmulc(x[c], tws[b * c]);
    }
    __syncthreads();
    for (int t = threadIdx.x; t < n * 8; t += 256) {
        const int c = t % 8, l = t / 8;
        cx<T> x[RB];
#pragma unroll
        for (int b = 0; b < RB; ++b) x[b] = e[l * LINE + c * LP + b];
        dft<RB, -1, RB>(x);
        cx<T>* o = spec + (int64_t(c0 + l) * n_groups + g) * S + c;
#pragma unroll
        for (int d = 0; d < RB; ++d) o[8 * d] = x[d];
    }
}

// ---------------------------------------------------------------------------
// Products and inverse z lines, FP64: bound by the FP64 pipe (1.06 TFLOP/s;
// 128^3: 1.20 ms, 0.54 G multiply-adds in the products alone take 1.0; the
// blocks' own products 8.0 ms).  A thread holds one frequency: the 14 stored
// kernel values in registers, and per set of 2^3 target groups its 4^3 source groups,
// each loaded once and used by every target within reach (216 products).
// acc += F K, or F conj(K)
template <bool CONJ>
__device__ __forceinline__ void mac(cx<double>& s, cx<double> f, cx<double> k) {
    s.x = fma(f.x, k.x, s.x);
    s.x = fma(CONJ ? f.y : -f.y, k.y, s.x);
    s.y = fma(CONJ ? -f.x : f.x, k.y, s.y);
    s.y = fma(f.y, k.x, s.y);
}
// one source at (TX, TY, TZ) of the 4^3 (0-based) into the targets C.. within
// reach.  The kernel of offset 0 is even: a real spectrum.
template <int TX, int TY, int TZ, int C>
__device__ __forceinline__ void reach(cx<double> (&acc)[8], cx<double> f, const cx<double> (&k)[kGroupRows]) {
    if constexpr (C < 8) {
        constexpr int dx = TX - 1 - (C & 1), dy = TY - 1 - ((C >> 1) & 1), dz = TZ - 1 - (C >> 2);
        if constexpr (dx >= -1 && dx <= 1 && dy >= -1 && dy <= 1 && dz >= -1 && dz <= 1) {
            constexpr int id = dx + 3 * dy + 9 * dz;   // stored rows: id >= 0
            if constexpr (id == 0) {
                acc[C].x = fma(f.x, k[0].x, acc[C].x);
                acc[C].y = fma(f.y, k[0].x, acc[C].y);
            } else {
                mac<(id < 0)>(acc[C], f, k[id < 0 ? -id : id]);
            }
        }
        reach<TX, TY, TZ, C + 1>(acc, f, k);
    }
}

// rows (ty, tz) of four sources (-1: absent), the next row in flight
template <int R>
__device__ __forceinline__ void rows(cx<double> (&acc)[8], cx<double> (&F)[2][4], const cx<double> (&k)[kGroupRows],
                                     const int4* __restrict__ ids, const cx<double>* spec, int stride) {
    auto load = [&](cx<double>(&n)[4], int4 q) {
        n[0] = q.x >= 0 ? ld_prev(spec + int64_t(q.x) * stride) : czero<double>();
        n[1] = q.y >= 0 ? ld_prev(spec + int64_t(q.y) * stride) : czero<double>();
        n[2] = q.z >= 0 ? ld_prev(spec + int64_t(q.z) * stride) : czero<double>();
        n[3] = q.w >= 0 ? ld_prev(spec + int64_t(q.w) * stride) : czero<double>();
    };
    if constexpr (R == 0) load(F[0], __ldg(ids));
    if constexpr (R < 16) {
        if constexpr (R + 1 < 16) load(F[(R + 1) % 2], __ldg(ids + R + 1));
        const int4 q = __ldg(ids + R);
        const cx<double>(&f)[4] = F[R % 2];
        if (q.x >= 0) reach<0, R % 4, R / 4, 0>(acc, f[0], k);
        if (q.y >= 0) reach<1, R % 4, R / 4, 0>(acc, f[1], k);
        if (q.z >= 0) reach<2, R % 4, R / 4, 0>(acc, f[2], k);
        if (q.w >= 0) reach<3, R % 4, R / 4, 0>(acc, f[3], k);
        rows<R + 1>(acc, F, k, ids, spec, stride);
    }
}

template <int NB>
__global__ void __launch_bounds__(Dim<double, NB>::MT)
    k_gmac(const cx<double>* spec, const cx<double>* __restrict__ kern, const cx<double>* __restrict__ tw,
           cx<double>* __restrict__ xy, const int4* __restrict__ sets, int n_super, int per, int n_groups) {
    using T = double;
    using D = Dim<T, NB>;
    constexpr int S = D::S, RB = D::RB, LP = D::LP, COLS = D::COLS, MT = D::MT, LINE = D::LINE;
    constexpr int64_t NW = D::NC * S;
    __shared__ cx<T> e[8 * COLS * LINE];
    __shared__ cx<T> tws[S];
    for (int i = threadIdx.x; i < S; i += MT) tws[i] = ld(tw + i);
    const int col0 = blockIdx.x * COLS, tid = int(threadIdx.x);
    const int lc = tid / S, kz = tid % S;
    const bool live = lc < COLS && col0 + lc < int(D::NC);
    const int64_t w = live ? int64_t(col0) * S + tid : 0;                   // frequency
    const int64_t ws = live ? int64_t(col0 + lc) * n_groups * S + kz : 0;   // of group 0 in spec
    cx<T> k[kGroupRows];
#pragma unroll
    for (int i = 0; i < kGroupRows; ++i) k[i] = ld(kern + int64_t(i) * NW + w);
    wait_previous();
    let_next_start();
    const int s1 = min(n_super, int(blockIdx.y + 1) * per);
    for (int s = blockIdx.y * per; s < s1; ++s) {
        const int4* ids = sets + int64_t(s) * (kSetInts / 4);
        const int* targets = reinterpret_cast<const int*>(ids + 16);
        cx<T> acc[8], F[2][4];
#pragma unroll
        for (int c = 0; c < 8; ++c) acc[c] = czero<T>();
        rows<0>(acc, F, k, ids, spec + ws, S);
        __syncthreads();   // the previous set's lines have been read (and tws is there)
        if (lc < COLS) {
#pragma unroll
            for (int c = 0; c < 8; ++c) e[(c * COLS + lc) * LINE + (kz % 8) * LP + kz / 8] = acc[c];
        }
        __syncthreads();
        // inverse z: the thread of (line, c) over d, in place
        for (int t = tid; t < 8 * COLS * 8; t += MT) {
            const int c = t % 8, l = t / 8;
            cx<T> x[RB];
            cx<T>* p = e + l * LINE + c * LP;
#pragma unroll
            for (int d = 0; d < RB; ++d) x[d] = p[d];
            dft<RB, 1, RB>(x);
#pragma unroll
            for (int b = 0; b < RB; ++b) p[b] = cmulw(x[b], tws[b * c]);
        }
        __syncthreads();
        // the thread of (line, b) over c -> z = RB a + b, a < 4
        for (int t = tid; t < 8 * COLS * RB; t += MT) {
            const int b = t % RB, l = t / RB, c = l / COLS, col = col0 + l % COLS;
            const int g = __ldg(targets + c);
            if (g < 0 || col >= int(D::NC)) continue;
            cx<T> x[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) x[i] = e[l * LINE + i * LP + b];
            dft<8, 1, 8>(x);
            cx<T>* o = xy + D::xy(g, col);
#pragma unroll
            for (int a = 0; a < 4; ++a) o[D::zoff(RB * a + b)] = x[a];
        }
    }
}

// ---------------------------------------------------------------------------
// FP32: the z lines are transformed into images, a band of columns at a time,
// and the products of the band read them from L2.  A thread holds two
// frequencies d, d + 1 of a line's row c, so that its packed operands (re, re)
// and (im, im) are loaded as they are.
//
// A line's image, in 8-byte units: row c holds RP = 2 U values (U pairs; an
// odd RB leaves the last half unused).  Between the two stages value (c, b)
// is complex; the transformed row holds, per pair j, the 16 bytes (X[2j].re,
// X[2j+1].re, X[2j].im, X[2j+1].im).  Each row belongs to one thread of the
// second stage, which rewrites it in place.  The low bits of the position are
// exchanged by c and lines are 8 mod 16 units apart: no bank conflicts at
// n_b = 16.
template <int NB>
struct ColDim {
    using D = Dim<float, NB>;
    static constexpr int S = D::S, RB = D::RB, U = (RB + 1) / 2, RP = 2 * U;
    static constexpr int COLS = S <= 24 ? (S == 16 ? 4 : 2) : S == 32 ? 2 : 1;
    static constexpr int SLOTS = 8 * U;                              // frequency pairs of a line
    static constexpr int SL = (COLS * SLOTS + 31) / 32;              // warps per unit
    static constexpr int LINE = ((8 * RP + 7) / 16) * 16 + 8;
    __host__ __device__ static constexpr int swz(int c) {
        return U == 8 ? c : U == 4 ? c >> 1 : U == 2 ? c >> 2 : 0;
    }
    __host__ __device__ static constexpr int at(int c, int b) { return c * RP + (b ^ swz(c)); }      // value
    __host__ __device__ static constexpr int pair(int c, int j) { return c * RP + 2 * (j ^ swz(c)); }   // pair
    static constexpr int IMG = 8 * RP;                               // values of an image in memory
    static constexpr int TH = 128, UNITS = TH / 32 / SL;             // sets in flight
};

__device__ __forceinline__ uint64_t pk(float lo, float hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void fma2(uint64_t& d, uint64_t a, uint64_t b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}
struct Acc2 { uint64_t re, im; };   // two frequencies
__device__ __forceinline__ uint64_t neg2(uint64_t a) {
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(0xbf800000bf800000ull));
    return r;
}
// Operation OP of acc += F K (F conj(K) for the offsets stored conjugated) for
// the source at (TX, TY, TZ) of the 4^3 and every target C within reach.  f =
// (re, im, -re, -im) pairs.  The kernel of offset 0 is even: a real spectrum.
template <int OP, int TX, int TY, int TZ, int C>
__device__ __forceinline__ void reach2(Acc2 (&acc)[8], const uint64_t (&f)[4], const uint64_t (&kx)[kGroupRows],
                                       const uint64_t (&ky)[kGroupRows]) {
    if constexpr (C < 8) {
        constexpr int dx = TX - 1 - (C & 1), dy = TY - 1 - ((C >> 1) & 1), dz = TZ - 1 - (C >> 2);
        if constexpr (dx >= -1 && dx <= 1 && dy >= -1 && dy <= 1 && dz >= -1 && dz <= 1) {
            constexpr int id = dx + 3 * dy + 9 * dz, row = id < 0 ? -id : id;   // stored rows: id >= 0
            if constexpr (OP == 0) fma2(acc[C].re, f[0], kx[row]);
            if constexpr (OP == 1) fma2(acc[C].im, f[1], kx[row]);
            if constexpr (OP == 2 && id != 0) fma2(acc[C].re, id < 0 ? f[1] : f[3], ky[row]);
            if constexpr (OP == 3 && id != 0) fma2(acc[C].im, id < 0 ? f[2] : f[0], ky[row]);
        }
        reach2<OP, TX, TY, TZ, C + 1>(acc, f, kx, ky);
    }
}
// one operation of a row's four sources: neighbouring instructions belong to
// different sums
template <int OP, int I>
__device__ __forceinline__ void row_op(Acc2 (&acc)[8], const uint64_t (&f)[4][4], const uint64_t (&kx)[kGroupRows],
                                       const uint64_t (&ky)[kGroupRows]) {
    reach2<OP, 0, I % 4, I / 4, 0>(acc, f[0], kx, ky);
    reach2<OP, 1, I % 4, I / 4, 0>(acc, f[1], kx, ky);
    reach2<OP, 2, I % 4, I / 4, 0>(acc, f[2], kx, ky);
    reach2<OP, 3, I % 4, I / 4, 0>(acc, f[3], kx, ky);
}

// Rows (ty, tz) of four sources; ids: their groups, an absent one the line of
// zeros behind the last group; a row of four absent ones is skipped (ids and
// branch are the same for the whole warp).  Two rows are in flight while one
// is used.
constexpr int kAhead = 2;
struct Row { ulonglong2 v[4]; };
template <int IMG>
__device__ __forceinline__ Row load_row(const int4 q, const cx<float>* base) {
    // loaded as the 64-bit pairs that are used: a move would wait for the load
    auto get = [&](int g) { return ld_prev(reinterpret_cast<const ulonglong2*>(base + int64_t(g) * IMG)); };
    return {{get(q.x), get(q.y), get(q.z), get(q.w)}};
}
template <int I, int IMG>
__device__ __forceinline__ void sources2(Acc2 (&acc)[8], const uint64_t (&kx)[kGroupRows],
                                         const uint64_t (&ky)[kGroupRows], const int4* ids, unsigned rows,
                                         const cx<float>* base, Row (&ring)[kAhead + 1]) {
    if constexpr (I < 16) {
        if constexpr (I + kAhead < 16)
            if (rows >> (I + kAhead) & 1) ring[(I + kAhead) % (kAhead + 1)] = load_row<IMG>(ids[I + kAhead], base);
        if (rows >> I & 1) {
            const Row& cur = ring[I % (kAhead + 1)];
            uint64_t f[4][4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                f[k][0] = cur.v[k].x;
                f[k][1] = cur.v[k].y;
                f[k][2] = neg2(cur.v[k].x);
                f[k][3] = neg2(cur.v[k].y);
            }
            row_op<0, I>(acc, f, kx, ky);
            row_op<1, I>(acc, f, kx, ky);
            row_op<2, I>(acc, f, kx, ky);
            row_op<3, I>(acc, f, kx, ky);
        }
        sources2<I + 1, IMG>(acc, kx, ky, ids, rows, base, ring);
    }
}

// The z lines go through both stages within a warp (no CTA barrier): a team
// of TL lanes takes LN lines at a time, R1 rounds of the first stage's RB
// tasks a line and R2 rounds of the second stage's eight.
template <int NB>
struct Team {
    static constexpr int RB = ColDim<NB>::RB;
    static constexpr int TL = RB <= 8 ? 8 : 16, LN = RB <= 8 ? 8 / RB : 2;
    static constexpr int R1 = (LN * RB + TL - 1) / TL, R2 = LN * 8 / TL;
    static constexpr int WARP_LINES = 32 / TL * LN;   // lines of a warp's step
};
// task of a round: line within the warp's step and position (b or c), -1: none
template <int NB, int PER>
__device__ __forceinline__ bool team_task(int round, int& line, int& pos) {
    using M = Team<NB>;
    const int lane = int(threadIdx.x % 32), i = round * M::TL + lane % M::TL;
    line = lane / M::TL * M::LN + i / PER;
    pos = i % PER;
    return i < M::LN * PER;
}

// the twiddles w_S^{p c}, c < 8, of this lane's position p in a round, where
// they are the same for every round (one line per team); else read per use
template <int NB, int PER>
struct TeamTw {
    static constexpr bool FIXED = Team<NB>::LN == 1;
    cx<float> w[FIXED ? PER : 1];
    const cx<float>* tws;
    // j-th factor of position p
    __device__ __forceinline__ TeamTw(const cx<float>* t, int p) : tws(t) {
        if constexpr (FIXED) {
#pragma unroll
            for (int j = 1; j < PER; ++j) w[j] = t[p * j];
        }
    }
    __device__ __forceinline__ cx<float> get(int p, int j) const {
        if constexpr (FIXED) return w[j];
        else return tws[p * j];
    }
};

// forward z lines first, first + step, ...: a warp's steps of WARP_LINES lines
// below n; value z of line l is get(l, z); the images go to e, LINE apart.  UN
// steps run interleaved.
template <int NB, int UN, typename Get>
__device__ __forceinline__ void z_forward(cx<float>* e, const cx<float>* tws, int first, int step, int n, Get&& get) {
    using C = ColDim<NB>;
    using M = Team<NB>;
    constexpr int RB = C::RB, LINE = C::LINE;
    int l0, p0;
    team_task<NB, RB>(0, l0, p0);
    const TeamTw<NB, 8> w(tws, p0);
    for (int base = first; base < n; base += step * UN) {
        cx<float> x[UN * M::R1][8];
#pragma unroll
        for (int r = 0; r < UN * M::R1; ++r) {
            int l, b;
            const bool ok = team_task<NB, RB>(r % M::R1, l, b);
            l += base + r / M::R1 * step;
#pragma unroll
            for (int a = 0; a < 4; ++a) x[r][a] = ok && l < n ? get(l, RB * a + b) : czero<float>();
        }
#pragma unroll
        for (int r = 0; r < UN * M::R1; ++r) {
            int l, b;
            const bool ok = team_task<NB, RB>(r % M::R1, l, b);
            l += base + r / M::R1 * step;
#pragma unroll
            for (int a = 4; a < 8; ++a) x[r][a] = czero<float>();
            dft<8, -1, 4>(x[r]);
            if (ok && l < n) {
                e[l * LINE + C::at(0, b)] = x[r][0];
#pragma unroll
                for (int c = 1; c < 8; ++c) e[l * LINE + C::at(c, b)] = cmulc(x[r][c], w.get(b, c));
            }
        }
        __syncwarp();
        cx<float> y[UN * M::R2][RB];
#pragma unroll
        for (int r = 0; r < UN * M::R2; ++r) {
            int l, c;
            team_task<NB, 8>(r % M::R2, l, c);
            l += base + r / M::R2 * step;
#pragma unroll
            for (int b = 0; b < RB; ++b) y[r][b] = l < n ? e[l * LINE + C::at(c, b)] : czero<float>();
        }
#pragma unroll
        for (int r = 0; r < UN * M::R2; ++r) {
            int l, c;
            team_task<NB, 8>(r % M::R2, l, c);
            l += base + r / M::R2 * step;
            dft<RB, -1, RB>(y[r]);
            if (l < n) {
#pragma unroll
                for (int j = 0; j < C::U; ++j) {
                    const cx<float> u = y[r][2 * j];
                    const cx<float> v = 2 * j + 1 < RB ? y[r][2 * j + 1 < RB ? 2 * j + 1 : 0] : czero<float>();
                    *reinterpret_cast<float4*>(e + l * LINE + C::pair(c, j)) = make_float4(u.x, v.x, u.y, v.y);
                }
            }
        }
    }
}

// inverse z lines, the images e (LINE apart) rewritten on the way; x[a] = value
// z = RB a + b of line l, a < 4, goes to put(l, b, x)
template <int NB, int UN, typename Put>
__device__ __forceinline__ void z_inverse(cx<float>* e, const cx<float>* tws, int first, int step, int n, Put&& put) {
    using C = ColDim<NB>;
    using M = Team<NB>;
    constexpr int RB = C::RB, U = C::U, LINE = C::LINE;
    int l0, p0;
    team_task<NB, 8>(0, l0, p0);
    const TeamTw<NB, RB> w(tws, p0);
    for (int base = first; base < n; base += step * UN) {
        cx<float> y[UN * M::R2][RB];
#pragma unroll
        for (int r = 0; r < UN * M::R2; ++r) {
            int l, c;
            team_task<NB, 8>(r % M::R2, l, c);
            l += base + r / M::R2 * step;
#pragma unroll
            for (int j = 0; j < U; ++j) {
                const float4 v = l < n ? *reinterpret_cast<const float4*>(e + l * LINE + C::pair(c, j))
                                       : make_float4(0.f, 0.f, 0.f, 0.f);
                y[r][2 * j] = {v.x, v.z};
                if (2 * j + 1 < RB) y[r][2 * j + 1 < RB ? 2 * j + 1 : 0] = {v.y, v.w};
            }
        }
#pragma unroll
        for (int r = 0; r < UN * M::R2; ++r) {
            int l, c;
            team_task<NB, 8>(r % M::R2, l, c);
            l += base + r / M::R2 * step;
            dft<RB, 1, RB>(y[r]);
            if (l < n) {
                e[l * LINE + C::at(c, 0)] = y[r][0];
#pragma unroll
                for (int b = 1; b < RB; ++b) e[l * LINE + C::at(c, b)] = cmulw(y[r][b], w.get(c, b));
            }
        }
        __syncwarp();
        cx<float> x[UN * M::R1][8];
#pragma unroll
        for (int r = 0; r < UN * M::R1; ++r) {
            int l, b;
            const bool ok = team_task<NB, RB>(r % M::R1, l, b);
            l += base + r / M::R1 * step;
#pragma unroll
            for (int c = 0; c < 8; ++c) x[r][c] = ok && l < n ? e[l * LINE + C::at(c, b)] : czero<float>();
        }
#pragma unroll
        for (int r = 0; r < UN * M::R1; ++r) {
            int l, b;
            const bool ok = team_task<NB, RB>(r % M::R1, l, b);
            l += base + r / M::R1 * step;
            dft<8, 1, 8>(x[r]);
            if (ok && l < n) put(l, b, x[r]);
        }
    }
}

// Products and inverse z lines of a band of columns.  A unit (a warp, or two
// where a column has more than 32 pairs of frequencies) keeps the kernel rows
// of its frequencies and takes sets of 2^3 target groups: 64 sources, 216
// products, the sums to shared memory, eight lines back.  Units share nothing
// but L1, which holds the sources that neighbouring sets have in common, so
// there is no CTA barrier.  Bound by the latency of the source loads (12 warps
// of 168 registers per SM, FMA pipe 40% busy); 128^3 box: 2 bands of 31 us, with
// the images 93 us where the blocks' own products take 206 us; 512^3 tori (2112
// groups) 3.6 ms against 7.6 ms.  Sources staged per tile of sets in shared
// memory measured the same for large domains (its barriers cost what the
// loads' latency does here), more loads in flight with fewer warps too.
//   img   [band column][n_groups + 1][IMG], the last line of a column zero
//   kern  [column][row][pair of frequencies] as (re, re, im, im)
//   per   sets per unit of a CTA
template <int NB>
__global__ void __launch_bounds__(ColDim<NB>::TH, 3)
    k_gprod(const cx<float>* img, const float4* __restrict__ kern, const cx<float>* __restrict__ tw,
            cx<float>* __restrict__ out, const int4* __restrict__ sets, int n_sets, int per, int n_groups,
            int first_col) {
    using C = ColDim<NB>;
    using D = Dim<float, NB>;
    constexpr int S = D::S, COLS = C::COLS, LINE = C::LINE, TH = C::TH, UW = C::SL, VEC = kSetInts / 4;
    __shared__ __align__(16) cx<float> lines[C::UNITS * 8 * COLS * LINE];   // [unit][target][column][LINE]
    __shared__ cx<float> tws[S];
    __shared__ int4 recs[TH / 32][2][VEC];
    const int tid = int(threadIdx.x), warp = tid / 32, lane = tid % 32, unit = warp / UW;
    for (int i = tid; i < S; i += TH) tws[i] = ld(tw + i);
    __syncthreads();
    // this thread's pair of frequencies: column, row and pair of a line
    const int slot = (warp % UW) * 32 + lane, live = slot < COLS * C::SLOTS, fl = live ? slot : 0;
    const int fcol = fl / C::SLOTS, fpair = fl % C::SLOTS, fpos = C::pair(fpair / C::U, fpair % C::U);
    const int bc = int(blockIdx.x) * COLS;                    // column in the band
    const int64_t col0 = first_col + bc;
    uint64_t kx[kGroupRows], ky[kGroupRows];
    {
        const float4* kp = kern + (col0 + fcol) * (kGroupRows * C::SLOTS) + fpair;
#pragma unroll
        for (int i = 0; i < kGroupRows; ++i) {
            const float4 v = __ldg(kp + i * C::SLOTS);
            kx[i] = pk(v.x, v.y);
            ky[i] = pk(v.z, v.w);
        }
    }
    const cx<float>* base = img + int64_t(bc + fcol) * (n_groups + 1) * C::IMG + fpos;
    cx<float>* mine = lines + unit * 8 * COLS * LINE;
    auto meet = [&] {   // the unit's warps
        if constexpr (UW > 1) asm volatile("bar.sync %0, %1;" ::"r"(1 + unit), "n"(UW * 32) : "memory");
        else __syncwarp();
    };
    int s = int(blockIdx.y) * per * C::UNITS + unit;
    const int end = min(n_sets, int(blockIdx.y + 1) * per * C::UNITS);
    int4 next = lane < VEC && s < end ? __ldg(sets + int64_t(s) * VEC + lane) : make_int4(0, 0, 0, 0);
    wait_previous();
    let_next_start();
    // the record of a set and its first rows come while the set before it is
    // transformed back
    Row ring[kAhead + 1];
    auto begin = [&](int buf) {
        if (lane < VEC) recs[warp][buf][lane] = next;
        __syncwarp();
#pragma unroll
        for (int i = 0; i < kAhead; ++i) ring[i] = load_row<C::IMG>(recs[warp][buf][i], base);
    };
    if (s < end) begin(0);
    for (int buf = 0; s < end; s += C::UNITS, buf ^= 1) {
        const bool more = s + C::UNITS < end;
        if (more && lane < VEC) next = __ldg(sets + int64_t(s + C::UNITS) * VEC + lane);
        const int4* ids = recs[warp][buf];
        const unsigned rows = unsigned(ids[18].x);
        Acc2 acc[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) acc[c] = {0ull, 0ull};
        sources2<0, C::IMG>(acc, kx, ky, ids, rows, base, ring);
        if (live) {
#pragma unroll
            for (int c = 0; c < 8; ++c)
                *reinterpret_cast<ulonglong2*>(mine + (c * COLS + fcol) * LINE + fpos) = make_ulonglong2(acc[c].re, acc[c].im);
        }
        if (more) begin(buf ^ 1);
        meet();
        const int* targets = reinterpret_cast<const int*>(ids + 16);
        z_inverse<NB, 2 / UW>(mine, tws, (warp % UW) * Team<NB>::WARP_LINES, UW * Team<NB>::WARP_LINES, 8 * COLS,
                              [&](int l, int b, const cx<float>(&x)[8]) {
                                  const int g = targets[l / COLS];
                                  if (g < 0) return;
                                  cx<float>* o = out + D::xy(g, int(col0) + l % COLS);
#pragma unroll
                                  for (int a = 0; a < 4; ++a) o[D::zoff(D::RB * a + b)] = x[a];
                              });
        meet();
    }
}

// Forward z lines of a band of columns of every group, as images
// [band column][n_groups + 1][IMG] (the last line of a column stays zero); a
// CTA transforms some tens of consecutive columns of a group.
template <int NB>
__host__ __device__ constexpr int image_lines() { return ColDim<NB>::LINE <= 72 ? 64 : 32; }
template <int NB>
__global__ void __launch_bounds__(256) k_gz_image(const cx<float>* xy, const cx<float>* __restrict__ tw,
                                                  cx<float>* __restrict__ img, int first_col, int band_cols,
                                                  int n_groups) {
    using C = ColDim<NB>;
    using D = Dim<float, NB>;
    constexpr int L = image_lines<NB>(), LINE = C::LINE, S = D::S, IMG = C::IMG;
    __shared__ __align__(16) cx<float> e[L * LINE];
    __shared__ cx<float> tws[S];
    const int per = (band_cols + L - 1) / L, g = blockIdx.x / per, c0 = blockIdx.x % per * L, n = min(L, band_cols - c0);
    for (int i = threadIdx.x; i < S; i += 256) tws[i] = ld(tw + i);
    wait_previous();
    let_next_start();
    __syncthreads();
    const cx<float>* in = xy + D::xy(g, first_col + c0);
    z_forward<NB, 2>(e, tws, int(threadIdx.x / 32) * Team<NB>::WARP_LINES, 8 * Team<NB>::WARP_LINES, n,
                     [&](int l, int z) { return ld_prev(in + l * D::PZ + D::zoff(z)); });
    __syncthreads();
    for (int i = threadIdx.x; i < n * (IMG / 2); i += 256) {
        const int l = i / (IMG / 2), v = i % (IMG / 2);
        reinterpret_cast<float4*>(img + (int64_t(c0 + l) * (n_groups + 1) + g) * IMG)[v] =
            *reinterpret_cast<const float4*>(e + l * LINE + 2 * v);
    }
}

// ---------------------------------------------------------------------------
// Inverse y and x transforms of PZ planes of a group into its blocks.
template <typename T, int NB>
__global__ void __launch_bounds__(Dim<T, NB>::TH, sizeof(T) == 4 && NB <= 16 ? 4 : 1)
    k_gxy_inv(const cx<T>* xy, const int* __restrict__ blk, const int* __restrict__ aux,
              const cx<T>* __restrict__ tw, T* __restrict__ u, const T* __restrict__ add, int add_n,
              int64_t add_stride) {
    using D = Dim<T, NB>;
    using P = Plane<T, NB>;
    constexpr int N = D::N, S = D::S, NX = D::NX, RB = D::RB, PZ = D::PZ, WARPS = D::TH / 32;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    P p(smem_raw, tw);
    const int g = blockIdx.x / (N / PZ), z = int(blockIdx.x % (N / PZ)) * PZ + p.pz, cz = z >= NB ? 4 : 0;
    const int warp = int(threadIdx.x / 32), zl = z - (cz ? NB : 0);
    __syncthreads();
    wait_previous();
    // y: ky = c + 8 d -> y = RB a + b; the rows y and y + n_b (half spectra A
    // and B of real rows) as one complex line A + i B
    const cx<T>* in = xy + D::xy(g, 0) + D::zoff(z);
    for (int k0 = warp * P::LINES; k0 < NX; k0 += WARPS * P::LINES) {
#pragma unroll
        for (int r = 0; r < D::R2; ++r) {
            int line, c;
            p.template task<8>(r, line, c);
            if (k0 + line >= NX) continue;
            const cx<T>* q = in + ((k0 + line) * S + c) * PZ;
            cx<T> x[RB];
#pragma unroll
            for (int d = 0; d < RB; ++d) x[d] = ld_prev(q + 8 * d * PZ);
            dft<RB, 1, RB>(x);
#pragma unroll
            for (int b = 0; b < RB; ++b) p.x(line, c, b) = cmulw(x[b], p.tw[b * c]);
        }
        __syncwarp();
#pragma unroll
        for (int r = 0; r < D::R1; ++r) {
            int line, b;
            if (!p.template task<RB>(r, line, b) || k0 + line >= NX) continue;
            const int kx = k0 + line;
            cx<T> x[8];
#pragma unroll
            for (int c = 0; c < 8; ++c) x[c] = p.x(line, c, b);
            dft<8, 1, 8>(x);
            const bool edge = kx == 0 || 2 * kx == S;   // real for a real row
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                cx<T> A = x[h], B = x[h + 2];
                if (edge) A.y = B.y = T(0);
                p.z(2 * h, b, kx) = {A.x - B.y, A.y + B.x};
                p.z(2 * h + 1, b, kx) = {A.x + B.y, B.x - A.y};
            }
        }
        __syncwarp();
    }
    __syncthreads();
    // x: the rows y = l (real part) and l + n_b (imaginary part)
    for (int l0 = warp * P::LINES; l0 < NB; l0 += WARPS * P::LINES) {
#pragma unroll
        for (int r = 0; r < D::R2; ++r) {
            int line, c;
            p.template task<8>(r, line, c);
            if (l0 + line >= NB) continue;
            cx<T> x[RB];
#pragma unroll
            for (int d = 0; d < RB; ++d) x[d] = p.line_at(l0 + line, c + 8 * d);
            dft<RB, 1, RB>(x);
#pragma unroll
            for (int b = 0; b < RB; ++b) p.x(line, c, b) = cmulw(x[b], p.tw[b * c]);
        }
        __syncwarp();
#pragma unroll
        for (int r = 0; r < D::R1; ++r) {
            int line, b;
            if (!p.template task<RB>(r, line, b) || l0 + line >= NB) continue;
            const int l = l0 + line;
            cx<T> x[8];
#pragma unroll
            for (int c = 0; c < 8; ++c) x[c] = p.x(line, c, b);
            dft<8, 1, 8>(x);
#pragma unroll
            for (int ch = 0; ch < 4; ++ch) {   // child (x, y) of the plane
                const int id = ch + cz;
                const int bi = __ldg(blk + int64_t(g) * 8 + id);
                if (bi < 0) continue;
                const int sl = add != nullptr ? __ldg(aux + int64_t(g) * 8 + id) : -1;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int a = 2 * (ch & 1) + h, xl = RB * h + b;
                    T v = (ch & 2) ? x[a].y : x[a].x;
                    if (sl >= 0) v += __ldg(add + int64_t(sl) * add_stride + (int64_t(zl) * add_n + l) * add_n + xl);
                    u[int64_t(bi) * (NB * NB * NB) + (int64_t(zl) * NB + l) * NB + xl] = v;
                }
            }
        }
        __syncwarp();
    }
}

}  // namespace grp

// early: behind the previous kernel of the stream with programmatic serialization
template <typename... P, typename... A>
static cudaError_t launch_after(void (*kernel)(P...), dim3 grid, int block, size_t smem, cudaStream_t st, bool early,
                                A... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(unsigned(block));
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = early ? 1 : 0;
    return launched(cudaLaunchKernelEx(&cfg, kernel, P(args)...));
}

template <typename T, int NB>
cudaError_t GroupSize<T, NB>::forward(const GroupTables& g, const T* f, void* xy, void* spec, int early,
                                      cudaStream_t st) {
    using D = grp::Dim<T, NB>;
    constexpr size_t smem = D::smem(D::PZ);
    auto k = grp::k_gxy_fwd<T, NB>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
    if (e != cudaSuccess || g.n_groups == 0) return e;
    auto* p = static_cast<dev::cx<T>*>(xy);
    const auto* tw = static_cast<const dev::cx<T>*>(g.tw);
    k<<<unsigned(g.n_groups * (D::N / D::PZ)), D::TH, smem, st>>>(f, g.blk, tw, p);
    if ((e = launched()) != cudaSuccess || group_banded<T>()) return e;
    if constexpr (!group_banded<T>()) {
        constexpr int L = grp::z_lines<NB>(), per = (int(D::NC) + L - 1) / L;
        e = launch_after(grp::k_gz_fwd<NB>, dim3(unsigned(g.n_groups * per)), 256, 0, st, early, p, tw,
                         static_cast<dev::cx<T>*>(spec), g.n_groups);
    }
    return e;
}

template <typename T, int NB>
cudaError_t GroupSize<T, NB>::products(const GroupTables& g, const void* in, const void* kern, void* out, int early,
                                       cudaStream_t st) {
    using D = grp::Dim<T, NB>;
    const auto* src = static_cast<const dev::cx<T>*>(in);
    const auto* kp = static_cast<const dev::cx<T>*>(kern);
    const auto* tw = static_cast<const dev::cx<T>*>(g.tw);
    auto* dst = static_cast<dev::cx<T>*>(out);
    if (g.n_super == 0) return cudaSuccess;
    if constexpr (group_banded<T>()) {
        using C = grp::ColDim<NB>;
        const int nc = int(D::NC), sets_at_once = C::UNITS;
        auto* img = static_cast<dev::cx<float>*>(g.images);
        cudaError_t e = cudaSuccess;
        for (int c0 = 0; c0 < nc; c0 += g.band_cols) {
            const int n = std::min(g.band_cols, nc - c0), cols = n / C::COLS;
            constexpr int L = grp::image_lines<NB>();
            e = launch_after(grp::k_gz_image<NB>, dim3(unsigned(g.n_groups * ((n + L - 1) / L))), 256, 0, st, early, src,
                             tw, img, c0, n, g.n_groups);
            if (e != cudaSuccess) return e;
            // sets per unit: one load of the kernel rows for all of them,
            // while the launch keeps some waves of CTAs
            int per = 1;
            auto chunks = [&](int p) { return (g.n_super + p * sets_at_once - 1) / (p * sets_at_once); };
            while (per * sets_at_once < g.n_super && (int64_t(cols) * chunks(2 * per) >= 4 * 3 * 152 || chunks(per) > 65535))
                per *= 2;
            e = launch_after(grp::k_gprod<NB>, dim3(unsigned(cols), unsigned(chunks(per))), C::TH, 0, st, early, img,
                             static_cast<const float4*>(kern), tw, dst, g.sets, g.n_super, per, g.n_groups, c0);
            if (e != cudaSuccess) return e;
        }
    } else {
        // sets of targets per CTA: one kernel-table load for all of them, while
        // the launch keeps about eight waves of CTAs
        const unsigned cols = unsigned((D::NC + D::COLS - 1) / D::COLS);
        int per = 1;
        auto chunks = [&](int p) { return (g.n_super + p - 1) / p; };
        while (per < g.n_super && (int64_t(cols) * chunks(2 * per) >= 8 * 152 * 4 || chunks(per) > 65535)) per *= 2;
        const dim3 grid(cols, unsigned(chunks(per)));
        return launch_after(grp::k_gmac<NB>, grid, D::MT, 0, st, early, src, kp, tw, dst, g.sets, g.n_super, per,
                            g.n_groups);
    }
    return cudaSuccess;
}

template <typename T, int NB>
cudaError_t GroupSize<T, NB>::inverse(const GroupTables& g, const void* xy, T* u, const T* add, int add_n,
                                      int64_t add_stride, int early, cudaStream_t st) {
    using D = grp::Dim<T, NB>;
    constexpr size_t smem = D::smem(D::PZ);
    auto k = grp::k_gxy_inv<T, NB>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
    if (e != cudaSuccess || g.n_groups == 0) return e;
    return launch_after(k, dim3(unsigned(g.n_groups * (D::N / D::PZ))), D::TH, smem, st, early,
                        static_cast<const dev::cx<T>*>(xy), g.blk, g.aux, static_cast<const dev::cx<T>*>(g.tw), u, add,
                        add_n, add_stride);
}

}  // namespace lgf
