// In-register DFTs of the grouped level-0 transforms (group_impl.cuh), every
// length 2 .. 16, with compile-time twiddles.
//
// The roots of unity are constant expressions (Taylor series of sin and cos on
// [0, pi/4] in FP64, octant symmetry), so after unrolling they are immediate
// operands and need no table.  A composite length is a decimation in time
// n = R m with R the radices 4, 2 or the smallest odd prime; an odd prime pairs
// the terms r and R - r, which share their cosines and sines.  NZ is the number
// of leading inputs that may be non-zero: all-zero branches are dropped.
#pragma once

#include <cuda_runtime.h>

#include "fft_device.cuh"   // cx<T>

namespace lgf {
namespace grp {

using dev::cx;
using dev::czero;
using dev::ld_prev;

// ---- exp(2 pi i j / n) as constant expressions ----
// sin and cos of a in [0, pi/4]: 14 terms of the series, below 1e-19
LGF_HD constexpr double taylor_sin(double a) {
    double s = 0, t = a;
    for (int k = 1; k < 28; k += 2) {
        s += t;
        t *= -a * a / double((k + 1) * (k + 2));
    }
    return s;
}
LGF_HD constexpr double taylor_cos(double a) {
    double s = 0, t = 1;
    for (int k = 0; k < 28; k += 2) {
        s += t;
        t *= -a * a / double((k + 1) * (k + 2));
    }
    return s;
}
constexpr double kPi = 3.14159265358979323846;
// cos(2 pi j / n), 0 <= j < n, by symmetry from [0, n/8]
LGF_HD constexpr double root_cos(int j, int n) {
    if (2 * j > n) j = n - j;                       // cos is even
    if (4 * j > n) return -root_cos(n - 2 * j, 2 * n);   // cos(pi - a) = -cos(a)
    // a = 2 pi j / n in [0, pi/2]
    return 8 * j <= n ? taylor_cos(2 * kPi * j / n) : taylor_sin(kPi * (n - 4 * j) / (2.0 * n));
}
LGF_HD constexpr double root_sin(int j, int n) {
    if (2 * j > n) return -root_sin(n - j, n);
    if (4 * j > n) return root_sin(n - 2 * j, 2 * n);    // sin(pi - a) = sin(a)
    return 8 * j <= n ? taylor_sin(2 * kPi * j / n) : taylor_cos(kPi * (n - 4 * j) / (2.0 * n));
}

// a * exp(SIGN 2 pi i j / n)
template <int N, int J, int SIGN, typename T>
__device__ __forceinline__ cx<T> rot(cx<T> a) {
    constexpr int j = J % N;
    if constexpr (j == 0) return a;
    else if constexpr (2 * j == N) return {-a.x, -a.y};
    else if constexpr (4 * j == N) return {T(-SIGN) * a.y, T(SIGN) * a.x};
    else if constexpr (4 * j == 3 * N) return {T(SIGN) * a.y, T(-SIGN) * a.x};
    else {
        constexpr T c = T(root_cos(j, N)), s = T(SIGN * root_sin(j, N));
        return {fma(a.x, c, -a.y * s), fma(a.x, s, a.y * c)};
    }
}

__host__ __device__ constexpr int dft_radix(int n) {
    if (n % 4 == 0) return 4;
    if (n % 2 == 0) return 2;
    for (int p = 3; p < n; p += 2)
        if (n % p == 0) return p;
    return n;
}
__host__ __device__ constexpr int imin(int a, int b) { return a < b ? a : b; }

// outputs k and R - k of an odd prime radix, k >= K, from the sums s and
// differences d of the inputs r and R - r
template <int R, int RNZ, int K, int r, int H, typename T>
__device__ __forceinline__ void odd_terms(cx<T>& p, cx<T>& q, const cx<T> (&s)[H], const cx<T> (&d)[H]) {
    if constexpr (r <= H && r < RNZ) {
        constexpr T c = T(root_cos(r * K % R, R)), w = T(root_sin(r * K % R, R));
        p.x = fma(s[r - 1].x, c, p.x);
        p.y = fma(s[r - 1].y, c, p.y);
        q.x = fma(d[r - 1].x, w, q.x);
        q.y = fma(d[r - 1].y, w, q.y);
        odd_terms<R, RNZ, K, r + 1>(p, q, s, d);
    }
}
template <int R, int SIGN, int RNZ, int K, int H, typename T>
__device__ __forceinline__ void odd_outputs(cx<T> (&z)[R], const cx<T> (&s)[H], const cx<T> (&d)[H], cx<T> z0) {
    if constexpr (K <= H) {
        cx<T> p = z0, q = czero<T>();
        odd_terms<R, RNZ, K, 1>(p, q, s, d);
        z[K] = {p.x - T(SIGN) * q.y, p.y + T(SIGN) * q.x};
        z[R - K] = {p.x + T(SIGN) * q.y, p.y - T(SIGN) * q.x};
        odd_outputs<R, SIGN, RNZ, K + 1>(z, s, d, z0);
    }
}

// radix-R butterfly, inputs z[r >= RNZ] zero
template <int R, int SIGN, int RNZ, typename T>
__device__ __forceinline__ void radix(cx<T> (&z)[R]) {
    if constexpr (RNZ <= 1) {
#pragma unroll
        for (int k = 1; k < R; ++k) z[k] = z[0];
    } else if constexpr (R == 2) {
        const cx<T> a = z[0], b = z[1];
        z[0] = a + b;
        z[1] = a - b;
    } else if constexpr (R == 4) {
        const cx<T> a = z[0], b = z[1];
        const cx<T> s0 = RNZ > 2 ? a + z[2] : a, d0 = RNZ > 2 ? a - z[2] : a;
        const cx<T> s1 = RNZ > 3 ? b + z[3] : b, d1 = RNZ > 3 ? b - z[3] : b;
        const cx<T> e = {T(-SIGN) * d1.y, T(SIGN) * d1.x};
        z[0] = s0 + s1;
        z[1] = d0 + e;
        z[2] = s0 - s1;
        z[3] = d0 - e;
    } else {
        constexpr int H = (R - 1) / 2;
        cx<T> s[H], d[H];
        cx<T> sum = z[0];
        const cx<T> z0 = z[0];
#pragma unroll
        for (int r = 1; r <= H; ++r) {
            s[r - 1] = r < RNZ ? (R - r < RNZ ? z[r] + z[R - r] : z[r]) : czero<T>();
            d[r - 1] = r < RNZ ? (R - r < RNZ ? z[r] - z[R - r] : z[r]) : czero<T>();
            if (r < RNZ) sum = sum + s[r - 1];
        }
        odd_outputs<R, SIGN, RNZ, 1>(z, s, d, z0);
        z[0] = sum;
    }
}

template <int N, int SIGN, int NZ, typename T>
__device__ __forceinline__ void dft(cx<T> (&x)[N]);

template <int N, int R, int M, int SIGN, int NZ, int r, typename T>
__device__ __forceinline__ void dft_sub(cx<T> (&y)[R][M]) {
    if constexpr (r < R) {
        dft<M, SIGN, NZ <= r ? 0 : (NZ - r + R - 1) / R>(y[r]);
        dft_sub<N, R, M, SIGN, NZ, r + 1>(y);
    }
}
template <int N, int R, int M, int SIGN, int NZ, int k1, int r, typename T>
__device__ __forceinline__ void dft_twist(cx<T> (&z)[R], const cx<T> (&y)[R][M]) {
    if constexpr (r < R) {
        z[r] = rot<N, r * k1, SIGN>(y[r][k1]);
        dft_twist<N, R, M, SIGN, NZ, k1, r + 1>(z, y);
    }
}
template <int N, int R, int M, int SIGN, int NZ, int k1, typename T>
__device__ __forceinline__ void dft_join(cx<T> (&x)[N], const cx<T> (&y)[R][M]) {
    if constexpr (k1 < M) {
        cx<T> z[R];
        dft_twist<N, R, M, SIGN, NZ, k1, 0>(z, y);
        radix<R, SIGN, imin(NZ, R)>(z);
#pragma unroll
        for (int k2 = 0; k2 < R; ++k2) x[k1 + M * k2] = z[k2];
        dft_join<N, R, M, SIGN, NZ, k1 + 1>(x, y);
    }
}

// x <- sum_n x[n] exp(SIGN 2 pi i k n / N), x[n >= NZ] taken as zero
template <int N, int SIGN, int NZ, typename T>
__device__ __forceinline__ void dft(cx<T> (&x)[N]) {
    if constexpr (NZ <= 0) {
#pragma unroll
        for (int k = 0; k < N; ++k) x[k] = czero<T>();
    } else if constexpr (NZ == 1 || N == 1) {
#pragma unroll
        for (int k = 1; k < N; ++k) x[k] = x[0];
    } else {
        constexpr int R = dft_radix(N), M = N / R;
        if constexpr (M == 1) {
            radix<R, SIGN, NZ>(x);
        } else {
            cx<T> y[R][M];
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int m = 0; m < M; ++m) y[r][m] = r + R * m < NZ ? x[r + R * m] : czero<T>();
            dft_sub<N, R, M, SIGN, NZ, 0>(y);
            dft_join<N, R, M, SIGN, NZ, 0>(x, y);
        }
    }
}

}  // namespace grp
}  // namespace lgf
