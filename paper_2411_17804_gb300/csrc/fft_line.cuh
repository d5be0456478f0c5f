// Register-resident line transforms of 16 to 256 points (exponent +), shared
// by the two XFFT imagers.
//
// A line of N = L E points is held by L lanes, lane t holding x[t + L m],
// m < E.  With k = k1 + E k2: lane t takes the E-point DFT over m, multiplies
// output k1 by wN^(t k1), and after one exchange lane j takes the L-point DFTs
// over t of k1 = j + L u (u < E / L), ending with X[j + L u + E k2] in
// a[L u + k2].  One exchange instead of log2 N passes over shared memory.
#pragma once

#include "fft512.cuh"

namespace hai_fft {

using hai_fft512::cmul;

template <int N>
struct Line {
    static constexpr int L = N >= 256 ? 16 : N >= 64 ? 8 : 4;   // lanes
    static constexpr int E = N / L;                             // points per lane: 4, 8, 8, 16, 16
    static constexpr int U = E / L;                             // L-point DFTs per lane after the exchange
    static_assert(N >= 16 && N <= 256 && U >= 1, "line length");
};

// 16-point DFT in registers, natural order: 4 x 4.
__device__ __forceinline__ void dft16(float2 (&a)[16]) {
    const float c = 0.92387953251128674f, s = 0.38268343236508977f, h = 0.70710678118654752f;   // pi/8, pi/4
    // over m2 of x[m1 + 4 m2]
#pragma unroll
    for (int m = 0; m < 4; m++) hai_fft512::dft4(a[m], a[m + 4], a[m + 8], a[m + 12]);
    // a[m1 + 4 k1] *= w16^(m1 k1)
    a[5] = cmul(a[5], make_float2(c, s));
    a[9] = make_float2(h * (a[9].x - a[9].y), h * (a[9].x + a[9].y));
    a[13] = cmul(a[13], make_float2(s, c));
    a[6] = make_float2(h * (a[6].x - a[6].y), h * (a[6].x + a[6].y));
    a[10] = hai_fft512::cmuli(a[10]);
    a[14] = make_float2(-h * (a[14].x + a[14].y), h * (a[14].x - a[14].y));
    a[7] = cmul(a[7], make_float2(s, c));
    a[11] = make_float2(-h * (a[11].x + a[11].y), h * (a[11].x - a[11].y));
    a[15] = cmul(a[15], make_float2(-c, -s));
    // over m1: X[k1 + 4 k2]
#pragma unroll
    for (int k = 0; k < 4; k++) hai_fft512::dft4(a[4 * k], a[4 * k + 1], a[4 * k + 2], a[4 * k + 3]);
    // a[4 k1 + k2] -> natural order k1 + 4 k2
#pragma unroll
    for (int i = 0; i < 4; i++)
#pragma unroll
        for (int j = i + 1; j < 4; j++) {
            const float2 t = a[4 * i + j];
            a[4 * i + j] = a[4 * j + i];
            a[4 * j + i] = t;
        }
}

template <int R>
__device__ __forceinline__ void dft(float2 (&a)[R]) {
    if constexpr (R == 16) dft16(a);
    else if constexpr (R == 8) hai_fft512::dft8(a);
    else hai_fft512::dft4(a[0], a[1], a[2], a[3]);
}

// wN^k, k < N, into shared memory.
template <int N>
__device__ __forceinline__ void fill_twiddles(float2 *tw) {
    for (int k = threadIdx.x; k < N; k += blockDim.x) {
        float s, c;
        sincospif((float)(2 * k) / (float)N, &s, &c);
        tw[k] = make_float2(c, s);
    }
}

// First half: the E-point DFT and the twiddles of lane t.
template <int N>
__device__ __forceinline__ void line_first(float2 (&a)[Line<N>::E], int t, const float2 *tw) {
    dft<Line<N>::E>(a);
#pragma unroll
    for (int k = 1; k < Line<N>::E; k++) a[k] = cmul(a[k], tw[t * k]);      // t k < N
}

// Second half, after the exchange has put value k1 = j + L u of lane t in
// a[L u + t]: a[L u + k2] = X[j + L u + E k2].
template <int N>
__device__ __forceinline__ void line_second(float2 (&a)[Line<N>::E]) {
    constexpr int L = Line<N>::L;
#pragma unroll
    for (int u = 0; u < Line<N>::U; u++) {
        float2 b[L];
#pragma unroll
        for (int i = 0; i < L; i++) b[i] = a[L * u + i];
        dft<L>(b);
#pragma unroll
        for (int i = 0; i < L; i++) a[L * u + i] = b[i];
    }
}

}  // namespace hai_fft
