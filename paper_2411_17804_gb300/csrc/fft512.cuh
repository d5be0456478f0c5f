// Register-resident 512-point FFT building blocks (exponent +), shared by the
// FP32 large-grid EPIC kernels and the FFT correlator.
//
// A 512-point transform by 64 threads, each holding 8 points, in three
// radix-8 passes (512 = 8 x 8 x 8) with two exchanges through shared memory.
// Pass 1: thread tau takes x[tau + 64 m], m < 8, an 8-point DFT over m,
// twiddle w512^(tau k1); pass 2: thread (k1, t1) the 8 values of k1 at
// tau = t1 + 8 t2, an 8-point DFT over t2, twiddle w64^(t1 k2); pass 3: thread
// (k1, k2) the 8 values at t1, an 8-point DFT over t1.  Thread tau ends with
// X[tau + 64 j], j < 8 (natural order, stride 64).  The exchange layouts (rows
// 66 apart, then k1 74 + k2 9 + t1; 65 and 73 for pairs) serve every pass's
// accesses without bank conflicts.
#pragma once

#include <cuda_runtime.h>

namespace hai_fft512 {

constexpr int kFftBuf = 589;                 // float2 per transform's exchange buffer

__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cmuli(float2 a) { return make_float2(-a.y, a.x); }          // a * i
__device__ __forceinline__ float2 cadd_i(float2 a, float2 b) { return make_float2(a.x - b.y, a.y + b.x); }   // a + i b
__device__ __forceinline__ float2 csub_i(float2 a, float2 b) { return make_float2(a.x + b.y, a.y - b.x); }   // a - i b
template <int N8>                                                 // a * e^(+i pi N8 / 4), N8 = 1 or 3
__device__ __forceinline__ float2 crot(float2 a) {
    const float h = 0.70710678118654752f;                         // cos(pi / 4)
    return N8 == 1 ? make_float2(h * (a.x - a.y), h * (a.x + a.y)) : make_float2(-h * (a.x + a.y), h * (a.x - a.y));
}

// The same value of two polarisations, real parts and imaginary parts as packed
// pairs: one instruction (two FP32 lanes, each rounded as the scalar one) for both.
// The rate of the FP32 pipe is the same (125 operations a cycle and SM measured
// either way); what halves is the instructions to issue.
struct c2 {
    unsigned long long re, im;                                    // (X, Y), (X, Y)
};
__device__ __forceinline__ unsigned long long pack2(float lo, float hi) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ float2 unpack2(unsigned long long v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b) {
    unsigned long long r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ unsigned long long sub2(unsigned long long a, unsigned long long b) {
    unsigned long long r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ unsigned long long mul2(unsigned long long a, unsigned long long b) {
    unsigned long long r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ c2 cadd(c2 a, c2 b) { return {add2(a.re, b.re), add2(a.im, b.im)}; }
__device__ __forceinline__ c2 csub(c2 a, c2 b) { return {sub2(a.re, b.re), sub2(a.im, b.im)}; }
__device__ __forceinline__ c2 cadd_i(c2 a, c2 b) { return {sub2(a.re, b.im), add2(a.im, b.re)}; }
__device__ __forceinline__ c2 csub_i(c2 a, c2 b) { return {add2(a.re, b.im), sub2(a.im, b.re)}; }
template <int N8>
__device__ __forceinline__ c2 crot(c2 a) {
    const float h = 0.70710678118654752f;
    const unsigned long long hh = pack2(h, h), d = sub2(a.re, a.im), s = add2(a.re, a.im);
    return N8 == 1 ? c2{mul2(hh, d), mul2(hh, s)} : c2{mul2(pack2(-h, -h), s), mul2(hh, d)};
}
// one factor for both: scalar, a factor's pairs would cost more moves than they save
__device__ __forceinline__ c2 cmul(c2 a, float2 w) {
    const float2 r = unpack2(a.re), i = unpack2(a.im);
    return {pack2(fmaf(r.x, w.x, -i.x * w.y), fmaf(r.y, w.x, -i.y * w.y)),
            pack2(fmaf(r.x, w.y, i.x * w.x), fmaf(r.y, w.y, i.y * w.x))};
}

// |F_X|^2, |F_Y|^2 (a pair) and F_X conj(F_Y) of one pixel added to its sums.
__device__ __forceinline__ void add_products(c2 f, unsigned long long &pw, float &xr, float &xi) {
    pw = fma2(f.re, f.re, fma2(f.im, f.im, pw));
    const float2 r = unpack2(f.re), i = unpack2(f.im);
    xr = fmaf(r.x, r.y, fmaf(i.x, i.y, xr));           // Re X conj(Y)
    xi = fmaf(i.x, r.y, fmaf(-r.x, i.y, xi));          // Im X conj(Y)
}

// 4-point DFT, exponent +: X_k = sum_m x_m i^(m k), natural order; I2: x2 is
// taken times i.
template <bool I2 = false, typename V>
__device__ __forceinline__ void dft4(V &x0, V &x1, V &x2, V &x3) {
    const V p = I2 ? cadd_i(x0, x2) : cadd(x0, x2), r = I2 ? csub_i(x0, x2) : csub(x0, x2);
    const V q = cadd(x1, x3), s = csub(x1, x3);
    x0 = cadd(p, q);
    x1 = cadd_i(r, s);
    x2 = csub(p, q);
    x3 = csub_i(r, s);
}

// 8-point DFT, exponent +, natural order in and out (decimation in frequency:
// the even outputs are the 4-point DFT of a_m + a_(m+4), the odd ones that of
// (a_m - a_(m+4)) w8^m)
template <typename V>
__device__ __forceinline__ void dft8(V (&a)[8]) {
    V u0 = cadd(a[0], a[4]), u1 = cadd(a[1], a[5]), u2 = cadd(a[2], a[6]), u3 = cadd(a[3], a[7]);
    V v0 = csub(a[0], a[4]), v1 = csub(a[1], a[5]), v2 = csub(a[2], a[6]), v3 = csub(a[3], a[7]);
    v1 = crot<1>(v1);
    v3 = crot<3>(v3);
    dft4(u0, u1, u2, u3);
    dft4<true>(v0, v1, v2, v3);
    a[0] = u0; a[2] = u1; a[4] = u2; a[6] = u3;
    a[1] = v0; a[3] = v1; a[5] = v2; a[7] = v3;
}

// The 8-point DFT when only a[0] and a[1] can be non-zero (the first pass of
// a transform whose non-zero inputs all lie in its first quarter).
template <typename V>
__device__ __forceinline__ void dft8_first2(V (&a)[8]) {
    const V u0 = a[0], u1 = a[1], v1 = crot<1>(u1);
    a[0] = cadd(u0, u1);
    a[2] = cadd_i(u0, u1);
    a[4] = csub(u0, u1);
    a[6] = csub_i(u0, u1);
    a[1] = cadd(u0, v1);
    a[3] = cadd_i(u0, v1);
    a[5] = csub(u0, v1);
    a[7] = csub_i(u0, v1);
}

// Exchange buffers: kFftBuf values a transform; row strides for which the
// accesses of 8-byte (16-byte) values are conflict-free.
template <typename V>
struct Xchg;
template <>
struct Xchg<float2> {
    using T = float2;
    static constexpr int kA = 66, kB = 74;
    static __device__ __forceinline__ T put(float2 v) { return v; }
    static __device__ __forceinline__ float2 get(T v) { return v; }
};
template <>
struct Xchg<c2> {
    using T = ulonglong2;
    static constexpr int kA = 65, kB = 73;
    static __device__ __forceinline__ T put(c2 v) { return make_ulonglong2(v.re, v.im); }
    static __device__ __forceinline__ c2 get(T v) { return {v.x, v.y}; }
};

// Twiddle tables of the 512-point transform in shared memory:
//   tw[n] = w512^n (n < 512), T1[(k - 1) 64 + tau] = w512^(tau k),
//   T2[(k - 1) 8 + t1] = w64^(t1 k) (k = 1..7): read by consecutive threads
//   without bank conflicts (T2 is a broadcast within groups of 8).
constexpr int kTwFloat2 = 512 + 7 * 64 + 7 * 8;

__device__ __forceinline__ void fill_fft512_tables(float2 *tw) {
    for (int k = threadIdx.x; k < 512; k += blockDim.x) {
        float s, c;
        sincospif((float)k / 256.0f, &s, &c);
        tw[k] = make_float2(c, s);
    }
    __syncthreads();
    float2 *T1 = tw + 512, *T2 = T1 + 7 * 64;
    for (int i = threadIdx.x; i < 7 * 64; i += blockDim.x) T1[i] = tw[((i & 63) * (1 + (i >> 6))) & 511];
    for (int i = threadIdx.x; i < 7 * 8; i += blockDim.x) T2[i] = tw[(8 * (i & 7) * (1 + (i >> 3))) & 511];
}

// One 512-point transform by the 64 threads of a group (tau = thread in the
// group), `buf` its exchange buffer, tw the tables above; ends with a[j] =
// X[tau + 64 j].  bar() synchronises every group of the CTA together.  Z2:
// the inputs a[2..7] are zero (skipped in the first pass).
template <bool Z2, typename V, typename Bar>
__device__ __forceinline__ void fft512(V (&a)[8], int tau, typename Xchg<V>::T *buf, const float2 *tw, Bar bar) {
    using X = Xchg<V>;
    const float2 *T1 = tw + 512, *T2 = T1 + 7 * 64;
    if (Z2) dft8_first2(a);
    else dft8(a);
#pragma unroll
    for (int k = 1; k < 8; k++) a[k] = cmul(a[k], T1[(k - 1) * 64 + tau]);
#pragma unroll
    for (int k = 0; k < 8; k++) buf[k * X::kA + tau] = X::put(a[k]);
    bar();
    const int k1 = tau & 7, q = tau >> 3;
#pragma unroll
    for (int t2 = 0; t2 < 8; t2++) a[t2] = X::get(buf[k1 * X::kA + q + 8 * t2]);
    dft8(a);
#pragma unroll
    for (int k = 1; k < 8; k++) a[k] = cmul(a[k], T2[(k - 1) * 8 + q]);
    bar();
#pragma unroll
    for (int k2 = 0; k2 < 8; k2++) buf[k1 * X::kB + k2 * 9 + q] = X::put(a[k2]);
    bar();
#pragma unroll
    for (int t1 = 0; t1 < 8; t1++) a[t1] = X::get(buf[k1 * X::kB + q * 9 + t1]);
    dft8(a);
}

}  // namespace hai_fft512
