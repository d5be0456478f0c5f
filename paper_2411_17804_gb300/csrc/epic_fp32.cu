// EPIC direct imager, FP32 on CUDA cores (Eq. intra-station EPIC followed by
// the squaring and temporal sum of Eq. intra-station squaring), for grids of
// N = 16, 32, 64 (larger grids: epic_large.cu).
//
// In every kernel here one CTA sums a contiguous range of the flattened
// (channel, sample) index.  The lines are held in registers, at N = 64 by groups
// of 8 lanes (epic64_kernel) and at N = 16 and 32 by groups of 4
// (epic_small_kernel), both described below.  Where even their forms with the
// gather table in global memory do not fit shared memory, epic_fp32_kernel does,
// per group of kSamples samples:
//   1. stages the int8 voltages of the group in shared memory;
//   2. row pass: one thread per (sample, pol, box row) gathers the gridded
//      row sum_a conj(W~) E_a from the layout's gather table and transforms
//      it along x with an N-point radix-2 FFT held in registers;
//   3. column pass: one thread per (sample, pol, column) transforms along y,
//      reading and writing its own column of the same shared buffer;
//   4. squaring: every thread owns N*N/256 pixels and adds F_X conj(F_Y)
//      products to register accumulators.
// Only the kernel's bounding box is transformed, placed at the grid origin.
// Shifting the input by (bx0, by0) multiplies F by exp(+2 pi i l.b / N), a
// phase common to both polarisations that cancels in every F_a conj(F_b);
// the (-1)^(jx+jy) phase-centre factor is an output shift by N/2.
#include <math.h>

#include <algorithm>

#include "fft512.cuh"
#include "hai_internal.h"

namespace {

constexpr int kThreads = 256;
constexpr int kSamples = 2;        // samples per group
constexpr int kTwN = 64;           // twiddle table resolution

__constant__ float2 c_tw[kTwN / 2];   // exp(+2 pi i m / 64), m < 32

__host__ __device__ constexpr int bitrev(int i, int n) {
    int r = 0;
    for (int b = 1; b < n; b <<= 1) r = (r << 1) | ((i & b) ? 1 : 0);
    return r;
}

__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}

// In-register radix-2 decimation-in-time FFT, X[k] = sum_n x[n] e^{+2 pi i nk/N}.
template <int N>
__device__ __forceinline__ void fft_reg(float2 (&x)[N]) {
#pragma unroll
    for (int i = 0; i < N; i++) {
        const int j = bitrev(i, N);
        if (i < j) {
            float2 t = x[i];
            x[i] = x[j];
            x[j] = t;
        }
    }
#pragma unroll
    for (int len = 2; len <= N; len <<= 1) {
        const int half = len / 2;
#pragma unroll
        for (int k = 0; k < half; k++) {
#pragma unroll
            for (int s = 0; s < N; s += len) {
                float2 a = x[s + k], b = x[s + k + half], bw;
                if (k == 0) {
                    bw = b;
                } else if (4 * k == len) {
                    bw = make_float2(-b.y, b.x);               // times +i
                } else {
                    bw = cmul(b, c_tw[k * (kTwN / len)]);
                }
                x[s + k] = make_float2(a.x + bw.x, a.y + bw.y);
                x[s + k + half] = make_float2(a.x - bw.x, a.y - bw.y);
            }
        }
    }
}

template <int N, int P>
struct EpicSmem {
    static constexpr int NP = N + 1;                       // padded row stride
    static constexpr int kBuf = kSamples * P * N * NP;     // float2 count
};

// Gridded value of one cell: sum over the cell's gather entries.
__device__ __forceinline__ float2 grid_cell(int cell, const int32_t *__restrict__ cstart,
                                            const int32_t *__restrict__ celem,
                                            const float2 *__restrict__ cw, const char2 *e) {
    float2 acc = make_float2(0.f, 0.f);
    const int b = __ldg(cstart + cell), end = __ldg(cstart + cell + 1);
    for (int i = b; i < end; i++) {
        const int a = __ldg(celem + i);
        const float2 w = __ldg(cw + i);
        const char2 v = e[a];
        const float er = (float)v.x, ei = (float)v.y;
        acc.x = fmaf(w.x, er, fmaf(-w.y, ei, acc.x));
        acc.y = fmaf(w.x, ei, fmaf(w.y, er, acc.y));
    }
    return acc;
}

template <int N, int P>
__global__ void __launch_bounds__(kThreads, 1)
epic_fp32_kernel(const int8_t *__restrict__ volt, int C, int T, int ne, long long len,
                 int box_w, int box_h, const int32_t *__restrict__ cstart,
                 const int32_t *__restrict__ celem, const float2 *__restrict__ cw,
                 float *__restrict__ out, int direct, int accumulate) {
    constexpr int Q = (P == 2) ? 4 : 1;
    constexpr int NP = EpicSmem<N, P>::NP;
    constexpr int PIX = N * N / kThreads;
    static_assert(N * N % kThreads == 0, "pixels per thread");
    extern __shared__ __align__(16) unsigned char smem[];
    float2 *buf = reinterpret_cast<float2 *>(smem);
    char2 *vs = reinterpret_cast<char2 *>(smem + sizeof(float2) * EpicSmem<N, P>::kBuf);

    const int tid = threadIdx.x;
    const long long total = (long long)C * T;
    const long long s0 = (long long)blockIdx.x * len;
    const long long s1 = min(total, s0 + len);
    const int sample_elems = P * ne;                 // char2 per sample

    float acc[PIX][Q];
#pragma unroll
    for (int m = 0; m < PIX; m++)
#pragma unroll
        for (int q = 0; q < Q; q++) acc[m][q] = 0.f;

    int seg = 0;
    int cur_c = (int)(s0 / T);
    auto flush = [&](int c, int sgm) {
        float *dst;
        if (direct) dst = out + (size_t)c * Q * N * N;
        else dst = out + ((size_t)blockIdx.x * 2 + sgm) * Q * N * N;
#pragma unroll
        for (int m = 0; m < PIX; m++) {
            const int pix = tid + m * kThreads;
#pragma unroll
            for (int q = 0; q < Q; q++) {
                float v = acc[m][q];
                if (direct && accumulate) v += dst[(size_t)q * N * N + pix];
                dst[(size_t)q * N * N + pix] = v;
                acc[m][q] = 0.f;
            }
        }
    };

    for (long long s = s0; s < s1;) {
        const int c = (int)(s / T);
        if (c != cur_c) {
            flush(cur_c, seg);
            seg++;
            cur_c = c;
        }
        const long long chan_end = (long long)(c + 1) * T;
        const int ng = (int)min((long long)kSamples, min(s1, chan_end) - s);

        // 1. stage voltages of the group (contiguous bytes)
        {
            const size_t nbytes = (size_t)ng * sample_elems * 2;
            const int8_t *src = volt + (size_t)s * sample_elems * 2;
            int8_t *dst = reinterpret_cast<int8_t *>(vs);
            if ((((uintptr_t)src) & 15) == 0 && (nbytes & 15) == 0) {
                const int4 *s4 = reinterpret_cast<const int4 *>(src);
                int4 *d4 = reinterpret_cast<int4 *>(dst);
                for (size_t i = tid; i < nbytes / 16; i += kThreads) d4[i] = __ldg(s4 + i);
            } else {
                for (size_t i = tid; i < nbytes; i += kThreads) dst[i] = src[i];
            }
        }
        __syncthreads();

        // 2. row pass: grid + FFT along x
        for (int task = tid; task < ng * P * box_h; task += kThreads) {
            const int g = task / (P * box_h);
            const int p = (task / box_h) % P;
            const int y = task % box_h;
            const char2 *e = vs + (size_t)(g * P + p) * ne;
            float2 x[N];
#pragma unroll
            for (int u = 0; u < N; u++)
                x[u] = (u < box_w) ? grid_cell(y * box_w + u, cstart, celem, cw, e) : make_float2(0.f, 0.f);
            fft_reg<N>(x);
            float2 *row = buf + (size_t)(g * P + p) * N * NP + (size_t)y * NP;
#pragma unroll
            for (int k = 0; k < N; k++) row[k] = x[k];
        }
        __syncthreads();

        // 3. column pass: FFT along y (rows >= box_h are zero)
        for (int task = tid; task < ng * P * N; task += kThreads) {
            const int gp = task / N;
            const int k = task % N;
            float2 *col = buf + (size_t)gp * N * NP + k;
            float2 x[N];
#pragma unroll
            for (int r = 0; r < N; r++) x[r] = (r < box_h) ? col[(size_t)r * NP] : make_float2(0.f, 0.f);
            fft_reg<N>(x);
#pragma unroll
            for (int r = 0; r < N; r++) col[(size_t)r * NP] = x[r];
        }
        __syncthreads();

        // 4. squaring and accumulation (pixel l reads F at l + N/2 mod N)
#pragma unroll
        for (int m = 0; m < PIX; m++) {
            const int pix = tid + m * kThreads;
            const int ly = pix / N, lx = pix % N;
            const int src = ((ly + N / 2) & (N - 1)) * NP + ((lx + N / 2) & (N - 1));
            for (int g = 0; g < ng; g++) {
                const float2 fx = buf[(size_t)(g * P) * N * NP + src];
                acc[m][0] = fmaf(fx.x, fx.x, fmaf(fx.y, fx.y, acc[m][0]));
                if (P == 2) {
                    const float2 fy = buf[(size_t)(g * P + 1) * N * NP + src];
                    acc[m][Q > 1 ? 1 : 0] = fmaf(fy.x, fy.x, fmaf(fy.y, fy.y, acc[m][Q > 1 ? 1 : 0]));
                    acc[m][Q > 2 ? 2 : 0] = fmaf(fx.x, fy.x, fmaf(fx.y, fy.y, acc[m][Q > 2 ? 2 : 0]));
                    acc[m][Q > 3 ? 3 : 0] = fmaf(fx.y, fy.x, fmaf(-fx.x, fy.y, acc[m][Q > 3 ? 3 : 0]));
                }
            }
        }
        __syncthreads();
        s += ng;
    }
    if (s1 > s0) flush(cur_c, seg);
}

// ------------------------------------------------------------------ N = 64
// The 64 x 64 grid with every 64-point line in registers: a group of 8 lanes
// per line, lane t holding points t + 8 m (m < 8).  With k = k1 + 8 k2,
// w64^((t + 8 m) k) = w64^(t k1) w8^(t k2) w8^(m k1): lane t takes the
// 8-point DFT over m (only m < 4 when the box spans at most 32 cells along
// the line), multiplies output k1 by w64^(t k1), and after one exchange
// through the group's shared scratch (within the warp) lane j takes the
// 8-point DFT over t of the values of k1 = j, ending with X[j + 8 k2] in
// a[k2].  Exponent + throughout.
//
// Per phase of one or two samples: row pass (a group per box row and sample,
// or per (box row, pol): gather, transform along x, row written to H), then
// column pass (a group per column, both pols, sample by sample: transform
// along y, then |F_X|^2, |F_Y|^2 and F_X conj(F_Y) of its 8 pixels into
// register accumulators).  The row pass of phase i and the column pass of
// phase i - 1 run together (H and the staged voltages double-buffered), so a
// phase costs one block barrier.
//
// Shared layouts, all accesses in the minimum two wavefronts per 8-byte
// access: H[sample][p][y][(k + 2 (y & 7)) & 63] with pol (or re, im) and sample planes
// 8 (mod 16) float2 apart (a half-warp writes one row of both samples, or of
// both pols, or rows y and y + 4 of one pol, and reads rows t + 8 m of two
// adjacent columns); the exchange scratch of a group holds value k of lane t
// at 9 k + t, groups 72 float2 (8 mod 16) apart, one pol at a time.
constexpr int k64Threads = 512;                  // 64 groups of 8 lanes
constexpr int k64Xs = 72;                        // float2 of exchange scratch per group (one pol at a time)

template <typename V>
__device__ __forceinline__ void dft8_first4(V (&a)[8]) {
    // inputs a[4..7] zero: the even outputs are the 4-point DFT of a[0..3],
    // the odd ones that of a[m] w8^m
    V v0 = a[0], v1 = hai_fft512::crot<1>(a[1]), v2 = a[2], v3 = hai_fft512::crot<3>(a[3]);
    V u0 = a[0], u1 = a[1], u2 = a[2], u3 = a[3];
    hai_fft512::dft4(u0, u1, u2, u3);
    hai_fft512::dft4<true>(v0, v1, v2, v3);
    a[0] = u0; a[2] = u1; a[4] = u2; a[6] = u3;
    a[1] = v0; a[3] = v1; a[5] = v2; a[7] = v3;
}

__device__ __forceinline__ void cp_async16_64(void *dst, const void *src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src) : "memory");
}

// Starts the copy of `bytes` voltages (2-byte aligned, as all voltages are)
// to a 16-byte aligned shared buffer, kept at their source's offset in 16
// bytes (staged_offset): the body goes by 16-byte cp.async whatever the
// station's sample size, the at most 14 bytes at each end by 2-byte copies (a
// station of 251 elements, 1,004 bytes a sample, 37 channels x 999 samples at
// N = 64: 697.0 -> 657.9 us against 2-byte loads for the whole copy).
__device__ __forceinline__ int staged_offset(const int8_t *src) { return (int)((uintptr_t)src & 15); }
__device__ __forceinline__ void stage_volt(const int8_t *src, int bytes, unsigned char *buf, int tid, int nthreads) {
    const int mis = staged_offset(src);
    unsigned char *dst = buf + mis;
    const int head = min(bytes, (16 - mis) & 15), body = (bytes - head) >> 4, tail = bytes - head - 16 * body;
    for (int i = tid; i < body; i += nthreads) cp_async16_64(dst + head + 16 * i, src + head + 16 * i);
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    if (tid < (head + tail) >> 1) {
        const int o = 2 * tid < head ? 2 * tid : 2 * tid + 16 * body;
        *reinterpret_cast<char2 *>(dst + o) = *reinterpret_cast<const char2 *>(src + o);
    }
}

// Shared memory of the N = 64 kernel.  SP samples per phase (2 when the box
// is at most 32 rows and shared memory allows, else 1); sample si of a phase
// and pol p keep their H plane at si SO + p PO, SO = 8 (mod 16) too, so that
// a half-warp writing one row of two samples stays within two wavefronts.
// TS: the gather table (cell starts, then {element, conj(W~)} as int4 per
// entry) is copied into shared memory at the start.
template <int P, bool PX, bool PY, int SP, bool TS>
struct Epic64Smem {
    static constexpr int HR = PY ? 32 : 64;                  // rows of H
    static constexpr int PO = HR * 64 + 8;                   // pol plane stride (float2)
    static constexpr int SO = (P * PO + 15) / 16 * 16 + 8;   // sample stride
    static constexpr int HB = SP * SO;                        // one of the two H buffers
    static constexpr size_t fixed = sizeof(float2) * (2 * (size_t)HB + 64 * (size_t)k64Xs);
    __host__ __device__ static size_t vbuf(int ne) { return ((size_t)SP * P * ne * 2 + 31) / 16 * 16; }
    __host__ __device__ static size_t cbytes(int ncell) { return TS ? ((size_t)(ncell + 1) * 4 + 15) / 16 * 16 : 0; }
    __host__ __device__ static size_t bytes(int ne, int ncell, int nnz) {
        return fixed + 2 * vbuf(ne) + cbytes(ncell) + (TS ? (size_t)nnz * 16 : 0);
    }
};

// Same arguments and outputs as epic_fp32_kernel<64, P> (nnz = the table's
// entry count); PX / PY: the box spans at most 32 cells along x / y.  The
// int8 voltages of the next phase are copied into shared memory while the
// current one is imaged.
//
// Row tasks: warp w takes rows w and 31 - w, so that the rows beyond a box of
// fewer than 32 spread over the four schedulers.  SP = 2: group g takes its row of
// sample g & 1 of the phase, both pols (one walk of the gather table for both); SP
// = 1: a row a group, both pols at once too for boxes of more than 32 rows (rows g
// and g + 4 paired in a half-warp), else pol g & 1.
//
// kPair: both pols go through one transform as packed pairs (one instruction for
// both), the two planes of H and the two halves of an exchange holding real and
// imaginary parts of (X, Y).  Bound: shared-memory wavefronts (exchanges, H and the
// gather's random reads: four fifths of the cycles) and issue slots.  37 channels x
// 999 samples of a station of 251 elements: 658 us with a transform per pol and the
// channel of a sample found by a 64-bit division, 617 us with packed pairs, 598 us
// with the channel's samples counted.
template <int P, bool PX, bool PY, int SP, bool TS>
__global__ void __launch_bounds__(k64Threads, 1)
epic64_kernel(const int8_t *__restrict__ volt, int C, int T, int ne, long long len, int box_w, int box_h,
              const int32_t *__restrict__ cstart_g, const int32_t *__restrict__ celem,
              const float2 *__restrict__ cw, int nnz, float *__restrict__ out, int direct, int accumulate) {
    constexpr int Q = (P == 2) ? 4 : 1;
    using S = Epic64Smem<P, PX, PY, SP, TS>;
    constexpr int PO = S::PO, SO = S::SO, HB = S::HB;
    constexpr bool kPair = P == 2 && (SP == 2 || !PY);       // both pols in one transform of packed pairs
    constexpr int GP = kPair ? 2 : 1;                        // pols per row task
    static_assert(SP == 1 || PY, "two samples per phase need a box of at most 32 rows");
    extern __shared__ __align__(16) unsigned char smem[];
    float2 *Hs = reinterpret_cast<float2 *>(smem);                        // [2][HB]
    float2 *xs = Hs + 2 * HB + (threadIdx.x >> 3) * k64Xs;                // this group's scratch
    unsigned char *vs = smem + S::fixed;                                  // [2][vstride]
    const int vbytes = P * ne * 2;                                        // one sample
    const int vstride = (int)S::vbuf(ne);
    const int ncell = box_w * box_h;
    int32_t *cs_s = reinterpret_cast<int32_t *>(vs + 2 * (size_t)vstride);
    int4 *ent_s = reinterpret_cast<int4 *>(reinterpret_cast<unsigned char *>(cs_s) + S::cbytes(ncell));

    const int tid = threadIdx.x, t = tid & 7, g = tid >> 3;
    const long long total = (long long)C * T;
    const long long s0 = (long long)blockIdx.x * len;
    const long long s1 = min(total, s0 + len);
    if (s0 >= s1) return;
    const int n = (int)(s1 - s0);
    const int nph = (n + SP - 1) / SP;

    if (TS) {
        for (int i = tid; i <= ncell; i += k64Threads) cs_s[i] = __ldg(cstart_g + i);
        for (int i = tid; i < nnz; i += k64Threads) {
            const float2 w = __ldg(cw + i);
            ent_s[i] = make_int4(__ldg(celem + i), __float_as_int(w.x), __float_as_int(w.y), 0);
        }
    }
    const int32_t *cstart = TS ? cs_s : cstart_g;

    // w64^(t k), k = 1..7, from the table of w64^m, m < 32
    float2 tw[8];
#pragma unroll
    for (int k = 1; k < 8; k++) {
        const int m = t * k;
        const float2 v = c_tw[m & 31];
        tw[k] = m < 32 ? v : make_float2(-v.x, -v.y);
    }

    auto load = [&](int ph, int b) {
        stage_volt(volt + (size_t)(s0 + (long long)SP * ph) * vbytes, min(SP, n - SP * ph) * vbytes,
                   vs + (size_t)b * vstride, tid, k64Threads);
    };

    float acc[8][Q];
#pragma unroll
    for (int k = 0; k < 8; k++)
#pragma unroll
        for (int q = 0; q < Q; q++) acc[k][q] = 0.f;
    const int col = g;                                   // column pass: column of this group
    int cur_c = (int)(s0 / T), seg = 0, left = T - (int)(s0 % T);   // left: samples of channel cur_c to add
    auto flush = [&](int c, int sgm) {
        float *dst = direct ? out + (size_t)c * Q * 4096 : out + ((size_t)blockIdx.x * 2 + sgm) * Q * 4096;
        const int lx = (col + 32) & 63;
#pragma unroll
        for (int k2 = 0; k2 < 8; k2++) {
            const int pix = ((t + 8 * k2 + 32) & 63) * 64 + lx;
#pragma unroll
            for (int q = 0; q < Q; q++) {
                float v = acc[k2][q];
                if (direct && accumulate) v += dst[(size_t)q * 4096 + pix];
                dst[(size_t)q * 4096 + pix] = v;
                acc[k2][q] = 0.f;
            }
        }
    };
    // second half of a 64-point line: a[k1] (twiddled) of lane t in, X[t + 8 k2] in a[k2] out
    auto finish = [&](float2 (&a)[8]) {
        __syncwarp();
#pragma unroll
        for (int k = 0; k < 8; k++) xs[9 * k + t] = a[k];
        __syncwarp();
#pragma unroll
        for (int u = 0; u < 8; u++) a[u] = xs[9 * t + u];
        hai_fft512::dft8(a);
    };

    // the same for a pair: real parts, then imaginary parts through the scratch
    using hai_fft512::c2;
    auto finish2 = [&](c2 (&a)[8]) {
        unsigned long long *x = reinterpret_cast<unsigned long long *>(xs);
        __syncwarp();
#pragma unroll
        for (int k = 0; k < 8; k++) x[9 * k + t] = a[k].re;
        __syncwarp();
#pragma unroll
        for (int u = 0; u < 8; u++) a[u].re = x[9 * t + u];
        __syncwarp();
#pragma unroll
        for (int k = 0; k < 8; k++) x[9 * k + t] = a[k].im;
        __syncwarp();
#pragma unroll
        for (int u = 0; u < 8; u++) a[u].im = x[9 * t + u];
        hai_fft512::dft8(a);
    };

    load(0, 0);
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    __syncthreads();
    for (int it = 0; it <= nph; it++) {
        if (it + 1 < nph) load(it + 1, (it + 1) & 1);
        if (it < nph) {
            // row pass of phase it
            const unsigned char *V = vs + (size_t)(it & 1) * vstride +
                                     staged_offset(volt + (size_t)(s0 + (long long)SP * it) * vbytes);
            float2 *H = Hs + (size_t)(it & 1) * HB;
            const int ns = min(SP, n - SP * it);
            do {
                int y, p0, si;
                const int w = g >> 2, yw = ((g & 2) ? 31 - w : w);
                if (SP == 2) {
                    si = g & 1;
                    p0 = 0;
                    y = yw;
                } else if (kPair) {
                    si = 0;
                    p0 = 0;
                    y = (g & ~7) | ((g & 1) << 2) | ((g >> 1) & 3);
                } else if (P == 2) {
                    si = 0;
                    p0 = g & 1;
                    y = yw;
                } else {
                    si = 0;
                    p0 = 0;
                    y = (g & ~7) | ((g & 1) << 2) | ((g >> 1) & 3);
                }
                const bool live = y < box_h && si < ns;
                if (!__any_sync(0xffffffffu, live)) break;                // warp-uniform
                float2 a[GP][8];
#pragma unroll
                for (int q = 0; q < GP; q++)
#pragma unroll
                    for (int m = 0; m < 8; m++) a[q][m] = make_float2(0.f, 0.f);
                if (live) {
                    const char2 *E = reinterpret_cast<const char2 *>(V + (size_t)si * vbytes) + (size_t)p0 * ne;
                    constexpr int MX = PX ? 4 : 8;
                    int cb[MX], ce[MX];                                   // the cells' entry ranges, loaded first
#pragma unroll
                    for (int m = 0; m < MX; m++) {
                        const int x = t + 8 * m;
                        cb[m] = ce[m] = 0;
                        if (x < box_w) {
                            cb[m] = cstart[y * box_w + x];
                            ce[m] = cstart[y * box_w + x + 1];
                        }
                    }
#pragma unroll
                    for (int m = 0; m < MX; m++) {
                        float2 acg[GP];
#pragma unroll
                        for (int q = 0; q < GP; q++) acg[q] = make_float2(0.f, 0.f);
                        for (int i = cb[m]; i < ce[m]; i++) {
                            int el;
                            float2 wv;                                    // conj(W~)
                            if (TS) {
                                const int4 d = ent_s[i];
                                el = d.x;
                                wv = make_float2(__int_as_float(d.y), __int_as_float(d.z));
                            } else {
                                el = __ldg(celem + i);
                                wv = __ldg(cw + i);
                            }
#pragma unroll
                            for (int q = 0; q < GP; q++) {
                                const char2 v = E[q * ne + el];
                                const float er = (float)v.x, ei = (float)v.y;
                                acg[q].x = fmaf(wv.x, er, fmaf(-wv.y, ei, acg[q].x));
                                acg[q].y = fmaf(wv.x, ei, fmaf(wv.y, er, acg[q].y));
                            }
                        }
#pragma unroll
                        for (int q = 0; q < GP; q++) a[q][m] = acg[q];
                    }
                }
                if constexpr (kPair) {
                    c2 b[8];
#pragma unroll
                    for (int m = 0; m < 8; m++)
                        b[m] = {hai_fft512::pack2(a[0][m].x, a[1][m].x), hai_fft512::pack2(a[0][m].y, a[1][m].y)};
                    if (PX) dft8_first4(b);
                    else hai_fft512::dft8(b);
#pragma unroll
                    for (int k = 1; k < 8; k++) b[k] = hai_fft512::cmul(b[k], tw[k]);
                    finish2(b);
                    if (live) {
                        const int sw = 2 * (y & 7);
                        unsigned long long *row = reinterpret_cast<unsigned long long *>(H + (size_t)si * SO + (size_t)y * 64);
#pragma unroll
                        for (int k2 = 0; k2 < 8; k2++) {
                            row[(t + 8 * k2 + sw) & 63] = b[k2].re;
                            row[PO + ((t + 8 * k2 + sw) & 63)] = b[k2].im;
                        }
                    }
                } else {
                    if (PX) dft8_first4(a[0]);
                    else hai_fft512::dft8(a[0]);
#pragma unroll
                    for (int k = 1; k < 8; k++) a[0][k] = hai_fft512::cmul(a[0][k], tw[k]);
                    finish(a[0]);
                    if (live) {
                        const int sw = 2 * (y & 7);
                        float2 *row = H + (size_t)si * SO + (size_t)p0 * PO + (size_t)y * 64;
#pragma unroll
                        for (int k2 = 0; k2 < 8; k2++) row[(t + 8 * k2 + sw) & 63] = a[0][k2];
                    }
                }
            } while (false);
        }
        if (it >= 1) {
            // column pass of phase it - 1, sample by sample
            const float2 *Hp = Hs + (size_t)((it - 1) & 1) * HB;
            const int ns = min(SP, n - SP * (it - 1));
            const int pos = (col + 2 * t) & 63;                           // row y = t + 8 m: y & 7 = t
#pragma unroll
            for (int si = 0; si < SP; si++) {
                if (si >= ns) break;                                      // CTA-uniform
                if (left == 0) {
                    flush(cur_c, seg);
                    seg++;
                    cur_c++;
                    left = T;
                }
                left--;
                const float2 *H = Hp + (size_t)si * SO;
                if constexpr (kPair) {
                    const unsigned long long *Hq = reinterpret_cast<const unsigned long long *>(H) + pos;
                    c2 x[8];
#pragma unroll
                    for (int m = 0; m < 8; m++) {
                        const int y = t + 8 * m;
                        x[m] = m < (PY ? 4 : 8) && y < box_h ? c2{Hq[y * 64], Hq[PO + y * 64]} : c2{0, 0};
                    }
                    if (PY) dft8_first4(x);
                    else hai_fft512::dft8(x);
#pragma unroll
                    for (int k = 1; k < 8; k++) x[k] = hai_fft512::cmul(x[k], tw[k]);
                    finish2(x);
#pragma unroll
                    for (int k2 = 0; k2 < 8; k2++) {
                        unsigned long long pw = hai_fft512::pack2(acc[k2][0], acc[k2][Q > 1 ? 1 : 0]);
                        hai_fft512::add_products(x[k2], pw, acc[k2][Q > 2 ? 2 : 0], acc[k2][Q > 3 ? 3 : 0]);
                        const float2 v = hai_fft512::unpack2(pw);
                        acc[k2][0] = v.x;
                        acc[k2][Q > 1 ? 1 : 0] = v.y;
                    }
                } else {
                    float2 f[P][8];
#pragma unroll
                    for (int p = 0; p < P; p++) {
#pragma unroll
                        for (int m = 0; m < 8; m++) {
                            const int y = t + 8 * m;
                            f[p][m] = (m < (PY ? 4 : 8) && y < box_h) ? H[(size_t)p * PO + (size_t)y * 64 + pos]
                                                                      : make_float2(0.f, 0.f);
                        }
                        if (PY) dft8_first4(f[p]);
                        else hai_fft512::dft8(f[p]);
#pragma unroll
                        for (int k = 1; k < 8; k++) f[p][k] = hai_fft512::cmul(f[p][k], tw[k]);
                    }
#pragma unroll
                    for (int p = 0; p < P; p++) finish(f[p]);
#pragma unroll
                    for (int k2 = 0; k2 < 8; k2++) {
                        const float2 fx = f[0][k2];
                        acc[k2][0] = fmaf(fx.x, fx.x, fmaf(fx.y, fx.y, acc[k2][0]));
                        if (P == 2) {
                            const float2 fy = f[P - 1][k2];
                            acc[k2][Q > 1 ? 1 : 0] = fmaf(fy.x, fy.x, fmaf(fy.y, fy.y, acc[k2][Q > 1 ? 1 : 0]));
                            acc[k2][Q > 2 ? 2 : 0] = fmaf(fx.x, fy.x, fmaf(fx.y, fy.y, acc[k2][Q > 2 ? 2 : 0]));
                            acc[k2][Q > 3 ? 3 : 0] = fmaf(fx.y, fy.x, fmaf(-fx.x, fy.y, acc[k2][Q > 3 ? 3 : 0]));
                        }
                    }
                }
            }
        }
        asm volatile("cp.async.wait_all;\n" ::: "memory");
        __syncthreads();
    }
    flush(cur_c, seg);
}

// ------------------------------------------------------- N = 16 and N = 32
// Lines in registers as at N = 64, by groups of 4 lanes: with E = N / 4 lane t
// holds points t + 4 m (m < E) and k = k1 + E k2, so it takes the E-point DFT
// over m, multiplies output k1 by wN^(t k1), and after one exchange through
// the group's scratch lane j takes the 4-point DFTs over t of k1 = j + 4 u,
// ending with X[j + 4 u + E k2].  A phase takes 128 / N samples: 128 groups
// hold the phase's columns, one (column, sample) each, and the box rows of its
// (sample, pol) fields are dealt to the same groups.  As at N = 64 the row
// pass of phase i runs beside the column pass of phase i - 1 (H and the staged
// voltages double-buffered): one block barrier per phase.  A phase never
// straddles two channels; at a channel's end the sample slots' sums are added
// in slot order in shared memory.
//
// These grids are latency-bound: one CTA per SM has a few samples of a short
// cadence, so the time is the chain gather -> row -> column of a phase times
// the number of phases.  The kernel before this one (above; one thread per
// whole row and column, two samples per phase) left all but 32 threads idle in
// its passes and re-walked 32 cells serially per thread.  One 64-element
// station, one pol, 1024 samples at N = 32: 100.3 -> 18.0 us a call, with the
// reduction below.
//
// Shared layouts: H[plane][y][(k + 4 y) & (N - 1)]: a half-warp writes rows
// y .. y + 3 (4 adjacent values each) and reads rows t + 4 m of 4 adjacent
// columns, 16 distinct 8-byte banks both ways; the exchange keeps value k1 of
// lane t at 4 k1 + ((t + k1) & 3), groups N + 4 float2 apart, conflict-free
// for the writes (one k1) and the reads (one t).
constexpr int kSmThreads = 512;                  // 128 groups of 4 lanes

template <int N, int P, bool TS>
struct EpicSmallSmem {
    static constexpr int SP = 128 / N;                       // samples per phase
    static constexpr int XS = N + 4;                         // exchange scratch of a group (float2)
    static constexpr int HB = SP * P * N * N;                // one of the two H buffers (float2)
    static constexpr size_t fixed = sizeof(float2) * (2 * (size_t)HB + 128 * (size_t)XS) +
                                    sizeof(float) * (size_t)(P == 2 ? 4 : 1) * N * N;
    // staged voltages of a phase, at their source's offset in 16 bytes
    __host__ __device__ static size_t vbuf(int ne) { return ((size_t)SP * P * ne * 2 + 31) / 16 * 16; }
    __host__ __device__ static size_t cbytes(int ncell) { return TS ? ((size_t)(ncell + 1) * 4 + 15) / 16 * 16 : 0; }
    __host__ __device__ static size_t bytes(int ne, int ncell, int nnz) {
        return fixed + 2 * vbuf(ne) + cbytes(ncell) + (TS ? (size_t)nnz * 16 : 0);
    }
};

// E-point DFT of a line's points in one lane; half: the second half is zero.
template <int E>
__device__ __forceinline__ void dft_small(float2 (&a)[E], bool half) {
    if constexpr (E == 8) {
        if (half) dft8_first4(a);
        else hai_fft512::dft8(a);
    } else {
        hai_fft512::dft4(a[0], a[1], a[2], a[3]);
    }
}

// Same arguments and outputs as epic64_kernel.
template <int N, int P, bool TS>
__global__ void __launch_bounds__(kSmThreads, 1)
epic_small_kernel(const int8_t *__restrict__ volt, int C, int T, int ne, long long len, int box_w, int box_h,
                  const int32_t *__restrict__ cstart_g, const int32_t *__restrict__ celem,
                  const float2 *__restrict__ cw, int nnz, float *__restrict__ out, int direct, int accumulate) {
    constexpr int Q = (P == 2) ? 4 : 1, E = N / 4, U = E / 4, NN = N * N;
    using S = EpicSmallSmem<N, P, TS>;
    constexpr int SP = S::SP, XS = S::XS, HB = S::HB;
    extern __shared__ __align__(16) unsigned char smem[];
    float2 *Hs = reinterpret_cast<float2 *>(smem);                        // [2][SP][P][N][N]
    float2 *xs = Hs + 2 * HB + (threadIdx.x >> 2) * XS;                   // this group's scratch
    float *fimg = reinterpret_cast<float *>(Hs + 2 * HB + 128 * XS);      // [Q][N][N], flush
    unsigned char *vs = smem + S::fixed;                                  // [2][vstride]
    const int vbytes = P * ne * 2;                                        // one sample
    const int vstride = (int)S::vbuf(ne);
    const int ncell = box_w * box_h;
    int32_t *cs_s = reinterpret_cast<int32_t *>(vs + 2 * (size_t)vstride);
    int4 *ent_s = reinterpret_cast<int4 *>(reinterpret_cast<unsigned char *>(cs_s) + S::cbytes(ncell));

    const int tid = threadIdx.x, t = tid & 3, g = tid >> 2;
    const long long total = (long long)C * T;
    const long long s0 = (long long)blockIdx.x * len;
    const long long s1 = min(total, s0 + len);
    if (s0 >= s1) return;
    // the range touches at most two channels: phases of the first, then of the second
    const int c0 = (int)(s0 / T);
    const long long sb = min(s1, (long long)(c0 + 1) * T);
    const int n0 = (int)(sb - s0), n1 = (int)(s1 - sb);
    const int nph0 = (n0 + SP - 1) / SP, nph = nph0 + (n1 + SP - 1) / SP;
    auto phase = [&](int ph, long long &start) {                          // first sample and count of a phase
        if (ph < nph0) {
            start = s0 + (long long)SP * ph;
            return min(SP, n0 - SP * ph);
        }
        start = sb + (long long)SP * (ph - nph0);
        return min(SP, n1 - SP * (ph - nph0));
    };

    if (TS) {
        for (int i = tid; i <= ncell; i += kSmThreads) cs_s[i] = __ldg(cstart_g + i);
        for (int i = tid; i < nnz; i += kSmThreads) {
            const float2 w = __ldg(cw + i);
            ent_s[i] = make_int4(__ldg(celem + i), __float_as_int(w.x), __float_as_int(w.y), 0);
        }
    }
    const int32_t *cstart = TS ? cs_s : cstart_g;

    float2 tw[E];                                                         // wN^(t k), k < E
#pragma unroll
    for (int k = 1; k < E; k++) {
        const int m = t * k * (kTwN / N);                                 // < 64
        const float2 v = c_tw[m & 31];
        tw[k] = m < 32 ? v : make_float2(-v.x, -v.y);
    }

    auto load = [&](int ph, int b) {
        long long start;
        const int bytes = phase(ph, start) * vbytes;
        stage_volt(volt + (size_t)start * vbytes, bytes, vs + (size_t)b * vstride, tid, kSmThreads);
    };

    float acc[E][Q];
#pragma unroll
    for (int k = 0; k < E; k++)
#pragma unroll
        for (int q = 0; q < Q; q++) acc[k][q] = 0.f;
    const int col = g & (N - 1), slot = g / N;           // column pass: column and sample slot of this group
    auto flush = [&](int c, int sgm) {
        for (int sl = 0; sl < SP; sl++) {
            if (slot == sl) {
                const int lx = (col + N / 2) & (N - 1);
#pragma unroll
                for (int u = 0; u < U; u++)
#pragma unroll
                    for (int k2 = 0; k2 < 4; k2++) {
                        const int pix = ((t + 4 * u + E * k2 + N / 2) & (N - 1)) * N + lx;
#pragma unroll
                        for (int q = 0; q < Q; q++) {
                            float *f = fimg + q * NN + pix;
                            *f = sl ? *f + acc[4 * u + k2][q] : acc[4 * u + k2][q];
                            acc[4 * u + k2][q] = 0.f;
                        }
                    }
            }
            __syncthreads();
        }
        float *dst = direct ? out + (size_t)c * Q * NN : out + ((size_t)blockIdx.x * 2 + sgm) * Q * NN;
        for (int i = tid; i < Q * NN; i += kSmThreads) dst[i] = direct && accumulate ? dst[i] + fimg[i] : fimg[i];
        __syncthreads();
    };
    // second half of a line: a[k1] (twiddled) of lane t in, a[4 u + k2] = X[t + 4 u + E k2] out
    auto finish = [&](float2 (&a)[E]) {
        __syncwarp();
#pragma unroll
        for (int k = 0; k < E; k++) xs[4 * k + ((t + k) & 3)] = a[k];
        __syncwarp();
#pragma unroll
        for (int u = 0; u < U; u++) {
#pragma unroll
            for (int i = 0; i < 4; i++) a[4 * u + i] = xs[4 * (t + 4 * u) + ((i + t) & 3)];
            hai_fft512::dft4(a[4 * u], a[4 * u + 1], a[4 * u + 2], a[4 * u + 3]);
        }
    };

    load(0, 0);
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    __syncthreads();
    for (int it = 0; it <= nph; it++) {
        if (it + 1 < nph) load(it + 1, (it + 1) & 1);
        if (it < nph) {
            // row pass of phase it: task = (sample, pol, box row), rows adjacent
            long long start;
            const int ns = phase(it, start);
            const unsigned char *V = vs + (size_t)(it & 1) * vstride + staged_offset(volt + (size_t)start * vbytes);
            float2 *H = Hs + (size_t)(it & 1) * HB;
            const int ntask = ns * P * box_h;
            for (int base = 0; base < ntask; base += 128) {               // CTA-uniform
                const int task = base + g;
                const bool live = task < ntask;
                if (!__any_sync(0xffffffffu, live)) continue;             // warp-uniform
                const int f = live ? task / box_h : 0, y = task - f * box_h;
                float2 a[E];
#pragma unroll
                for (int m = 0; m < E; m++) a[m] = make_float2(0.f, 0.f);
                if (live) {
                    const char2 *Ev = reinterpret_cast<const char2 *>(V) + (size_t)f * ne;
                    int cb[E], ce[E];                                     // the cells' entry ranges, loaded first
#pragma unroll
                    for (int m = 0; m < E; m++) {
                        const int x = t + 4 * m;
                        cb[m] = ce[m] = 0;
                        if (x < box_w) {
                            cb[m] = cstart[y * box_w + x];
                            ce[m] = cstart[y * box_w + x + 1];
                        }
                    }
#pragma unroll
                    for (int m = 0; m < E; m++)
                        for (int i = cb[m]; i < ce[m]; i++) {
                            int el;
                            float2 wv;                                    // conj(W~)
                            if (TS) {
                                const int4 d = ent_s[i];
                                el = d.x;
                                wv = make_float2(__int_as_float(d.y), __int_as_float(d.z));
                            } else {
                                el = __ldg(celem + i);
                                wv = __ldg(cw + i);
                            }
                            const char2 v = Ev[el];
                            const float er = (float)v.x, ei = (float)v.y;
                            a[m].x = fmaf(wv.x, er, fmaf(-wv.y, ei, a[m].x));
                            a[m].y = fmaf(wv.x, ei, fmaf(wv.y, er, a[m].y));
                        }
                }
                dft_small<E>(a, box_w <= N / 2);
#pragma unroll
                for (int k = 1; k < E; k++) a[k] = hai_fft512::cmul(a[k], tw[k]);
                finish(a);
                if (live) {
                    float2 *row = H + ((size_t)f * N + y) * N;
#pragma unroll
                    for (int u = 0; u < U; u++)
#pragma unroll
                        for (int k2 = 0; k2 < 4; k2++) row[(t + 4 * u + E * k2 + 4 * y) & (N - 1)] = a[4 * u + k2];
                }
            }
        }
        if (it >= 1) {
            // column pass of phase it - 1: sample `slot`, column `col`
            if (it - 1 == nph0) flush(c0, 0);                             // the second channel begins
            long long start;
            const int ns = phase(it - 1, start);
            if (slot < ns) {                                              // warp-uniform: a warp holds 8 columns of a slot
                const float2 *H = Hs + (size_t)((it - 1) & 1) * HB + (size_t)slot * P * NN;
                float2 f[P][E];
#pragma unroll
                for (int p = 0; p < P; p++) {
#pragma unroll
                    for (int m = 0; m < E; m++) {
                        const int y = t + 4 * m;
                        f[p][m] = y < box_h ? H[(size_t)p * NN + y * N + ((col + 4 * y) & (N - 1))] : make_float2(0.f, 0.f);
                    }
                    dft_small<E>(f[p], box_h <= N / 2);
#pragma unroll
                    for (int k = 1; k < E; k++) f[p][k] = hai_fft512::cmul(f[p][k], tw[k]);
                }
#pragma unroll
                for (int p = 0; p < P; p++) finish(f[p]);
#pragma unroll
                for (int k = 0; k < E; k++) {
                    const float2 fx = f[0][k];
                    acc[k][0] = fmaf(fx.x, fx.x, fmaf(fx.y, fx.y, acc[k][0]));
                    if (P == 2) {
                        const float2 fy = f[P - 1][k];
                        acc[k][Q > 1 ? 1 : 0] = fmaf(fy.x, fy.x, fmaf(fy.y, fy.y, acc[k][Q > 1 ? 1 : 0]));
                        acc[k][Q > 2 ? 2 : 0] = fmaf(fx.x, fy.x, fmaf(fx.y, fy.y, acc[k][Q > 2 ? 2 : 0]));
                        acc[k][Q > 3 ? 3 : 0] = fmaf(fx.y, fy.x, fmaf(-fx.x, fy.y, acc[k][Q > 3 ? 3 : 0]));
                    }
                }
            }
        }
        asm volatile("cp.async.wait_all;\n" ::: "memory");
        __syncthreads();
    }
    flush(n1 > 0 ? c0 + 1 : c0, n1 > 0 ? 1 : 0);
}

// img[c] = (accumulate ? img[c] : 0) + sum of the partials of channel c.  CTA
// b covers samples [b*len, (b+1)*len) of the flat index, so only a channel's
// first CTA can hold it in its second slot.  Thread (x, y) of a block adds the
// partials b0 + y, b0 + y + G, ... of V adjacent pixels, and row y = 0 adds
// the G sums in order (deterministic).  A long cadence of few channels has up
// to one partial per SM and channel: with one thread per pixel walking them all
// the loads ran one after another on four SMs, and took longer than the
// imaging they followed; a 64-channel cadence (3 or 4 partials a channel) gains
// from the wider accesses alone (tensor cores at 64^2: 1093.8 -> 1085.9 us).
template <int V>
__global__ void __launch_bounds__(1024) epic_reduce_kernel(const float *__restrict__ part, float *__restrict__ img,
                                                           int T, long long len, int plane, int accumulate) {
    extern __shared__ float red[];                          // [G][blockDim.x][V]
    const int c = blockIdx.y, G = blockDim.y;
    const int i = (blockIdx.x * blockDim.x + threadIdx.x) * V;
    const int b0 = (int)(((long long)c * T) / len);
    const int b1 = (int)(((long long)(c + 1) * T - 1) / len);
    const int slot0 = c - (int)(((long long)b0 * len) / T);
    float s[V];
#pragma unroll
    for (int v = 0; v < V; v++) s[v] = 0.f;
    if (i < plane) {
#pragma unroll 4
        for (int b = b0 + threadIdx.y; b <= b1; b += G) {
            const float *src = part + ((size_t)b * 2 + (b == b0 ? slot0 : 0)) * plane + i;
            if constexpr (V == 4) {
                const float4 x = *reinterpret_cast<const float4 *>(src);
                s[0] += x.x;
                s[1] += x.y;
                s[2] += x.z;
                s[3] += x.w;
            } else {
                s[0] += *src;
            }
        }
    }
    if (G > 1) {
#pragma unroll
        for (int v = 0; v < V; v++) red[(threadIdx.y * blockDim.x + threadIdx.x) * V + v] = s[v];
        __syncthreads();
        if (threadIdx.y > 0) return;
        for (int y = 1; y < G; y++)
#pragma unroll
            for (int v = 0; v < V; v++) s[v] += red[(y * blockDim.x + threadIdx.x) * V + v];
    }
    if (i >= plane) return;
    float *o = img + (size_t)c * plane + i;
    if constexpr (V == 4) {
        float4 x = accumulate ? *reinterpret_cast<const float4 *>(o) : make_float4(0.f, 0.f, 0.f, 0.f);
        x.x += s[0];
        x.y += s[1];
        x.z += s[2];
        x.w += s[3];
        *reinterpret_cast<float4 *>(o) = x;
    } else {
        *o = accumulate ? *o + s[0] : s[0];
    }
}

// Four pixels a thread when the buffers allow 16-byte accesses (planes are
// multiples of 256 floats); G partials side by side while a channel has four
// or more for each and the pixels alone leave SMs without threads.
hai_status reduce_launch(const float *part, float *img, const EpicSplit &sp, int C, int T, int plane, int accumulate,
                         int sms, cudaStream_t st) {
    const bool vec = (((uintptr_t)part | (uintptr_t)img) & 15) == 0;
    const int V = vec ? 4 : 1;
    const long long work = (long long)C * (plane / V), nb = T / sp.len + 2;
    int G = 1;
    while (G < 32 && 4 * G <= nb && work * G < 1024ll * sms) G *= 2;
    const int X = G < 8 ? 256 / G : 32;
    const dim3 grid((plane / V + X - 1) / X, C), block(X, G);
    const size_t smem = G > 1 ? sizeof(float) * V * X * G : 0;
    if (vec)
        epic_reduce_kernel<4><<<grid, block, smem, st>>>(part, img, T, sp.len, plane, accumulate);
    else
        epic_reduce_kernel<1><<<grid, block, smem, st>>>(part, img, T, sp.len, plane, accumulate);
    HAI_CUDA_TRY(cudaGetLastError());
    return HAI_OK;
}

// The N = 16, 32 kernel, the gather table in shared memory if it fits;
// *launched = false if even the voltages do not fit.
template <int N, int P, bool TS>
hai_status try_small(const int8_t *volt, int C, int T, int ne, const EpicSplit &sp, int box_w, int box_h,
                     const int32_t *cstart, const int32_t *celem, const float2 *cw, int nnz, float *dst,
                     int accumulate, int smem_optin, cudaStream_t st, bool *launched) {
    const size_t smem = EpicSmallSmem<N, P, TS>::bytes(ne, box_w * box_h, nnz);
    if (*launched || smem > (size_t)smem_optin) return HAI_OK;
    auto kern = epic_small_kernel<N, P, TS>;
    HAI_CUDA_TRY(hai_allow_dyn_smem(kern, smem_optin));
    kern<<<sp.n_cta, kSmThreads, smem, st>>>(volt, C, T, ne, sp.len, box_w, box_h, cstart, celem, cw, nnz, dst,
                                             sp.direct, accumulate);
    HAI_CUDA_TRY(cudaGetLastError());
    *launched = true;
    return HAI_OK;
}

template <int N, int P>
hai_status launch_small(const int8_t *volt, int C, int T, int ne, const EpicSplit &sp, int box_w, int box_h,
                        const int32_t *cstart, const int32_t *celem, const float2 *cw, int nnz, float *dst,
                        int accumulate, int smem_optin, cudaStream_t st, bool *launched) {
    *launched = false;
    const hai_status s = try_small<N, P, true>(volt, C, T, ne, sp, box_w, box_h, cstart, celem, cw, nnz, dst,
                                               accumulate, smem_optin, st, launched);
    if (s != HAI_OK) return s;
    return try_small<N, P, false>(volt, C, T, ne, sp, box_w, box_h, cstart, celem, cw, nnz, dst, accumulate,
                                  smem_optin, st, launched);
}

// The N = 64 kernel in the form the box and the shared memory allow:
// *launched = false if even the smallest form does not fit (the caller keeps
// the general kernel).
template <int P, bool PX, bool PY, int SP, bool TS>
void launch64_form(const int8_t *volt, int C, int T, int ne, const EpicSplit &sp, int box_w, int box_h,
                   const int32_t *cstart, const int32_t *celem, const float2 *cw, int nnz, float *dst,
                   int accumulate, size_t smem, cudaStream_t st) {
    epic64_kernel<P, PX, PY, SP, TS><<<sp.n_cta, k64Threads, smem, st>>>(
        volt, C, T, ne, sp.len, box_w, box_h, cstart, celem, cw, nnz, dst, sp.direct, accumulate);
}

template <int P, bool PX, bool PY, int SP, bool TS>
hai_status try64(const int8_t *volt, int C, int T, int ne, const EpicSplit &sp, int box_w, int box_h,
                 const int32_t *cstart, const int32_t *celem, const float2 *cw, int nnz, float *dst, int accumulate,
                 int smem_optin, cudaStream_t st, bool *launched) {
    const size_t smem = Epic64Smem<P, PX, PY, SP, TS>::bytes(ne, box_w * box_h, nnz);
    if (*launched || smem > (size_t)smem_optin) return HAI_OK;
    auto kern = epic64_kernel<P, PX, PY, SP, TS>;
    HAI_CUDA_TRY(hai_allow_dyn_smem(kern, smem_optin));
    launch64_form<P, PX, PY, SP, TS>(volt, C, T, ne, sp, box_w, box_h, cstart, celem, cw, nnz, dst, accumulate,
                                     smem, st);
    HAI_CUDA_TRY(cudaGetLastError());
    *launched = true;
    return HAI_OK;
}

// Forms in order of preference: two samples per phase (boxes of at most 32
// rows) with the table in shared memory, then without it; one sample with the
// table (taller boxes); one sample.  One pol: one sample, table in global
// memory.
template <int P, bool PX, bool PY>
hai_status launch64_box(const int8_t *volt, int C, int T, int ne, const EpicSplit &sp, int box_w, int box_h,
                        const int32_t *cstart, const int32_t *celem, const float2 *cw, int nnz, float *dst,
                        int accumulate, int smem_optin, cudaStream_t st, bool *launched) {
    *launched = false;
    if constexpr (P == 1) {       // one pol: the plain forms only
        return try64<P, PX, PY, 1, false>(volt, C, T, ne, sp, box_w, box_h, cstart, celem, cw, nnz, dst, accumulate,
                                          smem_optin, st, launched);
    } else {
#define HAI_TRY64(SPV, TSV)                                                                                    \
    {                                                                                                          \
        const hai_status s_ = try64<P, PX, PY, SPV, TSV>(volt, C, T, ne, sp, box_w, box_h, cstart, celem, cw,  \
                                                         nnz, dst, accumulate, smem_optin, st, launched);      \
        if (s_ != HAI_OK) return s_;                                                                           \
    }
        if constexpr (PY) {
            HAI_TRY64(2, true);
            HAI_TRY64(2, false);
        } else {
            HAI_TRY64(1, true);
        }
        HAI_TRY64(1, false);
#undef HAI_TRY64
        return HAI_OK;
    }
}

template <int P>
hai_status launch64(const int8_t *volt, int C, int T, int ne, const EpicSplit &sp, int box_w, int box_h,
                    const int32_t *cstart, const int32_t *celem, const float2 *cw, int nnz, float *dst,
                    int accumulate, int smem_optin, cudaStream_t st, bool *launched) {
    const bool px = box_w <= 32, py = box_h <= 32;
    if (px && py)
        return launch64_box<P, true, true>(volt, C, T, ne, sp, box_w, box_h, cstart, celem, cw, nnz, dst, accumulate,
                                           smem_optin, st, launched);
    if (px)
        return launch64_box<P, true, false>(volt, C, T, ne, sp, box_w, box_h, cstart, celem, cw, nnz, dst,
                                            accumulate, smem_optin, st, launched);
    if (py)
        return launch64_box<P, false, true>(volt, C, T, ne, sp, box_w, box_h, cstart, celem, cw, nnz, dst,
                                            accumulate, smem_optin, st, launched);
    return launch64_box<P, false, false>(volt, C, T, ne, sp, box_w, box_h, cstart, celem, cw, nnz, dst, accumulate,
                                         smem_optin, st, launched);
}

template <int N, int P>
hai_status launch_n(const hai_layout *L, const int8_t *volt, int C, int T, float *img, int accumulate,
                    cudaStream_t st) {
    const int optin = L->ctx->smem_optin;
    const EpicSplit sp = epic_make_split(C, T, epic_fp32_target_ctas(L->ctx, N));
    if (!sp.direct && (size_t)sp.n_cta * 2 > L->partial_slots)
        return hai_fail(HAI_ERR_INVALID_ARG, "epic fp32: partial buffer too small");
    float *dst = sp.direct ? img : L->d_partials;
    bool launched = false;
    const int pidx = prof_begin(L->ctx, st);
    auto refuse = [&](hai_status s) {
        prof_cancel(L->ctx, pidx);
        return s;
    };
    hai_status s = HAI_OK;
    if constexpr (N == 64)
        s = launch64<P>(volt, C, T, L->n_elem, sp, L->box_w, L->box_h, L->d_cell_start, L->d_entry_elem,
                        L->d_entry_w, L->nnz, dst, accumulate, optin, st, &launched);
    else
        s = launch_small<N, P>(volt, C, T, L->n_elem, sp, L->box_w, L->box_h, L->d_cell_start, L->d_entry_elem,
                               L->d_entry_w, L->nnz, dst, accumulate, optin, st, &launched);
    if (s != HAI_OK) return refuse(s);
    if (!launched) {
        const size_t smem = sizeof(float2) * EpicSmem<N, P>::kBuf +
                            ((size_t)kSamples * P * L->n_elem * 2 + 15) / 16 * 16;
        if (smem > (size_t)optin)
            return refuse(hai_fail(HAI_ERR_UNSUPPORTED, "epic fp32: shared memory need exceeds the device limit"));
        auto kern = epic_fp32_kernel<N, P>;
        HAI_CUDA_TRY(hai_allow_dyn_smem(kern, optin));
        kern<<<sp.n_cta, kThreads, smem, st>>>(volt, C, T, L->n_elem, sp.len, L->box_w, L->box_h,
                                               L->d_cell_start, L->d_entry_elem, L->d_entry_w, dst,
                                               sp.direct, accumulate);
        HAI_CUDA_TRY(cudaGetLastError());
    }
    prof_end(L->ctx, pidx, st);
    prof_count(L->ctx, 1);
    if (!sp.direct) return epic_reduce_launch(L, sp, C, T, img, accumulate, st);
    return HAI_OK;
}

}  // namespace

hai_status epic_fp32_init_tables(void) {
    float2 tw[kTwN / 2];
    for (int m = 0; m < kTwN / 2; m++) {
        const double ang = 2.0 * 3.14159265358979323846 * m / kTwN;
        tw[m] = make_float2((float)cos(ang), (float)sin(ang));
    }
    HAI_CUDA_TRY(cudaMemcpyToSymbol(c_tw, tw, sizeof(tw)));
    return HAI_OK;
}

int epic_fp32_target_ctas(const hai_ctx *ctx, int) { return ctx->num_sms; }

hai_status epic_reduce_launch(const hai_layout *L, const EpicSplit &sp, int C, int T, float *img,
                              int accumulate, cudaStream_t st) {
    const int plane = (L->n_pol == 2 ? 4 : 1) * L->grid_n * L->grid_n;
    const hai_status s = reduce_launch(L->d_partials, img, sp, C, T, plane, accumulate, L->ctx->num_sms, st);
    if (s != HAI_OK) return s;
    prof_count(L->ctx, 1);
    return HAI_OK;
}

hai_status epic_fp32_launch(const hai_layout *L, const int8_t *volt, int C, int T, float *img,
                            int accumulate, cudaStream_t st) {
    const int n = L->grid_n, p = L->n_pol;
    if (n == 16) return p == 2 ? launch_n<16, 2>(L, volt, C, T, img, accumulate, st)
                               : launch_n<16, 1>(L, volt, C, T, img, accumulate, st);
    if (n == 32) return p == 2 ? launch_n<32, 2>(L, volt, C, T, img, accumulate, st)
                               : launch_n<32, 1>(L, volt, C, T, img, accumulate, st);
    if (n == 64) return p == 2 ? launch_n<64, 2>(L, volt, C, T, img, accumulate, st)
                               : launch_n<64, 1>(L, volt, C, T, img, accumulate, st);
    if (epic_large_supported(n)) return epic_large_launch(L, volt, C, T, img, accumulate, st);
    return hai_fail(HAI_ERR_UNSUPPORTED, "epic fp32: grid size");
}

// ============================================================================
// Allocation-free entry point.
//
// hai_layout_create reserves the gather table and the time-split partial
// images with cudaMalloc, so callers that must not allocate device memory
// cannot use hai_epic_image.  This entry point runs the same FP32 kernel with
// both kept in one fixed file-scope device array: the gather table is built
// on the host from the caller's layout description into a static host
// buffer and copied in on the caller's stream, and the partial images of the
// time split live after it.  Every call on a device shares the array (and
// the host buffer), which keeps the last call's contents; nothing in it has
// to start at zero, because each launch rewrites the table and every partial
// image slot it reads.  Calls that overlap on the GPU, or that come from two
// host threads at once, race on it.
// ============================================================================
namespace {

constexpr int kStaticMaxN = 64;                  // grid side
constexpr int kStaticMaxNnz = 102400;            // n_elem x K^2 gather entries
constexpr int kStaticMaxCells = kStaticMaxN * kStaticMaxN;
constexpr int kStaticCtas = 64;                  // CTAs of the time split
// cell starts | elements | (pad to 8 bytes) conj taps as float2, rounded to 16 bytes
constexpr size_t kStaticTableWords = ((size_t)(kStaticMaxCells + 1) + 3 * (size_t)kStaticMaxNnz + 1 + 3) & ~(size_t)3;
constexpr size_t kStaticPartialFloats = 2 * (size_t)kStaticCtas * 4 * kStaticMaxN * kStaticMaxN;
constexpr size_t kStaticFloats = kStaticTableWords + kStaticPartialFloats;   // 2,408,452 (9.2 MiB)
constexpr int kStaticMaxDevices = 64;

static __device__ __align__(256) float g_epic_static_scratch[kStaticFloats];

// host side: device address of the array per device, and the host staging
// buffer of the gather table (cell starts | elements | conj taps)
static float *g_static_ptr[kStaticMaxDevices];
alignas(16) static int32_t g_static_host[kStaticTableWords];
static int32_t g_static_cursor[kStaticMaxCells];

// word offset of the float2 taps inside the table: 8-byte aligned
inline size_t static_taps_word(int ncell, int nnz) { return ((size_t)(ncell + 1) + nnz + 1) & ~(size_t)1; }

hai_status static_scratch(int device, float **out) {
    if (!g_static_ptr[device]) {
        // the host-side name of the array is only a stand-in: fetch the device
        // address once, with this device current; the FFT twiddles live in
        // constant memory that no context has filled yet on this path
        hai_status s = epic_fp32_init_tables();
        if (s != HAI_OK) return s;
        void *p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_epic_static_scratch);
        if (e != cudaSuccess) return hai_cuda_fail(e, "hai_epic_image_fp32_static: cudaGetSymbolAddress");
        g_static_ptr[device] = static_cast<float *>(p);
    }
    *out = g_static_ptr[device];
    return HAI_OK;
}

template <int N, int P>
hai_status launch_static(float *scratch, int ne, int box_w, int box_h, int ncell, int nnz, const int8_t *volt,
                         int C, int T, float *img, int accumulate, int sms, int smem_optin, cudaStream_t st) {
    const EpicSplit sp = epic_make_split(C, T, std::min(sms, kStaticCtas));
    const int32_t *cstart = reinterpret_cast<const int32_t *>(scratch);
    const int32_t *celem = cstart + (ncell + 1);
    const float2 *cw = reinterpret_cast<const float2 *>(cstart + static_taps_word(ncell, nnz));
    float *partials = scratch + kStaticTableWords;
    bool launched = false;
    hai_status s = HAI_OK;
    if constexpr (N == 64)
        s = launch64<P>(volt, C, T, ne, sp, box_w, box_h, cstart, celem, cw, nnz, sp.direct ? img : partials,
                        accumulate, smem_optin, st, &launched);
    else
        s = launch_small<N, P>(volt, C, T, ne, sp, box_w, box_h, cstart, celem, cw, nnz, sp.direct ? img : partials,
                               accumulate, smem_optin, st, &launched);
    if (s != HAI_OK) return s;
    if (!launched) {
        const size_t smem = sizeof(float2) * EpicSmem<N, P>::kBuf + ((size_t)kSamples * P * ne * 2 + 15) / 16 * 16;
        if (smem > (size_t)smem_optin)
            return hai_fail(HAI_ERR_UNSUPPORTED,
                            "hai_epic_image_fp32_static: shared memory need exceeds the device limit");
        auto kern = epic_fp32_kernel<N, P>;
        HAI_CUDA_TRY(hai_allow_dyn_smem(kern, smem_optin));
        kern<<<sp.n_cta, kThreads, smem, st>>>(volt, C, T, ne, sp.len, box_w, box_h, cstart, celem, cw,
                                               sp.direct ? img : partials, sp.direct, accumulate);
        HAI_CUDA_TRY(cudaGetLastError());
    }
    if (!sp.direct) return reduce_launch(partials, img, sp, C, T, (P == 2 ? 4 : 1) * N * N, accumulate, sms, st);
    return HAI_OK;
}

}  // namespace

extern "C" hai_status hai_epic_image_fp32_static(int device, const hai_layout_desc *d, const int8_t *volt, int C,
                                                 int T, float *img, int accumulate, void *stream) {
    if (!d || !d->anchors || !d->taps) return hai_fail(HAI_ERR_INVALID_ARG, "hai_epic_image_fp32_static: NULL argument");
    if (device < 0 || device >= kStaticMaxDevices)
        return hai_fail(HAI_ERR_INVALID_ARG, "hai_epic_image_fp32_static: device index out of range");
    if (d->n_elem <= 0 || d->ksize <= 0 || (d->n_pol != 1 && d->n_pol != 2) || C < 0 || T < 0 ||
        (accumulate != 0 && accumulate != 1))
        return hai_fail(HAI_ERR_INVALID_ARG, "hai_epic_image_fp32_static: bad descriptor or size");
    const int n = d->grid_n, k = d->ksize, ne = d->n_elem;
    if (n != 16 && n != 32 && n != 64)
        return hai_fail(HAI_ERR_UNSUPPORTED, "hai_epic_image_fp32_static: grid_n must be 16, 32 or 64");
    if ((long long)ne * k * k > kStaticMaxNnz)
        return hai_fail(HAI_ERR_UNSUPPORTED, "hai_epic_image_fp32_static: n_elem * ksize^2 exceeds the static "
                                             "scratch maximum of 102400 gather entries");
    int bx0 = n, by0 = n, bx1 = 0, by1 = 0;
    for (int a = 0; a < ne; a++) {
        const int x0 = d->anchors[2 * a], y0 = d->anchors[2 * a + 1];
        if (x0 < 0 || y0 < 0 || (long)x0 + k > n || (long)y0 + k > n)
            return hai_fail(HAI_ERR_OFF_GRID, "hai_epic_image_fp32_static: a kernel tap lies outside the grid");
        bx0 = std::min(bx0, x0);
        by0 = std::min(by0, y0);
        bx1 = std::max(bx1, x0 + k);
        by1 = std::max(by1, y0 + k);
    }
    if (C == 0) return HAI_OK;
    if (!img || (T > 0 && !volt)) return hai_fail(HAI_ERR_INVALID_ARG, "hai_epic_image_fp32_static: NULL buffer");
    if ((((uintptr_t)volt) & 1) || (((uintptr_t)img) & 3))
        return hai_fail(HAI_ERR_INVALID_ARG, "hai_epic_image_fp32_static: volt must be 2-byte and img 4-byte aligned");
    HAI_CUDA_TRY(cudaSetDevice(device));
    cudaStream_t st = (cudaStream_t)stream;
    const int Q = (d->n_pol == 2) ? 4 : 1;
    if (T == 0) {
        if (!accumulate) HAI_CUDA_TRY(cudaMemsetAsync(img, 0, sizeof(float) * (size_t)C * Q * n * n, st));
        return HAI_OK;
    }
    float *scratch = nullptr;
    hai_status s = static_scratch(device, &scratch);
    if (s != HAI_OK) return s;
    // gather table, same order as hai_layout_create: cells of the box row-major,
    // entries by element, weights conj(W~)
    const int box_w = bx1 - bx0, box_h = by1 - by0, ncell = box_w * box_h;
    const int nnz = ne * k * k;
    int32_t *cstart = g_static_host;
    int32_t *celem = cstart + (ncell + 1);
    float2 *cw = reinterpret_cast<float2 *>(cstart + static_taps_word(ncell, nnz));
    for (int i = 0; i <= ncell; i++) cstart[i] = 0;
    for (int a = 0; a < ne; a++)
        for (int v = 0; v < k; v++)
            for (int u = 0; u < k; u++) cstart[(d->anchors[2 * a + 1] + v - by0) * box_w + (d->anchors[2 * a] + u - bx0) + 1]++;
    for (int i = 0; i < ncell; i++) cstart[i + 1] += cstart[i];
    for (int i = 0; i < ncell; i++) g_static_cursor[i] = cstart[i];
    for (int a = 0; a < ne; a++)
        for (int v = 0; v < k; v++)
            for (int u = 0; u < k; u++) {
                const int cell = (d->anchors[2 * a + 1] + v - by0) * box_w + (d->anchors[2 * a] + u - bx0);
                const float *t = d->taps + (((size_t)a * k + v) * k + u) * 2;
                const int slot = g_static_cursor[cell]++;
                celem[slot] = a;
                cw[slot] = make_float2(t[0], -t[1]);
            }
    const size_t words = static_taps_word(ncell, nnz) + 2 * (size_t)nnz;
    HAI_CUDA_TRY(cudaMemcpyAsync(scratch, g_static_host, sizeof(int32_t) * words, cudaMemcpyHostToDevice, st));
    int sms = 0, optin = 0;
    HAI_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device));
    HAI_CUDA_TRY(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device));
    const int p = d->n_pol;
#define HAI_STATIC_CASE(NN)                                                                                        \
    if (n == NN)                                                                                                   \
        return p == 2 ? launch_static<NN, 2>(scratch, ne, box_w, box_h, ncell, nnz, volt, C, T, img, accumulate, \
                                             sms, optin, st)                                                      \
                      : launch_static<NN, 1>(scratch, ne, box_w, box_h, ncell, nnz, volt, C, T, img, accumulate, \
                                             sms, optin, st);
    HAI_STATIC_CASE(16)
    HAI_STATIC_CASE(32)
    HAI_STATIC_CASE(64)
#undef HAI_STATIC_CASE
    return hai_fail(HAI_ERR_UNSUPPORTED, "hai_epic_image_fp32_static: grid size");
}
