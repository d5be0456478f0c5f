// FFT correlator (Section 4.1.2 and Section 5.2.2: visibilities obtained from
// the accumulated EPIC images by an inverse FFT).
//
// The accumulated image I_ab[l] = sum_t F_a[l] conj(F_b[l]) is the DFT (+) of
// the circular autocorrelation of the checkerboarded grids (-1)^j G[j], so
//   R_ab[d] = (-1)^(dx+dy) / N^2  sum_l I_ab[l] exp(-2 pi i l.d / N)
// is the grid sum_t sum_j G_a[j + d] conj(G_b[j]) at lag d, the same grid the
// correlator + XFFT path fills with V_ab K_ab[d] (zero lag at cell (0, 0)).
// On a lattice with one unit tap per element every lag holds the plain sum of
// the visibilities of the baselines separated by it.
//
// Two passes over the output buffer, which holds the rows in between:
//   rows:    one warp per (channel, product, row): the row of the real XX /
//            YY plane or of the complex XY plane, radix-2 FFT (exponent -)
//            in shared memory, complex row written to the output plane;
//   columns: one CTA per (channel, product, 16 columns), one warp per
//            column: FFT along y, times (-1)^(dx+dy) / N^2, written back; the
//            XY CTA also writes YX[-d] = conj(XY[d]) (I_YX = conj(I_XY)).
// N = 512 keeps each line in registers instead: 64 threads per line, three
// radix-8 passes and two shared-memory exchanges (fft512.cuh), the inverse
// transform taken as conj(FFT(conj(x))); 8 lines per CTA in both passes.  The XX
// and YY images are real, so their rows go two to a transform, only columns 0 ..
// 256 are kept between the passes, and the column pass writes the others as
// R[-d] = conj(R[d]).  Persistent CTAs build the twiddle tables once.  16 channels
// of the lattice: every product as a complex image, tables built by every CTA
// (3,072 a pass), 39 + 57 us; 28 + 52 us now (bound: L2 and the exchanges'
// barriers; 335 MB cross L2 where the image and the grid alone are 201).
#include <algorithm>

#include "fft512.cuh"
#include "hai_internal.h"

namespace {

constexpr int kThreads = 512;
constexpr int kCols = 16;                 // columns per column CTA = warps per CTA

__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}

// Twiddles exp(-2 pi i k / N), k < N / 2.
__device__ __forceinline__ void fill_twiddles(float2 *tw, int N) {
    for (int k = threadIdx.x; k < N / 2; k += blockDim.x) {
        float s, c;
        sincospif(2.0f * (float)k / (float)N, &s, &c);
        tw[k] = make_float2(c, -s);
    }
}

// In-place radix-2 FFT (exponent -) of N points held in bit-reversed order,
// by one warp, with the twiddle table of length N / 2.
__device__ __forceinline__ void warp_ifft(float2 *x, int n, int log2n, const float2 *tw, int lane) {
    for (int s = 0; s < log2n; s++) {
        const int half = 1 << s;
        const int tstep = n >> (s + 1);
        for (int b = lane; b < n / 2; b += 32) {
            const int pos = b & (half - 1);
            const int i0 = ((b - pos) << 1) + pos, i1 = i0 + half;
            const float2 a = x[i0];
            const float2 t = cmul(x[i1], tw[pos * tstep]);
            x[i0] = make_float2(a.x + t.x, a.y + t.y);
            x[i1] = make_float2(a.x - t.x, a.y - t.y);
        }
        __syncwarp();
    }
}

// Output plane (polarisation pair index alpha * P + beta) of source product
// pr (0 = XX, 1 = YY, 2 = XY).
__device__ __forceinline__ int out_plane(int pr, int P) { return P == 1 ? 0 : (pr == 0 ? 0 : (pr == 1 ? 3 : 1)); }

__global__ void __launch_bounds__(kThreads) fc_rows_kernel(const float *__restrict__ img, int N, int log2n, int P,
                                                           float2 *__restrict__ out) {
    extern __shared__ float2 sm[];
    float2 *tw = sm;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float2 *line = sm + N / 2 + (size_t)warp * N;
    fill_twiddles(tw, N);
    __syncthreads();
    const int np = (P == 2) ? 3 : 1, Q = (P == 2) ? 4 : 1;
    const int c = blockIdx.x / np, pr = blockIdx.x % np;
    const int y = blockIdx.y * (kThreads / 32) + warp;
    if (y >= N) return;
    const size_t NN = (size_t)N * N;
    const float *re = img + ((size_t)c * Q + (pr == 2 ? 2 : pr)) * NN + (size_t)y * N;
    const float *im = (pr == 2) ? re + NN : nullptr;
    // lane takes N / 32 consecutive points: their bit-reversed slots for one
    // step are a permutation of 32 adjacent entries (no bank conflicts; points
    // x = lane + 32 k would put the lanes N / 32 entries apart)
    if (N >= 32) {
        const int E = N / 32;
        for (int k = 0; k < E; k++) {
            const int x = E * lane + k;
            line[__brev(x) >> (32 - log2n)] = make_float2(__ldg(re + x), im ? __ldg(im + x) : 0.f);
        }
    } else {
        for (int x = lane; x < N; x += 32)
            line[__brev(x) >> (32 - log2n)] = make_float2(__ldg(re + x), im ? __ldg(im + x) : 0.f);
    }
    __syncwarp();
    warp_ifft(line, N, log2n, tw, lane);
    float2 *dst = out + ((size_t)c * P * P + out_plane(pr, P)) * NN + (size_t)y * N;
    for (int x = lane; x < N; x += 32) dst[x] = line[x];
}

__global__ void __launch_bounds__(kThreads) fc_cols_kernel(int N, int log2n, int P, float2 *__restrict__ out) {
    extern __shared__ float2 sm[];
    float2 *tw = sm;
    float2 *F = sm + N / 2;                         // [kCols][N + 1]: the pad spreads the columns over the banks
    const int Fs = N + 1;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    fill_twiddles(tw, N);
    const int np = (P == 2) ? 3 : 1;
    const int c = blockIdx.x / np, pr = blockIdx.x % np;
    const int x0 = blockIdx.y * kCols;
    const size_t NN = (size_t)N * N;
    float2 *plane = out + ((size_t)c * P * P + out_plane(pr, P)) * NN;
    for (int i = threadIdx.x; i < N * kCols; i += kThreads) {
        const int j = i % kCols, y = i / kCols;
        F[(size_t)j * Fs + (__brev(y) >> (32 - log2n))] = plane[(size_t)y * N + x0 + j];
    }
    __syncthreads();
    warp_ifft(F + (size_t)warp * Fs, N, log2n, tw, lane);
    __syncthreads();
    const float inv = 1.0f / (float)NN;
    float2 *mirror = (pr == 2) ? out + ((size_t)c * P * P + 2) * NN : nullptr;   // YX
    for (int i = threadIdx.x; i < N * kCols; i += kThreads) {
        const int j = i % kCols, dy = i / kCols, dx = x0 + j;
        const float s = ((dx + dy) & 1) ? -inv : inv;
        const float2 v = F[(size_t)j * Fs + dy];
        const float2 r = make_float2(v.x * s, v.y * s);
        plane[(size_t)dy * N + dx] = r;
        if (mirror) mirror[(size_t)((N - dy) & (N - 1)) * N + ((N - dx) & (N - 1))] = make_float2(r.x, -r.y);
    }
}

// N = 512: items of a channel in each pass.  Rows: 32 of 16 rows for each of XX
// and YY, 64 of 8 rows for XY.  Columns: 33 of 8 columns (0 .. 256) for each of
// XX and YY, 64 for XY.
__host__ __device__ constexpr int fc512_items(int P, bool cols) { return P == 2 ? (cols ? 33 + 33 + 64 : 32 + 32 + 64) : cols ? 33 : 32; }

// Rows: thread (r, tau) of line r.  A real plane's line holds rows y, y + 1 as
// z = (row_y, row_y+1), whose transform splits into X_y[k] = (Z[k] + conj Z[-k])
// / 2 and X_y+1[k] = (Z[k] - conj Z[-k]) / 2i.
__global__ void __launch_bounds__(512, 3) fc512_rows_kernel(const float *__restrict__ img, int P, int C,
                                                            float2 *__restrict__ out) {
    constexpr int N = 512;
    extern __shared__ float2 sm[];
    float2 *tw = sm;                                          // [kTwFloat2]
    hai_fft512::fill_fft512_tables(tw);
    __syncthreads();
    const int r = threadIdx.x >> 6, tau = threadIdx.x & 63;
    float2 *buf = sm + hai_fft512::kTwFloat2 + r * hai_fft512::kFftBuf;
    const int per = fc512_items(P, false), Q = (P == 2) ? 4 : 1;
    const size_t NN = (size_t)N * N;
    for (int it = blockIdx.x; it < C * per; it += gridDim.x) {
        const int c = it / per, k = it % per, pr = k >> 5 > 2 ? 2 : k >> 5;
        const bool real = pr < 2;
        const int y = real ? 16 * (k & 31) + 2 * r : 8 * (k - 64) + r;
        // second component: the next row (real plane), or the next plane
        const float *re = img + ((size_t)c * Q + pr) * NN + (size_t)y * N, *im = re + (real ? N : NN);
        float2 a[8];
#pragma unroll
        for (int m = 0; m < 8; m++)                           // conj of the input: exponent -
            a[m] = make_float2(__ldg(re + tau + 64 * m), -__ldg(im + tau + 64 * m));
        hai_fft512::fft512<false>(a, tau, buf, tw, [] { __syncthreads(); });
        float2 *dst = out + ((size_t)c * P * P + out_plane(pr, P)) * NN + (size_t)y * N;
        if (!real) {                                          // CTA-uniform
#pragma unroll
            for (int j = 0; j < 8; j++) dst[tau + 64 * j] = make_float2(a[j].x, -a[j].y);
            __syncthreads();
            continue;
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < 8; j++) buf[tau + 64 * j] = make_float2(a[j].x, -a[j].y);
        __syncthreads();
#pragma unroll
        for (int j = 0; j < 5; j++) {
            const int kx = tau + 64 * j;
            if (kx > N / 2) break;
            const float2 z = buf[kx], w = buf[(N - kx) & (N - 1)];
            dst[kx] = make_float2(0.5f * (z.x + w.x), 0.5f * (z.y - w.y));
            dst[N + kx] = make_float2(0.5f * (z.y + w.y), 0.5f * (w.x - z.x));
        }
        __syncthreads();
    }
}

// N = 512, columns: CTA = 8 adjacent columns of one (channel, product).  The
// columns move between HBM and the registers through a shared tile [8][kTs]
// (which shares its memory with the exchange buffers): loads and stores of
// whole 64-byte row segments (a warp: 4 rows x 8 columns), and tile reads and
// writes of one column's rows by consecutive threads, both free of bank
// conflicts (kTs = 514: columns 4 banks apart).  Thread (col, tau) transforms
// its column; times (-1)^(dx+dy) / N^2; the XY CTA also writes the YX mirror.
constexpr int kTs = 514;

__global__ void __launch_bounds__(512, 3) fc512_cols_kernel(int P, int C, float2 *__restrict__ out) {
    constexpr int N = 512;
    extern __shared__ float2 sm[];
    float2 *tw = sm;
    float2 *bufs = sm + hai_fft512::kTwFloat2;                // exchange buffers, and the column tile
    float2 *tile = bufs;
    static_assert(8 * kTs <= 8 * hai_fft512::kFftBuf, "tile inside the exchange buffers");
    hai_fft512::fill_fft512_tables(tw);
    __syncthreads();
    const int col = threadIdx.x >> 6, tau = threadIdx.x & 63;
    const int lc = threadIdx.x & 7, lr = threadIdx.x >> 3;     // row-segment mapping: column, row of 64
    const int per = fc512_items(P, true);
    const size_t NN = (size_t)N * N;
    const float inv = 1.0f / (float)NN;
    for (int it = blockIdx.x; it < C * per; it += gridDim.x) {
        const int c = it / per, k0 = it % per, pr = k0 < 33 ? 0 : k0 < 66 ? 1 : 2;
        const bool real = pr < 2;
        const int x0 = 8 * (k0 - 33 * pr);
        const int ncol = real ? min(8, N / 2 + 1 - x0) : 8;
        float2 *plane = out + ((size_t)c * P * P + out_plane(pr, P)) * NN;
        float2 *mirror = real ? plane : out + ((size_t)c * P * P + 2) * NN;
        if (lc < ncol) {
#pragma unroll
            for (int k = 0; k < 8; k++) {
                const int y = lr + 64 * k;
                tile[lc * kTs + y] = plane[(size_t)y * N + x0 + lc];
            }
        }
        __syncthreads();
        float2 a[8];
#pragma unroll
        for (int m = 0; m < 8; m++) {                         // conj of the input: exponent -
            const float2 v = col < ncol ? tile[col * kTs + tau + 64 * m] : make_float2(0.f, 0.f);
            a[m] = make_float2(v.x, -v.y);
        }
        __syncthreads();
        hai_fft512::fft512<false>(a, tau, bufs + col * hai_fft512::kFftBuf, tw, [] { __syncthreads(); });
        __syncthreads();                                      // exchange buffers free: the tile again
        const int dxc = x0 + col;
#pragma unroll
        for (int j = 0; j < 8; j++) {
            const int dy = tau + 64 * j;
            const float s = ((dxc + dy) & 1) ? -inv : inv;
            tile[col * kTs + dy] = make_float2(a[j].x * s, -a[j].y * s);
        }
        __syncthreads();
        const int dx = x0 + lc;
        if (lc < ncol) {
            const bool twin = !real || (dx != 0 && dx != N / 2);
#pragma unroll
            for (int k = 0; k < 8; k++) {
                const int dy = lr + 64 * k;
                const float2 v = tile[lc * kTs + dy];
                plane[(size_t)dy * N + dx] = v;
                if (twin) mirror[(size_t)((N - dy) & (N - 1)) * N + ((N - dx) & (N - 1))] = make_float2(v.x, -v.y);
            }
        }
        __syncthreads();
    }
}

}  // namespace

extern "C" hai_status hai_fft_correlate(hai_ctx *ctx, const float *img, int C, int N, int P, float *grid,
                                        void *stream) {
    if (!ctx) return hai_fail(HAI_ERR_INVALID_ARG, "hai_fft_correlate: NULL ctx");
    if (C < 0 || (P != 1 && P != 2)) return hai_fail(HAI_ERR_INVALID_ARG, "hai_fft_correlate: bad C or P");
    int log2n = 0;
    while ((1 << log2n) < N && log2n < 30) log2n++;
    if (N < 16 || N > 512 || (1 << log2n) != N)
        return hai_fail(HAI_ERR_UNSUPPORTED, "hai_fft_correlate: N must be a power of two in [16, 512]");
    if (C == 0) return HAI_OK;
    if (!img || !grid) return hai_fail(HAI_ERR_INVALID_ARG, "hai_fft_correlate: NULL buffer");
    if ((reinterpret_cast<uintptr_t>(img) & 3) || (reinterpret_cast<uintptr_t>(grid) & 7))
        return hai_fail(HAI_ERR_INVALID_ARG, "hai_fft_correlate: img must be 4-byte and grid 8-byte aligned");
    if (hai_fault_injected("launch")) return hai_fail(HAI_ERR_CUDA, "hai_fft_correlate: injected launch failure");
    HAI_CUDA_TRY(cudaSetDevice(ctx->device));
    cudaStream_t st = (cudaStream_t)stream;
    float2 *out = reinterpret_cast<float2 *>(grid);
    if (N == 512) {
        const size_t smem512 = sizeof(float2) * (hai_fft512::kTwFloat2 + 8 * (size_t)hai_fft512::kFftBuf);
        HAI_CUDA_TRY(hai_allow_dyn_smem(fc512_rows_kernel, ctx->smem_optin));
        HAI_CUDA_TRY(hai_allow_dyn_smem(fc512_cols_kernel, ctx->smem_optin));
        if ((long long)C * fc512_items(P, true) > 0x7fffffffll)
            return hai_fail(HAI_ERR_UNSUPPORTED, "hai_fft_correlate: too many channels");
        const int pidx = prof_begin(ctx, st);
        const int resident = 3 * ctx->num_sms;
        fc512_rows_kernel<<<std::min(resident, C * fc512_items(P, false)), 512, smem512, st>>>(img, P, C, out);
        fc512_cols_kernel<<<std::min(resident, C * fc512_items(P, true)), 512, smem512, st>>>(P, C, out);
        prof_end(ctx, pidx, st);
        prof_count(ctx, 2);
        HAI_CUDA_TRY(cudaGetLastError());
        return HAI_OK;
    }
    const int np = (P == 2) ? 3 : 1;
    const size_t smem = sizeof(float2) * ((size_t)N / 2 + (size_t)kCols * (N + 1));   // both passes
    HAI_CUDA_TRY(hai_allow_dyn_smem(fc_rows_kernel, ctx->smem_optin));
    HAI_CUDA_TRY(hai_allow_dyn_smem(fc_cols_kernel, ctx->smem_optin));
    const int pidx = prof_begin(ctx, st);
    fc_rows_kernel<<<dim3(C * np, (N + kThreads / 32 - 1) / (kThreads / 32)), kThreads, smem, st>>>(img, N, log2n,
                                                                                                     P, out);
    fc_cols_kernel<<<dim3(C * np, N / kCols), kThreads, smem, st>>>(N, log2n, P, out);
    prof_end(ctx, pidx, st);
    prof_count(ctx, 2);
    HAI_CUDA_TRY(cudaGetLastError());
    return HAI_OK;
}
