// Correlator + FFT imager (Eq. intra-station XFFT).
//
// For every ordered element pair (a, b), autos included, the visibility
// V^{alpha beta}_{ab} is gridded with the autocorrelation of the two elements'
// illumination kernels, K_ab[d] = sum_j g_a[j + d] conj(g_b[j]) with g the
// placed conjugate taps, at lags d = (anchor_a - anchor_b) + (ex, ey),
// |ex|, |ey| < K, on the circular N grid; then the grid is multiplied by
// (-1)^(dx+dy) and transformed with exp(+2 pi i l.d / N).  With this kernel
// the result equals the EPIC image of the same voltages.
//
// Only the lower triangle a >= b is stored; the pair (b, a) contributes
// conj(V^{beta alpha}_{ab} K_ab[d]) at lag -d (Hermitian mirror).
//
// K_ab and the cells it lands on depend on the layout only.  On a layout's
// first call the footprints of K_ab (2K - 1 cells a side, stored pairs only) are
// binned to patches of 4 x 2 cells of the circular grid, and their values on
// every cell of a patch are computed on the GPU; the imaging is then two kernels
// per batch of channels:
//   gather: a warp holds a patch's 8 cells of 32 channels in registers (a lane
//           per channel), the sums D of all four products (XX, XY, YX, YY) over
//           the stored pairs, and walks the patch's records, the record's 8
//           coefficients the same for all lanes;
//   FFT:    one CTA per (channel, product) adds the mirrors' part as it loads
//           the grid, G_XX[d] = D_XX[d] + conj(D_XX[-d]) and G_XY[d] = D_XY[d] +
//           conj(D_YX[-d]) (autos enter D with half their weight), applies the
//           (-1)^(dx+dy) checkerboard and transforms rows then columns in
//           registers (fft_line.cuh) into the image planes.
// The polarisations keep their own sums and transforms throughout, so a weak
// one loses nothing to a strong one.  Sums run in a fixed order: deterministic.
#include <math.h>

#include <algorithm>
#include <vector>

#include "fft_line.cuh"
#include "hai_internal.h"

namespace {

constexpr int kPw = 4, kPh = 2, kPcells = kPw * kPh;   // patch sides, cells
constexpr int kChunk = 256;                       // records of one patch that a CTA sums
constexpr int kGatherWarps = 8;
constexpr uint32_t kAuto = 1u << 30;              // record flag beside the stored pair's index

// One chunk: records [q0, q1) of a patch.
struct Chunk {
    int32_t patch, q0, q1;
};

// Coefficients of the records: the value of K_ab on every cell of the record's
// patch, summed over the lags that fall on the cell of the circular grid; half
// of it for an auto (which is its own mirror); only real parts for a layout of
// real taps.
template <bool REAL>
__global__ void __launch_bounds__(256) xfft_coef_kernel(const Chunk *__restrict__ chunks, const uint32_t *__restrict__ rec,
                                                        const int32_t *__restrict__ anchors,
                                                        const float2 *__restrict__ taps, int N, int K,
                                                        float *__restrict__ coef) {
    const Chunk ch = chunks[blockIdx.x];
    const int npx = N / kPw, W = 2 * K - 1;
    for (int i = threadIdx.x; i < (ch.q1 - ch.q0) * kPcells; i += blockDim.x) {
        const int q = ch.q0 + i / kPcells, cell = i % kPcells;
        const uint32_t r = rec[q];
        const long long bl = r & (kAuto - 1);
        int a = (int)((sqrt(8.0 * (double)bl + 1.0) - 1.0) * 0.5);
        while ((long long)(a + 1) * (a + 2) / 2 <= bl) a++;
        while ((long long)a * (a + 1) / 2 > bl) a--;
        const int b = (int)(bl - (long long)a * (a + 1) / 2);
        const int x = ch.patch % npx * kPw + cell % kPw, y = ch.patch / npx * kPh + cell / kPw;
        const int dx = anchors[2 * a] - anchors[2 * b], dy = anchors[2 * a + 1] - anchors[2 * b + 1];
        const float2 *ta = taps + (size_t)a * K * K, *tb = taps + (size_t)b * K * K;
        float2 k = make_float2(0.f, 0.f);
        // every lag (ex, ey) in (-K, K)^2 congruent to the cell
        for (int ey = ((y - dy + K - 1) & (N - 1)) - (K - 1); ey <= W - K; ey += N)
            for (int ex = ((x - dx + K - 1) & (N - 1)) - (K - 1); ex <= W - K; ex += N)
                for (int vb = max(0, -ey); vb < min(K, K - ey); vb++)
                    for (int ub = max(0, -ex); ub < min(K, K - ex); ub++) {
                        // sum over tap pairs with (ua - ub, va - vb) = e of conj(w_a) w_b
                        const float2 wa = ta[(vb + ey) * K + (ub + ex)], wb = tb[vb * K + ub];
                        k.x += wa.x * wb.x + wa.y * wb.y;
                        k.y += wa.x * wb.y - wa.y * wb.x;
                    }
        const float half = r & kAuto ? 0.5f : 1.f;
        if (REAL) coef[(size_t)q * kPcells + cell] = half * k.x;
        else reinterpret_cast<float2 *>(coef)[(size_t)q * kPcells + cell] = make_float2(half * k.x, half * k.y);
    }
}

// Partial sums of one chunk for 32 channels: part[product][channel][chunk][8
// cells] (XX, XY, YX, YY, or XX alone for one pol).  The warps take the chunk's
// records in turn and their sums are added in warp order.  An auto's XX and YY
// are real and its YX is conj(XY) in what the correlator writes; only those
// parts enter, as only they reach the image.
//
// The work is 8 (real taps) complex multiply-adds a record, lane and product, on
// operands that are uniform (coefficients) or one 32-byte sector a lane (a
// pair's products of one channel): bound by issue, then L2.  A per-cell list
// walked by threads over (channel, product), after a transpose of the
// visibilities, read each pair's products for each of its 25 cells: 583 us
// after a 37 us transpose for the 64 channels of a 256-element station, now
// 141 us.  A chunk of 256 records keeps the patches around zero lag,
// which hold several thousand, from setting the time.
template <int P, bool REAL, bool VEC>
__global__ void __launch_bounds__(32 * kGatherWarps, 2) xfft_gather_kernel(
    const int32_t *__restrict__ vis, long long nbl, int c0, int cb, const Chunk *__restrict__ chunks, int nchunk,
    const uint32_t *__restrict__ rec, const float *__restrict__ coef, float2 *__restrict__ part) {
    constexpr int H = P * P;                           // products
    extern __shared__ float2 sums[];                   // [warps][H][8][33]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const Chunk ch = chunks[blockIdx.x];
    const int cg = blockIdx.y * 32, c = min(cg + lane, cb - 1);
    const int32_t *v = vis + (size_t)(c0 + c) * nbl * (2 * H);
    float2 acc[H][kPcells];
#pragma unroll
    for (int h = 0; h < H; h++)
#pragma unroll
        for (int i = 0; i < kPcells; i++) acc[h][i] = make_float2(0.f, 0.f);
    constexpr int D = 2;                               // records in flight per warp
    for (int q = ch.q0 + warp; q < ch.q1; q += D * kGatherWarps) {
        uint32_t r[D];
        int4 va[D], vb[D];
#pragma unroll
        for (int d = 0; d < D; d++) r[d] = __ldg(rec + min(q + d * kGatherWarps, ch.q1 - 1));
#pragma unroll
        for (int d = 0; d < D; d++) {
            const int32_t *p = v + (size_t)(r[d] & (kAuto - 1)) * (2 * H);
            if (P == 1) {
                const int2 x = __ldg(reinterpret_cast<const int2 *>(p));
                va[d] = make_int4(x.x, x.y, 0, 0);
            } else if (VEC) {
                va[d] = __ldg(reinterpret_cast<const int4 *>(p));
                vb[d] = __ldg(reinterpret_cast<const int4 *>(p) + 1);
            } else {
                const int2 *w = reinterpret_cast<const int2 *>(p);
                const int2 x = __ldg(w), y = __ldg(w + 1), z = __ldg(w + 2), u = __ldg(w + 3);
                va[d] = make_int4(x.x, x.y, y.x, y.y);
                vb[d] = make_int4(z.x, z.y, u.x, u.y);
            }
        }
#pragma unroll
        for (int d = 0; d < D; d++) {
            const int qd = q + d * kGatherWarps;
            if (qd >= ch.q1) break;
            const bool self = r[d] & kAuto;
            float2 g[H];
            g[0] = make_float2((float)va[d].x, self ? 0.f : (float)va[d].y);
            if (P == 2) {
                g[H > 1 ? 1 : 0] = make_float2((float)va[d].z, (float)va[d].w);
                g[H > 2 ? 2 : 0] = self ? make_float2((float)va[d].z, -(float)va[d].w) : make_float2((float)vb[d].x, (float)vb[d].y);
                g[H - 1] = make_float2((float)vb[d].z, self ? 0.f : (float)vb[d].w);
            }
            const float4 *cf = reinterpret_cast<const float4 *>(coef) + (size_t)qd * (REAL ? 2 : 4);
#pragma unroll
            for (int j = 0; j < (REAL ? 2 : 4); j++) {
                const float4 k = __ldg(cf + j);
                if (REAL) {
                    const float kk[4] = {k.x, k.y, k.z, k.w};
#pragma unroll
                    for (int i = 0; i < 4; i++)
#pragma unroll
                        for (int h = 0; h < H; h++)
                            acc[h][4 * j + i] = __ffma2_rn(make_float2(kk[i], kk[i]), g[h], acc[h][4 * j + i]);
                } else {
#pragma unroll
                    for (int i = 0; i < 2; i++) {
                        const float kr = i ? k.z : k.x, ki = i ? k.w : k.y;
#pragma unroll
                        for (int h = 0; h < H; h++) {
                            float2 &a = acc[h][2 * j + i];
                            a.x = fmaf(kr, g[h].x, fmaf(-ki, g[h].y, a.x));
                            a.y = fmaf(kr, g[h].y, fmaf(ki, g[h].x, a.y));
                        }
                    }
                }
            }
        }
    }
#pragma unroll
    for (int h = 0; h < H; h++)
#pragma unroll
        for (int i = 0; i < kPcells; i++) sums[((warp * H + h) * kPcells + i) * 33 + lane] = acc[h][i];
    __syncthreads();
    for (int i = threadIdx.x; i < H * 32 * kPcells; i += 32 * kGatherWarps) {
        const int cell = i % kPcells, l = i / kPcells % 32, h = i / (kPcells * 32);
        if (cg + l >= cb) continue;
        float2 t = sums[(h * kPcells + cell) * 33 + l];
#pragma unroll
        for (int w = 1; w < kGatherWarps; w++) {
            const float2 u = sums[((w * H + h) * kPcells + cell) * 33 + l];
            t.x += u.x;
            t.y += u.y;
        }
        part[(((size_t)h * cb + cg + l) * nchunk + blockIdx.x) * kPcells + cell] = t;
    }
}

// One CTA per (channel, image product h = XX, YY, XY): the cells' partial sums
// (in chunk order), each added to its own cell and, conjugated, to the mirrored
// one; checkerboard, rows, columns.  XX, YY -> their plane (the transform is
// real), XY -> Re XY, Im XY.  Lines in registers, exchanged in their own row or
// column of the shared tile; the row stride keeps a half-warp's rows on distinct
// banks.
template <int N>
__global__ void __launch_bounds__(N *hai_fft::Line<N>::L) xfft_fft_kernel(const float2 *__restrict__ part,
                                                                         const int32_t *__restrict__ pstart, int nchunk,
                                                                         int cb, int P, int c0, float *__restrict__ img,
                                                                         int accumulate) {
    constexpr int L = hai_fft::Line<N>::L, E = hai_fft::Line<N>::E, S = N + (L == 8 ? 8 : 4), NT = N * L;
    __shared__ float2 sm[N * S], tw[N];
    const int c = blockIdx.x, h = blockIdx.y, tid = threadIdx.x;
    hai_fft::fill_twiddles<N>(tw);
    // products of the pair and of its mirror: XX, XX; YY, YY; XY, YX
    const int hd = h == 0 ? 0 : h == 1 ? 3 : 1, hm = h == 2 ? 2 : hd;
    auto sum = [&](int prod, int i) {                 // cell i in patch order: 64-byte runs
        const float2 *src = part + ((size_t)prod * cb + c) * nchunk * kPcells + i % kPcells;
        float2 s = make_float2(0.f, 0.f);
        for (int q = pstart[i / kPcells]; q < pstart[i / kPcells + 1]; q++) {
            const float2 v = src[(size_t)q * kPcells];
            s.x += v.x;
            s.y += v.y;
        }
        return s;
    };
    auto at = [&](int i, int &x, int &y) {
        const int p = i / kPcells, cell = i % kPcells;
        x = p % (N / kPw) * kPw + cell % kPw;
        y = p / (N / kPw) * kPh + cell / kPw;
    };
    for (int i = tid; i < N * N; i += NT) {
        int x, y;
        at(i, x, y);
        sm[y * S + x] = sum(hd, i);
    }
    __syncthreads();
    // the mirrored cell's value: from the tile before it is overwritten (XX,
    // YY), or from the YX sums; signs with the checkerboard (the same for d, -d)
    constexpr int kC = N * N / NT;
    float2 m[kC];
#pragma unroll
    for (int k = 0; k < kC; k++) {
        int x, y;
        at(tid + k * NT, x, y);
        const int j = ((N - y) & (N - 1)) * S + ((N - x) & (N - 1));
        if (h < 2) m[k] = sm[j];
        else m[k] = sum(hm, tid + k * NT);
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kC; k++) {
        int x, y;
        at(tid + k * NT, x, y);
        // XX, YY: own cell += conj(mirrored); XY: mirrored cell += conj(own YX sum)
        const int j = h < 2 ? y * S + x : ((N - y) & (N - 1)) * S + ((N - x) & (N - 1));
        const float sg = (x + y) & 1 ? -1.f : 1.f;
        sm[j] = make_float2(sg * (sm[j].x + m[k].x), sg * (sm[j].y - m[k].y));
    }
    __syncthreads();
    float2 a[E];
    {
        const int t = tid % L;
        float2 *row = sm + (tid / L) * S;
#pragma unroll
        for (int m = 0; m < E; m++) a[m] = row[t + L * m];
        hai_fft::line_first<N>(a, t, tw);
        __syncwarp();
#pragma unroll
        for (int k = 0; k < E; k++) row[L * k + ((t + k) & (L - 1))] = a[k];
        __syncwarp();
#pragma unroll
        for (int u = 0; u < E / L; u++)
#pragma unroll
            for (int i = 0; i < L; i++) a[L * u + i] = row[L * (t + L * u) + ((i + t) & (L - 1))];
        hai_fft::line_second<N>(a);
        __syncwarp();
#pragma unroll
        for (int u = 0; u < E / L; u++)
#pragma unroll
            for (int i = 0; i < L; i++) row[t + L * u + E * i] = a[L * u + i];
    }
    __syncthreads();
    const int t = tid / N, x = tid % N;
    float2 *col = sm + x;
#pragma unroll
    for (int m = 0; m < E; m++) a[m] = col[(t + L * m) * S];
    hai_fft::line_first<N>(a, t, tw);
    __syncthreads();
#pragma unroll
    for (int k = 0; k < E; k++) col[(L * k + t) * S] = a[k];
    __syncthreads();
#pragma unroll
    for (int u = 0; u < E / L; u++)
#pragma unroll
        for (int i = 0; i < L; i++) a[L * u + i] = col[(L * (t + L * u) + i) * S];
    hai_fft::line_second<N>(a);
    const int Q = P == 2 ? 4 : 1;
    float *o0 = img + ((size_t)(c0 + c) * Q + h) * N * N + x;
#pragma unroll
    for (int u = 0; u < E / L; u++)
#pragma unroll
        for (int i = 0; i < L; i++) {
            const float2 v = a[L * u + i];
            float *o = o0 + (size_t)(t + L * u + E * i) * N;
            *o = accumulate ? *o + v.x : v.x;
            if (h == 2) o[(size_t)N * N] = accumulate ? o[(size_t)N * N] + v.y : v.y;
        }
}

template <int P, bool REAL, bool VEC>
hai_status launch_gather(hai_ctx *ctx, const hai_layout *L, const int32_t *vis, long long nbl, int c0, int cb,
                         float2 *part, cudaStream_t st) {
    auto kern = xfft_gather_kernel<P, REAL, VEC>;
    HAI_CUDA_TRY(hai_allow_dyn_smem(kern, ctx->smem_optin));
    const size_t smem = sizeof(float2) * kGatherWarps * P * P * kPcells * 33;
    kern<<<dim3(L->xfft_nchunk, (cb + 31) / 32), 32 * kGatherWarps, smem, st>>>(
        vis, nbl, c0, cb, static_cast<const Chunk *>(L->d_xchunk), L->xfft_nchunk, L->d_xrec, L->d_xcoef, part);
    return HAI_OK;
}

template <int N>
void launch_fft(const hai_layout *L, const float2 *part, int cb, int c0, float *img, int accumulate, cudaStream_t st) {
    xfft_fft_kernel<N><<<dim3(cb, L->n_pol == 2 ? 3 : 1), N * hai_fft::Line<N>::L, 0, st>>>(part, L->d_xpatch, L->xfft_nchunk, cb,
                                                                              L->n_pol, c0, img, accumulate);
}

}  // namespace

// The layout's patch records (binned on the host) and their coefficients (on
// the GPU), built once and kept with the layout.
static hai_status ensure_table(const hai_layout *L) {
    std::lock_guard<std::mutex> lock(L->xfft_mu);
    if (L->d_xpatch) return HAI_OK;
    const int N = L->grid_n, K = L->ksize, ne = L->n_elem, W = 2 * K - 1, npx = N / kPw, npy = N / kPh, np = npx * npy;
    // contributions of all pairs to cells: 2 (2K-1)^2 per stored pair at most
    const double max_ent = (double)ne * (ne + 1) / 2 * 2.0 * W * W;
    if (max_ent > 2.0e8)
        return hai_fail(HAI_ERR_UNSUPPORTED, "hai_xfft_image: the layout's gridding list would exceed 2e8 entries");
    const int32_t *anc = L->h_anchors.data();
    // f(patch, record) for every patch that a footprint touches, each once
    auto each_record = [&](auto &&f) {
        uint32_t bl = 0;
        for (int a = 0; a < ne; a++)
            for (int b = 0; b <= a; b++, bl++) {
                const int x = (anc[2 * a] - anc[2 * b] - (K - 1)) & (N - 1);
                const int y = (anc[2 * a + 1] - anc[2 * b + 1] - (K - 1)) & (N - 1);
                const int nx = std::min(npx, (x + W - 1) / kPw - x / kPw + 1);
                const int ny = std::min(npy, (y + W - 1) / kPh - y / kPh + 1);
                const uint32_t r = bl | (a == b ? kAuto : 0u);
                for (int j = 0; j < ny; j++)
                    for (int i = 0; i < nx; i++) f((y / kPh + j) % npy * npx + (x / kPw + i) % npx, r);
            }
    };
    std::vector<long long> fill((size_t)np + 1, 0);
    each_record([&](int p, uint32_t) { fill[p + 1]++; });
    std::vector<Chunk> chunks;
    std::vector<int32_t> pstart((size_t)np + 1, 0);
    for (int p = 0; p < np; p++) {
        fill[p + 1] += fill[p];
        for (long long q = fill[p]; q < fill[p + 1]; q += kChunk)
            chunks.push_back(Chunk{p, (int32_t)q, (int32_t)std::min(q + kChunk, fill[p + 1])});
        pstart[p + 1] = (int32_t)chunks.size();
    }
    const size_t nrec = (size_t)fill[np];
    std::vector<uint32_t> rec(nrec);
    each_record([&](int p, uint32_t r) { rec[fill[p]++] = r; });
    bool real = true;
    for (size_t i = 1; i < L->h_taps.size(); i += 2) real &= L->h_taps[i] == 0.f;
    const size_t coef_bytes = sizeof(float) * nrec * kPcells * (real ? 1 : 2);
    int32_t *d_patch = nullptr;
    uint32_t *d_rec = nullptr;
    Chunk *d_chunk = nullptr;
    float *d_coef = nullptr;
    cudaError_t e = cudaMalloc(&d_patch, sizeof(int32_t) * pstart.size());
    if (e == cudaSuccess) e = cudaMalloc(&d_rec, sizeof(uint32_t) * nrec);
    if (e == cudaSuccess) e = cudaMalloc(&d_chunk, sizeof(Chunk) * chunks.size());
    if (e == cudaSuccess) e = cudaMalloc(&d_coef, coef_bytes);
    if (e == cudaSuccess) e = cudaMemcpy(d_patch, pstart.data(), sizeof(int32_t) * pstart.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(d_rec, rec.data(), sizeof(uint32_t) * nrec, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(d_chunk, chunks.data(), sizeof(Chunk) * chunks.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) {
        (real ? xfft_coef_kernel<true> : xfft_coef_kernel<false>)<<<(unsigned)chunks.size(), 256>>>(
            d_chunk, d_rec, L->d_anchors, L->d_taps, N, K, d_coef);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(nullptr);
    if (e != cudaSuccess) {
        cudaFree(d_patch);
        cudaFree(d_rec);
        cudaFree(d_chunk);
        cudaFree(d_coef);
        return hai_cuda_fail(e, "hai_xfft_image: gridding table");
    }
    L->d_xrec = d_rec;
    L->d_xchunk = d_chunk;
    L->d_xcoef = d_coef;
    L->xfft_nchunk = (int)chunks.size();
    L->xfft_real = real;
    L->d_xpatch = d_patch;
    L->dev_bytes += sizeof(int32_t) * pstart.size() + sizeof(uint32_t) * nrec + sizeof(Chunk) * chunks.size() + coef_bytes;
    return HAI_OK;
}

extern "C" hai_status hai_xfft_image(hai_ctx *ctx, const hai_layout *L, const int32_t *vis, int C, float *img,
                                     int accumulate, void *stream) {
    if (!ctx || !L) return hai_fail(HAI_ERR_INVALID_ARG, "hai_xfft_image: NULL ctx or layout");
    if (L->ctx != ctx) return hai_fail(HAI_ERR_INVALID_ARG, "hai_xfft_image: layout of another context");
    if (C < 0 || (accumulate != 0 && accumulate != 1))
        return hai_fail(HAI_ERR_INVALID_ARG, "hai_xfft_image: bad channel count or flag");
    const int N = L->grid_n;
    if (N != 16 && N != 32 && N != 64) return hai_fail(HAI_ERR_UNSUPPORTED, "hai_xfft_image: grid size");
    if (C == 0) return HAI_OK;
    if (!vis || !img) return hai_fail(HAI_ERR_INVALID_ARG, "hai_xfft_image: NULL buffer");
    if (hai_fault_injected("launch")) return hai_fail(HAI_ERR_CUDA, "hai_xfft_image: injected launch failure");
    HAI_CUDA_TRY(cudaSetDevice(ctx->device));
    const hai_status ts = ensure_table(L);
    if (ts != HAI_OK) return ts;
    const hai_status ws = hai_workspace(ctx);
    if (ws != HAI_OK) return ws;
    cudaStream_t st = (cudaStream_t)stream;
    const int P = L->n_pol;
    const long long nbl = (long long)L->n_elem * (L->n_elem + 1) / 2;
    // channels per batch: partial sums in the context's workspace
    const size_t per_chan = sizeof(float2) * (size_t)P * P * L->xfft_nchunk * kPcells;
    const int cmax = (int)std::min<size_t>({(size_t)C, ctx->corr_ws_bytes / per_chan, (size_t)32768});
    // the interface's limit: one channel's visibilities and grids as floats would fit
    // the workspace (the partial sums take less)
    if (cmax < 1 || sizeof(float2) * ((size_t)nbl * P * P + (size_t)(P == 2 ? 3 : 1) * N * N) > ctx->corr_ws_bytes)
        return hai_fail(HAI_ERR_UNSUPPORTED, "hai_xfft_image: one channel exceeds the workspace");
    float2 *part = static_cast<float2 *>(ctx->d_corr_ws);
    const bool vec = ((uintptr_t)vis & 15) == 0;
    const int pidx = prof_begin(ctx, st);
    for (int c0 = 0; c0 < C; c0 += cmax) {
        const int cb = std::min(cmax, C - c0);
        hai_status s;
        if (P == 1)
            s = L->xfft_real ? launch_gather<1, true, false>(ctx, L, vis, nbl, c0, cb, part, st)
                             : launch_gather<1, false, false>(ctx, L, vis, nbl, c0, cb, part, st);
        else if (L->xfft_real)
            s = vec ? launch_gather<2, true, true>(ctx, L, vis, nbl, c0, cb, part, st)
                    : launch_gather<2, true, false>(ctx, L, vis, nbl, c0, cb, part, st);
        else
            s = vec ? launch_gather<2, false, true>(ctx, L, vis, nbl, c0, cb, part, st)
                    : launch_gather<2, false, false>(ctx, L, vis, nbl, c0, cb, part, st);
        if (s != HAI_OK) return s;
        if (N == 16) launch_fft<16>(L, part, cb, c0, img, accumulate, st);
        else if (N == 32) launch_fft<32>(L, part, cb, c0, img, accumulate, st);
        else launch_fft<64>(L, part, cb, c0, img, accumulate, st);
        prof_count(ctx, 2);
    }
    prof_end(ctx, pidx, st);
    HAI_CUDA_TRY(cudaGetLastError());
    return HAI_OK;
}
