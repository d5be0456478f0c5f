// Inter-station stage of the hierarchical array (Section 6, Eq. inter-station
// visibilities and Eq. inter-station XFFT).
//
// hai_beams_to_corr: station beams [S][C][T][K][P][2] int8 (the beamformer's
// output) -> correlator input [K][C][T][P][S][2] int8, so that hai_correlate
// with the (beam, channel) pairs as channels and the stations as elements
// gives V_mn(s_k) = sum_t E_m(s_k) conj(E_n(s_k)).
//
// hai_xfft_station_image: dirty images of those visibilities.  Every ordered
// station pair (m, n), autos included, is phased towards the beam direction,
// V~ = V exp(+2 pi i s_k.(r_m - r_n) / lambda), and gridded with a 2x2
// bilinear kernel at uv = (r_m - r_n) / cell; pairs whose 2x2 footprint (or
// its mirror's) leaves [-N/2, N/2 - 1]^2 are dropped and counted.  The steering
// phasors are computed once per (beam, pair) by an FP64 kernel at layout
// creation: the phase reaches ~10^5 rad on 65 km baselines, where FP32 would
// lose ~10^-2 rad; the FP64 phase is reduced to a fraction of a turn before
// sincospi and the phasor is stored in FP32.
//
// Both XX and YY grids are Hermitian (the mirror of a pair carries the
// conjugate), so their images are real and one complex FFT of G_XX + i G_YY
// gives XX in the real and YY in the imaginary part; XY needs its own complex
// grid.  The two complex grids are built in the caller's image planes
// [XX, YY, Re XY, Im XY] (as split re / im planes), which the FFT then
// transforms in place: no scratch memory.  Gridding runs over tiles of the uv
// grid with a thread per cell, the pairs binned to tiles on the host, and
// writes its cells with the (-1)^(u+v) checkerboard that puts the phase
// centre at pixel (N/2, N/2).  The FFTs hold their lines in registers
// (fft_line.cuh).
#include <math.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "fft_line.cuh"
#include "hai_internal.h"

namespace {

// Tiles of the periodic uv grid (x = u mod N, y = v mod N), 16 x 16 cells with a
// thread per cell.  The unit of gridding work is a tile and its mirror: tile t
// along an axis holds the lower corners 16 t .. 16 t + 15, whose mirrors' lower
// corners fall in tile -t - 1, so that a pair's visibilities are read once for
// both of its footprints.
constexpr int kTile = 16, kTcells = kTile * kTile;
constexpr int kGridThreads = 2 * kTcells;         // the tile's cells, then the mirror tile's
constexpr int kGridWarps = kGridThreads / 32;
constexpr int kImgs = 4;                          // images (beam, channel) a CTA grids together
constexpr int kFoot = 512;                        // pairs staged at a time
constexpr int kFootRow = kFoot + 4;               // float4 per staged row: direct and mirrored values 4 banks apart

// One chunk of a unit's pairs and, per warp, its gather entries: slot k of lane
// l at entry base[w] + 32 k + l (zero weights pad the shorter lists).
struct TileChunk {
    int32_t foot, nfoot;
    int32_t base[kGridWarps + 1];
};
struct TileEnt {
    float w;             // bilinear weight
    int32_t slot;        // pair within the chunk; + kFootRow: its mirror's value
};
// Tiles of a unit (mirror < 0: none), and its first chunk.
struct TileUnit {
    int32_t tile, mirror, chunk;
};

__device__ __forceinline__ void pair_of(long long bl, int &m, int &n) {
    int a = (int)((sqrt(8.0 * (double)bl + 1.0) - 1.0) * 0.5);
    while ((long long)(a + 1) * (a + 2) / 2 <= bl) a++;
    while ((long long)a * (a + 1) / 2 > bl) a--;
    m = a;
    n = (int)(bl - (long long)a * (a + 1) / 2);
}

// exp(+2 pi i s_k.(r_m - r_n) / lambda) for every (beam, stored pair), FP64.
__global__ void steering_kernel(const double *__restrict__ pos, const double *__restrict__ dir, int K,
                                long long nbl, double inv_lambda, float2 *__restrict__ out) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (long long)K * nbl) return;
    const int k = (int)(i / nbl);
    const long long bl = i - (long long)k * nbl;
    int m, n;
    pair_of(bl, m, n);
    const double turns = (dir[2 * k] * (pos[2 * m] - pos[2 * n]) + dir[2 * k + 1] * (pos[2 * m + 1] - pos[2 * n + 1])) *
                         inv_lambda;
    const double frac = turns - rint(turns);          // |frac| <= 1/2: exact reduction in FP64
    double s, c;
    sincospi(2.0 * frac, &s, &c);
    out[i] = make_float2((float)c, (float)s);
}

__device__ __forceinline__ float2 cmulf(float2 a, float2 b) {
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// G_XX + i G_YY into planes 0 / 1 and G_XY into planes 2 / 3 of kImgs images per
// CTA, one tile of the grid and its mirror, with the checkerboard.  The unit's
// pairs are phased once into shared memory, a chunk at a time, as the value of
// the pair (XX + i YY, XY) and that of its mirror (conj(XX) + i conj(YY),
// conj(YX)), and every cell (thread) then adds its own list of them: no atomics,
// and a fixed order, so the images are bit-reproducible.  Two lanes share a
// pair's 32-byte sector (XX, XY | YX, YY) and exchange XX for YY; one then holds
// the pair's value and the other the mirror's.  The lists are the same for every
// image: entries and phasors are read once per kImgs images; cells are dealt to
// the lanes by list length, so a warp's lanes end together.  Units are the fast
// grid index, so a group's visibilities (1 MB an image for 256 stations) come
// from HBM once and from L2 for the neighbouring tiles.  Grid rows whose tiles
// are all empty are left unwritten: the FFT passes do not read them.
//
// Bound: shared-memory wavefronts (one 16-byte random read per entry and image).
// Hierarchical cadence (256 stations, 512 images at 256^2): adding the
// footprints with shared-memory atomics took 902 us after an 85 us memset of
// all planes; a lane per image with the cells in registers 798 us (32 lanes a
// megabyte apart, 1.4 GB read from HBM); a tile at a time with a lane per
// footprint's two 16-byte loads 616 us (32 lines a load); this form 511 us.
template <bool VEC>
__global__ void __launch_bounds__(kGridThreads, 2) station_grid_kernel(
    const int32_t *__restrict__ vis, const uint32_t *__restrict__ foot, const TileEnt *__restrict__ ent,
    const TileChunk *__restrict__ chunks, const TileUnit *__restrict__ unit, const uint8_t *__restrict__ cell_of,
    int nunit, const float2 *__restrict__ phasor, int C, int images, long long nbl, int N, float *__restrict__ img) {
    extern __shared__ __align__(16) float4 stage[];     // [kImgs][2][kFootRow]; at the end [kImgs][4][512] floats
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int grp = blockIdx.x / nunit, o = blockIdx.x - grp * nunit;
    const int i0 = grp * kImgs, i1 = min(i0 + kImgs, images) - 1;
    const bool same = i0 / C == i1 / C;                 // one beam: one phasor for all images
    float4 acc[kImgs];
#pragma unroll
    for (int i = 0; i < kImgs; i++) acc[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    const int half = lane & 1;                          // XX, XY or YX, YY
    const int q0 = unit[o].chunk, q1 = unit[o + 1].chunk;
    for (int q = q0; q < q1; q++) {
        const TileChunk *ch = chunks + q;
        const int f0 = ch->foot, nf = ch->nfoot;
        if (q > q0) __syncthreads();                    // the last chunk's gather is done
        // whole warps stay in the loop for the exchange
        for (int fw = (tid >> 1) & ~15; fw < nf; fw += kGridThreads / 2) {
            const int f = fw + (lane >> 1);
            const size_t bl = __ldg(foot + f0 + min(f, nf - 1));
            int4 x[kImgs];
            float2 w[kImgs];
#pragma unroll
            for (int i = 0; i < kImgs; i++) {
                const int im = min(i0 + i, images - 1);
                const int32_t *v = vis + ((size_t)im * nbl + bl) * 8 + 4 * half;
                if (VEC) {
                    x[i] = __ldg(reinterpret_cast<const int4 *>(v));
                } else {
                    const int2 a = __ldg(reinterpret_cast<const int2 *>(v)), b = __ldg(reinterpret_cast<const int2 *>(v) + 1);
                    x[i] = make_int4(a.x, a.y, b.x, b.y);
                }
                w[i] = i > 0 && same ? w[0] : __ldg(phasor + (size_t)(im / C) * nbl + bl);
            }
#pragma unroll
            for (int i = 0; i < kImgs; i++) {
                const float2 u = cmulf(make_float2((float)x[i].x, (float)x[i].y), w[i]);      // XX or YX
                const float2 v = cmulf(make_float2((float)x[i].z, (float)x[i].w), w[i]);      // XY or YY
                const float sx = __shfl_xor_sync(0xffffffffu, half ? v.x : u.x, 1);
                const float sy = __shfl_xor_sync(0xffffffffu, half ? v.y : u.y, 1);           // YY or XX
                if (f < nf)
                    stage[(i * 2 + half) * kFootRow + f] = half ? make_float4(sx + v.y, v.x - sy, u.x, -u.y)
                                                                : make_float4(u.x - sy, u.y + sx, v.x, v.y);
            }
        }
        __syncthreads();
        const int e1 = ch->base[warp + 1];
#pragma unroll 2
        for (int e = ch->base[warp] + lane; e < e1; e += 32) {
            const float2 x = __ldg(reinterpret_cast<const float2 *>(ent) + e);
            const int slot = __float_as_int(x.y);
#pragma unroll
            for (int i = 0; i < kImgs; i++) {
                const float4 g = stage[i * 2 * kFootRow + slot];
                acc[i].x = fmaf(x.x, g.x, acc[i].x);
                acc[i].y = fmaf(x.x, g.y, acc[i].y);
                acc[i].z = fmaf(x.x, g.z, acc[i].z);
                acc[i].w = fmaf(x.x, g.w, acc[i].w);
            }
        }
    }
    // the cells back in row order, then out
    const int side = tid / kTcells, tc = tid % kTcells;
    float *cells = reinterpret_cast<float *>(stage);
    if (q1 > q0) {
        __syncthreads();
        const int cell = cell_of[(size_t)o * kGridThreads + tid];
        const float sgn = ((cell ^ (cell / kTile)) & 1) ? -1.f : 1.f;     // tiles start on even cells
#pragma unroll
        for (int i = 0; i < kImgs; i++) {
            float *d = cells + (size_t)i * 4 * kGridThreads + side * kTcells + cell;
            d[0] = sgn * acc[i].x;
            d[kGridThreads] = sgn * acc[i].y;
            d[2 * kGridThreads] = sgn * acc[i].z;
            d[3 * kGridThreads] = sgn * acc[i].w;
        }
        __syncthreads();
    }
    const int t = side ? unit[o].mirror : unit[o].tile;
    if (t < 0) return;
    const int x = t % (N / kTile) * kTile + tc % kTile, y = t / (N / kTile) * kTile + tc / kTile;
#pragma unroll
    for (int i = 0; i < kImgs; i++) {
        if (i0 + i >= images) break;
#pragma unroll
        for (int p = 0; p < 4; p++)
            img[(((size_t)(i0 + i) * 4 + p) * N + y) * N + x] = q1 > q0 ? cells[(i * 4 + p) * kGridThreads + tid] : 0.f;
    }
}

// Row pass, in place on a plane pair (re plane, im plane): lines in registers
// (fft_line.cuh), 256 / L rows per CTA.  The exchange keeps value k1 of lane t
// at (L + 1) k1 + t, lines 8 (mod 16) float2 apart at L = 8 and 4 (mod 16) at
// L = 4: conflict-free both ways.  Global accesses are runs of L floats, whole
// sectors.  The bound is HBM: every plane is read and written once (1.07 GB on
// the hierarchical cadence's 512 images at 256^2).  The radix-2 form it
// replaces made log2 N passes over shared memory and took 604 us there;
// now 169 us (6.3 TB/s).  Only the rows that the gridding wrote are transformed.
constexpr int kFftThreads = 256;

template <int N>
struct RowSmem {
    static constexpr int L = hai_fft::Line<N>::L, E = hai_fft::Line<N>::E;
    static constexpr int XS = (E * (L + 1) + 15) / 16 * 16 + (L == 8 ? 8 : L == 4 ? 4 : 0);
};

template <int N>
__global__ void __launch_bounds__(kFftThreads) fft_rows_kernel(float *__restrict__ img,
                                                               const int32_t *__restrict__ rows, int nrow) {
    constexpr int L = hai_fft::Line<N>::L, E = hai_fft::Line<N>::E, XS = RowSmem<N>::XS, W = kFftThreads / L;
    __shared__ float2 tw[N], xbuf[W * XS];
    hai_fft::fill_twiddles<N>(tw);
    const int t = threadIdx.x % L, w = threadIdx.x / L;
    const int pair = blockIdx.x;       // image * 2 + h
    const int r = blockIdx.y * W + w;
    const bool live = r < nrow;
    float *pre = img + ((size_t)pair * 2 * N + rows[live ? r : 0]) * N;
    float *pim = pre + (size_t)N * N;
    float2 a[E];
#pragma unroll
    for (int m = 0; m < E; m++) a[m] = make_float2(pre[t + L * m], pim[t + L * m]);
    __syncthreads();
    hai_fft::line_first<N>(a, t, tw);
    float2 *x = xbuf + w * XS;
#pragma unroll
    for (int k = 0; k < E; k++) x[(L + 1) * k + t] = a[k];
    __syncwarp();
#pragma unroll
    for (int u = 0; u < E / L; u++)
#pragma unroll
        for (int i = 0; i < L; i++) a[L * u + i] = x[(L + 1) * (t + L * u) + i];
    hai_fft::line_second<N>(a);
    if (!live) return;
#pragma unroll
    for (int u = 0; u < E / L; u++)
#pragma unroll
        for (int i = 0; i < L; i++) {
            const int k = t + L * u + E * i;
            pre[k] = a[L * u + i].x;
            pim[k] = a[L * u + i].y;
        }
}

// Column pass, in place: 16 columns per CTA, the column fastest over the
// threads (64-byte row segments; the exchange, value k1 of lane t at
// (L k1 + t) 16 + column, is conflict-free).  Before: 595 us on the
// cadence above (32 columns through a padded tile, radix-2); now 231 us.
template <int N>
__global__ void __launch_bounds__(16 * hai_fft::Line<N>::L) fft_cols_kernel(float *__restrict__ img,
                                                                                      const uint8_t *__restrict__ live) {
    constexpr int L = hai_fft::Line<N>::L, E = hai_fft::Line<N>::E;
    __shared__ float2 tw[N], x[N * 16];
    hai_fft::fill_twiddles<N>(tw);
    const int c = threadIdx.x % 16, t = threadIdx.x / 16;
    float *pre = img + (size_t)blockIdx.x * 2 * N * N + blockIdx.y * 16 + c;
    float *pim = pre + (size_t)N * N;
    float2 a[E];
#pragma unroll
    for (int m = 0; m < E; m++) {
        const size_t y = t + L * m;
        a[m] = live[y] ? make_float2(pre[y * N], pim[y * N]) : make_float2(0.f, 0.f);
    }
    __syncthreads();
    hai_fft::line_first<N>(a, t, tw);
#pragma unroll
    for (int k = 0; k < E; k++) x[(L * k + t) * 16 + c] = a[k];
    __syncthreads();
#pragma unroll
    for (int u = 0; u < E / L; u++)
#pragma unroll
        for (int i = 0; i < L; i++) a[L * u + i] = x[(L * (t + L * u) + i) * 16 + c];
    hai_fft::line_second<N>(a);
#pragma unroll
    for (int u = 0; u < E / L; u++)
#pragma unroll
        for (int i = 0; i < L; i++) {
            const size_t k = (size_t)(t + L * u + E * i) * N;
            pre[k] = a[L * u + i].x;
            pim[k] = a[L * u + i].y;
        }
}

template <int N>
void launch_fft(float *img, int images, const int32_t *rows, int nrow, const uint8_t *live, cudaStream_t st) {
    constexpr int W = kFftThreads / hai_fft::Line<N>::L;
    fft_rows_kernel<N><<<dim3(images * 2, (nrow + W - 1) / W), kFftThreads, 0, st>>>(img, rows, nrow);
    fft_cols_kernel<N><<<dim3(images * 2, N / 16), 16 * hai_fft::Line<N>::L, 0, st>>>(img, live);
}

// beams [S][C][T][K][P][2] -> [K][C][T][P][S][2]; one CTA per (c, t).  VEC:
// S and K P multiples of 8, 16-byte aligned buffers: every station's K P
// values and every output row move as 16-byte vectors through a shared slab
// [K P][Spad] (rows padded to keep 16-byte alignment).
template <bool VEC>
__global__ void __launch_bounds__(256) beams_to_corr_kernel(const char2 *__restrict__ in, int S, int C, int T, int KP,
                                                            int P, char2 *__restrict__ out) {
    extern __shared__ __align__(16) char2 slab[];
    const int Spad = VEC ? ((S + 7) & ~7) + 8 : S + 1;
    const long long ct = blockIdx.x;   // c * T + t
    const int c = (int)(ct / T), t = (int)(ct - (long long)c * T);
    if (VEC) {
        const int vpr = KP / 8;        // vectors per station segment
        for (int i = threadIdx.x; i < S * vpr; i += blockDim.x) {
            const int st = i / vpr, j0 = (i - st * vpr) * 8;
            const uint4 v = reinterpret_cast<const uint4 *>(in + ((size_t)st * C * T + ct) * KP)[i - st * vpr];
            const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int e = 0; e < 8; e++) {
                const uint32_t h = (w[e >> 1] >> (16 * (e & 1))) & 0xffffu;
                slab[(j0 + e) * Spad + st] = *reinterpret_cast<const char2 *>(&h);
            }
        }
    } else {
        for (int i = threadIdx.x; i < S * KP; i += blockDim.x) {
            const int st = i / KP, j = i - st * KP;
            slab[j * Spad + st] = in[((size_t)st * C * T + ct) * KP + j];
        }
    }
    __syncthreads();
    if (VEC) {
        const int vpr = S / 8;
        for (int i = threadIdx.x; i < KP * vpr; i += blockDim.x) {
            const int j = i / vpr, s0 = (i - j * vpr) * 8;   // j = (k, p)
            const int k = j / P, p = j - k * P;
            char2 *o = out + ((((size_t)k * C + c) * T + t) * P + p) * S + s0;
            *reinterpret_cast<uint4 *>(o) = *reinterpret_cast<const uint4 *>(slab + j * Spad + s0);
        }
    } else {
        for (int i = threadIdx.x; i < S * KP; i += blockDim.x) {
            const int j = i / S, st = i - j * S;     // j = (k, p)
            const int k = j / P, p = j - k * P;
            out[((((size_t)k * C + c) * T + t) * P + p) * S + st] = slab[j * Spad + st];
        }
    }
}

}  // namespace

struct hai_vis_layout {
    hai_ctx *ctx = nullptr;
    int S = 0, N = 0, P = 0, K = 0;
    long long nbl = 0;
    long long n_offgrid = 0;
    int nunit = 0, nrow = 0;                 // tile units in written rows; written rows
    uint32_t *d_foot = nullptr;              // stored pairs, unit after unit
    TileEnt *d_ent = nullptr;                // gather entries
    TileChunk *d_chunk = nullptr;
    TileUnit *d_unit = nullptr;              // units by pair count [nunit + 1]
    uint8_t *d_cell = nullptr;               // [nunit][512] cell of each thread
    int32_t *d_rows = nullptr;               // the written rows
    uint8_t *d_live = nullptr;               // [N] whether a row is written
    float2 *d_phasor = nullptr;
};

void vis_layout_dims(const hai_vis_layout *L, int *S, int *N, int *K) {
    *S = L->S;
    *N = L->N;
    *K = L->K;
}

static void vis_layout_free(hai_vis_layout *L) {
    if (!L) return;
    cudaFree(L->d_foot);
    cudaFree(L->d_ent);
    cudaFree(L->d_chunk);
    cudaFree(L->d_unit);
    cudaFree(L->d_cell);
    cudaFree(L->d_rows);
    cudaFree(L->d_live);
    cudaFree(L->d_phasor);
    delete L;
}

extern "C" hai_status hai_vis_layout_create(hai_ctx *ctx, const hai_vis_layout_desc *d, hai_vis_layout **out) {
    if (!ctx || !d || !out) return hai_fail(HAI_ERR_INVALID_ARG, "hai_vis_layout_create: NULL argument");
    *out = nullptr;
    const int S = d->n_station, N = d->grid_n, K = d->n_dir;
    if (S <= 0 || !d->pos_m || !(d->lambda_m > 0) || !(d->cell_m > 0) || (d->n_pol != 1 && d->n_pol != 2) ||
        K <= 0 || N < 16 || N > 256 || (N & (N - 1)))
        return hai_fail(HAI_ERR_INVALID_ARG, "hai_vis_layout_create: bad descriptor (grid_n a power of two in 16..256)");
    if (d->n_pol != 2) return hai_fail(HAI_ERR_UNSUPPORTED, "hai_vis_layout_create: station images need 2 pols");
    if (hai_fault_injected("alloc")) return hai_fail(HAI_ERR_NO_MEMORY, "hai_vis_layout_create: injected allocation failure");
    const long long nbl = (long long)S * (S + 1) / 2;
    // footprints in FP64 on the host: lower corner floor(uv) and fraction; a pair
    // is recorded once in every unit (tile and mirror tile) that its footprint or
    // its mirror's touches (counted, then placed)
    const int nt = N / kTile;
    auto mirror_of = [&](int t) { return (nt - 1 - t / nt) * nt + nt - 1 - t % nt; };
    auto unit_of = [&](int t) { return std::min(t, mirror_of(t)); };
    struct Hit {
        int tile, mirrored, cx, cy;            // lower corner in the tile, -1 .. 15
        float fu, fv;
    };
    // the tiles that the two footprints of a pair touch
    auto hits_of = [&](double du, double dv, bool autos, Hit (&h)[8]) {
        int n = 0;
        for (int m = 0; m < (autos ? 1 : 2); m++) {
            const double u = m ? -du : du, v = m ? -dv : dv, fu = floor(u), fv = floor(v);
            const int x = (((int)fu % N) + N) % N, y = (((int)fv % N) + N) % N;
            const int x1 = (x + 1) % N, y1 = (y + 1) % N;
            // with one tile a side the wrapped column is in the same tile: its own hit
            const int nx = x % kTile == kTile - 1 ? 2 : 1, ny = y % kTile == kTile - 1 ? 2 : 1;
            for (int j = 0; j < ny; j++)
                for (int i = 0; i < nx; i++)
                    h[n++] = Hit{((j ? y1 : y) / kTile) * nt + (i ? x1 : x) / kTile, m, i ? -1 : x % kTile,
                                 j ? -1 : y % kTile, (float)(u - fu), (float)(v - fv)};
        }
        return n;
    };
    long long dropped = 0;
    auto each_pair = [&](auto &&f) {           // f(pair, hits, n) of the kept pairs
        dropped = 0;
        long long bl = 0;
        Hit h[8];
        for (int m = 0; m < S; m++)
            for (int n = 0; n <= m; n++, bl++) {
                const double du = (d->pos_m[2 * m] - d->pos_m[2 * n]) / d->cell_m;
                const double dv = (d->pos_m[2 * m + 1] - d->pos_m[2 * n + 1]) / d->cell_m;
                if (!station_pair_kept(N, du, dv)) {
                    dropped++;
                    continue;
                }
                f((uint32_t)bl, h, hits_of(du, dv, m == n, h));    // an auto pair has no mirror
            }
    };
    auto each_unit = [&](const Hit *h, int n, auto &&f) {          // f(unit) once for every unit hit
        for (int i = 0; i < n; i++) {
            bool seen = false;
            for (int j = 0; j < i; j++) seen |= unit_of(h[j].tile) == unit_of(h[i].tile);
            if (!seen) f(unit_of(h[i].tile));
        }
    };
    std::vector<int32_t> count((size_t)nt * nt, 0);
    each_pair([&](uint32_t, const Hit *h, int n) { each_unit(h, n, [&](int u) { count[u]++; }); });
    // written rows: those of a tile row (or its mirror's) with a pair in it
    std::vector<uint8_t> live(N, 0);
    std::vector<int32_t> rows, tiles;
    for (int t = 0; t < nt * nt; t++)
        if (count[t])
            for (int r : {t / nt, nt - 1 - t / nt}) std::fill(live.begin() + r * kTile, live.begin() + (r + 1) * kTile, 1);
    for (int y = 0; y < N; y++)
        if (live[y]) rows.push_back(y);
    for (int t = 0; t < nt * nt; t++)
        if (unit_of(t) == t && live[t / nt * kTile]) tiles.push_back(t);
    std::stable_sort(tiles.begin(), tiles.end(), [&](int x, int y) { return count[x] > count[y]; });
    std::vector<long long> fill(count.size(), 0);
    long long nfoot = 0;
    for (int t : tiles) {
        fill[t] = nfoot;
        nfoot += count[t];
    }
    if (nfoot > 0x0fffffffll) return hai_fail(HAI_ERR_UNSUPPORTED, "hai_vis_layout_create: too many station pairs");
    std::vector<uint32_t> foot(std::max<long long>(1, nfoot));
    struct Where {
        int m, n;
    };
    std::vector<Where> who(foot.size());
    {
        long long bl = 0;
        std::vector<Where> of((size_t)nbl);
        for (int m = 0; m < S; m++)
            for (int n = 0; n <= m; n++) of[bl++] = Where{m, n};
        each_pair([&](uint32_t pair, const Hit *h, int n) {
            each_unit(h, n, [&](int u) {
                who[fill[u]] = of[pair];
                foot[fill[u]++] = pair;
            });
        });
    }
    std::vector<TileEnt> ent;
    std::vector<TileChunk> chunks;
    std::vector<TileUnit> units;
    std::vector<uint8_t> cell_of(tiles.size() * kGridThreads);
    long long f0 = 0;
    for (size_t o = 0; o < tiles.size(); o++) {
        const long long f1 = f0 + count[tiles[o]];
        const int ta = tiles[o], tb = mirror_of(ta) == ta ? -1 : mirror_of(ta);
        units.push_back(TileUnit{ta, tb, (int32_t)chunks.size()});
        // f(cell of the unit, weight, mirrored) of the non-zero cells of pair k in the unit
        auto each_cell = [&](long long k, auto &&f) {
            Hit h[8];
            const int m = who[k].m, n = who[k].n;
            const double du = (d->pos_m[2 * m] - d->pos_m[2 * n]) / d->cell_m;
            const double dv = (d->pos_m[2 * m + 1] - d->pos_m[2 * n + 1]) / d->cell_m;
            const int nh = hits_of(du, dv, m == n, h);
            for (int i = 0; i < nh; i++) {
                const Hit &r = h[i];
                if (r.tile != ta && r.tile != tb) continue;
                for (int t = 0; t < 4; t++) {
                    const int x = r.cx + (t & 1), y = r.cy + (t >> 1);
                    const float w = ((t & 1) ? r.fu : 1.f - r.fu) * ((t >> 1) ? r.fv : 1.f - r.fv);
                    if (x >= 0 && x < kTile && y >= 0 && y < kTile && w != 0.f)
                        f((r.tile == ta ? 0 : kTcells) + y * kTile + x, w, r.mirrored);
                }
            }
        };
        int total[kGridThreads] = {}, order[kGridThreads], thread_of[kGridThreads];
        for (long long k = f0; k < f1; k++) each_cell(k, [&](int c, float, int) { total[c]++; });
        for (int side = 0; side < 2; side++) {
            int *o0 = order + side * kTcells;
            for (int c = 0; c < kTcells; c++) o0[c] = side * kTcells + c;
            std::stable_sort(o0, o0 + kTcells, [&](int x, int y) { return total[x] > total[y]; });
        }
        for (int i = 0; i < kGridThreads; i++) {
            thread_of[order[i]] = i;
            cell_of[o * kGridThreads + i] = (uint8_t)(order[i] % kTcells);
        }
        for (long long q = f0; q < f1; q += kFoot) {
            TileChunk ch;
            ch.foot = (int32_t)q;
            ch.nfoot = (int32_t)std::min<long long>(kFoot, f1 - q);
            int n[kGridThreads] = {};
            for (int f = 0; f < ch.nfoot; f++) each_cell(q + f, [&](int c, float, int) { n[thread_of[c]]++; });
            for (int w = 0; w < kGridWarps; w++) {
                ch.base[w] = (int32_t)ent.size();
                ent.resize(ent.size() + 32 * (size_t)*std::max_element(n + 32 * w, n + 32 * w + 32), TileEnt{0.f, 0});
            }
            ch.base[kGridWarps] = (int32_t)ent.size();
            std::fill(n, n + kGridThreads, 0);
            for (int f = 0; f < ch.nfoot; f++)
                each_cell(q + f, [&](int c, float w, int mirrored) {
                    const int i = thread_of[c];
                    ent[ch.base[i / 32] + 32 * n[i]++ + i % 32] = TileEnt{w, mirrored * kFootRow + f};
                });
            chunks.push_back(ch);
            if (ent.size() > 0x7fffffffull) return hai_fail(HAI_ERR_UNSUPPORTED, "hai_vis_layout_create: too many station pairs");
        }
        f0 = f1;
    }
    units.push_back(TileUnit{-1, -1, (int32_t)chunks.size()});
    hai_vis_layout *L = new hai_vis_layout();
    L->ctx = ctx;
    L->S = S;
    L->N = N;
    L->P = d->n_pol;
    L->K = K;
    L->nbl = nbl;
    L->n_offgrid = dropped;
    L->nunit = (int)tiles.size();
    L->nrow = (int)rows.size();
    double *d_pos = nullptr, *d_dir = nullptr;
    std::vector<double> dirs(2 * (size_t)K, 0.0);
    if (d->dir) std::copy(d->dir, d->dir + 2 * (size_t)K, dirs.begin());
    cudaError_t e = cudaSetDevice(ctx->device);
    auto put = [&](auto *&dst, const auto &src) {
        if (e == cudaSuccess) e = cudaMalloc(&dst, sizeof(src[0]) * src.size());
        if (e == cudaSuccess) e = cudaMemcpy(dst, src.data(), sizeof(src[0]) * src.size(), cudaMemcpyHostToDevice);
    };
    put(L->d_foot, foot);
    put(L->d_ent, ent);
    put(L->d_chunk, chunks);
    put(L->d_unit, units);
    put(L->d_cell, cell_of);
    put(L->d_rows, rows);
    put(L->d_live, live);
    if (e == cudaSuccess) e = cudaMalloc(&L->d_phasor, sizeof(float2) * (size_t)K * nbl);
    if (e == cudaSuccess) e = cudaMalloc(&d_pos, sizeof(double) * 2 * S);
    if (e == cudaSuccess) e = cudaMalloc(&d_dir, sizeof(double) * 2 * K);
    if (e == cudaSuccess) e = cudaMemcpy(d_pos, d->pos_m, sizeof(double) * 2 * S, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(d_dir, dirs.data(), sizeof(double) * 2 * K, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) {
        const long long n = (long long)K * nbl;
        steering_kernel<<<(unsigned)((n + 255) / 256), 256>>>(d_pos, d_dir, K, nbl, 1.0 / d->lambda_m, L->d_phasor);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    cudaFree(d_pos);
    cudaFree(d_dir);
    if (e != cudaSuccess) {
        vis_layout_free(L);
        return hai_cuda_fail(e, "hai_vis_layout_create");
    }
    *out = L;
    return HAI_OK;
}

extern "C" void hai_vis_layout_destroy(hai_vis_layout *L) {
    if (!L) return;
    cudaSetDevice(L->ctx->device);
    vis_layout_free(L);
}

extern "C" hai_status hai_vis_layout_offgrid(const hai_vis_layout *L, long long *n_offgrid) {
    if (!L || !n_offgrid) return hai_fail(HAI_ERR_INVALID_ARG, "hai_vis_layout_offgrid: NULL argument");
    *n_offgrid = L->n_offgrid;
    return HAI_OK;
}

extern "C" hai_status hai_xfft_station_image(hai_ctx *ctx, const hai_vis_layout *L, const int32_t *vis, int C,
                                             float *img, void *stream) {
    if (!ctx || !L) return hai_fail(HAI_ERR_INVALID_ARG, "hai_xfft_station_image: NULL ctx or layout");
    if (L->ctx != ctx) return hai_fail(HAI_ERR_INVALID_ARG, "hai_xfft_station_image: layout of another context");
    if (C < 0) return hai_fail(HAI_ERR_INVALID_ARG, "hai_xfft_station_image: negative channel count");
    if (C == 0) return HAI_OK;
    if (!vis || !img) return hai_fail(HAI_ERR_INVALID_ARG, "hai_xfft_station_image: NULL buffer");
    if (hai_fault_injected("launch")) return hai_fail(HAI_ERR_CUDA, "hai_xfft_station_image: injected launch failure");
    HAI_CUDA_TRY(cudaSetDevice(ctx->device));
    cudaStream_t st = (cudaStream_t)stream;
    const int N = L->N, images = L->K * C;
    const int groups = (images + kImgs - 1) / kImgs;
    if ((long long)images * 2 > 0x7fffffffll || (long long)L->nunit * groups > 0x7fffffffll)
        return hai_fail(HAI_ERR_UNSUPPORTED, "hai_xfft_station_image: too many images");
    const int pidx = prof_begin(ctx, st);
    auto grid = (((uintptr_t)vis & 15) == 0) ? station_grid_kernel<true> : station_grid_kernel<false>;
    HAI_CUDA_TRY(hai_allow_dyn_smem(grid, ctx->smem_optin));
    grid<<<(unsigned)(L->nunit * groups), kGridThreads, sizeof(float4) * kImgs * 2 * kFootRow, st>>>(
        vis, L->d_foot, L->d_ent, L->d_chunk, L->d_unit, L->d_cell, L->nunit, L->d_phasor, C, images, L->nbl, N, img);
    prof_end(ctx, pidx, st);
    HAI_CUDA_TRY(cudaGetLastError());
    switch (N) {
    case 16: launch_fft<16>(img, images, L->d_rows, L->nrow, L->d_live, st); break;
    case 32: launch_fft<32>(img, images, L->d_rows, L->nrow, L->d_live, st); break;
    case 64: launch_fft<64>(img, images, L->d_rows, L->nrow, L->d_live, st); break;
    case 128: launch_fft<128>(img, images, L->d_rows, L->nrow, L->d_live, st); break;
    default: launch_fft<256>(img, images, L->d_rows, L->nrow, L->d_live, st); break;
    }
    prof_count(ctx, 3);
    HAI_CUDA_TRY(cudaGetLastError());
    return HAI_OK;
}

extern "C" hai_status hai_beams_to_corr(hai_ctx *ctx, const int8_t *beams, int S, int C, int T, int K, int P,
                                        int8_t *out, void *stream) {
    if (!ctx) return hai_fail(HAI_ERR_INVALID_ARG, "hai_beams_to_corr: NULL ctx");
    if (S <= 0 || C < 0 || T < 0 || K <= 0 || (P != 1 && P != 2))
        return hai_fail(HAI_ERR_INVALID_ARG, "hai_beams_to_corr: bad sizes");
    if ((long long)C * T == 0) return HAI_OK;
    if (!beams || !out) return hai_fail(HAI_ERR_INVALID_ARG, "hai_beams_to_corr: NULL buffer");
    const bool vec = S % 8 == 0 && (K * P) % 8 == 0 && (((uintptr_t)beams | (uintptr_t)out) & 15) == 0;
    const size_t smem = sizeof(char2) * (size_t)K * P * (vec ? ((S + 7) & ~7) + 8 : S + 1);
    if (smem > 48 * 1024) return hai_fail(HAI_ERR_UNSUPPORTED, "hai_beams_to_corr: S x K x P too large for one tile");
    if ((long long)C * T > 0x7fffffffll) return hai_fail(HAI_ERR_UNSUPPORTED, "hai_beams_to_corr: too many samples");
    HAI_CUDA_TRY(cudaSetDevice(ctx->device));
    cudaStream_t st = (cudaStream_t)stream;
    const unsigned grid = (unsigned)((long long)C * T);
    const char2 *in = reinterpret_cast<const char2 *>(beams);
    char2 *o = reinterpret_cast<char2 *>(out);
    if (vec)
        beams_to_corr_kernel<true><<<grid, 256, smem, st>>>(in, S, C, T, K * P, P, o);
    else
        beams_to_corr_kernel<false><<<grid, 256, smem, st>>>(in, S, C, T, K * P, P, o);
    prof_count(ctx, 1);
    HAI_CUDA_TRY(cudaGetLastError());
    return HAI_OK;
}
