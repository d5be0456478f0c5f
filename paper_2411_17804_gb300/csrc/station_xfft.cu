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
// grid with threads per cell, the pairs binned to tiles on the host and listed
// per cell on the GPU when the layout is made, and writes its cells with the
// (-1)^(u+v) checkerboard that puts the phase centre at pixel (N/2, N/2).  The
// FFTs hold their lines in registers (fft_line.cuh).
#include <math.h>
#include <string.h>

#include <algorithm>
#include <new>
#include <vector>

#include "fft_line.cuh"
#include "hai_internal.h"

namespace {

// Tiles of the periodic uv grid (x = u mod N, y = v mod N), 16 x 16 cells.  The
// unit of gridding work is a tile and its mirror: tile t along an axis holds the
// lower corners 16 t .. 16 t + 15, whose mirrors' lower corners fall in tile
// -t - 1, so that a pair's visibilities are read once for both of its footprints.
constexpr int kTile = 16, kTcells = kTile * kTile;
constexpr int kUcells = 2 * kTcells;              // cells of a unit: the tile's, then the mirror tile's
constexpr int kGridThreads = kUcells;
constexpr int kGridWarps = kGridThreads / 32;
constexpr int kImgs = 4;                          // images (beam, channel) a CTA grids together, at most
constexpr int kCellLists = 64;                    // lists of one cell, at most
constexpr int kFoot = 512;                        // pairs staged at a time
constexpr int kFootRow = kFoot + 4;               // float4 per staged row: direct and mirrored values 4 banks apart

// One chunk of a unit's pairs and, per warp, its gather entries: slot k of lane
// l at entry base[w] + 32 k + l (zero weights pad the shorter lists).
struct TileChunk {
    long long foot;
    int32_t nfoot, unit;
    long long base[kGridWarps + 1];
};
struct TileEnt {
    float w;             // bilinear weight
    int32_t slot;        // pair within the chunk; + kFootRow: its mirror's value
};
// Tiles of a unit (mirror < 0: none), and its first chunk.
struct TileUnit {
    int32_t tile, mirror, chunk;
};
// A pair in a unit's list: lower corners of its footprint and of its mirror's
// (periodic grid), and the fractions; mfu < 0: no mirror (an auto).
struct FootRec {
    uint8_t x, y, mx, my;
    float fu, fv, mfu, mfv;
};
static_assert(sizeof(FootRec) == 20, "copied by words");

__host__ __device__ __forceinline__ float bilinear(int dx, int dy, float fu, float fv) {
    return (dx ? fu : 1.f - fu) * (dy ? fv : 1.f - fv);
}

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

// ---- The gather lists, made once per layout (a CTA per chunk, a thread per cell
// or list).  Each thread compares its cell with every pair of the chunk, so the
// lists are in pair order whatever the threads' timing.  By the host, in passes
// over the pairs, they took 9 ms for 256 stations and 562 ms for 2,048; here, with
// the binning, 1 and 43 ms.
__device__ __forceinline__ FootRec foot_rec(long long pair, const double *__restrict__ pos, double cell, int N) {
    int m, n;
    pair_of(pair, m, n);
    // the host's operations (nothing to contract): the same corners
    const double du = (pos[2 * m] - pos[2 * n]) / cell, dv = (pos[2 * m + 1] - pos[2 * n + 1]) / cell;
    const double a = floor(du), b = floor(dv), ma = floor(-du), mb = floor(-dv);
    FootRec r;
    r.x = (uint8_t)((int)a & (N - 1));
    r.y = (uint8_t)((int)b & (N - 1));
    r.mx = (uint8_t)((int)ma & (N - 1));
    r.my = (uint8_t)((int)mb & (N - 1));
    r.fu = (float)(du - a);
    r.fv = (float)(dv - b);
    r.mfu = m == n ? -1.f : (float)(-du - ma);
    r.mfv = (float)(-dv - mb);
    return r;
}
__global__ void foot_rec_kernel(const uint32_t *__restrict__ foot, long long nfoot, const double *__restrict__ pos, double cell,
                                int N, FootRec *__restrict__ recs) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < nfoot) recs[i] = foot_rec(foot[i], pos, cell, N);
}

__device__ __forceinline__ bool unit_cell(const TileUnit &u, int cell, int N, int &X, int &Y) {
    const int t = cell < kTcells ? u.tile : u.mirror, c = cell % kTcells;
    X = t % (N / kTile) * kTile + c % kTile;
    Y = t / (N / kTile) * kTile + c / kTile;
    return t >= 0;
}

// f(weight, slot) for the entries of cell (X, Y) from the n staged pairs
template <typename F>
__device__ __forceinline__ void each_entry(const FootRec *rec, int n, int N, int X, int Y, F &&f) {
    for (int i = 0; i < n; i++) {
        const FootRec r = rec[i];
        const int dx = (X - r.x) & (N - 1), dy = (Y - r.y) & (N - 1);
        if (dx < 2 && dy < 2) {
            const float w = bilinear(dx, dy, r.fu, r.fv);
            if (w != 0.f) f(w, i);
        }
        const int mx = (X - r.mx) & (N - 1), my = (Y - r.my) & (N - 1);
        if (mx < 2 && my < 2 && r.mfu >= 0.f) {
            const float w = bilinear(mx, my, r.mfu, r.mfv);
            if (w != 0.f) f(w, i + kFootRow);
        }
    }
}

__device__ __forceinline__ int stage_recs(const TileChunk &ch, const FootRec *recs, FootRec *rec) {
    const uint32_t *src = reinterpret_cast<const uint32_t *>(recs + ch.foot);
    uint32_t *dst = reinterpret_cast<uint32_t *>(rec);
    for (int i = threadIdx.x; i < ch.nfoot * (int)(sizeof(FootRec) / 4); i += blockDim.x) dst[i] = src[i];
    __syncthreads();
    return ch.nfoot;
}

// entries of every cell of a unit: total[unit][kUcells]
__global__ void __launch_bounds__(kUcells) tile_total_kernel(const TileChunk *__restrict__ chunks,
                                                            const TileUnit *__restrict__ unit,
                                                            const FootRec *__restrict__ recs, int N, int *__restrict__ total) {
    __shared__ FootRec rec[kFoot];
    const TileChunk &ch = chunks[blockIdx.x];
    const int nf = stage_recs(ch, recs, rec), cell = threadIdx.x;
    int X, Y, n = 0;
    if (!unit_cell(unit[ch.unit], cell, N, X, Y)) return;
    each_entry(rec, nf, N, X, Y, [&](float, int) { n++; });
    if (n) atomicAdd(&total[(size_t)ch.unit * kUcells + cell], n);
}

// Lists of a unit's cells, a thread each: a cell without entries has none, one
// with more entries than `load` has several, dealt in turn, for the smallest load
// (of 8 or more) with which the unit's lists are at most its 512 threads.  Longest lists first,
// so that a warp's lanes end together.  lists[unit][thread] = cell | part << 9 |
// parts << 16 (0: none), cells[unit][cell] = first thread | parts << 16.
//
// A short array puts every pair on a few cells: with one thread a cell, 256
// stations within 57 m (49 cells of 19 m, 128 images) took 4,370 us and 512 within
// 270 m (32 images) 1,820, where shared-memory atomics had taken 1,118 and 915;
// now 275 and 760 (whole calls).
__global__ void __launch_bounds__(kUcells) tile_assign_kernel(const int *__restrict__ total, uint32_t *__restrict__ lists,
                                                             uint32_t *__restrict__ cells) {
    __shared__ int2 cell_load[kUcells];                // entries per list, lists
    __shared__ int need[32], most;                     // lists needed in each try; the largest cell
    const size_t o = (size_t)blockIdx.x * kUcells;
    const int cell = threadIdx.x, mine = total[o + cell];
    if (cell < 32) need[cell] = 0;
    if (cell == 0) most = 0;
    lists[o + cell] = 0;
    __syncthreads();
    atomicMax(&most, mine);
    __syncthreads();
    auto lists_at = [&](int load) { return mine ? min((mine - 1) / load + 1, kCellLists) : 0; };
    int hi = max(1, most), lo = min(8, hi);            // at hi a cell has one list
    for (int k = 0; lo < hi; k++) {                    // the same in every thread; at most 31 halvings
        const int mid = lo + (hi - lo) / 2;
        const int n = __reduce_add_sync(0xffffffffu, lists_at(mid));
        if ((cell & 31) == 0) atomicAdd(&need[k], n);
        __syncthreads();
        if (need[k] <= kUcells) hi = mid;
        else lo = mid + 1;
    }
    const int parts = lists_at(hi), each = parts ? (mine - 1) / parts + 1 : 0;
    cell_load[cell] = make_int2(each, parts);
    __syncthreads();
    int first = 0;
    for (int c = 0; c < kUcells; c++) {
        const int2 x = cell_load[c];
        if (x.x > each || (x.x == each && c < cell)) first += x.y;
    }
    for (int k = 0; k < parts; k++) lists[o + first + k] = cell | k << 9 | parts << 16;
    cells[o + cell] = first | parts << 16;
}

// FILL false: the longest list of every warp, slots[chunk][warp]; true: the
// entries at the chunk's bases, padded to that length.
template <bool FILL>
__global__ void __launch_bounds__(kGridThreads) tile_lists_kernel(const TileChunk *__restrict__ chunks,
                                                                 const TileUnit *__restrict__ unit,
                                                                 const FootRec *__restrict__ recs, int N,
                                                                 const uint32_t *__restrict__ lists,
                                                                 int *__restrict__ slots, TileEnt *__restrict__ ent) {
    __shared__ FootRec rec[kFoot];
    const TileChunk &ch = chunks[blockIdx.x];
    const int nf = stage_recs(ch, recs, rec), warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    TileEnt *dst = FILL ? ent + ch.base[warp] + lane : nullptr;
    const uint32_t list = lists[(size_t)ch.unit * kGridThreads + threadIdx.x];
    const int parts = list >> 16;
    int X, Y, n = 0, turn = (list >> 9) & 127;         // entries of other lists before the next one of this
    if (parts && unit_cell(unit[ch.unit], list & (kUcells - 1), N, X, Y))
        each_entry(rec, nf, N, X, Y, [&](float w, int slot) {
            if (turn-- > 0) return;
            turn = parts - 1;
            if (FILL) dst[32ll * n] = TileEnt{w, slot};
            n++;
        });
    if (FILL) {
        const int most = (int)((ch.base[warp + 1] - ch.base[warp]) / 32);
        for (; n < most; n++) dst[32ll * n] = TileEnt{0.f, 0};
    } else {
        n = __reduce_max_sync(0xffffffffu, n);
        if (lane == 0) slots[(size_t)blockIdx.x * kGridWarps + warp] = n;
    }
}

// G_XX + i G_YY into planes 0 / 1 and G_XY into planes 2 / 3 of IMGS images per
// CTA, one tile of the grid and its mirror, with the checkerboard.  The unit's
// pairs are phased once into shared memory, a chunk at a time, as the value of
// the pair (XX + i YY, XY) and that of its mirror (conj(XX) + i conj(YY),
// conj(YX)), and every thread then adds one list of a cell of them; a cell's lists
// are added in order at the end.  No atomics, and a fixed order, so the images are
// bit-reproducible.  Two lanes share a
// pair's 32-byte sector (XX, XY | YX, YY) and exchange XX for YY; one then holds
// the pair's value and the other the mirror's.  The lists are the same for every
// image: entries and phasors are read once per IMGS images; lists are dealt to
// the lanes by length, so a warp's lanes end together.  With one image a CTA (few
// CTAs, each a long walk) a chunk's loads are issued before the last one's gather.  Units are the fast
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
template <bool VEC, int IMGS>
__global__ void __launch_bounds__(kGridThreads, 2) station_grid_kernel(
    const int32_t *__restrict__ vis, const uint32_t *__restrict__ foot, const TileEnt *__restrict__ ent,
    const TileChunk *__restrict__ chunks, const TileUnit *__restrict__ unit, const uint32_t *__restrict__ cell_tab,
    int nunit, const float2 *__restrict__ phasor, int C, int images, long long nbl, int N, float *__restrict__ img) {
    extern __shared__ __align__(16) float4 stage[];     // [IMGS][2][kFootRow]; at the end [IMGS][4][512] floats
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int grp = blockIdx.x / nunit, o = blockIdx.x - grp * nunit;
    const int i0 = grp * IMGS, i1 = min(i0 + IMGS, images) - 1;
    const bool same = i0 / C == i1 / C;                 // one beam: one phasor for all images
    float4 acc[IMGS];
#pragma unroll
    for (int i = 0; i < IMGS; i++) acc[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    const int half = lane & 1;                          // XX, XY or YX, YY
    const int q0 = unit[o].chunk, q1 = unit[o + 1].chunk;
    constexpr int kPass = 2 * kFoot / kGridThreads;     // pairs a lane pair stages of a chunk
    constexpr bool kAhead = IMGS == 1;                  // a chunk's loads issued before the last one's gather
    struct Pair {
        int4 x[IMGS];
        float2 w[IMGS];
    };
    auto index = [&](int q, int p) -> size_t {
        const TileChunk *ch = chunks + q;
        return __ldg(foot + ch->foot + min(p * (kGridThreads / 2) + (tid >> 1), ch->nfoot - 1));
    };
    auto fetch = [&](size_t bl, Pair &r) {
#pragma unroll
        for (int i = 0; i < IMGS; i++) {
            const int im = min(i0 + i, images - 1);
            const int32_t *v = vis + ((size_t)im * nbl + bl) * 8 + 4 * half;
            if (VEC) {
                r.x[i] = __ldg(reinterpret_cast<const int4 *>(v));
            } else {
                const int2 a = __ldg(reinterpret_cast<const int2 *>(v)), b = __ldg(reinterpret_cast<const int2 *>(v) + 1);
                r.x[i] = make_int4(a.x, a.y, b.x, b.y);
            }
            r.w[i] = i > 0 && same ? r.w[0] : __ldg(phasor + (size_t)(im / C) * nbl + bl);
        }
    };
    auto put = [&](const Pair &r, int f, int nf) {
#pragma unroll
        for (int i = 0; i < IMGS; i++) {
            const float2 u = cmulf(make_float2((float)r.x[i].x, (float)r.x[i].y), r.w[i]);      // XX or YX
            const float2 v = cmulf(make_float2((float)r.x[i].z, (float)r.x[i].w), r.w[i]);      // XY or YY
            const float sx = __shfl_xor_sync(0xffffffffu, half ? v.x : u.x, 1);
            const float sy = __shfl_xor_sync(0xffffffffu, half ? v.y : u.y, 1);                 // YY or XX
            if (f < nf)
                stage[(i * 2 + half) * kFootRow + f] = half ? make_float4(sx + v.y, v.x - sy, u.x, -u.y)
                                                            : make_float4(u.x - sy, u.y + sx, v.x, v.y);
        }
    };
    Pair ahead[kAhead ? kPass : 1];
    size_t next[kAhead ? kPass : 1];
    if constexpr (kAhead)
        if (q0 < q1)
#pragma unroll
            for (int p = 0; p < kPass; p++) {
                fetch(index(q0, p), ahead[p]);
                next[p] = index(min(q0 + 1, q1 - 1), p);
            }
    for (int q = q0; q < q1; q++) {
        const TileChunk *ch = chunks + q;
        const int nf = ch->nfoot;
        if (q > q0) __syncthreads();                    // the last chunk's gather is done
#pragma unroll (kAhead ? kPass : 1)
        for (int p = 0; p < kPass; p++) {
            const int f = p * (kGridThreads / 2) + (tid >> 1);
            if constexpr (!kAhead) {
                if (f - (lane >> 1) >= nf) break;       // whole warps, for the exchange
                fetch(index(q, p), ahead[0]);
            }
            put(ahead[kAhead ? p : 0], f, nf);
        }
        __syncthreads();
        if constexpr (kAhead)
            if (q + 1 < q1)
#pragma unroll
                for (int p = 0; p < kPass; p++) {
                    fetch(next[p], ahead[p]);
                    next[p] = index(min(q + 2, q1 - 1), p);
                }
        const float2 *el = reinterpret_cast<const float2 *>(ent + ch->base[warp]) + lane;
        const int ne = (int)(ch->base[warp + 1] - ch->base[warp]);
#pragma unroll (8 / IMGS)
        for (int e = 0; e < ne; e += 32) {
            const float2 x = __ldg(el + e);
            const int slot = __float_as_int(x.y);
#pragma unroll
            for (int i = 0; i < IMGS; i++) {
                const float4 g = stage[i * 2 * kFootRow + slot];
                acc[i].x = fmaf(x.x, g.x, acc[i].x);
                acc[i].y = fmaf(x.x, g.y, acc[i].y);
                acc[i].z = fmaf(x.x, g.z, acc[i].z);
                acc[i].w = fmaf(x.x, g.w, acc[i].w);
            }
        }
    }
    // the sums back in row order of the cells, then out
    float *cells = reinterpret_cast<float *>(stage);
    if (q1 > q0) {
        __syncthreads();
#pragma unroll
        for (int i = 0; i < IMGS; i++) {
            float *d = cells + (size_t)i * 4 * kGridThreads + tid;
            d[0] = acc[i].x;
            d[kGridThreads] = acc[i].y;
            d[2 * kGridThreads] = acc[i].z;
            d[3 * kGridThreads] = acc[i].w;
        }
        __syncthreads();
    }
    const int t = tid < kTcells ? unit[o].tile : unit[o].mirror, tc = tid % kTcells;
    if (t < 0) return;
    const uint32_t list = q1 > q0 ? cell_tab[(size_t)o * kUcells + tid] : 0u;
    const int l0 = list & 0xffff, l1 = l0 + (int)(list >> 16);
    const float sgn = ((tc ^ (tc / kTile)) & 1) ? -1.f : 1.f;             // tiles start on even cells
    const int x = t % (N / kTile) * kTile + tc % kTile, y = t / (N / kTile) * kTile + tc / kTile;
    float v[4 * IMGS];
#pragma unroll
    for (int k = 0; k < 4 * IMGS; k++) v[k] = l1 > l0 ? sgn * cells[k * kGridThreads + l0] : 0.f;
    for (int l = l0 + 1; l < l1; l++)
#pragma unroll
        for (int k = 0; k < 4 * IMGS; k++) v[k] += sgn * cells[k * kGridThreads + l];
#pragma unroll
    for (int k = 0; k < 4 * IMGS; k++) {
        if (i0 + k / 4 >= images) break;
        img[(((size_t)i0 * 4 + k) * N + y) * N + x] = v[k];
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
    int nchunk = 0, most_chunks = 0;         // chunks of all units, of the largest
    uint32_t *d_foot = nullptr;              // stored pairs, unit after unit
    TileEnt *d_ent = nullptr;                // gather entries
    TileChunk *d_chunk = nullptr;
    TileUnit *d_unit = nullptr;              // units by pair count [nunit + 1]
    uint32_t *d_cell = nullptr;              // [nunit][kUcells] lists of each cell
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
    std::vector<int32_t> unit_of((size_t)nt * nt), mirror_of((size_t)nt * nt);
    for (int t = 0; t < nt * nt; t++) {
        mirror_of[t] = (nt - 1 - t / nt) * nt + nt - 1 - t % nt;
        unit_of[t] = std::min(t, mirror_of[t]);
    }
    struct Kept {
        uint32_t pair;
        uint8_t c[4];                          // lower corners: footprint x, y, its mirror's
    };
    // f(unit) once for every unit that the two footprints touch (an auto's mirror
    // lies on the auto)
    auto each_unit = [&](const Kept &r, auto &&f) {
        int seen[8], n = 0;
        for (int k = 0; k < 4; k += 2) {
            const int x = r.c[k], y = r.c[k + 1];
            const int nx = x % kTile == kTile - 1 ? 2 : 1, ny = y % kTile == kTile - 1 ? 2 : 1;
            for (int j = 0; j < ny; j++)
                for (int i = 0; i < nx; i++) {
                    const int u = unit_of[((y + j) & (N - 1)) / kTile * nt + ((x + i) & (N - 1)) / kTile];
                    bool known = false;
                    for (int q = 0; q < n; q++) known |= seen[q] == u;
                    if (known) continue;
                    seen[n++] = u;
                    f(u);
                }
        }
    };
    std::vector<Kept> kept;
    std::vector<int32_t> rows;
    std::vector<uint8_t> live(N, 0);
    std::vector<uint32_t> foot;
    std::vector<TileUnit> units;
    std::vector<TileChunk> chunks;
    try {
        kept.reserve((size_t)nbl);
        std::vector<long long> count((size_t)nt * nt, 0), fill((size_t)nt * nt, 0);
        long long bl = 0;
        for (int m = 0; m < S; m++)
            for (int n = 0; n <= m; n++, bl++) {
                const double du = (d->pos_m[2 * m] - d->pos_m[2 * n]) / d->cell_m;
                const double dv = (d->pos_m[2 * m + 1] - d->pos_m[2 * n + 1]) / d->cell_m;
                if (!station_pair_kept(N, du, dv)) continue;
                auto corner = [&](double u) { return (uint8_t)((int)floor(u) & (N - 1)); };
                const Kept r = {(uint32_t)bl, {corner(du), corner(dv), corner(-du), corner(-dv)}};
                kept.push_back(r);
                each_unit(r, [&](int u) { count[u]++; });
            }
        // written rows: those of a tile row (or its mirror's) with a pair in it
        std::vector<int32_t> tiles;
        for (int t = 0; t < nt * nt; t++)
            if (count[t])
                for (int r : {t / nt, nt - 1 - t / nt}) std::fill(live.begin() + r * kTile, live.begin() + (r + 1) * kTile, 1);
        for (int y = 0; y < N; y++)
            if (live[y]) rows.push_back(y);
        for (int t = 0; t < nt * nt; t++)
            if (unit_of[t] == t && live[t / nt * kTile]) tiles.push_back(t);
        std::stable_sort(tiles.begin(), tiles.end(), [&](int x, int y) { return count[x] > count[y]; });
        long long nfoot = 0;
        for (int t : tiles) {
            fill[t] = nfoot;
            units.push_back(TileUnit{t, mirror_of[t] == t ? -1 : mirror_of[t], (int32_t)chunks.size()});
            for (long long q = 0; q < count[t]; q += kFoot) {
                TileChunk ch = {};
                ch.foot = nfoot + q;
                ch.nfoot = (int32_t)std::min<long long>(kFoot, count[t] - q);
                ch.unit = (int32_t)units.size() - 1;
                chunks.push_back(ch);
            }
            nfoot += count[t];
        }
        units.push_back(TileUnit{-1, -1, (int32_t)chunks.size()});
        foot.resize((size_t)nfoot);
        for (const Kept &r : kept) each_unit(r, [&](int u) { foot[fill[u]++] = r.pair; });
    } catch (const std::bad_alloc &) {
        return hai_fail(HAI_ERR_NO_MEMORY, "hai_vis_layout_create: host memory for the station pairs");
    }
    hai_vis_layout *L = new hai_vis_layout();
    L->ctx = ctx;
    L->S = S;
    L->N = N;
    L->P = d->n_pol;
    L->K = K;
    L->nbl = nbl;
    L->n_offgrid = nbl - (long long)kept.size();
    L->nunit = (int)units.size() - 1;
    L->nchunk = (int)chunks.size();
    L->most_chunks = L->nunit ? units[1].chunk : 0;      // the units are in order of their pairs
    L->nrow = (int)rows.size();
    double *d_pos = nullptr, *d_dir = nullptr;
    std::vector<double> dirs(2 * (size_t)K, 0.0);
    if (d->dir) std::copy(d->dir, d->dir + 2 * (size_t)K, dirs.begin());
    cudaError_t e = cudaSetDevice(ctx->device);
    auto room = [&](auto *&dst, size_t n) {
        if (e == cudaSuccess) e = cudaMalloc(&dst, sizeof(*dst) * n);
    };
    auto put = [&](auto *&dst, const auto &src) {
        room(dst, src.size());
        if (e == cudaSuccess) e = cudaMemcpy(dst, src.data(), sizeof(src[0]) * src.size(), cudaMemcpyHostToDevice);
    };
    put(L->d_foot, foot);
    put(L->d_chunk, chunks);
    put(L->d_unit, units);
    put(L->d_rows, rows);
    put(L->d_live, live);
    room(d_pos, 2 * (size_t)S);
    if (e == cudaSuccess) e = cudaMemcpy(d_pos, d->pos_m, sizeof(double) * 2 * S, cudaMemcpyHostToDevice);
    // the gather lists: sizes, then entries
    const unsigned nchunk = (unsigned)chunks.size();
    const size_t ncell = (size_t)L->nunit * kUcells, nslot = (size_t)nchunk * kGridWarps;
    std::vector<int> slots(nslot);
    uint32_t *d_tmp = nullptr;                 // entries per cell, lists, slots, records
    room(d_tmp, 2 * ncell + nslot + foot.size() * (sizeof(FootRec) / 4));
    room(L->d_cell, ncell);
    if (e == cudaSuccess && nchunk) {
        int *total = reinterpret_cast<int *>(d_tmp), *d_slots = reinterpret_cast<int *>(d_tmp + 2 * ncell);
        uint32_t *list = d_tmp + ncell;
        FootRec *rec = reinterpret_cast<FootRec *>(d_slots + nslot);
        e = cudaMemset(total, 0, sizeof(int) * ncell);
        foot_rec_kernel<<<(unsigned)((foot.size() + 255) / 256), 256>>>(L->d_foot, (long long)foot.size(), d_pos, d->cell_m, N, rec);
        tile_total_kernel<<<nchunk, kUcells>>>(L->d_chunk, L->d_unit, rec, N, total);
        tile_assign_kernel<<<(unsigned)L->nunit, kUcells>>>(total, list, L->d_cell);
        tile_lists_kernel<false><<<nchunk, kGridThreads>>>(L->d_chunk, L->d_unit, rec, N, list, d_slots, nullptr);
        if (e == cudaSuccess) e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaMemcpy(slots.data(), d_slots, sizeof(int) * nslot, cudaMemcpyDeviceToHost);
        long long nent = 0;
        for (unsigned q = 0; q < nchunk; q++)
            for (int w = 0; w <= kGridWarps; w++) {
                chunks[q].base[w] = nent;
                if (w < kGridWarps) nent += 32ll * slots[(size_t)q * kGridWarps + w];
            }
        room(L->d_ent, (size_t)nent);
        if (e == cudaSuccess) e = cudaMemcpy(L->d_chunk, chunks.data(), sizeof(TileChunk) * nchunk, cudaMemcpyHostToDevice);
        if (e == cudaSuccess) {
            tile_lists_kernel<true><<<nchunk, kGridThreads>>>(L->d_chunk, L->d_unit, rec, N, list, d_slots, L->d_ent);
            e = cudaGetLastError();
        }
    }
    if (e == cudaSuccess) e = cudaMalloc(&L->d_phasor, sizeof(float2) * (size_t)K * nbl);
    if (e == cudaSuccess) e = cudaMalloc(&d_dir, sizeof(double) * 2 * K);
    if (e == cudaSuccess) e = cudaMemcpy(d_dir, dirs.data(), sizeof(double) * 2 * K, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) {
        const long long n = (long long)K * nbl;
        steering_kernel<<<(unsigned)((n + 255) / 256), 256>>>(d_pos, d_dir, K, nbl, 1.0 / d->lambda_m, L->d_phasor);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    cudaFree(d_tmp);
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
    if ((long long)images * 2 > 0x7fffffffll || (long long)L->nunit * ((images + kImgs - 1) / kImgs) > 0x7fffffffll)
        return hai_fail(HAI_ERR_UNSUPPORTED, "hai_xfft_station_image: too many images");
    // images per CTA: four share a unit's entries and phasors; fewer when the walk
    // over the largest unit is longer than what the work comes to per resident CTA
    int imgs = kImgs;
    while (imgs > 1 && 2ll * ctx->num_sms * L->most_chunks > (long long)L->nchunk * ((images + imgs - 1) / imgs)) imgs /= 2;
    const bool vec = ((uintptr_t)vis & 15) == 0;
    const int pidx = prof_begin(ctx, st);
    const auto grid = imgs == 4   ? vec ? station_grid_kernel<true, 4> : station_grid_kernel<false, 4>
                      : imgs == 2 ? vec ? station_grid_kernel<true, 2> : station_grid_kernel<false, 2>
                                  : vec ? station_grid_kernel<true, 1> : station_grid_kernel<false, 1>;
    HAI_CUDA_TRY(hai_allow_dyn_smem(grid, ctx->smem_optin));
    grid<<<(unsigned)(L->nunit * ((images + imgs - 1) / imgs)), kGridThreads, sizeof(float4) * imgs * 2 * kFootRow, st>>>(
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
