// Pieces shared by the tensor-core EPIC kernels (epic_tc.cu for N = 32 and
// 64, epic_tc128.cu for N = 128) and the batched plan (plan.cu).
//
// A launch images one or more stations ("a class": same grid side) over one
// cadence of C channels x T samples.  The flattened sample index runs over
// blocks (station, channel) of T samples each, block = station * C + channel,
// and every CTA (or CTA group) takes a contiguous range of it.
#pragma once

#include <cuda_fp16.h>
#include <stdint.h>

#include <vector>

#include "hai_internal.h"

// Static shared memory of the tensor-core EPIC kernels (mbarriers, TMEM
// address), which the device's per-block opt-in limit also has to hold.
constexpr size_t kStaticSmem = 1024;

// One station of a launch, in device memory.
struct TcStation {
    const uint8_t *table;   // gather table (GatherLayout) in global memory
    long long volt_off;     // byte offset of the station's voltages [C][T][2][ne][2] int8
    long long img_off;      // float offset of the station's images [C][4][N][N]
    int ne;                 // elements
    int ntile, nent;        // gather tiles and entries
    int cplx;               // complex taps
    uint32_t table_bytes;   // multiple of 16
};

// One step of a CTA's range: samples [t, t + nv) of channel chan of station
// stn (a step never straddles a block); src = its first voltage byte.
struct TcStep {
    int stn, chan, t, nv, ne;
    const int8_t *src;
    __device__ long long blk(int C) const { return (long long)stn * C + chan; }
};

// Walks a CTA's range [f, end) of the flattened index step by step, keeping
// the current station's element count and voltage offset in registers: one
// division at the start, none per step, a station-record load only when the
// station changes.
struct TcWalker {
    const TcStation *stations;
    int C, T;
    long long left;         // samples of the range still to walk
    int stn, chan, t, ne;
    const int8_t *next_src;
    const int8_t *volt;
    __device__ void init(const int8_t *v, const TcStation *st, int C_, int T_, long long s0, long long s1) {
        volt = v;
        stations = st;
        C = C_;
        T = T_;
        left = max(0ll, s1 - s0);
        const long long blk = s0 / T;
        t = (int)(s0 - blk * T);
        stn = (int)(blk / C);
        chan = (int)(blk - (long long)stn * C);
        ne = 0;
        next_src = v;
        if (left > 0) load();
    }
    // voltages are contiguous over a station's (channel, sample) index
    __device__ void load() {
        ne = stations[stn].ne;
        next_src = volt + stations[stn].volt_off + ((long long)chan * T + t) * 4ll * ne;
    }
    __device__ TcStep next(int sps) {
        TcStep s;
        s.stn = stn;
        s.chan = chan;
        s.t = t;
        s.nv = (int)min((long long)min(sps, T - t), left);
        s.ne = ne;
        s.src = next_src;
        next_src += s.nv * 4 * ne;
        left -= s.nv;
        t += s.nv;
        if (t == T) {
            t = 0;
            if (++chan == C) {
                chan = 0;
                ++stn;
                if (left > 0) load();
            }
        }
        return s;
    }
};

// Start of a step's voltages rounded down to 16 bytes when the layout has
// guard bytes (delta = bytes skipped).
__device__ __forceinline__ const int8_t *tc_aligned_src(const int8_t *src, int guard, uint32_t &delta) {
    delta = guard ? (uint32_t)((uintptr_t)src & 15u) : 0u;
    return src - delta;
}

// Steps of size `sps` in the range [s0, s1): whole blocks of T samples.
__device__ __forceinline__ int tc_count_steps(long long s0, long long s1, int T, int sps) {
    int n = 0;
    for (long long f = s0; f < s1;) {
        const long long lim = min((f / T + 1) * (long long)T, s1);
        n += (int)((lim - f + sps - 1) / sps);
        f = lim;
    }
    return n;
}

// Gather table of the gridding step.  The non-empty cells of the kernel's
// bounding box are dealt into tiles of 32 (one per warp lane), sorted by
// entry count so a tile's lanes run the same number of slots; a tile's
// entries are stored slot-major, entry (slot k, lane l) at tile_base + 32 k
// + l, with zero-weight padding.  Within a lane's list the order is chosen so
// that the lanes that one shared-memory phase serves together (128 bytes of
// voltages) read distinct banks, or one element, where they can.
//   cell offsets   uint32 [ntile * 32]  byte offset of the lane's cell in the
//                                       stage-1 operand (field 0), or
//                                       0xffffffff for an unused lane
//   tile bases     int32 [ntile + 1]    first entry of each tile
//   warp ranges    uint16 [kGatherWarps + 1] warp w grids tiles [r[w], r[w+1]);
//                                       tiles are dealt to the warps by
//                                       longest-first (slots + 2 per tile)
//   (pad to 16)
//   weights        float [nent]         a of conj(W~) = a + ib; for complex
//                                       taps float2 [nent] (a, b)
//   elements       uint16 [nent]
constexpr int kGatherWarps = 11;        // at most: a kernel may deal to fewer
struct GatherLayout {
    uint32_t off_cell, off_base, off_warp, off_w, off_e, bytes;
};
__host__ __device__ inline GatherLayout gather_layout(int ntile, int nent, int cplx) {
    GatherLayout t;
    t.off_cell = 0;
    t.off_base = 4u * 32u * ntile;
    t.off_warp = t.off_base + 4u * (ntile + 1);
    t.off_w = (t.off_warp + 2u * (kGatherWarps + 1) + 15u) & ~15u;
    t.off_e = t.off_w + (cplx ? 8u : 4u) * nent;
    t.bytes = (t.off_e + 2u * nent + 15u) & ~15u;
    return t;
}

// Sums of one lane's cell over its slots q, q + 32, .. (< qe): g[f] += conj(W~)
// E[field f], an element's F half2 voltages in one vector V (uint4: 4 fields,
// uint2: 2).  tab is the table in shared memory, through its own address (a
// pointer chosen at run time would make the loads generic).  Each term rounds
// as fmaf(w.x, x.x, fmaf(-w.y, x.y, re)), fmaf(w.x, x.y, fmaf(w.y, x.x, im)).
// Slots go four at a time, their loads issued before the first use.
template <bool CPLX, int F, typename V>
__device__ __forceinline__ void cell_sum_as(const uint8_t *tab, const GatherLayout &gl, int q, int qe, const V *E,
                                            float2 (&g)[F]) {
    static_assert(sizeof(V) == 4 * F, "one half2 a field");
    const float *wr = reinterpret_cast<const float *>(tab + gl.off_w);
    const float2 *wc = reinterpret_cast<const float2 *>(tab + gl.off_w);
    const uint16_t *el = reinterpret_cast<const uint16_t *>(tab + gl.off_e);
    auto weight = [&](int i) { return CPLX ? wc[i] : make_float2(wr[i], 0.f); };
    auto mac = [&](const float2 w, const V &e) {
        const uint32_t *x = reinterpret_cast<const uint32_t *>(&e);
#pragma unroll
        for (int f = 0; f < F; f++) {
            const float2 v = __half22float2(*reinterpret_cast<const __half2 *>(x + f));
            if (CPLX) g[f] = __ffma2_rn(make_float2(-w.y, w.y), make_float2(v.y, v.x), g[f]);
            g[f] = __ffma2_rn(make_float2(w.x, w.x), v, g[f]);
        }
    };
    for (; q + 96 < qe; q += 128) {
        float2 w[4];
        int en[4];
        V e[4];
#pragma unroll
        for (int j = 0; j < 4; j++) {
            en[j] = el[q + 32 * j];
            w[j] = weight(q + 32 * j);
        }
#pragma unroll
        for (int j = 0; j < 4; j++) e[j] = E[en[j]];
#pragma unroll
        for (int j = 0; j < 4; j++) mac(w[j], e[j]);
    }
    if (q + 32 < qe) {
        const int e0 = el[q], e1 = el[q + 32];
        const float2 w0 = weight(q), w1 = weight(q + 32);
        const V v0 = E[e0], v1 = E[e1];
        mac(w0, v0);
        mac(w1, v1);
        q += 64;
    }
    if (q < qe) mac(weight(q), E[el[q]]);
}
template <int F, typename V>
__device__ __forceinline__ void cell_sum(const uint8_t *tab, const GatherLayout &gl, int cplx, int q, int qe,
                                         const V *E, float2 (&g)[F]) {
    if (cplx) cell_sum_as<true>(tab, gl, q, qe, E, g);
    else cell_sum_as<false>(tab, gl, q, qe, E, g);
}

// Builds the gather table of one station from its CSR cell lists (cells of
// the box row-major, cstart[box_w * box_h + 1]).  Cell (x, y) of the box
// lands at byte tc::off_kmajor(y, 2 x, k_stride, mn_stride) of the stage-1
// operand.
// Entries of zero weight are left out.  F: half2 fields read per element (the
// phase is 32 / F lanes).  room: the most bytes a kernel can keep; a larger table
// is not ordered, as none can read it.  n_warps (<= kGatherWarps) get tiles; the
// others none.
void epic_tc_build_gather(int box_w, int box_h, const std::vector<int32_t> &cstart,
                          const std::vector<int32_t> &elem, const std::vector<float2> &w, uint32_t k_stride,
                          uint32_t mn_stride, int F, size_t room, std::vector<uint8_t> &out, int &ntile, int &nent, int &cplx,
                          int n_warps = kGatherWarps);

// fp16 W'[j][l] = (-1)^j exp(+2 pi i l j / N) as a real matrix entry: row
// (c_out, l), column (j, c_in) of the complex product y = W'^T x written for
// (re, im) pairs.
double epic_tc_dft_entry(int N, int c_out, int l, int j, int c_in);

// DFT operands of the tensor-core kernels for grid side N (built once per
// context, device memory owned by the context).
const void *epic_tc_dft(hai_ctx *ctx, int N, bool bf16 = false);
hai_status epic_tc_dft_prepare(hai_ctx *ctx, int N);

// Launchers over a list of stations of one grid side.  cta_begin (device,
// n_cta + 1 flat sample indices) gives each CTA's range; when it is null the
// ranges are b * len.  direct = 1: every block lies inside one CTA's range
// and is written straight into the station's image (with accumulate);
// direct = 0: blocks go to two partial slots per CTA for epic_reduce.
// guard = 1: every station's voltage block has 16 spare bytes before and
// after it, so voltage copies may round their start down and their end up
// to 16 bytes.
struct TcLaunch {
    const int8_t *volt;
    float *img;
    const TcStation *stations;
    int n_station;
    int ne_max;
    uint32_t table_max;
    const long long *cta_begin;
    long long len;
    int n_cta;
    int C, T;
    int direct, accumulate, guard;
    float *partials;
    int no_attr;            // 1: the kernel's shared-memory attribute is already set
    int split;              // 1: hi/lo split products (N = 32, 64)
    int bf16;               // 1: BF16 operands (N = 32, 64)
};
// Raises the kernel's dynamic shared-memory limit to the device's.
hai_status epic_tc_set_attr(hai_ctx *ctx, int N);
hai_status epic_tc_run(hai_ctx *ctx, int N, const TcLaunch &l, cudaStream_t st);
size_t epic_tc_smem(hai_ctx *ctx, int N, int ne_max, uint32_t table_max);
// Stage-1 operand strides of the gather table for grid side N.
void epic_tc_a1_strides(int N, uint32_t &k_stride, uint32_t &mn_stride);
// CTAs that image one channel together (1, or 4 for N = 128).
int epic_tc_group(int N);
hai_status epic_tc128_run(hai_ctx *ctx, const TcLaunch &l, cudaStream_t st);
hai_status epic_tc128_set_attr(hai_ctx *ctx);
size_t epic_tc128_smem(int ne_max, uint32_t table_max);
// Gather table (N = 128: blob) of one station: fills the record's table fields;
// shared_bytes = what the kernel keeps in shared memory.
void epic_tc_station_table(int grid_n, int box_w, int box_h, const std::vector<int32_t> &cstart,
                           const std::vector<int32_t> &elem, const std::vector<float2> &w, size_t room,
                           std::vector<uint8_t> &out, TcStation &rec, uint32_t &shared_bytes, long long &entries);
// Per-rank gather blob of one station for the N = 128 kernel;
// max_rank_bytes = the largest rank table (what a CTA keeps in shared memory).
void epic_tc128_build_blob(int box_w, int box_h, const std::vector<int32_t> &cstart,
                           const std::vector<int32_t> &elem, const std::vector<float2> &w, size_t room,
                           std::vector<uint8_t> &out, uint32_t &max_rank_bytes, long long &max_rank_entries);
// Clusters of the N = 128 kernel resident at once (0 if it cannot run).
int epic_tc128_max_groups(hai_ctx *ctx, int ne_max, uint32_t table_max);
