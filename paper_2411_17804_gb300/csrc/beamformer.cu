// Voltage beamformer (Eq. intra-station BF) with diagonal polarisation
// weights, B^p_k(t) = sum_a conj(w^p_{k,a}) E^p_a(t), exact in int32, with an
// optional requantisation to int8 fused into the epilogue.
//
// Per (station s, channel c, tile of 128 samples) and polarisation p the beams
// are one real GEMM on tcgen05 tensor cores:
//   D_p[t][n] = sum_kappa A_p[t][kappa] B_p[n][kappa],  kappa = (element, re/im)
// with A_p the voltages (int8 widened to fp16, exact) and B_p the weights:
// row n = 2k holds (w_r, w_i) per element (real part of conj(w) E), row 2k+1
// holds (-w_i, w_r) (imaginary part).  Products are at most 2^14 in magnitude and
// an output sums 2 N_e of them, so for N_e <= 512 every FP32 partial sum is an
// integer of at most 2^24: exact.
//
// CTA = 24 warps, persistent over a contiguous range of (s, c, tile) units:
//   warps 0-15 producers, in four groups of 4 warps: group g fills slot g of the
//              4-deep A ring, every fourth 64-element chunk, by 16-byte loads of
//              the voltage rows into registers (two chunks of the group in
//              flight; zero past T), widened to fp16 straight into the K-major
//              slot; the station's weights are widened into B when the station
//              changes;
//   warp 16    one thread issues the MMAs (8 per chunk);
//   warps 20-23 epilogue: TMEM -> int32, optional requantisation; each thread
//              assembles its sample's [k][p][re, im] row from both pols and
//              writes it with 16-byte stores (rows are contiguous per unit).
//
// Bound: HBM requests and the producers' registers (4.0 TB/s of voltages).  64
// stations x 256 elements x 32 channels x 1000 samples to 16 int8 beams: 745 us
// when eight warps landed the rows as int8 in shared memory by cp.async first, with
// two block barriers a chunk; 739 us with 16 warps loading into registers for every
// slot in turn; 760 us in groups, all with a warp on half lines of 8 rows; 521 us
// with a warp on whole 128-byte lines of 4 rows.  Neighbouring units dealt to the
// CTAs side by side instead of in ranges change stations more often: 546 us.  The
// launch's 80 registers a thread hold for the whole kernel, so the producers (two
// buffers of 32, the walkers) spill 112 bytes.
#include "hai_internal.h"
#include "tc.cuh"

namespace {

constexpr int kThreads = 768;
constexpr int kProd = 512;             // warps 0-15
constexpr int kMmaWarp = 16;
constexpr int kEpi = 128;              // warps 20-23
constexpr int kLaunchRegs = 80, kProdRegs = 96, kMmaRegs = 32, kEpiRegs = 64;
static_assert(512 * kProdRegs + 128 * kMmaRegs + 128 * kEpiRegs <= kThreads * kLaunchRegs, "register shares");
constexpr int kGroup = 128;            // producers of one slot
constexpr int kItems = 8;              // (row, 16-byte group) items per producer thread and chunk
constexpr int kItemRows = 16;          // rows between a thread's items
constexpr int kTile = 128;             // samples per unit (MMA M)
constexpr int kChunkE = 64;            // elements per K chunk (128 real K)
constexpr int kAStages = 4;            // fp16 operand ring
constexpr uint32_t kAKs = 144;         // A: K-group stride
constexpr uint32_t kAMNs = 16 * kAKs;  // A: row-group stride (16 K groups)
constexpr uint32_t kABytes = 16 * kAMNs;             // 36 KB fp16 chunk
constexpr uint32_t kBKs = 128;         // B: K-group stride

struct BfParams {
    const int8_t *volt;
    const int8_t *w;
    int S, C, T, K, ne, P;
    int tiles;                 // sample tiles per (s, c)
    long long nunits;
    int shift;                 // < 0: int32 output
    void *beams;
    unsigned long long *nsat;
    unsigned *status;
};

// 16 voltage bytes, not kept in L1 (every byte is read once).
__device__ __forceinline__ int4 load16(const int8_t *p) {
    int4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.s32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}
__device__ __forceinline__ void bar_prod() { asm volatile("bar.sync 1, 512;" ::: "memory"); }

// 16 int8 -> 16 fp16 (two 8-value K groups), exact
__device__ __forceinline__ void widen16(const int4 raw, uint4 &lo, uint4 &hi) {
    tc::widen4(raw.x, lo.x, lo.y);
    tc::widen4(raw.y, lo.z, lo.w);
    tc::widen4(raw.z, hi.x, hi.y);
    tc::widen4(raw.w, hi.z, hi.w);
}

__device__ __forceinline__ int requant(int x, int shift, int &sat) {
    int m = x < 0 ? -x : x;
    if (shift > 0) m = (m + (1 << (shift - 1))) >> shift;
    if (m > 127) {
        m = 127;
        sat++;
    }
    return x < 0 ? -m : m;
}

__global__ void __launch_bounds__(kThreads, 1) bf_kernel(const BfParams p) {
    extern __shared__ __align__(1024) uint8_t smem[];
    __shared__ __align__(8) uint64_t mb_full[kAStages], mb_empty[kAStages], mb_dfull[2], mb_dempty[2];
    __shared__ uint32_t tmem_slot;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nchunk = (p.ne + kChunkE - 1) / kChunkE;        // per polarisation
    const int ne_pad = nchunk * kChunkE;                      // B covers whole chunks, zero-padded
    const uint32_t bmns = (uint32_t)ne_pad * 32u;             // B: row-group stride (2 ne_pad / 8 groups)
    const uint32_t bbytes = (uint32_t)(2 * p.K / 8) * bmns;   // B of one polarisation
    uint8_t *sA = smem;                                       // [kAStages][kABytes]
    uint8_t *sB = sA + kAStages * kABytes;                    // [P][bbytes]
    const int ncols = 2 * p.K;                                // MMA N per polarisation
    const uint32_t dcols = (uint32_t)(p.P * ncols);           // TMEM columns per unit

    if (tid == 0) {
        for (int s = 0; s < kAStages; s++) {
            tc::mbar_init(&mb_full[s], kGroup / 32);
            tc::mbar_init(&mb_empty[s], 1);
        }
        for (int b = 0; b < 2; b++) {
            tc::mbar_init(&mb_dfull[b], 1);
            tc::mbar_init(&mb_dempty[b], kEpi / 32);
        }
        tc::mbar_fence_init();
    }
    uint32_t alloc = 32;
    while (alloc < 2 * dcols) alloc <<= 1;
    if (warp == 0) tc::tmem_alloc(&tmem_slot, alloc);
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tmem = tmem_slot;
    const long long u0 = p.nunits * blockIdx.x / gridDim.x, u1 = p.nunits * (blockIdx.x + 1) / gridDim.x;
    const size_t row_bytes = (size_t)p.ne * 2;                 // one (t, p) row of voltages
    const uint32_t idesc = tc::idesc_f16(128, ncols, 0, 0);

    if (warp < kMmaWarp) {
        tc::setmaxnreg_inc<kProdRegs>();
        // ============================================================ producers
        // Group grp fills slot grp of the ring: chunks grp, grp + 4, ... of the
        // CTA in order (unit, pol, element chunk).  Two chunks of the group are in
        // flight in registers; the loads of a buffer's next chunk start as soon as
        // it has been widened.
        const int grp = tid / kGroup, gt = tid % kGroup;
        const int per_unit = p.P * nchunk;
        const uint32_t t_stride = (uint32_t)(p.P * row_bytes);  // bytes between samples of one pol
        static_assert(kTile * 8 == kItems * kGroup && kProd == kAStages * kGroup, "items per chunk, a slot per group");
        // items: rows tw0 + 16 j, group gw: a warp loads whole 128-byte lines of 4
        // rows; 8 lanes store 2 rows of 4 groups (K groups 144 bytes apart: no bank
        // conflicts)
        const int tw0 = 4 * (gt >> 5) + 2 * ((lane >> 3) & 1) + (lane & 1), gw = 4 * (lane >> 4) + ((lane >> 1) & 3);
        const uint32_t src0 = (uint32_t)tw0 * t_stride + (uint32_t)gw * 16;
        const uint32_t wr0 = (uint32_t)(tw0 >> 3) * kAMNs + (uint32_t)(tw0 & 7) * 16 + (uint32_t)(2 * gw) * kAKs;
        int4 buf0[kItems], buf1[kItems];
        // load walker: the group's next chunk (unit lu, chunk lr of the unit)
        long long lu = u0, lsc = u0 / p.tiles;                 // station * C + channel
        int ltile = (int)(u0 - lsc * p.tiles), lr = grp;
        auto load = [&](int4 (&d)[kItems]) {
            while (lr >= per_unit) {
                lr -= per_unit;
                lu++;
                if (++ltile == p.tiles) {
                    ltile = 0;
                    lsc++;
                }
            }
            if (lu >= u1) return;
            const int t0 = ltile * kTile, pol = lr >= nchunk ? 1 : 0, kc = lr - pol * nchunk;
            const int8_t *src = p.volt + (size_t)(lsc * p.T + t0) * t_stride + pol * row_bytes + kc * (kChunkE * 2) + src0;
            const int rows = p.T - t0, left = p.ne - kc * kChunkE;
            if (rows >= kTile && left >= kChunkE) {            // the same for the group
#pragma unroll
                for (int j = 0; j < kItems; j++) d[j] = load16(src + (uint32_t)(kItemRows * j) * t_stride);
            } else {
#pragma unroll
                for (int j = 0; j < kItems; j++)
                    d[j] = tw0 + kItemRows * j < rows && gw * 8 < left ? load16(src + (uint32_t)(kItemRows * j) * t_stride)
                                                                       : make_int4(0, 0, 0, 0);
            }
            lr += kAStages;
        };
        uint8_t *A = sA + grp * kABytes + wr0;
        auto widen = [&](int4 (&d)[kItems]) {
#pragma unroll
            for (int j = 0; j < kItems; j++) {                 // rows tw0 + 16 j: A row groups + 2 j
                uint4 lo, hi;
                widen16(d[j], lo, hi);
                *reinterpret_cast<uint4 *>(A + (kItemRows / 8) * kAMNs * j) = lo;
                *reinterpret_cast<uint4 *>(A + (kItemRows / 8) * kAMNs * j + kAKs) = hi;
            }
            load(d);
        };
        // The station's weights into B: 8 elements of one (pol, beam) at a time,
        // row 2k: (wr, wi), row 2k + 1: (-wi, wr); zero beyond the elements.
        auto fill_b = [&](int s) {
            const int g8 = ne_pad / 8, rows8 = p.P * p.K * g8;
            const bool wide = ((uintptr_t)p.w & 15) == 0;
            for (int it = tid; it < rows8; it += kProd) {
                const int a8 = it % g8, row = it / g8, kk = row % p.K, pp = row / p.K;
                int4 raw = make_int4(0, 0, 0, 0);
                if (a8 * 8 < p.ne) {
                    const int8_t *src = p.w + ((((size_t)s * p.K + kk) * p.P + pp) * p.ne + a8 * 8) * 2;
                    if (wide) raw = *reinterpret_cast<const int4 *>(src);
                    else {
                        const ushort *e = reinterpret_cast<const ushort *>(src);
                        auto two = [&](int i) { return (int)((uint32_t)e[i] | ((uint32_t)e[i + 1] << 16)); };
                        raw = make_int4(two(0), two(2), two(4), two(6));
                    }
                }
                uint4 o[2];
                widen16(raw, o[0], o[1]);
                uint8_t *B = sB + pp * bbytes + tc::off_kmajor(2 * kk, 16 * a8, kBKs, bmns);
#pragma unroll
                for (int h = 0; h < 2; h++) {
                    // (wr, wi) -> (-wi, wr): halves swapped, the low one's sign flipped (0 stays +0)
                    const uint32_t v[4] = {o[h].x, o[h].y, o[h].z, o[h].w};
                    uint32_t m[4];
#pragma unroll
                    for (int i = 0; i < 4; i++) {
                        const __half2 x = *reinterpret_cast<const __half2 *>(&v[i]);
                        const __half2 y = __halves2half2(__hsub(__ushort_as_half(0), __high2half(x)), __low2half(x));
                        m[i] = *reinterpret_cast<const uint32_t *>(&y);
                    }
                    *reinterpret_cast<uint4 *>(B + h * kBKs) = o[h];
                    *reinterpret_cast<uint4 *>(B + h * kBKs + 16) = make_uint4(m[0], m[1], m[2], m[3]);
                }
            }
        };
        load(buf0);
        load(buf1);
        const long long per_station = (long long)p.C * p.tiles;
        long long u = u0, cu = u0 % per_station;               // unit, within its station
        int s = (int)(u0 / per_station), n = 0, r = grp;       // n chunks done, r the next one's place in the unit
        // Every group comes by every unit: a new station's B can be rewritten once
        // the MMAs of every group's last chunk have completed.
        auto enter = [&] {
            if (n > 0) tc::mbar_wait(&mb_empty[grp], (uint32_t)((n - 1) & 1), p.status);
            bar_prod();
            fill_b(s);
            tc::fence_proxy_async();
            bar_prod();
        };
        auto more = [&] {
            while (r >= per_unit) {
                r -= per_unit;
                if (++u == u1) return false;
                if (++cu == per_station) {
                    cu = 0;
                    s++;
                    enter();
                }
            }
            return true;
        };
        auto step = [&](int4 (&d)[kItems]) {
            if (n > 0) tc::mbar_wait(&mb_empty[grp], (uint32_t)((n - 1) & 1), p.status);
            widen(d);
            tc::fence_proxy_async();
            tc::mbar_arrive_warp(&mb_full[grp]);
            r += kAStages;
            n++;
        };
        // each buffer in its own half of the loop: one pass over both would copy a
        // buffer still being loaded, and wait for it
        if (u < u1) {
            enter();
            while (more()) {
                step(buf0);
                if (!more()) break;
                step(buf1);
            }
        }
    } else if (warp < kMmaWarp + 4) {
        // ============================================================ MMA
        tc::setmaxnreg_dec<kMmaRegs>();
        if (warp == kMmaWarp && tc::elect()) {
            long long gq = 0, gu = 0;
            const uint64_t da = tc::desc(tc::smem_u32(sA), kAKs, kAMNs), db = tc::desc(tc::smem_u32(sB), kBKs, bmns);
            for (long long u = u0; u < u1; u++, gu++) {
                const int b = (int)(gu & 1);
                if (gu >= 2) tc::mbar_wait(&mb_dempty[b], (uint32_t)(((gu >> 1) - 1) & 1), p.status);
                tc::fence_after();
                for (int pol = 0; pol < p.P; pol++) {
                    const uint32_t d = tmem + (uint32_t)b * dcols + (uint32_t)pol * ncols;
                    for (int kc = 0; kc < nchunk; kc++, gq++) {
                        const int slot = (int)(gq % kAStages);
                        tc::mbar_wait(&mb_full[slot], (uint32_t)((gq / kAStages) & 1), p.status);
                        tc::fence_after();
                        const uint64_t a = tc::desc_add(da, slot * kABytes);
                        const uint64_t bb = tc::desc_add(db, pol * bbytes + kc * 16 * kBKs);
#pragma unroll
                        for (int s = 0; s < 8; s++)
                            tc::mma_f16(d, tc::desc_add(a, s * 2 * kAKs), tc::desc_add(bb, s * 2 * kBKs), idesc,
                                        (kc > 0 || s > 0) ? 1u : 0u);
                        tc::mma_commit(&mb_empty[slot]);
                    }
                }
                tc::mma_commit(&mb_dfull[b]);
            }
        }
    } else {
        // ============================================================ epilogue
        tc::setmaxnreg_dec<kEpiRegs>();
        const int q = warp & 3;
        const uint32_t lane_base = (uint32_t)(q * 32) << 16;
        const int t_local = q * 32 + lane;
        long long gu = 0;
        int sat = 0;
        for (long long u = u0; u < u1; u++, gu++) {
            const int b = (int)(gu & 1);
            tc::mbar_wait(&mb_dfull[b], (uint32_t)((gu >> 1) & 1), p.status);
            tc::fence_after();
            const int s = (int)(u / ((long long)p.C * p.tiles));
            const int c = (int)((u / p.tiles) % p.C);
            const int t = (int)(u % p.tiles) * kTile + t_local;
            const size_t row = (((size_t)s * p.C + c) * p.T + t) * p.K * p.P * 2;   // [s][c][t][k][p][2]
            // 8 beams at a time: both pols' (re, im) of beams k0..k0+7, in output order
            for (int c0 = 0; c0 < ncols; c0 += 16) {
                int v[2][16];
#pragma unroll
                for (int pol = 0; pol < 2; pol++) {
                    if (pol < p.P) {
                        uint32_t r[16];
                        tc::tmem_ld16(tmem + lane_base + (uint32_t)b * dcols + (uint32_t)(pol * ncols + c0), r);
                        tc::tmem_wait_ld();
#pragma unroll
                        for (int j = 0; j < 16; j++) v[pol][j] = __float2int_rn(__uint_as_float(r[j]));
                    } else {
#pragma unroll
                        for (int j = 0; j < 16; j++) v[pol][j] = 0;
                    }
                }
                if (t >= p.T) continue;
                const int k0 = c0 >> 1;
                if (p.shift < 0) {
                    int32_t *o = reinterpret_cast<int32_t *>(p.beams) + row + (size_t)k0 * p.P * 2;
                    if (p.P == 2) {
#pragma unroll
                        for (int j = 0; j < 8; j++)             // beam k0 + j: X (re, im), Y (re, im)
                            reinterpret_cast<int4 *>(o)[j] = make_int4(v[0][2 * j], v[0][2 * j + 1], v[1][2 * j],
                                                                       v[1][2 * j + 1]);
                    } else {
#pragma unroll
                        for (int j = 0; j < 4; j++)
                            reinterpret_cast<int4 *>(o)[j] = make_int4(v[0][4 * j], v[0][4 * j + 1], v[0][4 * j + 2],
                                                                       v[0][4 * j + 3]);
                    }
                } else {
                    uint32_t wds[8];                             // P = 2: 8 words; P = 1: 4
#pragma unroll
                    for (int j = 0; j < 8; j++) {                // beam k0 + j
                        const uint32_t b0 = (uint8_t)requant(v[0][2 * j], p.shift, sat);
                        const uint32_t b1 = (uint8_t)requant(v[0][2 * j + 1], p.shift, sat);
                        if (p.P == 2) {
                            const uint32_t b2 = (uint8_t)requant(v[1][2 * j], p.shift, sat);
                            const uint32_t b3 = (uint8_t)requant(v[1][2 * j + 1], p.shift, sat);
                            wds[j] = b0 | (b1 << 8) | (b2 << 16) | (b3 << 24);
                        } else {
                            const uint32_t h = b0 | (b1 << 8);
                            if (j & 1) wds[j >> 1] |= h << 16;
                            else wds[j >> 1] = h;
                        }
                    }
                    int8_t *o = reinterpret_cast<int8_t *>(p.beams) + row + (size_t)k0 * p.P * 2;
                    if (p.P == 2) {                              // 32 bytes
                        reinterpret_cast<uint4 *>(o)[0] = make_uint4(wds[0], wds[1], wds[2], wds[3]);
                        reinterpret_cast<uint4 *>(o)[1] = make_uint4(wds[4], wds[5], wds[6], wds[7]);
                    } else {                                     // P = 1: 16 bytes
                        reinterpret_cast<uint4 *>(o)[0] = make_uint4(wds[0], wds[1], wds[2], wds[3]);
                    }
                }
            }
            tc::fence_before();
            tc::mbar_arrive_warp(&mb_dempty[b]);
        }
        if (p.nsat) {
            for (int o = 16; o; o >>= 1) sat += __shfl_xor_sync(0xffffffffu, sat, o);
            if (lane == 0 && sat) atomicAdd(p.nsat, (unsigned long long)sat);
        }
    }

    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    if (warp == 0) tc::tmem_dealloc(tmem, alloc);
}

}  // namespace

extern "C" hai_status hai_beamform(hai_ctx *ctx, const int8_t *volt, const int8_t *w, int S, int C, int T, int K,
                                   int N, int P, int requant_shift, void *beams, long long *n_saturated,
                                   void *stream) {
    if (!ctx) return hai_fail(HAI_ERR_INVALID_ARG, "hai_beamform: ctx is NULL");
    if (S < 0 || C < 0 || T < 0 || K <= 0 || N <= 0 || (P != 1 && P != 2) || requant_shift > 30)
        return hai_fail(HAI_ERR_INVALID_ARG, "hai_beamform: bad size, polarisation count or shift");
    if (N % 8 != 0 || N > 512 || (2 * K) % 16 != 0 || K > 64)
        return hai_fail(HAI_ERR_UNSUPPORTED,
                        "hai_beamform: this build needs N a multiple of 8 and <= 512 (exact FP32 block), "
                        "K a multiple of 8 and <= 64");
    if ((long long)S * C * T == 0) return HAI_OK;
    if (!volt || !w || !beams) return hai_fail(HAI_ERR_INVALID_ARG, "hai_beamform: NULL buffer");
    if ((((uintptr_t)volt) & 15) != 0 || (((uintptr_t)beams) & 15) != 0)
        return hai_fail(HAI_ERR_INVALID_ARG, "hai_beamform: volt and beams must be 16-byte aligned");
    if (hai_fault_injected("launch")) return hai_fail(HAI_ERR_CUDA, "hai_beamform: injected launch failure");
    HAI_CUDA_TRY(cudaSetDevice(ctx->device));
    cudaStream_t st = (cudaStream_t)stream;
    BfParams p;
    p.volt = volt;
    p.w = w;
    p.S = S;
    p.C = C;
    p.T = T;
    p.K = K;
    p.ne = N;
    p.P = P;
    p.tiles = (T + kTile - 1) / kTile;
    p.nunits = (long long)S * C * p.tiles;
    const int grid = (int)std::min<long long>(p.nunits, ctx->num_sms);
    p.shift = requant_shift;
    p.beams = beams;
    p.nsat = reinterpret_cast<unsigned long long *>(n_saturated);
    p.status = ctx->d_status;
    const size_t bbytes = (size_t)(2 * K / 8) * ((N + kChunkE - 1) / kChunkE * kChunkE) * 32;
    const size_t smem = kAStages * kABytes + (size_t)P * bbytes;
    if (smem > (size_t)ctx->smem_optin)
        return hai_fail(HAI_ERR_UNSUPPORTED, "hai_beamform: weights of one station exceed shared memory");
    if (!ctx->bf_ready || hai_fault_injected("registers")) {      // once: both are the build's and the device's
        const hai_status ready = hai_allow_dyn_smem_regs(bf_kernel, ctx->smem_optin, kLaunchRegs);
        if (ready != HAI_OK) return ready;
        ctx->bf_ready = true;
    }
    const int pidx = prof_begin(ctx, st);
    bf_kernel<<<grid, kThreads, smem, st>>>(p);
    prof_end(ctx, pidx, st);
    prof_count(ctx, 1);
    HAI_CUDA_TRY(cudaGetLastError());
    return HAI_OK;
}
