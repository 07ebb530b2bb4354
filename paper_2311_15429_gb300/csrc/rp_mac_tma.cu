// Spectral multiply-accumulate + inverse column FFT, fed by the tensor memory
// accelerator.
//
// For every padded shape with a column class (rp_internal.h).  Same
// arithmetic as k_mac_inv_column (the sum over a target's (source, lag)
// entries of G_m * S(l - m), Eq. 12 in the spectral domain, then the inverse
// FFT along z kept to the target's z < nz), restructured so that the operands
// stream through shared memory asynchronously:
//
//   * persistent blocks, one per SM, each walking (kx, 16-ky) column tiles
//     (or two fields or one of a tile, mac_tma_fields);
//   * the last warp is the producer: one lane issues bulk copies
//     (cp.async.bulk) into two rings of shared-memory stages, one for the
//     entries' kernel tiles (M rows x 128 B, or 64 B for a real kernel) and
//     one for their source field tiles.  The ring stores a tile's four field
//     tiles next to each other, so one copy brings FPC of them (4 up to
//     M = 96, 2 at 128, 1 at 192): the copy engine spends a roughly fixed time
//     per copy, and copies under about 16 KB leave HBM bandwidth unused.  Each
//     stage is guarded by a "full" mbarrier (transaction bytes) and an "empty"
//     mbarrier (one arrival per consumer warp);
//   * the other CW warps (8, 12 or 16, picked per size class by timing the
//     variants on the context's own plan) are consumers: they multiply-accumulate in registers,
//     then write the tile to a separate shared-memory region, where the FFT
//     warps run the inverse column transform (the two-stage tile transform of
//     rp_fft.cuh) and store T2, so the producer keeps prefetching the next
//     tile's operands meanwhile.
//
// Every wait is bounded (clock64 limit).  On a timeout the kernel sets the
// context's error flag, stops waiting, and the producer waits (bounded) for
// the copies it has in flight before the block exits.
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#define RP_SCALAR_COMPLEX
#include "rp_fft.cuh"
#include "rp_internal.h"

namespace rp {

namespace {

constexpr long long kWaitLimit = 4000000000LL;   // SM clock cycles (about 2 s)
constexpr int kMaxStages = 24;
constexpr int kKernelStages = 2;   // depth of the kernel-tile ring
constexpr int kFftWarps = 7;       // warps of the inverse column FFT and the T2 store: with the
                                   // producer, 8 + 8/12/16 MAC warps, a whole number of warps per
                                   // scheduler for the register split; 7 keep up with tiles of few
                                   // entries (the self lags alone), where 3 left the MAC warps waiting

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t *bar, int count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Wait for the phase of `parity` to complete; false after kWaitLimit cycles.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, long long limit = kWaitLimit)
{
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, parity))
        if (clock64() - t0 > limit) return false;
    return true;
}

// Self-test of the bounded wait: one mbarrier that nothing arrives on, waited
// through mbar_wait with a short limit; it runs out, raises the error flag
// and the block exits.
__global__ void k_wait_selftest(long long limit, int *err)
{
    __shared__ uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (threadIdx.x == 0 && !mbar_wait(&bar, 0, limit)) atomicExch(err, 1);
}

// Contiguous copy of `bytes` (multiple of 16, both addresses 16-byte aligned)
// by the bulk-copy engine, completing on `bar`, with an L2 eviction-priority
// policy for the source lines.
__device__ __forceinline__ void bulk_load(void *dst, const void *src, uint32_t bytes, uint64_t *bar, uint64_t policy)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(
            smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(smem_u32(bar)), "l"(policy)
        : "memory");
}

__device__ __forceinline__ uint64_t policy_evict_first()
{
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}

__device__ __forceinline__ uint64_t policy_evict_last()
{
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
    return p;
}

__device__ __forceinline__ uint64_t policy_evict_normal()
{
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(p));
    return p;
}

template <class T>
__device__ __forceinline__ int owner(const T *arr, int lo, int hi, int b, int T::*field)
{
    while (hi - lo > 1) {
        int mid = (lo + hi) >> 1;
        if (arr[mid].*field <= b) lo = mid; else hi = mid;
    }
    return lo;
}

// Kahan-compensated addition of two values at a time in packed FP32: s + c
// carries the sum of the added terms with the rounding of each addition kept
// in c (the error stays near one rounding of the sum of magnitudes, whatever
// the number of terms); the total is s - c.  A difference a - b is b * -1 + a,
// the same one rounding.
__device__ __forceinline__ void kahan_add2(float &s0, float &s1, float &c0, float &c1, float2 x)
{
    const float2 minus = make_float2(-1.0f, -1.0f), s = make_float2(s0, s1), c = make_float2(c0, c1);
    const float2 y = __ffma2_rn(c, minus, x);
    const float2 t = __fadd2_rn(s, y);
    const float2 d = __ffma2_rn(y, minus, __ffma2_rn(s, minus, t));
    s0 = t.x; s1 = t.y;
    c0 = d.x; c1 = d.y;
}

// barrier `id` among the first (or last) `threads` threads of the block
__device__ __forceinline__ void named_sync(int id, int threads)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// Inverse FFT along z of the NF field tiles of `acc` ([field][M][16], dense;
// fields f0 .. f0 + NF - 1) by the two-stage tile transform (rp_fft.cuh), its
// tasks shared by warps w = 0 .. nw-1 (this one is w; barrier `bar` of nw
// warps between the stages), then rows z < nz (row z of the transform sits at
// tile_row(z)) to T2.
template <int M, int NF>
__device__ __forceinline__ void column_tile_store(float2 *acc, const float2 *tw, const InvTarget &T, int local, int f0,
                                                  int w, int nw, int lane, int bar)
{
    constexpr int B = M / 16, FS = M * kTileY;
    const int tid = w * 32 + lane, nt = nw * 32;
    // the target's extents before the transform, not on its way out (two 28^3
    // 35.8 -> 34.9 us per step, one 64^3 74.0 -> 72.9)
    const int nz = T.nz, my = T.ay.M, nty = my / kTileY, kxi = local / nty, ky0 = (local - kxi * nty) * kTileY;
    const long long t2_field = (long long)T.kx * nz * my;
    float2 *dst = T.t2 + (long long)f0 * t2_field + (long long)kxi * nz * my + ky0;
    for (int i = tid; i < NF * 16 * B; i += nt) {
        const int c = i & 15, rest = i >> 4, f = rest / B, n2 = rest - f * B;
        tile_stage1<B, true, false>(acc + f * FS, tw, M, c, n2);
    }
    named_sync(bar, nt);
    for (int i = tid; i < NF * 256; i += nt) tile_stage2<B, true>(acc + (i >> 8) * FS, i & 15, (i >> 4) & 15);
    named_sync(bar, nt);
    for (int i = tid; i < NF * nz * (kTileY / 2); i += nt) {
        const int f = i / (nz * (kTileY / 2)), rem = i - f * nz * (kTileY / 2);
        const int zi = rem >> 3, pp = rem & 7;
        *reinterpret_cast<float4 *>(dst + f * t2_field + (long long)zi * my + 2 * pp) =
            *reinterpret_cast<const float4 *>(acc + f * FS + tile_row<B>(zi) * kTileY + 2 * pp);
    }
}

// Warps of the inverse column FFT (FW): seven beside the plain sum's MAC
// warps; beside the compensated ones, whose accumulators need the registers,
// three, which keep up with tiles of many entries and leave the multiply-adds
// the issue slots.  Tiles of few entries (the self lags alone) wait for them
// where a block has several: there as many as the registers leave, seven at
// M = 64 and five at 96 (at 128 and 192 none are left; 32 and 48 transform as
// fast with three).  32 x 48^3, 4 entries a tile: MAC 382 us with three, 354
// with five; 2 x 48^3, 9 entries: 52.6 and 54.4; 64^3 class of the mixed
// sizes, 4 entries: 27.3 with three, 25.9 with seven; four 27^3 neighbours, 19
// entries: 62.2 and 66.1; four far 24^3, 3 entries: the step 39.1 with three,
// 41.0 with seven.  A block's last unit is every warp's: with one unit a block
// (one 24^3) 17.9 with three, 23.1 with seven.
constexpr int kFewEntries = 6;
__host__ __device__ constexpr int few_fft_warps(int M) { return M == 64 ? 7 : M == 96 ? 5 : 3; }

// A block's unit of work is FH fields of one tile: all four (the kernel tile
// read once), unless
//   * M = 192, compensated: a MAC thread would hold 128 floats of sums and
//     compensation for four fields and spill them, so a unit is two;
//   * the plan's tiles are so few that half of the SMs would have none
//     (elongated and small grids): two fields or one, the kernel tile then
//     read again from L2 by the neighbouring block (mac_tma_fields).
// Every field is summed in the same order whatever the unit.
//
// Units go target by target, except (share) where the targets of a launch
// have the same tiles and two of them read the same source slots, as
// neighbouring domains do: then the same tile of every target in turn, so that
// a slot's tile is read from HBM once and by the other targets from L2 (as
// long as blocks in flight hold: 152 x some 0.4 MB).  Four 27^3 neighbours, 76
// entries of 4.3 MB over 155 MB of distinct slots: 93.4 -> 85.3 us per step.

// M: padded FFT size along z; CW: multiply-accumulate warps (the block has
// CW + FW + 1); FPC: field tiles per ring copy (1, 2 or 4; they are
// contiguous in the ring); FH: fields of a unit; COMP: the sum over (source,
// lag) entries is Kahan-compensated per spectral coefficient (the default;
// RP_FLAG_PLAIN_SUM selects the plain chain).
template <int M, int CW, int FPC, int FH, int FW, bool COMP>
__global__ void __launch_bounds__((CW + FW + 1) * 32, 1)
    k_mac_tma(const InvTarget *__restrict__ tgts, int t0, int t1, int tile_lo, int nunits, int share,
              const MacEntry *__restrict__ entries, long long step, int clamp, int ns, int *err)
{
    constexpr int STAGE = M * 128;                  // one M x 16 complex tile
    constexpr int SSTAGE = FPC * STAGE;             // FPC field tiles of one entry
    constexpr int NG = kKernelStages;
    constexpr int kConsumerWarps = CW;
    constexpr int RSTEP = kConsumerWarps * 32 / 8;   // rows covered by one pass of the consumers
    constexpr int ROWS = (M + RSTEP - 1) / RSTEP;
    constexpr int FS = M * kTileY;                   // float2 per field of the FFT tile (dense rows)
    constexpr int NFG = 4 / FH;                      // units per tile: unit u is fields FH (u % NFG) .. of tile u / NFG
    static_assert(FH % FPC == 0, "k_mac_tma: whole field copies per unit");
    extern __shared__ __align__(128) unsigned char smem[];
    unsigned char *sstages = smem;                                   // [ns][SSTAGE]
    unsigned char *gstages = smem + (size_t)ns * SSTAGE;             // [NG][STAGE]
    float2 *acc = reinterpret_cast<float2 *>(gstages + (size_t)NG * STAGE);
    float2 *tw = acc + FH * FS;                                      // acc: [FH][M][16]
    uint64_t *sfull = reinterpret_cast<uint64_t *>(tw + M);
    uint64_t *sempty = sfull + ns;
    uint64_t *gfull = sempty + ns;
    uint64_t *gempty = gfull + NG;
    uint64_t *accfull = gempty + NG;    // the FFT tile holds a tile's sums (one arrival per MAC warp)
    uint64_t *accempty = accfull + 1;   // the FFT warps are done with it (one arrival per FFT warp)
    volatile int *abort_flag = reinterpret_cast<volatile int *>(accempty + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < ns; ++s) {
            mbar_init(&sfull[s], 1);
            mbar_init(&sempty[s], kConsumerWarps);
        }
        for (int s = 0; s < NG; ++s) {
            mbar_init(&gfull[s], 1);
            mbar_init(&gempty[s], kConsumerWarps);
        }
        mbar_init(accfull, kConsumerWarps);
        mbar_init(accempty, FW);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    load_twiddles(tw, tgts[t0].tw_z, M);
    pdl_trigger();
    pdl_wait();   // the newest ring slot is written by the column pass; T2 was read by the last plane pass
    if (step < 0) step = *tgts[t0].d_step;   // graph replay: the step from the device counter
    __syncthreads();

    // unit u: its target, tile of the target and first field; target by target,
    // or (share) the same tile of every target in turn
    auto unit = [&](int u, int &local, int &f0) -> const InvTarget & {
        const int w = u / NFG, nt = t1 - t0;
        f0 = (u - w * NFG) * FH;
        if (share) {
            local = w / nt;
            return tgts[t0 + w - local * nt];
        }
        const InvTarget &T = tgts[owner(tgts, t0, t1, w + tile_lo, &InvTarget::tile0)];
        local = w + tile_lo - T.tile0;
        return T;
    };

    // wait for a phase; false (and the error raised) on abort/timeout
    auto wait_or_abort = [&](uint64_t *bar, uint32_t parity) {
        if (*abort_flag) return false;
        if (!mbar_wait(bar, parity)) {
            *abort_flag = 1;
            atomicExch(err, 1);
            return false;
        }
        return true;
    };

    if (warp == kConsumerWarps + FW) {
        // ------------------------------------------------------------ producer
        if (lane != 0) return;
        uint32_t qg = 0, qs = 0;
        bool ok = true;
        // The kernel tiles (tens of MB, read every step) stay in L2; the ring
        // tiles pass through without evicting them, unless another target is
        // about to read the same ones.
        const uint64_t keep = policy_evict_last(), stream = share ? policy_evict_normal() : policy_evict_first();
        // wait until stage q of a ring is free; false (and the error raised) on abort/timeout
        auto acquire = [&](uint64_t *empty, int n, uint32_t q) {
            if (*abort_flag || !mbar_wait(&empty[q % n], ((q / n) & 1) ^ 1)) {
                *abort_flag = 1;
                atomicExch(err, 1);
                return false;
            }
            return true;
        };
        for (int u = blockIdx.x; u < nunits && ok; u += gridDim.x) {
            int local, f0;
            const InvTarget &T = unit(u, local, f0);
            const long long tile_off = (long long)local * M * kTileY;
            const int nr = T.er - T.e0, nc = T.e1 - T.er;   // real (self) entries come first
            for (int k = 0; k < nr + nc && ok; ++k) {
                const MacEntry &E = entries[T.e0 + k];
                long long j = step - E.lag;
                if (clamp && j < 0) j = 0;
                const int slot = (int)(j % E.depth);
                // the kernel tile
                if (!(ok = acquire(gempty, NG, qg))) break;
                {
                    const int s = qg % NG;
                    const uint32_t bytes = E.is_real ? M * 64 : M * 128;
                    const void *src = E.is_real ? (const void *)(static_cast<const float *>(E.g) + tile_off)
                                                : (const void *)(static_cast<const float2 *>(E.g) + tile_off);
                    mbar_expect_tx(&gfull[s], bytes);
                    bulk_load(gstages + (size_t)s * STAGE, src, bytes, &gfull[s], keep);
                    ++qg;
                }
                // the unit's field tiles of the source spectrum, FPC per copy
                const float2 *fields = E.ring + (long long)slot * E.slot_elems + 4 * tile_off;
                for (int o = 0; o < FH / FPC; ++o) {
                    if (!(ok = acquire(sempty, ns, qs))) break;
                    const int s = qs % ns;
                    mbar_expect_tx(&sfull[s], SSTAGE);
                    bulk_load(sstages + (size_t)s * SSTAGE, fields + (long long)(f0 + o * FPC) * M * kTileY,
                              SSTAGE, &sfull[s], stream);
                    ++qs;
                }
            }
        }
        // no copy may still be landing when the block exits
        for (uint32_t r = qg > (uint32_t)NG ? qg - NG : 0; r < qg; ++r)
            if (!mbar_wait(&gfull[r % NG], (r / NG) & 1)) atomicExch(err, 1);
        for (uint32_t r = qs > (uint32_t)ns ? qs - ns : 0; r < qs; ++r)
            if (!mbar_wait(&sfull[r % ns], (r / ns) & 1)) atomicExch(err, 1);
        return;
    }

    // Hand-over, per unit: the MAC warps accumulate it in registers, store it
    // to the FFT tile and signal accfull; the FFT warps transform and store it
    // while the MAC warps accumulate the next, then signal accempty.  A
    // block's last unit has no successor, so all its consumer warps share
    // that transform (barrier 2 in place of the two signals).
    constexpr int kBarFft = 1, kBarAll = 2;
    if (warp >= kConsumerWarps) {
        // ------------------------------------------------------------ FFT warps
        const int fw = warp - kConsumerWarps;
        uint32_t it = 0;
        for (int u = blockIdx.x; u < nunits; u += gridDim.x, ++it) {
            int local, f0;
            const InvTarget &T = unit(u, local, f0);
            if (u + (int)gridDim.x >= nunits) {
                named_sync(kBarAll, (kConsumerWarps + FW) * 32);
                column_tile_store<M, FH>(acc, tw, T, local, f0, warp, kConsumerWarps + FW, lane, kBarAll);
                return;
            }
            const bool have = wait_or_abort(accfull, it & 1);
            // on an abort the sums are not used: skip the transform, keep the barriers
            if (have) column_tile_store<M, FH>(acc, tw, T, local, f0, fw, FW, lane, kBarFft);
            else {
                named_sync(kBarFft, FW * 32);
                named_sync(kBarFft, FW * 32);
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(accempty);
        }
        return;
    }

    // ---------------------------------------------------------------- MAC warps
    const int p = threadIdx.x & 7, r0 = threadIdx.x >> 3;   // ky pair p, rows r0 + RSTEP i
    uint32_t qg = 0, qs = 0, it = 0;

    // wait for stage q of a ring; its address (or nullptr after an abort/timeout)
    auto take = [&](unsigned char *base, int bytes, uint64_t *full, int n, uint32_t q) -> const unsigned char * {
        if (!wait_or_abort(&full[q % n], (q / n) & 1)) return nullptr;
        return base + (size_t)(q % n) * bytes;
    };
    auto give = [&](uint64_t *empty, int n, uint32_t q) {
        __syncwarp();
        if (lane == 0) mbar_arrive(&empty[q % n]);
    };

    for (int u = blockIdx.x; u < nunits; u += gridDim.x, ++it) {
        int local, f0;
        const InvTarget &T = unit(u, local, f0);
        {   // fields f0 .. f0 + FH - 1
            float4 a[ROWS][FH];
            float4 cmp[COMP ? ROWS : 1][FH];   // Kahan compensation (COMP only)
#pragma unroll
            for (int i = 0; i < ROWS; ++i)
#pragma unroll
                for (int f = 0; f < FH; ++f) a[i][f] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int i = 0; i < (COMP ? ROWS : 1); ++i)
#pragma unroll
                for (int f = 0; f < FH; ++f) cmp[i][f] = make_float4(0.f, 0.f, 0.f, 0.f);

            for (int e = T.e0; e < T.er; ++e) {   // real kernels (self pair)
                float2 g[ROWS];
                const unsigned char *st = take(gstages, STAGE, gfull, NG, qg);
                const float *Gt = reinterpret_cast<const float *>(st);   // [M][16]
#pragma unroll
                for (int i = 0; i < ROWS; ++i) {
                    const int r = r0 + RSTEP * i;
                    g[i] = (st && r < M) ? *reinterpret_cast<const float2 *>(Gt + r * 16 + 2 * p)
                                         : make_float2(0.f, 0.f);
                }
                give(gempty, NG, qg++);
#pragma unroll
                for (int o = 0; o < FH / FPC; ++o) {
                    const unsigned char *sf = take(sstages, SSTAGE, sfull, ns, qs);
#pragma unroll
                    for (int ff = 0; ff < FPC; ++ff) {
                        const int f = o * FPC + ff;
                        const float4 *S4 = reinterpret_cast<const float4 *>(sf + ff * STAGE);   // [M][8]
#pragma unroll
                        for (int i = 0; i < ROWS; ++i) {
                            const int r = r0 + RSTEP * i;
                            if (sf && r < M) {
                                const float4 s = S4[r * 8 + p];
                                if constexpr (COMP) {
                                    float4 &c = cmp[COMP ? i : 0][f];
                                    kahan_add2(a[i][f].x, a[i][f].y, c.x, c.y, make_float2(g[i].x * s.x, g[i].x * s.y));
                                    kahan_add2(a[i][f].z, a[i][f].w, c.z, c.w, make_float2(g[i].y * s.z, g[i].y * s.w));
                                } else {
                                    a[i][f].x = fmaf(g[i].x, s.x, a[i][f].x);
                                    a[i][f].y = fmaf(g[i].x, s.y, a[i][f].y);
                                    a[i][f].z = fmaf(g[i].y, s.z, a[i][f].z);
                                    a[i][f].w = fmaf(g[i].y, s.w, a[i][f].w);
                                }
                            }
                        }
                    }
                    give(sempty, ns, qs++);
                }
            }
            for (int e = T.er; e < T.e1; ++e) {   // complex kernels (other sources)
                float4 g[ROWS];
                const unsigned char *st = take(gstages, STAGE, gfull, NG, qg);
                const float4 *G4 = reinterpret_cast<const float4 *>(st);
#pragma unroll
                for (int i = 0; i < ROWS; ++i) {
                    const int r = r0 + RSTEP * i;
                    g[i] = (st && r < M) ? G4[r * 8 + p] : make_float4(0.f, 0.f, 0.f, 0.f);
                }
                give(gempty, NG, qg++);
#pragma unroll
                for (int o = 0; o < FH / FPC; ++o) {
                    const unsigned char *sf = take(sstages, SSTAGE, sfull, ns, qs);
#pragma unroll
                    for (int ff = 0; ff < FPC; ++ff) {
                        const int f = o * FPC + ff;
                        const float4 *S4 = reinterpret_cast<const float4 *>(sf + ff * STAGE);
#pragma unroll
                        for (int i = 0; i < ROWS; ++i) {
                            const int r = r0 + RSTEP * i;
                            if (sf && r < M) {
                                const float4 s = S4[r * 8 + p];
                                float4 &x = a[i][f];
                                if constexpr (COMP) {
                                    float4 &c = cmp[COMP ? i : 0][f];
                                    kahan_add2(x.x, x.y, c.x, c.y, make_float2(fmaf(g[i].x, s.x, -g[i].y * s.y),
                                                                               fmaf(g[i].x, s.y, g[i].y * s.x)));
                                    kahan_add2(x.z, x.w, c.z, c.w, make_float2(fmaf(g[i].z, s.z, -g[i].w * s.w),
                                                                               fmaf(g[i].z, s.w, g[i].w * s.z)));
                                } else {
                                    x.x = fmaf(g[i].x, s.x, fmaf(-g[i].y, s.y, x.x));
                                    x.y = fmaf(g[i].x, s.y, fmaf(g[i].y, s.x, x.y));
                                    x.z = fmaf(g[i].z, s.z, fmaf(-g[i].w, s.w, x.z));
                                    x.w = fmaf(g[i].z, s.w, fmaf(g[i].w, s.z, x.w));
                                }
                            }
                        }
                    }
                    give(sempty, ns, qs++);
                }
            }

            // hand the sums to the FFT warps once they are done with the previous unit
            if (it == 0 || wait_or_abort(accempty, (it - 1) & 1)) {
#pragma unroll
                for (int i = 0; i < ROWS; ++i) {
                    const int r = r0 + RSTEP * i;
                    if (r >= M) continue;
#pragma unroll
                    for (int f = 0; f < FH; ++f) {
                        if constexpr (COMP) {   // the compensated total
                            const float4 &c = cmp[COMP ? i : 0][f];
                            a[i][f] = make_float4(a[i][f].x - c.x, a[i][f].y - c.y, a[i][f].z - c.z, a[i][f].w - c.w);
                        }
                        *reinterpret_cast<float4 *>(acc + f * FS + r * kTileY + 2 * p) = a[i][f];
                    }
                }
            }
            if (u + (int)gridDim.x >= nunits) {
                named_sync(kBarAll, (kConsumerWarps + FW) * 32);
                column_tile_store<M, FH>(acc, tw, T, local, f0, warp, kConsumerWarps + FW, lane, kBarAll);
                return;
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(accfull);
        }
    }
}

constexpr int fields_per_copy(int M, int fh)
{
    const int f = M <= 96 ? 4 : (M == 128 ? 2 : 1);
    return f < fh ? f : fh;
}

// every (class, fields of a unit) that runs: M = 192, compensated, has no unit of four
#define RP_TMA_CLASSES(X) X(32) X(48) X(64) X(96) X(128) X(192)
#define RP_TMA_FIELDS(X, M) X(M, 4) X(M, 2) X(M, 1)
constexpr bool unit_runs(int M, int fh, bool comp) { return !(comp && M == 192 && fh == 4); }

template <int M, int FH, class F>
cudaError_t for_variants(F &&f)   // f(kernel, multiply-add warps, FFT warps, compensated)
{
    constexpr int FPC = fields_per_copy(M, FH);
    cudaError_t e;
    constexpr int FW = kFftWarps, FEW = few_fft_warps(M);
    if ((e = f(k_mac_tma<M, 8, FPC, FH, FW, false>, 8, FW, false)) ||
        (e = f(k_mac_tma<M, 12, FPC, FH, FW, false>, 12, FW, false)) ||
        (e = f(k_mac_tma<M, 16, FPC, FH, FW, false>, 16, FW, false)))
        return e;
    if constexpr (unit_runs(M, FH, true)) {
        if ((e = f(k_mac_tma<M, kCompWarps, FPC, FH, 3, true>, kCompWarps, 3, true))) return e;
        if constexpr (FEW != 3 && FH == 4) return f(k_mac_tma<M, kCompWarps, FPC, FH, FEW, true>, kCompWarps, FEW, true);
    }
    return cudaSuccess;
}

}  // namespace

cudaError_t launch_wait_selftest(long long limit_cycles, int *d_err, cudaStream_t s)
{
    k_wait_selftest<<<1, 32, 0, s>>>(limit_cycles, d_err);
    return cudaGetLastError();
}

// Fields of a unit: as many as the registers hold, halved while the units
// would still not outnumber the SMs: a block alone reads about 1/152 of the
// HBM bandwidth, so idle SMs cost it.  Two 16 x 16 x 60 boxes (68 tiles of M =
// 128, 40 entries): 54.7 us per step with four fields, 44.2 with two; one 8 x
// 8 x 90 box (17 tiles of M = 192): 40.3 with two, 33.5 with one.  Beyond one
// unit per SM the shorter copies only cost (16 x 16 x 96 pair: 67.7 with two,
// 80.6 with one).  Nor are tiles of few entries split (160 KB, some 4 us for
// one block) in a plan whose plane passes have fewer blocks than three quarters
// of the SMs: those start beside the MAC, on the SMs that it leaves free, and
// wait there.  Two 14^3 (112 plane blocks, 6 entries of 20 KB): 20.5 with two
// fields, 18.2 with four; one 20^3 (80, 3 of 30 KB) 18.1 and 17.0; two 16^3
// (128, 6 of 20 KB), whose blocks pile up on those SMs, 17.3 and 21.4.
int mac_tma_fields(int M, bool comp, int ntiles, double entries, int plane_blocks, int sms)
{
    int fh = unit_runs(M, 4, comp) ? 4 : 2;
    const double bytes = entries * 5 * M * 128;   // kernel and four field tiles of M x 16 an entry
    if (bytes <= 160 * 1024 && 4 * plane_blocks < 3 * sms) return fh;
    while (fh > 1 && ntiles * (4 / fh) * 2 <= sms) fh /= 2;
    return fh;
}

// FFT warps of a launch whose targets have `entries` (source, lag) terms on average.
int mac_tma_fft_warps(int M, bool comp, int fh, int ntiles, double entries, int sms)
{
    if (!comp) return kFftWarps;
    return fh == 4 && ntiles > sms && entries <= kFewEntries ? few_fft_warps(M) : 3;
}

int mac_tma_stages(int M, int smem_optin, int fh)
{
    const long long sstage = (long long)fields_per_copy(M, fh) * M * 128;
    const long long fixed = (long long)mac_tma_smem(M, 0, fh);   // kernel-tile ring, FFT tile, twiddles, barriers
    long long n = (smem_optin - fixed) / (sstage + 16);      // + two mbarriers per stage
    if (n > kMaxStages) n = kMaxStages;
    return (int)n;
}

size_t mac_tma_smem(int M, int nstages, int fh)
{
    const size_t stage = (size_t)M * 128;
    return (size_t)nstages * fields_per_copy(M, fh) * stage + kKernelStages * stage +
           sizeof(float2) * (fh * (size_t)M * kTileY + M) + 16 * ((size_t)nstages + kKernelStages) + 16 + 16;
}

cudaError_t open_mac_tma_smem_limit(int max_optin)
{
    cudaError_t e;
    const auto open = [&](auto kern, int, int, bool) {
        return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, max_optin);
    };
#define X(M, FH) \
    if ((e = for_variants<M, FH>(open))) return e;
#define Y(M) RP_TMA_FIELDS(X, M)
    RP_TMA_CLASSES(Y)
#undef Y
#undef X
    return cudaSuccess;
}

cudaError_t launch_mac_tma(int cls, int cw, bool comp, const InvTarget *d_tgts, int t0, int t1, int tile_lo,
                           int ntiles, bool share, const MacEntry *d_entries, long long step, int clamp, int fh, int fw,
                           int nstages, int sms, int *d_err, cudaStream_t s)
{
    if (ntiles <= 0) return cudaSuccess;
    if (comp ? cw != kCompWarps : (cw != 8 && cw != 12 && cw != 16)) return cudaErrorInvalidValue;
    if (nstages < 2 || nstages > kMaxStages || (fh != 4 && fh != 2 && fh != 1) || !unit_runs(cls, fh, comp))
        return cudaErrorInvalidValue;
    const size_t smem = mac_tma_smem(cls, nstages, fh);
    const int threads = (cw + fw + 1) * 32;
    const int nunits = ntiles * (4 / fh), grid = nunits < sms ? nunits : sms;
    cudaError_t e = cudaErrorInvalidValue;
    const auto go = [&](auto kern, int w, int f, bool c) {
        if (w == cw && f == fw && c == comp)
            e = launch_pdl(kern, dim3(grid), dim3(threads), smem, s, d_tgts, t0, t1, tile_lo, nunits, share ? 1 : 0,
                           d_entries, step, clamp, nstages, d_err);
        return cudaSuccess;
    };
#define X(M, FH) \
    if (cls == M && fh == FH) for_variants<M, FH>(go);
#define Y(M) RP_TMA_FIELDS(X, M)
    RP_TMA_CLASSES(Y)
#undef Y
#undef X
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace rp
