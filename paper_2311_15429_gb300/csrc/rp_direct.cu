// Direct retarded sum (the plain path of every pair in RP_MODE_DIRECT, and
// of pairs of unequal spacing in RP_MODE_FFT):
//
//   P(r_k, l) += sum_{k' in source} h_s^3 S(k', l - tau) / R,   tau = R/(c dt),
//   S(l - tau) = (1 - w) S_{l-m} + w S_{l-m-1},  m = floor(tau), w = tau - m
//
// (Eq. 8 with the hat interpolation of Eq. 7; at R = 0 of the self pair the
// cell-averaged weight C h^2 at lag 0).
//
// Bound by instruction issue and by what shared memory returns to registers
// (128 B/clk per SM, broadcasts included), about 1e9 node pairs per step of
// two 32^3 grids against some 5 MB of samples.  What that asks for:
//   * a thread owns four target nodes and walks the sources with the geometry
//     of two in packed FP32 pairs (add/mul/fma.f32x2), and floor by a
//     round-down addition of 2^23 (no conversion);
//   * the samples lie as 16 bytes (rho, Jx, Jy, Jz) per [lag][source]; four
//     neighbours along x no farther apart than light goes in a step (SHARED)
//     see at most two lag intervals, so three samples serve all four.  Where
//     they are farther apart, or rows so short that groups of four would be
//     mostly padding, each target loads its own two (direct_groups);
//   * the eight warps of a block share 128 targets and divide a staged tile of
//     sources, and the sources run in parts in blocks beside one another
//     (direct_parts), so that small grids fill the chip too; k_direct_sum adds
//     the parts in order;
//   * every term's product and addition is compensated (direct_add), as are
//     the additions of the warps' and the parts' sums;
//   * lengths are in bohr but for a power of two (DirectPair::scale), so that
//     positions on a dyadic grid and their differences stay exact, and no
//     square of a distance underflows whatever c dt is.  (In units of c dt,
//     with runs of 8 terms in plain FP32, the sum took 1713 us in place of
//     1870, at 2 to 5 times the error on white noise at h = 0.25, and NaN from
//     c dt = 1e19 bohr on.)
// 32^3 (h 0.25) and 27^3 (h 0.3), both cross pairs, 1.29e9 node pairs a step:
// 6990 us with one thread per target, scalar samples and a Kahan addition per
// term; 1870 us in this form.  One small target under a large source, 9^3 and
// 36^3: 1525 us with the sources of every target in as many parts as the
// smallest source allows, 237 with parts by target.
#include <cuda_runtime.h>

#include "rp_internal.h"

namespace rp {

namespace {

constexpr int kDirThreads = 256;
constexpr int kDirWarps = kDirThreads / 32;
constexpr int kDirOwn = 4;                  // target nodes of a thread
constexpr int kDirTargets = 32 * kDirOwn;   // target places of a block
constexpr int kDirOut = 4 * kDirTargets / kDirThreads;   // sums (target, field) a thread adds up
constexpr float kFloorShift = 8388608.0f;   // 2^23: x + 2^23 rounded down holds floor(x) in its low bits

// sum + comp += x, the rounding of the addition kept whichever is larger (a
// warp's or a part's sums are of one size, which Kahan's needs not to be)
__device__ __forceinline__ void two_add(float &sum, float &comp, float x)
{
    const float t = sum + x, b = t - sum;
    comp += (sum - (t - b)) + (x - b);
    sum = t;
}

__device__ __forceinline__ float rsqrt_ftz(float x)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// 4-byte asynchronous global -> shared copy
__device__ __forceinline__ void cp_async4(void *smem, const void *gmem)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((unsigned)__cvta_generic_to_shared(smem)), "l"(gmem)
                 : "memory");
}

__device__ __forceinline__ float2 dup(float x) { return make_float2(x, x); }
__device__ __forceinline__ float2 lo2(float4 v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ float2 hi2(float4 v) { return make_float2(v.z, v.w); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, dup(-1.0f), a); }   // one rounding

// A thread's sums: two fields a pair, lo what hi's additions rounded away.
struct DirectSums {
    float2 hi[kDirOwn][2], lo[kDirOwn][2];
};

// hi + lo += a v: the rounding of the fused product and sum goes to lo (exact
// while hi is the larger, as in Kahan's sum, and with no rounding of the
// product before it).
__device__ __forceinline__ void direct_add(float2 &hi, float2 &lo, float2 a, float2 v)
{
    const float2 t = __ffma2_rn(a, v, hi);
    lo = __fadd2_rn(lo, __ffma2_rn(a, v, sub2(hi, t)));
    hi = t;
}

// Shared memory of a block: two buffers of the sample rows (lag_lo twice,
// lag_lo + 1, ..., lag_hi three times; the repeats serve a tau that rounding
// put just outside the window) and the tile's negated source positions, with
// the threads' sums in their place at the end, and the rows' offsets into the
// raw ring.
__host__ __device__ constexpr int direct_buf_elems(int nlag, int tile) { return (nlag + 3) * (tile + 1) + tile; }
constexpr int kDirSums = 2 * kDirWarps * kDirTargets;   // float4
__host__ __device__ constexpr int direct_elems(int nlag, int tile)
{
    return 2 * direct_buf_elems(nlag, tile) > kDirSums ? 2 * direct_buf_elems(nlag, tile) : kDirSums;
}

// A thread's targets, in packed pairs, relative to the source origin
// (in units of 1 / DirectPair::scale).
struct DirectNodes {
    float2 x[2], y[2], z[2];
};

// Source jj of a staged tile onto the thread's targets, which SELF leaves out
// where they are the source (own[i] == jj).
template <bool SELF, bool SHARED>
__device__ __forceinline__ void direct_source(const float4 *__restrict__ S, const float4 *__restrict__ pos, int tile,
                                              int jj, const DirectNodes &r, float2 inv_cdt, float2 vol, unsigned base,
                                              unsigned top, const int (&own)[kDirOwn], DirectSums &sum)
{
    const float4 q = pos[jj];
    float a[kDirOwn], tau[kDirOwn];
    float2 line = dup(0.0f);   // SHARED: the four lie on one row
    if constexpr (SHARED) {
        const float dy = r.y[0].x + q.y, dz = r.z[0].x + q.z;
        line = dup(fmaf(dy, dy, dz * dz));
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const float2 dx = __fadd2_rn(r.x[h], dup(q.x));
        if constexpr (!SHARED) {
            const float2 dy = __fadd2_rn(r.y[h], dup(q.y)), dz = __fadd2_rn(r.z[h], dup(q.z));
            line = __ffma2_rn(dy, dy, __fmul2_rn(dz, dz));
        }
        const float2 R2 = __ffma2_rn(dx, dx, line);
        const float2 v = make_float2(rsqrt_ftz(R2.x), rsqrt_ftz(R2.y));
        const float2 t = __fmul2_rn(__fmul2_rn(R2, v), inv_cdt), w = __fmul2_rn(vol, v);
        a[2 * h] = w.x; a[2 * h + 1] = w.y;
        tau[2 * h] = t.x; tau[2 * h + 1] = t.y;
    }
    if constexpr (SELF) {
#pragma unroll
        for (int i = 0; i < kDirOwn; ++i)
            if (own[i] == jj) a[i] = tau[i] = 0.0f;
    }
    if constexpr (SHARED) {
        // the earliest of the four lag intervals, or the one after it; a
        // sample outside a target's own interval does not enter its sum
        // (it may not be finite)
        const float t = __fadd_rd(fminf(fminf(tau[0], tau[1]), fminf(tau[2], tau[3])), kFloorShift);
        const float m0 = t - kFloorShift, m1 = m0 + 1.0f;
        const float4 *s = S + min(__float_as_uint(t) - base, top) * (unsigned)(tile + 1) + jj;
        const float4 x0 = s[0], x1 = s[tile + 1], x2 = s[2 * (tile + 1)];
        const float2 da = sub2(lo2(x1), lo2(x0)), db = sub2(hi2(x1), hi2(x0));
        const float2 ea = sub2(lo2(x2), lo2(x1)), eb = sub2(hi2(x2), hi2(x1));
#pragma unroll
        for (int i = 0; i < kDirOwn; ++i) {
            const float2 w = dup(tau[i] - m0);
            float2 va = __ffma2_rn(w, da, lo2(x0)), vb = __ffma2_rn(w, db, hi2(x0));
            if (tau[i] >= m1) {
                const float2 e = dup(tau[i] - m1);
                va = __ffma2_rn(e, ea, lo2(x1));
                vb = __ffma2_rn(e, eb, hi2(x1));
            }
            if (SELF && own[i] == jj) va = vb = dup(0.0f);
            direct_add(sum.hi[i][0], sum.lo[i][0], dup(a[i]), va);
            direct_add(sum.hi[i][1], sum.lo[i][1], dup(a[i]), vb);
        }
    } else {
#pragma unroll
        for (int i = 0; i < kDirOwn; ++i) {
            const float t = __fadd_rd(tau[i], kFloorShift);
            const float2 w = dup(tau[i] - (t - kFloorShift));
            const float4 *s = S + min(__float_as_uint(t) - base, top) * (unsigned)(tile + 1) + jj;
            const float4 x0 = s[0], x1 = s[tile + 1];
            float2 va = __ffma2_rn(w, sub2(lo2(x1), lo2(x0)), lo2(x0));
            float2 vb = __ffma2_rn(w, sub2(hi2(x1), hi2(x0)), hi2(x0));
            if (SELF && own[i] == jj) va = vb = dup(0.0f);
            direct_add(sum.hi[i][0], sum.lo[i][0], dup(a[i]), va);
            direct_add(sum.hi[i][1], sum.lo[i][1], dup(a[i]), vb);
        }
    }
}

// Sources j .. end - 1 of a staged tile.
template <bool SELF, bool SHARED>
__device__ __forceinline__ void direct_run(const float4 *__restrict__ S, const float4 *__restrict__ pos, int tile,
                                           int j, int end, const DirectNodes &r, float2 inv_cdt, float2 vol,
                                           unsigned base, unsigned top, const int (&own)[kDirOwn], DirectSums &sum)
{
#pragma unroll 4
    for (; j < end; ++j) direct_source<SELF, SHARED>(S, pos, tile, j, r, inv_cdt, vol, base, top, own, sum);
}

// The target node at place i (0 .. 127) of block b (of its own) of target T,
// or -1: groups of four along a row, the last of a row padded (T.groups per
// row), or consecutive nodes (T.groups = 0).
__device__ __forceinline__ long long direct_node(const DirectTarget &T, int b, int i)
{
    const long long p = (long long)b * kDirTargets + i;
    if (T.groups == 0) return p < T.n ? p : -1;
    const long long g = p / kDirOwn, line = g / T.groups;
    const int x = (int)(g - line * T.groups) * kDirOwn + (i & (kDirOwn - 1));
    return x < T.nx && line < (long long)T.ny * T.nz ? line * T.nx + x : -1;
}

__device__ __forceinline__ void direct_store(const DirectTarget &T, const OutPtrs &out, int f, long long k, float v,
                                             float inv_c)
{
    float *o = f == 0 ? out.phi[T.dom] + k : out.A[T.dom] + (long long)(f - 1) * T.n + k;
    if (f > 0) v *= inv_c;
    if (T.accumulate) v += *o;
    *o = v;
}

// A block: 128 target places and one part of the target's sources (its pairs'
// one after another), or (TURN: no workspace) every part in turn, the same
// sums added in the same order.  part, of targets with more than one:
// [T.part0 + ((part * 4 + f) * 2 + {hi, lo}) * n + k].
template <bool TURN>
__global__ void __launch_bounds__(kDirThreads, 2)
    k_direct(const DirectTarget *__restrict__ tgts, int ntgt, const DirectPair *__restrict__ pairs, OutPtrs out,
             float *__restrict__ part, int tile, int max_nlag, long long step, int clamp, float inv_c)
{
    extern __shared__ float4 smem_f4[];
    float4 *S = smem_f4;   // two buffers of samples [nlag + 3][tile + 1] and positions [tile] (-x, -y, -z)
    const int rows_max = max_nlag + 3, buf_elems = direct_buf_elems(max_nlag, tile);
    float4 *sums = S;                                                                   // [warp][own][hi, lo][lane]
    long long *row = reinterpret_cast<long long *>(S + direct_elems(max_nlag, tile));   // [nlag + 3]: slot offsets
    int lo = 0, hi = ntgt;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (tgts[mid].block0 <= (int)blockIdx.x) lo = mid; else hi = mid;
    }
    const DirectTarget &T = tgts[lo];
    if (step < 0) step = *T.d_step;   // graph replay: the step from the device counter
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int share = tile / kDirWarps;   // sources of a warp in a full tile
    const int local = (int)blockIdx.x - T.block0, split0 = TURN ? 0 : local / T.blocks, b = local - split0 * T.blocks;
    float tot[kDirOut] = {}, err[kDirOut] = {};

    for (int split = split0; split < (TURN ? T.parts : split0 + 1); ++split) {
        DirectSums sum;
#pragma unroll
        for (int i = 0; i < kDirOwn; ++i) sum.hi[i][0] = sum.hi[i][1] = sum.lo[i][0] = sum.lo[i][1] = dup(0.0f);
        long long before = 0;   // sources of the pairs before
        for (int p = T.p0; p < T.p1; before += pairs[p].n_s, ++p) {
            const DirectPair &P = pairs[p];
            const long long j_first = max(T.sources * split / T.parts - before, 0LL);
            const long long j_end = min(T.sources * (split + 1) / T.parts - before, P.n_s);
            if (j_first >= j_end) continue;
            const int rows = P.nlag + 3;
            DirectNodes r;   // once in FP64
            {
                float v[3][kDirOwn];
                long long repeat = 0;
#pragma unroll
                for (int i = 0; i < kDirOwn; ++i) {   // a place without a node repeats the thread's first (or the last of all)
                    long long node = direct_node(T, b, lane * kDirOwn + i);
                    if (node < 0) node = i > 0 ? repeat : T.n - 1;
                    if (i == 0) repeat = node;
                    const long long line = node / T.nx;
                    v[0][i] = (float)((P.dx + T.ht * (int)(node - line * T.nx)) * P.scale);
                    v[1][i] = (float)((P.dy + T.ht * (int)(line % T.ny)) * P.scale);
                    v[2][i] = (float)((P.dz + T.ht * (int)(line / T.ny)) * P.scale);
                }
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    r.x[h] = make_float2(v[0][2 * h], v[0][2 * h + 1]);
                    r.y[h] = make_float2(v[1][2 * h], v[1][2 * h + 1]);
                    r.z[h] = make_float2(v[2][2 * h], v[2][2 * h + 1]);
                }
            }
            // low bits of floor(tau) + 2^23, less the lag of sample row 0
            const unsigned base = __float_as_uint(kFloorShift) + (unsigned)(P.lag_lo - 1), top = (unsigned)P.nlag;
            __syncthreads();   // the rows of the pair before, or the sums of the part before, are read
            for (int i = threadIdx.x; i < rows; i += kDirThreads) {
                long long j = step - (P.lag_lo + max(0, min(i - 1, P.nlag - 1)));
                if (clamp && j < 0) j = 0;
                row[i] = (j % P.depth) * 4 * P.n_s;
            }
            // sources j0 .. of a tile into buffer `buf`: positions, and the samples
            // by asynchronous copies (a tile ahead of the sums)
            const float hs = P.hs;
            const auto stage = [&](long long j0, int buf) {
                const int cnt = (int)min((long long)tile, j_end - j0);
                float4 *Sb = S + buf * buf_elems, *pb = Sb + rows_max * (tile + 1);
                for (int i = threadIdx.x; i < cnt; i += kDirThreads) {
                    const long long q = j0 + i;
                    int x, y, z;
                    if (q < 0x7fffffffLL) {
                        const unsigned q32 = (unsigned)q, l = q32 / (unsigned)P.nx_s;
                        x = (int)(q32 - l * (unsigned)P.nx_s);
                        z = (int)(l / (unsigned)P.ny_s);
                        y = (int)l - z * P.ny_s;
                    } else {
                        x = (int)(q % P.nx_s); y = (int)((q / P.nx_s) % P.ny_s); z = (int)(q / ((long long)P.nx_s * P.ny_s));
                    }
                    pb[i] = make_float4(-hs * (float)x, -hs * (float)y, -hs * (float)z, 0.0f);
                }
                for (int i = threadIdx.x; i < rows * tile; i += kDirThreads) {
                    const int jj = i & (tile - 1), l = i / tile;
                    if (jj >= cnt) continue;
                    const float *src = P.raw + row[l] + j0 + jj;
                    float *dst = reinterpret_cast<float *>(Sb + l * (tile + 1) + jj);
#pragma unroll
                    for (int f = 0; f < 4; ++f) cp_async4(dst + f, src + f * P.n_s);
                }
                asm volatile("cp.async.commit_group;" ::: "memory");
            };
            __syncthreads();   // the rows' offsets
            stage(j_first, 0);
            int buf = 0;
            for (long long j0 = j_first; j0 < j_end; j0 += tile, buf ^= 1) {
                const int cnt = (int)min((long long)tile, j_end - j0);
                asm volatile("cp.async.wait_all;" ::: "memory");
                __syncthreads();   // the tile is in, and the sums of the tile before are done with the other buffer
                if (j0 + tile < j_end) stage(j0 + tile, buf ^ 1);
                const float4 *Sb = S + buf * buf_elems, *pb = Sb + rows_max * (tile + 1);
                const int j = warp * share, end = min(j + share, cnt);
                const float2 ic = dup(P.inv_cdt), vol = dup(P.vol);
                int own[kDirOwn] = {-1, -1, -1, -1};   // the targets' places in the warp's share, if there (self pair)
                if (P.is_self) {
#pragma unroll
                    for (int i = 0; i < kDirOwn; ++i) {
                        const long long d = direct_node(T, b, lane * kDirOwn + i) - j0;
                        own[i] = d >= j && d < end ? (int)d : -1;
                    }
                    if (T.shared) direct_run<true, true>(Sb, pb, tile, j, end, r, ic, vol, base, top, own, sum);
                    else direct_run<true, false>(Sb, pb, tile, j, end, r, ic, vol, base, top, own, sum);
#pragma unroll
                    for (int i = 0; i < kDirOwn; ++i) {
                        if (own[i] < 0) continue;
                        const float4 x = Sb[tile + 1 + own[i]];   // weight C h^2 at lag 0 (sample row 1)
                        direct_add(sum.hi[i][0], sum.lo[i][0], dup(P.self_w), lo2(x));
                        direct_add(sum.hi[i][1], sum.lo[i][1], dup(P.self_w), hi2(x));
                    }
                } else {
                    if (T.shared) direct_run<false, true>(Sb, pb, tile, j, end, r, ic, vol, base, top, own, sum);
                    else direct_run<false, false>(Sb, pb, tile, j, end, r, ic, vol, base, top, own, sum);
                }
            }
        }
        // the eight warps' sums of each target, in warp order
        __syncthreads();
        {
            float4 *mine = sums + warp * (kDirSums / kDirWarps) + lane;
#pragma unroll
            for (int i = 0; i < kDirOwn; ++i) {
                mine[64 * i] = make_float4(sum.hi[i][0].x, sum.hi[i][0].y, sum.hi[i][1].x, sum.hi[i][1].y);
                mine[64 * i + 32] = make_float4(sum.lo[i][0].x, sum.lo[i][0].y, sum.lo[i][1].x, sum.lo[i][1].y);
            }
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < kDirOut; ++u) {
            const int c = threadIdx.x + u * kDirThreads, f = c / kDirTargets, i = c % kDirTargets;
            float s = 0.0f, e = 0.0f;
#pragma unroll
            for (int wv = 0; wv < kDirWarps; ++wv) {
                const float *v4 = reinterpret_cast<const float *>(
                    sums + wv * (kDirSums / kDirWarps) + 64 * (i % kDirOwn) + i / kDirOwn);
                two_add(s, e, v4[f]);
                e += v4[32 * 4 + f];
            }
            if constexpr (TURN) {
                two_add(tot[u], err[u], s);
                err[u] += e;
                continue;
            }
            const long long k = direct_node(T, b, i);
            if (k < 0) continue;
            if (T.parts == 1) {
                direct_store(T, out, f, k, s + e, inv_c);
                continue;
            }
            float *w = part + T.part0 + ((long long)split * 4 + f) * 2 * T.n + k;
            w[0] = s;
            w[T.n] = e;
        }
    }
    if constexpr (!TURN) return;
#pragma unroll
    for (int u = 0; u < kDirOut; ++u) {
        const int c = threadIdx.x + u * kDirThreads;
        const long long k = direct_node(T, b, c % kDirTargets);
        if (k >= 0) direct_store(T, out, c / kDirTargets, k, tot[u] + err[u], inv_c);
    }
}

// The parts of each target in order (32 B per node and part, a few percent of
// the sums' time).
__global__ void __launch_bounds__(kDirThreads)
    k_direct_sum(const DirectTarget *__restrict__ tgts, int ntgt, OutPtrs out, const float *__restrict__ part,
                 float inv_c)
{
    int lo = 0, hi = ntgt;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (tgts[mid].sum0 <= (int)blockIdx.x) lo = mid; else hi = mid;
    }
    const DirectTarget &T = tgts[lo];
    const int b = (int)blockIdx.x - T.sum0;
#pragma unroll
    for (int u = 0; u < kDirOut; ++u) {
        const int c = threadIdx.x + u * kDirThreads, f = c / kDirTargets;
        const long long k = direct_node(T, b, c % kDirTargets);
        if (k < 0) continue;
        float s = 0.0f, e = 0.0f;
        for (int i = 0; i < T.parts; ++i) {
            const float *w = part + T.part0 + ((long long)i * 4 + f) * 2 * T.n + k;
            two_add(s, e, w[0]);
            e += w[T.n];
        }
        direct_store(T, out, f, k, s + e, inv_c);
    }
}

constexpr size_t direct_smem(int nlag, int tile)
{
    return 16 * (size_t)direct_elems(nlag, tile) + 8 * (size_t)(nlag + 3);
}

// The largest tile of which three blocks would fit an SM (larger tiles stage
// more per barrier); for the longest lag windows, one that fits at all.
constexpr int direct_tile_of(int nlag)
{
    for (int tile : {128, 64})
        if (direct_smem(nlag, tile) <= 72 * 1024) return tile;
    return direct_smem(nlag, 32) <= 200 * 1024 ? 32 : 16;
}
static_assert(direct_smem(kDirMaxLags, direct_tile_of(kDirMaxLags)) <= 227 * 1024, "the longest window fits a block");

}  // namespace

// Groups of four nodes per row of nx nodes, or 0 for consecutive nodes: four
// along x share samples if light crosses them (3 h) within a step, and the
// padding of the rows stays under a third of the places.
int direct_groups(int nx, double h, double cdt, bool *shared)
{
    const int g = (nx + kDirOwn - 1) / kDirOwn;
    *shared = 3.0 * h <= 0.999 * cdt && 2 * g * kDirOwn <= 3 * nx;
    return *shared ? g : 0;
}

int direct_blocks(const int n[3], int groups)
{
    const long long places = groups ? (long long)groups * kDirOwn * n[1] * n[2] : (long long)n[0] * n[1] * n[2];
    return (int)((places + kDirTargets - 1) / kDirTargets);
}

// Parts of a target's sources: enough blocks for eight per SM of a 152-SM
// device, so that blocks of unequal length leave no long tail, each part with
// at least 512 sources.  From the target and its own sources alone: the order
// of its sum, so its bits, are the same whatever else a context holds, on any
// device, and with or without room for the workspace.
int direct_parts(int blocks, long long sources)
{
    const long long want = (8 * 152 + blocks - 1) / (blocks > 0 ? blocks : 1), most = sources / 512;
    const long long s = want < most ? want : most;
    return (int)(s < 1 ? 1 : s > 64 ? 64 : s);
}

cudaError_t open_direct_smem_limit(int max_optin)
{
    cudaError_t e = cudaFuncSetAttribute(k_direct<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, max_optin);
    return e ? e : cudaFuncSetAttribute(k_direct<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, max_optin);
}

cudaError_t launch_direct(const DirectTarget *d_tgts, int ntgt, const DirectPair *d_pairs, const OutPtrs &out,
                          float *part, bool turn, int nblocks, int sum_blocks, int max_nlag, long long step,
                          int clamp, float inv_c, cudaStream_t s)
{
    if (nblocks <= 0) return cudaSuccess;
    const int tile = direct_tile_of(max_nlag);
    const auto go = [&](auto kern) {
        kern<<<nblocks, kDirThreads, direct_smem(max_nlag, tile), s>>>(d_tgts, ntgt, d_pairs, out, part, tile, max_nlag,
                                                                       step, clamp, inv_c);
    };
    if (turn) go(k_direct<true>);
    else go(k_direct<false>);
    cudaError_t e = cudaGetLastError();
    if (e || sum_blocks <= 0) return e;
    k_direct_sum<<<sum_blocks, kDirThreads, 0, s>>>(d_tgts, ntgt, out, part, inv_c);
    return cudaGetLastError();
}

}  // namespace rp
