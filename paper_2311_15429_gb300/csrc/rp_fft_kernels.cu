// FFT-path kernels: the zero-padded (Hockney) convolution of each target with
// the lag kernels G_m of Eq. 11 of every FFT-path source, itself included,
// summed in the spectral domain over (source, lag) as in Eq. 12.
//
//   push   : k_ring_push   raw (rho, J) slice -> raw history ring (direct pairs only)
//            k_fwd_plane   R2C along x + FFT along y of one z-plane of a source
//            k_fwd_column  FFT along z of a (kx, 16 ky) column block, 4 fields -> spectral ring
//   eval   : k_mac_inv_col sum over (source, lag) of G_m * S(l - m) for a column
//                          block, then inverse FFT along z (kept z < nz of the target)
//            k_inv_plane   inverse FFT along y then C2R along x of one z-plane,
//                          crop to the target grid, scale (1/c for A), write phi / A
//
// Layouts: a spectrum is [field][kx][kz][ky] with ky fastest and kx <= mx/2;
// the scratch after a plane pass is [field][kx][z][ky]; every field array of
// a domain is [z][y][x].
//
// The column pass runs the two-stage shared-memory tile transform of
// rp_fft.cuh for 64, 96, 128 and 192 points along z (k_fwd_column16) and the
// lane-shuffle line transform otherwise; the plane passes here (lane-shuffle
// lines) serve a cross-section of 48, with M = 0 any supported shape read at
// run time, and the smallest forward launches at 32; the other square ones are
// in rp_plane.cu.  The MAC here serves
// shapes with no column class.
#include <cuda_runtime.h>

#include <algorithm>

#include "rp_fft.cuh"
#include "rp_internal.h"

namespace rp {

namespace {

__host__ __device__ constexpr int radix_R(int M) { return lane_radix(M); }
__host__ __device__ constexpr int radix_L(int M) { return M / radix_R(M); }
__host__ __device__ constexpr int ilog2c(int x) { return x <= 1 ? 0 : 1 + ilog2c(x / 2); }

template <int M>
__device__ __forceinline__ Axis axis_of(const Axis &rt)
{
    if constexpr (M == 0) return rt;
    else return Axis{M, radix_R(M), radix_L(M), ilog2c(radix_L(M))};
}

template <int M, class F>
__device__ __forceinline__ void run_radix(int R_rt, F &f)
{
    if constexpr (M == 0) dispatch_radix(R_rt, f);
    else f.template run<radix_R(M)>();
}

__host__ __device__ constexpr int lane_class(int M) { return M > 0 ? M : 32; }

// One line FFT: the compiled-size transform with precomputed lane twiddles
// for M > 0, else the table-driven runtime transform.
template <int M, bool INV, int RR>
__device__ __forceinline__ void do_line(float2 (&v)[RR], int g, const Axis &a, const float2 *tw,
                                        const LaneTw<lane_class(M), INV> *lt)
{
    if constexpr (M > 0) line_fft_c<M, INV>(v, *lt);
    else line_fft<RR, INV>(v, g, a, tw);
}

// index r in [lo, hi) of the last record whose first block (field) is <= b
template <class T>
__device__ __forceinline__ int owner_of(const T *arr, int lo, int hi, int b, int T::*field)
{
    while (hi - lo > 1) {
        int mid = (lo + hi) >> 1;
        if (arr[mid].*field <= b) lo = mid; else hi = mid;
    }
    return lo;
}

__device__ __forceinline__ float4 ldg4(const float2 *p) { return __ldg(reinterpret_cast<const float4 *>(p)); }

// 16-byte asynchronous global -> shared copy (both addresses 16-byte aligned)
__device__ __forceinline__ void cp_async16(void *smem, const void *gmem)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(smem)),
                 "l"(gmem)
                 : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// ---------------------------------------------------------------- raw ring push

struct PushPrefix {
    int block0[kMaxDomains + 1];
};

__global__ void __launch_bounds__(kThreads) k_ring_push(const RawRing *__restrict__ rings, IoPtrs in,
                                                          PushPrefix pre, int d0, int d1, long long step)
{
    int b = blockIdx.x;
    int lo = d0, hi = d1;
    while (hi - lo > 1) {
        int mid = (lo + hi) >> 1;
        if (pre.block0[mid] <= b) lo = mid; else hi = mid;
    }
    const int d = lo;
    const RawRing rr = rings[d];
    if (rr.ring == nullptr) return;
    if (step < 0) step = *rr.d_step;   // graph replay: the step from the device counter
    const long long n = rr.n;
    float *dst = rr.ring + (long long)(step % rr.depth) * 4 * n;
    const long long chunk = (long long)kThreads * 8;
    const long long base = (long long)(b - pre.block0[d]) * chunk;
    for (long long i = base + threadIdx.x; i < base + chunk && i < 4 * n; i += kThreads) {
        const float *src = i < n ? in.rho[d] + i : in.J[d] + (i - n);
        dst[i] = *src;
    }
}

// ---------------------------------------------------------------- forward plane pass

template <int M>
struct FwdPlaneX {
    const LaneTw<lane_class(M), false> *lt;
    Axis a;
    int nx, ny, kx;
    const float *plane;
    float2 *Q;      // [ny][qs]
    int qs;
    float2 *W;      // per-group scratch, M each
    const float2 *tw;
    int lane, warp, nwarps;

    template <int RX>
    __device__ __forceinline__ void run()
    {
        const int G = 32 >> a.logL;
        const int grp = lane >> a.logL, g = lane & (a.L - 1);
        const int pairs = (ny + 1) >> 1;
        const int per_iter = nwarps * G;
        float2 *Wg = W + (warp * G + grp) * a.M;
        for (int base = 0; base < pairs; base += per_iter) {
            const int p = base + warp * G + grp;
            const bool valid = p < pairs;
            const int ya = 2 * p, yb = 2 * p + 1;
            const bool vb = valid && yb < ny;
            float2 v[RX];
#pragma unroll
            for (int n = 0; n < RX; ++n) {
                const int xi = n * a.L + g;
                const bool in_x = xi < nx;
                v[n].x = (valid && in_x) ? plane[ya * nx + xi] : 0.0f;
                v[n].y = (vb && in_x) ? plane[yb * nx + xi] : 0.0f;
            }
            do_line<M, false>(v, g, a, tw, lt);
            const int kb = bitrev_lanes(g, a.logL) * RX;
#pragma unroll
            for (int k1 = 0; k1 < RX; ++k1) Wg[k1 + kb] = v[k1];
            __syncwarp();
            // two real rows from one complex transform:
            //   A[k] = (Z[k] + conj Z[M-k]) / 2,  B[k] = (Z[k] - conj Z[M-k]) / (2i)
            for (int k = g; k < kx; k += a.L) {
                const float2 zk = Wg[k];
                const float2 zc = cconj(Wg[k == 0 ? 0 : a.M - k]);
                const float2 A = cscale(cadd(zk, zc), 0.5f);
                const float2 D = csub(zk, zc);
                const float2 B = make_float2(0.5f * D.y, -0.5f * D.x);
                if (valid) Q[ya * qs + k] = A;
                if (vb) Q[yb * qs + k] = B;
            }
            __syncwarp();
        }
    }
};

template <int M>
struct FwdPlaneY {
    const LaneTw<lane_class(M), false> *lt;
    Axis a;
    int ny, kx, nz;
    const float2 *Q;
    int qs;
    float2 *out;    // row kx at out + kx*nz*my
    const float2 *tw;
    int lane, warp, nwarps;

    template <int RY>
    __device__ __forceinline__ void run()
    {
        const int G = 32 >> a.logL;
        const int grp = lane >> a.logL, g = lane & (a.L - 1);
        const int per_iter = nwarps * G;
        const long long row_stride = (long long)nz * a.M;
        for (int base = 0; base < kx; base += per_iter) {
            const int kxi = base + warp * G + grp;
            const bool valid = kxi < kx;
            float2 v[RY];
#pragma unroll
            for (int n = 0; n < RY; ++n) {
                const int yi = n * a.L + g;
                v[n] = (valid && yi < ny) ? Q[yi * qs + kxi] : make_float2(0.0f, 0.0f);
            }
            do_line<M, false>(v, g, a, tw, lt);
            const int kb = bitrev_lanes(g, a.logL) * RY;
            if (valid) {
                float2 *row = out + kxi * row_stride;
#pragma unroll
                for (int k1 = 0; k1 < RY; ++k1) row[k1 + kb] = v[k1];
            }
        }
    }
};

template <int M>
__global__ void __launch_bounds__(kPlaneThreads) k_fwd_plane(const FwdRing *__restrict__ rings, IoPtrs in,
                                                          int r0, int r1, int block_lo, int far_slot)
{
    extern __shared__ float4 smem_f4[];
    float2 *sm = reinterpret_cast<float2 *>(smem_f4);
    const int b = blockIdx.x + block_lo;
    const int r = owner_of(rings, r0, r1, b, &FwdRing::plane0);
    const FwdRing &R = rings[r];
    const Axis ax = axis_of<M>(R.ax), ay = axis_of<M>(R.ay);
    const int nx = R.nx, ny = R.ny, nz = R.nz;
    const int kx = ax.M / 2 + 1;
    const int local = b - R.plane0;
    const int f = local / nz, z = local % nz;
    const long long N = (long long)nx * ny * nz;

    float2 *twx = sm;
    float2 *twy = twx + ax.M;
    const int qs = kx | 1;
    float2 *Q = twy + ay.M;
    float2 *W = Q + ny * qs;
    load_twiddles(twx, R.tw_x, ax.M);
    load_twiddles(twy, R.tw_y, ay.M);
    pdl_trigger();
    pdl_wait();   // the input slice may come from the previous kernel; t1 was read by it
    __syncthreads();

    const float *src = f == 0 ? in.rho[R.src] : in.J[R.src] + (long long)(f - 1) * N;
    const float *plane = src + (long long)z * nx * ny;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;

    LaneTw<lane_class(M), false> lt;
    if constexpr (M > 0) lt.init(twx, lane & (ax.L - 1));
    FwdPlaneX<M> px{&lt, ax, nx, ny, kx, plane, Q, qs, W, twx, lane, warp, nwarps};
    run_radix<M>(ax.R, px);
    __syncthreads();
    float2 *out = R.t1 + ((long long)f * kx * nz + z) * ay.M;
    FwdPlaneY<M> py{&lt, ay, ny, kx, nz, Q, qs, out, twy, lane, warp, nwarps};
    run_radix<M>(ay.R, py);
    if (R.far_x) {
        // far path: this plane as bf16 hi/lo into row (slot, field) of the batch matrix
        __nv_bfloat16 *row = R.far_x + ((long long)far_slot * 4 + f) * 2 * R.far_ks + (long long)z * nx * ny;
        for (int i = threadIdx.x; i < nx * ny; i += blockDim.x) {
            const float v = __ldg(plane + i);
            const __nv_bfloat16 hi = __float2bfloat16(v);
            row[i] = hi;
            row[R.far_ks + i] = __float2bfloat16(v - __bfloat162float(hi));
        }
    }
}

// ---------------------------------------------------------------- column passes

// Line FFTs down the columns of a shared-memory tile [field][M][kTileYPad].
template <int M, bool INV>
struct ColumnFFT {
    const LaneTw<lane_class(M), INV> *lt;
    Axis a;
    float2 *V;
    int field_stride;  // float2 between fields in V
    int ncols;         // columns per field
    int nfields;
    int keep;          // outputs kept: index < keep
    const float2 *tw;
    int lane, warp, nwarps;

    template <int RR>
    __device__ __forceinline__ void run()
    {
        const int G = 32 >> a.logL;
        const int grp = lane >> a.logL, g = lane & (a.L - 1);
        const int lines = ncols * nfields;
        const int per_iter = nwarps * G;
        for (int base = 0; base < lines; base += per_iter) {
            const int line = base + warp * G + grp;
            const bool valid = line < lines;
            const int fld = valid ? line / ncols : 0, c = valid ? line % ncols : 0;
            float2 *col = V + fld * field_stride + c;
            float2 v[RR];
#pragma unroll
            for (int n = 0; n < RR; ++n) v[n] = col[(n * a.L + g) * kTileYPad];
            do_line<M, INV>(v, g, a, tw, lt);
            __syncwarp();
            const int kb = bitrev_lanes(g, a.logL) * RR;
            if (valid) {
#pragma unroll
                for (int k1 = 0; k1 < RR; ++k1)
                    if (k1 + kb < keep) col[(k1 + kb) * kTileYPad] = v[k1];
            }
            __syncwarp();
        }
    }
};

// Forward FFT along z of the four fields of one (kx, 16-ky) column block.
// CUBE: the cross-section is the padded length along z squared, its extents
// constants.  A launch of few blocks is all latency: with extents read at run
// time for every shape a step of one 24^3 grid took 20.3 us, with these 19.2
// (two 22^3 23.7 and 22.6, two 16^3 19.4 and 18.0).
template <int M, bool CUBE>
__global__ void __launch_bounds__(kColumnThreads) k_fwd_column(const FwdRing *__restrict__ rings, int r0, int r1,
                                                           int block_lo, long long step)
{
    extern __shared__ float4 smem_f4[];
    float2 *sm = reinterpret_cast<float2 *>(smem_f4);
    const int b = blockIdx.x + block_lo;
    const int r = owner_of(rings, r0, r1, b, &FwdRing::tile0);
    const FwdRing &R = rings[r];
    const Axis az = axis_of<M>(R.az);
    const int my = CUBE ? M : R.ay.M, mz = az.M, nz = R.nz;   // M > 0: mz = M, my a multiple of 16
    const int kx = CUBE ? M / 2 + 1 : R.kx;
    const int ntile = (my + kTileY - 1) / kTileY;
    const int local = b - R.tile0;
    const int kxi = local / ntile, ky0 = (local % ntile) * kTileY;
    const int ncols = min(kTileY, my - ky0);
    const int fs = mz * kTileYPad;

    float2 *tw = sm;
    float2 *V = tw + mz;
    load_twiddles(tw, R.tw_z, mz);
    pdl_trigger();
    pdl_wait();   // t1 is written by the plane pass
    if (step < 0) step = *R.d_step;   // graph replay: the step from the device counter
    const long long t1_field = (long long)kx * nz * my;
    const float2 *src = R.t1 + (long long)kxi * nz * my + ky0;
    if constexpr (M > 0) {
        // 16-byte loads of column pairs; rows z >= nz are the zero padding
        for (int i = threadIdx.x; i < 4 * mz * (kTileY / 2); i += blockDim.x) {
            const int f = i / (mz * (kTileY / 2)), rem = i % (mz * (kTileY / 2));
            const int zi = rem / (kTileY / 2), p = rem % (kTileY / 2);
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (zi < nz) v = ldg4(src + f * t1_field + (long long)zi * my + 2 * p);
            float2 *d = V + f * fs + zi * kTileYPad + 2 * p;
            d[0] = make_float2(v.x, v.y);
            d[1] = make_float2(v.z, v.w);
        }
    } else {
        for (int i = threadIdx.x; i < 4 * mz * kTileY; i += blockDim.x) {
            const int f = i / (mz * kTileY), rem = i % (mz * kTileY);
            const int zi = rem / kTileY, c = rem % kTileY;
            float2 v = make_float2(0.0f, 0.0f);
            if (zi < nz && c < ncols) v = src[f * t1_field + (long long)zi * my + c];
            V[f * fs + zi * kTileYPad + c] = v;
        }
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    LaneTw<lane_class(M), false> lt;
    if constexpr (M > 0) lt.init(tw, lane & (az.L - 1));
    ColumnFFT<M, false> cf{&lt, az, V, fs, ncols, 4, mz, tw, lane, warp, nwarps};
    run_radix<M>(az.R, cf);
    __syncthreads();
    // the tile's four field tiles sit next to each other in the slot
    const long long ring_field = (long long)mz * kTileY;
    float2 *dst = R.ring + (long long)((step - R.lag_off) % R.depth) * R.slot_elems +
                  (long long)(kxi * ntile + ky0 / kTileY) * 4 * ring_field;
    if constexpr (M > 0) {
        for (int i = threadIdx.x; i < 4 * mz * (kTileY / 2); i += blockDim.x) {
            const int f = i / (mz * (kTileY / 2)), rem = i % (mz * (kTileY / 2));
            const int kz = rem / (kTileY / 2), p = rem % (kTileY / 2);
            const float2 *s = V + f * fs + kz * kTileYPad + 2 * p;
            *reinterpret_cast<float4 *>(dst + f * ring_field + kz * kTileY + 2 * p) =
                make_float4(s[0].x, s[0].y, s[1].x, s[1].y);
        }
    } else {
        for (int i = threadIdx.x; i < 4 * mz * kTileY; i += blockDim.x) {
            const int f = i / (mz * kTileY), rem = i % (mz * kTileY);
            const int kz = rem / kTileY, c = rem % kTileY;
            dst[f * ring_field + kz * kTileY + c] = c < ncols ? V[f * fs + kz * kTileYPad + c] : make_float2(0.f, 0.f);
        }
    }
}

// The forward column pass for M = 16 B, B even (M = 64, 96, 128, 192): the
// tile [field][z][16] dense in shared memory, one warp per field with the
// two-stage tile transform (rows z >= nz are the zero padding: neither loaded
// nor read; when nz <= M/2 the first layer skips the zero half), then each
// spectral row copied from its tile row to the ring slot.
constexpr int kColumn16Threads = 256;   // two warps per field

__host__ __device__ constexpr bool tile16_class(int M) { return M == 64 || M == 96 || M == 128 || M == 192; }

template <int M, bool CUBE>
__global__ void __launch_bounds__(kColumn16Threads) k_fwd_column16(const FwdRing *__restrict__ rings, int r0, int r1,
                                                                    int block_lo, long long step)
{
    constexpr int B = M / 16;
    static_assert(tile16_class(M), "k_fwd_column16: M = 16 B, B even");
    extern __shared__ float4 smem_f4[];
    float2 *sm = reinterpret_cast<float2 *>(smem_f4);
    const int b = blockIdx.x + block_lo;
    const int r = owner_of(rings, r0, r1, b, &FwdRing::tile0);
    const FwdRing &R = rings[r];
    const int nz = R.nz, my = CUBE ? M : R.ay.M, kx = CUBE ? M / 2 + 1 : R.kx, ntile = my / kTileY;
    const int local = b - R.tile0;
    const int kxi = local / ntile, kyt = local % ntile;
    float2 *tw = sm;
    float2 *V = tw + M;   // [field][M rows][16]
    load_twiddles(tw, R.tw_z, M);
    pdl_trigger();
    pdl_wait();   // t1 is written by the plane pass
    if (step < 0) step = *R.d_step;   // graph replay: the step from the device counter
    __syncthreads();   // the twiddles
    // the warp pair 2f, 2f + 1 owns field f from copy-in to store (named
    // barrier 1 + f): no block barrier, so the fields' copies, transforms and
    // stores interleave
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, f = warp >> 1, half = warp & 1;
    const int t64 = threadIdx.x & 63, p = t64 & 7, zr = t64 >> 3;   // column pair p, rows zr + 8 j
    float2 *Vf = V + f * M * kTileY;
    {
        const long long t1_field = (long long)kx * nz * my;
        const float2 *src = R.t1 + f * t1_field + (long long)kxi * nz * my + kyt * kTileY + 2 * p;
        for (int z = zr; z < nz; z += 8) cp_async16(Vf + z * kTileY + 2 * p, src + (long long)z * my);
        cp_async_wait_all();
    }
    asm volatile("bar.sync %0, 64;" ::"r"(1 + f) : "memory");
    // a source as large as the target's padded half (the usual case) skips the
    // zero half in the first layer; a larger source of a cross pair does not
    if (nz <= M / 2) tile_fft16_pair<B, false, true>(Vf, tw, nz, lane, half, 1 + f);
    else tile_fft16_pair<B, false, false>(Vf, tw, nz, lane, half, 1 + f);
    float2 *dst = R.ring + (long long)((step - R.lag_off) % R.depth) * R.slot_elems +
                  (long long)(kxi * ntile + kyt) * 4 * M * kTileY + f * M * kTileY;
#pragma unroll 4
    for (int kz = zr; kz < M; kz += 8)
        *reinterpret_cast<float4 *>(dst + kz * kTileY + 2 * p) =
            *reinterpret_cast<const float4 *>(Vf + tile_row<B>(kz) * kTileY + 2 * p);
}

// Kahan-compensated addition (the total is s - c; see k_mac_tma).
__device__ __forceinline__ void kahan_add(float &s, float &c, float x)
{
    const float y = x - c;
    const float t = s + y;
    c = (t - s) - y;
    s = t;
}

// Spectral multiply-accumulate over the target's (source, lag) entries for
// one (kx, 16-ky) column block and all four fields, any shape (the shapes with
// no column class; the others run k_mac_tma), then the inverse FFT
// along z of the 64 columns; rows z < nz of the target go to T2.  COMP: the
// sum over entries is Kahan-compensated per spectral coefficient.
template <bool COMP>
__global__ void __launch_bounds__(kThreads) k_mac_inv_column(const InvTarget *__restrict__ tgts, int t0, int t1,
                                                               int block_lo, const MacEntry *__restrict__ entries,
                                                               long long step, int clamp)
{
    extern __shared__ float4 smem_f4[];
    float2 *sm = reinterpret_cast<float2 *>(smem_f4);
    const int b = blockIdx.x + block_lo;
    const int t = owner_of(tgts, t0, t1, b, &InvTarget::tile0);
    const InvTarget &T = tgts[t];
    const Axis az = T.az;
    const int my = T.ay.M, mz = az.M;
    const int kx = T.kx;
    const int ntile = (my + kTileY - 1) / kTileY;
    const int local = b - T.tile0;
    const int kxi = local / ntile, ky0 = (local % ntile) * kTileY;
    const int ncols = min(kTileY, my - ky0);
    const long long col0 = (long long)(kxi * ntile + ky0 / kTileY) * mz * kTileY;   // tile in a kernel spectrum
    const long long fstride = (long long)mz * kTileY;                             // field tile in a ring slot
    const int fs = mz * kTileYPad;

    float2 *tw = sm;
    float2 *acc = tw + mz;                 // [4][mz][kTileYPad]
    load_twiddles(tw, T.tw_z, mz);
    pdl_trigger();
    pdl_wait();   // the newest ring slot is written by the column pass
    if (step < 0) step = *T.d_step;   // graph replay: the step from the device counter

    for (int i = threadIdx.x; i < 4 * fs; i += blockDim.x) acc[i] = make_float2(0.0f, 0.0f);
    __syncthreads();
    // Each thread owns the (kz, c) cells i = threadIdx.x + k*blockDim.x and
    // sums every entry of one cell in registers (entries in order, the
    // warp's lanes reading consecutive cells of an entry), then stores it.
    for (int i = threadIdx.x; i < mz * kTileY; i += blockDim.x) {
        const int kz = i / kTileY, c = i % kTileY;
        if (c >= ncols) continue;
        const long long off = kz * kTileY + c;
        float2 v[4], cv[4];
#pragma unroll
        for (int f = 0; f < 4; ++f) v[f] = cv[f] = make_float2(0.0f, 0.0f);
        for (int e = T.e0; e < T.e1; ++e) {
            const MacEntry E = entries[e];
            long long j = step - E.lag;
            if (clamp && j < 0) j = 0;
            const float2 *S = E.ring + (j % E.depth) * E.slot_elems + 4 * col0;
            const float2 g = E.is_real ? make_float2(__ldg(static_cast<const float *>(E.g) + col0 + off), 0.0f)
                                       : __ldg(static_cast<const float2 *>(E.g) + col0 + off);
#pragma unroll
            for (int f = 0; f < 4; ++f) {
                const float2 t = cmul(g, __ldg(S + f * fstride + off));
                if constexpr (COMP) {
                    kahan_add(v[f].x, cv[f].x, t.x);
                    kahan_add(v[f].y, cv[f].y, t.y);
                } else {
                    v[f] = cadd(v[f], t);
                }
            }
        }
        const int a_ = kz * kTileYPad + c;
#pragma unroll
        for (int f = 0; f < 4; ++f) acc[f * fs + a_] = COMP ? make_float2(v[f].x - cv[f].x, v[f].y - cv[f].y) : v[f];
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    ColumnFFT<0, true> cf{nullptr, az, acc, fs, ncols, 4, T.nz, tw, lane, warp, nwarps};
    run_radix<0>(az.R, cf);
    __syncthreads();
    const int nz = T.nz;
    const long long t2_field = (long long)kx * nz * my;
    float2 *dst = T.t2 + (long long)kxi * nz * my + ky0;
    for (int i = threadIdx.x; i < 4 * nz * kTileY; i += blockDim.x) {
        const int f = i / (nz * kTileY), rem = i % (nz * kTileY);
        const int zi = rem / kTileY, c = rem % kTileY;
        if (c < ncols) dst[f * t2_field + (long long)zi * my + c] = acc[f * fs + zi * kTileYPad + c];
    }
}

// ---------------------------------------------------------------- inverse plane pass

template <int M>
struct InvPlaneY {
    const LaneTw<lane_class(M), true> *lt;
    Axis a;
    int kx, ny;
    float2 *P;
    int ps;
    const float2 *tw;
    int lane, warp, nwarps;

    template <int RY>
    __device__ __forceinline__ void run()
    {
        const int G = 32 >> a.logL;
        const int grp = lane >> a.logL, g = lane & (a.L - 1);
        const int per_iter = nwarps * G;
        for (int base = 0; base < kx; base += per_iter) {
            const int kxi = base + warp * G + grp;
            const bool valid = kxi < kx;
            float2 *row = P + (valid ? kxi : 0) * ps;
            float2 v[RY];
#pragma unroll
            for (int n = 0; n < RY; ++n) v[n] = row[n * a.L + g];
            do_line<M, true>(v, g, a, tw, lt);
            __syncwarp();
            const int kb = bitrev_lanes(g, a.logL) * RY;
            if (valid) {
#pragma unroll
                for (int k1 = 0; k1 < RY; ++k1)
                    if (k1 + kb < ny) row[k1 + kb] = v[k1];
            }
            __syncwarp();
        }
    }
};

template <int M>
struct InvPlaneX {
    const LaneTw<lane_class(M), true> *lt;
    Axis a;
    int nx, ny;
    const float2 *P;
    int ps;
    float *O;       // [ny][nx]
    float scale;
    const float2 *tw;
    int lane, warp, nwarps;

    template <int RX>
    __device__ __forceinline__ void run()
    {
        const int G = 32 >> a.logL;
        const int grp = lane >> a.logL, g = lane & (a.L - 1);
        const int pairs = (ny + 1) >> 1;
        const int half = a.M >> 1;
        const int per_iter = nwarps * G;
        for (int base = 0; base < pairs; base += per_iter) {
            const int p = base + warp * G + grp;
            const bool valid = p < pairs;
            const int ya = valid ? 2 * p : 0, yb = ya + 1;
            const bool vb = valid && yb < ny;
            float2 v[RX];
#pragma unroll
            for (int n = 0; n < RX; ++n) {
                const int k = n * a.L + g;
                const bool lower = k <= half;
                const int kk = lower ? k : a.M - k;
                float2 A = P[kk * ps + ya];
                float2 B = vb ? P[kk * ps + yb] : make_float2(0.0f, 0.0f);
                if (!lower) { A = cconj(A); B = cconj(B); }
                if (k == 0 || k == half) { A.y = 0.0f; B.y = 0.0f; }
                v[n] = make_float2(A.x - B.y, A.y + B.x);   // A + iB
            }
            do_line<M, true>(v, g, a, tw, lt);
            const int kb = bitrev_lanes(g, a.logL) * RX;
            if (valid) {
#pragma unroll
                for (int k1 = 0; k1 < RX; ++k1) {
                    const int x = k1 + kb;
                    if (x < nx) {
                        O[ya * nx + x] = scale * v[k1].x;
                        if (vb) O[yb * nx + x] = scale * v[k1].y;
                    }
                }
            }
        }
    }
};

template <int M>
__global__ void __launch_bounds__(kPlaneThreads) k_inv_plane(const InvTarget *__restrict__ tgts, int t0, int t1,
                                                          int block_lo, OutPtrs out, float inv_c, long long step)
{
    extern __shared__ float4 smem_f4[];
    float2 *sm = reinterpret_cast<float2 *>(smem_f4);
    const int b = blockIdx.x + block_lo;
    const int t = owner_of(tgts, t0, t1, b, &InvTarget::plane0);
    const InvTarget &T = tgts[t];
    const Axis ax = axis_of<M>(T.ax), ay = axis_of<M>(T.ay);
    const int nx = T.nx, ny = T.ny, nz = T.nz;
    const int kx = ax.M / 2 + 1, my = ay.M;
    const int local = b - T.plane0;
    const int f = local / nz, z = local % nz;
    const int ps = my | 1;

    float2 *twx = sm;
    float2 *twy = twx + ax.M;
    float2 *P = twy + my;                                   // [kx][ps]
    float *O = reinterpret_cast<float *>(P + kx * ps);      // [ny][nx]
    load_twiddles(twx, T.tw_x, ax.M);
    load_twiddles(twy, T.tw_y, my);
    // far pairs: the target's Lagrange weights (constant) into shared memory
    // now, so that the interpolation at the end reads no global table
    const FarTarget *Fp = T.far;
    int fpx = 0, fpy = 0, fpz = 0, fr = 0, fdepth = 1;
    const float *fcring = nullptr;
    float *cz = O + nx * ny;                                // [py][px]
    float *ux = cz + kMaxFarPts * kMaxFarPts;               // [py][nx]
    float *sLx = ux + kMaxFarPts * nx;                      // [nx][px]
    float *sLy = sLx + kMaxFarPts * nx;                     // [ny][py]
    float *sLz = sLy + kMaxFarPts * ny;                     // [pz], row z
    float *sc = sLz + kMaxFarPts;                           // [r]: this step's coefficients of field f
    if (Fp) {
        fpx = Fp->px; fpy = Fp->py; fpz = Fp->pz; fr = Fp->r; fdepth = Fp->depth; fcring = Fp->cring;
        for (int i = threadIdx.x; i < nx * fpx; i += blockDim.x) sLx[i] = __ldg(Fp->Lx + i);
        for (int i = threadIdx.x; i < ny * fpy; i += blockDim.x) sLy[i] = __ldg(Fp->Ly + i);
        for (int i = threadIdx.x; i < fpz; i += blockDim.x) sLz[i] = __ldg(Fp->Lz + z * fpz + i);
    }
    pdl_trigger();
    pdl_wait();   // T2 is written by the MAC, the coefficient ring by the far scatter or the learned field
    if (step < 0) step = *T.d_step;   // graph replay: the step from the device counter
    const float2 *src = T.t2 + ((long long)f * kx * nz + z) * my;
    const long long row_stride = (long long)nz * my;
    if constexpr (M > 0) {
        for (int i = threadIdx.x; i < kx * (M / 2); i += blockDim.x) {
            const int kxi = i / (M / 2), q = i % (M / 2);
            const float4 v = ldg4(src + kxi * row_stride + 2 * q);
            P[kxi * ps + 2 * q] = make_float2(v.x, v.y);
            P[kxi * ps + 2 * q + 1] = make_float2(v.z, v.w);
        }
    } else {
        for (int i = threadIdx.x; i < kx * my; i += blockDim.x) {
            const int kxi = i / my, ky = i % my;
            P[kxi * ps + ky] = src[kxi * row_stride + ky];
        }
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    LaneTw<lane_class(M), true> lt;
    if constexpr (M > 0) lt.init(twx, lane & (ax.L - 1));
    InvPlaneY<M> py{&lt, ay, kx, ny, P, ps, twy, lane, warp, nwarps};
    run_radix<M>(ay.R, py);
    __syncthreads();
    InvPlaneX<M> px{&lt, ax, nx, ny, P, ps, O, f == 0 ? 1.0f : inv_c, twx, lane, warp, nwarps};
    run_radix<M>(ax.R, px);
    __syncthreads();
    const long long N = (long long)nx * ny * nz;
    float *dst = (f == 0 ? out.phi[T.dom] : out.A[T.dom] + (long long)(f - 1) * N) + (long long)z * nx * ny;
    if (!Fp) {
        for (int i = threadIdx.x; i < nx * ny; i += blockDim.x) dst[i] = O[i];
        return;
    }
    // far pairs: tensor-product Lagrange interpolation of this step's node
    // coefficients (field f), contracted over z first
    const float *c = fcring + (step % fdepth) * (fr * 4);
    for (int i = threadIdx.x; i < fr; i += blockDim.x) sc[i] = c[i * 4 + f];
    __syncthreads();
    const int pxy = fpx * fpy;
    for (int i = threadIdx.x; i < pxy; i += blockDim.x) {
        float s = 0.0f;
        for (int cc = 0; cc < fpz; ++cc) s = fmaf(sLz[cc], sc[cc * pxy + i], s);
        cz[i] = s;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < fpy * nx; i += blockDim.x) {
        const int bb = i / nx, x = i % nx;
        float u = 0.0f;
        for (int aa = 0; aa < fpx; ++aa) u = fmaf(sLx[x * fpx + aa], cz[bb * fpx + aa], u);
        ux[i] = u;
    }
    __syncthreads();
    const float scale = f == 0 ? 1.0f : inv_c;
    for (int i = threadIdx.x; i < nx * ny; i += blockDim.x) {
        const int x = i % nx, y = i / nx;
        float v = 0.0f;
        for (int bb = 0; bb < fpy; ++bb) v = fmaf(sLy[y * fpy + bb], ux[bb * nx + x], v);
        dst[i] = fmaf(scale, v, O[i]);
    }
}

// lengths compiled here: of the plane passes (the others are in rp_plane.cu)
// and of the column pass
#define RP_PLANE_CLASSES(X) X(0) X(48)
#define RP_COLUMN_CLASSES(X) X(0) X(32) X(48) X(64) X(96) X(128) X(192)

}  // namespace

// ---------------------------------------------------------------- host side

int size_class(const Axis &ax, const Axis &ay, const Axis &az)
{
    const auto compiled = [](int M) {
        switch (M) {
        case 32: case 48: case 64: case 96: case 128: case 192: return M;
        default: return 0;
        }
    };
    const int plane = ax.M == ay.M ? compiled(ax.M) : 0, column = ay.M % kTileY == 0 ? compiled(az.M) : 0;
    return column << 8 | plane;
}

size_t smem_fwd_plane(int cls, int ny, const Axis &ax)
{
    const size_t line = plane_line_class(cls) ? smem_fwd_plane_line(cls, ny) : 0;
    if (line && cls != 32) return line;   // 32: either form
    const int kx = ax.M / 2 + 1;
    const int qs = kx | 1;
    // twiddles (x and y, bounded by kMaxFFT each) + Q + per-group scratch
    return std::max(line, sizeof(float2) * (2 * kMaxFFT + (size_t)ny * qs + (size_t)(kPlaneThreads / 32) * 32 * ax.R));
}

size_t smem_fwd_column(const Axis &az) { return sizeof(float2) * ((size_t)az.M + 4 * (size_t)az.M * kTileYPad); }

static size_t smem_fwd_column16(int M) { return sizeof(float2) * ((size_t)M + 4 * (size_t)M * kTileY); }

size_t smem_mac_inv_column(const Axis &az)
{
    return sizeof(float2) * ((size_t)az.M + 4 * (size_t)az.M * kTileYPad);
}

size_t smem_inv_plane(int cls, int nx, int ny, const Axis &ax, const Axis &ay)
{
    if (plane_line_class(cls)) return smem_inv_plane_line(cls, ny);
    const int kx = ax.M / 2 + 1;
    const int ps = ay.M | 1;
    // + the far path: coefficients contracted over z, then over x; the
    // Lagrange weights per axis; this step's node coefficients
    return sizeof(float2) * ((size_t)ax.M + ay.M + (size_t)kx * ps) + sizeof(float) * (size_t)nx * ny +
           sizeof(float) * kMaxFarPts * (kMaxFarPts + 2 * (size_t)nx + ny + 1 + kMaxFarPts * kMaxFarPts);
}

template <int M, bool CUBE>
static auto fwd_column_kernel()
{
    if constexpr (tile16_class(M)) return k_fwd_column16<M, CUBE>;
    else return k_fwd_column<M, CUBE>;
}

// The dynamic shared-memory limit is an attribute of the kernel function,
// shared by every context in the process, so each kernel is opened up to the
// device's opt-in maximum once (contexts never lower it for one another).
cudaError_t open_kernel_smem_limits(int max_optin)
{
    cudaError_t e;
    const auto open = [&](auto kern) { return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                                    max_optin); };
#define X(M) \
    if ((e = open(k_fwd_plane<M>)) || (e = open(k_inv_plane<M>))) return e;
    RP_PLANE_CLASSES(X)
#undef X
    if ((e = open(k_fwd_plane<32>))) return e;
#define X(M) \
    if ((e = open(fwd_column_kernel<M, false>())) || (e = open(fwd_column_kernel<M, (M > 0)>()))) return e;
    RP_COLUMN_CLASSES(X)
#undef X
    if ((e = open(k_mac_inv_column<false>)) || (e = open(k_mac_inv_column<true>))) return e;
    return open_plane_line_smem(max_optin);
}

cudaError_t launch_ring_push(const RawRing *d_rings, const IoPtrs &in, int d0, int d1,
                             const int *h_block0, int nblocks, long long step, cudaStream_t s)
{
    if (nblocks <= 0) return cudaSuccess;
    PushPrefix pre;
    for (int d = 0; d <= kMaxDomains; ++d) pre.block0[d] = 0;
    for (int d = d0; d <= d1; ++d) pre.block0[d] = h_block0[d];
    k_ring_push<<<nblocks, kThreads, 0, s>>>(d_rings, in, pre, d0, d1, step);
    return cudaGetLastError();
}

cudaError_t launch_fwd_plane(int cls, bool lane32, const FwdRing *d_rings, const IoPtrs &in, int r0, int r1, int block_lo,
                             int nblocks, size_t smem, int far_slot, cudaStream_t s)
{
    if (nblocks <= 0) return cudaSuccess;
    if (plane_line_class(cls) && !(lane32 && cls == 32))
        return launch_fwd_plane_line(cls, d_rings, in, r0, r1, block_lo, nblocks, smem, far_slot, s);
    switch (cls) {
    case 32:
        return launch_pdl(k_fwd_plane<32>, dim3(nblocks), dim3(kPlaneThreads), smem, s, d_rings, in, r0, r1, block_lo,
                          far_slot);
#define X(M)                                                                                                      \
    case M:                                                                                                       \
        return launch_pdl(k_fwd_plane<M>, dim3(nblocks), dim3(kPlaneThreads), smem, s, d_rings, in, r0, r1,       \
                          block_lo, far_slot);
        RP_PLANE_CLASSES(X)
#undef X
    default: return cudaErrorInvalidValue;
    }
}

// The general column and MAC kernels hold 552 B of shared memory per point
// along z and run for tens of microseconds in few blocks: launched while the
// kernel before still holds the SMs, several land on an SM that has room,
// beside idle ones, and which step that hits changes with every other kernel's
// size.  From 64 points along z (of the longest target: the plan's shared
// memory) they start after it.  9 x 9 x 33 box: step 67 -> 47 us (12 x 12 x 64
// 65 -> 63, two 6 x 6 x 48 69 -> 57, two 9 x 9 x 96 135 -> 126); at 48 points
// and fewer the launch gap costs more than it gives (6 x 6 x 20 22.5 -> 26.7).
constexpr size_t kGeneralApart = 64 * sizeof(float2) * (1 + 4 * kTileYPad);

cudaError_t launch_fwd_column(int cls, const FwdRing *d_rings, int r0, int r1, int block_lo, int nblocks,
                              size_t smem, long long step, cudaStream_t s)
{
    if (nblocks <= 0) return cudaSuccess;
    const int M = column_class(cls);
    const bool cube = M > 0 && plane_class(cls) == M, overlap = M > 0 || smem < kGeneralApart;
    if (tile16_class(M)) smem = smem_fwd_column16(M);
    const dim3 threads(tile16_class(M) ? kColumn16Threads : kColumnThreads);
    switch (M) {
#define X(M)                                                                                                  \
    case M:                                                                                                   \
        return launch_kernel(overlap, cube ? fwd_column_kernel<M, (M > 0)>() : fwd_column_kernel<M, false>(), \
                             dim3(nblocks), threads, smem, s, d_rings, r0, r1, block_lo, step);
        RP_COLUMN_CLASSES(X)
#undef X
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_mac_inv_column(bool comp, const InvTarget *d_tgts, int t0, int t1, int block_lo,
                                  const MacEntry *d_entries, int nblocks, size_t smem, long long step, int clamp,
                                  cudaStream_t s)
{
    if (nblocks <= 0) return cudaSuccess;
    return launch_kernel(smem < kGeneralApart, comp ? k_mac_inv_column<true> : k_mac_inv_column<false>, dim3(nblocks),
                         dim3(kThreads), smem, s, d_tgts, t0, t1, block_lo, d_entries, step, clamp);
}

cudaError_t launch_inv_plane(int cls, const InvTarget *d_tgts, int t0, int t1, int block_lo, const OutPtrs &out,
                             int nblocks, size_t smem, float inv_c, long long step, cudaStream_t s)
{
    if (nblocks <= 0) return cudaSuccess;
    if (plane_line_class(cls))
        return launch_inv_plane_line(cls, d_tgts, t0, t1, block_lo, out, nblocks, smem, inv_c, step, s);
    switch (cls) {
#define X(M)                                                                                                       \
    case M:                                                                                                        \
        return launch_pdl(k_inv_plane<M>, dim3(nblocks), dim3(kPlaneThreads), smem, s, d_tgts, t0, t1, block_lo,   \
                          out, inv_c, step);
        RP_PLANE_CLASSES(X)
#undef X
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace rp
