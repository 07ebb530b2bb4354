// The plane passes of the FFT path for square cross-sections of M = 16 B
// points, B even (M = 32, 64, 96, 128, 192): one (field, z-plane) per block.
//
//   forward: rows in pairs (one complex line: row 2c real, row 2c + 1
//     imaginary) along x, split into the two rows' half spectra, then along y
//     for every kx <= M/2 into T1 ([field][kx][z][ky]);
//   inverse: T2 along y for every kx, rows y < ny kept, then back along x as
//     one complex line per pair of output rows, cropped, scaled, the far
//     coefficients' interpolation added, straight to phi / A.
//
// Neither memory nor arithmetic bounds them but what shared memory exchanges
// between the threads of a line, so a line is exchanged once per axis and no
// pass exists for copying, packing or splitting alone: a thread loads its
// points of a line from global memory (or the previous axis' result), makes
// one sub-transform in registers and writes it to the exchange, a second
// thread reads across and makes the other sub-transform, whose results go on
// as they leave the registers.  With M = 16 B the sub-transforms are of 16
// and B points, in the order that suits each axis' neighbour:
//
//   "B first":  n = 16 n1 + n2, k = k1 + B k2: loads of 16 consecutive points
//   "16 first": n = B n1 + n2, k = k1 + 16 k2: stores of 16 consecutive points
//
// so that global loads and stores are 128-byte runs (64 for real rows).  The
// row strides (17 for a column of 16, 17 B = B mod 16 for a line, 16 B + 1)
// keep every access free of bank conflicts.  Zero padding (inputs n >= M/2)
// skips half of the first layer, cropping (outputs k >= M/2) half of the last.
//
// Shared memory per plane of n = M/2 and the blocks an SM holds: M = 96 40 KB
// forward (5) and 44 inverse (4), M = 128 70 and 73 KB (3), M = 192 111 KB (2);
// the exchange of the y axis goes in chunks of kx lines to keep it there.
// Per launch, before (tile and lane-shuffle forms) and now: 32 x 48^3 with far
// pairs forward 111 -> 91 us, inverse 173 -> 112 (288 MB each: 42 us at the
// copy rate); 8 x 64^3 92 -> 49 and 125 -> 61 (170 MB: 25 us); 3 x 96^3 100 ->
// 67 and 188 -> 90 (198 MB: 29 us); 2 x 48^3 12.2 -> 11.3 and 13.7 -> 10.2.
// Launches of about one wave are latency: 128 blocks of 64 points 6.7 -> 7.2
// and 6.8 -> 7.5, 256 7.7 -> 7.1 and 7.6 -> 7.7, though the step of one 32^3
// went from 22.8 to 19.8.  Below that, at 32 points, the forward pass has the
// lane-shuffle form (kLanePlane32).  Half of the issue slots are used at many
// waves; what is left is waits on the loads of T2 and on barriers at 24 to 27
// warps per SM (prefetching a round of lines, or fewer blocks with more
// registers, changed nothing or lost).
#include <cuda_runtime.h>

#include "rp_fft.cuh"
#include "rp_internal.h"

namespace rp {

namespace {

// Threads per block and kx lines per chunk of the y exchange: whole rounds of
// tasks at n = M/2 (16 and B tasks a line), two chunks at 96 and 128, and at
// 192 what leaves room for two blocks.  The inverse pass at 96 takes four
// blocks of 208 threads: two rounds a chunk where 160 need three (2 x 48^3
// 12.6 -> 11.1 us, 32 x 48^3 118 -> 112).
__host__ __device__ constexpr int plane_threads(int M)
{
    return M == 32 ? 128 : M == 64 ? 144 : M == 96 ? 160 : M == 128 ? 288 : 320;
}
__host__ __device__ constexpr int inv_plane_threads(int M) { return M == 96 ? 208 : M == 192 ? 224 : plane_threads(M); }
__host__ __device__ constexpr int plane_blocks(int M) { return M <= 64 ? 6 : M == 96 ? 5 : M == 128 ? 3 : 2; }
__host__ __device__ constexpr int inv_plane_blocks(int M) { return M == 96 ? 4 : plane_blocks(M); }
__host__ __device__ constexpr int fwd_chunk(int M) { return M <= 64 ? M / 2 + 1 : M == 96 ? 25 : M == 128 ? 33 : 20; }
__host__ __device__ constexpr int inv_chunk(int M) { return M <= 64 ? M / 2 + 1 : M == 96 ? 25 : M == 128 ? 33 : 14; }
// rows y of a kx line between the axes of the inverse pass: even, and B mod 16
// (2 mod 16 at M = 128, where the padding to 8 would cost the third block)
__host__ __device__ constexpr int inv_row_stride(int M, int ny)
{
    const int r = M == 128 ? 2 : M / 16, n = ny + (ny & 1);
    return n + ((r - n) % 16 + 16) % 16;
}

constexpr int kFarRow = kMaxFarPts;   // far coefficients of a row, zero past the target's px

template <class T>
__device__ __forceinline__ int plane_owner(const T *arr, int lo, int hi, int b)
{
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (arr[mid].plane0 <= b) lo = mid; else hi = mid;
    }
    return lo;
}

// B-point DFT in natural order; HALF: v[B/2 ..] count as zero.
template <int B, bool INV, bool HALF>
__device__ __forceinline__ void dft_part(float2 (&v)[B])
{
    if constexpr (!HALF) {
        dft_b<B, INV>(v);
    } else if constexpr (B == 2) {
        v[1] = v[0];
    } else if constexpr (B == 4) {
        r4<INV, true>(v[0], v[1], v[2], v[3]);
    } else if constexpr (B == 6) {
        // n = 3a + b, k = c + 2d: radix 2 over a copies, twiddle W_6^{bc}, radix 3 over b
        const float s = INV ? 1.0f : -1.0f;
        float2 y0[3] = {v[0], v[1], v[2]};
        float2 y1[3] = {v[0], cmul(v[1], make_float2(0.5f, s * kSin60)), cmul(v[2], make_float2(-0.5f, s * kSin60))};
        dft3<INV>(y0[0], y0[1], y0[2]);
        dft3<INV>(y1[0], y1[1], y1[2]);
        v[0] = y0[0]; v[2] = y0[1]; v[4] = y0[2];
        v[1] = y1[0]; v[3] = y1[1]; v[5] = y1[2];
    } else if constexpr (B == 8) {
        // n = 2p + q, k = k1 + 4 k2
        r4<INV, true>(v[0], v[2], v[4], v[6]);
        r4<INV, true>(v[1], v[3], v[5], v[7]);
        const float s = INV ? -1.0f : 1.0f;
        v[3] = cmul(v[3], make_float2(kRt2, -s * kRt2));
        v[5] = mul_mi<INV>(v[5]);
        v[7] = cmul(v[7], make_float2(-kRt2, -s * kRt2));
        float2 y[8];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            y[k] = cadd(v[2 * k], v[2 * k + 1]);
            y[k + 4] = csub(v[2 * k], v[2 * k + 1]);
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) v[k] = y[k];
    } else {
        static_assert(B == 12, "dft_part: B = 2, 4, 6, 8 or 12");
        // n = 3p + q, k = k1 + 4 k2
#pragma unroll
        for (int q = 0; q < 3; ++q) r4<INV, true>(v[q], v[3 + q], v[6 + q], v[9 + q]);
        const float s = INV ? -1.0f : 1.0f;
        v[4] = cmul(v[4], make_float2(kSin60, -s * 0.5f));
        v[5] = cmul(v[5], make_float2(0.5f, -s * kSin60));
        v[7] = cmul(v[7], make_float2(0.5f, -s * kSin60));
        v[8] = cmul(v[8], make_float2(-0.5f, -s * kSin60));
        v[10] = mul_mi<INV>(v[10]);
        v[11] = make_float2(-v[11].x, -v[11].y);
#pragma unroll
        for (int k = 0; k < 4; ++k) dft3<INV>(v[3 * k], v[3 * k + 1], v[3 * k + 2]);
        float2 y[12];
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int d = 0; d < 3; ++d) y[k + 4 * d] = v[3 * k + d];
#pragma unroll
        for (int k = 0; k < 12; ++k) v[k] = y[k];
    }
}

// ---------------------------------------------------------------- forward

// Along x, B first: row pair c of the plane into Z[c * 17 B + k], k < M.
// HALF: nx <= M/2.  E and Z share the pairs' rows.
template <int M, bool HALF>
__device__ __forceinline__ void fwd_rows(const float *__restrict__ plane, int nx, int ny, const float2 (&w)[M / 16],
                                         float2 *Z)
{
    constexpr int B = M / 16, S = 17 * B, T = plane_threads(M), NB = HALF ? B / 2 : B;
    const int pairs = (ny + 1) >> 1, n2 = threadIdx.x & 15;
    for (int c = threadIdx.x >> 4; c < pairs; c += T / 16) {
        const float *ra = plane + 2 * c * nx, *rb = ra + nx;
        const bool vb = 2 * c + 1 < ny;
        float2 v[B];
#pragma unroll
        for (int n1 = 0; n1 < B; ++n1) {
            const int x = 16 * n1 + n2;
            const bool in = n1 < NB && x < nx;
            v[n1].x = in ? ra[x] : 0.0f;
            v[n1].y = in && vb ? rb[x] : 0.0f;
        }
        dft_part<B, false, HALF>(v);
        float2 *E = Z + c * S + n2;
        E[0] = v[0];
#pragma unroll
        for (int k1 = 1; k1 < B; ++k1) E[17 * k1] = cmul(v[k1], w[k1]);
    }
    __syncthreads();
    constexpr int PR = T / B;   // pairs per round: a round's rows are read before they are overwritten
    for (int c0 = 0; c0 < pairs; c0 += PR) {
        const int c = c0 + threadIdx.x / B, k1 = threadIdx.x % B;
        const bool on = threadIdx.x < PR * B && c < pairs;
        float2 x[16];
        if (on) {
#pragma unroll
            for (int i = 0; i < 16; ++i) x[i] = Z[c * S + 17 * k1 + i];
        }
        __syncthreads();
        if (on) {
            dft16<false, false>(x);
#pragma unroll
            for (int k2 = 0; k2 < 16; ++k2) Z[c * S + k1 + B * k2] = x[k2];
        }
    }
    __syncthreads();
}

// Along y, 16 first: lines kx = l0 .. l0 + nl - 1 of the rows' spectra through
// E2 (nl lines of 16 B + 1) to T1.  HALF: ny <= M/2.  A thread takes the line's
// points of both parities, n2 = 2j and 2j + 1, so that each pair's values
// Z[kx], Z[M - kx] are read once and give row 2c and row 2c + 1.
template <int M, bool HALF>
__device__ __forceinline__ void fwd_lines(const float2 *Z, float2 *E2, const float2 *tw, int l0, int nl, int pairs,
                                          float2 *__restrict__ out, long long rs)
{
    constexpr int B = M / 16, S = 17 * B, SE = 16 * B + 1, T = plane_threads(M), NR = HALF ? 8 : 16;
    for (int t = threadIdx.x; t < nl * (B / 2); t += T) {
        const int j = t / nl, l = t - j * nl, k = l0 + l, km = k == 0 ? 0 : M - k;
        float2 a[16], b[16];
#pragma unroll
        for (int n1 = 0; n1 < 16; ++n1) {
            const int c = (B / 2) * n1 + j;
            a[n1] = b[n1] = make_float2(0.0f, 0.0f);
            if (n1 < NR && c < pairs) {
                //   A[k] = (Z[k] + conj Z[M-k]) / 2,  B[k] = (Z[k] - conj Z[M-k]) / (2i)
                const float2 z = Z[c * S + k], y = cconj(Z[c * S + km]), d = csub(z, y);
                a[n1] = cscale(cadd(z, y), 0.5f);
                b[n1] = make_float2(0.5f * d.y, -0.5f * d.x);
            }
        }
        dft16<false, HALF>(a);
        float2 *E = E2 + l * SE + 32 * j;
        E[0] = a[0];
#pragma unroll
        for (int k1 = 1; k1 < 16; ++k1) E[k1] = cmul(a[k1], tw[2 * j * k1]);
        dft16<false, HALF>(b);
        E[16] = b[0];
#pragma unroll
        for (int k1 = 1; k1 < 16; ++k1) E[16 + k1] = cmul(b[k1], tw[(2 * j + 1) * k1]);
    }
    __syncthreads();
    const int k1 = threadIdx.x & 15;
    for (int l = threadIdx.x >> 4; l < nl; l += T / 16) {
        float2 v[B];
#pragma unroll
        for (int n2 = 0; n2 < B; ++n2) v[n2] = E2[l * SE + 16 * n2 + k1];
        dft_b<B, false>(v);
        float2 *row = out + (l0 + l) * rs + k1;
#pragma unroll
        for (int k2 = 0; k2 < B; ++k2) row[16 * k2] = v[k2];
    }
    __syncthreads();
}

template <int M>
__global__ void __launch_bounds__(plane_threads(M), plane_blocks(M))
    k_fwd_plane_line(const FwdRing *__restrict__ rings, IoPtrs in, int r0, int r1, int block_lo, int far_slot)
{
    constexpr int B = M / 16, H = M / 2, T = plane_threads(M), CH = fwd_chunk(M);
    extern __shared__ float4 smem_f4[];
    float2 *tw = reinterpret_cast<float2 *>(smem_f4);
    const int b = blockIdx.x + block_lo;
    const FwdRing &R = rings[plane_owner(rings, r0, r1, b)];
    const int nx = R.nx, ny = R.ny, nz = R.nz;
    const int local = b - R.plane0, f = local / nz, z = local - f * nz, pairs = (ny + 1) >> 1;
    float2 *Z = tw + M;                       // [pairs][17 B]
    float2 *E2 = Z + pairs * 17 * B;          // [CH][16 B + 1]
    load_twiddles(tw, R.tw_x, M);
    float2 w[B];                              // W_M^{n2 k1} of this thread's n2
#pragma unroll
    for (int k1 = 1; k1 < B; ++k1) w[k1] = __ldg(R.tw_x + (threadIdx.x & 15) * k1);
    pdl_trigger();
    pdl_wait();   // the input slice may come from the previous kernel; t1 was read by it
    const long long N = (long long)nx * ny * nz;
    const float *plane = (f == 0 ? in.rho[R.src] : in.J[R.src] + (long long)(f - 1) * N) + (long long)z * nx * ny;
    if (nx <= H) fwd_rows<M, true>(plane, nx, ny, w, Z);
    else fwd_rows<M, false>(plane, nx, ny, w, Z);
    float2 *out = R.t1 + ((long long)f * (H + 1) * nz + z) * M;
    const long long rs = (long long)nz * M;
    for (int l0 = 0; l0 <= H; l0 += CH) {
        const int nl = min(CH, H + 1 - l0);
        if (ny <= H) fwd_lines<M, true>(Z, E2, tw, l0, nl, pairs, out, rs);
        else fwd_lines<M, false>(Z, E2, tw, l0, nl, pairs, out, rs);
    }
    if (R.far_x) {
        // far path: this plane as bf16 hi/lo into row (slot, field) of the batch matrix
        __nv_bfloat16 *row = R.far_x + ((long long)far_slot * 4 + f) * 2 * R.far_ks + (long long)z * nx * ny;
        for (int i = threadIdx.x; i < nx * ny; i += T) {
            const float v = __ldg(plane + i);
            const __nv_bfloat16 hi = __float2bfloat16(v);
            row[i] = hi;
            row[R.far_ks + i] = __float2bfloat16(v - __bfloat162float(hi));
        }
    }
}

// ---------------------------------------------------------------- inverse

// Along y, B first: lines kx = l0 .. l0 + nl - 1 of T2 through E (nl lines of
// 17 B) into Y[kx * SY + y], y < nyp (ny rounded up to even).  CROP: nyp <= M/2.
template <int M, bool CROP>
__device__ __forceinline__ void inv_lines(const float2 *__restrict__ src, long long rs, const float2 (&w)[M / 16],
                                          float2 *E, float2 *Y, int SY, int l0, int nl, int nyp)
{
    constexpr int B = M / 16, S = 17 * B, T = inv_plane_threads(M);
    const int n2 = threadIdx.x & 15;
    for (int l = threadIdx.x >> 4; l < nl; l += T / 16) {
        const float2 *line = src + (l0 + l) * rs + n2;
        float2 v[B];
#pragma unroll
        for (int n1 = 0; n1 < B; ++n1) v[n1] = __ldg(line + 16 * n1);
        dft_b<B, true>(v);
        float2 *e = E + l * S + n2;
        e[0] = v[0];
#pragma unroll
        for (int k1 = 1; k1 < B; ++k1) e[17 * k1] = cmul(v[k1], w[k1]);
    }
    __syncthreads();
    for (int t = threadIdx.x; t < nl * B; t += T) {
        const int l = t / B, k1 = t - l * B;
        float2 x[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) x[i] = E[17 * t + i];
        dft16<true, false>(x);
        float2 *y = Y + (l0 + l) * SY + k1;
#pragma unroll
        for (int k2 = 0; k2 < (CROP ? 8 : 16); ++k2)
            if (k1 + B * k2 < nyp) y[B * k2] = x[k2];
    }
    __syncthreads();
}

// Along x, 16 first: output row pairs p0 .. p0 + np - 1 (rows 2p real, 2p + 1
// imaginary part) through E (np lines of 16 B + 1) to the output plane.
// CROP: nx <= M/2.  far: each row's coefficients vy ([ny][kFarRow]) are
// interpolated along x onto its values, with the weights lx of this thread's
// x = k1 + 16 k2 for up to four nodes, read from the table for more.
template <int M, bool CROP>
__device__ __forceinline__ void inv_rows(const float2 *Y, int SY, float2 *E, const float2 *tw, int p0, int np, int nx,
                                         int ny, float scale, const FarTarget *__restrict__ far, const float *vy,
                                         const float4 (&lx)[M / 32], float *__restrict__ dst)
{
    constexpr int B = M / 16, SE = 16 * B + 1, T = inv_plane_threads(M);
    for (int t = threadIdx.x; t < np * B; t += T) {
        const int n2 = t / np, p = t - n2 * np;
        float2 v[16];
#pragma unroll
        for (int n1 = 0; n1 < 16; ++n1) {
            const int k = B * n1 + n2;
            // rows A and B of the pair at kx = k or its mirror: A + iB
            const bool low = n1 < 8 || (n1 == 8 && n2 == 0);
            const float4 ab = *reinterpret_cast<const float4 *>(Y + (low ? k : M - k) * SY + 2 * (p0 + p));
            v[n1] = low ? make_float2(ab.x - ab.w, ab.y + ab.z) : make_float2(ab.x + ab.w, ab.z - ab.y);
            if (n2 == 0 && (n1 == 0 || n1 == 8)) v[n1] = make_float2(ab.x, ab.z);   // real: kx = 0 and M/2
        }
        dft16<true, false>(v);
        float2 *e = E + p * SE + 16 * n2;
        e[0] = v[0];
#pragma unroll
        for (int k1 = 1; k1 < 16; ++k1) e[k1] = cmul(v[k1], twid<true>(tw, n2 * k1));
    }
    __syncthreads();
    const int k1 = threadIdx.x & 15, px = far ? far->px : 0;
    for (int p = threadIdx.x >> 4; p < np; p += T / 16) {
        float2 v[B];
#pragma unroll
        for (int n2 = 0; n2 < B; ++n2) v[n2] = E[p * SE + 16 * n2 + k1];
        dft_b<B, true>(v);
        const int ya = 2 * (p0 + p);
        const bool vb = ya + 1 < ny;
        float *row = dst + ya * nx;
        float4 va = make_float4(0.0f, 0.0f, 0.0f, 0.0f), vc = va;
        if (far) {
            va = *reinterpret_cast<const float4 *>(vy + ya * kFarRow);
            vc = *reinterpret_cast<const float4 *>(vy + (ya + (vb ? 1 : 0)) * kFarRow);
        }
#pragma unroll
        for (int k2 = 0; k2 < (CROP ? B / 2 : B); ++k2) {
            const int x = k1 + 16 * k2;
            if (x >= nx) continue;
            float a = v[k2].x, c = v[k2].y;
            if (far) {
                const float4 l = lx[k2 % (M / 32)];
                if (CROP && px <= 4) {
                    a += fmaf(l.w, va.w, fmaf(l.z, va.z, fmaf(l.y, va.y, l.x * va.x)));
                    c += fmaf(l.w, vc.w, fmaf(l.z, vc.z, fmaf(l.y, vc.y, l.x * vc.x)));
                } else {
                    float sa = 0.0f, sc = 0.0f;
                    for (int i = 0; i < px; ++i) {
                        const float w = __ldg(far->Lx + x * px + i);
                        sa = fmaf(w, vy[ya * kFarRow + i], sa);
                        sc = fmaf(w, vy[(ya + (vb ? 1 : 0)) * kFarRow + i], sc);
                    }
                    a += sa;
                    c += sc;
                }
            }
            row[x] = scale * a;
            if (vb) row[nx + x] = scale * c;
        }
    }
    __syncthreads();
}

template <int M>
__global__ void __launch_bounds__(inv_plane_threads(M), inv_plane_blocks(M))
    k_inv_plane_line(const InvTarget *__restrict__ tgts, int t0, int t1, int block_lo, OutPtrs out, float inv_c,
                     long long step)
{
    constexpr int B = M / 16, H = M / 2, T = inv_plane_threads(M), CH = inv_chunk(M);
    extern __shared__ float4 smem_f4[];
    float2 *tw = reinterpret_cast<float2 *>(smem_f4);
    const int b = blockIdx.x + block_lo;
    const InvTarget &I = tgts[plane_owner(tgts, t0, t1, b)];
    const int nx = I.nx, ny = I.ny, nz = I.nz;
    const int local = b - I.plane0, f = local / nz, z = local - f * nz;
    const int pairs = (ny + 1) >> 1, SY = inv_row_stride(M, ny);
    float2 *Y = tw + M;                                        // [H + 1][SY]
    float2 *E = Y + (H + 1) * SY;                              // [CH][17 B]
    float *vy = reinterpret_cast<float *>(E + CH * 17 * B);    // far: [ny][kFarRow]
    load_twiddles(tw, I.tw_x, M);
    float2 w[B];                                               // conj W_M^{n2 k1} of this thread's n2
#pragma unroll
    for (int k1 = 1; k1 < B; ++k1) w[k1] = cconj(__ldg(I.tw_x + (threadIdx.x & 15) * k1));
    pdl_trigger();
    pdl_wait();   // T2 is written by the MAC, the coefficient ring by the far path
    if (step < 0) step = *I.d_step;   // graph replay: the step from the device counter
    const float2 *src = I.t2 + ((long long)f * (H + 1) * nz + z) * M;
    const long long rs = (long long)nz * M;
    for (int l0 = 0; l0 <= H; l0 += CH) {
        const int nl = min(CH, H + 1 - l0);
        if (2 * pairs <= H) inv_lines<M, true>(src, rs, w, E, Y, SY, l0, nl, 2 * pairs);
        else inv_lines<M, false>(src, rs, w, E, Y, SY, l0, nl, 2 * pairs);
    }
    const FarTarget *far = I.far;
    float4 lx[M / 32];                                         // far: x weights of this thread's x < M/2
    if (far) {
        const int px = far->px;
#pragma unroll
        for (int k2 = 0; k2 < M / 32; ++k2) {
            const int x = (threadIdx.x & 15) + 16 * k2;
            const float *l = far->Lx + (x < nx ? x : 0) * px;
            lx[k2] = make_float4(__ldg(l), px > 1 ? __ldg(l + 1) : 0.0f, px > 2 ? __ldg(l + 2) : 0.0f,
                                 px > 3 ? __ldg(l + 3) : 0.0f);
        }
    }
    // far pairs: this step's node coefficients of field f contracted over z
    // (scratch in E), then over y for every row
    if (far) {
        const int px = far->px, py = far->py, pz = far->pz, pxy = px * py;
        const float *c = far->cring + (step % far->depth) * (far->r * 4) + f;
        float *cz = reinterpret_cast<float *>(E);
        for (int i = threadIdx.x; i < pxy; i += T) {
            float s = 0.0f;
            for (int k = 0; k < pz; ++k) s = fmaf(__ldg(far->Lz + z * pz + k), c[4 * (k * pxy + i)], s);
            cz[i] = s;
        }
        __syncthreads();
        for (int i = threadIdx.x; i < ny * kFarRow; i += T) {
            const int y = i / kFarRow, a = i % kFarRow;
            float u = 0.0f;
            if (a < px)
                for (int k = 0; k < py; ++k) u = fmaf(__ldg(far->Ly + y * py + k), cz[k * px + a], u);
            vy[i] = u;
        }
        __syncthreads();
    }
    const long long N = (long long)nx * ny * nz;
    float *dst = (f == 0 ? out.phi[I.dom] : out.A[I.dom] + (long long)(f - 1) * N) + (long long)z * nx * ny;
    const float scale = f == 0 ? 1.0f : inv_c;
    constexpr int CP = CH;   // pairs per chunk: 16 B + 1 <= 17 B
    for (int p0 = 0; p0 < pairs; p0 += CP) {
        const int np = min(CP, pairs - p0);
        if (nx <= H) inv_rows<M, true>(Y, SY, E, tw, p0, np, nx, ny, scale, far, vy, lx, dst);
        else inv_rows<M, false>(Y, SY, E, tw, p0, np, nx, ny, scale, far, vy, lx, dst);
    }
}

#define RP_PLANE_CLASSES(X) X(32) X(64) X(96) X(128) X(192)

}  // namespace

bool plane_line_class(int M) { return M == 32 || M == 64 || M == 96 || M == 128 || M == 192; }

size_t smem_fwd_plane_line(int M, int ny)
{
    const size_t B = M / 16;
    return sizeof(float2) * (M + (size_t)((ny + 1) / 2) * 17 * B + (size_t)fwd_chunk(M) * (16 * B + 1));
}

size_t smem_inv_plane_line(int M, int ny)
{
    const size_t B = M / 16;
    return sizeof(float2) * (M + (size_t)(M / 2 + 1) * inv_row_stride(M, ny) + (size_t)inv_chunk(M) * 17 * B) +
           sizeof(float) * (size_t)kFarRow * ny;
}

cudaError_t open_plane_line_smem(int max_optin)
{
    cudaError_t e;
#define X(M)                                                                                                        \
    if ((e = cudaFuncSetAttribute(k_fwd_plane_line<M>, cudaFuncAttributeMaxDynamicSharedMemorySize, max_optin)) || \
        (e = cudaFuncSetAttribute(k_inv_plane_line<M>, cudaFuncAttributeMaxDynamicSharedMemorySize, max_optin)))   \
        return e;
    RP_PLANE_CLASSES(X)
#undef X
    return cudaSuccess;
}

cudaError_t launch_fwd_plane_line(int M, const FwdRing *d_rings, const IoPtrs &in, int r0, int r1, int block_lo,
                                  int nblocks, size_t smem, int far_slot, cudaStream_t s)
{
    switch (M) {
#define X(M)                                                                                                        \
    case M:                                                                                                         \
        return launch_pdl(k_fwd_plane_line<M>, dim3(nblocks), dim3(plane_threads(M)), smem, s, d_rings, in, r0, r1, \
                          block_lo, far_slot);
        RP_PLANE_CLASSES(X)
#undef X
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_inv_plane_line(int M, const InvTarget *d_tgts, int t0, int t1, int block_lo, const OutPtrs &out,
                                  int nblocks, size_t smem, float inv_c, long long step, cudaStream_t s)
{
    switch (M) {
#define X(M)                                                                                                       \
    case M:                                                                                                        \
        return launch_pdl(k_inv_plane_line<M>, dim3(nblocks), dim3(inv_plane_threads(M)), smem, s, d_tgts, t0, t1, \
                          block_lo, out, inv_c, step);
        RP_PLANE_CLASSES(X)
#undef X
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace rp
