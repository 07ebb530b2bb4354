// The fields of App. B from the potentials on one domain's grid:
//
//   E = -grad phi - (1/c) dA/dt,    B = curl A        (atomic units)
//
// Space derivatives: second-order central differences, second-order
// one-sided ones on the grid faces.  Time derivative: the second-order
// backward difference (3 A_l - 4 A_{l-1} + A_{l-2}) / (2 dt), or the
// first-order one (A_l - A_{l-1}) / dt without A_{l-2}.
//
// 64 B per node from and to HBM; a domain's grid is one wave of blocks, so
// latency bounds it: few instructions before the loads (32-bit indices; three
// 64-bit divisions a node were most of the kernel), and, where rows and
// pointers allow 16-byte accesses (nx a multiple of 4), four nodes along x per
// thread with all of its loads independent.  Neighbours come through L1, the
// launch overlaps the kernel before it.  64^3 (16.8 MB, 2.5 us at the copy
// rate): 8.2 -> 5.4 us per call.
#include <cuda_runtime.h>

#include "rp_fft.cuh"
#include "rp_internal.h"

namespace rp {

namespace {

constexpr int kFieldThreads = 128;

__device__ __forceinline__ float4 ld4(const float *p) { return __ldg(reinterpret_cast<const float4 *>(p)); }
__device__ __forceinline__ void st4(float *p, float4 v) { *reinterpret_cast<float4 *>(p) = v; }
__device__ __forceinline__ float4 sub4(float4 a, float4 b)
{
    return make_float4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w);
}
// 3 a - 4 b + c of nearly equal values: 4 b is exact, so that 3 a - 4 b rounds
// once and the last addition cancels (any other order rounds at the size of
// the terms)
__device__ __forceinline__ float three(float a, float b, float c) { return __fadd_rn(fmaf(3.0f, a, -4.0f * b), c); }
// -3 a + 4 b - c, the one-sided difference (negated on the far face)
__device__ __forceinline__ float edge(float a, float b, float c) { return -three(a, b, c); }
__device__ __forceinline__ float4 edge4(float4 a, float4 b, float4 c)
{
    return make_float4(edge(a.x, b.x, c.x), edge(a.y, b.y, c.y), edge(a.z, b.z, c.z), edge(a.w, b.w, c.w));
}

// 2 h df/d(axis) at index i of n along a stride s; f points at the node(s)
__device__ __forceinline__ float diff(const float *__restrict__ f, int i, int n, long long s)
{
    if (i == 0) return edge(__ldg(f), __ldg(f + s), __ldg(f + 2 * s));
    if (i == n - 1) return -edge(__ldg(f), __ldg(f - s), __ldg(f - 2 * s));
    return __ldg(f + s) - __ldg(f - s);
}
__device__ __forceinline__ float4 diff4(const float *__restrict__ f, int i, int n, long long s)
{
    if (i == 0) return edge4(ld4(f), ld4(f + s), ld4(f + 2 * s));
    if (i == n - 1) return sub4(make_float4(0.f, 0.f, 0.f, 0.f), edge4(ld4(f), ld4(f - s), ld4(f - 2 * s)));
    return sub4(ld4(f + s), ld4(f - s));
}
// the same along x for nodes x .. x + 3 of the row
__device__ __forceinline__ float4 diffx4(const float *__restrict__ f, int x, int nx)
{
    const float4 v = ld4(f);
    const float l = x > 0 ? __ldg(f - 1) : 0.0f, r = x + 4 < nx ? __ldg(f + 4) : 0.0f;
    return make_float4(x > 0 ? v.y - l : edge(v.x, v.y, v.z), v.z - v.x, v.w - v.y,
                       x + 4 < nx ? r - v.z : -edge(v.w, v.z, v.y));
}

template <bool VEC, class Index>
__global__ void __launch_bounds__(kFieldThreads)
    k_fields(int nx, int ny, int nz, float inv_2h, float inv_c, float inv_dt, const float *__restrict__ phi,
             const float *__restrict__ A, const float *__restrict__ A1, const float *__restrict__ A2,
             float *__restrict__ E, float *__restrict__ B)
{
    constexpr int V = VEC ? 4 : 1;
    const Index row = (Index)nx / V, q = (Index)blockIdx.x * kFieldThreads + threadIdx.x;
    const Index line = q / row;
    const int x = (int)(q - line * row) * V, z = (int)(line / ny), y = (int)(line - (Index)z * ny);
    pdl_trigger();
    pdl_wait();   // the potentials are written by the kernels before
    if (z >= nz) return;
    const long long sy = nx, sz = (long long)nx * ny, N = sz * nz, k = (long long)line * nx + x;
    const float *Ax = A + k, *Ay = Ax + N, *Az = Ay + N;
    if constexpr (VEC) {
        const float4 g[3] = {diffx4(phi + k, x, nx), diff4(phi + k, y, ny, sy), diff4(phi + k, z, nz, sz)};
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float4 a0 = ld4(A + a * N + k), a1 = ld4(A1 + a * N + k);
            const float4 a2 = A2 ? ld4(A2 + a * N + k) : a1;
            const auto rate = [&](float u, float v, float w) {
                return A2 ? three(u, v, w) * (0.5f * inv_dt) : (u - v) * inv_dt;
            };
            st4(E + a * N + k, make_float4(fmaf(-inv_c, rate(a0.x, a1.x, a2.x), -__fmul_rn(g[a].x, inv_2h)),
                                           fmaf(-inv_c, rate(a0.y, a1.y, a2.y), -__fmul_rn(g[a].y, inv_2h)),
                                           fmaf(-inv_c, rate(a0.z, a1.z, a2.z), -__fmul_rn(g[a].z, inv_2h)),
                                           fmaf(-inv_c, rate(a0.w, a1.w, a2.w), -__fmul_rn(g[a].w, inv_2h))));
        }
        if (B) {
            const auto curl = [&](long long at, float4 u, float4 v) {
                const float4 d = sub4(u, v);
                st4(B + at + k, make_float4(d.x * inv_2h, d.y * inv_2h, d.z * inv_2h, d.w * inv_2h));
            };
            curl(0, diff4(Az, y, ny, sy), diff4(Ay, z, nz, sz));
            curl(N, diff4(Ax, z, nz, sz), diffx4(Az, x, nx));
            curl(2 * N, diffx4(Ay, x, nx), diff4(Ax, y, ny, sy));
        }
    } else {
        const float g[3] = {diff(phi + k, x, nx, 1), diff(phi + k, y, ny, sy), diff(phi + k, z, nz, sz)};
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float a0 = __ldg(A + a * N + k), a1 = __ldg(A1 + a * N + k);
            const float rate = A2 ? three(a0, a1, __ldg(A2 + a * N + k)) * (0.5f * inv_dt) : (a0 - a1) * inv_dt;
            E[a * N + k] = fmaf(-inv_c, rate, -__fmul_rn(g[a], inv_2h));
        }
        if (B) {
            B[k] = (diff(Az, y, ny, sy) - diff(Ay, z, nz, sz)) * inv_2h;
            B[N + k] = (diff(Ax, z, nz, sz) - diff(Az, x, nx, 1)) * inv_2h;
            B[2 * N + k] = (diff(Ay, x, nx, 1) - diff(Ax, y, ny, sy)) * inv_2h;
        }
    }
}

bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

}  // namespace

cudaError_t launch_fields(int nx, int ny, int nz, double h, double c, double dt, const float *phi, const float *A,
                          const float *A1, const float *A2, float *E, float *B, cudaStream_t s)
{
    const long long N = (long long)nx * ny * nz;
    if (N <= 0) return cudaSuccess;
    const bool vec = nx % 4 == 0 && aligned16(phi) && aligned16(A) && aligned16(A1) && aligned16(A2) && aligned16(E) &&
                     aligned16(B);
    const long long items = vec ? N / 4 : N;
    const unsigned blocks = (unsigned)((items + kFieldThreads - 1) / kFieldThreads);
    const float i2h = (float)(0.5 / h), ic = (float)(1.0 / c), idt = (float)(1.0 / dt);
    const auto go = [&](auto kern) {
        return launch_pdl(kern, dim3(blocks), dim3(kFieldThreads), 0, s, nx, ny, nz, i2h, ic, idt, phi, A, A1, A2, E, B);
    };
    if (items + kFieldThreads > 0xffffffffLL)   // 64-bit indices
        return vec ? go(k_fields<true, unsigned long long>) : go(k_fields<false, unsigned long long>);
    return vec ? go(k_fields<true, unsigned>) : go(k_fields<false, unsigned>);
}

}  // namespace rp
