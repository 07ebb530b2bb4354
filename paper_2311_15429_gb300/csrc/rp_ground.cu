// Small elementwise kernels of the step bookkeeping.
//
//   k_ground_delta: the ground-state split of Eqs. 9-12 -- with the first
//                   sample S(0) taken as the ground state, the histories hold
//                   Delta S = S - S(0): Delta S of the pushed slices (rho and J
//                   at their own pointers) into the library's [4][N] scratch;
//   k_step_advance: graph replay -- the device step counter, +1 per replay.
#include <cuda_runtime.h>

#include "rp_fft.cuh"
#include "rp_internal.h"

namespace rp {

namespace {

constexpr int kGroundThreads = 256, kGroundChunk = 8 * kGroundThreads;

// Every domain of the push that has a slice, in one launch (a launch of its own
// per domain, 2 to 3 us each, was a tenth of the step of four 27^3 neighbours).
__global__ void __launch_bounds__(kGroundThreads)
    k_ground_delta(const GroundDomain *__restrict__ doms, int d0, int d1, IoPtrs in)
{
    const int b = blockIdx.x + doms[d0].block0;
    int lo = d0, hi = d1;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (doms[mid].block0 <= b) lo = mid; else hi = mid;
    }
    const GroundDomain D = doms[lo];
    const float *rho = in.rho[lo], *J = in.J[lo];
    if (!rho) return;   // another context's source
    const long long base = (long long)(b - D.block0) * kGroundChunk + threadIdx.x;
    pdl_trigger();
    pdl_wait();   // the slices, and the last readers of delta
#pragma unroll
    for (int k = 0; k < kGroundChunk / kGroundThreads; ++k) {
        const long long i = base + k * kGroundThreads;
        if (i < 4 * D.n) D.delta[i] = (i < D.n ? __ldg(rho + i) : __ldg(J + (i - D.n))) - __ldg(D.ground + i);
    }
}

// Graph replay: the step the replayed kernels read.
__global__ void k_step_advance(long long *d_step) { *d_step += 1; }

}  // namespace

cudaError_t launch_step_advance(long long *d_step, cudaStream_t s)
{
    k_step_advance<<<1, 1, 0, s>>>(d_step);
    return cudaGetLastError();
}

int ground_blocks(long long n) { return (int)((4 * n + kGroundChunk - 1) / kGroundChunk); }

cudaError_t launch_ground_delta(const GroundDomain *d_doms, int d0, int d1, int nblocks, const IoPtrs &in,
                                cudaStream_t s)
{
    if (nblocks <= 0) return cudaSuccess;
    return launch_pdl(k_ground_delta, dim3(nblocks), dim3(kGroundThreads), 0, s, d_doms, d0, d1, in);
}

}  // namespace rp
