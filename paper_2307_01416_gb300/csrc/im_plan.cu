// Reach of each energy layer along its field's axis, for the influence-matrix
// column boxes.
//
// The influence matrix (paper Sec. 2.C) stores each spot's dose per primary
// as a sparse column.  The transport scores a spot's deposits into a dense
// box of the scoring grid first; a box that covers the field's whole depth
// holds, beyond the spots' Bragg peaks, voxels that no proton reaches, and
// each of them is cleared and read by every pass that builds the CSR.  This
// kernel finds, per (scenario, field, layer), the depth where a proton with
// the layer's largest residual range must have stopped: it marches rays
// parallel to the field's axis through the CT, one per lateral column of the
// opening, sums the water-equivalent path (SPR x scenario scale x length),
// and keeps, over the columns, the largest depth at which the sum reaches the
// layer's range.  A deposit beyond it (a bound that was too tight) is not
// lost: the transport records deposits outside an item's box one by one and
// the CSR build merges them.
#include <cstddef>

#include "vpmc_internal.cuh"

namespace vpmc {
namespace {

// One warp per lateral column of a job (blockIdx.x: the job).  Depths are
// stored as t - t0 >= 0, whose FP32 bit patterns order as the values do, so an
// integer maximum over the columns is the float maximum.
//
// A thread that marches a ray waits for two dependent loads (the voxel, its
// table entry) at every 0.5 mm, and there are few rays: 345 us for a field of
// 97 layers over 350 mm of water, with one thread per column.  Here the lanes
// take 32 consecutive steps, sum them in a warp scan, and find the first step
// that exhausts each of the job's (ascending) ranges with a ballot: 30 us (133
// to 199 us with eight steps' loads in flight per thread).
__global__ void k_depth_bounds(const uint16_t* __restrict__ ct, const float2* __restrict__ hu, Grid3 ctg,
                               const DepthJob* __restrict__ jobs, const float* __restrict__ r_lim,
                               unsigned* __restrict__ reach)
{
    const DepthJob J = jobs[blockIdx.x];
    const int ncol = J.na * J.nb;
    const int nstep = (int)ceilf((J.t1 - J.t0) / J.dt);
    const int lane = threadIdx.x & 31, per_block = blockDim.x >> 5;
    for (int c = blockIdx.y * per_block + (threadIdx.x >> 5); c < ncol; c += gridDim.y * per_block) {
        const float a = J.a0 + (float)(c % J.na) * J.da, b = J.b0 + (float)(c / J.na) * J.da;
        float q[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) q[k] = J.base[k] + a * J.u[k] + b * J.v[k];
        float wet = 0.0f;                            // of the steps before i0
        int r = 0;
        for (int i0 = 0; i0 < nstep && r < J.run_n; i0 += 32) {
            const float t = J.t0 + ((float)(i0 + lane) + 0.5f) * J.dt;
            long long idx = 0;
            bool inside = i0 + lane < nstep;
#pragma unroll
            for (int k = 2; k >= 0; --k) {
                const int v = (int)floorf((q[k] + t * J.w[k] - ctg.lo[k]) / ctg.d[k]);
                inside = inside && v >= 0 && v < ctg.n[k];
                idx = idx * ctg.n[k] + v;
            }
            float sum = inside ? hu[ct[idx]].y * J.spr_scale * J.dt : 0.0f;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const float below = __shfl_up_sync(0xffffffffu, sum, o);
                if (lane >= o) sum += below;
            }
            sum += wet;
            wet = __shfl_sync(0xffffffffu, sum, 31);
            for (; r < J.run_n; ++r) {
                const unsigned reached = __ballot_sync(0xffffffffu, sum >= r_lim[J.run_off + r]);
                if (!reached) break;
                if (lane == __ffs(reached) - 1)
                    atomicMax(reach + J.run_off + r, __float_as_uint(t + 0.5f * J.dt - J.t0));
            }
        }
        // a range the column never exhausts: the field's far end
        for (r += lane; r < J.run_n; r += 32) atomicMax(reach + J.run_off + r, __float_as_uint(J.t1 - J.t0));
    }
}

}  // namespace

cudaError_t launch_depth_bounds(const uint16_t* ct, const TablesImage* tables, Grid3 ctg, const DepthJob* jobs,
                                int n_jobs, int max_columns, const float* r_lim, unsigned* reach, cudaStream_t s)
{
    if (n_jobs <= 0) return cudaSuccess;
    const float2* hu = reinterpret_cast<const float2*>(reinterpret_cast<const char*>(tables) + offsetof(TablesImage, hu));
    const dim3 grid((unsigned)n_jobs, (unsigned)(max_columns < 4 * 4096 ? (max_columns + 3) / 4 : 4096));
    k_depth_bounds<<<grid, 128, 0, s>>>(ct, hu, ctg, jobs, r_lim, reach);
    return cudaGetLastError();
}

}  // namespace vpmc
