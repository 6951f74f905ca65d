// Sec. 2.2 -- ray tracing of the masked fine texels with temporal
// accumulation (Eq. 1) and the front/back sign vote.
//
// Each masked coarse voxel contributes its 8 fine children ("texel slots");
// each slot casts R rays, so the frame's work is a flat list of
// 8 * masked * R ray ids (consecutive ids share a texel).  Per ray:
//   * the direction comes from Philox-4x32-10 (Salmon et al., SC'11) with
//     counter (draw, ray, frame, texel) and key (seed lo, seed hi), mapped to
//     the sphere by Marsaglia's (1972) rejection method -- integer accept
//     test, fp32 map, so every direction is bit-reproducible;
//   * the closest hit comes from a traversal of the 4-wide BVH that starts
//     from a front of it, shared by the rays of neighbouring texels
//     (front_dev.cuh); one 128-byte node fetch tests four child boxes, the
//     nearest hit child is entered next, the others pushed farthest-first
//     with their entry distance and skipped on pop once they cannot hold a
//     closer hit; leaves are tested with Moller-Trumbore in fp32 with the
//     operation order written out (explicit fma / rounding intrinsics);
//     equal distances keep the smaller original triangle index.
// Rays of very different lengths would leave most lanes of a lock-step warp
// idle, so warps are persistent and refill idle lanes with new rays once
// enough lanes are idle.  The traversal runs in two
// phases (a lane parks the leaf it reaches and keeps descending; the warp
// tests triangles when enough lanes hold a parked leaf), NODE_STEPS (three)
// node steps per phase decision.  A finished ray commits its distance (minimum of the
// float bits, t >= 0) and its front/back hit to its warp's shared memory;
// once a unit's rays have all finished, the warp applies Eq. 1 to its texels:
// u_t = min(u, r_t) (the alpha decay was applied by the mask kernel), the
// counts, and f_t = +-u_t (c_t while no ray has hit), negative when back
// hits outnumber front hits.  In the nearest-face sign mode a ray starts
// with the texel's u as its best hit and commits (t, face) as one key.
#include <math_constants.h>

#include "internal.cuh"
#include "front_dev.cuh"

namespace rtsdf {
namespace {

using namespace dev;

#ifndef TRACE_MIN_BLOCKS
#define TRACE_MIN_BLOCKS 8
#endif

// Units of one scene's rays, handed out in order from the frame's counter.
struct SceneUnits {
    const TraceArgs& a;
    unsigned long long total;
    __device__ __forceinline__ const TraceArgs& args(int) const { return a; }
    __device__ __forceinline__ int root(int) const { return a.nt > 1 ? 0 : (a.nt == 1 ? ~0 : WIDE_EMPTY); }
    __device__ __forceinline__ bool next(WarpTrace& w, uint32_t unit, unsigned lane, int& scene) const {
        unsigned long long c0 = 0;
        if (lane == 0) c0 = atomicAdd(a.next_ray, (unsigned long long)unit);
        c0 = __shfl_sync(0xFFFFFFFFu, c0, 0);
        if (c0 >= total) return false;
        if (lane == 0) {
            w.g0 = c0;
            w.len = (uint32_t)min((unsigned long long)unit, total - c0);
        }
        __syncwarp();
        scene = 0;
        return true;
    }
};

template <bool COUNT, bool TEX>
__global__ void __launch_bounds__(TRACE_THREADS, TRACE_MIN_BLOCKS) k_trace(TraceArgs a) {
    __shared__ BlockTrace s_trace;
    __shared__ TraceArgs s_args;   // what the unit source reads at refills
    chain_wait();
    if (threadIdx.x == 0) s_args = a;
    __syncthreads();
    SceneUnits src{s_args, (unsigned long long)(*a.count) * 8u * (unsigned long long)a.rays};
    const uint32_t unit = unit_rays(src.total, (uint32_t)a.rays, (uint32_t)a.ray_chunk);
    trace_units<COUNT, TEX>(src, a, unit, a.refill_min, a.leaf_min, s_trace, a.counters);
}

}  // namespace

cudaError_t trace_occupancy(int* per_sm) {
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, k_trace<false, true>, TRACE_THREADS, 0);
}

cudaError_t launch_trace(rtsdf_ctx* c, int rays, int frame) {
    TraceArgs a;
    a.masked = c->masked;
    a.count = c->d_masked_count;
    a.nc = c->nc;
    a.rays = rays;
    int lg = 0;
    while ((1 << lg) < rays) lg++;
    a.log2_rays = lg;
    a.key0 = (uint32_t)c->cfg.seed;
    a.key1 = (uint32_t)(c->cfg.seed >> 32);
    a.frame = (uint32_t)frame;
    a.bx = c->cfg.bmin[0];
    a.by = c->cfg.bmin[1];
    a.bz = c->cfg.bmin[2];
    a.hf = c->hf;
    a.wide = c->bvh.wide;
    a.wtex = texture_fetch_on() ? c->bvh.wtex : 0;
    a.tri = c->bvh.tri;
    a.nt = c->bvh.nt;
    a.coarse = c->coarse;
    a.accum = c->accum;
    a.counts = c->counts;
    a.fine = c->fine;
    a.err = c->d_err;
    a.counters = c->d_counters;
    a.next_ray = c->d_next_ray;
    a.refill_min = c->tune.refill_min;
    a.ray_chunk = c->tune.ray_chunk;
    a.leaf_min = c->tune.leaf_min;
    a.nc_mag = (uint32_t)((0x100000000ull + (unsigned long long)c->nc - 1) / (unsigned long long)c->nc);
    a.nearest = c->sign_mode == RTSDF_SIGN_NEAREST;
    // (the mask stage has cleared the ray counter)
    {
        int sms = 0, per_sm = 0;
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device);
        if (a.wtex) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_trace<false, true>, TRACE_THREADS, 0);
        else cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_trace<false, false>, TRACE_THREADS, 0);
        if (per_sm < 1) per_sm = 4;
        const int use = (c->tune.trace_blocks_per_sm > 0 && c->tune.trace_blocks_per_sm < per_sm)
                            ? c->tune.trace_blocks_per_sm : per_sm;
        c->trace_grid = (unsigned)(sms > 0 ? sms : 132) * (unsigned)use;
    }
    // the texture path when the node texture exists (plain loads otherwise)
    if (a.wtex) {
        if (c->counting) launch_chain(c, k_trace<true, true>, c->trace_grid, TRACE_THREADS, 0, a);
        else launch_chain(c, k_trace<false, true>, c->trace_grid, TRACE_THREADS, 0, a);
    } else {
        if (c->counting) launch_chain(c, k_trace<true, false>, c->trace_grid, TRACE_THREADS, 0, a);
        else launch_chain(c, k_trace<false, false>, c->trace_grid, TRACE_THREADS, 0, a);
    }
    return cudaGetLastError();
}

}  // namespace rtsdf
