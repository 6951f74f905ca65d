// Sec. 2.3 -- soft shadows by sphere tracing the fine SDF, and the
// reverse-mode derivative of that march.
//
// Forward, per shading point p with normal n and unit light direction L:
//   o = p + 2 eps n, t = 0, res = 1, ph = 1e20
//   for i < steps:
//     q = o + t L; stop when q leaves the scene cube
//     h = S(q) (trilinear, cell-centred texels, clamped to the first/last centre)
//     h < eps: visibility 0 (the march met a surface; eps >= one texel, Sec. 2.3)
//     y = h^2 / (2 ph), dd = sqrt(max(h^2 - y^2, 0))
//     t - y > 0: res = min(res, k dd / (t - y))   (triangulation of the
//                current and previous samples, Aaltonen 2018, as in Sec. 2.3)
//     ph = h; t += min(h, step_max)                (restricted step, Sec. 2.3)
//   visibility = clamp(res, 0, 1)
// The grid is gathered through the read-only path; a 1080p floor image at
// 512^3 reads a few hundred MB of texels from L2/L1, not HBM.
//
// Backward: the march is re-run per point (nothing is stored by the forward
// pass), the t_i of the steps that carry a derivative kept in per-thread local
// memory, then the single penumbra term that produced the visibility (its arg-min step i*) is
// differentiated and swept back to step 0 through h_j = S(o + t_j L) and
// t_{j+1} = t_j + min(h_j, step_max):
//   dsdf[texel] += hbar_j w_texel(q_j)            (fp32 atomics)
//   qbar_j = hbar_j grad S(q_j),  tbar_j += qbar_j . L,  Lbar += t_j qbar_j
// Lbar is reduced per block and mapped through L = v / |v| to the
// unnormalised light vector.  Points stopped by h < eps, points whose res
// stayed 1 and clamped square roots carry no derivative.
#include <math_constants.h>
#include <string.h>

#include "internal.cuh"
#include "trace_dev.cuh"   // Philox-4x32-10

namespace rtsdf {
namespace {

constexpr int SHADOW_THREADS = 128;

struct ShadowArgs {
    const float* sdf;
    int n;
    float bx, by, bz, ext, inv_h;
    const float* pos;
    const float* nrm;
    long long npix;
    float Lx, Ly, Lz;
    float k, smax, eps;
    int steps;
    float jitter;              // origin jitter toward the light, world units (0: none)
    uint32_t frame, key0, key1;
};

// Sec. 2.3: the origin moves toward the light by xi x jitter, with xi in
// [0, 1) the top 24 bits of the first word of Philox-4x32-10, counter
// (pixel lo, pixel hi, frame, 0x53484457 "SHDW"), key = the context seed.
__device__ __forceinline__ float jitter_shift(const ShadowArgs& a, long long i) {
    uint32_t c[4] = {(uint32_t)i, (uint32_t)((unsigned long long)i >> 32), a.frame, 0x53484457u};
    dev::philox4x32_10(c, a.key0, a.key1);
    return __fmul_rn(__fmul_rn(__uint2float_rn(c[0] >> 8), 0x1p-24f), a.jitter);
}

struct Taps {
    int idx[8];
    float w[8];
    float grad[3];   // d S / d q
};

// S at offset (dx, dy, dz) from the lower corner of the scene cube.  The fine
// grid has n = 2 N >= 2 texels per axis, so a cell's upper neighbour is always
// the next texel, and the eight taps are four rows of two.
// GRAD: also the taps and the gradient.  NC: read the grid through the
// read-only path (not in a chained kernel, see chain_begin).
template <bool GRAD, bool NC>
__device__ __forceinline__ float sample(const ShadowArgs& a, float dx_, float dy_, float dz_, Taps* tp) {
    const int n = a.n;
    const float d[3] = {dx_, dy_, dz_};
    const float top = (float)(n - 1);
    int i0[3];
    float fr[3], dg[3];
#pragma unroll
    for (int ax = 0; ax < 3; ax++) {
        const float g0 = __fsub_rn(__fmul_rn(d[ax], a.inv_h), 0.5f);
        if (GRAD) dg[ax] = g0 > 0.f && !(g0 >= top) ? a.inv_h : 0.f;
        const float g = fminf(fmaxf(g0, 0.f), top);   // NaN goes to 0
        i0[ax] = min((int)g, n - 2);
        fr[ax] = g - (float)i0[ax];
    }
    const int id0 = i0[0] + n * (i0[1] + n * i0[2]);
    const float* p = a.sdf + id0;
    float val = 0.f;
    float gx = 0.f, gy = 0.f, gz = 0.f;
#pragma unroll
    for (int c = 0; c < 8; c++) {
        const int dx = c & 1, dy = (c >> 1) & 1, dz = c >> 2;
        const float wx = dx ? fr[0] : 1.f - fr[0], wy = dy ? fr[1] : 1.f - fr[1], wz = dz ? fr[2] : 1.f - fr[2];
        const int off = dx + n * (dy + n * dz);
        const float fv = NC ? __ldg(p + off) : p[off];
        const float w = wx * wy * wz;
        val = fmaf(w, fv, val);
        if (GRAD) {
            tp->idx[c] = id0 + off;
            tp->w[c] = w;
            gx = fmaf((dx ? 1.f : -1.f) * wy * wz, fv, gx);
            gy = fmaf(wx * (dy ? 1.f : -1.f) * wz, fv, gy);
            gz = fmaf(wx * wy * (dz ? 1.f : -1.f), fv, gz);
        }
    }
    if (GRAD) {
        tp->grad[0] = gx * dg[0];
        tp->grad[1] = gy * dg[1];
        tp->grad[2] = gz * dg[2];
    }
    return val;
}

// Whether the penumbra term of a step, k dd / (t - y), may be below res (or
// anything is not finite).  The march's divisions and root cost a third of a
// step, and in most steps the term is far above res: it is bounded from below
// here with an approximate reciprocal and squares (relative errors below 1e-6,
// taken as 1e-5), and only evaluated where the bound does not settle it, so the
// result keeps every bit.  r: 1 / (2 ph), approximate.
__device__ __forceinline__ bool may_lower(float k, float h, float t, float r, float res) {
    const float h2 = h * h, y = h2 * r;
    const float a2 = fmaf(-1e-5f, h2, fmaf(-y, y, h2));                // at most h^2 - y^2
    const float den = fmaf(1e-5f, t + y, t - y);                       // at least t - y
    const float rd = res * den * 1.00001f, rd2 = rd * rd;
    // (squares near the underflow are left to the exact form)
    return !(den < 0.f || ((k * k) * a2 >= rd2 && fminf(a2, rd2) > 1e-30f));
}

__device__ __forceinline__ float approx_half_rcp(float ph) { return 0.5f * __fdividef(1.f, ph); }

// The bounds of the scene cube as the march tests them: x >= b, by the sign of
// x - b (exact), and x <= b + ext.
struct Inside {
    float hx, hy, hz;
    __device__ __forceinline__ explicit Inside(const ShadowArgs& a) : hx(a.bx + a.ext), hy(a.by + a.ext), hz(a.bz + a.ext) {}
    __device__ __forceinline__ bool operator()(float qx, float qy, float qz, float dx, float dy, float dz) const {
        return dev::fmin3(dx, dy, dz) >= 0.f && qx <= hx && qy <= hy && qz <= hz;
    }
};

// Bound by the taps: a step waits for its eight loads (63 % of the L1 pipe's
// wavefronts, 3.2 a load: neighbouring marches drift apart) and issues 118
// instructions (73 % of the issue slots).  1920 x 1080 points, 256^3 grid, 64
// steps: 350 us with every penumbra term evaluated and per-axis clamps, 261 us
// now; blocks of 128 instead of 256 take 2 % off (10 % for 427 x 240 points).
// Tried, no change: floor without the conversion unit, 32 registers (64 warps
// an SM), two steps unrolled, the sample after a restricted step taken ahead
// (427 x 240: 28.6 instead of 17.0 us).
__global__ void __launch_bounds__(SHADOW_THREADS) k_shadow(ShadowArgs a, float* __restrict__ vis) {
    chain_begin();
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= a.npix) return;
    const float two_eps = 2.f * a.eps;
    float ox = fmaf(a.nrm[3 * i], two_eps, a.pos[3 * i]);
    float oy = fmaf(a.nrm[3 * i + 1], two_eps, a.pos[3 * i + 1]);
    float oz = fmaf(a.nrm[3 * i + 2], two_eps, a.pos[3 * i + 2]);
    if (a.jitter != 0.f) {
        const float sh = jitter_shift(a, i);
        ox = fmaf(sh, a.Lx, ox);
        oy = fmaf(sh, a.Ly, oy);
        oz = fmaf(sh, a.Lz, oz);
    }
    const Inside inside(a);
    float t = 0.f, res = 1.f, ph = 1e20f;
    for (int s = 0; s < a.steps; s++) {
        const float qx = fmaf(t, a.Lx, ox), qy = fmaf(t, a.Ly, oy), qz = fmaf(t, a.Lz, oz);
        const float dx = __fsub_rn(qx, a.bx), dy = __fsub_rn(qy, a.by), dz = __fsub_rn(qz, a.bz);
        if (!inside(qx, qy, qz, dx, dy, dz)) break;
        const float h = sample<false, false>(a, dx, dy, dz, nullptr);
        if (h < a.eps) {
            res = 0.f;
            break;
        }
        if (may_lower(a.k, h, t, approx_half_rcp(ph), res)) {
            const float y = h * h / (2.f * ph);
            const float dd = sqrtf(fmaxf(h * h - y * y, 0.f));
            if (t - y > 0.f) res = fminf(res, a.k * dd / (t - y));
        }
        ph = h;
        t += fminf(h, a.smax);
    }
    vis[i] = fminf(fmaxf(res, 0.f), 1.f);
}

// Bound by the latency of the re-marched steps (49 % of the issue slots, 52 %
// of the warps): 42 registers let 12 blocks of 128 reside.  1024^2 points,
// 512^3 grid: 439 us with (t, h) of every step in local memory and every step
// swept back, 210 us now (221 us at 56 registers).
__global__ void __launch_bounds__(128, 12) k_shadow_bwd(ShadowArgs a, const float* __restrict__ dvis,
                                                   float* __restrict__ dsdf, float* __restrict__ dlight,
                                                   float inv_norm) {
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    float lbx = 0.f, lby = 0.f, lbz = 0.f;
    if (i < a.npix && dvis[i] != 0.f) {
        // The sweep back visits step j < s - 1 only through t_{j+1} = t_j +
        // min(h_j, step_max), so only steps with h_j < step_max matter to it:
        // their t_j are kept (and, with the sign set, those of steps whose h_j
        // is not finite, which pass on what 0 times their taps gives).
        float ts[MAX_SHADOW_STEPS];
        const float two_eps = 2.f * a.eps;
        const float ox = fmaf(a.nrm[3 * i], two_eps, a.pos[3 * i]);
        const float oy = fmaf(a.nrm[3 * i + 1], two_eps, a.pos[3 * i + 1]);
        const float oz = fmaf(a.nrm[3 * i + 2], two_eps, a.pos[3 * i + 2]);
        const Inside inside(a);
        float t = 0.f, res = 1.f, ph = 1e20f, tprev = 0.f;
        int kept = 0, kept_prev = 0;           // kept steps before this one, before the previous one
        // the arg-min step: index, t, h, the previous step's h and t, kept steps before that
        int am = -1, am_kept = 0;
        float am_t = 0.f, am_h = 0.f, am_p = 0.f, am_tp = 0.f;
        bool term = false;
        for (int s = 0; s < a.steps; s++) {
            const float qx = fmaf(t, a.Lx, ox), qy = fmaf(t, a.Ly, oy), qz = fmaf(t, a.Lz, oz);
            const float dx = __fsub_rn(qx, a.bx), dy = __fsub_rn(qy, a.by), dz = __fsub_rn(qz, a.bz);
            if (!inside(qx, qy, qz, dx, dy, dz)) break;
            const float h = sample<false, true>(a, dx, dy, dz, nullptr);
            if (h < a.eps) {
                term = true;
                break;
            }
            if (may_lower(a.k, h, t, approx_half_rcp(ph), res)) {
                const float y = h * h / (2.f * ph);
                const float dd = sqrtf(fmaxf(h * h - y * y, 0.f));
                if (t - y > 0.f) {
                    const float g = a.k * dd / (t - y);
                    if (g < res) {
                        res = g;
                        am = s;
                        am_kept = kept_prev;
                        am_t = t;
                        am_h = h;
                        am_p = ph;
                        am_tp = tprev;
                    }
                }
            }
            kept_prev = kept;
            if (!(h >= a.smax && h < CUDART_INF_F)) ts[kept++] = h < a.smax ? t : -t;
            ph = h;
            tprev = t;
            t += fminf(h, a.smax);
        }
        if (!term && am >= 0) {
            const float h = am_h, tt = am_t, p = am_p;
            const float y = h * h / (2.f * p);
            const float a2 = h * h - y * y;
            if (a2 > 0.f) {
                const float dd = sqrtf(a2), den = tt - y;
                const float dy_dh = h / p, dy_dp = -y / p;
                const float ddd_dh = (h - y * dy_dh) / dd, ddd_dp = (-y * dy_dp) / dd;
                const float gb = dvis[i];
                const float kd = a.k / den, kd2 = a.k * dd / (den * den);
                float hbar = gb * (kd * ddd_dh + kd2 * dy_dh);
                const float pbar = am > 0 ? gb * (kd * ddd_dp + kd2 * dy_dp) : 0.f;
                float tbar = -gb * kd2;
                float tj = tt;
                // the arg-min step, the one before it, then the kept ones
                for (int j = am_kept + 1; j >= -1; j--) {
                    Taps tp;
                    const float dx = __fsub_rn(fmaf(tj, a.Lx, ox), a.bx), dy = __fsub_rn(fmaf(tj, a.Ly, oy), a.by),
                                dz = __fsub_rn(fmaf(tj, a.Lz, oz), a.bz);
                    sample<true, true>(a, dx, dy, dz, &tp);
#pragma unroll
                    for (int c = 0; c < 8; c++) atomicAdd(dsdf + tp.idx[c], hbar * tp.w[c]);
                    const float qbx = hbar * tp.grad[0], qby = hbar * tp.grad[1], qbz = hbar * tp.grad[2];
                    tbar += qbx * a.Lx + qby * a.Ly + qbz * a.Lz;
                    lbx = fmaf(qbx, tj, lbx);
                    lby = fmaf(qby, tj, lby);
                    lbz = fmaf(qbz, tj, lbz);
                    if (j == am_kept + 1) {
                        if (am == 0) break;
                        tj = am_tp;
                        hbar = pbar;
                        if (p < a.smax) hbar += tbar;
                    } else {
                        if (j == 0) break;
                        const float e = ts[j - 1];
                        tj = fabsf(e);
                        hbar = signbit(e) ? 0.f : tbar;
                    }
                }
            }
        }
    }
    // block reduction of dLoss/dL, then the map through L = v / |v|
    __shared__ float red[3][4];
    for (int off = 16; off >= 1; off >>= 1) {
        lbx += __shfl_xor_sync(0xFFFFFFFFu, lbx, off);
        lby += __shfl_xor_sync(0xFFFFFFFFu, lby, off);
        lbz += __shfl_xor_sync(0xFFFFFFFFu, lbz, off);
    }
    const int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) {
        red[0][w] = lbx;
        red[1][w] = lby;
        red[2][w] = lbz;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        float sx = 0.f, sy = 0.f, sz = 0.f;
        for (int k = 0; k < (int)(blockDim.x >> 5); k++) {
            sx += red[0][k];
            sy += red[1][k];
            sz += red[2][k];
        }
        if (sx != 0.f || sy != 0.f || sz != 0.f) {
            const float dl = sx * a.Lx + sy * a.Ly + sz * a.Lz;
            atomicAdd(dlight + 0, (sx - dl * a.Lx) * inv_norm);
            atomicAdd(dlight + 1, (sy - dl * a.Ly) * inv_norm);
            atomicAdd(dlight + 2, (sz - dl * a.Lz) * inv_norm);
        }
    }
}

// Temporal anti-aliasing of a visibility image (Sec. 2.3 steadies the
// jitter noise with TAA), static camera: the history is clamped to the
// current frame's 3x3 neighbourhood range (clamped at the border) and
// blended toward the current value in place, h = hc + blend (cur - hc).
__global__ void __launch_bounds__(256) k_taa(const float* cur, float* __restrict__ hist, int w,
                                             int h, float blend) {
    chain_begin();
    const int x = blockIdx.x * 32 + threadIdx.x;
    const int y = blockIdx.y * 8 + threadIdx.y;
    if (x >= w || y >= h) return;
    float mn = CUDART_INF_F, mx = -CUDART_INF_F;
#pragma unroll
    for (int dy = -1; dy <= 1; dy++) {
        const int yy = min(max(y + dy, 0), h - 1);
#pragma unroll
        for (int dx = -1; dx <= 1; dx++) {
            const int xx = min(max(x + dx, 0), w - 1);
            const float v = cur[(size_t)yy * w + xx];
            mn = fminf(mn, v);
            mx = fmaxf(mx, v);
        }
    }
    const size_t i = (size_t)y * w + x;
    const float c = cur[i];
    const float hc = fminf(fmaxf(hist[i], mn), mx);
    hist[i] = fmaf(blend, __fsub_rn(c, hc), hc);
}

ShadowArgs make_args(rtsdf_ctx* c, const float* sdf, const float* pos, const float* nrm, int64_t npix,
                     const float L[3], float k, int steps, float smax, float eps) {
    ShadowArgs a;
    a.sdf = sdf ? sdf : c->fine;
    a.n = c->nf;
    a.bx = c->cfg.bmin[0];
    a.by = c->cfg.bmin[1];
    a.bz = c->cfg.bmin[2];
    a.ext = c->cfg.extent;
    a.inv_h = (float)c->nf / c->cfg.extent;
    a.pos = pos;
    a.nrm = nrm;
    a.npix = npix;
    a.Lx = L[0];
    a.Ly = L[1];
    a.Lz = L[2];
    a.k = k;
    a.smax = smax;
    a.eps = eps;
    a.steps = steps;
    a.jitter = 0.f;
    a.frame = 0;
    a.key0 = (uint32_t)c->cfg.seed;
    a.key1 = (uint32_t)(c->cfg.seed >> 32);
    return a;
}

// Thin-surface fallback (Sec. 3: the march can step through a surface
// thinner than its epsilon and leave a hole in the umbra; the paper would
// shadow-map such regions).  Exact occlusion of the ray from the march's
// origin fmaf(n, 2 eps, p) along L: a BVH traversal that stops at the first
// hit (any hit decides), with the tracer's box and ray/triangle tests.  A
// blocked point gets visibility 0; the others keep the march's value.
// TEX: node fetches split between the load and texture pipes, as in the
// tracer.
constexpr int SHADOW_STACK = 24;   // entries in shared memory
struct ShadowStack : dev::Stack<SHADOW_STACK> {
    float3 o, d;   // the ray
    __device__ __forceinline__ float3 origin() const { return o; }
    __device__ __forceinline__ float3 direction() const { return d; }
    __device__ __forceinline__ bool below(float, int&) { return false; }   // nothing lies below the stack
};
template <bool TEX>
__global__ void __launch_bounds__(dev::TRACE_THREADS) k_shadow_exact(dev::TraceArgs t, const float* __restrict__ pos,
                                                                     const float* __restrict__ nrm, long long npix,
                                                                     float Lx, float Ly, float Lz, float two_eps,
                                                                     float* vis, uint8_t* blocked) {
    __shared__ int2 s_stack[SHADOW_STACK][dev::TRACE_THREADS];
    int2 deep[TRACE_STACK - SHADOW_STACK];
    ShadowStack stk;
    stk.e = &s_stack[0][threadIdx.x];
    stk.deep = deep;
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= npix) return;                      // no barrier below
    dev::Ray r;
    stk.o = make_float3(fmaf(nrm[3 * i], two_eps, pos[3 * i]), fmaf(nrm[3 * i + 1], two_eps, pos[3 * i + 1]),
                        fmaf(nrm[3 * i + 2], two_eps, pos[3 * i + 2]));
    stk.d = make_float3(Lx, Ly, Lz);
    r.id = make_float3(dev::safe_inv(Lx), dev::safe_inv(Ly), dev::safe_inv(Lz));
    r.oid = make_float3(stk.o.x * r.id.x, stk.o.y * r.id.y, stk.o.z * r.id.z);
    r.bt = CUDART_INF_F;
    r.bidx = 0x7FFFFFFF;
    r.bfront = false;
    r.node = t.nt > 1 ? 0 : WIDE_EMPTY;
    r.leaf = t.nt == 1 ? 0 : WIDE_EMPTY;
    r.sp = 0;
    r.steps = 0;
    uint32_t nv = 0, ntest = 0;
    // every step enters a node or tests a leaf (bounded by the step guard);
    // the loop ends at the first hit or when nothing is left
    while (r.bidx == 0x7FFFFFFF && !(r.node == WIDE_EMPTY && r.leaf == WIDE_EMPTY)) {
        if (dev::node_step<false, TEX>(t, r, stk, nv)) dev::advance(r, stk);
        if (r.leaf != WIDE_EMPTY && dev::leaf_step<false>(t, r, stk, nv, ntest)) dev::advance(r, stk);
        dev::step_guard(t, r);
    }
    const bool b = r.bidx != 0x7FFFFFFF;
    if (blocked) blocked[i] = (uint8_t)b;
    if (b && vis) vis[i] = 0.f;
}

}  // namespace

cudaError_t launch_shadow(rtsdf_ctx* c, const float* sdf, const float* pos, const float* nrm, int64_t npix,
                          const float L[3], float k, int steps, float smax, float eps, float jitter, int frame,
                          float* vis) {
    if (npix == 0) return cudaSuccess;
    ShadowArgs a = make_args(c, sdf, pos, nrm, npix, L, k, steps, smax, eps);
    a.jitter = jitter;
    a.frame = (uint32_t)frame;
    launch_chain(c, k_shadow, (unsigned)((npix + SHADOW_THREADS - 1) / SHADOW_THREADS), SHADOW_THREADS, 0, a, vis);
    return cudaGetLastError();
}

cudaError_t launch_shadow_bwd(rtsdf_ctx* c, const float* sdf, const float* pos, const float* nrm, int64_t npix,
                              const float L[3], float inv_norm, float k, int steps, float smax, float eps,
                              const float* dvis, float* dsdf, float* dlight) {
    if (npix == 0) return cudaSuccess;
    ShadowArgs a = make_args(c, sdf, pos, nrm, npix, L, k, steps, smax, eps);
    RTSDF_LAUNCH(c, k_shadow_bwd, (unsigned)((npix + 127) / 128), 128, 0, a, dvis, dsdf, dlight, inv_norm);
    return cudaGetLastError();
}

cudaError_t launch_taa(rtsdf_ctx* c, const float* cur, float* hist, int w, int h, float blend) {
    if (w == 0 || h == 0) return cudaSuccess;
    dim3 block(32, 8, 1), grid((unsigned)((w + 31) / 32), (unsigned)((h + 7) / 8), 1);
    launch_chain(c, k_taa, grid, block, 0, cur, hist, w, h, blend);
    return cudaGetLastError();
}

cudaError_t launch_shadow_exact(rtsdf_ctx* c, const float* pos, const float* nrm, int64_t npix, const float L[3],
                                float eps, float* vis, uint8_t* blocked) {
    if (npix == 0) return cudaSuccess;
    dev::TraceArgs t;
    memset(&t, 0, sizeof(t));
    t.wide = c->bvh.wide;
    t.wtex = texture_fetch_on() ? c->bvh.wtex : 0;
    t.tri = c->bvh.tri;
    t.nt = c->bvh.nt;
    t.err = c->d_err;
    const unsigned g = (unsigned)((npix + dev::TRACE_THREADS - 1) / dev::TRACE_THREADS);
    if (t.wtex)
        RTSDF_LAUNCH(c, k_shadow_exact<true>, g, dev::TRACE_THREADS, 0, t, pos, nrm, (long long)npix, L[0], L[1],
                     L[2], 2.f * eps, vis, blocked);
    else
        RTSDF_LAUNCH(c, k_shadow_exact<false>, g, dev::TRACE_THREADS, 0, t, pos, nrm, (long long)npix, L[0], L[1],
                     L[2], 2.f * eps, vis, blocked);
    return cudaGetLastError();
}

}  // namespace rtsdf
