// The Sec. 2.2 tracer's warp loop: every warp takes a unit of work (the rays
// of a few neighbouring texels), builds one front of the BVH for it, and
// traces the unit's rays from that front.  Shared by the per-scene tracer
// (trace.cu) and the batched one (batch.cu).
//
// All rays of a unit start within one or two coarse voxels, so the nodes
// around that place are entered by nearly all of them: from the root, half
// of a ray's node visits are to boxes that contain its origin, and most of
// the others to the large boxes near the root.  Those tests are taken out of
// the divergent traversal.  The front is a cut through the tree of at most
// FRONT_MAX nodes and leaves, opened where many of the unit's rays would
// enter (boxes over the unit's place first, then by the solid angle under
// which the unit sees the box).  Its boxes are tested for 32 rays at a time
// in a loop that is uniform over the warp (every lane tests the same box,
// from shared memory), and a ray keeps the boxes it meets as a 64-bit mask.
// The entries are sorted by their distance from the unit, so a ray's
// traversal takes them from the lowest bit, and ends at the first entry that
// lies farther away than its best hit.  A leaf found twice or in another
// order changes nothing: every triangle whose padded box the ray meets
// before its closest hit is tested, and equal distances go to the smaller
// index.
//
// Measured on the frame of 1M triangles (256^3 -> 512^3, 64 rays): 8.7 node
// visits a ray instead of 18.8, trace 357.8 instead of 375 ms; on a room of
// 100k (128^3 -> 256^3): 6.2 instead of 20.4, 138 instead of 170-192 ms; with
// rays that stop at the accumulated distance: 0.2 instead of 4.6, 2.3 instead
// of 2.9 ms (5.7M texels' worth of 32 rays, 75^3).  The visits that remain
// are the dear ones, to nodes that few other rays share: 7 resident blocks
// instead of 8 cost 7 %, so latency binds (72 % of the issue slots used),
// and what a front may cost in registers and shared memory is bounded by
// that.  A fifth of the time goes into making rays and testing the front.
// Tried: rays made in a called function (5 % slower: registers saved
// around the call), one stack entry a step instead of a loop (the same), runs
// of neighbouring units for the warps of an SM (L1 hits 27 instead of 11 %,
// the same time), fronts of 32 (3 % faster on the 1M frame, 14 % slower in
// the room).
#pragma once

#include "trace_dev.cuh"

namespace rtsdf {
namespace dev {

constexpr int FRONT_MAX = 64;        // entries of a front (one bit each)
constexpr int FRONT_ROUNDS = 32;     // rounds of opening nodes (a bound)
constexpr float FRONT_STEP = 0.4f;   // each time no node is left to open, the bar is lowered by this
constexpr float FRONT_LAST = 0.3f;   // share of the unit's rays below which a node stays closed
constexpr int UNIT_TEXELS = 32;      // texels of a unit, at most
constexpr int UNIT_RAYS = 512;       // rays of a unit, at most (but one texel's always)
constexpr int UNITS_PER_WARP = 2;    // units are made smaller until every warp gets this many (a front costs
                                     // as much as some 30 rays: trace of a tiny frame 147 us with 8, 123 with 2)
constexpr int FRONT_STACK = 8;       // stack entries in shared memory below a front

// One warp's shared state.
struct WarpTrace {
    // the front of the unit whose rays are being made
    union {
        struct {                     // while it is opened, by entry:
            float4 box0[FRONT_MAX];  // lo xyz, hi x
            float2 box1[FRONT_MAX];  // hi yz
        };
        float4 pair[FRONT_MAX / 2][3];   // then, by two entries: centre x x y y | z z, half extent x x | y y z z
    };
    // two units' entries (rays of the previous unit may still be under way):
    // (node or ~leaf, distance from the unit as float bits)
    int2 ent[2][FRONT_MAX];
    // rays made and not yet taken by a lane
    float dx[32], dy[32], dz[32];
    uint32_t mlo[32], mhi[32];
    uint32_t pack[32];               // texel x | y << 9 | z << 18 | texel of the unit << 27
    // per texel of the two units: smallest hit distance (or nearest-face key), hit counts
    uint32_t tmin[2][UNIT_TEXELS], tcnt[2][UNIT_TEXELS];
    unsigned long long g0;           // current unit: its first ray within its scene
    unsigned long long cnext, cend;  // rays fetched from the frame's counter and not yet in a unit
    // the warp's place in its work (uniform, read at refills only: kept out of
    // the registers of the traversal loop)
    uint32_t len, gi;                // rays of the current unit, rays made
    int buf, nfront;                 // its buffer, entries of its front
    int have, head;                  // rays waiting, position of the first
    int more;                        // units may be left
    uint32_t slot0[2], ntex[2];      // the units' texel slots
    int scene[2];
    uint8_t open[32];                // entries opened in a round
};

// A front's part of the traversal stack: the entries that the ray meets and
// has not visited, nearest first.
struct FrontStack : Stack<FRONT_STACK> {
    const int2* ent;
    uint32_t mlo, mhi;
    float* od;    // origin and direction, [6][thread] in shared memory: only leaf tests read them
    __device__ __forceinline__ float3 origin() const {
        return make_float3(od[0], od[TRACE_THREADS], od[2 * TRACE_THREADS]);
    }
    __device__ __forceinline__ float3 direction() const {
        return make_float3(od[3 * TRACE_THREADS], od[4 * TRACE_THREADS], od[5 * TRACE_THREADS]);
    }
    // the next entry, when the stack is empty
    __device__ __forceinline__ bool below(float bt, int& cand) {
        int i;
        if (mlo) {
            i = __ffs((int)mlo) - 1;
            mlo &= mlo - 1u;
        } else if (mhi) {
            i = 31 + __ffs((int)mhi);
            mhi &= mhi - 1u;
        } else {
            return false;
        }
        const int2 e = ent[i];
        if (__int_as_float(e.y) > bt) {   // and so are all that follow
            mlo = mhi = 0u;
            return false;
        }
        cand = e.x;
        return true;
    }
};

// Packed fp32 (sm_100 and later): two fused multiply-adds, each rounded as
// the scalar one.
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pair2(float a) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(a));
    return r;
}
__device__ __forceinline__ float2 split2(f32x2 a) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a));
    return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

__device__ __forceinline__ void texel_coords(const TraceArgs& a, uint32_t slot, uint32_t& jx, uint32_t& jy,
                                             uint32_t& jz) {
    const uint32_t parent = a.masked[slot >> 3];
    const uint32_t ch = slot & 7u;
    const uint32_t nc = (uint32_t)a.nc;
    const uint32_t pq = __umulhi(parent, a.nc_mag), pz = __umulhi(pq, a.nc_mag);
    jx = 2 * (parent - pq * nc) + (ch & 1);
    jy = 2 * (pq - pz * nc) + ((ch >> 1) & 1);
    jz = 2 * pz + (ch >> 2);
}

__device__ __forceinline__ float3 texel_centre(const TraceArgs& a, uint32_t jx, uint32_t jy, uint32_t jz) {
    return make_float3(__fadd_rn(a.bx, __fmul_rn(__fadd_rn((float)jx, 0.5f), a.hf)),
                       __fadd_rn(a.by, __fmul_rn(__fadd_rn((float)jy, 0.5f), a.hf)),
                       __fadd_rn(a.bz, __fmul_rn(__fadd_rn((float)jz, 0.5f), a.hf)));
}

// Distance of a box from the cube [ulo, uhi] (0: they meet).
__device__ __forceinline__ float box_distance(float3 ulo, float3 uhi, const float lo[3], const float hi[3]) {
    const float x = fmaxf(fmaxf(lo[0] - uhi.x, ulo.x - hi[0]), 0.f);
    const float y = fmaxf(fmaxf(lo[1] - uhi.y, ulo.y - hi[1]), 0.f);
    const float z = fmaxf(fmaxf(lo[2] - uhi.z, ulo.z - hi[2]), 0.f);
    return sqrtf(fmaf(x, x, fmaf(y, y, z * z)));
}

// Share of the unit's rays that meet a box: 1 where it meets the unit's
// cube, else its projected area over the sphere through a point between its
// nearest point and its centre.
__device__ __forceinline__ float box_share(float3 ulo, float3 uhi, const float lo[3], const float hi[3]) {
    if (box_distance(ulo, uhi, lo, hi) == 0.f) return 1.f;
    const float c[3] = {0.5f * (ulo.x + uhi.x), 0.5f * (ulo.y + uhi.y), 0.5f * (ulo.z + uhi.z)};
    float d[3], e[3];
#pragma unroll
    for (int k = 0; k < 3; k++) {
        d[k] = 0.5f * (fminf(fmaxf(c[k], lo[k]), hi[k]) + 0.5f * (lo[k] + hi[k])) - c[k];
        e[k] = hi[k] - lo[k];
    }
    const float d2 = fmaxf(fmaf(d[0], d[0], fmaf(d[1], d[1], d[2] * d[2])), 1e-30f);
    const float area = fabsf(d[0]) * e[1] * e[2] + fabsf(d[1]) * e[0] * e[2] + fabsf(d[2]) * e[0] * e[1];
    return fminf(0.5f, area * rsqrtf(d2) / (12.566371f * d2));
}

// Opens the tree from `root` (a node, or ~leaf) for rays that start in the
// cube [ulo, uhi] and look no farther than `far`, and leaves the front (at most
// `most` entries) sorted
// by distance in w.box0 / box1 and w.ent[buf].  Returns its size (the boxes behind it, up to the next
// multiple of 8, are met by nothing).  All 32 lanes call.
__device__ __forceinline__ int build_front(const WNode* __restrict__ wide, int root, float3 ulo, float3 uhi,
                                                  float far, int most, WarpTrace& w, int buf, unsigned lane, unsigned lt) {
    constexpr unsigned FULL = 0xFFFFFFFFu;
    int2* ent = w.ent[buf];              // while opening: (node or ~leaf, share of the rays)
    if (lane == 0) {
        ent[0] = make_int2(root, __float_as_int(1.f));
        w.box0[0] = make_float4(-1e18f, -1e18f, -1e18f, 1e18f);
        w.box1[0] = make_float2(1e18f, 1e18f);
    }
    __syncwarp();
    int n = 1;
    float bar = 1.f;
    for (int round = 0; round < FRONT_ROUNDS; round++) {
        bool open[2];
#pragma unroll
        for (int s = 0; s < 2; s++) {
            const int e = (int)lane + 32 * s;
            open[s] = false;
            if (e < n) {
                const int2 v = ent[e];
                open[s] = v.x >= 0 && __int_as_float(v.y) >= bar;
            }
        }
        const unsigned m0 = __ballot_sync(FULL, open[0]), m1 = __ballot_sync(FULL, open[1]);
        const int room = (most - n) / 3;
        if (room <= 0) break;
        const int found = __popc(m0) + __popc(m1);
        if (found == 0) {
            bar *= FRONT_STEP;
            if (bar < FRONT_LAST) break;
            continue;
        }
        const int c = min(found, room);
        const int r0 = __popc(m0 & lt), r1 = __popc(m0) + __popc(m1 & lt);
        if (open[0] && r0 < c) w.open[r0] = (uint8_t)lane;
        if (open[1] && r1 < c) w.open[r1] = (uint8_t)(lane + 32);
        __syncwarp();
        // four lanes per node, one child each; the first child takes the
        // node's place
        for (int b = 0; b < c; b += 8) {
            const int j = b + (int)(lane >> 2), k = (int)(lane & 3);
            int e = 0, id = 0;
            float lo[3], hi[3];
            float share = -1.f;
            if (j < c) {
                e = w.open[j];
                const WNode* nd = wide + ent[e].x;
                const float* row = &nd->lox.x + k;
                lo[0] = __ldg(row); hi[0] = __ldg(row + 4);
                lo[1] = __ldg(row + 8); hi[1] = __ldg(row + 12);
                lo[2] = __ldg(row + 16); hi[2] = __ldg(row + 20);
                id = __ldg(&nd->child.x + k);
                if (box_distance(ulo, uhi, lo, hi) * 0.999f > far) id = WIDE_EMPTY;
                if (id >= 0) share = box_share(ulo, uhi, lo, hi);
            }
            __syncwarp();
            if (j < c) {
                const int at = k == 0 ? e : n + 3 * j + k - 1;
                ent[at] = make_int2(id, __float_as_int(share));
                w.box0[at] = make_float4(lo[0], lo[1], lo[2], hi[0]);
                w.box1[at] = make_float2(hi[1], hi[2]);
            }
            __syncwarp();
        }
        n += 3 * c;
        if (c < found) break;
    }
    // sort by distance: keys are the distance's bits (rounded down a little,
    // so that it bounds every hit in the box from below) with the entry's
    // position in the low bits; empty child slots go last
    uint32_t key[2];
    int id[2];
    float4 b0[2];
    float2 b1[2];
#pragma unroll
    for (int s = 0; s < 2; s++) {
        const int e = (int)lane + 32 * s;
        key[s] = 0xFFFFFFFFu;
        if (e < n && ent[e].x != WIDE_EMPTY) {
            const float4 p = w.box0[e];
            const float2 q = w.box1[e];
            const float lo[3] = {p.x, p.y, p.z}, hi[3] = {p.w, q.x, q.y};
            const float d = box_distance(ulo, uhi, lo, hi) * 0.999f;
            key[s] = (__float_as_uint(d) & ~63u) | (uint32_t)e;
        }
    }
#pragma unroll
    for (int k = 2; k <= 64; k <<= 1)
#pragma unroll
        for (int j = k >> 1; j >= 1; j >>= 1) {
            if (j == 32) {
                const uint32_t a = min(key[0], key[1]), b = max(key[0], key[1]);
                key[0] = a;
                key[1] = b;
            } else {
                const bool low = (lane & (unsigned)j) == 0;
#pragma unroll
                for (int s = 0; s < 2; s++) {
                    const bool up = ((lane + 32u * (unsigned)s) & (unsigned)k) == 0;
                    const uint32_t o = __shfl_xor_sync(FULL, key[s], j);
                    key[s] = low == up ? min(key[s], o) : max(key[s], o);
                }
            }
        }
#pragma unroll
    for (int s = 0; s < 2; s++) {
        const int e = (int)(key[s] & 63u);
        id[s] = ent[e].x;
        b0[s] = w.box0[e];
        b1[s] = w.box1[e];
    }
    __syncwarp();
    int live = 0;
#pragma unroll
    for (int s = 0; s < 2; s++) {
        const int e = (int)lane + 32 * s;
        const bool real = key[s] != 0xFFFFFFFFu;
        live += __popc(__ballot_sync(FULL, real));
        float c[3] = {0.f, 0.f, 0.f}, h[3] = {-CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F};   // met by no ray
        if (real) {
            const float lo[3] = {b0[s].x, b0[s].y, b0[s].z}, hi[3] = {b0[s].w, b1[s].x, b1[s].y};
#pragma unroll
            for (int k = 0; k < 3; k++) {
                c[k] = 0.5f * (lo[k] + hi[k]);
                h[k] = fmaxf(hi[k] - c[k], c[k] - lo[k]) * (1.f + 0x1p-20f);
            }
        }
        float* p = &w.pair[e >> 1][0].x + (e & 1);
#pragma unroll
        for (int k = 0; k < 3; k++) {
            p[2 * k] = c[k];
            p[6 + 2 * k] = h[k];
        }
        ent[e] = make_int2(id[s], (int)(key[s] & ~63u));
    }
    __syncwarp();
    return live;
}

// Makes 32 rays of the current unit (those from gi on): directions, the mask
// of the front's n boxes that each meets; rays that meet one are put in
// w.dx .. w.pack.  Returns their number.  All 32 lanes call.
__device__ __forceinline__ int make_rays(const TraceArgs& a, WarpTrace& w, int buf, int n, uint32_t gi,
                                         unsigned lane, unsigned lt) {
    const uint32_t i = gi + lane;
    const bool valid = i < w.len;
    const unsigned long long g = w.g0 + (valid ? i : w.len - 1u);
    const uint32_t slot = (uint32_t)(g >> a.log2_rays);
    const uint32_t ray = (uint32_t)(g & (unsigned long long)(a.rays - 1));
    uint32_t jx, jy, jz;
    texel_coords(a, slot, jx, jy, jz);
    const uint32_t nf = 2u * (uint32_t)a.nc;
    const float3 o = texel_centre(a, jx, jy, jz);
    const float3 d = sphere_dir(a.key0, a.key1, jx + nf * (jy + nf * jz), a.frame, ray);
    const float3 id = make_float3(safe_inv(d.x), safe_inv(d.y), safe_inv(d.z));
    const float3 oid = make_float3(o.x * id.x, o.y * id.y, o.z * id.z);
    // two boxes at a time with packed fp32: the slab of an axis is centre +-
    // half extent, times the reciprocal direction.  Four boxes a turn: with
    // eight, their loads push the traversal's registers out (1M frame 358 and
    // 377 ms; one box at a time 358, but 6 % slower where most of the time goes
    // into making rays)
    const f32x2 ix = pair2(id.x), iy = pair2(id.y), iz = pair2(id.z);
    const f32x2 ox = pair2(-oid.x), oy = pair2(-oid.y), oz = pair2(-oid.z);
    const f32x2 ax = pair2(fabsf(id.x)), ay = pair2(fabsf(id.y)), az = pair2(fabsf(id.z));
    const f32x2 bx = pair2(-fabsf(id.x)), by = pair2(-fabsf(id.y)), bz = pair2(-fabsf(id.z));
    uint32_t m[2] = {0u, 0u};
#pragma unroll
    for (int s = 0; s < 2; s++) {
        for (int b = 32 * s; b < min(n, 32 * s + 32); b += 8) {
            uint32_t part = 0u;
#pragma unroll 2
            for (int k = 0; k < 4; k++) {
                const f32x2* p = reinterpret_cast<const f32x2*>(w.pair[(b >> 1) + k]);
                const ulonglong2 p0 = *reinterpret_cast<const ulonglong2*>(p);
                const ulonglong2 p1 = *reinterpret_cast<const ulonglong2*>(p + 2);
                const ulonglong2 p2 = *reinterpret_cast<const ulonglong2*>(p + 4);
                const f32x2 cx = fma2(p0.x, ix, ox), cy = fma2(p0.y, iy, oy), cz = fma2(p1.x, iz, oz);
                const float2 lx = split2(fma2(p1.y, bx, cx)), hx = split2(fma2(p1.y, ax, cx));
                const float2 ly = split2(fma2(p2.x, by, cy)), hy = split2(fma2(p2.x, ay, cy));
                const float2 lz = split2(fma2(p2.y, bz, cz)), hz = split2(fma2(p2.y, az, cz));
                if (fmax3(lx.x, ly.x, fmaxf(lz.x, 0.f)) <= fmin3(hx.x, hy.x, hz.x)) part |= 1u << (2 * k);
                if (fmax3(lx.y, ly.y, fmaxf(lz.y, 0.f)) <= fmin3(hx.y, hy.y, hz.y)) part |= 2u << (2 * k);
            }
            m[s] |= part << (b & 31);
        }
        if (n < 32 * s + 32) m[s] &= n > 32 * s ? (1u << (n - 32 * s)) - 1u : 0u;
    }
    const bool ok = valid && (m[0] | m[1]) != 0u;
    const unsigned bal = __ballot_sync(0xFFFFFFFFu, ok);
    if (ok) {
        const int at = __popc(bal & lt);
        w.dx[at] = d.x;
        w.dy[at] = d.y;
        w.dz[at] = d.z;
        w.mlo[at] = m[0];
        w.mhi[at] = m[1];
        w.pack[at] = jx | (jy << 9) | (jz << 18) | ((slot - w.slot0[buf]) << 27);
    }
    __syncwarp();
    return __popc(bal);
}

// Applies Eq. 1 to a unit's texels (a unit has all rays of its texels, so no
// other warp has a part in them) and frees its buffer.  All 32 lanes call; no
// ray of the unit is under way.  Through scratch of 8 bytes a fine texel and a
// launch after the tracer's, the frames took more: 24 batched scenes 58.9 ms
// against 57.1, a room of 100k triangles 114.2 against 113.8, the rigid refit
// frame 5.438 against 5.417.
__device__ __forceinline__ void flush_unit(const TraceArgs& a, WarpTrace& w, int buf, unsigned lane) {
    if (lane < w.ntex[buf]) {
        finalize_slot(a, w.slot0[buf] + lane, w.tmin[buf][lane], w.tcnt[buf][lane]);
    }
    __syncwarp();
    if (lane == 0) w.ntex[buf] = 0;
    __syncwarp();
}

// Rays of a unit: a power of two times the rays of a texel, at most
// UNIT_TEXELS texels and `most` rays (one texel's always), and small enough
// that every warp gets several units.
__device__ __forceinline__ uint32_t unit_rays(unsigned long long total, uint32_t rays, uint32_t most) {
    uint32_t u = rays < 32u ? 32u : rays;
    most = min(most, min((uint32_t)UNIT_RAYS, (uint32_t)UNIT_TEXELS * rays));
    const unsigned long long units = (unsigned long long)gridDim.x * (TRACE_THREADS / 32) * UNITS_PER_WARP;
    while (2u * u <= most && 2ull * u * units <= total) u *= 2u;
    return u;
}

// Traversal in two phases.  With one triangle per leaf, a warp in which
// every lane takes either a node step or a leaf step would pay both paths on
// almost every iteration.  So a lane that reaches a leaf parks it (one per
// lane) and keeps entering internal nodes; the warp runs the leaf phase only
// when enough lanes hold a parked leaf or some cannot continue.  The order of
// triangle tests does not change the closest hit (every triangle whose box
// the ray meets is tested unless its entry distance exceeds the best hit).
// Node steps per phase decision: 3 (1M triangles, 256^3: 364.8 ms with 2,
// 357.8 with 3, 359.4 with 4; 100k, 64^3: 25.1, 25.5, 26.3).
constexpr int NODE_STEPS = 3;

// One warp iteration for every lane (active or not: call it convergently).
// COUNT: visits / tests count this lane's node visits and triangle tests,
// leaf_slots the leaf rounds the warp ran (one or two per leaf phase).
// Returns true for a lane whose ray finished.
template <bool COUNT, bool TEX, class A>
__device__ __forceinline__ bool warp_step(const A& a, Ray& r, FrontStack& stack, bool active, int leaf_min,
                                          uint32_t& visits, uint32_t& tests, uint32_t& leaf_slots) {
    // the loops stay loops: the traversal's code has to fit the instruction
    // caches, which the warps of an SM pass through at different places
    if (active) {
#pragma unroll 1
        for (int i = 0; i < NODE_STEPS; i++)
            if (node_step<COUNT, TEX>(a, r, stack, visits)) advance(r, stack);
    }
    const bool parked = active && r.leaf != WIDE_EMPTY;
    const unsigned pm = __ballot_sync(0xFFFFFFFFu, parked);
    const unsigned im = __ballot_sync(0xFFFFFFFFu, active && r.node >= 0);
    // (pm & ~im: lanes that cannot go on before their leaf)
    if (pm && (__popc(pm) >= leaf_min || 2 * __popc(pm & ~im) >= leaf_min || im == 0)) {
        // a lane whose next node was a leaf waiting behind the tested one has
        // parked it then and tests it in a second round of this phase (any
        // lane: measured slightly faster than waiting for several)
        bool test = parked;
#pragma unroll 1
        for (int i = 0; i < 2; i++) {
            if (COUNT) leaf_slots++;
            if (test) {
                if (leaf_step<COUNT>(a, r, stack, visits, tests)) advance(r, stack);
                test = r.leaf != WIDE_EMPTY;
            }
            if (__ballot_sync(0xFFFFFFFFu, test) == 0) break;
        }
    }
    if (active) step_guard(a, r);
    return active && r.node == WIDE_EMPTY && r.leaf == WIDE_EMPTY;
}

// Block-wide shared state of the tracer.
struct BlockTrace {
    WarpTrace warp[TRACE_THREADS / 32];
    int2 stack[FRONT_STACK][TRACE_THREADS];
    float od[6][TRACE_THREADS];
};

__device__ __forceinline__ unsigned lanes_below() {
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// Gives idle lanes new rays: from those that wait, else 32 more of the
// current unit, else of the next unit (whose front is built then).  Returns
// true when nothing is left for an idle lane, now or later.
template <bool COUNT, class Src, class A>
__device__ __forceinline__ bool refill(Src& src, const A& bvh, uint32_t unit, WarpTrace& w, Ray& r, FrontStack& stk,
                                       uint32_t& tex, bool& active, uint32_t& n_rays) {
    constexpr unsigned FULL = 0xFFFFFFFFu;
    const unsigned lane = threadIdx.x & 31, lt = lanes_below();
    // commit the rays that finished since the last refill.  Vote: smallest
    // distance and hit counts; nearest face: the smallest (distance, face)
    // key, ties to the front face
    if (!active && r.bidx != 0x7FFFFFFF) {
        const int b = (int)(tex >> 5), j = (int)(tex & 31u);
        const uint32_t tb = __float_as_uint(r.bt) & 0x7FFFFFFFu;
        if (src.args(w.scene[b]).nearest) {
            atomicMin(&w.tmin[b][j], (tb << 1) | (r.bfront ? 0u : 1u));
        } else {
            atomicMin(&w.tmin[b][j], tb);
            atomicAdd(&w.tcnt[b][j], r.bfront ? 1u : 0x10000u);
        }
        r.bidx = 0x7FFFFFFF;
    }
    __syncwarp();
    unsigned idle = __ballot_sync(FULL, !active);
    while (idle) {
        const int have = w.have;
        if (have == 0) {
            if (w.gi >= w.len) {
                if (!w.more) return true;
                // the next unit takes the other buffer, once no ray of
                // the unit that had it is under way
                const int nb = w.buf ^ 1;
                if (__ballot_sync(FULL, active && (int)(tex >> 5) == nb)) return false;
                if (w.ntex[nb]) flush_unit(src.args(w.scene[nb]), w, nb, lane);
                int scene = 0;
                if (!src.next(w, unit, lane, scene)) {
                    if (lane == 0) {
                        w.more = 0;
                        w.gi = w.len;
                    }
                    __syncwarp();
                    return true;
                }
                const TraceArgs& a = src.args(scene);
                const uint32_t slot0 = (uint32_t)(w.g0 >> a.log2_rays), ntex = w.len >> a.log2_rays;
                uint32_t jx, jy, jz;
                texel_coords(a, slot0 + min(lane, ntex - 1u), jx, jy, jz);
                w.tmin[nb][lane] = ray_min_none(a.nearest != 0);
                w.tcnt[nb][lane] = 0u;
                const float3 ulo = texel_centre(a, __reduce_min_sync(FULL, jx), __reduce_min_sync(FULL, jy),
                                                __reduce_min_sync(FULL, jz));
                const float3 uhi = texel_centre(a, __reduce_max_sync(FULL, jx), __reduce_max_sync(FULL, jy),
                                                __reduce_max_sync(FULL, jz));
                // nearest-face variant: no ray looks beyond its texel's accumulated distance
                float far = CUDART_INF_F;
                if (a.nearest) {
                    const uint32_t nf = 2u * (uint32_t)a.nc;
                    // (a faded distance can be negative: such a texel's rays accept no hit)
                    const float u = fmaxf(a.accum[jx + nf * (jy + nf * jz)], 0.f);
                    far = __uint_as_float(__reduce_max_sync(FULL, __float_as_uint(u)));
                }
                // a front costs the same for few rays as for many: smaller for
                // few (room, 1 ray a texel: 4.53 ms with 22 or 64 entries, 4.41
                // with 40; 4 rays: 6.1 with 64, 5.7 with 40)
                const int most = w.len >= 256u ? FRONT_MAX : 40;
                const int root = src.root(scene);
                const int n = root == WIDE_EMPTY ? 0 : build_front(bvh.wide, root, ulo, uhi, far, most, w, nb, lane, lt);
                if (lane == 0) {
                    w.scene[nb] = scene;
                    w.slot0[nb] = slot0;
                    w.ntex[nb] = ntex;
                    w.nfront = n;
                    w.buf = nb;
                    w.gi = 0;
                }
                __syncwarp();
            }
            const uint32_t gi = w.gi;
            if (COUNT) n_rays += lane < min(32u, w.len - gi);
            const int made = make_rays(src.args(w.scene[w.buf]), w, w.buf, w.nfront, gi, lane, lt);
            if (lane == 0) {
                w.have = made;
                w.head = 0;
                w.gi = gi + 32u;
            }
            __syncwarp();
            continue;
        }
        const int take = min(have, __popc(idle)), head = w.head, buf = w.buf;
        if (!active) {
            const int rank = __popc(idle & lt);
            if (rank < take) {
                const int at = head + rank;
                const TraceArgs& a = src.args(w.scene[buf]);
                const uint32_t pk = w.pack[at];
                const uint32_t jx = pk & 511u, jy = (pk >> 9) & 511u, jz = (pk >> 18) & 511u;
                const float3 o = texel_centre(a, jx, jy, jz);
                const float3 d = make_float3(w.dx[at], w.dy[at], w.dz[at]);
                stk.od[0] = o.x;
                stk.od[TRACE_THREADS] = o.y;
                stk.od[2 * TRACE_THREADS] = o.z;
                stk.od[3 * TRACE_THREADS] = d.x;
                stk.od[4 * TRACE_THREADS] = d.y;
                stk.od[5 * TRACE_THREADS] = d.z;
                r.id = make_float3(safe_inv(d.x), safe_inv(d.y), safe_inv(d.z));
                r.oid = make_float3(o.x * r.id.x, o.y * r.id.y, o.z * r.id.z);
                // nearest-face variant: no hit beyond the texel's accumulated
                // distance can change its result, so the ray starts with that
                // distance as its best hit (hits at exactly that distance
                // still count: bidx is unset)
                const uint32_t nf = 2u * (uint32_t)a.nc;
                r.bt = a.nearest ? a.accum[jx + nf * (jy + nf * jz)] : CUDART_INF_F;
                r.bidx = 0x7FFFFFFF;
                r.bfront = false;
                r.node = r.leaf = WIDE_EMPTY;
                r.sp = 0;
                r.steps = 0;
                tex = (pk >> 27) | ((uint32_t)buf << 5);
                stk.mlo = w.mlo[at];
                stk.mhi = w.mhi[at];
                stk.ent = w.ent[buf];
                advance(r, stk);
                active = true;
            }
        }
        __syncwarp();
        if (lane == 0) {
            w.head = head + take;
            w.have = have - take;
        }
        __syncwarp();
        idle = __ballot_sync(FULL, !active);
    }
    return false;
}

// Traces all rays of the frame (all lanes of all warps call, once).  Src
// gives the units: next(w, unit, lane, scene) puts up to `unit` rays of one
// scene into w.g0 / w.len and that scene into `scene` (false: none left); args(scene)
// its tracer fields; root(scene) the node or ~leaf its rays start from
// (WIDE_EMPTY: an empty scene).  A: the BVH fields of the traversal.
template <bool COUNT, bool TEX, class Src, class A>
__device__ __forceinline__ void trace_units(Src& src, const A& bvh, uint32_t unit, int refill_min, int leaf_min,
                                            BlockTrace& s, TraceCounters* counters) {
    constexpr unsigned FULL = 0xFFFFFFFFu;
    WarpTrace& w = s.warp[threadIdx.x >> 5];
    int2 deep[TRACE_STACK - FRONT_STACK];
    FrontStack stk;
    stk.e = &s.stack[0][threadIdx.x];
    stk.deep = deep;
    stk.ent = w.ent[0];
    stk.mlo = stk.mhi = 0u;
    stk.od = &s.od[0][threadIdx.x];
    uint32_t n_visits = 0, n_tests = 0, n_rays = 0;
    uint32_t n_slots = 0, n_leaf_slots = 0;
    if ((threadIdx.x & 31) == 0) {
        w.cnext = w.cend = 0;
        w.ntex[0] = w.ntex[1] = 0;
        w.len = w.gi = 0;
        w.buf = 1;
        w.nfront = w.have = w.head = 0;
        w.more = 1;
    }
    __syncwarp();
    Ray r;
    r.bidx = 0x7FFFFFFF;
    r.node = r.leaf = WIDE_EMPTY;
    r.sp = 0;
    bool active = false;
    uint32_t tex = 0;                 // texel of the unit | unit's buffer << 5
    for (;;) {
        const bool drained = refill<COUNT>(src, bvh, unit, w, r, stk, tex, active, n_rays);
        if (drained && __ballot_sync(FULL, active) == 0) break;
        // trace until enough lanes are idle to be worth a refill
        for (;;) {
            const bool done = warp_step<COUNT, TEX>(bvh, r, stk, active, leaf_min, n_visits, n_tests, n_leaf_slots);
            if (COUNT) n_slots += NODE_STEPS;   // lane slots of the node steps
            if (done) active = false;
            const unsigned act = __ballot_sync(FULL, active);
            if (act == 0) break;
            if (!drained && (32 - __popc(act)) >= refill_min) break;
        }
    }
    __syncwarp();
    const unsigned lane = threadIdx.x & 31;
    for (int b = 0; b < 2; b++)
        if (w.ntex[b]) flush_unit(src.args(w.scene[b]), w, b, lane);
    if (COUNT) {
        // summed over the warp's lanes, the iteration counts become lane slots
        unsigned long long rr = n_rays, v = n_visits, t = n_tests, sl = n_slots, ls = n_leaf_slots;
        for (int off = 16; off >= 1; off >>= 1) {
            rr += __shfl_xor_sync(FULL, rr, off);
            v += __shfl_xor_sync(FULL, v, off);
            t += __shfl_xor_sync(FULL, t, off);
            sl += __shfl_xor_sync(FULL, sl, off);
            ls += __shfl_xor_sync(FULL, ls, off);
        }
        if (lane == 0) {
            atomicAdd(&counters->rays, rr);
            atomicAdd(&counters->visits, v);
            atomicAdd(&counters->tests, t);
            atomicAdd(&counters->slots, sl);
            atomicAdd(&counters->leaf_slots, ls);
        }
    }
}

}  // namespace dev
}  // namespace rtsdf
