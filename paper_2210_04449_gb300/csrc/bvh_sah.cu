// Binned surface-area-heuristic topology for the Sec. 2.2 ray casts (the
// paper leaves the ray-tracing structure open).
//
// Top-down: the triangles of a node (a contiguous range of leaf positions)
// are split where the surface-area heuristic (MacDonald & Booth 1990) is
// lowest, cost = half-area(left box) x left count + half-area(right box) x
// right count, evaluated over 32 bins of the range's centroid bounds per
// axis (binning as in Wald 2007).  Every range is split down to single
// triangles.  Node ids need no allocation: the node whose right child starts
// at leaf position s is node s - 1 (each boundary between neighbouring leaves
// belongs to exactly one node), so the tree has the layout of the Morton
// tree: [nt - 1] nodes, [nt] leaves, any node may be the root.
//
// Three tiers by range size m (blk: 256, or 1024 for large meshes):
//  * m > blk: level-synchronous over chunks of 256 or 1024 positions, the levels'
//    sizes kept on the device so that no level waits for the host.
//    k_sah_split bins a chunk in shared memory and merges into the range's
//    bins with global atomics (and keeps the chunk's histogram); the block
//    that finishes a range picks the split and every chunk's output offset;
//    k_sah_partition scatters stably into the other order buffer.
//  * 32 < m <= blk: one block per range (k_sah_block), boxes in shared
//    memory, the same binned split down to ranges of 32: by the whole block
//    above MID_MAX positions, by a warp per range below;
//  * 2 <= m <= 32: one warp per range, the exact heuristic over every split
//    of the centroids sorted along each axis (bitonic sort in registers).
// Float min/max merges go through an order-preserving map to uint32, so
// every merge is exact and independent of order: the build is
// deterministic, whatever order the atomics land in.
#include <math_constants.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "internal.cuh"

namespace rtsdf {

namespace {

constexpr int NB = 32;                        // bins per axis (one per lane)
constexpr int BW = 7;                         // words per bin: count, lo xyz, hi xyz
constexpr int SAH_BIN_WORDS = 3 * NB * BW;
constexpr int SAH_CH = 1024;                  // chunk size, largest block range
constexpr int SAH_THREADS = 256;
constexpr int SAH_ITEMS = SAH_CH / SAH_THREADS;
constexpr int SAH_WARPS = SAH_THREADS / 32;
constexpr int WARP_MAX = 32;                  // largest range of the exact warp build
// Largest range of the block tier that one warp bins and splits, so that the
// ranges of a level are split side by side and without block barriers (which
// bound the tier: 4.5 of its stalls per issue).  Whole build with 256 against
// the whole block for every range: 2.2k triangles 240 / 249 us, 104k 502 / 517,
// 300k 757 / 836, 1M 1752 / 1949 (with 128 and 1024: between).  Warps that take
// ranges from a list as they come, without rounds, were slower: 520 us at 2.2k.
constexpr int MID_MAX = 256;
constexpr int MID_CAP = 32;                   // disjoint ranges > 32 in 1024: at most 31
constexpr int BLK_STACK = SAH_CH / MID_MAX;   // disjoint ranges > MID_MAX in SAH_CH: at most 3
constexpr int WLIST_CAP = SAH_CH / 2;         // disjoint ranges >= 2 in 1024
constexpr unsigned FULL = 0xFFFFFFFFu;

static_assert(SAH_ITEMS * SAH_THREADS == SAH_CH, "one chunk per block pass");

// Largest range of the block tier.  A block splits its range one node after
// another, so a small mesh, whose few ranges leave most SMs idle, is split
// further by the levels (each of which costs two launches).  Whole build with
// 256 against 1024: 2.2k triangles 240 / 295 us, 104k 502 / 556 (512: 247 and
// 490); 300k 825 / 755, 1M 1940 / 1752.
constexpr int SAH_BLK_SMALL = 256;
constexpr int64_t SAH_SMALL_MESH = 200000;
__host__ __device__ constexpr int blk_of(int64_t n) { return n <= SAH_SMALL_MESH ? SAH_BLK_SMALL : SAH_CH; }
// Positions that a block bins and scatters at a level: 1024, or 256 where those
// would be too few blocks (the bin atomics of a chunk bound its time).  Whole
// build with 256 against 1024: 2.2k triangles 240 / 262 us, 12k 315 / 346, 104k
// 502 / 533, 300k 757 / 800, 1M 1960 / 1752.
constexpr int64_t SAH_SMALL_CHUNKS = 500000;
__host__ __device__ constexpr int chunk_of(int64_t n) { return n <= SAH_SMALL_CHUNKS ? SAH_THREADS : SAH_CH; }

// Device-side counters of a build: block ranges listed, a capacity guard that
// fired, block ranges taken, then (tasks, chunks) of each level of a batch.
constexpr int CT_BLOCKS = 0, CT_BAD = 1, CT_TAKEN = 2, CT_LEVELS = 4;
constexpr int LEVEL_BATCH = 28;               // levels enqueued without a look from the host, at most
constexpr int CT_WORDS = CT_LEVELS + 2 * (LEVEL_BATCH + 1);
static_assert(CT_WORDS <= 64, "counters fit 256 bytes");

// big range (m > blk_of(n)) of one level
struct SahTask {
    int32_t b, e, parent, side;
    int32_t buf, chunk0, nchunk, axis;   // buf: order buffer holding the range
    int32_t split, nl, child[2];         // split: first right bin (-1: median)
    uint32_t cb[6];                      // centroid bounds, ordered uint: lo xyz, hi xyz
    int32_t pad[2];
};
static_assert(sizeof(SahTask) == 80, "task record");

// range for the block tier: [b, e), parent node, side | buf << 1
struct SahRange {
    int32_t b, e, parent, sb;
};

__device__ __forceinline__ uint32_t f2o(float f) {
    const uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float o2f(uint32_t u) {
    return __uint_as_float((u & 0x80000000u) ? (u & 0x7FFFFFFFu) : ~u);
}
__device__ __forceinline__ float cen(float lo, float hi) { return __fmul_rn(0.5f, __fadd_rn(lo, hi)); }
__device__ __forceinline__ float half_area3(const float lo[3], const float hi[3]) {
    const float dx = hi[0] - lo[0], dy = hi[1] - lo[1], dz = hi[2] - lo[2];
    return dx * dy + dy * dz + dz * dx;
}
__device__ __forceinline__ uint32_t bin_init(int i) {
    const int w = i % BW;
    return w == 0 ? 0u : (w < 4 ? 0xFFFFFFFFu : 0u);
}

struct BinMap {
    float lo[3], scale[3];
};
__device__ __forceinline__ BinMap bin_map(const float clo[3], const float chi[3]) {
    BinMap m;
#pragma unroll
    for (int a = 0; a < 3; a++) {
        m.lo[a] = clo[a];
        const float ext = chi[a] - clo[a];
        float s = ext > 0.f ? (float)NB / ext : 0.f;
        if (!(s <= 3.0e38f)) s = 0.f;       // a denormal extent: treat as flat
        m.scale[a] = s;
    }
    return m;
}
__device__ __forceinline__ int bin_of(const BinMap& m, int a, float c) {
    const int k = (int)((c - m.lo[a]) * m.scale[a]);
    return min(max(k, 0), NB - 1);
}

struct Choice {
    float cost;
    int axis, split, nl;   // axis -1: no axis separates the range
};

// Lane l reads bin l of axis a; the split after bin l puts bins 0..l left.
// Ties go to the smaller bin.  All 32 lanes call.
__device__ Choice axis_choose(const uint32_t* bins, int a, int lane) {
    const uint32_t* p = bins + (a * NB + lane) * BW;
    const uint32_t cnt = p[0];
    float plo[3], phi[3], slo[3], shi[3];
#pragma unroll
    for (int k = 0; k < 3; k++) {
        plo[k] = slo[k] = cnt ? o2f(p[1 + k]) : CUDART_INF_F;
        phi[k] = shi[k] = cnt ? o2f(p[4 + k]) : -CUDART_INF_F;
    }
    uint32_t pc = cnt, sc = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t up = __shfl_up_sync(FULL, pc, o), dn = __shfl_down_sync(FULL, sc, o);
#pragma unroll
        for (int k = 0; k < 3; k++) {
            const float ul = __shfl_up_sync(FULL, plo[k], o), uh = __shfl_up_sync(FULL, phi[k], o);
            const float dl = __shfl_down_sync(FULL, slo[k], o), dh = __shfl_down_sync(FULL, shi[k], o);
            if (lane >= o) {
                plo[k] = fminf(plo[k], ul);
                phi[k] = fmaxf(phi[k], uh);
            }
            if (lane + o < 32) {
                slo[k] = fminf(slo[k], dl);
                shi[k] = fmaxf(shi[k], dh);
            }
        }
        if (lane >= o) pc += up;
        if (lane + o < 32) sc += dn;
    }
    // right side of the split after bin `lane`: the suffix from lane + 1
    const uint32_t rc = __shfl_down_sync(FULL, sc, 1);
    float rlo[3], rhi[3];
#pragma unroll
    for (int k = 0; k < 3; k++) {
        rlo[k] = __shfl_down_sync(FULL, slo[k], 1);
        rhi[k] = __shfl_down_sync(FULL, shi[k], 1);
    }
    float cost = CUDART_INF_F;
    if (lane < NB - 1 && pc > 0 && rc > 0)
        cost = half_area3(plo, phi) * (float)pc + half_area3(rlo, rhi) * (float)rc;
    // a cost that is not a number (a vertex moved out of all range) is infinite:
    // past it, the lanes would come to different splits
    float bc = fminf(cost, CUDART_INF_F);
    int bl = lane;
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) {
        const float c2 = __shfl_xor_sync(FULL, bc, o);
        const int l2 = __shfl_xor_sync(FULL, bl, o);
        if (c2 < bc || (c2 == bc && l2 < bl)) {
            bc = c2;
            bl = l2;
        }
    }
    const uint32_t nl = __shfl_sync(FULL, pc, bl);
    return bc < CUDART_INF_F ? Choice{bc, a, bl + 1, (int)nl} : Choice{CUDART_INF_F, -1, -1, 0};
}

// The cheapest of the three axes' splits (ties: the smaller axis); three warps
// of the block find them side by side.  Every thread of the block calls.
__device__ __forceinline__ Choice block_choose(const uint32_t* bins, Choice* s_axis) {
    const int warp = (int)(threadIdx.x >> 5), lane = (int)(threadIdx.x & 31);
    if (warp < 3) {
        const Choice c = axis_choose(bins, warp, lane);
        if (lane == 0) s_axis[warp] = c;
    }
    __syncthreads();
    Choice best = s_axis[0];
    if (s_axis[1].cost < best.cost) best = s_axis[1];
    if (s_axis[2].cost < best.cost) best = s_axis[2];
    return best;
}

// Where a build writes its topology.  A parent id >= 0 is a node, -1 the
// tree's root, <= -2 the root of segment -2 - parent (per-segment builds).
// A top-level build over segments (child_of set) names its nodes through
// node_ids (local id -> node) and makes each of its leaves the subtree
// child_of[item] of the listed segment `item`.
struct Links {
    BNode* nodes;
    int32_t* leaf_parent;
    int32_t* root;
    int32_t* seg_root;
    const int32_t* node_ids;
    const int32_t* child_of;
};

__device__ __forceinline__ void hook(const Links& L, int parent, int side, int child) {
    if (parent >= 0) {
        if (side) L.nodes[parent].d.y = child;
        else L.nodes[parent].d.x = child;
    } else if (parent == -1) {
        *L.root = child;
    } else {
        L.seg_root[-2 - parent] = child;
    }
}

__device__ __forceinline__ void make_node(const Links& L, int id, int parent, int side) {
    L.nodes[id].d.z = parent;
    L.nodes[id].d.w = 0;
    hook(L, parent, side, id);
}

// Leaf at global position pos, or in a top-level build the subtree of item.
__device__ __forceinline__ void make_leaf(const Links& L, int parent, int side, int pos, int item) {
    if (L.child_of) {
        const int c = L.child_of[item];
        hook(L, parent, side, c);
        if (c >= 0) L.nodes[c].d.z = parent;
        else L.leaf_parent[~c] = parent;
    } else {
        hook(L, parent, side, ~pos);
        L.leaf_parent[pos] = parent;
    }
}

// Exclusive block-wide sum (all SAH_THREADS threads call).
__device__ __forceinline__ int block_excl(int v, int* s_warp, int& total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(FULL, inc, o);
        if (lane >= o) inc += u;
    }
    if (lane == 31) s_warp[warp] = inc;
    __syncthreads();
    int off = 0, tot = 0;
#pragma unroll
    for (int w = 0; w < SAH_WARPS; w++) {
        const int s = s_warp[w];
        if (w < warp) off += s;
        tot += s;
    }
    __syncthreads();
    total = tot;
    return off + inc - v;
}

// ------------------------------------------------------------- setup

__global__ void k_sah_root(SahTask* t, int4* chunks, uint32_t* bins, SahRange* blist, int32_t n, int blk,
                           int32_t* counters) {
    chain_begin();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int size = chunk_of(n), nch = (n + size - 1) / size;
    if (i == 0) {
        SahTask r;
        r.b = 0; r.e = n; r.parent = -1; r.side = 0;
        r.buf = 0; r.chunk0 = 0; r.nchunk = nch; r.axis = -1;
        r.split = -1; r.nl = 0; r.child[0] = r.child[1] = -1;
        for (int k = 0; k < 3; k++) {
            r.cb[k] = 0xFFFFFFFFu;
            r.cb[3 + k] = 0u;
        }
        r.pad[0] = r.pad[1] = 0;
        t[0] = r;
        if (n <= blk) blist[0] = SahRange{0, n, -1, 0};
    }
    if (i < CT_WORDS) {
        int v = 0;
        if (i == CT_BLOCKS) v = n <= blk ? 1 : 0;
        if (i == CT_LEVELS) v = n <= blk ? 0 : 1;
        if (i == CT_LEVELS + 1) v = n <= blk ? 0 : nch;
        counters[i] = v;
    }
    if (n > blk) {
        if (i < nch) chunks[i] = make_int4(0, i * size, min(size, n - i * size), 0);
        if (i < SAH_BIN_WORDS) bins[i] = bin_init(i);
    }
}

// Per triangle: its box (unpadded); for a single-root build also the
// identity order and the root's centroid bounds (ord, root: nullptr for a
// segment build).
__global__ void __launch_bounds__(SAH_THREADS) k_sah_prims(const float* __restrict__ verts,
                                                           const int32_t* __restrict__ tris, int32_t n,
                                                           float4* __restrict__ pbox, int32_t* __restrict__ ord,
                                                           SahTask* root) {
    __shared__ float s_red[SAH_WARPS][6];
    chain_begin();
    const int i = blockIdx.x * SAH_THREADS + threadIdx.x;
    float r[6] = {CUDART_INF_F, CUDART_INF_F, CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F};
    if (i < n) {
        const float* p0 = verts + 3 * (int64_t)tris[3 * (int64_t)i];
        const float* p1 = verts + 3 * (int64_t)tris[3 * (int64_t)i + 1];
        const float* p2 = verts + 3 * (int64_t)tris[3 * (int64_t)i + 2];
        float lo[3], hi[3];
#pragma unroll
        for (int a = 0; a < 3; a++) {
            lo[a] = fminf(p0[a], fminf(p1[a], p2[a]));
            hi[a] = fmaxf(p0[a], fmaxf(p1[a], p2[a]));
            const float c = cen(lo[a], hi[a]);
            r[a] = c;
            r[3 + a] = c;
        }
        pbox[2 * (int64_t)i] = make_float4(lo[0], lo[1], lo[2], 0.f);
        pbox[2 * (int64_t)i + 1] = make_float4(hi[0], hi[1], hi[2], 0.f);
        if (ord) ord[i] = i;
    }
    if (!root) return;                          // block-uniform: segment builds set their own bounds
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1)
#pragma unroll
        for (int k = 0; k < 3; k++) {
            r[k] = fminf(r[k], __shfl_xor_sync(FULL, r[k], o));
            r[3 + k] = fmaxf(r[3 + k], __shfl_xor_sync(FULL, r[3 + k], o));
        }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0)
        for (int k = 0; k < 6; k++) s_red[warp][k] = r[k];
    __syncthreads();
    if (threadIdx.x < 6) {
        const int k = threadIdx.x;
        float v = s_red[0][k];
        for (int w = 1; w < SAH_WARPS; w++) v = k < 3 ? fminf(v, s_red[w][k]) : fmaxf(v, s_red[w][k]);
        if (v == v && fabsf(v) <= 3.4e38f) {   // skip the empty value of an all-idle block
            if (k < 3) atomicMin(&root->cb[k], f2o(v));
            else atomicMax(&root->cb[k], f2o(v));
        }
    }
}

// Centroid bounds of the first level's big ranges of a segment build (one
// block per range) and their bins reset.
__global__ void __launch_bounds__(SAH_THREADS) k_sah_task_init(SahTask* tasks, const int32_t* __restrict__ ord,
                                                               const float4* __restrict__ pbox, uint32_t* bins) {
    __shared__ float s_red[SAH_WARPS][6];
    SahTask& T = tasks[blockIdx.x];
    float r[6] = {CUDART_INF_F, CUDART_INF_F, CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F};
    for (int p = T.b + threadIdx.x; p < T.e; p += SAH_THREADS) {
        const int32_t t = ord[p];
        const float4 lo = pbox[2 * (int64_t)t], hi = pbox[2 * (int64_t)t + 1];
        const float c[3] = {cen(lo.x, hi.x), cen(lo.y, hi.y), cen(lo.z, hi.z)};
#pragma unroll
        for (int k = 0; k < 3; k++) {
            r[k] = fminf(r[k], c[k]);
            r[3 + k] = fmaxf(r[3 + k], c[k]);
        }
    }
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1)
#pragma unroll
        for (int k = 0; k < 3; k++) {
            r[k] = fminf(r[k], __shfl_xor_sync(FULL, r[k], o));
            r[3 + k] = fmaxf(r[3 + k], __shfl_xor_sync(FULL, r[3 + k], o));
        }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0)
        for (int k = 0; k < 6; k++) s_red[warp][k] = r[k];
    for (int i = threadIdx.x; i < SAH_BIN_WORDS; i += SAH_THREADS)
        bins[(size_t)blockIdx.x * SAH_BIN_WORDS + i] = bin_init(i);
    __syncthreads();
    if (threadIdx.x < 6) {
        const int k = threadIdx.x;
        float v = s_red[0][k];
        for (int w = 1; w < SAH_WARPS; w++) v = k < 3 ? fminf(v, s_red[w][k]) : fmaxf(v, s_red[w][k]);
        T.cb[k] = f2o(v);                       // a big range is never empty
    }
}

// A top-level tree over a single segment: the segment's subtree is the root.
__global__ void k_sah_top_single(const int32_t* child_of, BNode* nodes, int32_t* leaf_parent, int32_t* root) {
    const int c = child_of[0];
    *root = c;
    if (c >= 0) nodes[c].d.z = -1;
    else leaf_parent[~c] = -1;
}

// ------------------------------------------------------------- big ranges

// One block per chunk bins it; the block that finishes a range's last chunk
// then splits the range: split choice, node links, chunk output offsets, and
// the children (leaf, block range or next-level big range).
template <int ITEMS>
__global__ void __launch_bounds__(SAH_THREADS) k_sah_split(const int4* chunks, SahTask* tasks,
                                                           const int32_t* ord0, const int32_t* ord1,
                                                           const float4* pbox, uint32_t* bins,
                                                           uint32_t* hist, int32_t* __restrict__ left_off, Links L,
                                                           SahTask* next, int4* next_chunks, uint32_t* next_bins,
                                                           SahRange* blist, int32_t* counters, int lev,
                                                           int32_t cap_task, int32_t cap_chunk, int32_t cap_blist,
                                                           int blk) {
    constexpr int CH = ITEMS * SAH_THREADS;   // chunk size
    __shared__ uint32_t sb[SAH_BIN_WORDS];
    __shared__ Choice s_axis[3];
    __shared__ int s_last;
    chain_begin();
    const int4 chunk = chunks[blockIdx.x];     // (task, start, length); read beside the counters, before they are known
    if ((int)blockIdx.x >= counters[lev + 1] || counters[CT_BAD]) return;
    SahTask& T = tasks[chunk.x];
    for (int i = threadIdx.x; i < SAH_BIN_WORDS; i += SAH_THREADS) sb[i] = bin_init(i);
    float clo[3], chi[3];
#pragma unroll
    for (int a = 0; a < 3; a++) {
        clo[a] = o2f(T.cb[a]);
        chi[a] = o2f(T.cb[3 + a]);
    }
    const BinMap m = bin_map(clo, chi);
    const int32_t* ord = T.buf ? ord1 : ord0;
    // (all items' loads before the barrier and before the first of them is binned)
    int32_t t[ITEMS];
    float4 blo[ITEMS], bhi[ITEMS];
#pragma unroll
    for (int j = 0; j < ITEMS; j++) {
        const int i = (int)threadIdx.x + j * SAH_THREADS;
        t[j] = i < chunk.z ? ord[chunk.y + i] : -1;
    }
#pragma unroll
    for (int j = 0; j < ITEMS; j++) {
        const int64_t b = t[j] >= 0 ? 2 * (int64_t)t[j] : 0;
        blo[j] = pbox[b];
        bhi[j] = pbox[b + 1];
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < ITEMS; j++) {
        if (t[j] < 0) break;
        const float l[3] = {blo[j].x, blo[j].y, blo[j].z}, h[3] = {bhi[j].x, bhi[j].y, bhi[j].z};
#pragma unroll
        for (int a = 0; a < 3; a++) {
            uint32_t* p = sb + (a * NB + bin_of(m, a, cen(l[a], h[a]))) * BW;
            atomicAdd(p, 1u);
#pragma unroll
            for (int k = 0; k < 3; k++) {
                atomicMin(p + 1 + k, f2o(l[k]));
                atomicMax(p + 4 + k, f2o(h[k]));
            }
        }
    }
    __syncthreads();
    uint32_t* gb = bins + (size_t)chunk.x * SAH_BIN_WORDS;
    for (int i = threadIdx.x; i < SAH_BIN_WORDS; i += SAH_THREADS) {
        const int w = i % BW;
        const uint32_t cnt = sb[i - w];
        if (w == 0) __stcg(hist + (size_t)blockIdx.x * 3 * NB + i / BW, cnt);
        if (cnt == 0) continue;
        if (w == 0) atomicAdd(gb + i, cnt);
        else if (w < 4) atomicMin(gb + i, sb[i]);
        else atomicMax(gb + i, sb[i]);
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(&T.pad[0], 1) == T.nchunk - 1;
    __syncthreads();
    if (!s_last) return;
    // every chunk of the range is binned: its bins and histograms come from L2
    __threadfence();
    for (int i = threadIdx.x; i < SAH_BIN_WORDS; i += SAH_THREADS) sb[i] = __ldcg(gb + i);
    __syncthreads();
    const Choice ch = block_choose(sb, s_axis);
    if (threadIdx.x >= 32) return;
    const int lane = (int)threadIdx.x;
    const int b = T.b, e = T.e, msz = e - b;
    const int nl = ch.axis < 0 ? msz / 2 : ch.nl;
    // left items before each chunk (chunks of a range are in position order)
    int carry = 0;
    for (int k0 = 0; k0 < T.nchunk; k0 += 32) {
        const int k = k0 + lane;
        int lc = 0;
        if (k < T.nchunk) {
            const int4 cr = chunks[T.chunk0 + k];
            if (ch.axis < 0) {
                lc = min(max(nl - (cr.y - b), 0), cr.z);
            } else {
                // (all bins, so that their loads are under way together)
                const uint4* h = reinterpret_cast<const uint4*>(hist + (size_t)(T.chunk0 + k) * 3 * NB + ch.axis * NB);
#pragma unroll
                for (int j = 0; j < NB / 4; j++) {
                    const uint4 v = __ldcg(h + j);
                    lc += (4 * j < ch.split ? v.x : 0u) + (4 * j + 1 < ch.split ? v.y : 0u) +
                          (4 * j + 2 < ch.split ? v.z : 0u) + (4 * j + 3 < ch.split ? v.w : 0u);
                }
            }
        }
        int inc = lc;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(FULL, inc, o);
            if (lane >= o) inc += u;
        }
        if (k < T.nchunk) left_off[T.chunk0 + k] = carry + inc - lc;
        carry += __shfl_sync(FULL, inc, 31);
    }
    const int id = b + nl - 1;
    // lane s takes side s: a leaf, a block range or a place in the next level
    int child[2] = {-1, -1};
    int q = 0, c0 = 0;
    if (lane < 2) {
        const int cb = lane ? b + nl : b, ce = lane ? e : b + nl, cm = ce - cb;
        if (cm == 1) {
            make_leaf(L, id, lane, cb, -1);
        } else if (cm <= blk) {
            q = atomicAdd(counters + CT_BLOCKS, 1);
            if (q < cap_blist) blist[q] = SahRange{cb, ce, id, lane | ((T.buf ^ 1) << 1)};
            else atomicOr(counters + CT_BAD, 1);
        } else {
            q = atomicAdd(counters + lev + 2, 1);
            c0 = atomicAdd(counters + lev + 3, (cm + CH - 1) / CH);
        }
    }
#pragma unroll
    for (int s = 0; s < 2; s++) {
        const int cb = s ? b + nl : b, ce = s ? e : b + nl, cm = ce - cb;
        if (cm <= blk) continue;
        const int nch = (cm + CH - 1) / CH;
        const int qs = __shfl_sync(FULL, q, s), cs = __shfl_sync(FULL, c0, s);
        if (qs < cap_task && cs + nch <= cap_chunk) {
            child[s] = qs;
            if (lane == 0) {
                SahTask r;
                r.b = cb; r.e = ce; r.parent = id; r.side = s;
                r.buf = T.buf ^ 1; r.chunk0 = cs; r.nchunk = nch; r.axis = -1;
                r.split = -1; r.nl = 0; r.child[0] = r.child[1] = -1;
                for (int k = 0; k < 3; k++) {
                    r.cb[k] = 0xFFFFFFFFu;
                    r.cb[3 + k] = 0u;
                }
                r.pad[0] = r.pad[1] = 0;
                next[qs] = r;
            }
            for (int k = lane; k < nch; k += 32)
                next_chunks[cs + k] = make_int4(qs, cb + k * CH, min(CH, ce - (cb + k * CH)), 0);
            for (int i = lane; i < SAH_BIN_WORDS; i += 32) next_bins[(size_t)qs * SAH_BIN_WORDS + i] = bin_init(i);
        } else if (lane == 0) {
            atomicOr(counters + CT_BAD, 1);
        }
    }
    if (lane == 0) {
        make_node(L, id, T.parent, T.side);
        T.axis = ch.axis;
        T.split = ch.split;
        T.nl = nl;
        T.child[0] = child[0];
        T.child[1] = child[1];
    }
}

// Stable scatter of a chunk to the other order buffer; leaves get their
// final position; big children get their centroid bounds.
template <int ITEMS>
__global__ void __launch_bounds__(SAH_THREADS) k_sah_partition(const int4* __restrict__ chunks,
                                                               const SahTask* tasks, const int32_t* left_off,
                                                               int32_t* ord0, int32_t* ord1,
                                                               const float4* __restrict__ pbox,
                                                               int32_t* __restrict__ order_final, SahTask* next,
                                                               const int32_t* counters, int lev) {
    __shared__ int s_warp[SAH_WARPS];
    __shared__ uint32_t s_cb[2][6];
    chain_begin();
    const int4 ch = chunks[blockIdx.x];        // as in k_sah_split
    if ((int)blockIdx.x >= counters[lev + 1] || counters[CT_BAD]) return;
    const SahTask& T = tasks[ch.x];
    const int32_t* src = T.buf ? ord1 : ord0;
    int32_t* dst = T.buf ? ord0 : ord1;
    if (threadIdx.x < 12) s_cb[threadIdx.x / 6][threadIdx.x % 6] = (threadIdx.x % 6) < 3 ? 0xFFFFFFFFu : 0u;
    float clo[3], chi[3];
#pragma unroll
    for (int a = 0; a < 3; a++) {
        clo[a] = o2f(T.cb[a]);
        chi[a] = o2f(T.cb[3 + a]);
    }
    const BinMap m = bin_map(clo, chi);
    const int axis = T.axis, split = T.split, nl = T.nl, b = T.b, msz = T.e - T.b;
    const int child[2] = {T.child[0], T.child[1]};
    const int i0 = threadIdx.x * ITEMS;
    int32_t t[ITEMS];
    float c[ITEMS][3];
    bool left[ITEMS];
    int nleft = 0;
#pragma unroll
    for (int j = 0; j < ITEMS; j++) {
        const int i = i0 + j;
        left[j] = false;
        t[j] = -1;
        if (i < ch.z) {
            t[j] = src[ch.y + i];
            const float4 lo = pbox[2 * (int64_t)t[j]], hi = pbox[2 * (int64_t)t[j] + 1];
            c[j][0] = cen(lo.x, hi.x);
            c[j][1] = cen(lo.y, hi.y);
            c[j][2] = cen(lo.z, hi.z);
            left[j] = axis < 0 ? (ch.y + i - b) < nl : bin_of(m, axis, c[j][axis]) < split;
            nleft += left[j];
        }
    }
    int total = 0;
    const int lrank0 = block_excl(nleft, s_warp, total);   // also orders the s_cb init
    const int lo_base = b + left_off[blockIdx.x];
    const int ro_base = b + nl + (ch.y - b - left_off[blockIdx.x]);
    int lr = lrank0, rr = min(i0, ch.z) - lrank0;
    const bool need_cb = child[0] >= 0 || child[1] >= 0;
#pragma unroll
    for (int j = 0; j < ITEMS; j++) {
        if (t[j] < 0) continue;
        const int pos = left[j] ? lo_base + lr++ : ro_base + rr++;
        dst[pos] = t[j];
        if ((left[j] ? nl : msz - nl) == 1) order_final[pos] = t[j];
    }
    if (!need_cb) return;                      // block-uniform
    // the children's centroid bounds, over the warp first: all items of a
    // chunk meet in six words a side
#pragma unroll
    for (int s = 0; s < 2; s++) {
        if (child[s] < 0) continue;            // block-uniform
#pragma unroll
        for (int k = 0; k < 3; k++) {
            uint32_t lo = 0xFFFFFFFFu, hi = 0u;
#pragma unroll
            for (int j = 0; j < ITEMS; j++)
                if (t[j] >= 0 && left[j] == (s == 0)) {
                    lo = min(lo, f2o(c[j][k]));
                    hi = max(hi, f2o(c[j][k]));
                }
            lo = __reduce_min_sync(FULL, lo);
            hi = __reduce_max_sync(FULL, hi);
            if ((threadIdx.x & 31) == 0) {
                atomicMin(&s_cb[s][k], lo);
                atomicMax(&s_cb[s][3 + k], hi);
            }
        }
    }
    __syncthreads();
    if (threadIdx.x < 12) {
        const int s = threadIdx.x / 6, k = threadIdx.x % 6;
        const int q = s ? child[1] : child[0];
        const uint32_t v = s_cb[s][k];
        if (q >= 0 && v != (k < 3 ? 0xFFFFFFFFu : 0u)) {
            if (k < 3) atomicMin(&next[q].cb[k], v);
            else atomicMax(&next[q].cb[k], v);
        }
    }
}

// ------------------------------------------------------------- block ranges

struct BlockSmem {
    float lo[3][SAH_CH], hi[3][SAH_CH];   // by slot (load order)
    int32_t tri[SAH_CH];                  // triangle of each slot
    uint16_t perm[SAH_CH], tmp[SAH_CH];   // slot at each position
    uint32_t bins[SAH_WARPS][SAH_BIN_WORDS];   // of each warp's range; [0] also the block's
    SahRange stack[BLK_STACK];
    SahRange mid[2][MID_CAP];
    SahRange wlist[WLIST_CAP];
    float red[SAH_WARPS][6];
    int scan[SAH_WARPS];
    Choice axis[3];
    int top, nw, bad, take, nmid[2];
};

// Exact heuristic for a range of <= 32 positions, one warp, one item per lane:
// all sub-ranges of a tree level are split at once (segmented sorts, scans and
// minima), so that a range takes as many steps as its subtree is deep, not as
// many as it has nodes (a step is a long chain of shuffles, and a block's
// warps are too few to hide it; node by node, the block tier of 1M triangles
// took 1.7 ms, and that of 2.2k 0.5 ms).  The three axes' chains run side by
// side, and small segments take shorter sorts and scans (whole build: 2.2k
// triangles 251 -> 236 us, 104k 517 -> 499, 300k 803 -> 760, 1M 1817 -> 1757).
// Positions are local to the block's range (global position = gb + local).
__device__ void warp_exact(BlockSmem& S, SahRange r0, int gb, const Links& L, int lane) {
    const int lb = r0.b, m = r0.e - r0.b;
    int slot = lane < m ? (int)S.perm[lb + lane] : 0;
    float lo[3], hi[3];
#pragma unroll
    for (int k = 0; k < 3; k++) {
        lo[k] = S.lo[k][slot];
        hi[k] = S.hi[k][slot];
    }
    // this lane's segment: first lane, size (a lane without an item: itself, 0)
    int sb = lane < m ? 0 : lane, sm = lane < m ? m : 0;
    int parent = r0.parent, side = r0.sb & 1;
    // every level splits every segment of two or more: at most 31 levels
    for (int level = 0; level < WARP_MAX && __any_sync(FULL, sm >= 2); level++) {
        const int end = sb + sm - 1;                     // last lane of the segment
        float bestc = CUDART_INF_F;
        int bestj = sb, bestidx = lane;
        const int most = __reduce_max_sync(FULL, sm);   // items of the largest segment
        if (most >= 3) {
            // each axis's order: by (segment, centroid, lane); a pair keeps its
            // order.  Small segments by exchanges between neighbours (as many
            // steps as the largest has items), else a bitonic sort
            int order[3];
            uint32_t key[3];
#pragma unroll
            for (int a = 0; a < 3; a++) {
                key[a] = sm >= 3 ? f2o(cen(lo[a], hi[a])) : 0u;
                order[a] = lane;
            }
            if (most <= 8) {
                for (int step = 0; step < most; step++) {
                    const bool first = (((lane - sb) ^ step) & 1) == 0;   // of its pair
                    const int other = (first ? lane + 1 : lane - 1) & 31;
                    const bool pair = first ? lane < end : lane > sb && sm > 0;
#pragma unroll
                    for (int a = 0; a < 3; a++) {
                        const uint32_t ok = __shfl_sync(FULL, key[a], other);
                        const int oi = __shfl_sync(FULL, order[a], other);
                        if (pair && (first ? ok < key[a] : ok > key[a])) {
                            key[a] = ok;
                            order[a] = oi;
                        }
                    }
                }
            } else {
                unsigned long long v[3];
#pragma unroll
                for (int a = 0; a < 3; a++)
                    v[a] = ((unsigned long long)sb << 37) | ((unsigned long long)key[a] << 5) | (unsigned long long)lane;
#pragma unroll
                for (int k = 2; k <= 32; k <<= 1)
#pragma unroll
                    for (int j = k >> 1; j > 0; j >>= 1) {
                        const bool keep_min = ((lane & j) == 0) == ((lane & k) == 0);
#pragma unroll
                        for (int a = 0; a < 3; a++) {
                            const unsigned long long o = __shfl_xor_sync(FULL, v[a], j);
                            v[a] = keep_min == (o < v[a]) ? o : v[a];
                        }
                    }
#pragma unroll
                for (int a = 0; a < 3; a++) order[a] = (int)(v[a] & 31ull);
            }
#pragma unroll
            for (int a = 0; a < 3; a++) {
                const int idx = order[a];
                float plo[3], phi[3], slo[3], shi[3];
#pragma unroll
                for (int k = 0; k < 3; k++) {
                    plo[k] = slo[k] = __shfl_sync(FULL, lo[k], idx);
                    phi[k] = shi[k] = __shfl_sync(FULL, hi[k], idx);
                }
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    if (o >= most) break;
#pragma unroll
                    for (int k = 0; k < 3; k++) {
                        const float ul = __shfl_up_sync(FULL, plo[k], o), uh = __shfl_up_sync(FULL, phi[k], o);
                        const float dl = __shfl_down_sync(FULL, slo[k], o), dh = __shfl_down_sync(FULL, shi[k], o);
                        if (lane - o >= sb) {
                            plo[k] = fminf(plo[k], ul);
                            phi[k] = fmaxf(phi[k], uh);
                        }
                        if (lane + o <= end) {
                            slo[k] = fminf(slo[k], dl);
                            shi[k] = fmaxf(shi[k], dh);
                        }
                    }
                }
                float rlo[3], rhi[3];
#pragma unroll
                for (int k = 0; k < 3; k++) {
                    rlo[k] = __shfl_down_sync(FULL, slo[k], 1);
                    rhi[k] = __shfl_down_sync(FULL, shi[k], 1);
                }
                float cost = CUDART_INF_F;
                if (lane < end)
                    cost = half_area3(plo, phi) * (float)(lane - sb + 1) + half_area3(rlo, rhi) * (float)(end - lane);
                // equal costs: the split nearest the middle, then the smaller one
                float bc = cost;
                int bl = lane;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    if (o >= most) break;
                    const float c2 = __shfl_up_sync(FULL, bc, o);
                    const int l2 = __shfl_up_sync(FULL, bl, o);
                    const int d1 = abs(2 * (bl - sb) + 2 - sm), d2 = abs(2 * (l2 - sb) + 2 - sm);
                    if (lane - o >= sb && (c2 < bc || (c2 == bc && (d2 < d1 || (d2 == d1 && l2 < bl))))) {
                        bc = c2;
                        bl = l2;
                    }
                }
                bc = __shfl_sync(FULL, bc, max(end, 0) & 31);
                bl = __shfl_sync(FULL, bl, max(end, 0) & 31);
                if (sm >= 3 && bc < bestc) {
                    bestc = bc;
                    bestj = bl;
                    bestidx = idx;
                }
            }
        }
        // position lb + lane takes the item that sorted to this lane
        slot = __shfl_sync(FULL, slot, bestidx);
#pragma unroll
        for (int k = 0; k < 3; k++) {
            lo[k] = __shfl_sync(FULL, lo[k], bestidx);
            hi[k] = __shfl_sync(FULL, hi[k], bestidx);
        }
        if (sm >= 2) {
            const int nl = bestj - sb + 1;
            const int id = L.node_ids ? L.node_ids[lb + sb + nl - 1] : gb + lb + sb + nl - 1;
            if (lane == sb) make_node(L, id, parent, side);
            parent = id;
            side = lane < sb + nl ? 0 : 1;
            sm = side ? sm - nl : nl;
            if (side) sb += nl;
            if (sm == 1) make_leaf(L, id, side, gb + lb + lane, S.tri[slot]);
        }
    }
    if (lane < m) S.perm[lb + lane] = (uint16_t)slot;
}

// Hands a new range to its tier: a leaf, the exact warp build, the next round
// of the warps' binned splits (list `to`), or the block's stack.  One thread;
// others may add ranges at the same time, but not to the stack.
__device__ __forceinline__ void add_range(BlockSmem& S, const SahRange& r, int gb, const Links& L, int to) {
    const int m = r.e - r.b;
    if (m == 1) {
        make_leaf(L, r.parent, r.sb, gb + r.b, S.tri[S.tmp[r.b]]);   // tmp: the parent's new order
        return;
    }
    SahRange* list = m <= WARP_MAX ? S.wlist : (m <= MID_MAX ? S.mid[to] : S.stack);
    int* n = m <= WARP_MAX ? &S.nw : (m <= MID_MAX ? &S.nmid[to] : &S.top);
    const int at = atomicAdd(n, 1);
    if (at < (m <= WARP_MAX ? WLIST_CAP : (m <= MID_MAX ? MID_CAP : BLK_STACK))) list[at] = r;
    else S.bad = 1;
}

// One binned split of a range of at most MID_MAX positions by one warp, as the
// block splits larger ones (the same bins, choice and stable order); the
// children go to list `to`.  All 32 lanes call.
__device__ __forceinline__ void warp_split(BlockSmem& S, const SahRange& r, uint32_t* bins, int gb, const Links& L,
                                           int lane, int to) {
    const int lb = r.b, le = r.e, mm = le - lb;
    float cb[6] = {CUDART_INF_F, CUDART_INF_F, CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F};
    for (int p = lb + lane; p < le; p += 32) {
        const int s = S.perm[p];
#pragma unroll
        for (int k = 0; k < 3; k++) {
            const float c = cen(S.lo[k][s], S.hi[k][s]);
            cb[k] = fminf(cb[k], c);
            cb[3 + k] = fmaxf(cb[3 + k], c);
        }
    }
    for (int i = lane; i < SAH_BIN_WORDS; i += 32) bins[i] = bin_init(i);
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1)
#pragma unroll
        for (int k = 0; k < 3; k++) {
            cb[k] = fminf(cb[k], __shfl_xor_sync(FULL, cb[k], o));
            cb[3 + k] = fmaxf(cb[3 + k], __shfl_xor_sync(FULL, cb[3 + k], o));
        }
    const BinMap bm = bin_map(cb, cb + 3);
    __syncwarp();
    for (int p = lb + lane; p < le; p += 32) {
        const int s = S.perm[p];
        float l[3], h[3];
#pragma unroll
        for (int k = 0; k < 3; k++) {
            l[k] = S.lo[k][s];
            h[k] = S.hi[k][s];
        }
#pragma unroll
        for (int a = 0; a < 3; a++) {
            uint32_t* q = bins + (a * NB + bin_of(bm, a, cen(l[a], h[a]))) * BW;
            atomicAdd(q, 1u);
#pragma unroll
            for (int k = 0; k < 3; k++) {
                atomicMin(q + 1 + k, f2o(l[k]));
                atomicMax(q + 4 + k, f2o(h[k]));
            }
        }
    }
    __syncwarp();
    Choice c = axis_choose(bins, 0, lane);
#pragma unroll 1
    for (int a = 1; a < 3; a++) {
        const Choice d = axis_choose(bins, a, lane);
        if (d.cost < c.cost) c = d;
    }
    const int nl = c.axis < 0 ? mm / 2 : c.nl;
    const unsigned lt = (1u << lane) - 1u;
    int lr = 0, rr = nl;   // stable partition of positions [lb, le)
    for (int i0 = 0; i0 < mm; i0 += 32) {
        const int i = i0 + lane;
        bool left = false;
        int s = 0;
        if (i < mm) {
            s = S.perm[lb + i];
            left = c.axis < 0 ? i < nl : bin_of(bm, c.axis, cen(S.lo[c.axis][s], S.hi[c.axis][s])) < c.split;
        }
        const unsigned in = __ballot_sync(FULL, i < mm), ml = __ballot_sync(FULL, left), mr = in & ~ml;
        if (i < mm) S.tmp[lb + (left ? lr + __popc(ml & lt) : rr + __popc(mr & lt))] = (uint16_t)s;
        lr += __popc(ml);
        rr += __popc(mr);
    }
    __syncwarp();
    for (int p = lb + lane; p < le; p += 32) S.perm[p] = S.tmp[p];
    if (lane < 2) {
        const int id = L.node_ids ? L.node_ids[lb + nl - 1] : gb + lb + nl - 1;
        if (lane == 0) make_node(L, id, r.parent, r.sb & 1);
        add_range(S, lane ? SahRange{lb + nl, le, id, 1} : SahRange{lb, lb + nl, id, 0}, gb, L, to);
    }
    __syncwarp();   // the next range reuses the bins
}

__global__ void __launch_bounds__(SAH_THREADS) k_sah_block(const SahRange* blist, const int32_t* ord0,
                                                           const int32_t* ord1, const float4* pbox,
                                                           int32_t* __restrict__ order_final, Links L,
                                                           int32_t* counters) {
    extern __shared__ __align__(16) unsigned char sah_smem[];
    BlockSmem& S = *reinterpret_cast<BlockSmem*>(sah_smem);
    chain_begin();
    // the ranges are on the device; blocks take them from a counter
    const int count = counters[CT_BLOCKS];
    for (;;) {
        if (threadIdx.x == 0) S.take = atomicAdd(counters + CT_TAKEN, 1);
        __syncthreads();
        const int mine = S.take;
        if (mine >= count) return;                 // block-uniform
        const SahRange R = blist[mine];
        const int gb = R.b, m = R.e - R.b;
        const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
        const int32_t* ord = (R.sb >> 1) ? ord1 : ord0;
        for (int i = tid; i < m; i += SAH_THREADS) {
            const int32_t t = ord[gb + i];
            const float4 l = pbox[2 * (int64_t)t], h = pbox[2 * (int64_t)t + 1];
            S.lo[0][i] = l.x; S.lo[1][i] = l.y; S.lo[2][i] = l.z;
            S.hi[0][i] = h.x; S.hi[1][i] = h.y; S.hi[2][i] = h.z;
            S.tri[i] = t;
            S.perm[i] = (uint16_t)i;
        }
        if (tid == 0) {
            S.top = 0;
            S.nw = 0;
            S.bad = 0;
            S.nmid[0] = S.nmid[1] = 0;
            add_range(S, SahRange{0, m, R.parent, R.sb & 1}, gb, L, 0);   // (m >= 2)
        }
        __syncthreads();
        for (int guard = 0; guard < 2 * SAH_CH; guard++) {
            if (S.top == 0) break;                 // block-uniform: read after a barrier
            const SahRange r = S.stack[S.top - 1];
            const int lb = r.b, le = r.e, mm = le - lb;
            // centroid bounds of the range; bins reset
            float cb[6] = {CUDART_INF_F, CUDART_INF_F, CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F};
            for (int p = lb + tid; p < le; p += SAH_THREADS) {
                const int s = S.perm[p];
#pragma unroll
                for (int k = 0; k < 3; k++) {
                    const float c = cen(S.lo[k][s], S.hi[k][s]);
                    cb[k] = fminf(cb[k], c);
                    cb[3 + k] = fmaxf(cb[3 + k], c);
                }
            }
#pragma unroll
            for (int o = 16; o >= 1; o >>= 1)
#pragma unroll
                for (int k = 0; k < 3; k++) {
                    cb[k] = fminf(cb[k], __shfl_xor_sync(FULL, cb[k], o));
                    cb[3 + k] = fmaxf(cb[3 + k], __shfl_xor_sync(FULL, cb[3 + k], o));
                }
            if (lane == 0)
                for (int k = 0; k < 6; k++) S.red[warp][k] = cb[k];
            for (int i = tid; i < SAH_BIN_WORDS; i += SAH_THREADS) S.bins[0][i] = bin_init(i);
            __syncthreads();
            if (tid == 0) S.top--;
#pragma unroll
            for (int k = 0; k < 6; k++) {
                float v = S.red[0][k];
                for (int w = 1; w < SAH_WARPS; w++) v = k < 3 ? fminf(v, S.red[w][k]) : fmaxf(v, S.red[w][k]);
                cb[k] = v;
            }
            const BinMap bm = bin_map(cb, cb + 3);
            for (int p = lb + tid; p < le; p += SAH_THREADS) {
                const int s = S.perm[p];
                float l[3], h[3];
#pragma unroll
                for (int k = 0; k < 3; k++) {
                    l[k] = S.lo[k][s];
                    h[k] = S.hi[k][s];
                }
#pragma unroll
                for (int a = 0; a < 3; a++) {
                    uint32_t* q = S.bins[0] + (a * NB + bin_of(bm, a, cen(l[a], h[a]))) * BW;
                    atomicAdd(q, 1u);
#pragma unroll
                    for (int k = 0; k < 3; k++) {
                        atomicMin(q + 1 + k, f2o(l[k]));
                        atomicMax(q + 4 + k, f2o(h[k]));
                    }
                }
            }
            __syncthreads();
            const Choice c = block_choose(S.bins[0], S.axis);
            const int nl = c.axis < 0 ? mm / 2 : c.nl;
            // stable partition of positions [lb, le)
            const int i0 = tid * SAH_ITEMS;
            bool left[SAH_ITEMS];
            int nleft = 0;
#pragma unroll
            for (int j = 0; j < SAH_ITEMS; j++) {
                const int i = i0 + j;
                left[j] = false;
                if (i < mm) {
                    const int s = S.perm[lb + i];
                    left[j] = c.axis < 0 ? i < nl : bin_of(bm, c.axis, cen(S.lo[c.axis][s], S.hi[c.axis][s])) < c.split;
                    nleft += left[j];
                }
            }
            int total = 0;
            const int lr0 = block_excl(nleft, S.scan, total);
            int lr = lr0, rr = min(i0, mm) - lr0;
#pragma unroll
            for (int j = 0; j < SAH_ITEMS; j++) {
                const int i = i0 + j;
                if (i < mm) S.tmp[lb + (left[j] ? lr++ : nl + rr++)] = S.perm[lb + i];
            }
            __syncthreads();
            for (int p = lb + tid; p < le; p += SAH_THREADS) S.perm[p] = S.tmp[p];
            if (tid == 0) {
                const int id = L.node_ids ? L.node_ids[lb + nl - 1] : gb + lb + nl - 1;
                make_node(L, id, r.parent, r.sb & 1);
                add_range(S, SahRange{lb, lb + nl, id, 0}, gb, L, 0);
                add_range(S, SahRange{lb + nl, le, id, 1}, gb, L, 0);
            }
            __syncthreads();
        }
        // ranges of up to MID_MAX: a warp each, all of a level at once
        int from = 0;
        for (int guard = 0; guard < MID_MAX; guard++) {   // (each level takes at least one off the largest)
            const int nm = min(S.nmid[from], MID_CAP);
            if (nm == 0) break;                    // block-uniform
            for (int q = warp; q < nm; q += SAH_WARPS) warp_split(S, S.mid[from][q], S.bins[warp], gb, L, lane, from ^ 1);
            __syncthreads();
            if (tid == 0) S.nmid[from] = 0;
            __syncthreads();
            from ^= 1;
        }
        for (int q = warp; q < S.nw; q += SAH_WARPS) warp_exact(S, S.wlist[q], gb, L, lane);
        __syncthreads();
        if (order_final)
            for (int i = tid; i < m; i += SAH_THREADS) order_final[gb + i] = S.tri[S.perm[i]];
        if (tid == 0 && (S.bad || S.top != 0 || S.nmid[0] != 0 || S.nmid[1] != 0)) atomicOr(counters + CT_BAD, 2);
        __syncthreads();                           // the next range reuses S
    }
}

}  // namespace

size_t sah_scratch_bytes(int64_t n) {
    const int64_t cap_task = n / (blk_of(n) + 1) + 2;
    const int64_t cap_chunk = n / chunk_of(n) + cap_task + 4;
    const int64_t cap_blist = n / 2 + 2;
    return sizeof(float4) * 2 * n + sizeof(int32_t) * 3 * n + sizeof(uint32_t) * 3 * NB * cap_chunk +
           sizeof(int32_t) * cap_chunk + sizeof(SahTask) * 2 * cap_task + sizeof(int4) * 2 * cap_chunk +
           sizeof(uint32_t) * SAH_BIN_WORDS * 2 * cap_task + sizeof(SahRange) * cap_blist + CT_WORDS * sizeof(int32_t) +
           16 * 256;   // alignment slack
}

namespace {

struct SahArena {
    float4* pbox;
    int32_t *ord0, *ord1, *loff, *counters;
    uint32_t* hist;
    SahTask* tasks[2];
    int4* chunks[2];
    uint32_t* bins[2];
    SahRange* blist;
    int32_t cap_task, cap_chunk, cap_blist;
};

cudaError_t carve(void* scratch, int32_t n, SahArena& A) {
    A.cap_task = n / (blk_of(n) + 1) + 2;
    A.cap_chunk = n / chunk_of(n) + A.cap_task + 4;
    A.cap_blist = n / 2 + 2;
    unsigned char* p = (unsigned char*)scratch;
    auto take = [&](size_t bytes) {
        void* r = p;
        p += (bytes + 255) & ~(size_t)255;
        return r;
    };
    A.pbox = (float4*)take(sizeof(float4) * 2 * (size_t)n);
    A.ord0 = (int32_t*)take(sizeof(int32_t) * (size_t)n);
    A.ord1 = (int32_t*)take(sizeof(int32_t) * (size_t)n);
    A.hist = (uint32_t*)take(sizeof(uint32_t) * 3 * NB * (size_t)A.cap_chunk);
    A.loff = (int32_t*)take(sizeof(int32_t) * (size_t)A.cap_chunk);
    for (int k = 0; k < 2; k++) A.tasks[k] = (SahTask*)take(sizeof(SahTask) * (size_t)A.cap_task);
    for (int k = 0; k < 2; k++) A.chunks[k] = (int4*)take(sizeof(int4) * (size_t)A.cap_chunk);
    for (int k = 0; k < 2; k++) A.bins[k] = (uint32_t*)take(sizeof(uint32_t) * SAH_BIN_WORDS * (size_t)A.cap_task);
    A.blist = (SahRange*)take(sizeof(SahRange) * (size_t)A.cap_blist);
    A.counters = (int32_t*)take(CT_WORDS * sizeof(int32_t));
    return (size_t)(p - (unsigned char*)scratch) > sah_scratch_bytes(n) ? cudaErrorInvalidValue : cudaSuccess;
}

cudaError_t block_attr(rtsdf_ctx* c) {
    static bool attr_set[64] = {};             // per device ordinal
    const int dv = c->device >= 0 && c->device < 64 ? c->device : 0;
    if (!attr_set[dv]) {
        cudaError_t e = cudaFuncSetAttribute(k_sah_block, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)sizeof(BlockSmem));
        if (e != cudaSuccess) return e;
        attr_set[dv] = true;
    }
    return cudaSuccess;
}

// The levels over big ranges, then the block ranges; the first level (ntask
// ranges of at most `largest` positions) is in A and its counts in A.counters.
// Levels are enqueued in batches, each with the largest grid that it can need
// and kernels that read the level's size on the device; the host looks once
// per batch whether ranges are left (one batch nearly always does).  With a
// look after every level, the host round trips were a third of a build.
cudaError_t run_levels(rtsdf_ctx* c, SahArena& A, const Links& L, int32_t* order, int32_t n, int32_t ntask,
                       int32_t largest) {
    cudaError_t e;
    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device);
    const int blk = blk_of(n);
    int cur = 0;
    // a binned split is rarely further off the middle than these allow for (an
    // empty level costs 6 us, a second batch 150)
    int levels = 0;
    if (ntask > 0) {
        while (((int64_t)blk << levels) < largest) levels++;
        levels = std::min(levels + 6, LEVEL_BATCH);
    }
    const bool one = chunk_of(n) == SAH_THREADS;   // items a thread: one or SAH_ITEMS
    const auto split = one ? k_sah_split<1> : k_sah_split<SAH_ITEMS>;
    const auto part = one ? k_sah_partition<1> : k_sah_partition<SAH_ITEMS>;
    const int64_t block_grid = std::min<int64_t>(std::max<int64_t>(n / 64, 1), 4 * (int64_t)(sms > 0 ? sms : 132));
    for (int batch = 0;; batch++) {
        if (batch >= 4096) return cudaErrorUnknown;   // sizes shrink every level; only a fault gets here
        int64_t tasks = ntask;
        for (int l = 0; l < levels; l++) {
            const int lev = CT_LEVELS + 2 * l;
            const unsigned gc = (unsigned)std::min<int64_t>(n / chunk_of(n) + tasks + 1, A.cap_chunk);
            launch_chain(c, split, gc, SAH_THREADS, 0, A.chunks[cur], A.tasks[cur], A.ord0, A.ord1, A.pbox,
                         A.bins[cur], A.hist, A.loff, L, A.tasks[cur ^ 1], A.chunks[cur ^ 1], A.bins[cur ^ 1],
                         A.blist, A.counters, lev, A.cap_task, A.cap_chunk, A.cap_blist, blk);
            launch_chain(c, part, gc, SAH_THREADS, 0, A.chunks[cur], A.tasks[cur], A.loff, A.ord0, A.ord1,
                         A.pbox, order, A.tasks[cur ^ 1], A.counters, lev);
            tasks = std::min<int64_t>(2 * tasks, A.cap_task);
            cur ^= 1;
        }
        launch_chain(c, k_sah_block, (unsigned)block_grid, SAH_THREADS, sizeof(BlockSmem), A.blist, A.ord0, A.ord1,
                     A.pbox, order, L, A.counters);
        int32_t h[CT_WORDS];
        if ((e = cudaGetLastError())) return e;
        if ((e = cudaMemcpyAsync(h, A.counters, sizeof(h), cudaMemcpyDeviceToHost, c->stream))) return e;
        if ((e = cudaStreamSynchronize(c->stream))) return e;
        if (h[CT_BAD] != 0) return cudaErrorUnknown;   // a capacity guard fired: cannot happen for a valid range
        ntask = h[CT_LEVELS + 2 * levels];
        if (ntask == 0) return cudaSuccess;
        // the ranges that are left become the first level of another batch
        int32_t r[CT_WORDS] = {0};
        r[CT_BLOCKS] = r[CT_TAKEN] = h[CT_BLOCKS];
        r[CT_LEVELS] = ntask;
        r[CT_LEVELS + 1] = h[CT_LEVELS + 2 * levels + 1];
        if ((e = cudaMemcpyAsync(A.counters, r, sizeof(r), cudaMemcpyHostToDevice, c->stream))) return e;
        if ((e = cudaStreamSynchronize(c->stream))) return e;   // r is a local buffer
        levels = 4;
    }
}

}  // namespace

cudaError_t sah_topology(rtsdf_ctx* c, void* scratch, int32_t* order) {
    Bvh& bv = c->bvh;
    const int32_t n = (int32_t)bv.nt;
    SahArena A;
    cudaError_t e = carve(scratch, n, A);
    if (!e) e = block_attr(c);
    if (e) return e;
    const int nch0 = (n + chunk_of(n) - 1) / chunk_of(n);
    const int init_threads = nch0 > SAH_BIN_WORDS ? nch0 : SAH_BIN_WORDS;
    launch_chain(c, k_sah_root, (unsigned)((init_threads + 255) / 256), 256, 0, A.tasks[0], A.chunks[0], A.bins[0],
                 A.blist, n, blk_of(n), A.counters);
    launch_chain(c, k_sah_prims, (unsigned)((n + SAH_THREADS - 1) / SAH_THREADS), SAH_THREADS, 0, c->verts, c->tris,
                 n, A.pbox, A.ord0, A.tasks[0]);
    const Links L{bv.nodes, bv.leaf_parent, bv.root, nullptr, nullptr, nullptr};
    return run_levels(c, A, L, order, n, n > blk_of(n) ? 1 : 0, n);
}

cudaError_t sah_segments(rtsdf_ctx* c, void* scratch, int32_t* order, const int32_t* order_in,
                         const int32_t* bounds, int32_t nseg, int32_t* seg_root) {
    Bvh& bv = c->bvh;
    const int32_t n = (int32_t)bv.nt;
    SahArena A;
    cudaError_t e = carve(scratch, n, A);
    if (!e) e = block_attr(c);
    if (e) return e;
    // the first level, laid out on the host
    std::vector<SahTask> tasks;
    std::vector<int4> chunks;
    std::vector<SahRange> blist;
    std::vector<int32_t> root0((size_t)nseg, 0);
    int32_t largest = 0;
    const int size = chunk_of(n);
    for (int32_t k = 0; k < nseg; k++) {
        const int32_t b = bounds[k], en = bounds[k + 1], m = en - b;
        if (m == 1) {
            root0[(size_t)k] = ~b;                // a one-triangle segment is its own leaf
        } else if (m <= blk_of(n)) {
            blist.push_back(SahRange{b, en, -2 - k, 0});
        } else {
            largest = std::max(largest, m);
            SahTask t;
            memset(&t, 0, sizeof(t));
            t.b = b; t.e = en; t.parent = -2 - k; t.side = 0; t.buf = 0;
            t.chunk0 = (int32_t)chunks.size();
            t.nchunk = (m + size - 1) / size;
            t.axis = -1; t.split = -1; t.child[0] = t.child[1] = -1;
            for (int q = 0; q < t.nchunk; q++)
                chunks.push_back(make_int4((int)tasks.size(), b + q * size, std::min(size, en - (b + q * size)), 0));
            tasks.push_back(t);
        }
    }
    if ((int64_t)tasks.size() > A.cap_task || (int64_t)chunks.size() > A.cap_chunk ||
        (int64_t)blist.size() > A.cap_blist)
        return cudaErrorInvalidValue;   // cannot happen: the segments partition [0, n)
    int32_t h0[CT_WORDS] = {0};
    h0[CT_BLOCKS] = (int32_t)blist.size();
    h0[CT_LEVELS] = (int32_t)tasks.size();
    h0[CT_LEVELS + 1] = (int32_t)chunks.size();
    if ((e = cudaMemcpyAsync(A.counters, h0, sizeof(h0), cudaMemcpyHostToDevice, c->stream))) return e;
    if ((e = cudaMemcpyAsync(seg_root, root0.data(), sizeof(int32_t) * (size_t)nseg, cudaMemcpyHostToDevice,
                             c->stream)))
        return e;
    if (!tasks.empty() &&
        ((e = cudaMemcpyAsync(A.tasks[0], tasks.data(), sizeof(SahTask) * tasks.size(), cudaMemcpyHostToDevice,
                              c->stream)) ||
         (e = cudaMemcpyAsync(A.chunks[0], chunks.data(), sizeof(int4) * chunks.size(), cudaMemcpyHostToDevice,
                              c->stream))))
        return e;
    if (!blist.empty() && (e = cudaMemcpyAsync(A.blist, blist.data(), sizeof(SahRange) * blist.size(),
                                               cudaMemcpyHostToDevice, c->stream)))
        return e;
    if ((e = cudaMemcpyAsync(A.ord0, order_in, sizeof(int32_t) * (size_t)n, cudaMemcpyDeviceToDevice, c->stream)))
        return e;
    RTSDF_LAUNCH(c, k_sah_prims, (unsigned)((n + SAH_THREADS - 1) / SAH_THREADS), SAH_THREADS, 0, c->verts, c->tris,
                 n, A.pbox, (int32_t*)nullptr, (SahTask*)nullptr);
    if (!tasks.empty())
        RTSDF_LAUNCH(c, k_sah_task_init, (unsigned)tasks.size(), SAH_THREADS, 0, A.tasks[0], A.ord0, A.pbox, A.bins[0]);
    // one-triangle segments are final at once
    if ((e = cudaMemcpyAsync(order, order_in, sizeof(int32_t) * (size_t)n, cudaMemcpyDeviceToDevice, c->stream)))
        return e;
    const Links L{bv.nodes, bv.leaf_parent, bv.root, seg_root, nullptr, nullptr};
    // the host vectors must outlive the copies above: run_levels synchronises
    return run_levels(c, A, L, order, n, (int32_t)tasks.size(), largest);
}

size_t sah_top_bytes(int32_t nseg) {
    return 512 + sizeof(int32_t) * (size_t)nseg;   // counters | range | identity list
}

cudaError_t sah_top_prepare(rtsdf_ctx* c, void* scratch, int32_t nseg) {
    if (nseg < 1 || nseg > SAH_CH) return cudaErrorInvalidValue;
    std::vector<unsigned char> h(sah_top_bytes(nseg), 0);
    ((int32_t*)h.data())[CT_BLOCKS] = 1;
    SahRange r{0, nseg, -1, 0};
    memcpy(h.data() + 256, &r, sizeof(r));
    int32_t* list = (int32_t*)(h.data() + 512);
    for (int32_t j = 0; j < nseg; j++) list[j] = j;
    cudaError_t e = cudaMemcpyAsync(scratch, h.data(), h.size(), cudaMemcpyHostToDevice, c->stream);
    if (!e) e = cudaStreamSynchronize(c->stream);   // h is a local buffer
    return e;
}

cudaError_t sah_top(rtsdf_ctx* c, void* scratch, int32_t nseg, const float4* boxes, const int32_t* node_ids,
                    const int32_t* child_of) {
    Bvh& bv = c->bvh;
    if (nseg < 1 || nseg > SAH_CH) return cudaErrorInvalidValue;
    if (nseg == 1) {
        RTSDF_LAUNCH(c, k_sah_top_single, 1, 1, 0, child_of, bv.nodes, bv.leaf_parent, bv.root);
        return cudaGetLastError();
    }
    cudaError_t e = block_attr(c);
    if (e) return e;
    unsigned char* p = (unsigned char*)scratch;
    int32_t* counters = (int32_t*)p;
    SahRange* range = (SahRange*)(p + 256);
    int32_t* list = (int32_t*)(p + 512);
    const Links L{bv.nodes, bv.leaf_parent, bv.root, nullptr, node_ids, child_of};
    // counters, the range {0, nseg} and the identity list come from sah_top_prepare
    if ((e = cudaMemsetAsync(counters + CT_TAKEN, 0, sizeof(int32_t), c->stream))) return e;
    RTSDF_LAUNCH(c, k_sah_block, 1, SAH_THREADS, sizeof(BlockSmem), range, list, list, boxes, (int32_t*)nullptr, L,
                 counters);
    return cudaGetLastError();
}

}  // namespace rtsdf
