// Device helpers of the 3D jump flood (Sec. 2.1), shared by the per-scene
// pass kernel (jfa.cu) and the batched persistent kernel.
#pragma once

#include <math_constants.h>

#include "internal.cuh"

namespace rtsdf {
namespace dev {

__device__ __forceinline__ uint32_t seed_d2(uint32_t s, uint32_t v, uint32_t vv) {
    uint32_t ss = __dp4a(s, s, vv);
    uint32_t sv = __dp4a(s, v, 0u);
    return (ss - 2u * sv) | (s & 0xFF000000u);
}

// Coarse SDF from a packed seed: fp32, h * sqrt(D2) - beta * h, no contraction.
__device__ __forceinline__ float coarse_value(uint32_t best, uint32_t d2, float hc, float beta_h) {
    if (best == SEED_EMPTY) return CUDART_INF_F;
    return __fsub_rn(__fmul_rn(hc, __fsqrt_rn((float)d2)), beta_h);
}

// One voxel of a pass with step k (27 candidates, two-pass exact arg-min).
// An offset that leaves the grid is replaced, on that axis only, by offset 0:
// the voxel read is then another member of the same 27-voxel set, so the
// arg-min over the multiset equals the arg-min over the voxels inside the
// grid (voxels outside hold no seed), and no masking is needed.
// NC: read the input through the read-only path (only when no thread of the
// launch writes it).
template <bool FINAL, bool NC>
__device__ __forceinline__ void jfa_voxel(const uint32_t* __restrict__ in, uint32_t* __restrict__ out, int n, int k,
                                          int x, int y, int z, float* __restrict__ coarse, float hc, float beta_h) {
    const uint32_t v = pack_seed(x, y, z);
    const uint32_t vv = __dp4a(v, v, 0u);
    int xs[3], ys[3], zs[3];
#pragma unroll
    for (int i = 0; i < 3; i++) {
        const int o = (i - 1) * k;
        xs[i] = (x + o >= 0 && x + o < n) ? x + o : x;
        ys[i] = (y + o >= 0 && y + o < n) ? y + o : y;
        zs[i] = (z + o >= 0 && z + o < n) ? z + o : z;
    }
    uint32_t cs[27], cd[27];
#pragma unroll
    for (int iz = 0; iz < 3; iz++) {
#pragma unroll
        for (int iy = 0; iy < 3; iy++) {
            const uint32_t* row = in + (size_t)n * (ys[iy] + (size_t)n * zs[iz]);
#pragma unroll
            for (int ix = 0; ix < 3; ix++) {
                const int c = 9 * iz + 3 * iy + ix;
                const uint32_t sv = NC ? __ldg(row + xs[ix]) : row[xs[ix]];
                cs[c] = sv;
                cd[c] = seed_d2(sv, v, vv);
            }
        }
    }
    // smallest D2 (three-input minima), then the smallest seed at that D2
    uint32_t dmin = __vimin3_u32(cd[0], cd[1], cd[2]);
#pragma unroll
    for (int c = 3; c < 27; c += 2) dmin = __vimin3_u32(dmin, cd[c], cd[c + 1]);
    uint32_t best = SEED_EMPTY;
#pragma unroll
    for (int c = 0; c < 27; c++)
        if (cd[c] == dmin) best = min(best, cs[c]);
    const size_t idx = x + (size_t)n * (y + (size_t)n * z);
    out[idx] = best;
    if (FINAL) coarse[idx] = coarse_value(best, dmin, hc, beta_h);
}

// z-blocked pass: a thread floods T voxels of one z-lattice column,
// (x, y, z_t = rz + k (T g + t)) for t < T (jfa_zblock_column; the
// per-scene kernel uses blocks of 32 x 4 threads in (x, y) and
// blockIdx.z = g k + rz).  The T + 2 candidate z-slices (9 voxels
// each) are read once and shared by the column's voxels.
//
// Per candidate seed s = (sx, sy, sz, 0) of a slice, once:
//   A = s.s - 2 (x sx + y sy)                     dp4a, whose accumulator
//       adds s's top byte (as 0x7F000000: a seedless candidate, all ones, lands
//       above every real key), and dp2a.lo (16-bit -2 x, -2 y times bytes 0, 1)
// Per voxel z_t and candidate, one instruction:
//   key = A - 2 z_t sz = D2 - v.v                 dp2a.hi (16-bit -2 z_t times byte 2)
// Keys of one voxel share the v.v offset, so their order is D2's; the
// arg-min is the smallest key (three-input signed minima), then the smallest
// seed among the candidates at that key (one clamped add-min and one
// multiply-add per candidate, then unsigned minima) -- the lexicographic
// (D2, seed) minimum.  An x or y offset that leaves the grid reads the voxel's own
// coordinate on that axis (a duplicate of another candidate); a z-slice
// outside the grid holds no seed.  Slices roll through registers: voxel t
// needs slices t .. t + 2 only.
// NC: read the input through the read-only path (only when nothing writes it
// while the kernel lives: not in a chain, see chain_begin).
// AHEAD hides a slice's load latency where few warps do (32^3: 12.0 -> 9.4 us,
// 61^3: 28.4 -> 25.8); with the registers it takes, large grids are slower with
// it (200^3: 629 -> 683 us).  Tried: keys as whole numbers in fp32, three
// multiply-adds at the full rate for the two dot products and the clamped add
// (256^3: 1533 instead of 1237 us: 128 registers).
__device__ __forceinline__ int dp2a_hi_s_u(uint32_t a, uint32_t b, int c) {
    int d;
    asm("dp2a.hi.s32.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}

__device__ __forceinline__ int dp2a_lo_s_u(uint32_t a, uint32_t b, int c) {
    int d;
    asm("dp2a.lo.s32.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}

// the smallest key a seedless candidate can have: 0x7F000000 + 4 255^2, minus
// 2 255 (x + y + z) with x, y, z <= 255
constexpr int SEEDLESS_KEY_MIN = 0x7F000000 - 2 * 255 * 255;

// Candidates that cannot be are left out where a whole warp or pass knows it:
// NX, NY = 2: every lane's column is within k of a side in x / y, so that only
// two of its three offsets lie in the grid; ZEDGE: the column holds the whole
// lattice, so that its first voxel has no slice below and its last none above.
// With k = n / 2 that leaves 8 of 27, with n / 4 16 on average: all passes of
// 256^3 1208 -> 1131 us, 128^3 139 -> 124, 61^3 25.8 -> 23.9.
template <int N, class V>
__device__ __forceinline__ V min_of(const V (&a)[N]) {
    V m = a[0];
#pragma unroll
    for (int c = 1; c + 1 < N; c += 2) {
        if constexpr (sizeof(V) == 4 && V(-1) < V(0)) m = (V)__vimin3_s32((int)m, (int)a[c], (int)a[c + 1]);
        else m = (V)__vimin3_u32(m, a[c], a[c + 1]);
    }
    if (N % 2 == 0) m = min(m, a[N - 1]);
    return m;
}

// The voxel's arg-min over the slices [J0, J1) of the three at ss, aa: the
// smallest key, and the smallest seed at it.
template <int J0, int J1, int C>
__device__ __forceinline__ uint32_t jfa_argmin(const uint32_t (*ss)[C], const int (*aa)[C], int z, int& kmin) {
    constexpr int N = (J1 - J0) * C;
    // 16-bit -2 z in the low half, 0 in the high half (byte 3 is 0 or, for
    // a seedless candidate, already pushed out of range through A)
    const uint32_t wz = (uint32_t)(-2 * z) & 0xFFFFu;
    int key[N];
#pragma unroll
    for (int j = J0; j < J1; j++)
#pragma unroll
        for (int c = 0; c < C; c++) key[C * (j - J0) + c] = dp2a_hi_s_u(wz, ss[j][c], aa[j][c]);
    kmin = min_of(key);
    // smallest seed among the candidates at kmin: gap = min(key - kmin,
    // 255) is 0 exactly for them, and gap * 2^24 + seed then orders every
    // such candidate (a real seed, < 2^24) before every other one (>= 2^24;
    // a seedless one has gap 255 and wraps to 254 * 2^24 + 0xFFFFFF).
    // When kmin itself is a seedless key, every candidate is seedless.
    uint32_t v[N];
#pragma unroll
    for (int j = J0; j < J1; j++)
#pragma unroll
        for (int c = 0; c < C; c++) {
            const uint32_t gap = (uint32_t)__viaddmin_s32(key[C * (j - J0) + c], -kmin, 255);
            v[C * (j - J0) + c] = gap * 0x01000000u + ss[j][c];
        }
    const uint32_t vmin = min_of(v);
    return kmin >= SEEDLESS_KEY_MIN ? SEED_EMPTY : vmin;
}

template <bool FINAL, int T, bool AHEAD, bool NC, bool ZEDGE = false, int NX = 3, int NY = 3>
__device__ __forceinline__ void jfa_zblock_column(const uint32_t* in, uint32_t* __restrict__ out,
                                                  int n, int k, int x, int y, int rz, int g,
                                                  float* __restrict__ coarse, float hc, float beta_h) {
    constexpr int C = NX * NY;
    const uint32_t n2 = (uint32_t)n * (uint32_t)n;
    const uint32_t row = (uint32_t)y * (uint32_t)n;
    // offsets -k, 0, k; of two: the one in the grid (or 0 twice) and 0
    uint32_t xs[NX], ys[NY];
#pragma unroll
    for (int i = 0; i < NX; i++) {
        int o = (i - 1) * k;
        if (NX == 2) o = i == 1 ? 0 : (x - k >= 0 ? -k : k);
        xs[i] = (uint32_t)((x + o >= 0 && x + o < n) ? x + o : x);
    }
#pragma unroll
    for (int i = 0; i < NY; i++) {
        int o = (i - 1) * k;
        if (NY == 2) o = i == 1 ? 0 : (y - k >= 0 ? -k : k);
        ys[i] = (uint32_t)((y + o >= 0 && y + o < n) ? y + o : y) * (uint32_t)n;
    }
    const uint32_t wxy = ((uint32_t)(-2 * x) & 0xFFFFu) | ((uint32_t)(-2 * y) << 16);
    const int vv = x * x + y * y;
    // slice j (0 .. T + 1) holds z-lattice index T g + j - 1
    uint32_t ss[T + 2][C];
    int aa[T + 2][C];
    auto take = [&](int j, int c, uint32_t sv) {
        ss[j][c] = sv;
        aa[j][c] = dp2a_lo_s_u(wxy, sv, (int)__dp4a(sv, sv, sv & 0x7F000000u));
    };
    auto read = [](const uint32_t* p) { return NC ? __ldg(p) : *p; };
    auto load_slice = [&](int j) {
        const int z = rz + k * (T * g + j - 1);
        if (z >= 0 && z < n) {
            const uint32_t zo = (uint32_t)z * n2;
#pragma unroll
            for (int iy = 0; iy < NY; iy++)
#pragma unroll
                for (int ix = 0; ix < NX; ix++) take(j, NX * iy + ix, read(in + zo + ys[iy] + xs[ix]));
        } else {
#pragma unroll
            for (int c = 0; c < C; c++) {
                ss[j][c] = SEED_EMPTY;
                aa[j][c] = 0x7F000000;
            }
        }
    };
    // AHEAD: the seeds of a slice without a branch, read one step before use
    uint32_t nx[C];
    auto fetch = [&](int j) {
        const int z = rz + k * (T * g + j - 1);
        const bool in_grid = z >= 0 && z < n;
        const uint32_t* p = in + (uint32_t)(in_grid ? z : 0) * n2;
#pragma unroll
        for (int iy = 0; iy < NY; iy++)
#pragma unroll
            for (int ix = 0; ix < NX; ix++) nx[NX * iy + ix] = in_grid ? read(p + (ys[iy] + xs[ix])) : SEED_EMPTY;
    };
    auto take_slice = [&](int j) {
#pragma unroll
        for (int c = 0; c < C; c++) take(j, c, nx[c]);
    };
    if (AHEAD) {
        if (!ZEDGE) {
            fetch(0);
            take_slice(0);
        }
        fetch(1);
        take_slice(1);
        fetch(2);
    } else {
        if (!ZEDGE) load_slice(0);
        load_slice(1);
    }
#pragma unroll
    for (int t = 0; t < T; t++) {
        const bool above = !(ZEDGE && t == T - 1);   // slice t + 2 is wanted
        if (above) {
            if (AHEAD) take_slice(t + 2);
            else load_slice(t + 2);
        }
        const int z = rz + k * (T * g + t);
        if (z >= n) break;
        if (AHEAD && t + 1 < T && !(ZEDGE && t + 1 == T - 1)) fetch(t + 3);
        int kmin;
        uint32_t best;
        if (ZEDGE && t == 0) best = jfa_argmin<1, 3, C>(ss + t, aa + t, z, kmin);
        else if (ZEDGE && t == T - 1) best = jfa_argmin<0, 2, C>(ss + t, aa + t, z, kmin);
        else best = jfa_argmin<0, 3, C>(ss + t, aa + t, z, kmin);
        const uint32_t idx = (uint32_t)x + row + (uint32_t)z * n2;
        out[idx] = best;
        if (FINAL) coarse[idx] = dev::coarse_value(best, (uint32_t)(kmin + vv + z * z), hc, beta_h);
    }
}

}  // namespace dev
}  // namespace rtsdf
