// mpm_mcis.cu -- Monte Carlo Importance Sampling of interior fill points
// (§4.1 "Monte Carlo Importance Sampling", steps 1-4) for objects given as
// contiguous ranges of surface points (the cluster C_k) and candidates Q_k:
//   d_j = min_{c in C_k} |q_j - c|;  w_j = max(exp(-d_j^2 / 2 sigma^2), eps);
//   p_j = w_j / sum w;  n_k i.i.d. draws with P(s = q_j) = p_j.
//
// GPU layout:
//   * surface points are binned per object into a uniform grid over the unit
//     cube (App. C.1 normalises every scene to it; coordinates outside are
//     clamped into the border cells, which keeps every pair within the
//     cut-off in neighbouring cells) with a counting sort.  The grid is kept as
//     one occupancy bit per cell; occupied cells are numbered by their rank
//     among the bits and carry their points' range and bounding box;
//   * candidates are taken in cell order, a warp's worth of neighbours at a
//     time, and search rings of cells in order of distance until the best
//     distance is below the ring's lower bound.  Beyond
//     d_cut = sigma sqrt(2 ln(1/eps)) the weight is eps whatever the
//     distance, so the search radius is d_cut.  Distances are compared in
//     FP32; the points that FP32 cannot tell apart from the nearest are settled
//     in FP64 at the end, so the minimum is the exact FP64 one.  A second kernel
//     takes the candidates with nothing within d_cut, whose distance is that to
//     the nearest point in the coarse cells around them, and those with many
//     points at the same distance;
//   * weights are summed as integers round(w 2^40), which makes the
//     cumulative sums independent of the summation order, and each draw
//     binary-searches its object's cumulative sums for floor(u W_k).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <string>
#include <vector>

#include "../../include/mpm.h"
#include "mpm_ptr.h"
#include "mpm_scan.cuh"
#include "mpm_scratch.h"

namespace {

thread_local std::string g_mcis_msg;

constexpr double WSCALE = 1099511627776.0;   // 2^40
constexpr int RINGS = 6;                      // coarse cell edge >= d_cut / 6: rings 0..6 cover d_cut

__device__ __forceinline__ int find_range(const int64_t *off, int n, int64_t i) {
    int lo = 0, hi = n;   // off[lo] <= i < off[hi]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (off[mid] <= i) lo = mid; else hi = mid;
    }
    return lo;
}

__device__ __forceinline__ int cell_of(float x, float inv_h, int G) {
    int c = (int)floorf(x * inv_h);
    return c < 0 ? 0 : (c >= G ? G - 1 : c);
}

// The search radius d_cut spans RINGS coarse cells.  The cells the surface
// points are binned into are `sub` times finer along each axis, so that few
// points share one (see search).
struct Grid {
    int G;            // cells per axis
    float inv_h;
    int zwords;       // words of 32 cells per row of the occupancy mask
    int sub;          // cells per coarse cell and axis
};
// occupied cells as the search reads them: one bit per cell, zwords per
// (object, x, y) row, the last of a row always zero, so that any window of up to
// 32 cells of a row lies in two consecutive words; per word the number
// of occupied cells before it; per occupied cell (in that order) the box of its
// points with their first index (lo.w) and number (hi.w)
struct Cells {
    const unsigned *mask, *before;
    const float4 *lo, *hi;
    const float4 *point;   // surface points by cell
};
__device__ __forceinline__ long long mask_row(const Grid &g, int k, int x, int y) {
    return (((long long)k * g.G + x) * g.G + y) * g.zwords;
}

// unsigned integers that order like the floats they come from
__device__ __forceinline__ unsigned ordered(float x) {
    const unsigned u = __float_as_uint(x);
    return (u & 0x80000000u) ? ~u : u | 0x80000000u;
}
__device__ __forceinline__ float unordered(unsigned u) {
    return __uint_as_float((u & 0x80000000u) ? u & 0x7fffffffu : ~u);
}

// word and bit of a surface point's cell
__device__ __forceinline__ long long point_word(int n_obj, const int64_t *soff, const float *surf, const Grid &g,
                                                int64_t s, unsigned &bit) {
    const int k = find_range(soff, n_obj, s);
    const int cx = cell_of(surf[3 * s], g.inv_h, g.G), cy = cell_of(surf[3 * s + 1], g.inv_h, g.G),
              cz = cell_of(surf[3 * s + 2], g.inv_h, g.G);
    bit = 1u << (cz & 31);
    return mask_row(g, k, cx, cy) + (cz >> 5);
}

__global__ void k_mc_mark(int n_obj, const int64_t *soff, const float *surf, Grid g, unsigned *mask) {
    const int64_t n = soff[n_obj];
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < n; s += (int64_t)gridDim.x * blockDim.x) {
        unsigned bit;
        const long long w = point_word(n_obj, soff, surf, g, s, bit);
        atomicOr(&mask[w], bit);
    }
}
__global__ void k_mc_bits(const unsigned *mask, long long words, unsigned *bits) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < words; i += (long long)gridDim.x * blockDim.x)
        bits[i] = __popc(mask[i]);
}
// points per occupied cell, each point's cell and rank in it, and the cells'
// boxes (box: min xyz, max xyz as ordered integers, the minima complemented)
__global__ void k_mc_count(int n_obj, const int64_t *soff, const float *surf, Grid g, const unsigned *mask,
                           const unsigned *before, unsigned *cnt, unsigned *cell, unsigned *rank, unsigned *box) {
    const int64_t n = soff[n_obj];
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < n; s += (int64_t)gridDim.x * blockDim.x) {
        unsigned bit;
        const long long w = point_word(n_obj, soff, surf, g, s, bit);
        const unsigned c = before[w] + __popc(mask[w] & (bit - 1u));
        cell[s] = c;
        rank[s] = atomicAdd(&cnt[c], 1u);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const unsigned u = ordered(surf[3 * s + a]);
            atomicMax(&box[6 * (size_t)c + a], ~u);
            atomicMax(&box[6 * (size_t)c + 3 + a], u);
        }
    }
}
__global__ void k_mc_scatter(int64_t n, const float *surf, const unsigned *start, const unsigned *cell,
                             const unsigned *rank, const unsigned *cnt, const unsigned *box, float4 *sorted,
                             float4 *lo, float4 *hi) {
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < n; s += (int64_t)gridDim.x * blockDim.x) {
        const unsigned c = cell[s], r = rank[s], s0 = start[c];
        sorted[s0 + r] = make_float4(surf[3 * s], surf[3 * s + 1], surf[3 * s + 2], 0.f);
        if (r == 0) {   // one point per cell writes its box
            const unsigned *b = box + 6 * (size_t)c;
            lo[c] = make_float4(unordered(~b[0]), unordered(~b[1]), unordered(~b[2]), __uint_as_float(s0));
            hi[c] = make_float4(unordered(b[3]), unordered(b[4]), unordered(b[5]), __uint_as_float(cnt[c]));
        }
    }
}

// inclusive scan of int64 weights: per-block scans, block totals, offsets
__global__ void __launch_bounds__(1024) k_mc_scan_i64_block(const long long *in, long long *out, long long n,
                                                             long long *totals) {
    __shared__ long long sh[32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    long long x = i < n ? in[i] : 0;
    for (int o = 1; o < 32; o <<= 1) {
        const long long y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sh[w] = x;
    __syncthreads();
    if (w == 0) {
        long long t = lane < (int)(blockDim.x >> 5) ? sh[lane] : 0;
        for (int o = 1; o < 32; o <<= 1) {
            const long long y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        sh[lane] = t;
    }
    __syncthreads();
    if (i < n) out[i] = x + (w > 0 ? sh[w - 1] : 0);
    if (threadIdx.x == 0) totals[blockIdx.x] = sh[(blockDim.x >> 5) - 1];
}

__global__ void __launch_bounds__(1024) k_mc_scan_i64_totals(long long *totals, long long nb) {
    // exclusive scan of the block totals, in place, one CTA
    __shared__ long long sh[32];
    long long carry = 0;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (long long b = 0; b < nb; b += blockDim.x) {
        const long long i = b + threadIdx.x;
        const long long v = i < nb ? totals[i] : 0;
        long long x = v;
        for (int o = 1; o < 32; o <<= 1) {
            const long long y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) sh[w] = x;
        __syncthreads();
        if (w == 0) {
            long long t = lane < (int)(blockDim.x >> 5) ? sh[lane] : 0;
            for (int o = 1; o < 32; o <<= 1) {
                const long long y = __shfl_up_sync(0xffffffffu, t, o);
                if (lane >= o) t += y;
            }
            sh[lane] = t;
        }
        __syncthreads();
        if (i < nb) totals[i] = carry + (w > 0 ? sh[w - 1] : 0) + x - v;
        const long long total = sh[(blockDim.x >> 5) - 1];
        __syncthreads();
        carry += total;
    }
}

__global__ void k_mc_scan_i64_add(long long *out, long long n, const long long *totals) {
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i < n) out[i] += totals[blockIdx.x];
}

// candidates in (object, cell) order of a grid of G cells per axis, so that the
// candidates of a warp are neighbours
__global__ void k_mc_cand_count(int n_obj, const int64_t *coff, const float *cand, int G, unsigned *cnt,
                                unsigned *cell, unsigned *rank) {
    const int64_t n = coff[n_obj];
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x) {
        const int k = find_range(coff, n_obj, j);
        const float ih = (float)G;
        const unsigned key = (unsigned)((((long long)k * G + cell_of(cand[3 * j], ih, G)) * G + cell_of(cand[3 * j + 1], ih, G)) * G +
                                        cell_of(cand[3 * j + 2], ih, G));
        cell[j] = key;
        rank[j] = atomicAdd(&cnt[key], 1u);
    }
}
__global__ void k_mc_cand_scatter(int64_t n, const unsigned *start, const unsigned *cell, const unsigned *rank,
                                  unsigned *order) {
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x)
        order[start[cell[j]] + rank[j]] = (unsigned)j;
}

// squared distance along one axis from q to cell c of edge h, in FP32
__device__ __forceinline__ float box_d2f(float q, int c, float h) {
    const float lo = (float)c * h, hi = lo + h;
    const float e = q < lo ? lo - q : (q > hi ? q - hi : 0.f);
    return e * e;
}

// ... from q to the range [lo, hi], and from [a, b] to it
__device__ __forceinline__ float range_d2f(float q, float lo, float hi) {
    const float e = fmaxf(0.f, fmaxf(lo - q, q - hi));
    return e * e;
}
__device__ __forceinline__ float gap2(float a, float b, float lo, float hi) {
    const float e = fmaxf(0.f, fmaxf(lo - b, a - hi));
    return e * e;
}

__device__ __forceinline__ double dist2(float qx, float qy, float qz, float4 c) {
    const double fx = (double)qx - (double)c.x, fy = (double)qy - (double)c.y, fz = (double)qz - (double)c.z;
    return fx * fx + fy * fy + fz * fz;
}

// device counters: the scans' ticket, then candidates and items left to k_mc_open, its next item
enum { OPEN_COUNT = 1, OPEN_ITEMS, OPEN_NEXT, MC_COUNTERS };

// the three smallest FP32 squared distances seen, with the points of the two
// smallest; a NaN is never kept
struct Near3 {
    float d1, d2, d3;
    unsigned i1, i2;
    __device__ __forceinline__ void clear() {
        d1 = d2 = d3 = INFINITY;
        i1 = i2 = 0;
    }
    __device__ __forceinline__ void add(float d, unsigned i) {
        if (!(d < d3)) return;
        if (d < d1) {
            d3 = d2; d2 = d1; i2 = i1;
            d1 = d; i1 = i;
        } else if (d < d2) {
            d3 = d2;
            d2 = d; i2 = i;
        } else {
            d3 = d;
        }
    }
};

__device__ __forceinline__ unsigned lanes_before() {
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}
// the i-th lowest lane of a mask
__device__ __forceinline__ int nth_lane(unsigned lanes, int i) { return (int)__fns(lanes, 0, i + 1); }

// warp minimum and maximum of non-negative floats (their bit patterns order alike)
__device__ __forceinline__ float warp_min(float x) {
    return __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(x)));
}
__device__ __forceinline__ float warp_max(float x) {
    return __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(x)));
}

// A group of candidates that search together: the cells they lie in and their
// bounding box
struct Group {
    int k;                 // object
    int c0[3], c1[3];      // cells
    float a[3], b[3];      // box
};

constexpr int NN_WARPS = 4;        // warps per CTA of the search
constexpr int TURN = 8;            // candidates a warp takes at a time, four lanes each
constexpr int FIRST_RINGS = 2;     // reach of the first pass, unless the first bound is
constexpr int DIRECT_RINGS = 4;    // this close already
constexpr int SAMPLES = 8;         // surface points each lane tries for a first bound
struct WarpScratch {
    unsigned cell[1024];           // occupied cells still to be read: mask word of the object << 5 | bit
    float4 pt[32];                 // points (x y z, index) that every candidate meets
    float two[TURN / 2][8];        // candidates 2 u, 2 u + 1: x x y y z z, bounds
    unsigned char order[32];       // candidates by (cell, octant of the cell)
};

// packed pairs of FP32 operations, one instruction each
__device__ __forceinline__ unsigned long long pack2(float2 a) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a.x), "f"(a.y));
    return r;
}
__device__ __forceinline__ float2 unpack2(unsigned long long a) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a));
    return r;
}
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
    unsigned long long r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pack2(a)), "l"(pack2(b)));
    return unpack2(r);
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
    unsigned long long r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pack2(a)), "l"(pack2(b)));
    return unpack2(r);
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(pack2(a)), "l"(pack2(b)), "l"(pack2(c)));
    return unpack2(r);
}
// distances from two coordinates to the range [lo, -nhi]
__device__ __forceinline__ float2 range_pair(float2 q, float lo, float nhi) {
    const float2 over = add2(q, make_float2(nhi, nhi));
    return make_float2(fmaxf(0.f, fmaxf(lo - q.x, over.x)), fmaxf(0.f, fmaxf(lo - q.y, over.y)));
}

// Appends every lane's cells to the warp's list, each as `at` plus its bit's
// number; the list's new length.  The whole warp.
__device__ __forceinline__ int list_cells(unsigned *cell, int listed, unsigned bits, unsigned at) {
    const int lane = threadIdx.x & 31;
    unsigned incl = __popc(bits);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += u;
    }
    __syncwarp();
    for (int to = listed + (int)incl - __popc(bits); bits; bits &= bits - 1) cell[to++] = at + (unsigned)(__ffs(bits) - 1);
    listed += (int)__shfl_sync(0xffffffffu, incl, 31);
    __syncwarp();
    return listed;
}

// Distances from the lanes' candidates to the points of the cells of the lanes
// in `keep` (lane l: points s0 .. s0 + n), read 32 at a time.  BY_POINT: one
// candidate, each lane takes a point; otherwise the four lanes of a candidate
// take a quarter each, passed through shared memory.
template <bool BY_POINT>
__device__ __forceinline__ void meet(Near3 &m, float qx, float qy, float qz, unsigned keep, unsigned s0, unsigned n,
                                     const float4 *sorted, WarpScratch &W) {
    const int lane = threadIdx.x & 31;
    const unsigned mine = (keep >> lane) & 1u ? n : 0u;
    unsigned incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += u;
    }
    const unsigned first = s0 - (incl - mine);   // point of running index i in this lane's cell: first + i
    const unsigned total = __shfl_sync(0xffffffffu, incl, 31);
    for (unsigned p0 = 0; p0 < total; p0 += 32) {
        const unsigned i = p0 + lane;
        int c = 0;   // the cell that holds running index i
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            if (__shfl_sync(0xffffffffu, incl, c + o - 1) <= i) c += o;
        const unsigned s = __shfl_sync(0xffffffffu, first, c & 31) + i;
        if (BY_POINT) {
            if (i < total) {
                const float4 t = sorted[s];
                const float ex = qx - t.x, ey = qy - t.y, ez = qz - t.z;
                m.add(ex * ex + ey * ey + ez * ez, s);
            }
        } else {
            __syncwarp();
            if (i < total) {
                float4 t = sorted[s];
                t.w = __uint_as_float(s);
                W.pt[lane] = t;
            }
            __syncwarp();
            const int cnt = (int)min(32u, total - p0);
#pragma unroll 4
            for (int u = lane & 3; u < cnt; u += 4) {
                const float4 t = W.pt[u];
                const float ex = qx - t.x, ey = qy - t.y, ez = qz - t.z;
                m.add(ex * ex + ey * ey + ez * ez, __float_as_uint(t.w));
            }
        }
    }
}

// Searches the cells around a group for the nearest surface points within
// sqrt(cut2).  BY_POINT: one candidate for the whole warp; otherwise one per
// four lanes, where they are active.  seed: a squared distance that the
// candidate's nearest point is known not to exceed (INFINITY: none).  The whole warp calls it, and
// all of its memory accesses are made 32 at a time: the lanes look up one row
// of cells each in the occupancy mask, then the box of one occupied cell each,
// then one point each.  A pass takes the cells up to R away from the group's;
// a second one, over the rest, follows where R proved too small.  Cells are
// dropped whose points are farther than the best point so far of every
// candidate; the first to be read is the one closest to the group.
template <bool BY_POINT>
__device__ __forceinline__ void search(Near3 &m, bool active, float qx, float qy, float qz, float seed, const Group &p,
                                       float cut2, const Grid &g, const Cells &C, WarpScratch &W) {
    const int lane = threadIdx.x & 31;
    const float hf = 1.f / g.inv_h;
    // words are counted from the object's first: one object's mask has at most
    // 2^23 (512 cells per axis would be 4.5M), so that a cell's number fits 32
    // bits, while all objects together may have more than 2^27
    const long long words0 = mask_row(g, p.k, 0, 0);
    const unsigned *const mask = C.mask + words0, *const before = C.before + words0;
    seed = fminf(seed, cut2);
    auto bound = [&]() {   // squared distance beyond which no candidate needs a point, with the margin of FP32 box distances
        seed = fminf(seed, m.d1);
        if (!BY_POINT) {
            seed = fminf(seed, __shfl_xor_sync(0xffffffffu, seed, 1));
            seed = fminf(seed, __shfl_xor_sync(0xffffffffu, seed, 2));
        }
        return (BY_POINT ? warp_min(seed) : warp_max(active ? seed : 0.f)) * 1.00001f + 2e-7f;
    };
    // cells more than R away lie at least R h away; R_most h is past the
    // cut-off (or past the grid), which keeps a window of z cells below 32
    const int R_most = min(RINGS * g.sub + 2, g.G);
    float worst = bound();
    auto rings = [&](int least) {
        const float x = sqrtf(worst) * g.inv_h;
        return x < (float)R_most ? max(least, (int)x + 1) : R_most;
    };
    bool seeded = false;
    int done = -1;   // cells up to this far away have been taken
    for (int R = rings(1) <= DIRECT_RINGS ? rings(1) : FIRST_RINGS;;) {
        const int X0 = p.c0[0] - R, Y0 = p.c0[1] - R, X1 = p.c1[0] + R, Y1 = p.c1[1] + R;
        const int wy = Y1 - Y0 + 1, rows = (X1 - X0 + 1) * wy;
        const int z0 = max(p.c0[2] - R, 0), z1 = min(p.c1[2] + R, g.G - 1);
        const unsigned all = 0xffffffffu >> (31 - (z1 - z0));
        // the window's cells that an earlier pass took, in the rows it took
        const int d0 = max(p.c0[2] - done, 0), d1 = min(p.c1[2] + done, g.G - 1);
        const unsigned old = done < 0 ? 0u : (0xffffffffu >> (31 - (d1 - d0))) << (d0 - z0);
        const float iw = 1.f / (float)wy;
        int listed = 0;   // cells in the list
        for (int c0 = 0; c0 < rows; c0 += 32) {
            const int c = c0 + lane;
            const int ix = (int)(((float)c + 0.5f) * iw);   // c / wy: c < 2^10, never near an integer
            const int x = X0 + ix, y = Y0 + c - ix * wy;
            unsigned bits = 0;             // occupied cells z0 .. z1 of the row that belong to this pass
            unsigned at = 0;               // of z0's cell: mask word of the object << 5 | bit
            // a row at the cube's face also holds what lies beyond it and is always looked up
            if (c < rows && x >= 0 && y >= 0 && x < g.G && y < g.G &&
                (x == 0 || y == 0 || x == g.G - 1 || y == g.G - 1 ||
                 gap2(p.a[0], p.b[0], (float)x * hf, (float)(x + 1) * hf) +
                         gap2(p.a[1], p.b[1], (float)y * hf, (float)(y + 1) * hf) <= worst)) {
                const unsigned row = (unsigned)((x * g.G + y) * g.zwords + (z0 >> 5));
                at = row << 5 | (z0 & 31);
                bits = __funnelshift_r(mask[row], mask[row + 1], z0 & 31) & all;
                if (x >= p.c0[0] - done && x <= p.c1[0] + done && y >= p.c0[1] - done && y <= p.c1[1] + done) bits &= ~old;
            }
            if (__any_sync(0xffffffffu, bits != 0)) {
                listed = list_cells(W.cell, listed, bits, at);
            }
            // 32 cells at a time, what is left over after the last row
            const bool last = c0 + 32 >= rows;
            while (listed >= 32 || (last && listed > 0)) {
                const int take = min(listed, 32);
                listed -= take;
                float4 lo = make_float4(0.f, 0.f, 0.f, 0.f), hi = lo;
                float dist = INFINITY;
                if (lane < take) {
                    const unsigned e = W.cell[listed + lane];
                    const unsigned c = before[e >> 5] + __popc(mask[e >> 5] & ((1u << (e & 31)) - 1u));
                    lo = C.lo[c];
                    hi = C.hi[c];
                    dist = gap2(p.a[0], p.b[0], lo.x, hi.x) + gap2(p.a[1], p.b[1], lo.y, hi.y) +
                           gap2(p.a[2], p.b[2], lo.z, hi.z);
                }
                worst = bound();
                unsigned keep = __ballot_sync(0xffffffffu, dist <= worst);
                if (!keep) continue;
                const unsigned s0 = __float_as_uint(lo.w), n = __float_as_uint(hi.w);
                if (!seeded) {
                    // the closest cell first: its points bound what else is needed
                    const unsigned near = __reduce_min_sync(0xffffffffu, __float_as_uint(dist));
                    const unsigned one = __ballot_sync(0xffffffffu, __float_as_uint(dist) == near);
                    const unsigned lead = one & (0u - one);
                    meet<BY_POINT>(m, qx, qy, qz, lead, s0, n, C.point, W);
                    worst = bound();
                    keep = __ballot_sync(0xffffffffu, dist <= worst) & ~lead;
                    seeded = true;
                }
                if (!BY_POINT && keep) {
                    // the cells that some candidate of the group still needs:
                    // each lane holds its cell against all candidates
                    // (two candidates at a time in packed arithmetic)
                    __syncwarp();
                    if ((lane & 3) == 0) {
                        float *o = &W.two[lane >> 3][(lane >> 2) & 1];
                        o[0] = qx; o[2] = qy; o[4] = qz;
                        o[6] = active ? seed * 1.00001f + 2e-7f : -1.f;
                    }
                    __syncwarp();
                    const float nhx = -hi.x, nhy = -hi.y, nhz = -hi.z;
                    bool want = false;
#pragma unroll
                    for (int u = 0; u < TURN / 2; ++u) {
                        const float4 xy = *reinterpret_cast<const float4 *>(&W.two[u][0]);
                        const float4 zb = *reinterpret_cast<const float4 *>(&W.two[u][4]);
                        float2 e = range_pair(make_float2(xy.x, xy.y), lo.x, nhx);
                        float2 acc = mul2(e, e);
                        e = range_pair(make_float2(xy.z, xy.w), lo.y, nhy);
                        acc = fma2(e, e, acc);
                        e = range_pair(make_float2(zb.x, zb.y), lo.z, nhz);
                        acc = fma2(e, e, acc);
                        want |= acc.x <= zb.z || acc.y <= zb.w;
                    }
                    keep &= __ballot_sync(0xffffffffu, want);
                }
                if (keep) meet<BY_POINT>(m, qx, qy, qz, keep, s0, n, C.point, W);
            }
        }
        worst = bound();
        const float far = (float)R * hf;
        if (R >= R_most || worst <= far * far) break;
        done = R;
        R = rings(R + 1);
    }
}

// step 1 per candidate: exact squared distance to the nearest surface point
// within d_cut.  A CTA takes NN_WARPS x per consecutive candidates in (object, cell)
// order, orders them further by the octant of their cell, and each warp takes
// `per` of them: those within `reach` cells of the first one search together,
// four lanes each, when there are at least GROUP, else the first one alone with
// the lanes on the points.  Distances are compared in FP32, whose value is
// within 1e-6 relative of the exact one; the points that FP32 cannot tell apart
// from the nearest (mostly none besides it) are settled in FP64.
//
// What bounds it: issue slots and the latency of three dependent loads per 32
// cells (mask word, box, points).  750k candidates against 108k surface points:
// 4.2 ms -> 0.76 ms; a thread per candidate walking the same cells took 2.4 ms
// (divergent), 32 candidates of one lane each 1.3 ms (a few deep groups, whose
// points are nearly equidistant, ran twice as long as all others).
constexpr int GROUP = 2;
__global__ void __launch_bounds__(32 * NN_WARPS, 7) k_mc_nn(int n_obj, const int64_t *soff, const int64_t *coff,
                                                         const float *cand, const unsigned *order, Grid g, Cells C,
                                                         int per, int reach, float cells_sorted, float cut2,
                                                         uint2 *open, uint2 *items, unsigned *ctr, double *d2) {
    __shared__ WarpScratch scratch[NN_WARPS];
    WarpScratch &W = scratch[threadIdx.x >> 5];
    const int64_t n = coff[n_obj];
    const int lane = threadIdx.x & 31;
    const int64_t t0 = (int64_t)blockIdx.x * NN_WARPS * per;
    // the CTA's candidates (every warp looks at all of them), ordered within
    // their cell by octant
    float qx = 0.f, qy = 0.f, qz = 0.f;
    int64_t j = -1;
    int k = -1;
    {
        const bool in = lane < NN_WARPS * per && t0 + lane < n;
        unsigned cell = 0xffffffffu, octant = 0;
        if (in) {
            j = order[t0 + lane];
            k = find_range(coff, n_obj, j);
            qx = cand[3 * j]; qy = cand[3 * j + 1]; qz = cand[3 * j + 2];
            const float ux = qx * cells_sorted, uy = qy * cells_sorted, uz = qz * cells_sorted;
            // candidates of one cell are side by side: any label of the cell does
            cell = ((unsigned)(int)floorf(ux) * 73856093u ^ (unsigned)(int)floorf(uy) * 19349663u ^
                    (unsigned)(int)floorf(uz) * 83492791u) & 0x7fffffffu;
            octant = (ux - floorf(ux) >= 0.5f ? 1u : 0u) | (uy - floorf(uy) >= 0.5f ? 2u : 0u) |
                     (uz - floorf(uz) >= 0.5f ? 4u : 0u);
        }
        const unsigned peers = __match_any_sync(0xffffffffu, cell);
        int rank = 0;   // among the candidates of the cell, by (octant, lane)
#pragma unroll
        for (unsigned o = 0; o < 8; ++o) {
            const unsigned m = __ballot_sync(0xffffffffu, octant == o) & peers;
            if (o < octant) rank += __popc(m);
            if (o == octant) rank += __popc(m & lanes_before());
        }
        const int to = nth_lane(peers, rank);
        W.order[to] = (unsigned char)lane;
        __syncwarp();
        const int from = W.order[min(31, (threadIdx.x >> 5) * per + (lane >> 2))];
        qx = __shfl_sync(0xffffffffu, qx, from);
        qy = __shfl_sync(0xffffffffu, qy, from);
        qz = __shfl_sync(0xffffffffu, qz, from);
        j = __shfl_sync(0xffffffffu, j, from);
        k = __shfl_sync(0xffffffffu, k, from);
    }
    const bool mine = (lane >> 2) < per && k >= 0;
    const int cx = cell_of(qx, g.inv_h, g.G), cy = cell_of(qy, g.inv_h, g.G), cz = cell_of(qz, g.inv_h, g.G);
    double best = INFINITY;
    bool opened = false;   // the lane's candidate is left to k_mc_open
    unsigned todo = __ballot_sync(0xffffffffu, mine);   // four bits per candidate
    while (todo) {
        const int lead = __ffs(todo) - 1;
        Group p;
        p.k = __shfl_sync(0xffffffffu, k, lead);
        const int lx = __shfl_sync(0xffffffffu, cx, lead), ly = __shfl_sync(0xffffffffu, cy, lead),
                  lz = __shfl_sync(0xffffffffu, cz, lead);
        const float lqx = __shfl_sync(0xffffffffu, qx, lead), lqy = __shfl_sync(0xffffffffu, qy, lead),
                    lqz = __shfl_sync(0xffffffffu, qz, lead);
        const bool near_lead = k == p.k && abs(cx - lx) <= reach && abs(cy - ly) <= reach && abs(cz - lz) <= reach;
        const unsigned same = __ballot_sync(0xffffffffu, near_lead) & todo;
        const bool together = __popc(same) >= 4 * GROUP;
        // a first bound: the closest to the first candidate of a few surface
        // points spread over the object's cells
        float seed = INFINITY;
        const int64_t s_lo = soff[p.k], s_n = soff[p.k + 1] - s_lo;
        if (s_n > 0) {
            float near = INFINITY;
            float4 at = make_float4(INFINITY, INFINITY, INFINITY, 0.f);
#pragma unroll
            for (int u = 0; u < SAMPLES; ++u) {
                const float4 t = C.point[s_lo + (s_n * (u * 32 + lane)) / (32 * SAMPLES)];
                const float ex = lqx - t.x, ey = lqy - t.y, ez = lqz - t.z;
                const float e2 = ex * ex + ey * ey + ez * ez;
                if (e2 < near) { near = e2; at = t; }
            }
            const unsigned who = __ballot_sync(0xffffffffu, near == warp_min(near));
            const int src = __ffs(who) - 1;
            const float ex = qx - __shfl_sync(0xffffffffu, at.x, src), ey = qy - __shfl_sync(0xffffffffu, at.y, src),
                        ez = qz - __shfl_sync(0xffffffffu, at.z, src);
            seed = ex * ex + ey * ey + ez * ez;
            if (!(seed < INFINITY)) seed = INFINITY;   // nothing finite to go by
        }
        Near3 m;
        m.clear();
        float px = qx, py = qy, pz = qz;
        bool active = (same >> lane) & 1u;
        if (together) {
            todo &= ~same;
            if (!active) m.d3 = -1.f;   // keeps nothing
            const int cc[3] = {cx, cy, cz}, lc[3] = {lx, ly, lz};
            const float q[3] = {qx, qy, qz}, lq[3] = {lqx, lqy, lqz};
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                p.c0[a] = __reduce_min_sync(0xffffffffu, active ? cc[a] : lc[a]);
                p.c1[a] = __reduce_max_sync(0xffffffffu, active ? cc[a] : lc[a]);
                p.a[a] = unordered(__reduce_min_sync(0xffffffffu, ordered(active ? q[a] : lq[a])));
                p.b[a] = unordered(__reduce_max_sync(0xffffffffu, ordered(active ? q[a] : lq[a])));
            }
            search<false>(m, active, px, py, pz, seed, p, cut2, g, C, W);
        } else {
            todo &= ~(0xfu << lead);
            px = lqx;
            py = lqy;
            pz = lqz;
            active = true;
            p.c0[0] = p.c1[0] = lx; p.c0[1] = p.c1[1] = ly; p.c0[2] = p.c1[2] = lz;
            p.a[0] = p.b[0] = px; p.a[1] = p.b[1] = py; p.a[2] = p.b[2] = pz;
            seed = __shfl_sync(0xffffffffu, seed, lead);
            search<true>(m, active, px, py, pz, seed, p, cut2, g, C, W);
        }
        // what FP32 cannot tell apart from the nearest point, in FP64
        float d1 = m.d1;
        if (together) {
            d1 = fminf(d1, __shfl_xor_sync(0xffffffffu, d1, 1));
            d1 = fminf(d1, __shfl_xor_sync(0xffffffffu, d1, 2));
        } else {
            d1 = warp_min(d1);
        }
        const float limit = fmaf(d1, 3e-6f, d1) + 1e-36f;
        double e = INFINITY;
        const bool none = !(d1 < INFINITY && d1 <= cut2 * 0.99997f);   // nothing within d_cut (cut2 carries a margin of 1e-5)
        bool again = active && none;
        if (active && !again) {
            if (m.d1 <= limit) e = dist2(px, py, pz, C.point[m.i1]);
            if (m.d2 <= limit) e = fmin(e, dist2(px, py, pz, C.point[m.i2]));
            again = m.d3 <= limit;
        }
        const unsigned crowd = __ballot_sync(0xffffffffu, again);
        for (int o = 1; o < (together ? 4 : 32); o <<= 1) e = fmin(e, __shfl_xor_sync(0xffffffffu, e, o));
        // left to k_mc_open: those with nothing within d_cut, together, and the
        // others still open, one by one
        if (crowd) {
            const unsigned heads = together ? 0x11111111u : 1u << lead;   // the candidates' first lanes
            const unsigned far = __ballot_sync(0xffffffffu, again && none) & heads;
            const unsigned quad = crowd | crowd >> 1 | crowd >> 2 | crowd >> 3;
            const unsigned left = together ? quad & heads : heads, alone = left & ~far;
            unsigned o0 = 0, i0 = 0;
            if (lane == 0) {
                o0 = atomicAdd(&ctr[OPEN_COUNT], (unsigned)__popc(left));
                i0 = atomicAdd(&ctr[OPEN_ITEMS], (unsigned)__popc(alone) + (far ? 1u : 0u));
            }
            o0 = __shfl_sync(0xffffffffu, o0, 0);
            i0 = __shfl_sync(0xffffffffu, i0, 0);
            if ((far >> lane) & 1u) {
                const unsigned r = __popc(far & lanes_before());
                open[o0 + r] = make_uint2((unsigned)j, __float_as_uint(INFINITY));
                if (r == 0) items[i0] = make_uint2(o0, (unsigned)__popc(far));
            }
            o0 += __popc(far);
            i0 += far ? 1 : 0;
            if ((alone >> lane) & 1u) {
                const unsigned r = __popc(alone & lanes_before());
                open[o0 + r] = make_uint2((unsigned)j, __float_as_uint(limit));
                items[i0 + r] = make_uint2(o0 + r, 1u | 1u << 4);
            }
            if ((left >> lane) & 1u) opened = true;
        }
        if (together ? active : lane == lead) best = e;
        __syncwarp();
    }
    if (mine && (lane & 3) == 0 && !opened) d2[j] = best;
}

// the smallest of the lanes' values
__device__ __forceinline__ double warp_min(double x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x = fmin(x, __shfl_xor_sync(0xffffffffu, x, o));
    return x;
}

// the cells a .. b of a grid, up to 31 along z
struct Window {
    int a[3], b[3];
    __device__ __forceinline__ int rows() const { return (b[0] - a[0] + 1) * (b[1] - a[1] + 1); }
    __device__ __forceinline__ void row(int r, int &x, int &y) const {
        const int wy = b[1] - a[1] + 1;
        x = a[0] + r / wy;
        y = a[1] + r % wy;
    }
};
// occupied cells of row (x, y) of a window; word: of its first cell
__device__ __forceinline__ unsigned row_bits(const Window &w, const Grid &g, const Cells &C, int k, int x, int y, long long &word) {
    word = mask_row(g, k, x, y) + (w.a[2] >> 5);
    return __funnelshift_r(C.mask[word], C.mask[word + 1], w.a[2] & 31) & (0xffffffffu >> (31 - (w.b[2] - w.a[2])));
}
// box of the occupied cell z cells behind a window's first in a row
__device__ __forceinline__ void cell_box(const Window &w, const Cells &C, long long word, int z, float4 &lo, float4 &hi) {
    const int at = (w.a[2] & 31) + z;
    word += at >> 5;
    const unsigned c = C.before[word] + __popc(C.mask[word] & ((1u << (at & 31)) - 1u));
    lo = C.lo[c];
    hi = C.hi[c];
}
// the cells of the coarse cells up to RINGS away from a candidate's
__device__ __forceinline__ Window coarse_window(float qx, float qy, float qz, const Grid &g) {
    const int Gc = g.G / g.sub;
    const float inv_hc = g.inv_h / (float)g.sub;
    const int c[3] = {cell_of(qx, inv_hc, Gc), cell_of(qy, inv_hc, Gc), cell_of(qz, inv_hc, Gc)};
    Window w;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        w.a[d] = max(c[d] - RINGS, 0) * g.sub;
        w.b[d] = min(c[d] + RINGS, Gc - 1) * g.sub + g.sub - 1;
    }
    return w;
}

// Squared distance of one candidate to its nearest surface point, decided in
// FP64; the whole warp.  For a candidate whose three nearest points agree to FP32
// rounding (repeated points).  limit: an FP32 squared distance that the nearest
// point does not exceed.  Each lane looks up a row of the cells within the limit
// and holds the box of one occupied cell at a time against the best distance; the
// points of a cell are shared out over the lanes.
__device__ __forceinline__ double nn_exact(float qx, float qy, float qz, float limit, int k, const Grid &g, const Cells &C) {
    const int lane = threadIdx.x & 31;
    const float hf = 1.f / g.inv_h;
    // a point beyond the cube is in the cube's outermost cells, as q -+ reach then is
    const float reach = sqrtf(limit) * 1.00001f + 1e-6f, q[3] = {qx, qy, qz};
    Window w = coarse_window(qx, qy, qz, g);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        w.a[d] = max(w.a[d], cell_of(q[d] - reach, g.inv_h, g.G));
        w.b[d] = min(w.b[d], cell_of(q[d] + reach, g.inv_h, g.G));
    }
    double best = INFINITY;
    float screen = limit;   // best * (1 + 1e-6), rounded up to FP32
    // pruning threshold in FP32: the FP32 distance of a box within d_cut is within
    // 1.3e-7 of the exact one (cell edges and differences rounded), so this margin
    // never skips a cell that could hold a closer point
    float prune = limit * 1.00001f + 2e-7f;
    const int rows = w.rows();
    for (int r0 = 0; r0 < rows; r0 += 32) {
        unsigned bits = 0;
        long long word = 0;
        int x, y;
        w.row(r0 + lane, x, y);
        // (a row at the cube's face also holds what lies beyond it)
        if (r0 + lane < rows && (x == 0 || y == 0 || x == g.G - 1 || y == g.G - 1 ||
                                 box_d2f(qx, x, hf) + box_d2f(qy, y, hf) <= prune))
            bits = row_bits(w, g, C, k, x, y, word);
        while (__any_sync(0xffffffffu, bits != 0)) {
            bool near = false;
            unsigned s0 = 0, n = 0;
            if (bits) {
                float4 lo, hi;
                cell_box(w, C, word, __ffs(bits) - 1, lo, hi);
                bits &= bits - 1;
                near = range_d2f(qx, lo.x, hi.x) + range_d2f(qy, lo.y, hi.y) + range_d2f(qz, lo.z, hi.z) <= prune;
                s0 = __float_as_uint(lo.w);
                n = __float_as_uint(hi.w);
            }
            for (unsigned keep = __ballot_sync(0xffffffffu, near); keep; keep &= keep - 1) {
                const int l = __ffs(keep) - 1;
                const unsigned p0 = __shfl_sync(0xffffffffu, s0, l), m = __shfl_sync(0xffffffffu, n, l);
                for (unsigned i = lane; i < m; i += 32) {
                    const float4 t = C.point[p0 + i];
                    const float ex = qx - t.x, ey = qy - t.y, ez = qz - t.z;
                    // the FP32 value is within 1e-6 relative of the exact one, so a
                    // point closer than best passes this FP32 screen
                    if (ex * ex + ey * ey + ez * ez <= screen) best = fmin(best, dist2(qx, qy, qz, t));
                }
            }
            best = warp_min(best);
            if (best < INFINITY) {
                screen = fminf(screen, __double2float_ru(best * (1.0 + 1e-6)));
                prune = fminf(prune, (float)best * 1.00001f + 2e-7f);
            }
        }
    }
    return best;
}

constexpr int OPEN_WARPS = 4;      // warps per CTA
struct FarScratch {
    unsigned cell[1024];           // occupied cells still to be read: row of the window << 5 | z
    struct {
        float q[3], bound;
        int a[3], b[3];
    } far[TURN];
};
// Squared distances of the lanes' candidates (one per four lanes, those of `mine`)
// to the nearest surface points in their coarse windows, decided in FP64
// (INFINITY: none); the whole warp.  For candidates with nothing within d_cut:
// their windows then say how far they looked.  The candidates walk the occupied
// cells of all their windows together, 32 at a time, a cell per lane: once for a
// limit per candidate, the farthest corner of the box that is nearest by it, then
// for the points of the boxes within it.
__device__ __forceinline__ double nn_far(bool mine, float qx, float qy, float qz, int k, const Grid &g, const Cells &C,
                                         FarScratch &W) {
    const int lane = threadIdx.x & 31, own = lane >> 2;
    const float q[3] = {qx, qy, qz};
    Window o = coarse_window(qx, qy, qz, g);
    __syncwarp();
    if ((lane & 3) == 0) {
        auto &f = W.far[own];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            f.q[d] = q[d];
            f.a[d] = o.a[d];
            f.b[d] = o.b[d];
        }
        f.bound = INFINITY;
    }
    __syncwarp();
    float limit[TURN];
#pragma unroll
    for (int u = 0; u < TURN; ++u) limit[u] = INFINITY;
    bool held = false, odd = false;   // an occupied cell; one with a point that is not finite, whose box says nothing
    double best = INFINITY;
    for (int walk = 0; walk < 2; ++walk) {
        float screen = W.far[own].bound;
        if (walk) {
            // the cells within the limits; a point beyond the cube is in the cube's
            // outermost cells, as q -+ reach then is
            mine = mine && (odd || screen < INFINITY);
            const float reach = sqrtf(screen) * 1.00001f + 1e-6f;
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                o.a[d] = max(o.a[d], cell_of(q[d] - reach, g.inv_h, g.G));
                o.b[d] = min(o.b[d], cell_of(q[d] + reach, g.inv_h, g.G));
            }
        }
        const unsigned them = __ballot_sync(0xffffffffu, mine);
        if (!them) break;
        Window w;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            w.a[d] = __reduce_min_sync(0xffffffffu, mine ? o.a[d] : g.G);
            w.b[d] = __reduce_max_sync(0xffffffffu, mine ? o.b[d] : 0);
        }
        const int rows = w.rows();
        int listed = 0;   // cells in the list: row << 5 | z
        for (int r0 = 0; r0 < rows; r0 += 32) {
            unsigned bits = 0;
            if (r0 + lane < rows) {
                int x, y;
                long long word;
                w.row(r0 + lane, x, y);
                bits = row_bits(w, g, C, k, x, y, word);
            }
            if (__any_sync(0xffffffffu, bits != 0)) listed = list_cells(W.cell, listed, bits, (unsigned)(r0 + lane) << 5);
            // 32 cells at a time, what is left over after the last row
            const bool last = r0 + 32 >= rows;
            while (listed >= 32 || (last && listed > 0)) {
                const int take = min(listed, 32);
                listed -= take;
                unsigned wanted = 0;   // candidates that need this lane's cell
                unsigned s0 = 0, n = 0;
                if (lane < take) {
                    const unsigned e = W.cell[listed + lane];
                    const int z = e & 31, zz = w.a[2] + z;
                    int x, y;
                    w.row(e >> 5, x, y);
                    float4 lo, hi;
                    cell_box(w, C, mask_row(g, k, x, y) + (w.a[2] >> 5), z, lo, hi);
                    s0 = __float_as_uint(lo.w);
                    n = __float_as_uint(hi.w);
                    held = true;
                    odd |= !isfinite((hi.x - lo.x) + (hi.y - lo.y) + (hi.z - lo.z));
#pragma unroll
                    for (int u = 0; u < TURN; ++u) {
                        const auto &f = W.far[u];
                        if (!((them >> (4 * u)) & 1u)) continue;
                        if (x < f.a[0] || x > f.b[0] || y < f.a[1] || y > f.b[1] || zz < f.a[2] || zz > f.b[2]) continue;
                        if (walk == 0) {
                            const float fx = fmaxf(hi.x - f.q[0], f.q[0] - lo.x), fy = fmaxf(hi.y - f.q[1], f.q[1] - lo.y),
                                        fz = fmaxf(hi.z - f.q[2], f.q[2] - lo.z);
                            limit[u] = fminf(limit[u], fx * fx + fy * fy + fz * fz);
                        } else if (range_d2f(f.q[0], lo.x, hi.x) + range_d2f(f.q[1], lo.y, hi.y) +
                                       range_d2f(f.q[2], lo.z, hi.z) <= f.bound * 1.00001f + 2e-7f) {
                            wanted |= 1u << u;
                        }
                    }
                }
                __syncwarp();
                if (walk == 0) continue;
                for (unsigned keep = __ballot_sync(0xffffffffu, wanted != 0); keep; keep &= keep - 1) {
                    const int l = __ffs(keep) - 1;
                    const unsigned p0 = __shfl_sync(0xffffffffu, s0, l), m = __shfl_sync(0xffffffffu, n, l);
                    if ((__shfl_sync(0xffffffffu, wanted, l) >> own) & 1u)
                        for (unsigned i = lane & 3; i < m; i += 4) {
                            const float4 t = C.point[p0 + i];
                            const float ex = qx - t.x, ey = qy - t.y, ez = qz - t.z;
                            // (the FP32 value is within 1e-6 relative of the exact one)
                            if (ex * ex + ey * ey + ez * ez <= screen) {
                                const double d2 = dist2(qx, qy, qz, t);
                                if (d2 < best) {
                                    best = d2;
                                    screen = fminf(screen, __double2float_ru(best * (1.0 + 1e-6)));
                                }
                            }
                        }
                }
            }
        }
        if (walk == 0) {
            if (!__any_sync(0xffffffffu, held)) return INFINITY;   // deep inside an object
            odd = __any_sync(0xffffffffu, odd);
            __syncwarp();
#pragma unroll
            for (int u = 0; u < TURN; ++u) {
                // with the margin of the FP32 distances of the points
                const float t = odd ? INFINITY : warp_min(limit[u]) * 1.00001f + 1e-36f;
                if (lane == 0) W.far[u].bound = t;
            }
            __syncwarp();
        }
    }
    best = fmin(best, __shfl_xor_sync(0xffffffffu, best, 1));
    return fmin(best, __shfl_xor_sync(0xffffffffu, best, 2));
}

// The candidates that k_mc_nn leaves open: an item is a group of up to TURN of them
// with nothing within d_cut, or one whose nearest points FP32 cannot tell apart
// (y >> 4); open: candidate and limit.  A warp takes the next item when it is done
// with one, since some walk a few cells and some hundreds.
//
// In a kernel of its own so that the search keeps its registers (with both in one
// the search spilled 146 bytes, and a ball of radius 0.3 took 2.2 ms).  Fills of
// 250k candidates and 36,000 surface points, by one thread per candidate without
// occupied cells, with one lane per open candidate walking its window after the
// search, and so: a ball of radius 0.3, 27% of the candidates beyond d_cut, 1.5,
// 72.8 and 1.2 ms; a ball of radius 0.15, 3%, 2.3, 8.9 and 1.3 ms; every surface
// point three times, 5.3, 6.8 and 1.6 ms.
__global__ void __launch_bounds__(32 * OPEN_WARPS) k_mc_open(int n_obj, const int64_t *coff, const float *cand, Grid g, Cells C,
                                                             const uint2 *open, const uint2 *items, unsigned *ctr,
                                                             double *d2) {
    __shared__ FarScratch scratch[OPEN_WARPS];
    const int lane = threadIdx.x & 31;
    for (;;) {
        unsigned i = 0;
        if (lane == 0) i = atomicAdd(&ctr[OPEN_NEXT], 1u);
        i = __shfl_sync(0xffffffffu, i, 0);
        if (i >= ctr[OPEN_ITEMS]) return;
        const uint2 item = items[i];
        const unsigned n = item.y & 15u;
        const bool one = (item.y >> 4) != 0, mine = (unsigned)(lane >> 2) < n;
        const uint2 o = open[item.x + (mine ? lane >> 2 : 0)];
        const int64_t j = o.x;
        const float qx = cand[3 * j], qy = cand[3 * j + 1], qz = cand[3 * j + 2];
        const int k = find_range(coff, n_obj, j);
        const double x = one ? nn_exact(qx, qy, qz, __uint_as_float(o.y), k, g, C)
                             : nn_far(mine, qx, qy, qz, k, g, C, scratch[threadIdx.x >> 5]);
        if (mine && (lane & 3) == 0) d2[j] = x;
    }
}

// step 2: distance, weight and integer weight of the squared distance, in place
// of which the integer weight is stored.  FP64 throughout (some 80 operations
// per candidate at 2 per clock and SM), so with full warps
__global__ void k_mc_weight(long long n, double sigma, double eps, double *d, double *w, long long *wq) {
    for (long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x; j < n; j += (long long)gridDim.x * blockDim.x) {
        const double best = __longlong_as_double(wq[j]);
        // nothing within the searched rings: the distance is at least d_cut, so the weight is eps
        const double wt = isinf(best) ? eps : fmax(exp(-best / (2.0 * sigma * sigma)), eps);
        if (d) d[j] = sqrt(best);
        if (w) w[j] = wt;
        wq[j] = (long long)floor(wt * WSCALE + 0.5);
    }
}

// step 4: draw i of object k picks the first candidate whose cumulative weight
// (within the object) exceeds floor(u_i W_k)
__global__ void k_mc_draw(int n_obj, const int64_t *coff, const int64_t *doff, const double *u, const long long *cum,
                          int64_t *picked) {
    const int64_t n = doff[n_obj];
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int k = find_range(doff, n_obj, i);
        const int64_t c0 = coff[k], c1 = coff[k + 1];
        if (c1 == c0) { picked[i] = -1; continue; }
        const long long base = c0 > 0 ? cum[c0 - 1] : 0;
        const long long total = cum[c1 - 1] - base;
        const long long t = (long long)floor(u[i] * (double)total);
        int64_t lo = c0, hi = c1 - 1;   // first j with cum[j] - base > t; the last candidate if none
        while (lo < hi) {
            const int64_t mid = (lo + hi) >> 1;
            if (cum[mid] - base > t) hi = mid; else lo = mid + 1;
        }
        picked[i] = lo;
    }
}

bool is_dev(const void *p) { return mpm::on_this_device(p); }

int blocks_for(long long n, int t) {
    long long b = (n + t - 1) / t;
    if (b < 1) b = 1;
    if (b > 152 * 32) b = 152 * 32;
    return (int)b;
}

}  // namespace

extern "C" MPM_API mpm_status mpm_mcis(int32_t n_obj, const int64_t *surf_off, const float *surf,
                                       const int64_t *cand_off, const float *cand, const int64_t *draw_off,
                                       const double *u, double sigma, double eps, double *d, double *w,
                                       int64_t *picked, void *stream) {
    g_mcis_msg.clear();
    if (n_obj < 1 || !surf_off || !cand_off || !draw_off || !(sigma > 0.0) || !(eps > 0.0) || !(eps < 1.0)) {
        g_mcis_msg = "mcis: n_obj >= 1, offsets non-NULL, sigma > 0, 0 < eps < 1";
        return MPM_ERR_INVALID_ARG;
    }
    for (int k = 0; k < n_obj; ++k)
        if (surf_off[k + 1] < surf_off[k] || cand_off[k + 1] < cand_off[k] || draw_off[k + 1] < draw_off[k]) {
            g_mcis_msg = "mcis: offsets must be non-decreasing";
            return MPM_ERR_INVALID_ARG;
        }
    if (surf_off[0] != 0 || cand_off[0] != 0 || draw_off[0] != 0) {
        g_mcis_msg = "mcis: offsets must start at 0";
        return MPM_ERR_INVALID_ARG;
    }
    if (mpm::any_on_other_device({surf, cand, u, d, w, picked})) {
        g_mcis_msg = "mcis: an array lives on another device than the current one";
        return MPM_ERR_INVALID_ARG;
    }
    const long long ns = surf_off[n_obj], nc = cand_off[n_obj], nd = draw_off[n_obj];
    if ((ns > 0 && !surf) || (nc > 0 && !cand) || (nd > 0 && (!u || !picked)) || ns >= (1ll << 32)) {
        g_mcis_msg = "mcis: missing arrays or too many surface points";
        return MPM_ERR_INVALID_ARG;
    }
    cudaStream_t st = (cudaStream_t)stream;
    const double cut = sigma * std::sqrt(2.0 * std::log(1.0 / eps));
    Grid g;
    // coarse cell edge 1/G >= d_cut / RINGS, so rings 0..RINGS hold every point within d_cut
    g.G = (int)std::floor(RINGS / cut);
    if (g.G < 1) g.G = 1;
    if (g.G > 256) g.G = 256;
    if ((long long)g.G * g.G * g.G * n_obj >= (1ll << 31)) { g_mcis_msg = "mcis: grid too large"; return MPM_ERR_INVALID_ARG; }
    // twice as fine where an object has the points to fill the cells, while the mask
    // stays within 8M words (its clearing and scan then cost some 30 us).  Three
    // objects, coarse and fine: 4,000 points each and 50k candidates 324 and 367 us,
    // 12,000 and 250k 650 and 656, 36,000 and 250k 1,189 and 1,072.  A ball of
    // radius 0.1, 250k candidates: 12,000 points 555 and 595 us, 18,000 692 and 715,
    // 25,000 949 and 883, 36,000 1,555 and 1,248.  (A ball of 0.2, whose points are
    // sparser, gains from 100,000 points on.)
    const int Gc = g.G;
    auto mask_words = [&](int sub) {
        const long long G = (long long)Gc * sub;
        return n_obj * G * G * ((G + 31) / 32 + 1);
    };
    g.sub = ns / n_obj >= 24000 && mask_words(2) <= (1ll << 23) ? 2 : 1;
    g.G = Gc * g.sub;
    g.inv_h = (float)g.G;
    g.zwords = (g.G + 31) / 32 + 1;
    const long long words = mask_words(g.sub);
    const float cut2 = (float)(cut * cut * (1.0 + 1e-5));
    // the candidates' cells: up to twice the coarse grid's, about a warp's worth in
    // one.  Coarse and twice as fine, a ball with 36,000 points: 12k candidates 687
    // and 829 us, 25k 772 and 920, 50k 985 and 877, 100k 1,140 and 1,170; 4,000
    // points: 25k 351 and 364, 50k 348 and 317, 100k 381 and 353
    int Gs = Gc;
    if (8ll * Gc * Gc * Gc * n_obj <= (1ll << 23) && nc / n_obj >= 50000) Gs *= 2;
    const long long keys = (long long)n_obj * Gs * Gs * Gs;

    // scratch: one stream-ordered allocation carved into pieces
    auto al = [](size_t b) { return (b + 255) & ~size_t(255); };
    const long long nb = (nc + 1023) / 1024;
    size_t off = 0;
    const size_t o_soff = off; off += al((n_obj + 1) * 8);
    const size_t o_coff = off; off += al((n_obj + 1) * 8);
    const size_t o_doff = off; off += al((n_obj + 1) * 8);
    const size_t o_surf = off; off += al(ns * 12);
    const size_t o_cand = off; off += al(nc * 12);
    const size_t o_u = off; off += al(nd * 8);
    // cleared together: counters, mask, points per cell, boxes, candidates per cell
    const size_t o_ticket = off; off += al(MC_COUNTERS * 4);
    const size_t o_mask = off; off += al(words * 4);
    const size_t o_cnt = off; off += al(ns * 4);
    const size_t o_box = off; off += al(ns * 24);
    const size_t o_cnt2 = off; off += al(keys * 4);
    const size_t o_clear = off;
    const size_t o_bits = off; off += al(words * 4);
    const size_t o_before = off; off += al(words * 4);
    const size_t o_start = off; off += al(ns * 4);
    const size_t o_cell = off; off += al(ns * 4);
    const size_t o_rank = off; off += al(ns * 4);
    const size_t o_lo = off; off += al(ns * 16);
    const size_t o_hi = off; off += al(ns * 16);
    const size_t o_start2 = off; off += al(keys * 4);
    const size_t o_ccell = off; off += al(nc * 4);
    const size_t o_crank = off; off += al(nc * 4);
    const size_t o_order = off; off += al(nc * 4);
    const size_t o_open = off; off += al(nc * 8);
    const size_t o_items = off; off += al(nc * 8);
    const size_t o_sorted = off; off += al(ns * 16);
    const size_t o_wq = off; off += al(nc * 8);
    const size_t o_cum = off; off += al(nc * 8);
    const size_t o_tot = off; off += al((nb + 1) * 8);
    const long long scan_most = std::max(keys, std::max(words, ns));
    const size_t o_kb = off; off += al(scan_words(scan_most) * 8);   // scan block sums
    const size_t o_kt = off; off += al(8);
    const size_t o_d = off; off += al(nc * 8);
    const size_t o_w = off; off += al(nc * 8);
    const size_t o_pick = off; off += al(nd * 8);
    char *buf = nullptr;
    if (mpm::scratch_alloc((void **)&buf, off ? off : 256, st) != cudaSuccess) {
        cudaGetLastError();
        g_mcis_msg = "mcis: device allocation failed";
        return MPM_ERR_OOM;
    }
    auto P = [&](size_t o) { return (void *)(buf + o); };
    mpm_status status = MPM_OK;
#define MC_CK(call)                                                                  \
    do {                                                                             \
        if ((call) != cudaSuccess) {                                                 \
            g_mcis_msg = std::string("mcis: ") + cudaGetErrorString(cudaGetLastError()); \
            status = MPM_ERR_CUDA;                                                   \
            goto done;                                                               \
        }                                                                            \
    } while (0)
    {
        int64_t *dsoff = (int64_t *)P(o_soff), *dcoff = (int64_t *)P(o_coff), *ddoff = (int64_t *)P(o_doff);
        MC_CK(cudaMemcpyAsync(dsoff, surf_off, (n_obj + 1) * 8, cudaMemcpyHostToDevice, st));
        MC_CK(cudaMemcpyAsync(dcoff, cand_off, (n_obj + 1) * 8, cudaMemcpyHostToDevice, st));
        MC_CK(cudaMemcpyAsync(ddoff, draw_off, (n_obj + 1) * 8, cudaMemcpyHostToDevice, st));
        const float *dsurf = surf, *dcand = cand;
        const double *du = u;
        if (ns > 0 && !is_dev(surf)) { MC_CK(cudaMemcpyAsync(P(o_surf), surf, ns * 12, cudaMemcpyHostToDevice, st)); dsurf = (const float *)P(o_surf); }
        if (nc > 0 && !is_dev(cand)) { MC_CK(cudaMemcpyAsync(P(o_cand), cand, nc * 12, cudaMemcpyHostToDevice, st)); dcand = (const float *)P(o_cand); }
        if (nd > 0 && !is_dev(u)) { MC_CK(cudaMemcpyAsync(P(o_u), u, nd * 8, cudaMemcpyHostToDevice, st)); du = (const double *)P(o_u); }
        auto U = [&](size_t o) { return (unsigned *)P(o); };
        unsigned *mask = U(o_mask), *cnt = U(o_cnt), *start = U(o_start);
        unsigned long long *kb = (unsigned long long *)P(o_kb), *kt = (unsigned long long *)P(o_kt);
        const Cells cells = {mask, U(o_before), (const float4 *)P(o_lo), (const float4 *)P(o_hi), (const float4 *)P(o_sorted)};
        long long *wq = (long long *)P(o_wq), *cum = (long long *)P(o_cum), *tot = (long long *)P(o_tot);
        unsigned *ticket = U(o_ticket);
        MC_CK(cudaMemsetAsync(ticket, 0, o_clear - o_ticket, st));
        if (ns > 0) {
            k_mc_mark<<<blocks_for(ns, 256), 256, 0, st>>>(n_obj, dsoff, dsurf, g, mask);
            k_mc_bits<<<blocks_for(words, 256), 256, 0, st>>>(mask, words, U(o_bits));
            scan_counts(U(o_bits), U(o_before), words, kb, kt, ticket, st);
            k_mc_count<<<blocks_for(ns, 256), 256, 0, st>>>(n_obj, dsoff, dsurf, g, mask, U(o_before), cnt, U(o_cell),
                                                            U(o_rank), U(o_box));
            scan_counts(cnt, start, ns, kb, kt, ticket, st);
            k_mc_scatter<<<blocks_for(ns, 256), 256, 0, st>>>(ns, dsurf, start, U(o_cell), U(o_rank), cnt, U(o_box),
                                                              (float4 *)P(o_sorted), (float4 *)P(o_lo),
                                                              (float4 *)P(o_hi));
            MC_CK(cudaGetLastError());
        }
        double *dd = d && is_dev(d) ? d : (double *)P(o_d);
        double *dw = w && is_dev(w) ? w : (double *)P(o_w);
        int64_t *dp = picked && is_dev(picked) ? picked : (int64_t *)P(o_pick);
        if (nc > 0) {
            unsigned *cnt2 = U(o_cnt2), *start2 = U(o_start2), *order = U(o_order);
            k_mc_cand_count<<<blocks_for(nc, 256), 256, 0, st>>>(n_obj, dcoff, dcand, Gs, cnt2, U(o_ccell), U(o_crank));
            scan_counts(cnt2, start2, keys, kb, kt, ticket, st);
            k_mc_cand_scatter<<<blocks_for(nc, 256), 256, 0, st>>>(nc, start2, U(o_ccell), U(o_crank), order);
            MC_CK(cudaGetLastError());
            // candidates per warp: 8, fewer where that would leave SMs without warps
            const int per = (int)std::min<long long>(TURN, std::max<long long>(1, nc / (152 * 24)));
            const long long ctas = (nc + per * NN_WARPS - 1) / (per * NN_WARPS);
            k_mc_nn<<<(unsigned)ctas, 32 * NN_WARPS, 0, st>>>(n_obj, dsoff, dcoff, dcand, order, g, cells, per,
                                                              std::max(1, g.sub / 2), (float)Gs, cut2,
                                                              (uint2 *)P(o_open), (uint2 *)P(o_items), ticket, (double *)wq);
            k_mc_open<<<(unsigned)std::min<long long>(152 * 5, (nc + OPEN_WARPS - 1) / OPEN_WARPS), 32 * OPEN_WARPS, 0, st>>>(
                n_obj, dcoff, dcand, g, cells, (const uint2 *)P(o_open), (const uint2 *)P(o_items), ticket, (double *)wq);
            k_mc_weight<<<blocks_for(nc, 256), 256, 0, st>>>(nc, sigma, eps, dd, dw, wq);
            MC_CK(cudaGetLastError());
            k_mc_scan_i64_block<<<(unsigned)nb, 1024, 0, st>>>(wq, cum, nc, tot);
            k_mc_scan_i64_totals<<<1, 1024, 0, st>>>(tot, nb);
            k_mc_scan_i64_add<<<(unsigned)nb, 1024, 0, st>>>(cum, nc, tot);
            MC_CK(cudaGetLastError());
        }
        if (nd > 0) {
            k_mc_draw<<<blocks_for(nd, 256), 256, 0, st>>>(n_obj, dcoff, ddoff, du, cum, dp);
            MC_CK(cudaGetLastError());
        }
        if (d && dd != d) MC_CK(cudaMemcpyAsync(d, dd, nc * 8, cudaMemcpyDeviceToHost, st));
        if (w && dw != w) MC_CK(cudaMemcpyAsync(w, dw, nc * 8, cudaMemcpyDeviceToHost, st));
        if (nd > 0 && dp != picked) MC_CK(cudaMemcpyAsync(picked, dp, nd * 8, cudaMemcpyDeviceToHost, st));
    }
done:
    cudaFreeAsync(buf, st);
    if (status == MPM_OK && cudaStreamSynchronize(st) != cudaSuccess) {
        g_mcis_msg = std::string("mcis: ") + cudaGetErrorString(cudaGetLastError());
        status = MPM_ERR_CUDA;
    }
#undef MC_CK
    return status;
}

extern "C" MPM_API const char *mpm_mcis_last_error(void) { return g_mcis_msg.c_str(); }
