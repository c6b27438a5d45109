// mpm_render.cu -- splatting of the (deformed) Gaussian kernels into a
// headless image (§3.1): Sigma' = J W Sigma W^T J^T and front-to-back
// compositing Col = sum_i col_i alpha_i prod_{j<i} (1 - alpha_j).
//
// Pipeline (one stream, scratch from the stream-ordered allocator):
//   1. per Gaussian: camera position, projected covariance dilated by 0.3,
//      its inverse (conic), the 3-sigma square and the 16x16 tiles it
//      touches;
//   2. the Gaussians sorted by depth, a positive float, whose bit pattern
//      orders like its value (stable LSD radix sort, three 11-bit digits);
//   3. in that order one entry per touched tile, stably sorted by the tile (one
//      or two digits), and per tile the range of its entries.  Sorting by depth
//      first moves 300k 8-byte pairs three times and the 600k to 900k entries
//      twice, where (tile, depth) keys moved 12 bytes of every entry six times;
//   4. one CTA per tile, one thread per pixel: the tile's Gaussians are
//      composited front to back; a pixel stops once its transmittance would
//      drop below 1e-4, a warp once all its pixels have.
// Conventions where the paper defers to 3DGS: Gaussians nearer than 0.2 are
// not drawn; alpha = min(0.99, o exp(power)), skipped below 1/255 or for
// power > 0; the background is added with the remaining transmittance.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <string>
#include <utility>

#include "../../include/mpm.h"
#include "mpm_ptr.h"
#include "mpm_scan.cuh"
#include "mpm_scratch.h"

namespace {

thread_local std::string g_render_msg;
constexpr int TS = 16;            // tile edge in pixels
constexpr int RS_THREADS = 256;   // radix sort: threads per CTA
constexpr int RS_ITEMS = 8;       // pairs per thread per CTA tile
constexpr int RS_BITS = 11;       // largest digit: 8 KB of bases and 32 KB of counters
constexpr int RS_TILE = RS_THREADS * RS_ITEMS;

struct Cam {
    float R[9], T[3];
    float fx, fy, cx, cy;
    int W, H, gx, gy;
};

// 1. projection per Gaussian
// g: three words per Gaussian, u v and the conic's xx xy | its yy, opacity,
// depth, reach (two halves) | colour
__global__ void k_rd_pre(long long n, const float *mean, const float *cov, const float *color, const float *opac, Cam c,
                         float4 *g, int4 *rect, unsigned *cnt, unsigned *depth) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        cnt[i] = 0;
        depth[i] = 0xffffffffu;   // not drawn: behind all others
        const float px = mean[3 * i], py = mean[3 * i + 1], pz = mean[3 * i + 2];
        const float tx = c.R[0] * px + c.R[1] * py + c.R[2] * pz + c.T[0];
        const float ty = c.R[3] * px + c.R[4] * py + c.R[5] * pz + c.T[1];
        // the depth orders the compositing: rounded operation by operation in a
        // fixed order (no contraction), so that its value does not depend on
        // the compiler
        const float tz = __fadd_rn(__fadd_rn(__fadd_rn(__fmul_rn(c.R[6], px), __fmul_rn(c.R[7], py)),
                                             __fmul_rn(c.R[8], pz)), c.T[2]);
        if (!(tz > 0.2f)) continue;
        const float *s = cov + 6 * i;
        const float S[9] = {s[0], s[1], s[2], s[1], s[3], s[4], s[2], s[4], s[5]};
        float WS[9], Sc[9];
        for (int r = 0; r < 3; ++r)
            for (int q = 0; q < 3; ++q)
                WS[3 * r + q] = c.R[3 * r] * S[q] + c.R[3 * r + 1] * S[3 + q] + c.R[3 * r + 2] * S[6 + q];
        for (int r = 0; r < 3; ++r)
            for (int q = 0; q < 3; ++q)
                Sc[3 * r + q] = WS[3 * r] * c.R[3 * q] + WS[3 * r + 1] * c.R[3 * q + 1] + WS[3 * r + 2] * c.R[3 * q + 2];
        const float iz = 1.f / tz;
        const float J[6] = {c.fx * iz, 0.f, -c.fx * tx * iz * iz, 0.f, c.fy * iz, -c.fy * ty * iz * iz};
        float JS[6];
        for (int r = 0; r < 2; ++r)
            for (int q = 0; q < 3; ++q) JS[3 * r + q] = J[3 * r] * Sc[q] + J[3 * r + 1] * Sc[3 + q] + J[3 * r + 2] * Sc[6 + q];
        const float a = JS[0] * J[0] + JS[1] * J[1] + JS[2] * J[2] + 0.3f;
        const float b = JS[0] * J[3] + JS[1] * J[4] + JS[2] * J[5];
        const float d = JS[3] * J[3] + JS[4] * J[4] + JS[5] * J[5] + 0.3f;
        const float det = a * d - b * b;
        if (!(det > 0.f)) continue;
        const float mid = 0.5f * (a + d), disc = sqrtf(fmaxf(0.1f, mid * mid - det));
        const float rad = ceilf(3.f * sqrtf(fmaxf(mid + disc, mid - disc)));
        const float u = c.fx * tx * iz + c.cx, v = c.fy * ty * iz + c.cy;
        int x0 = (int)fminf((float)c.gx, fmaxf(0.f, floorf((u - rad) / TS)));
        int x1 = (int)fminf((float)c.gx, fmaxf(0.f, floorf((u + rad + TS - 1) / TS)));
        int y0 = (int)fminf((float)c.gy, fmaxf(0.f, floorf((v - rad) / TS)));
        int y1 = (int)fminf((float)c.gy, fmaxf(0.f, floorf((v + rad + TS - 1) / TS)));
        if (x1 <= x0 || y1 <= y0) continue;
        // Where alpha stays below 1/255 the Gaussian has no effect: beyond
        // |dx| = sqrt(2 ln(255 o) Sigma'_xx), and alike in y.  The compositing
        // skips it there; tiles wholly there get no key.  The reach is taken 1%
        // and 0.05 larger in the exponent, far above the rounding of the
        // exponent computed per pixel, which grows with the condition number of
        // Sigma' (relative 6e-8 times it); beyond 1e5 nothing is left out.
        const float o = opac[i];
        if (o < 1.f / 255.f) continue;
        const float q2 = 2.02f * logf(255.f * o) + 0.1f, cond = (a + d) * (a + d) / det;
        const bool known = cond <= 1e5f && q2 < INFINITY;     // (a NaN opacity composites with alpha 0.99)
        const float rx = known ? sqrtf(q2 * a) + 0.01f : INFINITY, ry = known ? sqrtf(q2 * d) + 0.01f : INFINITY;
        // pixel centres of tile t: 16 t + 0.5 .. 16 t + 15.5
        x0 = (int)fmaxf((float)x0, ceilf((u - rx - (TS - 0.4f)) / TS));
        x1 = (int)fminf((float)x1, floorf((u + rx - 0.4f) / TS) + 1.f);
        y0 = (int)fmaxf((float)y0, ceilf((v - ry - (TS - 0.4f)) / TS));
        y1 = (int)fminf((float)y1, floorf((v + ry - 0.4f) / TS) + 1.f);
        if (x1 <= x0 || y1 <= y0) continue;
        const float idet = 1.f / det;
        g[3 * i] = make_float4(u, v, d * idet, -b * idet);
        const __half2 reach = __halves2half2(__float2half_ru(rx), __float2half_ru(ry));
        g[3 * i + 2] = make_float4(color[3 * i], color[3 * i + 1], color[3 * i + 2], 0.f);
        g[3 * i + 1] = make_float4(a * idet, o, tz, __uint_as_float(*reinterpret_cast<const unsigned *>(&reach)));
        rect[i] = make_int4(x0, x1, y0, y1);
        depth[i] = __float_as_uint(tz);
        cnt[i] = (unsigned)((x1 - x0) * (y1 - y0));
    }
}


// 3. one entry per touched tile, Gaussians in depth order
__global__ void k_rd_dup(long long n, const unsigned *order, const int4 *rect, const unsigned *cnt, const unsigned *off,
                         const unsigned long long *btot, int gx, unsigned *tile, unsigned *vals) {
    for (long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x; s < n;
         s += (long long)gridDim.x * blockDim.x) {
        const unsigned i = order[s];
        if (cnt[i] == 0) continue;
        const int4 r = rect[i];
        unsigned o = scanned(off, btot, s);
        for (int y = r.z; y < r.w; ++y)
            for (int x = r.x; x < r.y; ++x) {
                tile[o] = (unsigned)(y * gx + x);
                vals[o] = i;
                ++o;
            }
    }
}

// Stable radix sort of (key, value) pairs by digits of up to RS_BITS bits.  A
// CTA takes RS_TILE pairs, each warp a contiguous part of them.
// Histogram: hist[digit * nblocks + block]
__global__ void __launch_bounds__(RS_THREADS) k_rs_hist(const unsigned *keys, long long n, int shift, int bits,
                                                          unsigned *hist, int nblocks) {
    extern __shared__ unsigned rs_mem[];
    const int bins = 1 << bits;
    for (int d = threadIdx.x; d < bins; d += RS_THREADS) rs_mem[d] = 0;
    __syncthreads();
    const long long base = (long long)blockIdx.x * RS_TILE;
    for (int j = 0; j < RS_ITEMS; ++j) {
        const long long i = base + j * RS_THREADS + threadIdx.x;
        if (i < n) atomicAdd(&rs_mem[(keys[i] >> shift) & (bins - 1)], 1u);
    }
    __syncthreads();
    for (int d = threadIdx.x; d < bins; d += RS_THREADS) hist[(long long)d * nblocks + blockIdx.x] = rs_mem[d];
}

// Stable scatter.  vals == NULL: the value is the index.  Each warp ranks its
// pairs by digit with its own counters in shared memory (a warp's lanes of one
// digit by their order), then the counters of the warps are summed per digit.
__global__ void __launch_bounds__(RS_THREADS) k_rs_scatter(const unsigned *keys, const unsigned *vals, long long n,
                                                             int shift, int bits, const unsigned *hoff,
                                                             const unsigned long long *hbt, int nblocks,
                                                             unsigned *okeys, unsigned *ovals) {
    extern __shared__ unsigned rs_mem[];
    const int bins = 1 << bits;
    unsigned *base = rs_mem;                                             // bins: first output of the digit
    unsigned short *cnt = reinterpret_cast<unsigned short *>(rs_mem + bins);   // warps x bins
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    constexpr int WARPS = RS_THREADS / 32;
    unsigned *cnt32 = rs_mem + bins;
    for (int q = threadIdx.x; q < WARPS * bins / 2; q += RS_THREADS) cnt32[q] = 0;
    __syncthreads();
    unsigned short *mine = cnt + w * bins;
    const long long first = (long long)blockIdx.x * RS_TILE + w * (RS_TILE / WARPS);
    unsigned key[RS_ITEMS], rank[RS_ITEMS];
#pragma unroll
    for (int j = 0; j < RS_ITEMS; ++j) {
        const long long i = first + j * 32 + lane;
        key[j] = i < n ? keys[i] : 0u;
    }
#pragma unroll
    for (int j = 0; j < RS_ITEMS; ++j) {
        const long long i = first + j * 32 + lane;
        const unsigned d = i < n ? (key[j] >> shift) & (bins - 1) : (unsigned)bins;   // bins: no pair
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        const unsigned lt = peers & ((1u << lane) - 1u);
        unsigned before = 0;
        if (i < n) before = mine[d];
        __syncwarp();
        if (i < n && lt == 0) mine[d] = (unsigned short)(before + __popc(peers));
        __syncwarp();
        rank[j] = before + __popc(lt);
    }
    __syncthreads();
    for (int d = threadIdx.x; d < bins; d += RS_THREADS) {
        base[d] = scanned(hoff, hbt, (long long)d * nblocks + blockIdx.x);
        unsigned sum = 0;
#pragma unroll
        for (int q = 0; q < WARPS; ++q) {
            const unsigned t = cnt[q * bins + d];
            cnt[q * bins + d] = (unsigned short)sum;
            sum += t;
        }
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < RS_ITEMS; ++j) {
        const long long i = first + j * 32 + lane;
        if (i < n) {
            const unsigned d = (key[j] >> shift) & (bins - 1);
            const unsigned pos = base[d] + mine[d] + rank[j];
            okeys[pos] = key[j];
            ovals[pos] = vals ? vals[i] : (unsigned)i;
        }
    }
}

// per tile the range [start, end) of its sorted entries
__global__ void k_rd_ranges(const unsigned *tile, long long n, uint2 *ranges) {
    for (long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x; s < n;
         s += (long long)gridDim.x * blockDim.x) {
        const unsigned t = tile[s];
        if (s == 0 || tile[s - 1] != t) ranges[t].x = (unsigned)s;
        if (s == n - 1 || tile[s + 1] != t) ranges[t].y = (unsigned)(s + 1);
    }
}

// 4. compositing, one CTA per tile, one pixel per thread, an 8 x 4 pixel patch
// per warp.  Each warp walks the tile's list by itself, 32 Gaussians at a time
// (the next 32 are read meanwhile): those that reach its patch are put side by
// side in shared memory and composited in order, HITS at a time.  The warps do
// not wait for one another, and one whose pixels are all done leaves.
//
// What bounds it: the longest lists, one dependent chain per warp (a dense
// object's tile holds thousands of Gaussians a few pixels wide, 80 to 90% of
// which miss a given patch).  300k Gaussians at 1024 x 768: 481 us with every
// pixel looking at every Gaussian of its tile, 278 with the test per patch, 204
// with HITS 4 in a double-buffered CTA-wide batch, 143 as it is.
constexpr int HITS = 4;
__global__ void __launch_bounds__(TS * TS) k_rd_blend(Cam c, const uint2 *ranges, const unsigned *vals, const float4 *g,
                                                      float bg0, float bg1, float bg2, float *img, float *trans) {
    __shared__ float4 hit_s[TS * TS / 32][3][32];
    const int tile = blockIdx.x, tx = tile % c.gx, ty = tile / c.gx;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int qx = tx * TS + (warp & 1) * 8, qy = ty * TS + (warp >> 1) * 4;   // the warp's patch
    const int px = qx + (lane & 7), py = qy + (lane >> 3);
    const bool inside = px < c.W && py < c.H;
    const uint2 r = ranges[tile];
    float T = 1.f, C0 = 0.f, C1 = 0.f, C2 = 0.f;
    bool done = !inside;
    const float fx = (float)px + 0.5f, fy = (float)py + 0.5f;
    const float mx = (float)qx + 4.f, my = (float)qy + 2.f;                    // its centre
    float4 (*S)[32] = hit_s[warp];
    // Gaussian of list entry s + lane, read one group ahead; its index two ahead
    const float4 none = make_float4(0.f, 0.f, 0.f, 0.f);
    float4 a = none, e = none, k = none;
    auto read = [&](unsigned s, unsigned i) {
        if (s + lane < r.y) {
            const float4 *p = g + 3 * (size_t)i;
            a = p[0];
            e = p[1];
            k = p[2];
        }
    };
    auto index = [&](unsigned s) { return s + lane < r.y ? vals[s + lane] : 0u; };
    unsigned next = 0;
    if (r.x < r.y) {
        read(r.x, index(r.x));
        next = index(r.x + 32);
    }
    for (unsigned b = r.x; b < r.y; b += 32) {
        if (__all_sync(0xffffffffu, done)) break;
        const unsigned w = __float_as_uint(e.w);
        const float2 reach = __half22float2(*reinterpret_cast<const __half2 *>(&w));
        const bool hit = b + lane < r.y && fabsf(a.x - mx) <= reach.x + 3.51f && fabsf(a.y - my) <= reach.y + 1.51f;
        const unsigned hits = __ballot_sync(0xffffffffu, hit);
        __syncwarp();
        if (hit) {
            const int at = __popc(hits & ((1u << lane) - 1u));
            S[0][at] = a;
            S[1][at] = e;
            S[2][at] = k;
        }
        __syncwarp();
        read(b + 32, next);
        next = index(b + 64);
        const int n = __popc(hits);
        for (int q = 0; q < n; q += HITS) {
            float alpha[HITS];
#pragma unroll
            for (int h = 0; h < HITS; ++h) {
                const float4 ga = S[0][min(q + h, 31)], ge = S[1][min(q + h, 31)];
                const float dx = fx - ga.x, dy = fy - ga.y;
                const float power = -0.5f * (ga.z * dx * dx + ge.x * dy * dy) - ga.w * dx * dy;
                alpha[h] = fminf(0.99f, ge.y * expf(power));
                if (q + h >= n || power > 0.f) alpha[h] = 0.f;
            }
#pragma unroll
            for (int h = 0; h < HITS; ++h) {
                if (done || alpha[h] < 1.f / 255.f) continue;
                const float tt = T * (1.f - alpha[h]);
                if (tt < 1e-4f) { done = true; continue; }
                const float4 gk = S[2][q + h];
                C0 += gk.x * alpha[h] * T;
                C1 += gk.y * alpha[h] * T;
                C2 += gk.z * alpha[h] * T;
                T = tt;
            }
        }
    }
    if (inside) {
        float *o = img + 3 * ((size_t)py * c.W + px);
        o[0] = C0 + T * bg0;
        o[1] = C1 + T * bg1;
        o[2] = C2 + T * bg2;
        if (trans) trans[(size_t)py * c.W + px] = T;
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

extern "C" MPM_API mpm_status mpm_render(int64_t n, const float *mean, const float *cov, const float *color,
                                         const float *opacity, const float view[12], float fx, float fy, float cx,
                                         float cy, int32_t width, int32_t height, const float bg[3], float *image,
                                         float *trans, void *stream) {
    g_render_msg.clear();
    if (n < 0 || (n > 0 && (!mean || !cov || !color || !opacity)) || !view || !bg || !image || width < 1 ||
        height < 1 || width > 16384 || height > 16384 || n >= (1ll << 31)) {
        g_render_msg = "render: bad arguments";
        return MPM_ERR_INVALID_ARG;
    }
    if (mpm::any_on_other_device({mean, cov, color, opacity, image, trans})) {
        g_render_msg = "render: an array lives on another device than the current one";
        return MPM_ERR_INVALID_ARG;
    }
    cudaStream_t st = (cudaStream_t)stream;
    Cam c;
    for (int r = 0; r < 3; ++r) {
        for (int q = 0; q < 3; ++q) c.R[3 * r + q] = view[4 * r + q];
        c.T[r] = view[4 * r + 3];
    }
    c.fx = fx; c.fy = fy; c.cx = cx; c.cy = cy;
    c.W = width; c.H = height;
    c.gx = (width + TS - 1) / TS;
    c.gy = (height + TS - 1) / TS;
    const long long tiles = (long long)c.gx * c.gy;
    int tile_bits = 0;
    while ((1ll << tile_bits) < tiles) ++tile_bits;
    const long long npix = (long long)width * height;
    auto al = [](size_t b) { return (b + 255) & ~size_t(255); };
    mpm_status status = MPM_OK;
    char *buf = nullptr, *kbuf = nullptr;
    unsigned long long total = 0;
#define RD_CK(call)                                                                   \
    do {                                                                              \
        if ((call) != cudaSuccess) {                                                  \
            g_render_msg = std::string("render: ") + cudaGetErrorString(cudaGetLastError()); \
            status = MPM_ERR_CUDA;                                                    \
            goto done;                                                                \
        }                                                                             \
    } while (0)
    {
        size_t off = 0;
        const size_t o_mean = off; off += al(n * 12);
        const size_t o_cov = off; off += al(n * 24);
        const size_t o_col = off; off += al(n * 12);
        const size_t o_op = off; off += al(n * 4);
        const size_t o_g = off; off += al(n * 48);
        const size_t o_rect = off; off += al(n * 16);
        const size_t o_cnt = off; off += al(n * 4);
        const size_t o_off = off; off += al(n * 4);
        size_t o_sort[4];   // depth keys and order, each twice
        for (size_t &o : o_sort) { o = off; off += al(n * 4); }
        const int nb_d = (int)((n + RS_TILE - 1) / RS_TILE);
        const size_t o_h = off; off += al((size_t)(1 << RS_BITS) * nb_d * 4);
        const size_t o_ho = off; off += al((size_t)(1 << RS_BITS) * nb_d * 4);
        const size_t o_bt = off; off += al(scan_words(std::max<long long>(n, (long long)(1 << RS_BITS) * nb_d)) * 8);
        const size_t o_ht = off; off += al(8);
        // cleared together: the tiles' ranges, the entry count, the scans' ticket
        const size_t o_rng = off; off += al(tiles * 8);
        const size_t o_tot = off; off += al(8);
        const size_t o_tick = off; off += al(4);
        const size_t o_clear = off;
        const size_t o_img = off; off += al(npix * 12);
        const size_t o_tr = off; off += al(npix * 4);
        if (mpm::scratch_alloc((void **)&buf, off, st) != cudaSuccess) {
            cudaGetLastError();
            buf = nullptr;
            g_render_msg = "render: device allocation failed";
            return MPM_ERR_OOM;
        }
        auto P = [&](size_t o) { return (void *)(buf + o); };
        const float *dmean = mean, *dcov = cov, *dcol = color, *dop = opacity;
        if (n > 0 && !is_dev(mean)) { RD_CK(cudaMemcpyAsync(P(o_mean), mean, n * 12, cudaMemcpyHostToDevice, st)); dmean = (const float *)P(o_mean); }
        if (n > 0 && !is_dev(cov)) { RD_CK(cudaMemcpyAsync(P(o_cov), cov, n * 24, cudaMemcpyHostToDevice, st)); dcov = (const float *)P(o_cov); }
        if (n > 0 && !is_dev(color)) { RD_CK(cudaMemcpyAsync(P(o_col), color, n * 12, cudaMemcpyHostToDevice, st)); dcol = (const float *)P(o_col); }
        if (n > 0 && !is_dev(opacity)) { RD_CK(cudaMemcpyAsync(P(o_op), opacity, n * 4, cudaMemcpyHostToDevice, st)); dop = (const float *)P(o_op); }
        float4 *g = (float4 *)P(o_g);
        int4 *rect = (int4 *)P(o_rect);
        unsigned *cnt = (unsigned *)P(o_cnt), *offs = (unsigned *)P(o_off);
        unsigned long long *dtot = (unsigned long long *)P(o_tot);
        uint2 *ranges = (uint2 *)P(o_rng);
        unsigned *ticket = (unsigned *)P(o_tick);
        unsigned long long *bt = (unsigned long long *)P(o_bt), *ht = (unsigned long long *)P(o_ht);
        RD_CK(cudaMemsetAsync(ranges, 0, o_clear - o_rng, st));
        // one pass of the radix sort: from (ka, va) to (kb, vb)
        auto sort_pass = [&](const unsigned *ka, const unsigned *va, unsigned *kb, unsigned *vb, long long m, int shift,
                             int bits, unsigned *h, unsigned *ho, unsigned long long *hb) {
            const int nb = (int)((m + RS_TILE - 1) / RS_TILE);
            const size_t bins = (size_t)1 << bits;
            k_rs_hist<<<nb, RS_THREADS, bins * 4, st>>>(ka, m, shift, bits, h, nb);
            scan_blocks(h, nullptr, ho, (long long)bins * nb, hb, ht, ticket, st);
            k_rs_scatter<<<nb, RS_THREADS, bins * 4 + (RS_THREADS / 32) * bins * 2, st>>>(ka, va, m, shift, bits, ho, hb, nb,
                                                                                         kb, vb);
        };
        unsigned *dk[2] = {(unsigned *)P(o_sort[0]), (unsigned *)P(o_sort[1])};
        unsigned *dv[2] = {(unsigned *)P(o_sort[2]), (unsigned *)P(o_sort[3])};
        if (n > 0) {
            k_rd_pre<<<blocks_for(n, 256), 256, 0, st>>>(n, dmean, dcov, dcol, dop, c, g, rect, cnt, dk[0]);
            for (int p = 0; p < 3; ++p)
                sort_pass(dk[p & 1], p ? dv[p & 1] : nullptr, dk[(p & 1) ^ 1], dv[(p & 1) ^ 1], n, 11 * p, p < 2 ? 11 : 10,
                          (unsigned *)P(o_h), (unsigned *)P(o_ho), bt);
            scan_blocks(cnt, dv[1], offs, n, bt, dtot, ticket, st);
            RD_CK(cudaGetLastError());
            RD_CK(cudaMemcpyAsync(&total, dtot, 8, cudaMemcpyDeviceToHost, st));
            RD_CK(cudaStreamSynchronize(st));
        }
        if (total >= (1ull << 32)) { g_render_msg = "render: too many tile overlaps"; status = MPM_ERR_CAPACITY; goto done; }
        if (total > 0) {
            const long long nk = (long long)total;
            const int nb = (int)((nk + RS_TILE - 1) / RS_TILE);
            // the tile's digits: one of up to RS_BITS bits, or two halves
            const int passes = tile_bits <= RS_BITS ? 1 : 2, bits = std::max(1, (tile_bits + passes - 1) / passes);
            const long long hn = (long long)nb << bits;
            size_t ko = 0;
            size_t o_e[4];   // tiles and Gaussians of the entries, each twice
            for (size_t &o : o_e) { o = ko; ko += al(nk * 4); }
            const size_t o_eh = ko; ko += al(hn * 4);
            const size_t o_eho = ko; ko += al(hn * 4);
            const size_t o_ehb = ko; ko += al(scan_words(hn) * 8);
            if (mpm::scratch_alloc((void **)&kbuf, ko, st) != cudaSuccess) {
                cudaGetLastError();
                kbuf = nullptr;
                g_render_msg = "render: device allocation failed";
                status = MPM_ERR_OOM;
                goto done;
            }
            auto E = [&](size_t o) { return (unsigned *)(kbuf + o); };
            unsigned *k0 = E(o_e[0]), *k1 = E(o_e[1]), *v0 = E(o_e[2]), *v1 = E(o_e[3]);
            k_rd_dup<<<blocks_for(n, 256), 256, 0, st>>>(n, dv[1], rect, cnt, offs, bt, c.gx, k0, v0);
            RD_CK(cudaGetLastError());
            for (int p = 0; p < passes; ++p) {
                sort_pass(k0, v0, k1, v1, nk, p * bits, bits, E(o_eh), E(o_eho), (unsigned long long *)(kbuf + o_ehb));
                RD_CK(cudaGetLastError());
                std::swap(k0, k1);
                std::swap(v0, v1);
            }
            k_rd_ranges<<<blocks_for(nk, 256), 256, 0, st>>>(k0, nk, ranges);
            RD_CK(cudaGetLastError());
            float *dimg = is_dev(image) ? image : (float *)P(o_img);
            float *dtr = trans ? (is_dev(trans) ? trans : (float *)P(o_tr)) : nullptr;
            k_rd_blend<<<(unsigned)tiles, TS * TS, 0, st>>>(c, ranges, v0, g, bg[0], bg[1], bg[2], dimg, dtr);
            RD_CK(cudaGetLastError());
            if (dimg != image) RD_CK(cudaMemcpyAsync(image, dimg, npix * 12, cudaMemcpyDeviceToHost, st));
            if (trans && dtr != trans) RD_CK(cudaMemcpyAsync(trans, dtr, npix * 4, cudaMemcpyDeviceToHost, st));
        } else {
            // nothing visible: the background everywhere
            float *dimg = is_dev(image) ? image : (float *)P(o_img);
            float *dtr = trans ? (is_dev(trans) ? trans : (float *)P(o_tr)) : nullptr;
            k_rd_blend<<<(unsigned)tiles, TS * TS, 0, st>>>(c, ranges, nullptr, g, bg[0], bg[1], bg[2], dimg, dtr);
            RD_CK(cudaGetLastError());
            if (dimg != image) RD_CK(cudaMemcpyAsync(image, dimg, npix * 12, cudaMemcpyDeviceToHost, st));
            if (trans && dtr != trans) RD_CK(cudaMemcpyAsync(trans, dtr, npix * 4, cudaMemcpyDeviceToHost, st));
        }
    }
done:
    if (kbuf) cudaFreeAsync(kbuf, st);
    if (buf) cudaFreeAsync(buf, st);
    if (status == MPM_OK && cudaStreamSynchronize(st) != cudaSuccess) {
        g_render_msg = std::string("render: ") + cudaGetErrorString(cudaGetLastError());
        status = MPM_ERR_CUDA;
    }
#undef RD_CK
    return status;
}

extern "C" MPM_API const char *mpm_render_last_error(void) { return g_render_msg.c_str(); }
