// mpm_scan.cuh -- exclusive scan of unsigned counts over many CTAs, shared
// by the splatting and MCIS translation units (internal linkage in each).
#pragma once
#include <cuda_runtime.h>

namespace {

// Exclusive scan of n unsigned counts over many CTAs.  Each CTA scans its SC_N
// counts and stores their sum; the last CTA to finish scans the sums (exclusive,
// in place) and writes the grand total, so that the scan is one launch.  A CTA's
// offset, its scanned sum, is added by a second launch (scan_counts) or by the
// kernel that reads the scan (scan_blocks, scanned).
constexpr int SC_T = 1024;            // threads per CTA
constexpr int SC_V = 4;               // consecutive counts per thread
constexpr int SC_N = SC_T * SC_V;
__device__ __forceinline__ unsigned long long block_exclusive_scan(unsigned long long v, unsigned long long &tot) {
    __shared__ unsigned long long sh[SC_T / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    unsigned long long x = v;
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sh[w] = x;
    __syncthreads();
    if (w == 0) {
        unsigned long long t = lane < (int)(blockDim.x >> 5) ? sh[lane] : 0ull;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        sh[lane] = t;
    }
    __syncthreads();
    const unsigned long long ex = (w > 0 ? sh[w - 1] : 0ull) + x - v;
    tot = sh[(blockDim.x >> 5) - 1];
    __syncthreads();
    return ex;
}
// order (nullable): count i is in[order[i]].  ticket: zero before the launch, and after it.
__global__ void __launch_bounds__(SC_T) k_sc_block(const unsigned *in, const unsigned *order, unsigned *out, long long n,
                                                   unsigned long long *btot, unsigned long long *total,
                                                   unsigned *ticket) {
    const long long i0 = blockIdx.x * (long long)SC_N + threadIdx.x * SC_V;
    unsigned v[SC_V];
    unsigned long long sum = 0;
#pragma unroll
    for (int u = 0; u < SC_V; ++u) {
        v[u] = i0 + u < n ? in[order ? order[i0 + u] : i0 + u] : 0u;
        sum += v[u];
    }
    unsigned long long tot;
    unsigned long long ex = block_exclusive_scan(sum, tot);
#pragma unroll
    for (int u = 0; u < SC_V; ++u) {
        if (i0 + u < n) out[i0 + u] = (unsigned)ex;
        ex += v[u];
    }
    __shared__ bool last;
    if (threadIdx.x == 0) {
        btot[blockIdx.x] = tot;
        __threadfence();
        last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    unsigned long long carry = 0;
    for (long long b0 = 0; b0 < gridDim.x; b0 += SC_T) {
        const long long i = b0 + threadIdx.x;
        const unsigned long long x = i < gridDim.x ? __ldcg(&btot[i]) : 0ull;
        unsigned long long t;
        const unsigned long long e = block_exclusive_scan(x, t);
        if (i < gridDim.x) btot[i] = carry + e;
        carry += t;
    }
    if (threadIdx.x == 0) {
        *total = carry;
        *ticket = 0;
    }
}
__global__ void __launch_bounds__(SC_T) k_sc_add(unsigned *out, long long n, const unsigned long long *btot) {
    for (long long i = blockIdx.x * (long long)SC_N + threadIdx.x; i < min(n, (blockIdx.x + 1) * (long long)SC_N); i += SC_T)
        out[i] += (unsigned)btot[blockIdx.x];
}

// 64-bit scratch words for the block sums of a scan of up to n counts
inline long long scan_words(long long n) { return (n + SC_N - 1) / SC_N + 1; }
// the scan without the CTAs' offsets: count i's prefix is out[i] + btot[i / SC_N] (scanned)
inline void scan_blocks(const unsigned *in, const unsigned *order, unsigned *out, long long n, unsigned long long *btot,
                        unsigned long long *total, unsigned *ticket, cudaStream_t st) {
    if (n > 0) k_sc_block<<<(unsigned)((n + SC_N - 1) / SC_N), SC_T, 0, st>>>(in, order, out, n, btot, total, ticket);
}
__device__ __forceinline__ unsigned scanned(const unsigned *out, const unsigned long long *btot, long long i) {
    return out[i] + (unsigned)btot[i / SC_N];
}
// exclusive scan of n counts into out (sums below 2^32), grand total to *total
// (unchanged for n = 0); btot: scan_words(n) scratch words; ticket: one zero word, left zero
inline void scan_counts(const unsigned *in, unsigned *out, long long n, unsigned long long *btot,
                        unsigned long long *total, unsigned *ticket, cudaStream_t st) {
    scan_blocks(in, nullptr, out, n, btot, total, ticket, st);
    if (n > SC_N) k_sc_add<<<(unsigned)((n + SC_N - 1) / SC_N), SC_T, 0, st>>>(out, n, btot);
}

}  // namespace
