// Depth-jump filter (section "Numerical stability", eqs. (dstab), (newdw), (newdc)), in FP64;
// shared by cliffs_set_bathy and cliffs_depth_filter_noalloc so that both launch the same code.
//
// A pass is a Jacobi pass along rows, then one along columns; one kernel does both, tile by
// tile in shared memory. Passes are launched several at a time, each noting whether it
// changed anything in a flag of its own; one that follows a pass without a change returns at
// once, so the host reads the flags once per group and not once per pass (129 x 269 nodes:
// 199 -> 106 us, most of it that round trip). The first groups are short: a depth that is smooth
// enough already takes one pass, rough relief five or six.
#pragma once
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

namespace cliffs {

constexpr int FILTER_PASSES = 100;                 // at most

// FP64 runs at a small fraction of the integer rate here, so the tests that nearly every node
// passes are made on the bits: d > 0, and "l < 2^e dj", which rules l > alpha^2 dj out
// (2^e <= alpha^2, e20 = e << 20; adding it to the high word of a normal number multiplies by
// 2^e).
__device__ __forceinline__ bool filter_pos(double d) {
    const long long b = __double_as_longlong(d);
    return b > 0 && b <= 0x7ff0000000000000LL;
}
__device__ __forceinline__ bool filter_deeper(double l, double dj, double a2, int e20) {
    const int hl = __double2hiint(l), hd = __double2hiint(dj);
    if (hd >= 0x100000 && hl - hd < e20) return false;
    return l > a2 * dj;
}
// Whether a node changes: wet, with a wet neighbour along the line deeper than alpha^2 d_j.
__device__ __forceinline__ bool filter_violates(double dj, double l, double r, bool hl, bool hr, double a2, int e20) {
    return filter_pos(dj) && ((hl && filter_pos(l) && filter_deeper(l, dj, a2, e20)) ||
                              (hr && filter_pos(r) && filter_deeper(r, dj, a2, e20)));
}
// What it changes to: the square of the mean square root of its two neighbours (open water) or
// the coastal neighbour's depth over alpha^2.
__device__ __forceinline__ double filter_value(double l, double r, bool hl, bool hr, double a2) {
    const bool lw = hl && filter_pos(l), rw = hr && filter_pos(r);
    if (lw && rw) {
        const double s = sqrt(l) + sqrt(r);
        return s * s / 4.0;
    }
    return (lw ? l : r) / a2;
}

// wet nodes (0 < d < min_depth) raised to min_depth; in may be out. Clears the passes' flags.
static __global__ void k_filter_raise(const double* in, double* out, long long n, double min_depth, int* flags) {
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (blockIdx.x == 0 && threadIdx.x < FILTER_PASSES) flags[threadIdx.x] = 0;
    if (i >= n) return;
    const double d = in[i];
    out[i] = (d > 0.0 && d < min_depth) ? min_depth : d;
}

// Pass p (from 0): in -> out; changed[p] is set when a node changed. A block filters 32 x 32
// nodes (34 rows along x). The nodes that change are few but scattered, and a square root in
// FP64 costs a warp the same for one lane as for 32, so they are first listed and then
// computed by consecutive threads (1000 x 1000 nodes of rough relief, 5 passes: 378 us without the list).
constexpr int FILTER_TILE = 32;
static __global__ void __launch_bounds__(256) k_filter_pass(const double* __restrict__ in, double* __restrict__ out,
                                                            int nx, int ny, double a2, int e20, int* changed, int p) {
    if (p > 0 && changed[p - 1] == 0) return;        // done: both buffers hold the result
    __shared__ double T[FILTER_TILE + 2][FILTER_TILE];   // rows r0-1 .. r0+32 after the pass along x
    __shared__ short list[(FILTER_TILE + 2) * FILTER_TILE];
    __shared__ int count[2];
    // tiles are numbered along x first, in one grid dimension: a line along y has too many for the second
    const unsigned across = (unsigned)(nx + FILTER_TILE - 1) / FILTER_TILE;
    const int c0 = (int)(blockIdx.x % across) * FILTER_TILE, r0 = (int)(blockIdx.x / across) * FILTER_TILE;
    bool any = false;
    if (threadIdx.x < 2) count[threadIdx.x] = 0;
    __syncthreads();
    const int c = c0 + (threadIdx.x & 31);
    for (int i = threadIdx.x; i < (FILTER_TILE + 2) * FILTER_TILE; i += 256) {
        const int r = r0 - 1 + (i >> 5);
        if (r < 0 || r >= ny || c >= nx) continue;
        const double* d = in + (long long)r * nx + c;
        const bool hl = c > 0, hr = c < nx - 1;
        const double dj = *d;
        T[i >> 5][i & 31] = dj;
        any |= (__double_as_longlong(dj) & 0x7fffffffffffffffLL) > 0x7ff0000000000000LL;   // a NaN differs from itself
        if (nx >= 3 && filter_violates(dj, hl ? d[-1] : 0.0, hr ? d[1] : 0.0, hl, hr, a2, e20))
            list[atomicAdd(&count[0], 1)] = (short)i;
    }
    __syncthreads();
    for (int k = threadIdx.x; k < count[0]; k += 256) {
        const int i = list[k], q = c0 + (i & 31);
        const double* d = in + (long long)(r0 - 1 + (i >> 5)) * nx + q;
        const bool hl = q > 0, hr = q < nx - 1;
        T[i >> 5][i & 31] = filter_value(hl ? d[-1] : 0.0, hr ? d[1] : 0.0, hl, hr, a2);
        any |= (i >> 5) >= 1 && (i >> 5) <= FILTER_TILE;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < FILTER_TILE * FILTER_TILE; i += 256) {
        const int t = (i >> 5) + 1, r = r0 + (i >> 5);
        if (r >= ny || c >= nx) continue;
        const double dj = T[t][i & 31];
        const bool hu = r > 0, hd = r < ny - 1;
        if (ny >= 3 && filter_violates(dj, hu ? T[t - 1][i & 31] : 0.0, hd ? T[t + 1][i & 31] : 0.0, hu, hd, a2, e20))
            list[atomicAdd(&count[1], 1)] = (short)i;
        else
            out[(long long)r * nx + c] = dj;
    }
    __syncthreads();
    for (int k = threadIdx.x; k < count[1]; k += 256) {
        const int i = list[k], t = (i >> 5) + 1, r = r0 + (i >> 5);
        const bool hu = r > 0, hd = r < ny - 1;
        out[(long long)r * nx + c0 + (i & 31)] =
            filter_value(hu ? T[t - 1][i & 31] : 0.0, hd ? T[t + 1][i & 31] : 0.0, hu, hd, a2);
        any = true;
    }
    if (any) changed[p] = 1;
}

// Filter d (k_filter_raise's output in blocks of 256, which cleared the flags) to a fixed point, with
// tmp as the second buffer and flags[100] on the device. Writes the passes made (-1: stopped at
// 100), the result is in d. Waits for the stream once per group of 2, 4, 8, .. passes: with a first
// group of 8 a 200^2 grid that needs one pass took 58 us (33 now, 35 with a launch and a wait per
// pass) and one of six passes 105 (107).
inline cudaError_t run_filter(double* d, double* tmp, int nx, int ny, double alpha, int* flags, cudaStream_t s,
                              int* passes) {
    cudaError_t e = cudaSuccess;
    const dim3 grid((unsigned)((nx + FILTER_TILE - 1) / FILTER_TILE) * (unsigned)((ny + FILTER_TILE - 1) / FILTER_TILE));
    const dim3 block(256);
    int h[FILTER_PASSES];
    const double a2 = alpha * alpha;
    const int e20 = std::ilogb(a2) << 20;
    *passes = -1;
    for (int p0 = 0, group = 2; p0 < FILTER_PASSES && e == cudaSuccess; p0 += group, group *= 2) {
        const int p1 = std::min(p0 + group, FILTER_PASSES);
        for (int p = p0; p < p1; ++p)
            k_filter_pass<<<grid, block, 0, s>>>(p & 1 ? tmp : d, p & 1 ? d : tmp, nx, ny, a2, e20, flags, p);
        e = cudaGetLastError();
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(h + p0, flags + p0, sizeof(int) * (p1 - p0), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) return e;
        for (int p = p0; p < p1; ++p)
            if (!h[p]) { *passes = p + 1; return e; }
    }
    return e;
}

}  // namespace cliffs
