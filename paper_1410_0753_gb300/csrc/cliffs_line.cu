// 1D grids, many steps in one launch. A line of a few thousand nodes is far too small for a
// launch per step: 4.5 us each for 613 nodes, of which the sweep is a fraction. Here one block
// takes a scenario's line through all the steps of the call in shared memory (two buffers of
// the state, depth, metric and maxima: 48 bytes per node, so up to about 4700 nodes), each
// warp 56 nodes at a time with the x-sweep of the other kernels (the same bits), one block
// barrier per step. What bounds it is the latency of one sweep, about 0.5 us.
#include <algorithm>

#include "step_kernels.cuh"

namespace cliffs {

constexpr int LINE_PAD = 4;                        // nodes a window starts before its outputs
constexpr int LINE_ARRAYS = 12;
constexpr int LINE_MAX_SMEM = 227 * 1024;          // of one block

static int line_floats(int n) { return (n + XOUT - 1) / XOUT * XOUT + 2 * LINE_PAD; }

template <bool FRIC, bool S1, bool OPEN>
__global__ void __launch_bounds__(1024, 1)
k_line(const __grid_constant__ StepArgs a, const __grid_constant__ BatchArgs B, long long step0, long long n, int nsamp,
       int along_y) {
    extern __shared__ __align__(16) float sm[];
    const SweepConst& K = a.K;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int b = blockIdx.x;
    if (a.limit) n = min(n, a.limit[b] - step0);
    if (n <= 0) return;
    const int N = along_y ? a.ny : a.nx, nstrips = (N + XOUT - 1) / XOUT, L = nstrips * XOUT + 2 * LINE_PAD;
    const long long stride = along_y ? a.pitch : 1;
    // eta, velocity along, velocity across, twice; then d, 1/(2 dx) left and right, k2, maxima
    float* D = sm + 6 * L;
    float* hl = sm + 7 * L;
    float* hr = sm + 8 * L;
    float* k2 = sm + 9 * L;
    float* em = sm + 10 * L;                        // eta; speed at em + L
    const float* in = B.eta[step0 & 1] + (long long)b * a.plane;
    float* gmax = B.emax + (long long)b * a.plane;
    const long long fw = along_y ? 2 * a.fs_out : a.fs_out, ft = along_y ? a.fs_out : 2 * a.fs_out;
    for (int i = threadIdx.x; i < L; i += blockDim.x) {
        const int c = i - LINE_PAD;
        const bool inside = c >= 0 && c < N;
        const long long o = c * stride;
        for (int f = 0; f < 6; ++f) sm[f * L + i] = 0.f;
        D[i] = OUTSIDE_D;
        hl[i] = hr[i] = k2[i] = 0.f;
        if (inside) {
            sm[i] = in[o];
            sm[L + i] = in[fw + o];
            sm[2 * L + i] = in[ft + o];
            D[i] = a.d[o];
            if (along_y) {
                const float4 q = a.ymet[c];
                hl[i] = q.x; hr[i] = q.y; k2[i] = q.z;
            } else {
                const float f = a.xrow[0];          // 1 on Cartesian grids
                hl[i] = a.xa[c] * f; hr[i] = a.xb[c] * f; k2[i] = a.xk[c] * f;
            }
            em[i] = gmax[o];
            em[L + i] = gmax[a.fs_max + o];
        }
    }
    __syncthreads();
    const bool lo = OPEN && (a.open_edges & (along_y ? 4 : 1)), hi = OPEN && (a.open_edges & (along_y ? 8 : 2));
    int bad = 0;
    for (long long s = 0; s < n; ++s) {
        const long long st = step0 + s + 1;
        const float* A = sm + (s & 1) * 3 * L;
        float* Z = sm + (1 - (s & 1)) * 3 * L;
        const bool mx = st % B.maxout == 0;
        for (int w = wib; w < nstrips; w += nwarps) {
            const int i = w * XOUT + 2 * lane, cA = i - LINE_PAD;
            auto at = [i](const float* p) { return *reinterpret_cast<const float2*>(p + i); };
            float2 E = at(A), W = at(A + L), T = at(A + 2 * L);
            const float2 d = at(D);
            const XMet2 m{at(hl), at(hr), at(k2)};
            unsigned ends = 0u;
            if (lo) ends |= (cA == 0 ? 1u : 0u) | (cA + 1 == 0 ? 4u : 0u);
            if (hi) ends |= (cA == N - 1 ? 2u : 0u) | (cA + 1 == N - 1 ? 8u : 0u);
            xsweep2<FRIC, S1, OPEN>(E, W, T, d, m, K, lane, ends);
            const bool own = lane >= 2 && lane < 30, va = own && cA < N, vb = own && cA + 1 < N;
            emit_pair(Z + i, L, va, vb, E, W, T);
            bad |= (va && runaway(E.x, W.x, T.x)) | (vb && runaway(E.y, W.y, T.y));
            if (mx && va) emit_max(K, em + i, L, va, vb, E, along_y ? T : W, along_y ? W : T, d, at(em), at(em + L));
        }
        __syncthreads();
        if (B.grec && st % B.gout == 0) {
            float* rec = B.grec + (st / B.gout) * B.grec_row + (long long)b * a.rec_g_bstride;
            for (int k = threadIdx.x; k < nsamp; k += blockDim.x) {
                const int4 it = __ldg(a.samp + k);   // (row, col, class, slot)
                const int i = (along_y ? it.x : it.y) + LINE_PAD;
                rec[3 * it.w + 0] = Z[i];
                rec[3 * it.w + (along_y ? 2 : 1)] = Z[L + i];
                rec[3 * it.w + (along_y ? 1 : 2)] = Z[2 * L + i];
            }
        }
    }
    float* out = B.eta[(step0 + n) & 1] + (long long)b * a.plane;
    const float* Z = sm + (n & 1) * 3 * L;
    for (int c = threadIdx.x; c < N; c += blockDim.x) {
        const int i = c + LINE_PAD;
        const long long o = c * stride;
        out[o] = Z[i];
        out[fw + o] = Z[L + i];
        out[ft + o] = Z[2 * L + i];
        gmax[o] = em[i];
        gmax[a.fs_max + o] = em[L + i];
    }
    if (bad) atomicOr(a.err, ERRF_NONFINITE);
}

static size_t line_smem(int nodes) { return (size_t)line_floats(nodes) * LINE_ARRAYS * 4; }
static int line_threads(int nodes) { return 32 * std::min(32, (nodes + XOUT - 1) / XOUT); }
static const void* line_kernel(const StepArgs& a) {
    static const void* const t[8] = {(const void*)k_line<false, false, false>, (const void*)k_line<true, false, false>,
                                     (const void*)k_line<false, true, false>, (const void*)k_line<true, true, false>,
                                     (const void*)k_line<false, false, true>, (const void*)k_line<true, false, true>,
                                     (const void*)k_line<false, true, true>, (const void*)k_line<true, true, true>};
    return t[(a.K.fric ? 1 : 0) + (a.K.inv_dt2 > 0.f ? 2 : 0) + (a.open_edges ? 4 : 0)];
}
// always the maximum, not this line's size: the attribute belongs to the kernel, and another
// thread may launch it for a longer line between this call and the launch
static cudaError_t optin(const void* k) {
    return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, LINE_MAX_SMEM);
}

// Whether n steps in one launch are faster than n launches. Along y always (a launch of the y-sweep
// takes 46 us and more). Along x a launch takes 4.2 us and 7 ns per 1000 nodes of the batch (8 with
// open edges or eq. (solver1)); one launch for all costs 3 us more than a small one and goes in rounds
// of the blocks that fit on the GPU at once, each loading its line and then passing over it with up
// to 32 warps at a time, n times.
// The constants are fitted to 60 .. 4600 nodes, batches of 1 .. 3000 and 2 .. 40 steps; us of a call
// by launches and in one: 613 nodes x 40 steps 176 and 55, 4600 x 40 176 and 139, x 4 33 and 38, with
// open edges x 40 178 and 225; 3000 lines of 1000 nodes x 40 986 and 965, with open edges 1160 and 1579.
bool line_pays(const StepArgs& a, int batch, long long n, int along_y) {
    const int N = along_y ? a.ny : a.nx;
    if (line_smem(N) > (size_t)LINE_MAX_SMEM || n < 2) return false;
    if (along_y) return true;
    int dev = 0, sms = 1, per_sm = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const void* k = line_kernel(a);
    if (batch > sms && (optin(k) != cudaSuccess || cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                                                       &per_sm, k, line_threads(N), line_smem(N)) != cudaSuccess))
        return false;
    const long long at_once = (long long)sms * std::max(1, per_sm), rounds = (batch + at_once - 1) / at_once;
    const bool s1 = a.K.inv_dt2 > 0.f, open = a.open_edges != 0;
    const double kn = 1e-3 * N;
    const double pass = 0.75 + (open ? 0.3 : 0.0) + kn * (0.47 + (s1 ? 0.19 : 0.0) + (open ? 0.40 : 0.0) + (s1 && open ? 0.14 : 0.0));
    const double step = 4.2 + kn * batch * (s1 || open ? 8e-3 : 7e-3);
    return 3.0 + (double)rounds * (1.7 + 1.34 * kn + (double)n * pass) < (double)n * step;
}

cudaError_t launch_line(const StepArgs& a, const BatchArgs& b, int batch, long long step0, long long n, int nsamp,
                        int along_y, cudaStream_t s) {
    const int N = along_y ? a.ny : a.nx;
    const void* k = line_kernel(a);
    const cudaError_t e = optin(k);
    if (e != cudaSuccess) return e;
    StepArgs aa = a;
    BatchArgs bb = b;
    void* args[] = {&aa, &bb, &step0, &n, &nsamp, &along_y};
    return cudaLaunchKernel(k, dim3(batch), dim3(line_threads(N)), args, line_smem(N), s);
}

}  // namespace cliffs
