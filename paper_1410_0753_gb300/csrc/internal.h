// Internal interface between the host runtime (cliffs_api.cu) and the kernel translation
// units. Not part of the public ABI.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace cliffs {

// Constants of a sweep. Those that enter packed FP32x2 arithmetic are kept as pairs, so that
// no instruction is spent on widening them.
struct SweepConst {
    float hmin;       // h_min ('ground')
    float dwall;      // nodes with d < dwall are permanent walls (-FLT_MAX when itopo != 0)
    float half_dt;    // dt / 2
    float inv_dt2;    // 1 / dt^2 with eq. (solver1) (1/(dx_{j-1}+dx_j) = k2 / dt^2), else 0
    int fric;         // friction on
    int transverse;   // eq. (pq3) on/off
    float2 hdt;       // dt / 2
    float2 ntr;       // -1 with eq. (pq3), 0 without
    float2 lgf;       // log2(dt g n^2 g^(4/3)) (friction, fric_k2)
};

// Interpolation of one step's boundary input per edge: record k and weight w toward k + 1.
struct BndRow {
    long long k[4];
    double w[4];
};

// Arguments of one sweep-kernel launch (all device pointers). Fields 2D are pitched:
// element (b, r, c) lives at b * plane + r * pitch + c.
struct StepArgs {
    const float* eta_in; const float* u_in; const float* v_in;
    long long fs_in;                 // floats from eta to u and from u to v of the input state
    float* eta_out;                  // u and v follow at the field stride
    long long fs_out;                // floats from eta to u and from u to v of the output state
    const float* d;                  // [ny][pitch], FP32 depth
    const float* xa; const float* xb; const float* xk;   // [nx] per-column x metric: 1/(2 dx_{j-1}), 1/(2 dx_j), dt^2/(dx_{j-1}+dx_j)
    // per-row tables, valid for row indices -MET_PAD .. ny + MET_PAD - 1 (edge rows repeated)
    const float* xrow;               // row factor of the x metric (1 or 1/(R cos phi))
    const float4* ymet;              // (1/(2 dy_{j-1}), 1/(2 dy_j), dt^2/(dy_{j-1}+dy_j), -dt tan(phi)/R)
    float* emax;                     // max-wave eta, or null when not due this step
    long long fs_max;                // floats from the max-wave eta to the max-wave speed
    const float4* ymp;               // (1/(2 dy_j) twice, dt^2/(dy_{j-1}+dy_j) twice): packed operands
    float* rec_g;                    // gauge record row of this step (scenario 0) or null
    float* rec_n;                    // enclosed-grid node record row or null
    long long rec_g_bstride;         // floats between scenarios in the gauge records
    const int* samp_ptr;             // [nwarps + 1] per-warp sample list (CSR)
    const int4* samp;                // (row, col, class 0 gauge / 1 node, slot)
    const long long* limit;          // [batch] step limits, or null
    long long step;                  // index of the step being produced (1-based)
    int* err;                        // device error flags
    int nx, ny, pitch;
    long long plane;
    int S;                           // output rows per warp (y kernel)
    int nstrips, nseg;
    const int4* items;               // fused kernel: per warp (strip, first row, end row)
    int nitems;
    int nslots, slot_floats;         // ring of a fused warp: slots and floats per slot
    int tile_rows;                   // rows of the largest tile, halo included (k_step_tile, k_batch)
    int walls;                       // itopo = 0: nodes with d < dwall are walls
    SweepConst K;
    int sph;                         // geographic grid: x metric scaled per row
    int yfirst;                      // this step sweeps y, then x (alternating order)
    int open_edges;                  // open outer edges: bits W 1, E 2, S 4, N 8
    // boundary input, taken by the tile kernels as they read the state (bnd: this launch's step)
    int bnd;
    BndRow bnd_row;
    const double* bnd_vals[4];       // records [nt][3][np] per edge, or null
    long long wait_cycles;           // limit of every mbarrier wait (clock cycles)
    unsigned tx_pad;                 // extra bytes each ring slot expects (fault injection; 0)
};

enum { ERRF_NONFINITE = 1, ERRF_TIMEOUT = 2 };
constexpr int MET_PAD = 8;
constexpr int TMA_BOX_COLS = 64;   // columns of one TMA box (a warp's window)
constexpr int TMA_BOX_ROWS = 4;    // rows of one TMA box (one ring slot)

// message returned by cliffs_last_error() on the calling thread (cliffs_api.cu)
void set_last_error(const char* msg);

// TMA descriptors of the fused step's inputs: the state as a 4D [3][batch][ny][pitch] tensor
// (eta, u, v), d as a 2D [ny][pitch] tensor and the max-wave fields as [2][batch][ny][pitch],
// each read as 64 x 4 boxes, every field of the state (of the maxima) in one box.
struct StepMaps {
    CUtensorMap s, d, mw;
};

struct StepMaps2 {
    StepMaps m[2];                   // [k]: buffer k is the input
};

// The batched persistent run (k_batch, k_batch_tile). ctl lives in device memory so that one captured
// graph serves every call: ctl[0] = steps done before the launch, ctl[1] = steps done after
// it, ctl[2] = grid barrier (arrival count in the low 32 bits, generation in the high 32).
struct BatchArgs {
    long long* ctl;
    const int* order;                // scenarios by decreasing step limit
    const int* nact;                 // [nact_len]: scenarios whose limit is >= the step; null: all
    long long nact_len;
    int nall;                        // the batch size
    float* eta[2];                   // u and v at the field stride (StepArgs.fs_out)
    float* emax;
    int maxout, gout, bndout;
    float* grec;                     // gauge records, row = step / gout (scenario stride in StepArgs)
    long long grec_row;              // floats per record row
    float* nrec;                     // enclosed-grid corner records, row = step / bndout
    long long nrec_row;
    int alternate;                   // y first on the odd steps (the alternating order)
    // boundary input (batch 1): before step step0 + 1 + j the edge nodes of its input take
    // record k, weight w of bnd_rows[j] (computed on the host as cliffs_step_n does)
    int bnd;
    const BndRow* bnd_rows;
    const double* bv[4];             // records [nt][3][np] per edge, or null
    int bnp[4];                      // nodes per edge
};

// The input (u, v, eta) of edge node q of edge e (0 W, 1 E, 2 S, 3 N; n nodes) from record k with
// weight w toward k + 1 (the interpolation in FP64, non-fused, then rounded to FP32). Shared by
// the per-step kernel and those that take it as they read, so all give the same bits.
__device__ __forceinline__ float bnd_value(const double* vals, int n, int f, int q, long long k, double w) {
    const double* r0 = vals + k * 3 * n;
    const double a = r0[f * n + q];
    return (float)((w > 0.0) ? __dadd_rn(__dmul_rn(__dsub_rn(1.0, w), a), __dmul_rn(w, r0[(3 + f) * n + q])) : a);
}
// Edge node q of edge e takes its input. S and N own the corners when they carry input.
__device__ __forceinline__ void bnd_apply(float* eta, float* u, float* v, int pitch, int nx, int ny, int e, int q,
                                          const double* const* vals, const int* np, long long k, double w) {
    if (!vals[e] || q >= np[e]) return;
    if (e < 2 && ((q == 0 && vals[2]) || (q == ny - 1 && vals[3])) && nx > 1 && ny > 1) return;
    const int ix = (e == 0) ? 0 : (e == 1) ? nx - 1 : q;
    const int iy = (e == 2) ? 0 : (e == 3) ? ny - 1 : q;
    const size_t o = (size_t)iy * pitch + ix;
    u[o] = bnd_value(vals[e], np[e], 0, q, k, w);
    v[o] = bnd_value(vals[e], np[e], 1, q, k, w);
    eta[o] = bnd_value(vals[e], np[e], 2, q, k, w);
}
// Node (iy, ix) as a step reads it under boundary input: its edge's input, else (e, u, v) as
// they are.
__device__ __forceinline__ void bnd_read(float& e, float& u, float& v, int nx, int ny, int ix, int iy,
                                         const double* const* vals, const BndRow& R) {
    const int g = (iy == 0 && vals[2]) ? 2 : (iy == ny - 1 && vals[3]) ? 3 : (ix == nx - 1 && vals[1]) ? 1 :
                  (ix == 0 && vals[0]) ? 0 : -1;
    if (g < 0) return;
    const int n = g < 2 ? ny : nx, q = g < 2 ? iy : ix;
    u = bnd_value(vals[g], n, 0, q, R.k[g], R.w[g]);
    v = bnd_value(vals[g], n, 1, q, R.k[g], R.w[g]);
    e = bnd_value(vals[g], n, 2, q, R.k[g], R.w[g]);
}

// launchers (cliffs_step.cu, cliffs_tile.cu)
cudaError_t launch_step_fused(const StepArgs& a, const StepMaps& m, int batch, cudaStream_t s);
cudaError_t launch_batch(const StepArgs& a, const StepMaps2& mm, const BatchArgs& b, int blocks, cudaStream_t s);
int batch_blocks_per_sm(bool sph);
int fused_blocks_per_sm(bool sph);
void fused_ring(bool maxwave, int* nslots, int* slot_floats);
int fused_warps_per_block();
cudaError_t launch_step_tile(const StepArgs& a, int batch, cudaStream_t s);
cudaError_t launch_batch_tile(const StepArgs& a, const BatchArgs& b, int blocks, cudaStream_t s);
int tile_warps_per_block();
int tile_blocks_per_sm(int tile_rows);
int tile_max_rows();             // the largest tile_rows of which two blocks fit on an SM
// n steps of a 1D grid's scenarios: the line fits in one block and one launch is the faster way (cliffs_line.cu)
bool line_pays(const StepArgs& a, int batch, long long n, int along_y);
// steps step0 + 1 .. step0 + n of a 1D grid's scenarios, the samples in a.samp
cudaError_t launch_line(const StepArgs& a, const BatchArgs& b, int batch, long long step0, long long n, int nsamp,
                        int along_y, cudaStream_t s);
cudaError_t launch_xsweep(const StepArgs& a, int batch, cudaStream_t s);
cudaError_t launch_ysweep(const StepArgs& a, int batch, cudaStream_t s);

}  // namespace cliffs
