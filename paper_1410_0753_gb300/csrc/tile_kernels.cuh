// The step by tiles: a block of eight warps takes a window of 64 columns and a range of rows,
// x-sweeps the rows into shared memory, each warp whole rows, and after a barrier each warp
// finishes the y-sweep of a run of them from there. The same arithmetic as the marching kernels
// (step_kernels.cuh), so the same bits; what differs is the split of the work:
//   - a row's x-sweep and y-sweep are done by different warps, so no warp's serial chain is
//     longer than its share of the tile's rows twice (a marching warp runs both sweeps of its
//     rows and of three more, one after the other);
//   - the rows above and below are swept once per tile, not once per warp.
// That pays where a launch of marching warps does not fill the GPU several times over (there a
// warp per scheduler runs at the latency of its chain), and in the persistent run, whose steps
// each end at a grid barrier. Rows are read with plain loads (past L1: other SMs wrote them in
// the step before), two ahead of the one being swept.
#pragma once
#include "step_kernels.cuh"

namespace cliffs {

constexpr int TILE_WARPS = 8;
constexpr int TROW_FLOATS = 5 * XWIN;              // eta, v, u, d, c of a row

__device__ __forceinline__ float2 ld_cg(const float* p) {
    return __ldcg(reinterpret_cast<const float2*>(p));
}

template <bool SPH, bool FRIC, bool YF, bool S1, bool OPEN>
struct Tile {
    const StepArgs& a;
    const SweepConst& K;
    float* rows;               // [nr][5][64]
    unsigned char* wet;        // [nr]: the nodes that count are wet at the start of the y-sweep
    int lane, wib, b, c0, r0, r1;
    bool colA, colB, vA, vB, wallx;
    unsigned ends, walls;
    XMet2 m0;
    YMarch2 ym;
    StepOut O;
    const BndRow* bnd;         // this step's boundary input, or null
    const float* in;           // eta of the input state (this lane's pair of row 0); u, v at fs_in
    int bad;
    float2 chk_x, chk_out;     // as in FusedWarp

    __device__ __forceinline__ Tile(const StepArgs& a_) : a(a_), K(a_.K) {}

    __device__ __forceinline__ void setup(unsigned char* smem_raw) {
        lane = threadIdx.x & 31;
        wib = uniform(threadIdx.x >> 5);
        rows = reinterpret_cast<float*>(smem_raw);
        wet = smem_raw + (size_t)a.tile_rows * TROW_FLOATS * 4;
        bad = 0;
        chk_x = chk_out = v2(0.f);
    }

    __device__ __forceinline__ void take_item(int idx) {
        const int4 item = __ldg(a.items + idx);          // (strip, first row, end row)
        c0 = uniform(item.x) * XOUT;
        r0 = uniform(item.y);
        r1 = uniform(item.z);
        const int cA = c0 + 2 * lane;
        colA = cA < a.nx;
        colB = cA + 1 < a.nx;
        const bool own = (lane >= 2 || c0 == 0) && (lane < 30 || c0 + XWIN >= a.nx);   // as in FusedWarp
        vA = own && colA;
        vB = own && colB;
        wallx = c0 == 0 || c0 + XWIN >= a.nx;
        walls = wall_ends_x(cA, a.nx);
        ends = OPEN ? open_ends_x(a, cA) : 0u;
        float2 hr = v2(0.f), k2 = v2(0.f);
        if (colA) { hr.x = __ldg(a.xb + cA); k2.x = __ldg(a.xk + cA); }
        if (colB) { hr.y = __ldg(a.xb + cA + 1); k2.y = __ldg(a.xk + cA + 1); }
        m0 = XMet2{v2(0.f), hr, k2};
    }

    // the metric of row k, and the left intervals for the general x-sweep
    __device__ __forceinline__ XMet2 met_row(int k) const {
        XMet2 m = m0;
        if (SPH) {
            const float2 f = v2(__ldg(a.xrow + k));
            m.hr = mul2(m.hr, f); m.k2 = mul2(m.k2, f);
        }
        m.hl.y = m.hr.x;
        m.hl.x = __shfl_up_sync(FULL, m.hr.y, 1);
        if (lane == 0) m.hl.x = m.hr.x;
        return m;
    }

    __device__ __forceinline__ bool wet_pair(float2 H, float2 D, bool cA_, bool cB_) const {
        const bool wA = H.x >= K.hmin && D.x >= K.dwall, wB = H.y >= K.hmin && D.y >= K.dwall;
        return (wA || !cA_) && (wB || !cB_);
    }

    __device__ __forceinline__ void sweep_x(float2& E, float2& U, float2& V, float2 D, int k) const {
        const XMet2 m = met_row(k);
        const float2 H = add2(E, D);
        if (!S1 && __all_sync(FULL, wet_pair(H, D, colA, colB)))
            xsweep2_open<FRIC, OPEN>(E, U, V, D, H, m, K, wallx, walls, ends);
        else
            xsweep2<FRIC, S1, OPEN>(E, U, V, D, m, K, lane, ends, wallx);
    }

    // row k of the input (zero state, dry depth outside the domain)
    __device__ __forceinline__ void load(int k, float2& E, float2& U, float2& V, float2& D) const {
        E = U = V = v2(0.f);
        D = v2(OUTSIDE_D);
        if (k >= 0 && k < a.ny && colA) {
            const long long o = (long long)k * a.pitch;
            E = ld_cg(in + o);
            U = ld_cg(in + a.fs_in + o);
            V = ld_cg(in + 2 * a.fs_in + o);
            D = __ldg(reinterpret_cast<const float2*>(a.d + o + c0 + 2 * lane));
            if (bnd && (wallx || k == 0 || k == a.ny - 1)) {
                const int cA = c0 + 2 * lane;
                bnd_read(E.x, U.x, V.x, a.nx, a.ny, cA, k, a.bnd_vals, *bnd);
                if (colB) bnd_read(E.y, U.y, V.y, a.nx, a.ny, cA + 1, k, a.bnd_vals, *bnd);
            }
            if (!colB) { E.y = U.y = V.y = 0.f; D.y = OUTSIDE_D; }
        }
    }

    // phase 1: rows r0-3 .. r1+2 into shared memory, x-swept (unless YF)
    __device__ __forceinline__ void sweep_rows() {
        const int nr = r1 - r0 + 6;
        float2 E, U, V, D, E1, U1, V1, D1;            // this row and the next of the warp
        if (wib < nr) load(r0 - 3 + wib, E, U, V, D);
        if (wib + TILE_WARPS < nr) load(r0 - 3 + wib + TILE_WARPS, E1, U1, V1, D1);
        for (int i = wib; i < nr; i += TILE_WARPS) {
            const int k = r0 - 3 + i;
            float2 E2, U2, V2, D2;
            if (i + 2 * TILE_WARPS < nr) load(k + 2 * TILE_WARPS, E2, U2, V2, D2);
            const bool inside = k >= 0 && k < a.ny;
            if (inside && !YF) sweep_x(E, U, V, D, k);
            // a non-finite x-sweep result reads as a dry node in the y-sweep and would be
            // refilled by step (b) there: it is caught here (0 * NaN or 0 * inf is NaN)
            if (vA) chk_x.x = fmaf(E.x, 0.f, chk_x.x);
            if (vB) chk_x.y = fmaf(E.y, 0.f, chk_x.y);
            const float2 H = add2(E, D);
            float2* s = reinterpret_cast<float2*>(rows + i * TROW_FLOATS) + lane;
            s[0] = E;
            s[XWIN / 2] = V;
            s[XWIN] = U;
            s[3 * XWIN / 2] = D;
            s[2 * XWIN] = wave_speed2(H);
            const bool all = __all_sync(FULL, wet_pair(H, D, YF ? colA : vA, YF ? colB : vB));
            if (lane == 0) wet[i] = inside && all;
            E = E1; U = U1; V = V1; D = D1;
            E1 = E2; U1 = U2; V1 = V2; D1 = D2;
        }
    }

    __device__ __forceinline__ void row_from(int k, YRow& r) const {
        const float2* s = reinterpret_cast<const float2*>(rows + (k - r0 + 3) * TROW_FLOATS) + lane;
        r.e = s[0];
        r.w = s[XWIN / 2];
        r.t = s[XWIN];
        r.d = s[3 * XWIN / 2];
        r.c = s[2 * XWIN];
    }
    // row k wet at the start of the y-sweep (rows past the domain count as dry)
    __device__ __forceinline__ bool is_wet(int k) const { return k >= r0 - 3 && wet[k - r0 + 3] != 0; }

    __device__ __forceinline__ void emit(int r, float2 oe, float2 ow, float2 ot, float2 od, float2 em, float2 sm) {
        if (YF) sweep_x(oe, ot, ow, od, r);           // u along the row (ot), v across (ow)
        float* po = O.eta_out + ((long long)b * a.plane + (long long)r * a.pitch + c0 + 2 * lane);
        emit_pair(po, a.fs_out, vA, vB, oe, ot, ow);
        if (vB) chk_out = fma2(oe, oe, fma2(ot, ot, fma2(ow, ow, chk_out)));
        else if (vA) chk_out.x = fmaf(oe.x, oe.x, fmaf(ot.x, ot.x, fmaf(ow.x, ow.x, chk_out.x)));
        if (O.emax) emit_max(K, O.emax + (po - O.eta_out), a.fs_max, vA, vB, oe, ot, ow, od, em, sm);
    }

    __device__ __forceinline__ void load_max(int r, float2& em, float2& sm) const {
        em = sm = v2(0.f);
        if (O.emax && r >= 0 && r < a.ny && colA) {
            const float* p = O.emax + ((long long)b * a.plane + (long long)r * a.pitch + c0 + 2 * lane);
            em = ld_cg(p);
            sm = ld_cg(p + a.fs_max);
        }
    }

    // Row r of the y-sweep: the row in bank[PH] (after (b)) with the flux above it in fb[PH];
    // rows [ra, rb) go out. True in open water.
    template <int PH>
    __device__ __forceinline__ void y_row(int r, int ra, int rb, bool& fast) {
        float2 em, sm;
        load_max(r, em, sm);
        // rows r-1, r and r+1 wet, or past a wall of the domain (set in fast())
        const bool noedge = S1 || OPEN;
        const bool w0 = is_wet(r), wm = (r == 0 && !noedge) || is_wet(r - 1);
        const bool last = r == a.ny - 1 && !noedge;
        const bool now = w0 && wm && (last || is_wet(r + 1)) && !ym.pend;
        if (fast && !now) ym.after_fast();
        fast = now;
        row_from(r + 1, ym.bank[1 - PH]);
        if (now) {
            const float4 q = __ldg(a.ymp + r);
            const float4 m2 = __ldg(a.ymet + r);
            const int edge = noedge ? 0 : (r == 0 ? 1 : 0) | (r == a.ny - 1 ? 2 : 0);
            float2 ne, nw, nt;
            const float2 dP = ym.bank[PH].d;
            ym.template fast<PH, SPH, FRIC, S1>(make_float2(q.x, q.y), make_float2(q.z, q.w), v2(m2.w), edge, m2.x, K,
                                                ne, nw, nt);
            if (r >= ra && r < rb) emit(r, ne, nw, nt, dP, em, sm);
        } else {
            YRow n;
            row_from(r + 2, n);
            const bool oA = wet_mark(n.e.x, n.d.x, K), oB = wet_mark(n.e.y, n.d.y, K);
            ym.template slow<PH, SPH, FRIC, S1, OPEN>(n.e, n.w, n.t, n.d, oA, oB, __ldg(a.ymet + r), K,
                [&](int lag, float2 oe, float2 ow, float2 ot, float2 od) {
                    const int q = r + 2 - lag;
                    if (q < ra || q >= rb) return;
                    float2 e1 = em, s1 = sm;
                    if (lag == 3) load_max(q, e1, s1);
                    emit(q, oe, ow, ot, od, e1, s1);
                }, OPEN ? open_end_y(a, r) : 0);
        }
    }

    // phase 2: the y-sweep of this warp's run of rows
    __device__ __forceinline__ void sweep_cols() {
        const int m = (r1 - r0 + TILE_WARPS - 1) / TILE_WARPS;
        const int ra = r0 + wib * m, rb = min(ra + m, r1);
        if (ra >= rb) return;
        ym.init();
        // In open water the run starts at its first row, with the flux above it (or the wall
        // above row 0, which fast() sets); else three rows above, whose own upper neighbours the
        // rows of the run do not see.
        const bool noedge = S1 || OPEN;
        bool fast = is_wet(ra) && ((ra == 0 && !noedge) || is_wet(ra - 1)) && ((ra == a.ny - 1 && !noedge) || is_wet(ra + 1));
        int r = ra;
        if (fast) {
            row_from(ra, ym.bank[0]);
            if (ra > 0) {
                YRow p;
                row_from(ra - 1, p);
                const float4 q = __ldg(a.ymp + ra - 1);
                ym.fb[0] = iface2(p.e, p.w, p.t, p.d, p.c, ym.bank[0].e, ym.bank[0].w, ym.bank[0].t, ym.bank[0].d,
                                  ym.bank[0].c, make_float2(q.x, q.y));
                if (S1) { ym.pe = p.e; ym.pw = p.w; ym.pt = p.t; ym.pd = p.d; ym.pc = p.c; }
            }
        } else {
            r = ra - 3;
            if (ra > r0 || r >= 0) {
                row_from(r, ym.bank[0]);
                ym.fl = YMarch2::mark_bits(wet_mark(ym.bank[0].e.x, ym.bank[0].d.x, K),
                                           wet_mark(ym.bank[0].e.y, ym.bank[0].d.y, K), 0, 0);
            }
        }
        while (true) {
            y_row<0>(r, ra, rb, fast);
            if (++r >= rb && !(ym.pend && !fast)) break;
            if (r > rb) break;
            y_row<1>(r, ra, rb, fast);
            if (++r >= rb && !(ym.pend && !fast)) break;
            if (r > rb) break;
        }
    }

    // item idx of scenario b_ (whole block)
    __device__ __forceinline__ void run_item(int idx, int b_, const StepOut& O_, const float* eta_in, const BndRow* bnd_) {
        O = O_;
        bnd = bnd_;
        b = b_;
        in = eta_in + ((long long)b * a.plane + c0 + 2 * lane);
        sweep_rows();
        __syncthreads();
        sweep_cols();
        bad |= !(chk_out.x + chk_out.y < RUNAWAY_SQ);
        chk_out = v2(0.f);
        if (a.samp_ptr && (O.rec_g || O.rec_n)) {
            __syncthreads();                          // the whole tile is stored
            if (wib == 0) write_samples(a, O, idx, b, lane);
        }
    }

    __device__ __forceinline__ void report() {
        bad |= !(chk_x.x + chk_x.y == 0.f);
        if (bad) atomicOr(a.err, ERRF_NONFINITE);
    }
};

template <bool SPH, bool FRIC, bool YF, bool S1, bool OPEN>
__global__ void __launch_bounds__(TILE_WARPS * 32, 2)
k_step_tile(const __grid_constant__ StepArgs a) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int b = blockIdx.y;
    if (a.limit && __all_sync(FULL, a.step > a.limit[b])) return;
    Tile<SPH, FRIC, YF, S1, OPEN> T(a);
    T.setup(smem_raw);
    T.take_item(blockIdx.x);
    T.run_item(blockIdx.x, b, step_out(nullptr, a), a.eta_in, a.bnd ? &a.bnd_row : nullptr);
    T.report();
}

// ------------------------------------------------------------------ batched, persistent
// k_batch (step_kernels.cuh) with blocks that take (scenario, tile) pairs in place of warps that
// take marching items: for runs whose tiles fit in one round of resident blocks.
template <bool SPH, bool FRIC, bool S1, bool OPEN, bool ALT>
__global__ void __launch_bounds__(TILE_WARPS * 32, 2)
k_batch_tile(const __grid_constant__ StepArgs a, const __grid_constant__ BatchArgs B) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const long long step0 = uniform64(B.ctl[0]), step_end = uniform64(B.ctl[1]);
    if (__any_sync(FULL, *reinterpret_cast<volatile int*>(a.err) & ERRF_TIMEOUT)) return;
    Tile<SPH, FRIC, false, S1, OPEN> T(a);
    Tile<SPH, FRIC, true, S1, OPEN> TY(a);
    T.setup(smem_raw);
    if (ALT) TY.setup(smem_raw);
    int taken = -1;                                // the tile taken last (small grids keep theirs)
    // fault injection: the barrier waits for an arrival that never comes
    const unsigned arrivals = gridDim.x + (a.tx_pad ? 1u : 0u);
    for (long long st = step0 + 1; st <= step_end; ++st) {
        const bool yf = ALT && (((st - 1) & 1) != 0);
        const bool odd = (st & 1) != 0;          // odd steps read buffer 0 and write buffer 1
        const BndRow* bnd = B.bnd ? &B.bnd_rows[st - step0 - 1] : nullptr;
        const bool mx = st % B.maxout == 0;
        const StepOut O{nullptr, odd ? B.eta[1] : B.eta[0], mx ? B.emax : nullptr,
                        (B.grec && st % B.gout == 0) ? B.grec + (st / B.gout) * B.grec_row : nullptr,
                        (B.nrec && st % B.bndout == 0) ? B.nrec + (st / B.bndout) * B.nrec_row : nullptr};
        const float* in = odd ? B.eta[0] : B.eta[1];
        const int na = B.nact ? (st < B.nact_len ? uniform(__ldg(B.nact + st)) : 0) : B.nall;
        const unsigned total = (unsigned)na * (unsigned)a.nitems;
        for (unsigned t = blockIdx.x; t < total; t += gridDim.x) {
            const int item = (int)(t % (unsigned)a.nitems), scen = uniform(__ldg(B.order + t / (unsigned)a.nitems));
            if (ALT || item != taken) {
                if (yf) TY.take_item(item);
                else T.take_item(item);
                taken = item;
            }
            if (t != blockIdx.x) __syncthreads();    // the tile before is done with shared memory
            if (yf) TY.run_item(item, scen, O, in, bnd);
            else T.run_item(item, scen, O, in, bnd);
        }
        if (!grid_sync(reinterpret_cast<unsigned long long*>(B.ctl + 2), arrivals, a.wait_cycles, a.err)) break;
    }
    T.report();
    if (ALT) TY.report();
}

}  // namespace cliffs
