// Kernel templates of the split step (arXiv 1410.0753, section "Numerics"); instantiated by
// cliffs_step.cu (reflecting outer edges) and cliffs_step_open.cu (open outer edges, OPEN).
// The kernels and their work split are described at the top of cliffs_step.cu.
#pragma once
#include "internal.h"
#include "sweep.cuh"

namespace cliffs {

constexpr int SLOT_ROWS = TMA_BOX_ROWS;       // rows per ring slot (one TMA box per tensor)
static_assert(TMA_BOX_COLS == XWIN && SLOT_ROWS == 4, "a TMA box spans the warp's window");
constexpr int ARR_FLOATS = SLOT_ROWS * XWIN;  // one array of a slot: eta, u, v, d [, eta_max, speed_max]
constexpr int FUSED_WARPS = 4;
constexpr int MAX_SLOTS = 8;                  // mbarriers kept per warp
constexpr int BAR_BYTES = FUSED_WARPS * MAX_SLOTS * 8;

// ------------------------------------------------------------------ TMA / mbarrier (PTX)
__device__ __forceinline__ unsigned smem_u32(const void* p) {
    return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t* b, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void fence_proxy_async() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_tx(uint64_t* b, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(b)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ bool mbar_test(uint64_t* b, unsigned parity) {
    unsigned r;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(r) : "r"(smem_u32(b)), "r"(parity) : "memory");
    return r != 0;
}
// bounded wait for the phase with the given parity
__device__ __forceinline__ bool mbar_wait(uint64_t* b, unsigned parity, long long limit) {
    if (mbar_test(b, parity)) return true;
    const long long t0 = clock64();
    while (!mbar_test(b, parity))
        if (clock64() - t0 > limit) return false;
    return true;
}
__device__ __forceinline__ void tma_box4(float* dst, const CUtensorMap* m, uint64_t* b, int x, int y, int z) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%3, %4, %5, %6}], [%2];"
        ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(m)), "r"(smem_u32(b)), "r"(x), "r"(y), "r"(z), "r"(0)
        : "memory");
}
__device__ __forceinline__ void tma_box2(float* dst, const CUtensorMap* m, uint64_t* b, int x, int y) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%3, %4}], [%2];"
        ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(m)), "r"(smem_u32(b)), "r"(x), "r"(y)
        : "memory");
}

__device__ __forceinline__ void prefetch_map(const CUtensorMap* m) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(m)) : "memory");
}
// A value that is the same in every lane, through an instruction whose result is uniform by
// construction: the compiler then keeps what derives from it (row counters, ring positions)
// in uniform registers and branches on it without convergence barriers.
__device__ __forceinline__ int uniform(int x) { return __reduce_max_sync(FULL, x); }
__device__ __forceinline__ long long uniform64(long long x) {
    const unsigned lo = __reduce_max_sync(FULL, (unsigned)x), hi = __reduce_max_sync(FULL, (unsigned)(x >> 32));
    return (long long)(((unsigned long long)hi << 32) | lo);
}

// ------------------------------------------------------------------ epilogue
// Nodes (r, c) and (r, c+1) of the step input, for the kernels without TMA; nodes outside
// the domain get depth OUTSIDE_D (dry, never wetted) and zero state.
__device__ __forceinline__ void load_pair(const StepArgs& a, size_t boff, int r, int c,
                                          float2& E, float2& U, float2& V, float2& D) {
    E = U = V = make_float2(0.f, 0.f);
    D = make_float2(OUTSIDE_D, OUTSIDE_D);
    if (r >= 0 && r < a.ny && c >= 0 && c < a.nx) {
        const size_t o = (size_t)r * a.pitch + c;
        E = __ldg(reinterpret_cast<const float2*>(a.eta_in + boff + o));
        U = __ldg(reinterpret_cast<const float2*>(a.u_in + boff + o));
        V = __ldg(reinterpret_cast<const float2*>(a.v_in + boff + o));
        D = __ldg(reinterpret_cast<const float2*>(a.d + o));
        if (c + 1 >= a.nx) { E.y = U.y = V.y = 0.f; D.y = OUTSIDE_D; }
    }
}

// Open outer edges of a lane's pair of columns for xsweep2 (bits 1 A left, 2 A right, 4 B
// left, 8 B right) and of a row for the y-sweep pipeline (1 first row, 2 last row, 0 none).
__device__ __forceinline__ unsigned open_ends_x(const StepArgs& a, int cA) {
    unsigned e = 0u;
    if (a.open_edges & 1) { if (cA == 0) e |= 1u; if (cA + 1 == 0) e |= 4u; }
    if (a.open_edges & 2) { if (cA == a.nx - 1) e |= 2u; if (cA + 1 == a.nx - 1) e |= 8u; }
    return e;
}
__device__ __forceinline__ int open_end_y(const StepArgs& a, int row) {
    return (row == 0 && (a.open_edges & 4)) ? 1 : (row == a.ny - 1 && (a.open_edges & 8)) ? 2 : 0;
}

__device__ __forceinline__ int runaway(float e, float u, float v) {
    return !(fabsf(e) + fabsf(u) + fabsf(v) < 3e5f);
}
// The same test accumulated branch-free over the rows of one work item: the sum of e^2 + u^2 +
// v^2 over a lane's stored nodes reaches 9e10 when any node reaches 3e5 in a component, and a
// non-finite value makes it non-finite. No physical state sums that high over an item's rows
// (land far above the sea counts with its eta = -d; over the steps of a persistent run it
// would), so the sum is tested and cleared after every item.
constexpr float RUNAWAY_SQ = 9e10f;

// What changes from one step to the next: the input state's TMA descriptors, the output
// planes (eta; u and v follow at the field stride), and the max-wave fields and record rows
// when they are due this step (else null).
struct StepOut {
    const StepMaps* M;
    float* eta_out;
    float* emax;
    float* rec_g;
    float* rec_n;
};

__device__ __forceinline__ StepOut step_out(const StepMaps* M, const StepArgs& a) {
    return StepOut{M, a.eta_out, a.emax, a.rec_g, a.rec_n};
}

// Store a finished pair of nodes at po (eta; u and v at the field stride fs). With max-wave
// due (section "Running Options", field maxout), (em, sm) hold the stored maxima of the pair
// and pm is where they live (speed at the stride ms): on wet nodes they take the new eta and
// speed sqrt(u^2 + v^2) where these are larger and are written back.
__device__ __forceinline__ void emit_pair(float* po, long long fs, bool va, bool vb,
                                          float2 E, float2 U, float2 V) {
    if (vb) {
        *reinterpret_cast<float2*>(po) = E;
        *reinterpret_cast<float2*>(po + fs) = U;
        *reinterpret_cast<float2*>(po + 2 * fs) = V;
    } else if (va) {
        po[0] = E.x; po[fs] = U.x; po[2 * fs] = V.x;
    }
}
__device__ __forceinline__ void emit_max(const SweepConst& K, float* pm, long long ms, bool va, bool vb,
                                         float2 E, float2 U, float2 V, float2 D, float2 em, float2 sm) {
    const float2 h = add2(E, D);
    const float2 s2 = fma2(U, U, mul2(V, V));
    const float2 sm2 = mul2(sm, sm);
    const bool wA = va && (D.x >= K.dwall) && (h.x >= K.hmin);
    const bool wB = vb && (D.y >= K.dwall) && (h.y >= K.hmin);
    const bool eA = wA && E.x > em.x, eB = wB && E.y > em.y;
    const bool sA = wA && s2.x > sm2.x, sB = wB && s2.y > sm2.y;
    if (eA || eB || sA || sB) {
        if (eA) em.x = E.x;
        if (eB) em.y = E.y;
        if (sA) sm.x = fmaxf(sm.x, sqrt_pos(s2.x));
        if (sB) sm.y = fmaxf(sm.y, sqrt_pos(s2.y));
        if (vb) {
            *reinterpret_cast<float2*>(pm) = em;
            *reinterpret_cast<float2*>(pm + ms) = sm;
        } else {
            pm[0] = em.x; pm[ms] = sm.x;
        }
    }
}

// The gauge / enclosed-grid records of a work item whose rows are all stored: every lane reads
// nodes of the item's sample list back from the output (written by this warp, so a warp
// barrier orders it; the lines are in L2) and writes their records. Sampling inside the row
// loop instead, from registers, took a call there and 18 warp-instructions per row whether
// the row has samples or not (147.7 against 164.0 us on a 4096^2 grid without any).
__device__ __forceinline__ void write_samples(const StepArgs& a, const StepOut& O, int item, int b, int lane) {
    if (!a.samp_ptr || !(O.rec_g || O.rec_n)) return;
    const int sp = __ldg(a.samp_ptr + item), se = __ldg(a.samp_ptr + item + 1);
    if (sp >= se) return;
    __syncwarp();
    const float* st = O.eta_out + (long long)b * a.plane;
    float* rg = O.rec_g ? O.rec_g + (long long)b * a.rec_g_bstride : nullptr;
    for (int i = sp + lane; i < se; i += 32) {
        const int4 it = __ldg(a.samp + i);           // (row, col, class 0 gauge / 1 node, slot)
        float* out = it.z == 0 ? rg : O.rec_n;
        if (!out) continue;
        const float* q = st + ((long long)it.x * a.pitch + it.y);
        const float e = __ldcg(q), u = __ldcg(q + a.fs_out), v = __ldcg(q + 2 * a.fs_out);
        out[3 * it.w + 0] = e;
        out[3 * it.w + 1] = u;
        out[3 * it.w + 2] = v;
    }
}

// ------------------------------------------------------------------ fused step
// One warp of the fused step. A work item is a strip and an output row range [r0, r1); the
// warp marches down the rows of its 64-column window, which arrive by TMA in slots of four
// rows (one box for eta, u, v and one for d, issued by one lane) through a ring per warp.
//
// One vote per row decides its path: when the incoming row k and the x-swept rows before it
// are wet, the row is open water and one straight block of code updates row k-2 in the y-sweep
// (which needs rows k-3 .. k-1 only) and x-sweeps row k, two independent chains of arithmetic
// side by side; else the general x-sweep and march step run (slow_row). In open water a row
// depends on one row above and below only, so the march starts at row r0-1 and ends with row
// r1+1 in place of r0-3 .. r1+2; should one of the first rows turn out not to be open water,
// it starts over from r0-3 (nothing has been written by then, and the first slot, which
// holds rows r0-3 .. r0, is still there). At the top and bottom of the domain the walls are
// set in the fast path, and rows past the domain only keep the march going.
//
// The ring's position and phase bits live as long as the warp, so a warp may process any
// number of items in a row. With YF (a y-first step of the alternating order) rows enter the
// march unswept and each finished row is x-swept across the warp on its way out.
template <bool SPH, bool FRIC, bool YF = false, bool S1 = false, bool OPEN = false>
struct FusedWarp {
    // the plain step has its open-water loop once per case (edge windows, max-wave due); the
    // other variants one loop for all
    static constexpr bool MAIN = !YF && !S1 && !OPEN;
    const StepArgs& a;
    const SweepConst& K;
    float* ring;
    uint64_t* bar;
    unsigned phase;            // phase parity of each ring slot (bits)
    int head;                  // the ring slot to fill next
    int cs;                    // the ring slot being read
    int nfill, nread, ntot;    // slots of the item filled, waited for, to be filled
    int lane, b, c0, r0, r1, k0, kpast;
    bool sw;                   // this lane's nodes of row k-1 that count are wet at the start of the y-sweep
    bool colA, colB, vA, vB;
    bool wallx;                // the window touches the domain's edge
    unsigned tx, ends, walls;
    XMet2 m0;                  // hl is formed where it is needed
    YMarch2 ym;
    StepOut O;
    int bad;
    float2 chk_x;              // sum of 0 * (x-swept eta) of the general rows: 0, or NaN once one is not finite
    float2 chk_out;            // sum of e^2 + u^2 + v^2 over the stored nodes (RUNAWAY_SQ)

    __device__ __forceinline__ FusedWarp(const StepArgs& a_) : a(a_), K(a_.K) {}
    __device__ __forceinline__ void setup(unsigned char* smem_raw, int wib) {
        lane = threadIdx.x & 31;
        bar = reinterpret_cast<uint64_t*>(smem_raw) + wib * MAX_SLOTS;
        ring = reinterpret_cast<float*>(smem_raw + BAR_BYTES) + wib * a.nslots * a.slot_floats + 2 * lane;
        phase = 0u;
        head = 0;
        bad = 0;
        chk_x = chk_out = v2(0.f);
        if (lane == 0) {
            for (int s = 0; s < a.nslots; ++s) mbar_init(&bar[s], 1);
            fence_mbar_init();
        }
        __syncwarp();
    }

    __device__ __forceinline__ int next_of(int s) const { return s + 1 == a.nslots ? 0 : s + 1; }
    // this lane's pair in row q of ring slot s
    __device__ __forceinline__ const float* at(int s, int q) const { return ring + s * a.slot_floats + q * XWIN; }

    // one lane starts the boxes of the item's next slot (rows k0 + 4 nfill ..; the max-wave
    // rows two rows behind, where the open-water path emits). The caller has the warp meet first:
    // the slot may hold a row that other lanes have just read. The fence orders those reads (the
    // generic proxy) before the copy's writes (the async proxy).
    __device__ __forceinline__ void fill() {
        if (lane == 0) {
            fence_proxy_async();
            float* dst = ring + head * a.slot_floats;
            const int row = k0 + SLOT_ROWS * nfill;
            mbar_arrive_tx(&bar[head], tx);
            tma_box4(dst, &O.M->s, &bar[head], c0, row, b);
            tma_box2(dst + 3 * ARR_FLOATS, &O.M->d, &bar[head], c0, row);
            if (O.emax) tma_box4(dst + 4 * ARR_FLOATS, &O.M->mw, &bar[head], c0, row - 2, b);
        }
        head = next_of(head);
        ++nfill;
    }
    // wait for ring slot cs (bounded); false when it expired
    __device__ __forceinline__ bool acquire() {
        const bool ok = mbar_wait(&bar[cs], (phase >> cs) & 1u, a.wait_cycles);
        if (!__all_sync(FULL, ok)) return false;
        phase ^= 1u << cs;
        ++nread;
        return true;
    }
    // The march enters the slot that row k begins (`open`: the row only keeps open water going, so
    // a row past the last slot is not read).
    __device__ __forceinline__ bool next_slot(int k, bool open) {
        cs = next_of(cs);
        const int i = (k - k0) >> 2;
        if (i < nread) return true;                     // started over: it is here already
        if (i >= ntot && k < a.ny && !open) {           // rows past r1, for the general path
            ntot = i + 1;
            __syncwarp();
            fill();
        }
        return i >= ntot || acquire();
    }
    // the slot before the one row k is in is free: its place takes a new one
    __device__ __forceinline__ void refill(int k) {
        if (nfill < ntot && nfill < ((k - k0) >> 2) + a.nslots) {
            __syncwarp();
            fill();
        }
    }

    __device__ __forceinline__ XMet2 met_row(int k) const {
        XMet2 m = m0;
        if (SPH) {
            const float2 f = v2(__ldg(a.xrow + k));
            m.hr = mul2(m.hr, f); m.k2 = mul2(m.k2, f);
        }
        return m;
    }
    // the left intervals (the general x-sweep's walls): those of the left neighbours
    __device__ __forceinline__ void met_left(XMet2& m) const {
        m.hl.y = m.hr.x;
        m.hl.x = __shfl_up_sync(FULL, m.hr.y, 1);
        if (lane == 0) m.hl.x = m.hr.x;
    }

    // Whether the lane's nodes that count are wet, given their heights. EDGE: the window has
    // columns past the domain's edge or the grid permanent walls.
    template <bool EDGE>
    __device__ __forceinline__ bool wet_pair(float2 H, float2 D, bool cA_, bool cB_) const {
        float m = min_nan(H.x, H.y);
        if (EDGE && !cB_) m = H.x;
        bool ok = m >= K.hmin;
        if (EDGE && a.walls) {
            float d = min_nan(D.x, D.y);
            if (!cB_) d = D.x;
            ok = ok && d >= K.dwall;
        }
        return ok || !cA_;
    }
    __device__ __forceinline__ float* out_row(int r) const {
        return O.eta_out + ((long long)b * a.plane + (long long)r * a.pitch + c0 + 2 * lane);
    }

    // Finished row r out at po, by the lanes whose nodes go out (va, vb); mw: its stored maxima
    // in the ring (eta, then speed). EDGE: a lane's A may go out alone. MW: max-wave is due.
    template <bool EDGE, bool MW>
    __device__ __forceinline__ void emit(int r, float* po, bool va, bool vb, const float* mw, float2 oe, float2 ow,
                                         float2 ot, float2 od) {
        if (YF) {
            // x-sweep of the y-swept row r: along-row velocity u (ot), across v (ow)
            XMet2 m = met_row(SPH ? max(r, 0) : r);
            const float2 H = add2(oe, od);
            if (!S1 && __all_sync(FULL, wet_pair<EDGE>(H, od, colA, colB))) {
                xsweep2_open<FRIC, OPEN>(oe, ot, ow, od, H, m, K, EDGE && wallx, walls, ends);
            } else {
                met_left(m);
                xsweep2<FRIC, S1, OPEN>(oe, ot, ow, od, m, K, lane, ends, wallx);
            }
        }
        if (vb) {
            *reinterpret_cast<float2*>(po) = oe;
            *reinterpret_cast<float2*>(po + a.fs_out) = ot;
            *reinterpret_cast<float2*>(po + 2 * a.fs_out) = ow;
            // the stored nodes only (an unstored column past the domain edge may hold anything)
            chk_out = fma2(oe, oe, fma2(ot, ot, fma2(ow, ow, chk_out)));
        }
        if (EDGE) {
            if (va && !vb) {
                po[0] = oe.x; po[a.fs_out] = ot.x; po[2 * a.fs_out] = ow.x;
                chk_out.x = fmaf(oe.x, oe.x, fmaf(ot.x, ot.x, fmaf(ow.x, ow.x, chk_out.x)));
            }
        }
        if (MW && (MAIN || O.emax)) {
            const float2 em = *reinterpret_cast<const float2*>(mw);
            const float2 sm = *reinterpret_cast<const float2*>(mw + ARR_FLOATS);
            emit_max(K, O.emax + (po - O.eta_out), a.fs_max, va, vb, oe, ot, ow, od, em, sm);
        }
    }

    // columns past the domain's edge: at rest, dry, never wetted
    __device__ __forceinline__ void outside(float2& E, float2& U, float2& V, float2& D) const {
        if (!colA) { E.x = U.x = V.x = 0.f; D.x = OUTSIDE_D; }
        if (!colB) { E.y = U.y = V.y = 0.f; D.y = OUTSIDE_D; }
    }

    // Row k in open water, at s in the ring: row k-2 in the y-sweep, row k in the x-sweep.
    // False, with nothing done, when it is not open water.
    template <int PH, bool EDGE, bool MW>
    __device__ __forceinline__ bool fast_row(int k, const float* s, int kgen, float*& po) {
        // a row before the first or after the last that counts only keeps the march going
        const bool past = (unsigned)k > (unsigned)kpast;
        float2 E = *reinterpret_cast<const float2*>(s + 0 * ARR_FLOATS);
        float2 U = *reinterpret_cast<const float2*>(s + 1 * ARR_FLOATS);
        float2 V = *reinterpret_cast<const float2*>(s + 2 * ARR_FLOATS);
        float2 D = *reinterpret_cast<const float2*>(s + 3 * ARR_FLOATS);
        if (YF && wallx) outside(E, U, V, D);           // its x-sweep comes later, with its votes
        float2 H = add2(E, D);
        bool wet = sw && (YF || past || wet_pair<EDGE>(H, D, colA, colB));
        if (S1 || OPEN) wet = wet && k < kgen;
        if (!__all_sync(FULL, wet)) return false;
        const float4 q = __ldg(a.ymp + k - 2);
        const float2 nsdt = SPH ? v2(__ldg(a.ymet + k - 2).w) : v2(0.f);
        int edge = 0;
        float hl = 0.f;
        if (k == 2 || k == a.ny + 1) {
            edge = (k == 2 ? 1 : 0) | (k == a.ny + 1 ? 2 : 0);
            hl = __ldg(a.ymet).x;
        }
        float2 ne, nw, nt;
        const float2 dP = ym.bank[PH].d;
        ym.template fast<PH, SPH, FRIC, S1>(make_float2(q.x, q.y), make_float2(q.z, q.w), nsdt, edge, hl, K, ne, nw, nt);
        if (!YF) {
            XMet2 m = met_row(SPH ? min(max(k, 0), a.ny - 1) : k);
            if (S1) {
                met_left(m);
                xsweep2<FRIC, S1, OPEN>(E, U, V, D, m, K, lane, ends, wallx);
            } else {
                xsweep2_open<FRIC, OPEN>(E, U, V, D, H, m, K, EDGE && wallx, walls, ends);
            }
            H = add2(E, D);
        }
        sw = past || wet_pair<EDGE>(H, D, YF ? colA : vA, YF ? colB : vB);
        ym.template store_row<PH>(E, V, U, D, H);
        const bool out = k - 2 >= r0;
        emit<EDGE, MW>(k - 2, po, vA && out, vB && out, s + 4 * ARR_FLOATS, ne, nw, nt, dP);
        po += a.pitch;
        return true;
    }

    // Row k in the general case, at s in the ring when it is inside the domain (q: its row in
    // ring slot cs). hist: rows k-2 (bit 0) and k-3 (bit 1) wet at the start of the y-sweep.
    template <int PH>
    __device__ __forceinline__ void slow_row(int k, int q, const float* s, unsigned& hist) {
        const unsigned h1 = __all_sync(FULL, sw) ? 1u : 0u;
        float2 E = v2(0.f), U = E, V = E, D = v2(OUTSIDE_D);
        if (k >= 0 && k < a.ny) {
            E = *reinterpret_cast<const float2*>(s + 0 * ARR_FLOATS);
            U = *reinterpret_cast<const float2*>(s + 1 * ARR_FLOATS);
            V = *reinterpret_cast<const float2*>(s + 2 * ARR_FLOATS);
            D = *reinterpret_cast<const float2*>(s + 3 * ARR_FLOATS);
            if (wallx) outside(E, U, V, D);
            if (!YF) {
                XMet2 m = met_row(k);
                met_left(m);
                xsweep2<FRIC, S1, OPEN>(E, U, V, D, m, K, lane, ends, wallx);
            }
        }
        // a non-finite x-sweep result reads as a dry node in the y-sweep and would be
        // refilled by step (b) there: it is caught here (0 * NaN or 0 * inf is NaN), with that
        // of row k-1, which the open-water x-sweep may have left (in the lanes that count)
        chk_x = fma2(E, v2(0.f), chk_x);
        if (vA) chk_x.x = fmaf(ym.bank[1 - PH].e.x, 0.f, chk_x.x);
        if (vB) chk_x.y = fmaf(ym.bank[1 - PH].e.y, 0.f, chk_x.y);
        const bool oA = wet_mark(E.x, D.x, K), oB = wet_mark(E.y, D.y, K);
        const float4 m2 = __ldg(a.ymet + k - 2);
        const int edge = OPEN ? open_end_y(a, k - 2) : 0;
        ym.template slow<PH, SPH, FRIC, S1, OPEN>(E, V, U, D, oA, oB, m2, K,
            [&](int lag, float2 oe, float2 ow, float2 ot, float2 od) {
                const int r = k - lag;
                if (r < r0 || r >= r1) return;
                // the row's place among the max-wave rows, two rows ahead of the state's
                const int qm = q + 2 - lag;
                const float* mw = qm >= 0 ? at(cs, qm) : at(cs == 0 ? a.nslots - 1 : cs - 1, qm + SLOT_ROWS);
                if (!MAIN || O.emax) emit<true, true>(r, out_row(r), vA, vB, mw + 4 * ARR_FLOATS, oe, ow, ot, od);
                else emit<true, false>(r, out_row(r), vA, vB, mw, oe, ow, ot, od);
            }, edge);
        hist = (((ym.pend ? hist & ~1u : hist) << 1) | h1) & 3u;
        sw = YF ? ((oA || !colA) && (oB || !colB)) : ((oA || !vA) && (oB || !vB));
    }

    // Pairs of rows in open water from row k (row q of the slot, at s), until a row is not open
    // water (odd: the second of its pair), the item is done (then k > r1) or a wait expires (false).
    template <bool EDGE, bool MW>
    __device__ __forceinline__ bool fast_rows(int& k, int& q, const float*& s, bool& odd, int kgen, int klim) {
        float* po = out_row(k - 2);
        while (true) {
            if (q == SLOT_ROWS) {
                if (!next_slot(k, __all_sync(FULL, sw) && k < kgen)) return false;
                q = 0;
                s = at(cs, 0);
            }
            odd = false;
            if (!fast_row<0, EDGE, MW>(k, s, kgen, po)) return true;
            if (k > r1) { ++k; return true; }
            if (q == 0 && k >= klim) refill(k);
            odd = true;
            if (!fast_row<1, EDGE, MW>(k + 1, s + XWIN, kgen, po)) return true;
            if (q == 0 && k < klim) refill(k);
            k += 2;
            if (k - 1 > r1) return true;
            q += 2;
            s += 2 * XWIN;
        }
    }

    // General rows from row k (row q of the slot, at s; odd: from the second of its pair) up to
    // the next pair after three rows of open water, the end of the item (k - 1 > r1) or an
    // expired wait (false).
    __device__ __forceinline__ bool slow_rows(int& k, int& q, const float*& s, bool odd, unsigned hist, int kgen) {
        while (true) {
            if (!odd) {
                if (q == SLOT_ROWS) {
                    if (!next_slot(k, false)) return false;
                    q = 0;
                    s = at(cs, 0);
                }
                slow_row<0>(k, q, s, hist);
                if (k > r1 && (!ym.pend || k == r1 + 2)) { ++k; return true; }
                if (q == 0 && k != k0) refill(k);
            }
            odd = false;
            slow_row<1>(k + 1, q + 1, s + XWIN, hist);
            const bool done = k >= r1 && (!ym.pend || k + 1 == r1 + 2);
            if (!done && q == 0 && k != k0) refill(k);
            k += 2;
            q += 2;
            s += 2 * XWIN;
            if (done || (hist == 3u && k < kgen && __all_sync(FULL, sw))) return true;
        }
    }

    // Take work item `idx` (strip, rows): what does not depend on the state.
    __device__ __forceinline__ void take_item(int idx) {
        const int4 item = __ldg(a.items + idx);          // (strip, first row, end row)
        c0 = uniform(item.x) * XOUT;                     // window columns c0 .. c0 + 63 (fused_strips)
        const int cA = c0 + 2 * lane;
        r0 = uniform(item.y);
        r1 = uniform(item.z);
        k0 = r0 - 3;
        kpast = min(r1, a.ny - 1);
        colA = cA < a.nx;
        colB = cA + 1 < a.nx;
        // the output columns: c0 + 4 .. c0 + 59, and from the domain's first column in the
        // first window, to its last column in the window that reaches it (past it the
        // window holds dry ghost columns, or its edge is the domain's)
        const bool own = (lane >= 2 || c0 == 0) && (lane < 30 || c0 + XWIN >= a.nx);
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

    // Process the item taken (number idx) of scenario b_ for the step described by O_. Returns
    // false when a wait expired (the warp's copies have landed when it returns).
    __device__ __forceinline__ bool run_item(int idx, int b_, const StepOut& O_) {
        O = O_;
        b = b_;
        tx = (O.emax ? 6u : 4u) * ARR_FLOATS * 4u + a.tx_pad;
        // the slots the open-water march reads (with max-wave due its rows count too)
        ntot = ((O.emax ? r1 + 1 : kpast) - k0) / SLOT_ROWS + 1;
        nfill = nread = 0;
        cs = head;
        const int first = head;
        __syncwarp();                              // the item before is done with the ring
        while (nfill < min(a.nslots, ntot)) fill();
        ym.init();
        // An open first or last row and eq. (solver1)'s flux around one take the general path: no
        // open water from row kgen on, and no start in open water above row 0.
        const int kgen = ((OPEN && (a.open_edges & 8) != 0) || S1) ? a.ny - 1 : 0x7fffffff;
        bool opt = !(((OPEN && (a.open_edges & 4) != 0) || S1) && r0 == 0);
        // the last row whose vote may still send the march back to row r0-3: a general row k
        // needs the flux (k-3 | k-2), or the wall above row 0, from the rows before it
        const int klim = r0 == 0 ? 2 : r0 + 1;
        int k = opt ? r0 - 1 : k0, q = k - k0;
        unsigned hist = 0u;
        sw = opt;
        bool ok = acquire(), odd = false;
        const float* s = at(cs, q);
        bool fast = opt;
        while (ok) {
            if (fast) {
                if (!MAIN)
                    ok = fast_rows<true, true>(k, q, s, odd, kgen, klim);
                else if (wallx || a.walls)
                    ok = O.emax ? fast_rows<true, true>(k, q, s, odd, kgen, klim) : fast_rows<true, false>(k, q, s, odd, kgen, klim);
                else
                    ok = O.emax ? fast_rows<false, true>(k, q, s, odd, kgen, klim) : fast_rows<false, false>(k, q, s, odd, kgen, klim);
                if (!ok || k - 1 > r1) break;
                ym.after_fast();
                hist = 3u;
                if (opt && k + (odd ? 1 : 0) <= klim) {     // start over from row r0-3
                    k = k0;
                    q = 0;
                    cs = first;
                    s = at(cs, 0);
                    odd = false;
                    hist = 0u;
                    sw = false;
                    ym.init();
                }
                opt = false;
            }
            ok = slow_rows(k, q, s, odd, hist, kgen);
            if (!ok || k - 1 > r1) break;
            odd = false;
            fast = true;
        }
        if (!ok) {
            // a wait expired: the slots filled may still be in flight; let each land (bounded)
            // before going on
            for (; nread < nfill; ++nread) {
                mbar_wait(&bar[cs], (phase >> cs) & 1u, a.wait_cycles);
                cs = next_of(cs);
            }
            bad |= 2;
            return false;
        }
        bad |= !(chk_out.x + chk_out.y < RUNAWAY_SQ);
        chk_out = v2(0.f);
        write_samples(a, O, idx, b, lane);
        return true;
    }

    __device__ __forceinline__ void report() {
        bad |= !(chk_x.x + chk_x.y == 0.f);
        if (bad) atomicOr(a.err, (bad & 2) ? (ERRF_TIMEOUT | ERRF_NONFINITE) : ERRF_NONFINITE);
    }
};

template <bool SPH, bool FRIC, bool YF, bool S1, bool OPEN>
__global__ void __launch_bounds__(FUSED_WARPS * 32, 4)
k_step_fused(const __grid_constant__ StepMaps M, const __grid_constant__ StepArgs a) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int wib = threadIdx.x >> 5;
    const int gw = uniform(blockIdx.x * FUSED_WARPS + wib);
    const int b = blockIdx.y;
    if (gw >= a.nitems) return;
    FusedWarp<SPH, FRIC, YF, S1, OPEN> W(a);
    W.setup(smem_raw, wib);
    W.take_item(gw);
    if (W.lane == 0) {
        prefetch_map(&M.s);
        prefetch_map(&M.d);
        if (a.emax) prefetch_map(&M.mw);
    }
    if (a.limit && __all_sync(FULL, a.step > a.limit[b])) return;
    // a wait of an earlier launch expired: do not start new copies
    if (__any_sync(FULL, *reinterpret_cast<volatile int*>(a.err) & ERRF_TIMEOUT)) return;
    W.run_item(gw, b, step_out(&M, a));
    W.report();
}

// ------------------------------------------------------------------ batched, persistent
// Grid-wide barrier of a cooperative launch. Thread 0 of every block adds one arrival to the
// low half of *bar; the last arrival clears the count and advances the generation in the high
// half, which the others wait on for at most `limit` cycles before setting the timeout flag.
// Returns false when the run must stop (a wait expired here or, as of the arrival, anywhere
// else: the flag is read while waiting, so it costs no latency of its own).
__device__ __forceinline__ bool grid_sync(unsigned long long* bar, unsigned nblocks, long long limit, int* err) {
    __shared__ int go;
    asm volatile("fence.proxy.async.global;" ::: "memory");    // outputs before the next TMA reads
    __syncthreads();
    if (threadIdx.x == 0) {
        int ok = 1;
        __threadfence();
        const unsigned long long old = atomicAdd(bar, 1ull);
        const int flag = *reinterpret_cast<volatile int*>(err);
        const unsigned gen = (unsigned)(old >> 32);
        if ((unsigned)old == nblocks - 1) {
            // last arrival: count back to zero and generation + 1, in one atomic
            atomicAdd(bar, (1ull << 32) - (unsigned long long)nblocks);
        } else {
            volatile unsigned* vgen = reinterpret_cast<volatile unsigned*>(bar) + 1;
            const long long t0 = clock64();
            while (*vgen == gen)
                if (clock64() - t0 > limit) { ok = 0; break; }
        }
        __threadfence();
        if (!ok) atomicOr(err, ERRF_TIMEOUT);
        go = ok && !(flag & ERRF_TIMEOUT);
    }
    __syncthreads();
    asm volatile("fence.proxy.async.global;" ::: "memory");
    return __all_sync(FULL, go);
}

// Steps ctl[0]+1 .. ctl[1] of a batch of scenarios in one launch. Scenarios are taken in
// decreasing order of duration, so those still running at a step are the first nact[step]
// of `order`; the step's (scenario, item) pairs are numbered scenario-major and warp w of W
// takes numbers w, w + W, .. (cut_items makes items cost about the same; where W is a multiple
// of the items of a scenario, a warp draws the same item of every scenario, and one with a shore
// stays the dearer one. Handing them out by an atomic counter put a round trip to L2 before every
// item, and on small grids queued every warp at one address), then the warps meet at the grid barrier before the next step reads
// what this one wrote. A scenario that has stopped keeps its last state in the buffer of its
// last step's parity.
// With ALT (the alternating order) the odd-indexed steps (st - 1 odd) sweep y first: a second
// per-warp worker of the y-first kind shares the warp's ring, barriers and ring position.
template <bool SPH, bool FRIC, bool S1, bool OPEN, bool ALT>
__global__ void __launch_bounds__(FUSED_WARPS * 32, 4)
k_batch(const __grid_constant__ StepMaps2 MM, const __grid_constant__ StepArgs a, const __grid_constant__ BatchArgs B) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int wib = threadIdx.x >> 5;
    const unsigned gw = (unsigned)uniform(blockIdx.x * FUSED_WARPS + wib), nw = gridDim.x * FUSED_WARPS;
    const long long step0 = uniform64(B.ctl[0]), step_end = uniform64(B.ctl[1]);
    if (__any_sync(FULL, *reinterpret_cast<volatile int*>(a.err) & ERRF_TIMEOUT)) return;
    int taken = -1;                                // the item taken last
    FusedWarp<SPH, FRIC, false, S1, OPEN> W(a);
    W.setup(smem_raw, wib);
    FusedWarp<SPH, FRIC, true, S1, OPEN> WY(a);
    if (ALT) {
        WY.lane = W.lane; WY.ring = W.ring; WY.bar = W.bar; WY.bad = 0;
        WY.chk_x = WY.chk_out = v2(0.f);
    }
    for (long long st = step0 + 1; st <= step_end; ++st) {
        const bool yf = ALT && (((st - 1) & 1) != 0);
        if (yf) { WY.head = W.head; WY.phase = W.phase; }
        if (B.bnd) {
            // boundary input: the edge nodes of this step's input take the input at its model
            // time, then every block waits so that no TMA load reads an edge before it is set
            const BndRow& R = B.bnd_rows[st - step0 - 1];
            float* ei = (st & 1) ? B.eta[0] : B.eta[1];
            float* ui = ei + a.fs_out;
            float* vi = ei + 2 * a.fs_out;
            const int per = 2 * a.ny + 2 * a.nx;
            for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < per; idx += gridDim.x * blockDim.x) {
                const int e = idx < a.ny ? 0 : idx < 2 * a.ny ? 1 : idx < 2 * a.ny + a.nx ? 2 : 3;
                const int q = e == 0 ? idx : e == 1 ? idx - a.ny : e == 2 ? idx - 2 * a.ny : idx - 2 * a.ny - a.nx;
                bnd_apply(ei, ui, vi, a.pitch, a.nx, a.ny, e, q, B.bv, B.bnp, R.k[e], R.w[e]);
            }
            if (!grid_sync(reinterpret_cast<unsigned long long*>(B.ctl + 2), gridDim.x, a.wait_cycles, a.err)) break;
        }
        const bool odd = (st & 1) != 0;          // odd steps read buffer 0 and write buffer 1
        const bool mx = st % B.maxout == 0;
        StepOut O{odd ? &MM.m[0] : &MM.m[1], odd ? B.eta[1] : B.eta[0], mx ? B.emax : nullptr,
                  (B.grec && st % B.gout == 0) ? B.grec + (st / B.gout) * B.grec_row : nullptr,
                  (B.nrec && st % B.bndout == 0) ? B.nrec + (st / B.bndout) * B.nrec_row : nullptr};
        const int na = B.nact ? (st < B.nact_len ? uniform(__ldg(B.nact + st)) : 0) : B.nall;
        const unsigned total = (unsigned)na * (unsigned)a.nitems;
        bool ok = true;
        for (unsigned t = gw; ok && t < total; t += nw) {
            const int item = (int)(t % (unsigned)a.nitems), scen = uniform(__ldg(B.order + t / (unsigned)a.nitems));
            if (ALT || item != taken) {
                if (yf) WY.take_item(item);
                else W.take_item(item);
                taken = item;
            }
            ok = yf ? WY.run_item(item, scen, O) : W.run_item(item, scen, O);
        }
        if (yf) { W.head = WY.head; W.phase = WY.phase; }
        if (!ok && W.lane == 0) atomicOr(a.err, ERRF_TIMEOUT);
        if (!grid_sync(reinterpret_cast<unsigned long long*>(B.ctl + 2), gridDim.x, a.wait_cycles, a.err)) break;
    }
    W.report();
    if (ALT) WY.report();
}

// x-sweep alone: one warp per (row, strip of 56 columns).
template <bool SPH, bool FRIC, bool S1, bool OPEN>
__global__ void __launch_bounds__(128) k_xsweep(const StepArgs a) {
    const int lane = threadIdx.x & 31;
    const int gw = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int b = blockIdx.y;
    if (gw >= a.nstrips * a.ny) return;
    if (a.limit && a.step > a.limit[b]) return;
    const int strip = gw % a.nstrips, r = gw / a.nstrips;
    const int c0 = strip * XOUT - 4;
    const int cA = c0 + 2 * lane;
    const size_t boff = (size_t)b * a.plane;
    const SweepConst& K = a.K;
    float2 il = v2(0.f), ir = v2(0.f), k2 = v2(0.f);
    if (cA >= 0 && cA < a.nx) { il.x = a.xa[cA]; ir.x = a.xb[cA]; k2.x = a.xk[cA]; }
    if (cA + 1 >= 0 && cA + 1 < a.nx) { il.y = a.xa[cA + 1]; ir.y = a.xb[cA + 1]; k2.y = a.xk[cA + 1]; }
    XMet2 m{il, ir, k2};
    if (SPH) {
        const float2 f = v2(a.xrow[r]);
        m.hl = mul2(m.hl, f); m.hr = mul2(m.hr, f); m.k2 = mul2(m.k2, f);
    }
    float2 E, U, V, D;
    load_pair(a, boff, r, cA, E, U, V, D);
    xsweep2<FRIC, S1, OPEN>(E, U, V, D, m, K, lane, OPEN ? open_ends_x(a, cA) : 0u);
    const bool own = lane >= 2 && lane < 30;
    const bool va = own && cA < a.nx, vb = own && cA + 1 < a.nx;
    const size_t o = boff + (size_t)r * a.pitch + cA;
    const StepOut O = step_out(nullptr, a);
    emit_pair(a.eta_out + o, a.fs_out, va, vb, E, U, V);
    int bad = (va && runaway(E.x, U.x, V.x)) | (vb && runaway(E.y, U.y, V.y));
    if (O.emax && va) {
        float2 em = make_float2(a.emax[o], 0.f), sm = make_float2(a.emax[o + a.fs_max], 0.f);
        if (vb) { em.y = a.emax[o + 1]; sm.y = a.emax[o + 1 + a.fs_max]; }
        emit_max(a.K, a.emax + o, a.fs_max, va, vb, E, U, V, D, em, sm);
    }
    write_samples(a, O, gw, b, lane);
    if (bad) atomicOr(a.err, ERRF_NONFINITE);
}

// y-sweep alone: one warp per (strip of 64 columns, S rows).
template <bool SPH, bool FRIC, bool S1, bool OPEN>
struct YOnly {
    const StepArgs& a;
    const SweepConst& K;
    int lane, b, c0, cA, r0, r1;
    size_t boff;
    bool vA, vB;
    unsigned hist;             // rows k-1, k-2, k-3 (bits 0-2) wet at the start of the sweep
    YMarch2 ym;
    StepOut O;
    int bad;
    __device__ __forceinline__ YOnly(const StepArgs& a_) : a(a_), K(a_.K) {}
    __device__ __forceinline__ void emit(int r, float2 oe, float2 ow, float2 ot, float2 od) {
        if (r < r0 || r >= r1) return;
        const size_t o = boff + (size_t)r * a.pitch + cA;
        emit_pair(a.eta_out + o, a.fs_out, vA, vB, oe, ot, ow);
        bad |= (vA && runaway(oe.x, ot.x, ow.x)) | (vB && runaway(oe.y, ot.y, ow.y));
        if (O.emax && vA) {
            float2 em = make_float2(a.emax[o], 0.f), sm = make_float2(a.emax[o + a.fs_max], 0.f);
            if (vB) { em.y = a.emax[o + 1]; sm.y = a.emax[o + 1 + a.fs_max]; }
            emit_max(K, a.emax + o, a.fs_max, vA, vB, oe, ot, ow, od, em, sm);
        }
    }
    template <int PH>
    __device__ __forceinline__ void row(int k) {
        float2 E, U, V, D;
        load_pair(a, boff, k, cA, E, U, V, D);
        const float4 m2 = __ldg(a.ymet + k - 2);
        const bool oA = wet_mark(E.x, D.x, K), oB = wet_mark(E.y, D.y, K);
        if (hist == 7u) {
            float2 ne, nw, nt;
            const float2 dP = ym.bank[PH].d;
            ym.template fast<PH, SPH, FRIC, S1>(v2(m2.y), v2(m2.z), v2(m2.w), 0, 0.f, K, ne, nw, nt);
            ym.template store_row<PH>(E, V, U, D, add2(E, D));
            ym.after_fast();
            emit(k - 2, ne, nw, nt, dP);
        } else {
            ym.template slow<PH, SPH, FRIC, S1, OPEN>(E, V, U, D, oA, oB, m2, K,
                [&](int lag, float2 oe, float2 ow, float2 ot, float2 od) { emit(k - lag, oe, ow, ot, od); },
                OPEN ? open_end_y(a, k - 2) : 0);
            if (ym.pend) hist &= ~2u;                  // row k-2 waits for its (e)
        }
        hist = ((hist << 1) | (__all_sync(FULL, (oA || !vA) && (oB || !vB)) ? 1u : 0u)) & 7u;
    }
};

template <bool SPH, bool FRIC, bool S1, bool OPEN>
__global__ void __launch_bounds__(128) k_ysweep(const StepArgs a) {
    const int lane = threadIdx.x & 31;
    const int gw = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int b = blockIdx.y;
    if (gw >= a.nstrips * a.nseg) return;
    if (a.limit && a.step > a.limit[b]) return;
    YOnly<SPH, FRIC, S1, OPEN> Y(a);
    const int strip = gw % a.nstrips, seg = gw / a.nstrips;
    Y.lane = lane;
    Y.b = b;
    Y.c0 = strip * XWIN;
    Y.cA = Y.c0 + 2 * lane;
    Y.r0 = seg * a.S;
    Y.r1 = min(Y.r0 + a.S, a.ny);
    Y.boff = (size_t)b * a.plane;
    Y.vA = Y.cA < a.nx;
    Y.vB = Y.cA + 1 < a.nx;
    Y.hist = 0u;
    Y.bad = 0;
    Y.O = step_out(nullptr, a);
    Y.ym.init();
    int k = Y.r0 - 3;
    for (; k + 1 < Y.r1 + 3; k += 2) {
        Y.template row<0>(k);
        Y.template row<1>(k + 1);
    }
    if (k < Y.r1 + 3) Y.template row<0>(k);
    write_samples(a, Y.O, gw, b, lane);
    if (Y.bad) atomicOr(a.err, ERRF_NONFINITE);
}

}  // namespace cliffs
