// Device building blocks of the split shallow-water step (arXiv 1410.0753, "Numerics").
//
// One sweep of one line applies, in order, the inundation steps of section "Inundation
// algorithm": (a) mark dry nodes (h < h_min), (b) add a dry node to a wet neighbour's
// segment when h_j - d_j + d_i > h_min, with height h_min and the neighbour's velocities,
// (c) treat wet/dry interfaces as reflecting walls half a node from the wet node (mirror
// ghosts), (d) update every wet node by eq. (solver2), (e) limit a newly wetted node to half
// its neighbour's height and to its neighbour's speed. The readings where the paper is
// silent (tie-break in (b), ghost values, friction law and clamp, spherical terms) are the
// ones the FP64 oracle states; this file restates them for FP32.
//
// FP32 form. eq. (solver2) is written in the paper on the Riemann invariants p, q = u +- 2c
// (c = sqrt(g h)). In deep water c is ~200 m/s while a wave changes it by ~1e-4, below the
// FP32 resolution of p, so the kernels keep eta (not h) and evaluate the algebraically
// identical perturbation form of eq. (eqQ):
//   Q(b,a) dx = 1/2 (lam_b + lam_a)(w_b - w_a) +- (w_b + w_a)(c_b - c_a) + g (eta_b - eta_a),
//   c_b - c_a = g ((eta_b - eta_a) + (d_b - d_a)) / (c_b + c_a),
// and recover by increments (eqs. (stateu), (stateh)): du = (dp + dq)/2, dc = (dp - dq)/4,
// deta = dc (2c + dc)/g. At rest every term is exactly zero, so the lake at rest is kept
// bit for bit.
// Both the flux and the update are taken on the half sum and the half difference of the two
// invariants, a = (Q_p + Q_q)/2 and b = (Q_p - Q_q)/2:
//   a dx = 1/2 (w_b - w_a)(w_b + w_a) + g (eta_b - eta_a),
//   b dx = 1/2 (w_b - w_a)(c_b + c_a) + (w_b + w_a)(c_b - c_a),
//   du = -dt/2 (a_L + a_R) + k2 (w (a_R - a_L) + c (b_R - b_L)),
//   2 dc = -dt/2 (b_L + b_R) + k2 (w (b_R - b_L) + c (a_R - a_L)),  k2 = dt^2/(dx_L + dx_R),
// which takes 42 packed operations per sweep (friction included) where p and q one by one
// take 59; friction enters du alone. The metric tables hold 1/(2 dx), which carries the
// halves (an exact scaling).
//
// Layout of the work. Every lane owns two neighbouring nodes (columns A and B of its pair)
// and evaluates the update of both with packed FP32x2 instructions (add/mul/fma .f32x2).
// Steps (b), (c) and (e) are corrections applied per node, and only inside warp-uniform
// branches taken when some node of the warp needs them (a dry node that can flood, a wet
// node next to a dry one, a newly wetted node), so open water runs the update alone.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>
#include "internal.h"

namespace cliffs {

constexpr float GRAV = 9.81f;
constexpr float INV_GRAV = 1.0f / 9.81f;
constexpr float OUTSIDE_D = -1.0e30f;     // depth given to nodes beyond the domain edge
constexpr unsigned FULL = 0xffffffffu;
constexpr int XWIN = 64;                  // columns a warp holds in an x-sweep (2 per lane)
constexpr int XOUT = 56;                  // columns it can finish: 4-column halo per side

// ------------------------------------------------------------------ packed FP32x2
__device__ __forceinline__ float2 v2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
    unsigned long long r;
    asm("sub.rn.f32x2 %0, %1, %2;"
        : "=l"(r) : "l"(reinterpret_cast<unsigned long long&>(a)), "l"(reinterpret_cast<unsigned long long&>(b)));
    return reinterpret_cast<float2&>(r);
}

#ifndef CLIFFS_IEEE_MATH
// Hardware approximations (MUFU): one instruction each.
__device__ __forceinline__ float rsqrt_approx(float x) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float rcp_approx(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
// sqrt(x) for x >= 0 (x = 0 gives 0 through the 1e-30 floor)
__device__ __forceinline__ float sqrt_pos(float x) { return x * rsqrt_approx(fmaxf(x, 1e-30f)); }
__device__ __forceinline__ float div_pos(float a, float b) { return a * rcp_approx(b); }
// base-2 logarithm (log2(0) = -inf) and exponential (2^-inf = 0)
__device__ __forceinline__ float log2_fast(float x) {
    float r;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float exp2_fast(float x) {
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
#else
// Build option CLIFFS_IEEE_MATH: correctly rounded square root, reciprocal and quotient
// (IEEE round-to-nearest) in place of the hardware approximations.
__device__ __forceinline__ float rsqrt_approx(float x) { return __frsqrt_rn(x); }
__device__ __forceinline__ float rcp_approx(float x) { return __frcp_rn(x); }
__device__ __forceinline__ float sqrt_pos(float x) { return __fsqrt_rn(x); }
__device__ __forceinline__ float div_pos(float a, float b) { return __fdiv_rn(a, b); }
__device__ __forceinline__ float log2_fast(float x) { return log2f(x); }
__device__ __forceinline__ float exp2_fast(float x) { return exp2f(x); }
#endif

// c = sqrt(g h) of both nodes (h > 0 for wet nodes; dry nodes give NaN and are not used)
__device__ __forceinline__ float2 wave_speed2(float2 h) {
    const float2 gh = mul2(v2(GRAV), h);
#ifndef CLIFFS_IEEE_MATH
    return mul2(gh, make_float2(rsqrt_approx(gh.x), rsqrt_approx(gh.y)));
#else
    return make_float2(__fsqrt_rn(gh.x), __fsqrt_rn(gh.y));
#endif
}
__device__ __forceinline__ float wave_speed(float h) {
    const float gh = GRAV * h;
#ifndef CLIFFS_IEEE_MATH
    return gh * rsqrt_approx(gh);
#else
    return __fsqrt_rn(gh);
#endif
}

__device__ __forceinline__ bool wet_mark(float eta, float d, const SweepConst& K) {
    return (d >= K.dwall) && (eta + d >= K.hmin);              // (a): dry when h < h_min
}

// Friction (reading 4: Manning at time level n, alpha = g n^2 w sqrt(w^2 + t^2) / h^(4/3),
// clamped so that |alpha dt| <= |w|), as alpha dt = w k with
//   k = min(dt g n^2 sqrt(s2) h^(-4/3), 1) = 2^min(ex, 0),
//   ex = log2(dt g n^2 g^(4/3)) + log2(s2) / 2 - 8/3 log2(c),   s2 = w^2 + t^2, c^2 = g h:
// one power of two carries the clamp (ex >= 0: clamped, alpha dt = w). s2 = 0 gives k = 0.
// The adjoint's recomputation calls the same function, so both take the same clamp decision.
__device__ __forceinline__ float2 fric_k2(float2 w, float2 t, float2 c, const SweepConst& K, float2& s2, float2& ex) {
    s2 = fma2(w, w, mul2(t, t));
    const float2 ls = make_float2(log2_fast(s2.x), log2_fast(s2.y));
    const float2 lc = make_float2(log2_fast(c.x), log2_fast(c.y));
    ex = fma2(v2(0.5f), ls, fma2(v2(-8.0f / 3.0f), lc, K.lgf));
    return make_float2(exp2_fast(fminf(ex.x, 0.f)), exp2_fast(fminf(ex.y, 0.f)));
}
__device__ __forceinline__ float fric_k(float w, float t, float c, const SweepConst& K, float& s2, float& ex) {
    float2 s2p, exp_;
    const float2 k = fric_k2(v2(w), v2(t), v2(c), K, s2p, exp_);
    s2 = s2p.x;
    ex = exp_.x;
    return k.x;
}

struct Flux2 { float2 a, b, t; };   // half sum and half difference of Q_p and Q_q; eq. (pq3)'s

// eq. (eqQ) as a and b and the eq. (pq3) flux for t across two interfaces at once,
// perturbation form, per unit length (hi is half the inverse interval), from the differences
// (right node minus left node) of eta, w, t, d and the sums of w and c.
__device__ __forceinline__ Flux2 iface_core(float2 de, float2 dw, float2 dt, float2 dd, float2 sw, float2 sc,
                                            float2 hi) {
    const float2 z = mul2(v2(2.f * GRAV), de);
    const float2 num = fma2(v2(2.f * GRAV), dd, z);
#ifndef CLIFFS_IEEE_MATH
    const float2 dc = mul2(num, make_float2(rcp_approx(sc.x), rcp_approx(sc.y)));
#else
    const float2 dc = make_float2(__fdiv_rn(num.x, sc.x), __fdiv_rn(num.y, sc.y));
#endif
    Flux2 F;
    F.a = mul2(fma2(dw, sw, z), hi);
    F.b = mul2(fma2(dw, sc, mul2(sw, dc)), hi);
    F.t = mul2(mul2(sw, dt), hi);
    return F;
}
// between a left node a and a right node b
__device__ __forceinline__ Flux2 iface2(float2 ea, float2 wa, float2 ta, float2 da, float2 ca,
                                        float2 eb, float2 wb, float2 tb, float2 db, float2 cb,
                                        float2 hi) {
    return iface_core(sub2(eb, ea), sub2(wb, wa), sub2(tb, ta), sub2(db, da), add2(wb, wa), add2(cb, ca), hi);
}
// The right interfaces of a lane's nodes A (.x) and B (.y): (A|B) and (B|R), R the next
// lane's A. The differences are formed one by one: the pair (B, R) is not one of aligned
// registers, and putting it together would cost as many moves as the packed form saves.
__device__ __forceinline__ Flux2 iface_right(float2 E, float2 W, float2 T, float2 D, float2 C,
                                             float eR, float wR, float tR, float dR, float cR, float2 hi) {
    auto dif = [](float2 p, float r) { return make_float2(__fsub_rn(p.y, p.x), __fsub_rn(r, p.y)); };
    auto sum = [](float2 p, float r) { return make_float2(__fadd_rn(p.y, p.x), __fadd_rn(r, p.y)); };
    return iface_core(dif(E, eR), dif(W, wR), dif(T, tR), dif(D, dR), sum(W, wR), sum(C, cR), hi);
}

// Flux when the neighbour is the mirror ghost of the node (eta_g = eta, d_g = d, w_g = -w,
// t_g = t): a wall on its left gives b = 2 w c / dx, on its right the negation; a = t = 0.
__device__ __forceinline__ void ghost_left(float w, float c, float hi, float& a, float& b, float& t) {
    a = 0.f; b = 4.f * w * c * hi; t = 0.f;
}
__device__ __forceinline__ void ghost_right(float w, float c, float hi, float& a, float& b, float& t) {
    a = 0.f; b = -4.f * w * c * hi; t = 0.f;
}

// Open outer edge (no condition in the paper): the ghost beyond a wet edge node carries the
// node's outgoing Riemann invariant and the incoming invariant of still water at its depth,
// c0 = sqrt(g max(d, 0)). With delta = c - c0 (= g eta / (c + c0) for d > 0, else c):
//   right end (p leaves, q = -2 c0 enters): w_g = w/2 + delta, c_g = c + w/4 - delta/2;
//   left end  (q leaves, p = 2 c0 enters):  w_g = w/2 - delta, c_g = c - w/4 - delta/2;
// eta_g = eta + (c_g - c)(c_g + c)/g, the node's depth and transverse velocity. A ghost
// whose c_g would be negative is dry (c_g = 0). At rest (eta = w = 0) the ghost equals the
// node exactly, so the edge flux vanishes.
__device__ __forceinline__ void open_ghost(float e, float w, float d, float c, bool right,
                                           float& eg, float& wg, float& cg) {
    const bool deep = d > 0.f;
    const float c0 = deep ? wave_speed(d) : 0.f;
    const float delta = deep ? div_pos(GRAV * e, c + c0) : c;
    const float s = right ? 1.f : -1.f;
    wg = fmaf(0.5f, w, s * delta);
    float gam = fmaf(s * 0.25f, w, -0.5f * delta);           // c_g - c
    if (c + gam < 0.f) gam = -c;
    cg = c + gam;
    eg = fmaf(gam * (2.f * c + gam), INV_GRAV, e);
}

// Fluxes at the open edge of a node (scalar; the .x lane of the packed form). Kept out of
// line: open edges are rare, and inlined they would take registers from the sweeps.
static __device__ __noinline__ void open_flux(float e, float w, float t, float d, float c, float hi, bool right,
                                          float& fa, float& fb, float& tf, float& eg, float& wg, float& cg) {
    open_ghost(e, w, d, c, right, eg, wg, cg);
    const Flux2 F = right ? iface2(v2(e), v2(w), v2(t), v2(d), v2(c), v2(eg), v2(wg), v2(t), v2(d), v2(cg), v2(hi))
                          : iface2(v2(eg), v2(wg), v2(t), v2(d), v2(cg), v2(e), v2(w), v2(t), v2(d), v2(c), v2(hi));
    fa = F.a.x; fb = F.b.x; tf = F.t.x;
}

// (d): eq. (solver2) at two nodes given their left and right interface fluxes.
//   k2 = dt^2 / (dx_{j-1} + dx_j); nsdt = -dt tan(phi) / R in the spherical y-sweep (SRC).
// Friction (fric_k2) at time level n. D = -du and N = -2 dc are formed.
// With S1, eq. (solver1): the first-order term is dt Q(j+1, j-1) over dx_{j-1} + dx_j, given
// as the flux F1 between the two neighbours (per unit length) instead of the mean of L and R.
template <bool SRC, bool FRIC, bool S1 = false>
__device__ __forceinline__ void node_update2(float2 e, float2 w, float2 t, float2 c,
                                             const Flux2& L, const Flux2& R, float2 k2, float2 nsdt,
                                             const SweepConst& K,
                                             float2& e2, float2& w2, float2& t2, const Flux2* F1 = nullptr) {
    const float2 wk = mul2(w, k2), ck = mul2(c, k2);
    const float2 da = sub2(L.a, R.a), db = sub2(L.b, R.b);
    float2 D, N, T;
    if (S1) {
        const float2 f = add2(K.hdt, K.hdt);
        D = fma2(wk, da, mul2(f, F1->a));
        N = fma2(wk, db, mul2(f, F1->b));
        T = fma2(wk, sub2(L.t, R.t), mul2(f, F1->t));
    } else {
        // dt/2 (L + R) + w k2 (L - R), the two factors taken together
        const float2 fl = add2(K.hdt, wk), fr = sub2(K.hdt, wk);
        D = fma2(R.a, fr, mul2(L.a, fl));
        N = fma2(R.b, fr, mul2(L.b, fl));
        T = fma2(R.t, fr, mul2(L.t, fl));
    }
    D = fma2(ck, db, D);
    N = fma2(ck, da, N);
    if (FRIC) {
        float2 s2, ex;
        D = fma2(w, fric_k2(w, t, c, K, s2, ex), D);
    }
    if (SRC) N = fma2(mul2(nsdt, c), w, N);
    w2 = sub2(w, D);
    e2 = fma2(mul2(N, fma2(v2(-4.f), c, N)), v2(0.25f * INV_GRAV), e);
    t2 = fma2(T, K.ntr, t);
}

// (e): a node wetted in (b) against its source neighbour's state after (d).
__device__ __forceinline__ void cushion(float& e, float& w, float d, float hj, float wj) {
    const float hi = e + d;
    if (hi > 0.5f * hj) e = 0.5f * hj - d;
    if (fabsf(w) > fabsf(wj)) w = wj;
}

// (b) for one node i, dry at the start of the sweep and not a wall, with neighbours L and R
// (start-of-sweep eta, w, t and wet marks): the wetter neighbour (larger eta) wins, the
// left one on a tie. Returns the direction of the source (-1, +1) or 0.
__device__ __forceinline__ int flood1(float& e, float& w, float& t, float d,
                                      float eL, float wL, float tL, bool oL,
                                      float eR, float wR, float tR, bool oR, float hmin) {
    const bool okL = oL && (eL + d > hmin);
    const bool okR = oR && (eR + d > hmin);
    if (!(okL || okR)) return 0;
    const bool useR = okR && (!okL || eR > eL);
    e = hmin - d;                                              // height h_min
    w = useR ? wR : wL;
    t = useR ? tR : tL;
    return useR ? 1 : -1;
}

struct XMet2 { float2 hl, hr, k2; };   // per pair: 1/(2 dx_{j-1}), 1/(2 dx_j), dt^2/(dx_{j-1}+dx_j)

// x-sweep of one row segment held by a warp: lane l has nodes A = window column 2l (.x)
// and B = 2l + 1 (.y). Neighbours across lanes come by shuffles. On return (E, W, T) hold
// the sweep result; it is valid for window columns 4..59 (the outer 4 columns on each side
// lack their 3-node dependency radius), and up to the window's edge on a side where that
// edge is the domain's (bounded). W is the velocity along the row, T across it.
// ends: this lane's nodes at open outer edges, bits 1 A left, 2 A right, 4 B left, 8 B right.
template <bool FRIC, bool S1 = false, bool OPEN = false>
__device__ __forceinline__ void xsweep2(float2& E, float2& W, float2& T, float2 D, const XMet2& m,
                                        const SweepConst& K, int lane, unsigned ends = 0u, bool bounded = false) {
    const bool oA = wet_mark(E.x, D.x, K), oB = wet_mark(E.y, D.y, K);
    const unsigned bA = __ballot_sync(FULL, oA), bB = __ballot_sync(FULL, oB);
    // bounded: the window starts or ends at the domain's edge, where the first (last) lane's
    // outer neighbour is the wall's mirror ghost: the general path, which takes it so
    const bool allwet = (bA & bB) == FULL && !bounded;
    bool wA = oA, wB = oB;                 // wet after (b)
    int dirA = 0, dirB = 0;
    if (!allwet) {
        if (!oA) { W.x = 0.f; T.x = 0.f; }   // (a): a dry node is at rest
        if (!oB) { W.y = 0.f; T.y = 0.f; }
        const bool oL = lane > 0 && ((bB >> (lane - 1)) & 1u);
        const bool oR = lane < 31 && ((bA >> (lane + 1)) & 1u);
        const bool cA = !oA && D.x >= K.dwall && (oL || oB);
        const bool cB = !oB && D.y >= K.dwall && (oA || oR);
        if (__any_sync(FULL, cA || cB)) {
            const float eL = __shfl_up_sync(FULL, E.y, 1), eR = __shfl_down_sync(FULL, E.x, 1);
            const bool qA = cA && ((oL && eL + D.x > K.hmin) || (oB && E.y + D.x > K.hmin));
            const bool qB = cB && ((oA && E.x + D.y > K.hmin) || (oR && eR + D.y > K.hmin));
            if (__any_sync(FULL, qA || qB)) {
                const float wL = __shfl_up_sync(FULL, W.y, 1), tL = __shfl_up_sync(FULL, T.y, 1);
                const float wR = __shfl_down_sync(FULL, W.x, 1), tR = __shfl_down_sync(FULL, T.x, 1);
                const float eA0 = E.x, wA0 = W.x, tA0 = T.x;     // A as the source of B
                if (qA) {
                    dirA = flood1(E.x, W.x, T.x, D.x, eL, wL, tL, oL, E.y, W.y, T.y, oB, K.hmin);
                    wA = true;
                }
                if (qB) {
                    dirB = flood1(E.y, W.y, T.y, D.y, eA0, wA0, tA0, oA, eR, wR, tR, oR, K.hmin);
                    wB = true;
                }
            }
        }
    }
    const float2 C = wave_speed2(add2(E, D));
    // post-(b) state of the right neighbour of B (node A of lane + 1)
    const float eR = __shfl_down_sync(FULL, E.x, 1), wR = __shfl_down_sync(FULL, W.x, 1);
    const float tR = __shfl_down_sync(FULL, T.x, 1), dR = __shfl_down_sync(FULL, D.x, 1);
    const float cR = __shfl_down_sync(FULL, C.x, 1);
    // right interfaces of A and B: (A|B) and (B|R)
    Flux2 FR = iface_right(E, W, T, D, C, eR, wR, tR, dR, cR, m.hr);
    // left interfaces: (B_{l-1}|A) from the lane below, and (A|B)
    Flux2 FL;
    FL.a = make_float2(__shfl_up_sync(FULL, FR.a.y, 1), FR.a.x);
    FL.b = make_float2(__shfl_up_sync(FULL, FR.b.y, 1), FR.b.x);
    FL.t = make_float2(__shfl_up_sync(FULL, FR.t.y, 1), FR.t.x);
    bool wetL = true, wetR = true;
    if (!allwet) {
        // (c): walls between wet and dry nodes
        const unsigned w1A = __ballot_sync(FULL, wA), w1B = __ballot_sync(FULL, wB);
        wetL = lane > 0 && ((w1B >> (lane - 1)) & 1u);
        wetR = lane < 31 && ((w1A >> (lane + 1)) & 1u);
        if (!wetL) ghost_left(W.x, C.x, m.hl.x, FL.a.x, FL.b.x, FL.t.x);
        if (!wB) ghost_right(W.x, C.x, m.hr.x, FR.a.x, FR.b.x, FR.t.x);
        if (!wA) ghost_left(W.y, C.y, m.hl.y, FL.a.y, FL.b.y, FL.t.y);
        if (!wetR) ghost_right(W.y, C.y, m.hr.y, FR.a.y, FR.b.y, FR.t.y);
    }
    float2 gE = v2(0.f), gW = v2(0.f), gC = v2(0.f);   // open-edge ghosts of A (.x) and B (.y)
    if (OPEN && ends) {
        if ((ends & 1u) && wA) open_flux(E.x, W.x, T.x, D.x, C.x, m.hl.x, false, FL.a.x, FL.b.x, FL.t.x, gE.x, gW.x, gC.x);
        if ((ends & 2u) && wA) open_flux(E.x, W.x, T.x, D.x, C.x, m.hr.x, true, FR.a.x, FR.b.x, FR.t.x, gE.x, gW.x, gC.x);
        if ((ends & 4u) && wB) open_flux(E.y, W.y, T.y, D.y, C.y, m.hl.y, false, FL.a.y, FL.b.y, FL.t.y, gE.y, gW.y, gC.y);
        if ((ends & 8u) && wB) open_flux(E.y, W.y, T.y, D.y, C.y, m.hr.y, true, FR.a.y, FR.b.y, FR.t.y, gE.y, gW.y, gC.y);
    }
    Flux2 F1;
    if (S1) {
        // eq. (solver1): flux between the two neighbours of each node, mirror ghosts for dry ones
        float2 le = make_float2(__shfl_up_sync(FULL, E.y, 1), E.x), lw = make_float2(__shfl_up_sync(FULL, W.y, 1), W.x);
        float2 lt = make_float2(__shfl_up_sync(FULL, T.y, 1), T.x), ld = make_float2(__shfl_up_sync(FULL, D.y, 1), D.x);
        float2 lc = make_float2(__shfl_up_sync(FULL, C.y, 1), C.x);
        float2 re = make_float2(E.y, eR), rw = make_float2(W.y, wR), rt = make_float2(T.y, tR);
        float2 rd = make_float2(D.y, dR), rc = make_float2(C.y, cR);
        if (!allwet) {
            if (!wetL) { le.x = E.x; lw.x = -W.x; lt.x = T.x; ld.x = D.x; lc.x = C.x; }
            if (!wB) { re.x = E.x; rw.x = -W.x; rt.x = T.x; rd.x = D.x; rc.x = C.x; }
            if (!wA) { le.y = E.y; lw.y = -W.y; lt.y = T.y; ld.y = D.y; lc.y = C.y; }
            if (!wetR) { re.y = E.y; rw.y = -W.y; rt.y = T.y; rd.y = D.y; rc.y = C.y; }
        }
        if (OPEN && ends) {                // an open edge's neighbour is its ghost
            if (ends & 1u) { le.x = gE.x; lw.x = gW.x; lt.x = T.x; ld.x = D.x; lc.x = gC.x; }
            if (ends & 2u) { re.x = gE.x; rw.x = gW.x; rt.x = T.x; rd.x = D.x; rc.x = gC.x; }
            if (ends & 4u) { le.y = gE.y; lw.y = gW.y; lt.y = T.y; ld.y = D.y; lc.y = gC.y; }
            if (ends & 8u) { re.y = gE.y; rw.y = gW.y; rt.y = T.y; rd.y = D.y; rc.y = gC.y; }
        }
        F1 = iface2(le, lw, lt, ld, lc, re, rw, rt, rd, rc, mul2(m.k2, v2(0.5f * K.inv_dt2)));
    }
    float2 E2, W2, T2;
    node_update2<false, FRIC, S1>(E, W, T, C, FL, FR, m.k2, v2(0.f), K, E2, W2, T2, &F1);
    if (!allwet) {
        if (!wA) { E2.x = E.x; W2.x = W.x; T2.x = T.x; }
        if (!wB) { E2.y = E.y; W2.y = W.y; T2.y = T.y; }
        if (__any_sync(FULL, (dirA | dirB) != 0)) {
            const float hA = E2.x + D.x, hB = E2.y + D.y;
            const float hL = __shfl_up_sync(FULL, hB, 1), wLn = __shfl_up_sync(FULL, W2.y, 1);
            const float hR = __shfl_down_sync(FULL, hA, 1), wRn = __shfl_down_sync(FULL, W2.x, 1);
            const float w2A0 = W2.x, w2B0 = W2.y;
            if (dirA < 0) cushion(E2.x, W2.x, D.x, hL, wLn);
            else if (dirA > 0) cushion(E2.x, W2.x, D.x, hB, w2B0);
            if (dirB < 0) cushion(E2.y, W2.y, D.y, hA, w2A0);
            else if (dirB > 0) cushion(E2.y, W2.y, D.y, hR, wRn);
        }
    }
    E = E2; W = W2; T = T2;
}

// min(a, b), NaN when either is NaN (a NaN depth must not read as wet)
__device__ __forceinline__ float min_nan(float a, float b) {
    float r;
    asm("min.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}

// Reflecting walls of a lane's pair of columns: bits 1 A left, 2 A right, 8 B right (a window
// starts at an even column, so column 0 is an A).
__device__ __forceinline__ unsigned wall_ends_x(int cA, int nx) {
    return (cA == 0 ? 1u : 0u) | (cA == nx - 1 ? 2u : 0u) | (cA + 1 == nx - 1 ? 8u : 0u);
}

// xsweep2 when every node of the window inside the domain is wet at the start of the sweep
// (eq. (solver2)): steps (a), (b) and (e) change nothing then and (c) only puts the domain's
// own walls (wallx: some lane has one) or open edges (ends, as in xsweep2), so this is the
// sequence of operations xsweep2 takes in that case, without its votes. Lanes past the
// domain's edge compute values nobody reads.
template <bool FRIC, bool OPEN = false>
__device__ __forceinline__ void xsweep2_open(float2& E, float2& W, float2& T, float2 D, float2 H, const XMet2& m,
                                             const SweepConst& K, bool wallx, unsigned walls, unsigned ends = 0u) {
    const float2 C = wave_speed2(H);
    const float eR = __shfl_down_sync(FULL, E.x, 1), wR = __shfl_down_sync(FULL, W.x, 1);
    const float tR = __shfl_down_sync(FULL, T.x, 1), dR = __shfl_down_sync(FULL, D.x, 1);
    const float cR = __shfl_down_sync(FULL, C.x, 1);
    Flux2 FR = iface_right(E, W, T, D, C, eR, wR, tR, dR, cR, m.hr);
    Flux2 FL;
    FL.a = make_float2(__shfl_up_sync(FULL, FR.a.y, 1), FR.a.x);
    FL.b = make_float2(__shfl_up_sync(FULL, FR.b.y, 1), FR.b.x);
    FL.t = make_float2(__shfl_up_sync(FULL, FR.t.y, 1), FR.t.x);
    if (wallx) {
        // the first node's left interval equals its right one
        if (walls & 1u) ghost_left(W.x, C.x, m.hr.x, FL.a.x, FL.b.x, FL.t.x);
        if (walls & 2u) ghost_right(W.x, C.x, m.hr.x, FR.a.x, FR.b.x, FR.t.x);
        if (walls & 8u) ghost_right(W.y, C.y, m.hr.y, FR.a.y, FR.b.y, FR.t.y);
        if (OPEN && ends) {
            float ge, gw, gc;
            if (ends & 1u) open_flux(E.x, W.x, T.x, D.x, C.x, m.hr.x, false, FL.a.x, FL.b.x, FL.t.x, ge, gw, gc);
            if (ends & 2u) open_flux(E.x, W.x, T.x, D.x, C.x, m.hr.x, true, FR.a.x, FR.b.x, FR.t.x, ge, gw, gc);
            if (ends & 8u) open_flux(E.y, W.y, T.y, D.y, C.y, m.hr.y, true, FR.a.y, FR.b.y, FR.t.y, ge, gw, gc);
        }
    }
    float2 E2, W2, T2;
    node_update2<false, FRIC, false>(E, W, T, C, FL, FR, m.k2, v2(0.f), K, E2, W2, T2);
    E = E2; W = W2; T = T2;
}

// One row of a pair of columns in the y-sweep.
struct YRow {
    float2 e, w, t, d, c;     // w: velocity along the column (v), t: across it (u)
};

// y-sweep of a pair of columns as a march down the rows. Push k takes the sweep input of row
// k; the interface flux between rows k-2 and k-1 is formed once and shared, and row k-2 is
// updated (d). Rows k-2 and k-1 live in two banks whose roles swap every push (PH), so the
// march advances without copying them.
//  fast()  rows k-1, k-2 and k-3 wet at the start of the sweep: steps (a), (b), (c), (e) change
//          nothing, row k-2 is finished, and row k itself is not needed yet.
//  slow()  the general case: (b) on row k-1 with neighbours k-2 and k, (c) and (d) on row k-2,
//          (e) on row k-3 against rows k-4 and k-2. It emits row k-2 at once when none of its
//          nodes was flooded in (b), else row k-2 waits for the next push (pend).
// What only slow() needs besides (the marks, row k-3 and row k-4 after (d)) is not carried
// through fast(): after_fast() sets it to what it then must be (wet, nothing flooded, and no
// (e) that would look at the rows), so it takes no registers in open water.
struct YMarch2 {
    YRow bank[2];             // [PH]: row k-2 after (b); [1-PH]: row k-1 as input (c: wet nodes)
    Flux2 fb[2];              // [PH]: flux (k-3 | k-2)
    unsigned fl;              // marks: bits 0-5 row k-2, bits 6-11 row k-3 (see mark_bits)
    bool pend;                // row k-3 waits for (e) (warp-uniform)
    float2 e3, w3, t3, d3;    // row k-3 after (d)
    float2 h4, w4;            // row k-4 after (d): height, velocity
    float2 pe, pw, pt, pd, pc;   // row k-3 after (b) (eq. (solver1) only)

    __device__ __forceinline__ void init() {
        for (int i = 0; i < 2; ++i) {
            bank[i].e = bank[i].w = bank[i].t = bank[i].c = v2(0.f);
            bank[i].d = v2(OUTSIDE_D);
            fb[i].a = fb[i].b = fb[i].t = v2(0.f);
        }
        pe = pw = pt = pc = v2(0.f);
        pd = v2(OUTSIDE_D);
        after_fast();
        fl = 0u;                                       // before the first row: dry
    }
    __device__ __forceinline__ void after_fast() {
        fl = 3u | (3u << 6);
        pend = false;
        e3 = w3 = t3 = d3 = h4 = w4 = v2(0.f);
    }

    // wet after (b) (A 1, B 2); flooded from row k-1 (A 4, B 8) or from row k+1 (A 16, B 32)
    static __device__ __forceinline__ unsigned mark_bits(bool wA, bool wB, int dA, int dB) {
        return (wA ? 1u : 0u) | (wB ? 2u : 0u) | (dA < 0 ? 4u : dA > 0 ? 16u : 0u) | (dB < 0 ? 8u : dB > 0 ? 32u : 0u);
    }

    // eq. (solver1): flux between rows k-3 and k-1 around row k-2 (P), with mirror ghosts
    // of P for a neighbour row that is dry after (b) (marks f3 and w1); at an open edge (pend_
    // 1: row k-2 is the first row, 2: the last) the neighbour beyond it is the open ghost
    __device__ __forceinline__ Flux2 f1(const YRow& P, const YRow& B1, bool open, float2 k2, const SweepConst& K,
                                        unsigned f3 = 3u, unsigned w1 = 3u, int edge = 0, float2 ge = v2(0.f),
                                        float2 gw = v2(0.f), float2 gc = v2(0.f)) const {
        float2 le = pe, lw = pw, lt = pt, ld = pd, lc = pc;
        float2 re = B1.e, rw = B1.w, rt = B1.t, rd = B1.d, rc = B1.c;
        if (!open) {
            if (!(f3 & 1u)) { le.x = P.e.x; lw.x = -P.w.x; lt.x = P.t.x; ld.x = P.d.x; lc.x = P.c.x; }
            if (!(f3 & 2u)) { le.y = P.e.y; lw.y = -P.w.y; lt.y = P.t.y; ld.y = P.d.y; lc.y = P.c.y; }
            if (!(w1 & 1u)) { re.x = P.e.x; rw.x = -P.w.x; rt.x = P.t.x; rd.x = P.d.x; rc.x = P.c.x; }
            if (!(w1 & 2u)) { re.y = P.e.y; rw.y = -P.w.y; rt.y = P.t.y; rd.y = P.d.y; rc.y = P.c.y; }
        }
        if (edge == 1) { le = ge; lw = gw; lt = P.t; ld = P.d; lc = gc; }
        if (edge == 2) { re = ge; rw = gw; rt = P.t; rd = P.d; rc = gc; }
        return iface2(le, lw, lt, ld, lc, re, rw, rt, rd, rc, mul2(k2, v2(0.5f * K.inv_dt2)));
    }

    // hi, k2, nsdt: 1/(2 dy), dt^2/(dy + dy) and the source factor of row k-2. edge: row k-2 is
    // the first row (bit 1, hl = its left 1/(2 dy)) or the last (bit 2) of a grid with walls.
    template <int PH, bool SRC, bool FRIC, bool S1>
    __device__ __forceinline__ void fast(float2 hi, float2 k2, float2 nsdt, int edge, float hl, const SweepConst& K,
                                         float2& ne, float2& nw, float2& nt) {
        YRow& P = bank[PH];
        YRow& B1 = bank[1 - PH];
        Flux2& F2 = fb[1 - PH];
        F2 = iface2(P.e, P.w, P.t, P.d, P.c, B1.e, B1.w, B1.t, B1.d, B1.c, hi);
        if (edge) {
            if (edge & 1) {
                ghost_left(P.w.x, P.c.x, hl, fb[PH].a.x, fb[PH].b.x, fb[PH].t.x);
                ghost_left(P.w.y, P.c.y, hl, fb[PH].a.y, fb[PH].b.y, fb[PH].t.y);
            }
            if (edge & 2) {
                ghost_right(P.w.x, P.c.x, hi.x, F2.a.x, F2.b.x, F2.t.x);
                ghost_right(P.w.y, P.c.y, hi.y, F2.a.y, F2.b.y, F2.t.y);
            }
        }
        Flux2 F1;
        if (S1) F1 = f1(P, B1, true, k2, K);
        node_update2<SRC, FRIC, S1>(P.e, P.w, P.t, P.c, fb[PH], F2, k2, nsdt, K, ne, nw, nt, &F1);
        if (S1) { pe = P.e; pw = P.w; pt = P.t; pd = P.d; pc = P.c; }
    }

    // row k takes the freed bank (c is used when its nodes are wet)
    template <int PH>
    __device__ __forceinline__ void store_row(float2 E0, float2 W0, float2 T0, float2 D0, float2 H0) {
        bank[PH].e = E0; bank[PH].w = W0; bank[PH].t = T0; bank[PH].d = D0;
        bank[PH].c = wave_speed2(H0);
    }

    // m2: metric of row k-2 (1/(2 dy_{j-1}), 1/(2 dy_j), dt^2/(dy_{j-1}+dy_j), -dt tan(phi)/R).
    // emit(lag, e, w, t, d) receives finished rows k - lag, in order; o0A/o0B: the incoming
    // row's wet marks. edge: row k-2 is the first row of the grid at an open edge (1) or the
    // last (2), else 0.
    template <int PH, bool SRC, bool FRIC, bool S1, bool OPEN, class Emit>
    __device__ __forceinline__ void slow(float2 E0, float2 W0, float2 T0, float2 D0, bool o0A, bool o0B,
                                         float4 m2, const SweepConst& K, Emit&& emit, int edge = 0) {
        YRow& P = bank[PH];
        YRow& B1 = bank[1 - PH];
        Flux2& F3 = fb[PH];
        Flux2& F2 = fb[1 - PH];
        const unsigned f = fl;
        const bool PwA = f & 1u, PwB = f & 2u, f3A = f & 64u, f3B = f & 128u;
        const bool PoA = PwA && !(f & 20u), PoB = PwB && !(f & 40u);
        // (a)/(b) on row k-1 (input held in B1), neighbours row k-2 (P) and row k (new). Row k-2 is
        // held after (b) only: when it was wet at the start its values are its start-of-sweep ones
        bool wA = wet_mark(B1.e.x, B1.d.x, K), wB = wet_mark(B1.e.y, B1.d.y, K);
        int dA = 0, dB = 0;
        if (!wA) {
            B1.w.x = 0.f; B1.t.x = 0.f;
            if (B1.d.x >= K.dwall) {
                dA = flood1(B1.e.x, B1.w.x, B1.t.x, B1.d.x, P.e.x, P.w.x, P.t.x, PoA, E0.x, W0.x, T0.x, o0A, K.hmin);
                wA = dA != 0;
            }
        }
        if (!wB) {
            B1.w.y = 0.f; B1.t.y = 0.f;
            if (B1.d.y >= K.dwall) {
                dB = flood1(B1.e.y, B1.w.y, B1.t.y, B1.d.y, P.e.y, P.w.y, P.t.y, PoB, E0.y, W0.y, T0.y, o0B, K.hmin);
                wB = dB != 0;
            }
        }
        B1.c = wave_speed2(add2(B1.e, B1.d));
        F2 = iface2(P.e, P.w, P.t, P.d, P.c, B1.e, B1.w, B1.t, B1.d, B1.c, v2(m2.y));
        // (c): walls, then (d) on row k-2
        Flux2 L = F3, R = F2;
        if (PwA && !f3A) ghost_left(P.w.x, P.c.x, m2.x, L.a.x, L.b.x, L.t.x);
        if (PwA && !wA) ghost_right(P.w.x, P.c.x, m2.y, R.a.x, R.b.x, R.t.x);
        if (PwB && !f3B) ghost_left(P.w.y, P.c.y, m2.x, L.a.y, L.b.y, L.t.y);
        if (PwB && !wB) ghost_right(P.w.y, P.c.y, m2.y, R.a.y, R.b.y, R.t.y);
        float2 ge = v2(0.f), gw = v2(0.f), gc = v2(0.f);
        if (OPEN && edge) {
            // an open outer edge: the flux across it from the open ghost (wet nodes only)
            const bool right = edge == 2;
            Flux2 Fo;
            open_flux(P.e.x, P.w.x, P.t.x, P.d.x, P.c.x, right ? m2.y : m2.x, right, Fo.a.x, Fo.b.x, Fo.t.x,
                      ge.x, gw.x, gc.x);
            open_flux(P.e.y, P.w.y, P.t.y, P.d.y, P.c.y, right ? m2.y : m2.x, right, Fo.a.y, Fo.b.y, Fo.t.y,
                      ge.y, gw.y, gc.y);
            Flux2& S = right ? R : L;
            if (PwA) { S.a.x = Fo.a.x; S.b.x = Fo.b.x; S.t.x = Fo.t.x; }
            if (PwB) { S.a.y = Fo.a.y; S.b.y = Fo.b.y; S.t.y = Fo.t.y; }
        }
        float2 ne, nw, nt;
        Flux2 F1;
        if (S1) F1 = f1(P, B1, false, v2(m2.z), K, f >> 6, (wA ? 1u : 0u) | (wB ? 2u : 0u), edge, ge, gw, gc);
        node_update2<SRC, FRIC, S1>(P.e, P.w, P.t, P.c, L, R, v2(m2.z), v2(m2.w), K, ne, nw, nt, &F1);
        if (!PwA) { ne.x = P.e.x; nw.x = P.w.x; nt.x = P.t.x; }
        if (!PwB) { ne.y = P.e.y; nw.y = P.w.y; nt.y = P.t.y; }
        // rows out: row k-3 after (e), against row k-4 (h4, w4) or row k-2 (ne, nw), if it waits;
        // then row k-2 unless it has to wait for its own (e)
        const bool wait = __any_sync(FULL, (f & 60u) != 0u);
        const int last = wait ? 3 : 2;
        for (int lag = pend ? 3 : 2; lag >= last; --lag) {
            float2 oe = ne, ow = nw, ot = nt, od = P.d;
            if (lag == 3) {
                oe = e3; ow = w3; ot = t3; od = d3;
                if (f & (20u << 6)) cushion(oe.x, ow.x, d3.x, (f & (4u << 6)) ? h4.x : ne.x + P.d.x, (f & (4u << 6)) ? w4.x : nw.x);
                if (f & (40u << 6)) cushion(oe.y, ow.y, d3.y, (f & (8u << 6)) ? h4.y : ne.y + P.d.y, (f & (8u << 6)) ? w4.y : nw.y);
            }
            emit(lag, oe, ow, ot, od);
        }
        h4 = add2(e3, d3);
        w4 = w3;
        e3 = ne; w3 = nw; t3 = nt; d3 = P.d;
        if (S1) { pe = P.e; pw = P.w; pt = P.t; pd = P.d; pc = P.c; }
        fl = mark_bits(wA, wB, dA, dB) | ((f & 63u) << 6);
        pend = wait;
        store_row<PH>(E0, W0, T0, D0, add2(E0, D0));
    }
};

}  // namespace cliffs
