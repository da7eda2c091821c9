// Node right-hand sides evaluated from exact window sums (FP64).
//
// Every model is written as: a coupled quantity f(x) of a node's stage input
// (the "exchange" variables of the paper's memory layout, Section III.B), whose
// window sums W = sum_{j in window incl. self} Q(f_j) arrive as exact
// fixed-point integers, and a local right-hand side.
#pragma once
#include "common.cuh"
#include "fastmath.cuh"
#include "hh_rates.cuh"

namespace simk {

// coupled_q() rounds a node's coupled quantity f(x) onto the grid 2^-F (sin and
// cos of the phase through the integer-only fixed_sincos for the Kuramoto
// models; u, v or V themselves otherwise), checking |f| < 2^lim (ok = false
// outside it or for a non-finite value).
// rhs() (general link matrices) takes the node's window sums W, its link count
// (wsize, the FHN/HH self-term multiplier) and a coupling scale cs = 1/K_i
// applied to the converted sums (the constants c then carry K = 1).  rhs_ring()
// takes the ring's window sums shifted right by ksh into int64 (ring_sums),
// OWN_OUT: without the node itself (unless it is one of its own links).

// Derived constants, computed once on the host in FP64.
struct ModelParams {
    double c[8];
    uint64_t a0[2];   // Kuramoto models: alpha = aq pi/2 + alpha0, alpha0 in [0, pi/2):
                      //   cos alpha0, sin alpha0 on the grid 2^-63 (non-negative multiples of 4)
    int64_t at[2];    //   (a0[0] - a0[1]) / 4 and (a0[0] + a0[1]) / 4 (turned_by_alpha0)
    int aq;           //   in 0..3
    int ksh;          // rings: right shift taking the exact window sums into int64
    uint64_t wsm;     // FHN and HH rings: wsize 2^(56 - ksh), for own_multiple
    int fx;           // FHN rings: 1 = the slope's bracket in integer arithmetic (kq, a54 in range)
    int64_t kq[4];    //   (sigma/K) b00, b01, b10, b11 times 2^(ksh + 67)
    int64_t a54;      //   a on the grid 2^-54
    MathTables tab;   // device tables of the fast elementary functions
    int64_t wsize;    // window size including the node itself (2R+1 or (2P+1)^3)
    int include_self; // 1: the node is one of its own links
};

template <int M> struct Model;

// Kuramoto coupling on a lattice.  On the ball and disk the window sums arrive
// rotated by -alpha: W' = W'c + i W's = sum over the window (the node itself
// included) of e^{-i alpha} Q(e^{i phi_j}), int64 on the grid 2^-F (their x pass
// rotates every node's quantity).  The cube keeps its sums unrotated and turns
// the node's own phase by +alpha instead (own_phase_turned), which gives the
// same T.  Then
//   T = Im[e^{-i phi_i} W'] = cos(phi_i) W's - sin(phi_i) W'c
//     = sum_j sin(phi_j - phi_i - alpha)   (the node's own term is -sin alpha),
// two 64 x 64 high products of the node's own (sin, cos) on the grid 2^-62 with
// the sums, on the grid 2^-(F-2).  The caller converts T once (correctly
// rounded, the grid's power of two folded into c[5]); the window without the
// node itself is T + sin alpha, the constant folded into c[4] on the host
// (quantisation makes the node's own rotated term differ from -sin alpha by a
// few units of 2^-F).
__device__ __forceinline__ double lattice_coupling(const int64_t (&f62)[2], int64_t W0, int64_t W1)
{
    return __ll2double_rn(mulhi_ss(f62[1], W0) - mulhi_ss(f62[0], W1));
}

// e^{i alpha0} (c + i s) from the grid 2^-62 onto 2^-61: four high products of the
// biased (s, c) with the non-negative cos alpha0, sin alpha0.  Each is short of its
// floor by at most one (2^-61 of the node's phase, whose own error is 2^-53.6).
__device__ __forceinline__ void turned_by_alpha0(const ModelParams &P, int64_t s, int64_t c, int64_t &s1, int64_t &c1)
{
    const uint64_t bs = biased62(s), bc = biased62(c);
    c1 = (int64_t)(umulhi_near(bc, P.a0[0]) - umulhi_near(bs, P.a0[1])) - P.at[0];
    s1 = (int64_t)(umulhi_near(bs, P.a0[0]) + umulhi_near(bc, P.a0[1])) - P.at[1];
}

// The node's own (sin, cos) on the grid 2^-62 turned by +alpha = aq pi/2 +
// alpha0: e^{i alpha0} (c + i s) by four high products with the non-negative cos
// alpha0, sin alpha0 (grid 2^-63, landing on 2^-61), back onto 2^-62 by one bit
// (|values| <= 1, so they stay below 2^62 + 2), then aq quarter turns.  With
// the turned phase the cross product of lattice_coupling takes the unrotated
// window sums: Im[e^{-i(phi + alpha)} S] = Im[e^{-i phi} e^{-i alpha} S] (the
// cube; the ball and disk rotate their sums instead).
__device__ __forceinline__ void own_phase_turned(const ModelParams &P, const int64_t (&f62)[2], int64_t (&t62)[2])
{
    int64_t s1, c1, ca, sa;
    turned_by_alpha0(P, f62[0], f62[1], s1, c1);
    switch (P.aq) { // times i^aq
    case 0: ca = c1; sa = s1; break;
    case 1: ca = -s1; sa = c1; break;
    case 2: ca = -c1; sa = -s1; break;
    default: ca = s1; sa = -c1; break;
    }
    t62[0] = (int64_t)((uint64_t)sa << 1);
    t62[1] = (int64_t)((uint64_t)ca << 1);
}

// Both Kuramoto models' coupling term on a lattice, c[5] T + c[4] (the whole
// slope of the plain model, the coupling part of dpsi/dt with inertia).
__device__ __forceinline__ double lattice_coupling_term(const ModelParams &P, const int64_t (&f62)[2], int64_t W0,
                                                        int64_t W1)
{
    return fma(P.c[5], lattice_coupling(f62, W0, W1), P.c[4]);
}

// Kuramoto coupling on a ring or a link matrix: T = Im[e^{-i(phi+alpha)} S] =
// cos(phi+alpha) S_sin - sin(phi+alpha) S_cos, with S the exact window sum
// (int128 on the grid 2^-F; without the node itself unless it is one of its own
// links) shifted right by sh bits into int64, and (cos, sin)(phi + alpha) from
// the node's own grid values by the angle-addition formula: four high products
// with the non-negative cos alpha0, sin alpha0 (grid 2^-61), then aq quarter
// turns.  Two signed high products give T on the grid 2^-(F - sh - 3).  No FP64
// instruction and no conversion until the caller's single one.
__device__ __forceinline__ int64_t ring_coupling(const ModelParams &P, const int64_t (&qo)[2], int F, int64_t S_s,
                                                 int64_t S_c)
{
    const int64_t s = qo[0] * (int64_t(1) << (62 - F)), c = qo[1] * (int64_t(1) << (62 - F));
    int64_t s1, c1, ca, sa;
    turned_by_alpha0(P, s, c, s1, c1);
    switch (P.aq) { // times i^aq
    case 0: ca = c1; sa = s1; break;
    case 1: ca = -s1; sa = c1; break;
    case 2: ca = -c1; sa = -s1; break;
    default: ca = s1; sa = -c1; break;
    }
    return mulhi_ss(ca, S_s) - mulhi_ss(sa, S_c);
}

// The same from a node's 128-bit window sums (node included), shifted here.
__device__ __forceinline__ int64_t ring_coupling_wide(const ModelParams &P, const int64_t (&qo)[2], int F,
                                                      const i128 (&W)[2], int sh)
{
    const i128 ss = P.include_self ? W[0] : W[0] - (i128)qo[0];
    const i128 sc = P.include_self ? W[1] : W[1] - (i128)qo[1];
    return ring_coupling(P, qo, F, (int64_t)(ss >> sh), (int64_t)(sc >> sh));
}

// floor(q wsize 2^-ksh) for a node's own quantity |q| < 2^54: one high product,
// (q 2^8) (wsize 2^(56 - ksh)) 2^-64.
__device__ __forceinline__ int64_t own_multiple(const ModelParams &P, int64_t q)
{
    return mulhi_su((int64_t)((uint64_t)q << 8), P.wsm);
}

// The shift and the scale of ring_coupling's T for a window of ws links (the
// node itself included or not): sh = max(0, ceil(log2 ws) + F - 61) keeps
// |S >> sh| < 2^62; the returned scale is coef 2^(sh + 3 - F), with coef the
// coupling constant (times the link-matrix node's 1/K_i).
__device__ __forceinline__ double ring_coupling_scale(int64_t ws, int F, double coef, int &sh)
{
    const int lg = ws > 1 ? 64 - __clzll((long long)(ws - 1)) : 0;
    sh = lg + F - 61 > 0 ? lg + F - 61 : 0;
    // coef 2^(sh + 3 - F) by the exponent field (coef is a normal double, the
    // power of two keeps it one)
    return __longlong_as_double(__double_as_longlong(coef) + ((long long)(sh + 3 - F) << 52));
}

// Kuramoto-Sakaguchi, Eq. (3) with m = 0, eps = 1 (Algorithm 1):
//   dphi_i/dt = omega - (mu/K) sum_{j in W(i)} sin(phi_i - phi_j + alpha)
//             = omega + (mu/K) [cos(phi_i+alpha) S_sin - sin(phi_i+alpha) S_cos],
// S_sin = sum_j sin phi_j, S_cos = sum_j cos phi_j (angle-difference identity,
// so the window only needs sums of sin and cos).
// c = {omega, mu/K, sin alpha, cos alpha}.  Coupled quantity (sin phi, cos phi).
template <> struct Model<0> {
    static constexpr int D = 1, NQ = 2, NX = 0, F = 53;
    static constexpr bool OWN_OUT = true;
    __device__ __forceinline__ static void coupled_q(const ModelParams &P, const double (&x)[D], int F, int,
                                                     bool &ok, int64_t (&q)[NQ])
    {
        int64_t s62, c62;
        fixed_sincos(x[0], P.tab, s62, c62, ok);
        q[0] = q62_to(s62, F);
        q[1] = q62_to(c62, F);
    }
    // Link matrices: a node of wsize links scales mu cs.
    __device__ __forceinline__ static void rhs(const ModelParams &P, int F_, const double (&)[NQ],
                                               const int64_t (&qo)[NQ], const i128 (&W)[NQ], const double *, double,
                                               double (&k)[D], int64_t wsize, double cs)
    {
        int sh;
        const double sc = ring_coupling_scale(wsize, F_, P.c[1] * cs, sh);
        k[0] = fma(sc, __ll2double_rn(ring_coupling_wide(P, qo, F_, W, sh)), P.c[0]);
    }
    // Rings: c[5] = (mu/K) 2^(ksh + 3 - F).
    __device__ __forceinline__ static void rhs_ring(const ModelParams &P, const int64_t (&qo)[NQ],
                                                    const int64_t (&S)[NQ], const double *, double, double (&k)[D])
    {
        k[0] = fma(P.c[5], __ll2double_rn(ring_coupling(P, qo, F, S[0], S[1])), P.c[0]);
    }
    // Lattices: c[4] = omega + (mu/K) sin alpha (omega with the node itself as a
    // link), c[5] = (mu/K) 2^-(F-2).
    __device__ __forceinline__ static void rhs_lattice(const ModelParams &P, const int64_t (&f62)[2], int64_t W0,
                                                       int64_t W1, const double *, double (&k)[D])
    {
        k[0] = lattice_coupling_term(P, f62, W0, W1);
    }
    __device__ __forceinline__ static void rhs_from_coupling(const ModelParams &, double c, const double *,
                                                             double (&k)[D])
    {
        k[0] = c;
    }
};

// FitzHugh-Nagumo, Eq. (2) with tau = 0, D = 0, I_app = 0 and the rotational
// coupling matrix B = [[b00, b01], [b10, b11]] = [[cos p, sin p], [-sin p, cos p]]:
//   du/dt = (u - u^3/3 - v + (sigma/K) [b00 Cu + b01 Cv]) / eps
//   dv/dt =  u + a        + (sigma/K) [b10 Cu + b11 Cv]
// with Cu = sum_{j in W(i)} (u_j - u_i) = W_u - wsize * Q(u_i), exact in fixed point.
// c = {1/eps, a, (sigma/K) b00/eps, (sigma/K) b01/eps, (sigma/K) b10, (sigma/K) b11}
// (constants folded on the host so that the RHS costs 9 FP64 instructions).
// Coupled quantity (u, v).
template <> struct Model<1> {
    static constexpr int D = 2, NQ = 2, NX = 0, F = 51;
    static constexpr bool OWN_OUT = false;
    __device__ __forceinline__ static void coupled_q(const ModelParams &, const double (&x)[D], int, int, bool &ok,
                                                     int64_t (&q)[NQ])
    {
        q[0] = to_fixed54(x[0], F, ok);
        q[1] = to_fixed54(x[1], F, ok);
    }
    __device__ __forceinline__ static void rhs(const ModelParams &P, int F_, const double (&fo)[NQ],
                                               const int64_t (&qo)[NQ], const i128 (&W)[NQ], const double *, double,
                                               double (&k)[D], int64_t wsize, double cs)
    {
        slope(P, fo[0], fo[1], cs * fixed_to_double_wide(W[0] - (i128)qo[0] * wsize, F_),
              cs * fixed_to_double_wide(W[1] - (i128)qo[1] * wsize, F_), k);
    }
    // Rings.  The stage was bound by the FP64 pipe (13 FP64 instructions and four
    // conversions per node), so the slope's bracket
    //   G_u = u - u^3/3 - v + (sigma/K) (b00 Cu + b01 Cv),  G_v = u + a + (sigma/K) (b10 Cu + b11 Cv)
    // is formed in integers on the grid 2^-54 from the grid values of u and v
    // (|u|, |v| < 8, so |u - u^3/3| < 171), and each slope takes one conversion; k_u = G_u / eps with
    // 1/eps in two parts (its rounding would be the largest systematic error left).
    // Every product is truncated at 2^-54 or finer (|error| of a bracket < 3 2^-54,
    // against roundings of 2^-53 |u| in FP64): rms error of k_u from this arithmetic
    // 2.3e-15 on the circle of radius 2, 3.3e-15 in FP64; 7e-16 against 3e-16 next to the
    // rest point, where the grid of u and v itself makes 3.3e-15.  Ring of 10^6: 35 -> 23 us
    // per stage launch.  fx = 0 (coupling constants or a beyond the range the host checks,
    // windows of fewer than 65 nodes): FP64, c[2..5] carrying 2^(ksh - F).
    __device__ __forceinline__ static void rhs_ring(const ModelParams &P, const int64_t (&qo)[NQ],
                                                    const int64_t (&S)[NQ], const double *, double, double (&k)[D])
    {
        const int64_t Cu = S[0] - own_multiple(P, qo[0]), Cv = S[1] - own_multiple(P, qo[1]); // grid 2^(ksh - 51)
        if (P.fx) {
            const int64_t qu = qo[0], qv = qo[1];
            const uint64_t ua = (uint64_t)(qu < 0 ? -qu : qu) << 9;            // |u| 2^60
            const uint64_t u2 = __umul64hi(ua, ua);                            // u^2 2^56
            const int64_t w = (1ll << 58) - (int64_t)(__umul64hi(u2, 0x5555555555555555ull) << 2); // (1 - u^2/3) 2^58
            const int64_t uw = mulhi_su(w, ua);                                // |u| (1 - u^2/3) 2^54
            const int64_t gu = (qu < 0 ? -uw : uw) - (qv << 3) + mulhi_ss(Cu, P.kq[0]) + mulhi_ss(Cv, P.kq[1]) + 1;
            const int64_t gv = (qu << 3) + P.a54 + mulhi_ss(Cu, P.kq[2]) + mulhi_ss(Cv, P.kq[3]) + 1;
            const double g = __ll2double_rn(gu);
            k[0] = fma(P.c[6], g, P.c[7] * g); // c[6] + c[7] = 2^-54 / eps
            k[1] = ll2double_scaled(gv, 54);
            return;
        }
        slope(P, ll2double_scaled(qo[0], F), ll2double_scaled(qo[1], F), __ll2double_rn(Cu), __ll2double_rn(Cv), k);
    }
    __device__ __forceinline__ static void slope(const ModelParams &P, double u, double v, double Cu, double Cv,
                                                 double (&k)[D])
    {
        const double w = fma(u * u, -1.0 / 3.0, 1.0);      // 1 - u^2/3
        const double local = fma(u, w, -v);                // u - u^3/3 - v
        k[0] = fma(P.c[0], local, fma(P.c[2], Cu, P.c[3] * Cv));
        k[1] = fma(P.c[4], Cu, fma(P.c[5], Cv, u + P.c[1]));
    }
};

// Hodgkin-Huxley, Eq. (1) as the classic neuron (V, m, h, n), textbook rates
// (V in mV, rates in 1/ms, rest near -65 mV):
//   Cm dV/dt = I_ext - gNa m^3 h (V-ENa) - gK n^4 (V-EK) - gL (V-EL) + (g/K) CV
//   dx/dt    = alpha_x(V) (1-x) - beta_x(V) x,   x in {m, h, n}
// with CV = sum_{j in W(i)} (V_j - V_i) = W_V - wsize * Q(V_i), exact in fixed point.
// c = {1/Cm, gNa, gK, gL, ENa, EK, EL, g/K}.  Coupled quantity V; the gates are
// local variables.  The rates come from integer arithmetic (hh_rates.cuh); 34
// FP64 instructions per node are left.
template <> struct Model<2> {
    static constexpr int D = 4, NQ = 1, NX = 3, F = 46;
    static constexpr bool OWN_OUT = false;
    __device__ __forceinline__ static void coupled_q(const ModelParams &, const double (&x)[D], int, int, bool &ok,
                                                     int64_t (&q)[NQ])
    {
        q[0] = to_fixed54(x[0], F, ok);
    }
    __device__ __forceinline__ static void rhs(const ModelParams &P, int F_, const double (&fo)[NQ],
                                               const int64_t (&qo)[NQ], const i128 (&W)[NQ], const double *X,
                                               double Iext, double (&k)[D], int64_t wsize, double cs)
    {
        slope(P, qo[0], fo[0], cs * fixed_to_double_wide(W[0] - (i128)qo[0] * wsize, F_), X, Iext, k);
    }
    // Rings: c[7] carries 2^(ksh - F).
    __device__ __forceinline__ static void rhs_ring(const ModelParams &P, const int64_t (&qo)[NQ],
                                                    const int64_t (&S)[NQ], const double *X, double Iext,
                                                    double (&k)[D])
    {
        slope(P, qo[0], ll2double_scaled(qo[0], F), __ll2double_rn(S[0] - own_multiple(P, qo[0])), X, Iext, k);
    }
    __device__ __forceinline__ static void slope(const ModelParams &P, int64_t q, double V, double CV, const double *X,
                                                 double Iext, double (&k)[D])
    {
        const double m = X[0], h = X[1], n = X[2];
        const HHRates r = hh_rates(q, P.tab);
        const double m3h = m * m * m * h, n4 = (n * n) * (n * n);
        const double I = Iext - P.c[1] * m3h * (V - P.c[4]) - P.c[2] * n4 * (V - P.c[5]) -
                         P.c[3] * (V - P.c[6]) + P.c[7] * CV;
        k[0] = I * P.c[0];
        // alpha (1 - x) - beta x, as it stands: from x = 1/2 on 1 - x is exact, and a gate near 1
        // keeps the relative accuracy of its slope.  alpha - (alpha + beta) x, one FP64
        // instruction less per gate, had 3.5 times the rms error at x in (0.95, 1) and took
        // 282 us per RK4 step at 10^6 neurons, this takes 305 (48.6 and 51.4 at 10^5); the sum
        // in integer arithmetic with the smaller of x and 1 - x: 306 and 51.1.
        k[1] = fma(r.am, 1.0 - m, -(r.bm * m));
        k[2] = fma(r.ah, 1.0 - h, -(r.bh * h));
        k[3] = fma(r.an, 1.0 - n, -(r.bn * n));
    }
};

// Kuramoto-Sakaguchi with inertia, Eq. (3) with m != 0, as a first-order system:
//   dphi/dt = psi,   dpsi/dt = ((mu/K) sum_{j in W(i)} sin(phi_j - phi_i - alpha) - eps psi) / m
// with sum_j sin(phi_j - phi_i - alpha) = cos(phi_i+alpha) S_sin - sin(phi_i+alpha) S_cos.
// c = {mu/(m K), eps/m, sin alpha, cos alpha}.  Coupled
// quantity (sin phi, cos phi);
// psi is a local variable.
template <> struct Model<3> {
    static constexpr int D = 2, NQ = 2, NX = 1, F = 53;
    static constexpr bool OWN_OUT = true;
    __device__ __forceinline__ static void coupled_q(const ModelParams &P, const double (&x)[D], int F, int,
                                                     bool &ok, int64_t (&q)[NQ])
    {
        int64_t s62, c62;
        fixed_sincos(x[0], P.tab, s62, c62, ok);
        q[0] = q62_to(s62, F);
        q[1] = q62_to(c62, F);
    }
    __device__ __forceinline__ static void rhs(const ModelParams &P, int F_, const double (&)[NQ],
                                               const int64_t (&qo)[NQ], const i128 (&W)[NQ], const double *X, double,
                                               double (&k)[D], int64_t wsize, double cs)
    {
        int sh;
        const double sc = ring_coupling_scale(wsize, F_, P.c[0] * cs, sh);
        k[0] = X[0];
        k[1] = fma(sc, __ll2double_rn(ring_coupling_wide(P, qo, F_, W, sh)), -P.c[1] * X[0]);
    }
    // Rings: c[5] = (mu/(m K)) 2^(ksh + 3 - F).
    __device__ __forceinline__ static void rhs_ring(const ModelParams &P, const int64_t (&qo)[NQ],
                                                    const int64_t (&S)[NQ], const double *X, double, double (&k)[D])
    {
        k[0] = X[0];
        k[1] = fma(P.c[5], __ll2double_rn(ring_coupling(P, qo, F, S[0], S[1])), -P.c[1] * X[0]);
    }
    // Lattices: c[4] = (mu/(m K)) sin alpha (0 with the node itself as a link),
    // c[5] = (mu/(m K)) 2^-(F-2).  The coupling term first, then the damping
    // (the order of the split cube node pass, which takes the coupling term
    // from the window pass).
    __device__ __forceinline__ static void rhs_lattice(const ModelParams &P, const int64_t (&f62)[2], int64_t W0,
                                                       int64_t W1, const double *X, double (&k)[D])
    {
        k[0] = X[0];
        k[1] = fma(-P.c[1], X[0], lattice_coupling_term(P, f62, W0, W1));
    }
    // The slope from the coupling term c of lattice_coupling_term.
    __device__ __forceinline__ static void rhs_from_coupling(const ModelParams &P, double c, const double *X,
                                                             double (&k)[D])
    {
        k[0] = X[0];
        k[1] = fma(-P.c[1], X[0], c);
    }
};

} // namespace simk
