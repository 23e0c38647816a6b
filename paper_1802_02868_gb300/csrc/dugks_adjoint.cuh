// dugks_adjoint.cuh -- reverse-mode (adjoint) sweep of one DUGKS step and of
// the initialisation, written by hand as the transpose of the forward step
// (Sec. 2.2 procedure).
//
// Forward step n leaves what the reverse step reads (k_step, MODE_PLANES):
//   mu, grad mu, lap mu, grad phi, u, p, grad p and bar-plus of every cell.
// Reverse, given the adjoint xb of the state at n+1:
//   ka_face  one thread per face: reconstruction and face macros again, then their
//            transpose -> what each face gives its bar values and aux fields
//   ka_cell  gathers the gifts of a cell's faces (the transpose of the
//            reconstruction), then bar-plus -> adjoint of tilde, of u, p, phi, mu
//            and the gradients
//   ka_tail  transpose grad p, then p, u, F -> adjoint of tilde f, phi, grad mu, ...;
//            transpose grad mu, lap mu, then mu -> adjoint of phi, lap phi;
//            transpose grad phi, lap phi, then phi = sum g -> adjoint of tilde g
// Nothing is scattered: every value has one writer, so a gradient comes out the
// same every time.  The parameters kappa and lambda (the mobility) collect their
// adjoints in FP64, one slot per warp of a kernel, added up per instance at the
// end.
//
// One warp takes a run of 32 cells or faces of a row (AdjSeg), so that the work of
// a small mesh spreads over all SM sub-partitions; the point transpose is that of
// the regrouped equilibria and sources (dugks_fp64.cuh), about a third of the
// operations of the transpose of the separate ones.
#pragma once
#include "dugks_fused.cuh"

namespace dugks {

// Gifts of a face, one plane each: to the bar f and bar g of the six flux
// directions (fset order), to every bar f (AS), to +-bar f along the face (AM), to
// every bar g (AP), and to the aux fields.
constexpr int AF = 0, AG = 6, AS = 12, AM = 13, AP = 14, AX = 15, NFP = 23;

// positions i .. i + 31 of row j of an instance; -1 is the face at a low wall.  Runs
// follow each other up a column of 32, so that the warps of a block read each
// other's rows.
struct AdjSeg {
    int inst, i, j, axis;   // axis: of the faces
};

template <typename T>
struct AdjPlanes {
    const T *xf, *xg;   // adjoint of the tracked state at step n+1 [Q][N]
    T *af, *ag;         // adjoint of the tracked state at step n   [Q][N]
    T *face[2];         // [NFP][NF] per axis: the face between a cell and its high neighbour at
                        // the cell's index; one at a low wall at N + the other axis' record
    T *phi, *mu, *lapmu, *gmx, *gmy, *gfx, *gfy, *gpx, *gpy, *p, *ux, *uy, *lapphi;  // [N]
    double *lam_face, *lam_cell, *lam_macro, *kap, *kap0;   // slots of the parameters' adjoints, per warp
    long long N, NF;
};

template <typename T>
__device__ __forceinline__ T recip(T x);
template <>
__device__ __forceinline__ float recip<float>(float x) { return __frcp_rn(x); }
template <>
__device__ __forceinline__ double recip<double>(double x) { return fp64::rcp(x); }

// add a warp's sum of v to its slot
template <typename T>
__device__ __forceinline__ void slot_add(double *slot, T v)
{
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) *slot += (double)v;
}

// A point of the scheme (a cell in bar-plus, or a face) and its adjoint.
template <typename T>
struct APt {
    T phi, ux, uy, p, mu, lmu, gmx, gmy, gfx, gfy, gpx, gpy;
};

// Transpose of bar-plus of a cell (A = -1: all directions) or of the originals of
// a face of axis A (its flux directions) with respect to the point's variables:
// a f + b f^eq + c F^f and ga g + ..., given their adjoints ob, yb.  Returns a
// (a cell: b = 1 - a); fsum is sum f ob, the adjoint of a.  B: the adjoint of the
// point, with that of rho and of the weights in phi's; of a cell's u and p, and at a
// face, whose p and u are formed from its bars, of sum f (in p) and sum xi f (in u).
// A cell's u lacks the share b rho sum w xi ob of the equilibrium's term linear in u,
// which the relaxation cancels in the adjoint of tilde (ka_cell): its effect on F and
// rho is in B already.
template <typename T, int A>
__device__ __forceinline__ T point_adj(const InstDev &I, const APt<T> &s, const T (&ob)[Q], const T (&yb)[Q], T fsum, bool wall,
                                       APt<T> &B, T &lam)
{
    constexpr bool CELL = A < 0;
    const ParT<T> &Pr = par<T>(I);
    const PtC<T> &C = CELL ? cellc<T>(I) : facec<T>(I);
    const T rho = Pr.rhoB + Pr.drho * (s.phi - Pr.phiB), irho = recip(rho);
    const T Fx = -s.phi * s.gmx + (rho - Pr.rho_ref) * Pr.gxa, Fy = -s.phi * s.gmy + (rho - Pr.rho_ref) * Pr.gya;
    const T D = (s.phi - Pr.phiB) * Pr.hmuB + (Pr.phiA - s.phi) * Pr.hmuA, X = D * rho;
    const T kx = CELL ? T(2) : T(1);
    const T r = recip(C.k6 + kx * X);
    const T a = (CELL ? C.k6 - X : C.k6) * r, b = C.nb * X * r, c = C.nc * r;
    const T ECx = Fx + C.cd * s.gfx, ECy = Fy + C.cd * s.gfy;      // F + c_s^2 grad rho
    const T uF = s.ux * Fx + s.uy * Fy, uE = s.ux * ECx + s.uy * ECy;
    const T rl = rho * s.lmu, src = C.cgl * rl + uF;
    const T rho3 = rho * T(1.0 / 3.0);
    const T KL = CELL ? b * rho3 : T(0), K1 = (CELL ? T(0) : b * rho3) - c * uE;   // KL: the share left out
    const T fx = c * Fx, fy = c * Fy, ex = c * ECx, ey = c * ECy;
    const T Gx = Fx - s.gpx, Gy = Fy - s.gpy, Pg = C.gc * s.phi * irho, gx = Pg * Gx, gy = Pg * Gy;
    const T ug = s.ux * gx + s.uy * gy, D2 = C.gb * s.phi - ug;
    const T s0 = T(-1.5) * (s.ux * s.ux + s.uy * s.uy);
    // directions: z, y are the adjoints times the weight over the diagonals'
    T K0b = 0, K1b = 0, fxb = 0, fyb = 0, exb = 0, eyb = 0, A2b = 0, D2b = 0, gxb = 0, gyb = 0, s0b = 0, uxb = 0, uyb = 0;
#pragma unroll
    for (int q = 0; q < Q; q++) {
        if (!CELL && ca(q, CELL ? 0 : A) == 0) continue;
        const T w = q == 0 ? T(16) : q < 5 ? T(4) : T(1);
        const T z = w * ob[q], y = w * yb[q];
        const T xu = xi_dot<T>(q, s.ux, s.uy), sq = s0 + (q == 0 ? T(0) : xu * (T(4.5) * xu + T(3)));
        const T zs = z * sq, ys = y * sq;
        K0b += z;
        K1b += zs;
        A2b += y;
        D2b += ys;
        T sb = z * K1 + y * D2;
        if (q > 0) {
            if (cx(q)) { fxb += T(cx(q)) * z; exb += T(cx(q)) * zs; gxb += T(cx(q)) * (y + ys); }
            if (cy(q)) { fyb += T(cy(q)) * z; eyb += T(cy(q)) * zs; gyb += T(cy(q)) * (y + ys); }
            sb += z * xi_dot<T>(q, ex, ey) + y * xi_dot<T>(q, gx, gy);
            const T xub = CELL ? T(9) * xu * (sb + z * KL) + T(3) * sb : sb * (T(9) * xu + T(3));
            if (cx(q)) uxb += T(cx(q)) * xub;
            if (cy(q)) uyb += T(cy(q)) * xub;
        }
        s0b += CELL ? sb + z * KL : sb;
    }
    uxb -= T(3) * s.ux * s0b;
    uyb -= T(3) * s.uy * s0b;
    T phib = C.gb * D2b, rhob = 0, Hb = A2b;
    if (CELL) {
        // H of the rest direction is phi - (1 - w_0) eta mu: the adjoint of eta mu
        // is sum w (yb_q - yb_0), formed from the differences, for yb hardly varies
        // with q and the sum of separately rounded weights would leave a bias
        phib += C.gb36 * yb[0];
        Hb = 0;
#pragma unroll
        for (int q = 1; q < Q; q++) Hb += (q < 5 ? T(4) : T(1)) * (yb[q] - yb[0]);
    }
    const T mub = C.gbe * Hb;
    lam += C.dgbe * s.mu * Hb;
    // g: D2 = gb phi - u.G', A2 = gbe mu - u.G', G' = P (F - grad p), P = gc phi / rho
    const T ugb = -(A2b + D2b);
    uxb += ugb * gx;
    uyb += ugb * gy;
    gxb += ugb * s.ux;
    gyb += ugb * s.uy;
    const T Pb = gxb * Gx + gyb * Gy;
    T Fxb = Pg * gxb, Fyb = Pg * gyb;
    B.gpx = -Fxb;
    B.gpy = -Fyb;
    phib += C.gc * irho * Pb;
    rhob -= Pg * irho * Pb;
    // f: K0 = b p - c (cgl rho lap mu + u.F), K1 = b rho / 3 - c u.E, c F, c E
    T bb = s.p * K0b + rho3 * K1b;
    T cb = -(src * K0b) - uE * K1b + Fx * fxb + Fy * fyb + ECx * exb + ECy * eyb;
    T pb = b * K0b;
    const T tb = -c * K0b, uEb = -c * K1b;
    rhob += C.cgl * s.lmu * tb + b * T(1.0 / 3.0) * K1b;
    T lmub = C.cgl * rho * tb;
    lam += C.dcgl * rl * tb;
    const T ExB = c * exb + uEb * s.ux, EyB = c * eyb + uEb * s.uy;
    Fxb += c * fxb + tb * s.ux + ExB;
    Fyb += c * fyb + tb * s.uy + EyB;
    uxb += tb * Fx + uEb * ECx;
    uyb += tb * Fy + uEb * ECy;
    if (CELL) {   // the share of u's adjoint that is left out, b rho sum xi z, through u = (3 m + dt/2 F) / rho
        const T lx = b * fxb, ly = b * fyb, hdt = T(0.5) * Pr.dt;
        Fxb += hdt * lx;
        Fyb += hdt * ly;
        rhob -= s.ux * lx + s.uy * ly;
    }
    T gfxb = C.cd * ExB, gfyb = C.cd * EyB;
    // weights: a, b, c over 6K + k X; b-bar and a-bar nearly cancel (f is near
    // equilibrium), so their difference is formed first
    const T Xb = r * r * (C.k6 * (C.nb * bb - (CELL ? T(3) : T(1)) * fsum) - kx * C.nc * cb);
    rhob += D * Xb;
    phib += (Pr.hmuB - Pr.hmuA) * rho * Xb;
    if (!CELL) {
        // p = sum f + kp1 u.grad phi - kp2 rho lap mu, u = (m + kf F) 3 / rho
        uxb += C.kp1 * pb * s.gfx;
        uyb += C.kp1 * pb * s.gfy;
        gfxb += C.kp1 * pb * s.ux;
        gfyb += C.kp1 * pb * s.uy;
        rhob -= C.kp2 * s.lmu * pb;
        lmub -= C.kp2 * rho * pb;
        lam -= C.dkp2 * rl * pb;
        if (wall) uxb = uyb = T(0);
        rhob -= (s.ux * uxb + s.uy * uyb) * irho;
        uxb *= T(3) * irho;   // the adjoint of the momentum sum
        uyb *= T(3) * irho;
        Fxb += C.kf * uxb;
        Fyb += C.kf * uyb;
    }
    // F = -phi grad mu + (rho - rho_ref) g, rho(phi)
    phib -= s.gmx * Fxb + s.gmy * Fyb;
    rhob += Pr.gxa * Fxb + Pr.gya * Fyb;
    B.phi = phib + Pr.drho * rhob;
    B.gmx = -s.phi * Fxb;
    B.gmy = -s.phi * Fyb;
    B.gfx = gfxb;
    B.gfy = gfyb;
    B.mu = mub;
    B.lmu = lmub;
    B.ux = uxb;
    B.uy = uyb;
    B.p = pb;
    return CELL ? T(36) * b : a;
}

// v minus its part in the sums of f and of xi f: v_q - sum w v - 3 xi_q . sum w xi v,
// from differences of v alone, so that a v which is such a part gives zero.
template <typename T>
__device__ __forceinline__ void nonconserved(const T (&v)[Q], T (&r)[Q])
{
    const T d1 = v[1] - v[3], d2 = v[2] - v[4], d5 = v[5] - v[7], d6 = v[6] - v[8];
    const T e1 = (v[1] - v[0]) + (v[3] - v[0]), e2 = (v[2] - v[0]) + (v[4] - v[0]);
    const T e5 = (v[5] - v[0]) + (v[7] - v[0]), e6 = (v[6] - v[0]) + (v[8] - v[0]);
    const T m = (T(4) * (e1 + e2) + (e5 + e6)) * T(1.0 / 36.0);   // sum w v - v_0
    const T o1 = (T(2) * d1 - (d5 - d6)) * T(1.0 / 12.0), o2 = (T(2) * d2 - (d5 + d6)) * T(1.0 / 12.0);
    const T o5 = (d5 - (d1 + d2)) * T(1.0 / 3.0), o6 = (d6 - (d2 - d1)) * T(1.0 / 3.0);
    r[0] = -m;
    r[1] = (T(0.5) * e1 - m) + o1;
    r[3] = (T(0.5) * e1 - m) - o1;
    r[2] = (T(0.5) * e2 - m) + o2;
    r[4] = (T(0.5) * e2 - m) - o2;
    r[5] = (T(0.5) * e5 - m) + o5;
    r[7] = (T(0.5) * e5 - m) - o5;
    r[6] = (T(0.5) * e6 - m) + o6;
    r[8] = (T(0.5) * e6 - m) - o6;
}

template <typename T>
__device__ __forceinline__ const AxisRecT<T> &rec(const InstDev &I, const AxisRecT<T> *__restrict__ geo, int axis, int k)
{
    return geo[(axis == 0 ? I.gx_off : I.gy_off) + k];
}

// Index of the face at a low wall of axis A, at position t of the other axis.
__device__ __forceinline__ long long low_face(const InstDev &I, long long N, int A, int t)
{
    return N + (A == 0 ? I.gy_off : I.gx_off) + t;
}

// The high face on axis A of the cell at position n of that axis and t of the
// other, or the face at the low wall for n = -1.
template <typename T, int A>
__device__ __forceinline__ void face_of(const InstDev &I, const AxisRecT<T> *__restrict__ geo, const Planes<T> &P, const AdjPlanes<T> &Ad,
                                        int n, int t, T &lam)
{
    const ParT<T> &Pr = par<T>(I);
    const long long N = P.N;
    auto cell = [&](int nn, int tt) -> long long { return A == 0 ? cell_of(I, nn, tt) : cell_of(I, tt, nn); };
    const AxisRecT<T> &rt = rec<T>(I, geo, 1 - A, t);
    const T em = rt.e1m, e0 = rt.e10, ep = rt.e1p, h = Pr.h;
    const int nc = n < 0 ? 0 : n;
    const AxisRecT<T> &rn = rec<T>(I, geo, A, nc);
    const int side = n < 0 ? -1 : rn.hi_wall ? 1 : 0;
    const long long cL = cell(nc, t), cLm = cell(nc, rt.km), cLp = cell(nc, rt.kp);
    T fb[Q], gb[Q], ob[Q], yb[Q];
    APt<T> s, B;
    T fsum = 0;
#pragma unroll
    for (int q = 0; q < Q; q++) ob[q] = yb[q] = T(0);
    if (side == 0) {
        const int nR = rn.kp;
        const long long cR = cell(nR, t), cRm = cell(nR, rt.km), cRp = cell(nR, rt.kp);
        const T wL = rn.wL, wR = rn.wR, k = h * rn.invd;
        const T Lm = h * wL * em, Lp = h * wL * ep, L0 = h * wL * e0, Rm = h * wR * em, Rp = h * wR * ep, R0 = h * wR * e0;
        const T kL = Pr.dt * recip(rn.d), kR = Pr.dt * recip(rec<T>(I, geo, A, nR).d);
#pragma unroll
        for (int q = 0; q < Q; q++) {
            const int nq = ca(q, A), tq = ca(q, 1 - A);
            const T cl = wL + T(nq) * k - T(tq) * L0, cr = wR - T(nq) * k - T(tq) * R0;
            const T *Pf = P.fbp + q * N, *Pg = P.gbp + q * N;
            T vf = cl * Pf[cL] + cr * Pf[cR], vg = cl * Pg[cL] + cr * Pg[cR];
            if (tq) {
                const T sg = T(-tq);
                vf += sg * (Lm * Pf[cLm] + Lp * Pf[cLp] + Rm * Pf[cRm] + Rp * Pf[cRp]);
                vg += sg * (Lm * Pg[cLm] + Lp * Pg[cLp] + Rm * Pg[cRm] + Rp * Pg[cRp]);
            }
            fb[q] = vf;
            gb[q] = vg;
            if (nq) {   // the flux enters J_L with + and J_R with -; J-bar = -dt/|V| x-bar
                ob[q] = T(nq) * (kR * Ad.xf[q * N + cR] - kL * Ad.xf[q * N + cL]);
                yb[q] = T(nq) * (kR * Ad.xg[q * N + cR] - kL * Ad.xg[q * N + cL]);
                fsum += vf * ob[q];
            }
        }
        s.mu = wL * P.mu[cL] + wR * P.mu[cR];
        s.lmu = wL * P.lapmu[cL] + wR * P.lapmu[cR];
        s.gmx = wL * P.gmux[cL] + wR * P.gmux[cR];
        s.gmy = wL * P.gmuy[cL] + wR * P.gmuy[cR];
        s.gfx = wL * P.gphix[cL] + wR * P.gphix[cR];
        s.gfy = wL * P.gphiy[cL] + wR * P.gphiy[cR];
        s.gpx = wL * P.gpx[cL] + wR * P.gpx[cR];
        s.gpy = wL * P.gpy[cL] + wR * P.gpy[cR];
    } else {
        // wall face: Taylor reconstruction of the outgoing and parallel directions,
        // bounce-back of the incoming ones
        const long long cnm = cell(rn.km, t), cnp = cell(rn.kp, t);
        const T half = T(0.5) * rn.d, kc = Pr.dt * recip(rn.d);
#pragma unroll
        for (int q = 0; q < Q; q++) {
            if (ca(q, A) * side < 0) continue;
            const T off = T(side) * half - h * T(ca(q, A)), ht = h * T(ca(q, 1 - A));
            const T *Pf = P.fbp + q * N, *Pg = P.gbp + q * N;
            const T bf = Pf[cL], bg = Pg[cL];
            fb[q] = bf + off * (rn.e1m * Pf[cnm] + rn.e10 * bf + rn.e1p * Pf[cnp]) - ht * (em * Pf[cLm] + e0 * bf + ep * Pf[cLp]);
            gb[q] = bg + off * (rn.e1m * Pg[cnm] + rn.e10 * bg + rn.e1p * Pg[cnp]) - ht * (em * Pg[cLm] + e0 * bg + ep * Pg[cLp]);
            if (ca(q, A) * side > 0) {   // carries its own flux and its opposite's
                const int o = opp(q);
                ob[q] = kc * (Ad.xf[o * N + cL] - Ad.xf[q * N + cL]);
                yb[q] = kc * (Ad.xg[o * N + cL] - Ad.xg[q * N + cL]);
                fsum += fb[q] * ob[q];
            }
        }
#pragma unroll
        for (int q = 0; q < Q; q++) {
            if (ca(q, A) * side < 0) {
                fb[q] = fb[opp(q)];
                gb[q] = gb[opp(q)];
            }
        }
        s.mu = P.mu[cL];
        s.lmu = P.lapmu[cL];
        s.gmx = A == 0 ? T(0) : P.gmux[cL];
        s.gmy = A == 1 ? T(0) : P.gmuy[cL];
        s.gfx = A == 0 ? T(0) : P.gphix[cL];
        s.gfy = A == 1 ? T(0) : P.gphiy[cL];
        s.gpx = A == 0 ? T(0) : P.gpx[cL];
        s.gpy = A == 1 ? T(0) : P.gpy[cL];
    }
    // face macros (Eq. conservedVariable with h)
    const PtC<T> &C = facec<T>(I);
    T sf = 0, mx = 0, my = 0;
    s.phi = 0;
#pragma unroll
    for (int q = 0; q < Q; q++) {
        s.phi += gb[q];
        sf += fb[q];
        if (cx(q)) mx += T(cx(q)) * fb[q];
        if (cy(q)) my += T(cy(q)) * fb[q];
    }
    const T rho = Pr.rhoB + Pr.drho * (s.phi - Pr.phiB), r3 = T(3) * recip(rho);
    s.ux = (mx + C.kf * (-s.phi * s.gmx + (rho - Pr.rho_ref) * Pr.gxa)) * r3;
    s.uy = (my + C.kf * (-s.phi * s.gmy + (rho - Pr.rho_ref) * Pr.gya)) * r3;
    if (side != 0) s.ux = s.uy = T(0);
    s.p = sf + C.kp1 * (s.ux * s.gfx + s.uy * s.gfy) - C.kp2 * rho * s.lmu;
    const T a = point_adj<T, A>(I, s, ob, yb, fsum, side != 0, B, lam);
    // gifts: bar f_q gets a ob_q + p-bar + xi_q . m-bar, bar g_q gets ga yb_q + phi-bar;
    // a wall's incoming bars are copies of the outgoing ones
    T *F = Ad.face[A];
    const long long NF = Ad.NF, at = n < 0 ? low_face(I, N, A, t) : cL;
    const T two = side != 0 ? T(2) : T(1);
#pragma unroll
    for (int k = 0; k < 6; k++) {
        const int q = fset<A>(k);
        const bool in = ca(q, A) * side < 0;
        const T m = T(cx(q)) * B.ux + T(cy(q)) * B.uy;
        F[(AF + k) * NF + at] = in ? T(0) : a * ob[q] + two * B.p + m;
        F[(AG + k) * NF + at] = in ? T(0) : C.ga * yb[q] + two * B.phi;
    }
    F[AS * NF + at] = B.p;
    F[AM * NF + at] = A == 0 ? B.uy : B.ux;
    F[AP * NF + at] = B.phi;
    const bool wx = side != 0 && A == 0, wy = side != 0 && A == 1;   // aux normal to a wall: not the cell's
    const T v[8] = {B.mu, B.lmu, wx ? T(0) : B.gmx, wy ? T(0) : B.gmy, wx ? T(0) : B.gfx, wy ? T(0) : B.gfy,
                    wx ? T(0) : B.gpx, wy ? T(0) : B.gpy};
#pragma unroll
    for (int k = 0; k < 8; k++) F[(AX + k) * NF + at] = v[k];
}

template <typename T>
__global__ void __launch_bounds__(128, sizeof(T) == 4 ? 4 : 2) ka_face(const InstDev *__restrict__ insts, const AdjSeg *__restrict__ segs, int n_seg,
                                               const AxisRecT<T> *__restrict__ geo, Planes<T> P, AdjPlanes<T> Ad)
{
    const int sg = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (sg >= n_seg) return;
    const AdjSeg g = segs[sg];
    const InstDev &I = insts[g.inst];
    const int i = g.i + (threadIdx.x & 31);
    T lam = 0;
    if (i < I.nx) {
        if (g.axis == 0) face_of<T, 0>(I, geo, P, Ad, i, g.j, lam);
        else face_of<T, 1>(I, geo, P, Ad, g.j, i, lam);
    }
    slot_add(Ad.lam_face + sg, lam);
}

// What the faces of axis A give the bar values p of one kind (0 f, 1 g) and four of
// the aux fields (0: mu, lap mu, grad mu; 1: grad phi, grad p) of a cell at position
// n of that axis and t of the other: the transpose of the reconstruction.  With T = (interpolation weight) E + (weight) W of the cell's
// high and low face values, an interior cell gets T + h xi_n (E - W) / distance
// - h xi_t (e0 T + e1m T of the next row + e1p T of the row before).
template <typename T, int A, int KIND>
__device__ __forceinline__ void gather(const InstDev &I, const AxisRecT<T> *__restrict__ geo, const AdjPlanes<T> &Ad, int n, int t,
                                       T (&p)[Q], T (&x)[4])
{
    const long long N = Ad.N, NF = Ad.NF;
    const T h = par<T>(I).h;
    const T *F = Ad.face[A];
    auto cell = [&](int nn, int tt) -> long long { return A == 0 ? cell_of(I, nn, tt) : cell_of(I, tt, nn); };
    const AxisRecT<T> &rn = rec<T>(I, geo, A, n), &rt = rec<T>(I, geo, 1 - A, t);
    const int km = rn.km, kp = rn.kp;
    const bool lo = rn.lo_wall, hi = rn.hi_wall;
    const AxisRecT<T> &rm = rec<T>(I, geo, A, km), &rp = rec<T>(I, geo, A, kp);
    // weights of the high (E) and low (W) face; a wall's face is the cell's alone
    const T aE = hi ? T(1) : rn.wL, aW = lo ? T(1) : rm.wR;
    const T kE = hi ? T(0) : h * rn.invd, kW = lo ? T(0) : h * rm.invd;
    const long long E0 = cell(n, t), W0 = lo ? low_face(I, N, A, t) : cell(km, t);
    // the rows whose tangential derivative reads this cell
    const bool hm = rt.km != t, hp = rt.kp != t;
    const long long Em = cell(n, rt.km), Ep = cell(n, rt.kp);
    const long long Wm = lo ? low_face(I, N, A, rt.km) : cell(km, rt.km), Wp = lo ? low_face(I, N, A, rt.kp) : cell(km, rt.kp);
    const T e0 = h * (rt.e10 + (hm ? T(0) : rt.e1m) + (hp ? T(0) : rt.e1p));
    const T em = hp ? h * rec<T>(I, geo, 1 - A, rt.kp).e1m : T(0);   // the next row's low neighbour
    const T ep = hm ? h * rec<T>(I, geo, 1 - A, rt.km).e1p : T(0);   // the row before's high neighbour
    auto at = [&](int pl, long long e, long long w) -> T { return aE * F[pl * NF + e] + aW * F[pl * NF + w]; };
    auto tang = [&](int pl, T c0) -> T { return e0 * c0 + em * at(pl, Ep, Wp) + ep * at(pl, Em, Wm); };
    // wall terms of direction q: the normal derivative of the wall's cell reads it
    // and its inner neighbour
    const bool nearw = lo || hi || rm.lo_wall || rp.hi_wall;
    auto normal = [&](int pl, int xn) -> T {
        T v = T(xn) * (kE * F[pl * NF + E0] - kW * F[pl * NF + W0]);
        if (nearw) {
            if (hi) v += (T(0.5) * rn.d - h * T(xn)) * rn.e10 * F[pl * NF + E0];
            else if (rp.hi_wall) v += (T(0.5) * rp.d - h * T(xn)) * rp.e1m * F[pl * NF + cell(kp, t)];
            if (lo) v += (T(-0.5) * rn.d - h * T(xn)) * rn.e10 * F[pl * NF + W0];
            else if (rm.lo_wall) v += (T(-0.5) * rm.d - h * T(xn)) * rm.e1p * F[pl * NF + low_face(I, N, A, t)];
        }
        return v;
    };
    constexpr int F0 = KIND == 0 ? AF : AG;
#pragma unroll
    for (int k = 0; k < 6; k++) {
        const int q = fset<A>(k), xn = ca(q, A), xt = ca(q, 1 - A);
        const T c = at(F0 + k, E0, W0);
        p[q] = c + normal(F0 + k, xn);
        if (xt) p[q] -= T(xt) * tang(F0 + k, c);
    }
    constexpr int tp = A == 0 ? 2 : 1, tn = A == 0 ? 4 : 3;   // along the face
    if (KIND == 0) {
        const T cS = at(AS, E0, W0), cM = at(AM, E0, W0);
        const T nS = cS + normal(AS, 0), nM = cM + normal(AM, 0), yS = tang(AS, cS), yM = tang(AM, cM);
        p[0] = nS;
        p[tp] = (nS + nM) - (yS + yM);
        p[tn] = (nS - nM) + (yS - yM);
    } else {
        const T cP = at(AP, E0, W0), nP = cP + normal(AP, 0), yP = tang(AP, cP);
        p[0] = nP;
        p[tp] = nP - yP;
        p[tn] = nP + yP;
    }
#pragma unroll
    for (int k = 0; k < 4; k++) x[k] = at(AX + 4 * KIND + k, E0, W0);
}

// bar-plus at the cell centre (Eq. relations1) after its faces, and the update
// x_new = 4/3 bar-plus - 1/3 x - dt/|V| J (Eqs. relations2, updatef).  A warp per
// run of 32 cells, or (SPLIT) a block: its four warps gather the two kinds from the
// two axes, then one of them (another one in the next block, so that the FP64 work of
// an SM's blocks spreads over its sub-partitions) transposes the point.  The split
// shortens the longest path (FP64 48x96: 43 -> 31 us), and leaves three of four warps
// without work at the end (FP32 256x512: 34 -> 54 us): it is for meshes of few runs.
template <typename T, bool SPLIT>
__global__ void __launch_bounds__(128, sizeof(T) == 4 && !SPLIT ? 4 : 2) ka_cell(const InstDev *__restrict__ insts,
                                                                                 const AdjSeg *__restrict__ segs, int n_seg,
                                                                                 const AxisRecT<T> *__restrict__ geo,
                                                                                 Planes<T> P, AdjPlanes<T> Ad)
{
    __shared__ T Gs[SPLIT ? 2 : 1][2][Q][32], Xs[SPLIT ? 2 : 1][8][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int sg = SPLIT ? blockIdx.x : blockIdx.x * (blockDim.x >> 5) + warp;
    if (sg >= n_seg) return;
    const AdjSeg g = segs[sg];
    const InstDev &I = insts[g.inst];
    const int i = g.i + lane, j = g.j;
    const bool own = i < I.nx;
    T Gf[Q], Gg[Q], X[8];
    if (own) {
        T v[Q], x[4];
        if constexpr (SPLIT) {
            if (warp == 0) gather<T, 0, 0>(I, geo, Ad, i, j, v, x);
            else if (warp == 1) gather<T, 0, 1>(I, geo, Ad, i, j, v, x);
            else if (warp == 2) gather<T, 1, 0>(I, geo, Ad, j, i, v, x);
            else gather<T, 1, 1>(I, geo, Ad, j, i, v, x);
#pragma unroll
            for (int q = 0; q < Q; q++) Gs[warp >> 1][warp & 1][q][lane] = v[q];
#pragma unroll
            for (int k = 0; k < 4; k++) Xs[warp >> 1][4 * (warp & 1) + k][lane] = x[k];
        } else {
            gather<T, 0, 0>(I, geo, Ad, i, j, Gf, x);
            T y[4];
            gather<T, 1, 0>(I, geo, Ad, j, i, v, y);
#pragma unroll
            for (int q = 0; q < Q; q++) Gf[q] += v[q];
#pragma unroll
            for (int k = 0; k < 4; k++) X[k] = x[k] + y[k];
            gather<T, 0, 1>(I, geo, Ad, i, j, Gg, x);
            gather<T, 1, 1>(I, geo, Ad, j, i, v, y);
#pragma unroll
            for (int q = 0; q < Q; q++) Gg[q] += v[q];
#pragma unroll
            for (int k = 0; k < 4; k++) X[4 + k] = x[k] + y[k];
        }
    }
    if constexpr (SPLIT) {
        __syncthreads();
        if (warp != (int)(blockIdx.x & 3)) return;
        if (own) {
#pragma unroll
            for (int q = 0; q < Q; q++) {
                Gf[q] = Gs[0][0][q][lane] + Gs[1][0][q][lane];
                Gg[q] = Gs[0][1][q][lane] + Gs[1][1][q][lane];
            }
#pragma unroll
            for (int k = 0; k < 8; k++) X[k] = Xs[0][k][lane] + Xs[1][k][lane];
        }
    }
    T lam = 0;
    if (own) {
        const long long c = cell_of(I, i, j), N = P.N;
        APt<T> s, B;
        s.phi = T(phi_val(P.phi[c]));
        s.ux = P.ux[c];
        s.uy = P.uy[c];
        s.p = P.p[c];
        s.mu = P.mu[c];
        s.lmu = P.lapmu[c];
        s.gmx = P.gmux[c];
        s.gmy = P.gmuy[c];
        s.gfx = P.gphix[c];
        s.gfy = P.gphiy[c];
        s.gpx = P.gpx[c];
        s.gpy = P.gpy[c];
        T pf[Q], pg[Q], xf[Q], xg[Q];
        T fsum = 0;
#pragma unroll
        for (int q = 0; q < Q; q++) {
            xf[q] = Ad.xf[q * N + c];
            xg[q] = Ad.xg[q * N + c];
            pf[q] = T(4.0 / 3.0) * xf[q] + Gf[q];
            pg[q] = T(4.0 / 3.0) * xg[q] + Gg[q];
            fsum += P.f[q * N + c] * pf[q];
        }
        const T b = point_adj<T, -1>(I, s, pf, pg, fsum, false, B, lam);
        // a p - x / 3 with p = 4/3 x + G and a = 1 - b: as an increment of x, so that
        // a uniform adjoint passes the step unchanged (4/3, 1/3 and a rounded one by
        // one would leave a bias that grows with the steps).  Of f, the
        // relaxation -b p and what the equilibrium's p and u give back of it, b times
        // p's part in the sums of f and of xi f, are formed as one here (the latter is
        // not added in ka_tail): they cancel on an adjoint that is such a part, and
        // rounded one by one they left an eigenvalue of 1 + 1e-8, an error of 2.5e-5 in
        // dL/dkappa after 2000 FP32 steps of Rayleigh-Taylor 256x512 (5e-7 as one; 133
        // us per step of a gradient either way, FP64 256x512 1.25 and 1.27 ms).
        const T bg = cellc<T>(I).gb36;
        T r[Q];
        nonconserved(pf, r);
#pragma unroll
        for (int q = 0; q < Q; q++) {
            Ad.af[q * N + c] = xf[q] + (Gf[q] - b * r[q]);
            Ad.ag[q * N + c] = xg[q] + (Gg[q] - bg * pg[q]);
        }
        T *const out[8] = {Ad.mu, Ad.lapmu, Ad.gmx, Ad.gmy, Ad.gfx, Ad.gfy, Ad.gpx, Ad.gpy};
        const T v[8] = {B.mu, B.lmu, B.gmx, B.gmy, B.gfx, B.gfy, B.gpx, B.gpy};
#pragma unroll
        for (int k = 0; k < 8; k++) out[k][c] = X[k] + v[k];
        Ad.phi[c] = B.phi;
        Ad.p[c] = B.p;
        Ad.ux[c] = B.ux;
        Ad.uy[c] = B.uy;
    }
    slot_add(Ad.lam_cell + sg, lam);
}

template <typename T>
struct PtBar {
    T phi, rho, ux, uy, p, mu, lapmu, Fx, Fy, grx, gry, gpx, gpy;
};

template <typename T>
struct InvBar {
    T uu15, prho, emu, srcF, fg, Gx, Gy, cgx, cgy;
};

template <typename T>
__device__ __forceinline__ PtBar<T> ptbar_zero()
{
    PtBar<T> b;
    b.phi = b.rho = b.ux = b.uy = b.p = b.mu = b.lapmu = b.Fx = b.Fy = b.grx = b.gry = b.gpx = b.gpy = T(0);
    return b;
}

template <typename T>
__device__ __forceinline__ InvBar<T> invbar_zero()
{
    InvBar<T> b;
    b.uu15 = b.prho = b.emu = b.srcF = b.fg = b.Gx = b.Gy = b.cgx = b.cgy = T(0);
    return b;
}

// transpose of eq_src: adjoints of (feq, geq, Ff, Fg) of direction q into s, v
template <typename T>
__device__ __forceinline__ void eq_src_adj(const Pt<T> &s, const PtInv<T> &v, int q, T feqb, T geqb, T Ffb, T Fgb,
                                           PtBar<T> &sb, InvBar<T> &vb)
{
    const T w = T(wq(q));
    const T xu = T(cx(q)) * s.ux + T(cy(q)) * s.uy;
    const T si = w * (T(3) * xu + T(4.5) * xu * xu - v.uu15);
    const T G = w + si;
    const T ex = T(cx(q)) - s.ux, ey = T(cy(q)) - s.uy;
    const T A = s.Fx * G + si * v.cgx, B = s.Fy * G + si * v.cgy;
    const T C = ex * v.Gx + ey * v.Gy;
    T sib = 0, Gb = 0;
    // feq = w p + prho si
    sb.p += w * feqb;
    vb.prho += si * feqb;
    sib += v.prho * feqb;
    // geq = H + phi si, H_0 = phi - (1 - w) emu, H_q = w emu
    sb.phi += si * geqb;
    sib += s.phi * geqb;
    if (q == 0) {
        sb.phi += geqb;
        vb.emu -= (T(1) - w) * geqb;
    } else {
        vb.emu += w * geqb;
    }
    // Ff = ex A + ey B - w srcF
    const T Ab = ex * Ffb, Bb = ey * Ffb;
    T exb = A * Ffb, eyb = B * Ffb;
    vb.srcF -= w * Ffb;
    sb.Fx += G * Ab;
    sb.Fy += G * Bb;
    Gb += s.Fx * Ab + s.Fy * Bb;
    sib += v.cgx * Ab + v.cgy * Bb;
    vb.cgx += si * Ab;
    vb.cgy += si * Bb;
    // Fg = fg C G
    vb.fg += C * G * Fgb;
    const T Cb = v.fg * G * Fgb;
    Gb += v.fg * C * Fgb;
    exb += v.Gx * Cb;
    eyb += v.Gy * Cb;
    vb.Gx += ex * Cb;
    vb.Gy += ey * Cb;
    sb.ux -= exb;
    sb.uy -= eyb;
    // G = w + si, si = w (3 xu + 4.5 xu^2 - uu15)
    sib += Gb;
    const T xub = w * (T(3) + T(9) * xu) * sib;
    vb.uu15 -= w * sib;
    sb.ux += T(cx(q)) * xub;
    sb.uy += T(cy(q)) * xub;
}

// transpose of pt_inv; lamb collects d/dlambda (eta = 3 lambda / tau_g, srcF)
template <typename T>
__device__ __forceinline__ void pt_inv_adj(const ParT<T> &Pr, const Pt<T> &s, const PtInv<T> &v, const InvBar<T> &vb,
                                           PtBar<T> &sb, T &lamb)
{
    const T cs2 = Cst<T>::cs2;
    sb.ux += T(3) * s.ux * vb.uu15;
    sb.uy += T(3) * s.uy * vb.uu15;
    sb.rho += cs2 * vb.prho;
    sb.mu += Pr.eta * vb.emu;
    lamb += T(3) / Pr.tau_g * s.mu * vb.emu;
    sb.rho += cs2 * Pr.gamma * Pr.lambda * s.lapmu * vb.srcF;
    sb.lapmu += cs2 * s.rho * Pr.gamma * Pr.lambda * vb.srcF;
    lamb += cs2 * s.rho * Pr.gamma * s.lapmu * vb.srcF;
    sb.phi += T(3) / s.rho * vb.fg;
    sb.rho -= v.fg / s.rho * vb.fg;
    sb.Fx += vb.Gx;
    sb.Fy += vb.Gy;
    sb.gpx -= vb.Gx;
    sb.gpy -= vb.Gy;
    sb.grx += cs2 * vb.cgx;
    sb.gry += cs2 * vb.cgy;
}

// transpose of F = -phi grad mu + (rho - rho_ref) g and grad rho = drho grad phi
template <typename T>
__device__ __forceinline__ void force_adj(const ParT<T> &Pr, T phi, T gmx, T gmy, PtBar<T> &sb, T &gmxb, T &gmyb,
                                          T &gfxb, T &gfyb)
{
    sb.phi += -gmx * sb.Fx - gmy * sb.Fy;
    gmxb += -phi * sb.Fx;
    gmyb += -phi * sb.Fy;
    sb.rho += Pr.gxa * sb.Fx + Pr.gya * sb.Fy;
    gfxb += Pr.drho * sb.grx;
    gfyb += Pr.drho * sb.gry;
}

// Transpose of a three-point stencil along axis a: the sum over the cells whose
// stencil reads cell (i, j), of their coefficient times the adjoint there.
// KIND 0: first derivative (c1m, c10, c1p); 1: first derivative in difference
// form (centre weight -(c1m + c1p)); 2: second derivative (c2m, c20, c2p);
// 3: second derivative in difference form.
template <typename T, int KIND>
__device__ __forceinline__ T coef(const AxisRecT<T> &r, int which)
{
    const T m = (KIND < 2) ? r.c1m : r.c2m, p = (KIND < 2) ? r.c1p : r.c2p;
    const T z = (KIND == 0) ? r.c10 : (KIND == 2) ? r.c20 : -(m + p);
    return which < 0 ? m : which > 0 ? p : z;
}

template <typename T, int KIND>
__device__ __forceinline__ T stencil_t(const InstDev &I, const AxisRecT<T> *__restrict__ geo, const T *__restrict__ Ab,
                                       int a, int i, int j)
{
    const long long off = a == 0 ? I.gx_off : I.gy_off;
    const int k = a == 0 ? i : j;
    const AxisRecT<T> &r = geo[off + k];
    auto at = [&](int kk) -> T { return Ab[a == 0 ? cell_of(I, kk, j) : cell_of(I, i, kk)]; };
    T s = coef<T, KIND>(r, 0) * at(k);
    if (r.km == k) s += coef<T, KIND>(r, -1) * at(k);
    else s += coef<T, KIND>(geo[off + r.km], +1) * at(r.km);
    if (r.kp == k) s += coef<T, KIND>(r, +1) * at(k);
    else s += coef<T, KIND>(geo[off + r.kp], -1) * at(r.kp);
    return s;
}

// Coefficients of the stencil transposes (see stencil_t) at one position of an axis:
// of the adjoint at the position before, after, and at the position itself, for the
// first and the second derivative; z*: the position itself, the difference forms.
template <typename T>
struct TCoef {
    T m1, p1, c1, z1, m2, p2, c2, z2;
};

// The rest of the step's transpose for a BX x BY tile per thread block, each on the
// ring that the next one reads: grad p, then p, u, F (Eqs. u, P) on a 2-cell ring;
// grad mu and lap mu, then mu = psi'(phi) - kappa lap(phi) (Eq. chemicalpotential) on
// a 1-cell ring; grad phi and lap phi, then phi = sum g~ on the tile.  The stencils'
// coefficients and the adjoint of grad p are staged first, so that a phase has one
// load latency and not a chain through the geometry records.
template <typename T, int BX, int BY, int NT>
__global__ void __launch_bounds__(NT) ka_tail(const InstDev *__restrict__ insts, const int4 *__restrict__ tiles,
                                              const AxisRecT<T> *__restrict__ geo, Planes<T> P, AdjPlanes<T> Ad)
{
    constexpr int W2 = BX + 4, H2 = BY + 4, A2 = W2 * H2, W1 = BX + 2, A1 = W1 * (BY + 2);
    constexpr int WX = BX + 6, AX_ = WX * H2, AY_ = W2 * (BY + 6);
    __shared__ T gmx[A2], gmy[A2], lmu[A2], gfx[A2], gfy[A2], lph[A1], phb[BX * BY], sgx[AX_], sgy[AY_];
    __shared__ TCoef<T> tc[W2 + H2];
    __shared__ int gi[W2 + H2];   // global index of positions -2 .. (-1 outside), columns then rows
    const int4 t = tiles[blockIdx.x];
    const InstDev &I = insts[t.x];
    const ParT<T> &Pr = par<T>(I);
    const int i0 = t.y, j0 = t.z, tid = threadIdx.x;
    const long long N = P.N;
    auto wrap = [](int g, int n, int bc) -> int {
        if (bc == 0) {
            while (g < 0) g += n;
            while (g >= n) g -= n;
            return g;
        }
        return g < 0 || g >= n ? -1 : g;
    };
    for (int r = tid; r < AX_ + AY_; r += NT) {
        const bool isx = r < AX_;
        const int k = isx ? r : r - AX_, w = isx ? WX : W2;
        const int i = wrap(i0 + k % w - (isx ? 3 : 2), I.nx, I.bcx), j = wrap(j0 + k / w - (isx ? 2 : 3), I.ny, I.bcy);
        const T v = i >= 0 && j >= 0 ? (isx ? Ad.gpx : Ad.gpy)[cell_of(I, i, j)] : T(0);
        (isx ? sgx : sgy)[k] = v;
    }
    for (int r = tid; r < W2 + H2; r += NT) {
        const bool isx = r < W2;
        const int g = isx ? wrap(i0 + r - 2, I.nx, I.bcx) : wrap(j0 + r - W2 - 2, I.ny, I.bcy);
        gi[r] = g;
        if (g < 0) continue;
        const AxisRecT<T> &c = rec<T>(I, geo, isx ? 0 : 1, g), &m = rec<T>(I, geo, isx ? 0 : 1, c.km), &p = rec<T>(I, geo, isx ? 0 : 1, c.kp);
        const bool hm = !c.lo_wall, hp = !c.hi_wall;   // a wall's ghost is the cell itself
        TCoef<T> k;
        const T s1 = (hm ? T(0) : c.c1m) + (hp ? T(0) : c.c1p), s2 = (hm ? T(0) : c.c2m) + (hp ? T(0) : c.c2p);
        k.m1 = hm ? m.c1p : T(0);
        k.p1 = hp ? p.c1m : T(0);
        k.c1 = c.c10 + s1;
        k.z1 = s1 - (c.c1m + c.c1p);
        k.m2 = hm ? m.c2p : T(0);
        k.p2 = hp ? p.c2m : T(0);
        k.c2 = c.c20 + s2;
        k.z2 = s2 - (c.c2m + c.c2p);
        tc[r] = k;
    }
    __syncthreads();
    const T cs2 = Cst<T>::cs2, hdt = T(0.5) * Pr.dt;
    T lamb = 0, kapb = 0;
    for (int r = tid; r < A2; r += NT) {
        const int x = r % W2 - 2, y = r / W2 - 2;
        const int i = gi[x + 2], j = gi[W2 + y + 2];
        if (i < 0 || j < 0) {   // its neighbours read it with a zero coefficient
            gmx[r] = gmy[r] = lmu[r] = gfx[r] = gfy[r] = T(0);
            continue;
        }
        const bool own = x >= 0 && x < BX && y >= 0 && y < BY && i0 + x < I.nx && j0 + y < I.ny;
        const long long c = cell_of(I, i, j);
        const TCoef<T> &kx = tc[x + 2], &ky = tc[W2 + y + 2];
        const T *sx = sgx + (y + 2) * WX + x + 3, *sy = sgy + (y + 3) * W2 + x + 2;
        // of sum f: the share that comes from bar-plus is in ka_cell's af already
        const T pg = (kx.c1 * sx[0] + kx.m1 * sx[-1] + kx.p1 * sx[1]) + (ky.c1 * sy[0] + ky.m1 * sy[-W2] + ky.p1 * sy[W2]);
        const T pb = Ad.p[c] + pg;
        T uxb = Ad.ux[c], uyb = Ad.uy[c];
        const T phi = T(phi_val(P.phi[c]));
        const T rho = Pr.rhoB + Pr.drho * (phi - Pr.phiB);
        const T ux = P.ux[c], uy = P.uy[c];
        const T grx = Pr.drho * P.gphix[c], gry = Pr.drho * P.gphiy[c];
        const T lm = P.lapmu[c];
        const T pk = hdt * cs2 * pb;
        // p = sum f + dt/2 c_s^2 (u . grad rho - gamma rho lambda lap mu)
        uxb += pk * grx;
        uyb += pk * gry;
        PtBar<T> sb = ptbar_zero<T>();
        sb.grx = pk * ux;
        sb.gry = pk * uy;
        sb.rho = -pk * Pr.gamma * Pr.lambda * lm;
        // u = (3 m + dt/2 F) / rho
        const T irho = recip(rho);
        const T mxb = T(3) * uxb * irho, myb = T(3) * uyb * irho;
        sb.Fx = hdt * uxb * irho;
        sb.Fy = hdt * uyb * irho;
        sb.rho -= (ux * uxb + uy * uyb) * irho;
        T gmxb = 0, gmyb = 0, gfxb = 0, gfyb = 0;
        force_adj<T>(Pr, phi, P.gmux[c], P.gmuy[c], sb, gmxb, gmyb, gfxb, gfyb);
        gmx[r] = Ad.gmx[c] + gmxb;
        gmy[r] = Ad.gmy[c] + gmyb;
        lmu[r] = Ad.lapmu[c] - pk * Pr.gamma * rho * Pr.lambda;
        gfx[r] = Ad.gfx[c] + gfxb;
        gfy[r] = Ad.gfy[c] + gfyb;
        if (own) {
            lamb -= pk * Pr.gamma * rho * lm;
            phb[y * BX + x] = Ad.phi[c] + (sb.phi + Pr.drho * sb.rho);
#pragma unroll
            for (int q = 0; q < Q; q++) Ad.af[q * N + c] += pg + T(cx(q)) * mxb + T(cy(q)) * myb;
        }
    }
    __syncthreads();
    for (int r = tid; r < A1; r += NT) {
        const int x = r % W1 - 1, y = r / W1 - 1;
        const int i = gi[x + 2], j = gi[W2 + y + 2];
        if (i < 0 || j < 0) {
            lph[r] = T(0);
            continue;
        }
        const bool own = x >= 0 && x < BX && y >= 0 && y < BY && i0 + x < I.nx && j0 + y < I.ny;
        const long long c = cell_of(I, i, j);
        const TCoef<T> &kx = tc[x + 2], &ky = tc[W2 + y + 2];
        const int e = (y + 2) * W2 + x + 2;
        const T mub = Ad.mu[c] + (kx.c1 * gmx[e] + kx.m1 * gmx[e - 1] + kx.p1 * gmx[e + 1])
                    + (ky.c1 * gmy[e] + ky.m1 * gmy[e - W2] + ky.p1 * gmy[e + W2])
                    + (kx.c2 * lmu[e] + kx.m2 * lmu[e - 1] + kx.p2 * lmu[e + 1])
                    + (ky.c2 * lmu[e] + ky.m2 * lmu[e - W2] + ky.p2 * lmu[e + W2]);
        lph[r] = -Pr.kappa * mub;
        if (own) {
            const AxisRecT<T> &ax = rec<T>(I, geo, 0, i), &ay = rec<T>(I, geo, 1, j);
            const phi_t<T> p0 = P.phi[c];
            const T phi = T(phi_val(p0));
            const T a = phi - Pr.phiA, b = phi - Pr.phiB, m = phi - T(0.5) * (Pr.phiA + Pr.phiB);
            const T d2psi = T(4) * Pr.beta * (b * m + a * m + a * b);
            const int im = ax.lo_wall ? i : gi[x + 1], ip = ax.hi_wall ? i : gi[x + 3];
            const int jm = ay.lo_wall ? j : gi[W2 + y + 1], jp = ay.hi_wall ? j : gi[W2 + y + 3];
            const T lap = (ax.c2m * phi_sub(P.phi[cell_of(I, im, j)], p0) + ax.c2p * phi_sub(P.phi[cell_of(I, ip, j)], p0))
                        + (ay.c2m * phi_sub(P.phi[cell_of(I, i, jm)], p0) + ay.c2p * phi_sub(P.phi[cell_of(I, i, jp)], p0));
            phb[y * BX + x] += d2psi * mub;
            kapb -= lap * mub;
        }
    }
    __syncthreads();
    for (int r = tid; r < BX * BY; r += NT) {
        const int x = r % BX, y = r / BX, i = i0 + x, j = j0 + y;
        if (i >= I.nx || j >= I.ny) continue;
        const long long c = cell_of(I, i, j);
        const TCoef<T> &kx = tc[x + 2], &ky = tc[W2 + y + 2];
        const int e2 = (y + 2) * W2 + x + 2, e1 = (y + 1) * W1 + x + 1;
        const T phib = phb[r] + (kx.z1 * gfx[e2] + kx.m1 * gfx[e2 - 1] + kx.p1 * gfx[e2 + 1])
                     + (ky.z1 * gfy[e2] + ky.m1 * gfy[e2 - W2] + ky.p1 * gfy[e2 + W2])
                     + (kx.z2 * lph[e1] + kx.m2 * lph[e1 - 1] + kx.p2 * lph[e1 + 1])
                     + (ky.z2 * lph[e1] + ky.m2 * lph[e1 - W1] + ky.p2 * lph[e1 + W1]);
#pragma unroll
        for (int q = 0; q < Q; q++) Ad.ag[q * N + c] += phib;
    }
    const int w = blockIdx.x * (NT / 32) + tid / 32;
    slot_add(Ad.lam_macro + w, lamb);
    slot_add(Ad.kap + w, kapb);
}

// The initialisation's mu = psi'(phi) - kappa lap(phi) (Eq. chemicalpotential),
// after the transposes of grad mu and lap mu; writes the adjoint of lap(phi)
template <typename T>
__global__ void __launch_bounds__(128) ka_mu(const InstDev *__restrict__ insts, const AdjSeg *__restrict__ segs, int n_seg,
        const AxisRecT<T> *__restrict__ geo, Planes<T> P, AdjPlanes<T> Ad)
{
    const int sg = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (sg >= n_seg) return;
    const AdjSeg g = segs[sg];
    const InstDev &I = insts[g.inst];
    const ParT<T> &Pr = par<T>(I);
    const int i = g.i + (threadIdx.x & 31), j = g.j;
    T kapb = 0;
    if (i < I.nx) {
        const long long c = cell_of(I, i, j);
        const AxisRecT<T> &ax = geo[I.gx_off + i];
        const AxisRecT<T> &ay = geo[I.gy_off + j];
        const T mub = Ad.mu[c] + stencil_t<T, 0>(I, geo, Ad.gmx, 0, i, j) + stencil_t<T, 0>(I, geo, Ad.gmy, 1, i, j)
                    + stencil_t<T, 2>(I, geo, Ad.lapmu, 0, i, j) + stencil_t<T, 2>(I, geo, Ad.lapmu, 1, i, j);
        const phi_t<T> p0 = P.phi[c];
        const T phi = T(phi_val(p0));
        const T a = phi - Pr.phiA, b = phi - Pr.phiB, m = phi - T(0.5) * (Pr.phiA + Pr.phiB);
        const T d2psi = T(4) * Pr.beta * (b * m + a * m + a * b);
        const T lap = (T(ax.c2m) * phi_sub(P.phi[cell_of(I, ax.km, j)], p0) + T(ax.c2p) * phi_sub(P.phi[cell_of(I, ax.kp, j)], p0))
                    + (T(ay.c2m) * phi_sub(P.phi[cell_of(I, i, ay.km)], p0) + T(ay.c2p) * phi_sub(P.phi[cell_of(I, i, ay.kp)], p0));
        Ad.phi[c] += d2psi * mub;
        Ad.lapphi[c] = -Pr.kappa * mub;
        kapb = -lap * mub;
    }
    slot_add(Ad.kap0 + sg, kapb);
}

// The initialisation's phi, after the transposes of grad phi and lap phi: the
// gradient with respect to the input field
template <typename T>
__global__ void __launch_bounds__(128) ka_phi0(const InstDev *__restrict__ insts, const AdjSeg *__restrict__ segs, int n_seg,
                                               const AxisRecT<T> *__restrict__ geo, AdjPlanes<T> Ad, double *phi0_out,
                                               const long long *__restrict__ dense0)
{
    const int sg = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (sg >= n_seg) return;
    const AdjSeg g = segs[sg];
    const InstDev &I = insts[g.inst];
    const int i = g.i + (threadIdx.x & 31), j = g.j;
    if (i >= I.nx) return;
    const long long c = cell_of(I, i, j);
    phi0_out[dense0[g.inst] + (long long)j * I.nx + i] =
        (double)(Ad.phi[c] + stencil_t<T, 1>(I, geo, Ad.gfx, 0, i, j) + stencil_t<T, 1>(I, geo, Ad.gfy, 1, i, j)
                 + stencil_t<T, 3>(I, geo, Ad.lapphi, 0, i, j) + stencil_t<T, 3>(I, geo, Ad.lapphi, 1, i, j));
}

// Step 1 (Eq. auxf a with the original distribution at equilibrium):
// tilde = eq - dt/2 F; the adjoint of the tracked state is in xf, xg.
template <typename T>
__global__ void __launch_bounds__(128) ka_init(const InstDev *__restrict__ insts, const AdjSeg *__restrict__ segs, int n_seg,
                                                  const AxisRecT<T> *__restrict__ geo, Planes<T> P, AdjPlanes<T> Ad)
{
    const int sg = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (sg >= n_seg) return;
    const AdjSeg g = segs[sg];
    const InstDev &I = insts[g.inst];
    const ParT<T> &Pr = par<T>(I);
    const int i = g.i + (threadIdx.x & 31), j = g.j;
    T lamb = 0;
    if (i < I.nx) {
        const AxisRecT<T> &ax = geo[I.gx_off + i];
        const AxisRecT<T> &ay = geo[I.gy_off + j];
        const long long c = cell_of(I, i, j);
        const long long N = P.N;
        Pt<T> s;
        s.phi = T(phi_val(P.phi[c]));
        s.rho = rho_of<T>(I, s.phi);
        s.ux = P.ux[c];
        s.uy = P.uy[c];
        s.p = P.p[c];
        s.mu = P.mu[c];
        T gmx, gmy, gfx, gfy, gpx, gpy;
        grad_field(I, P.mu, ax, ay, i, j, s.mu, gmx, gmy);
        grad_phi<T>(I, P.phi, ax, ay, i, j, P.phi[c], gfx, gfy);
        grad_field(I, P.p, ax, ay, i, j, s.p, gpx, gpy);
        s.lapmu = (T(ax.c2m) * P.mu[cell_of(I, ax.km, j)] + T(ax.c20) * s.mu + T(ax.c2p) * P.mu[cell_of(I, ax.kp, j)])
                + (T(ay.c2m) * P.mu[cell_of(I, i, ay.km)] + T(ay.c20) * s.mu + T(ay.c2p) * P.mu[cell_of(I, i, ay.kp)]);
        s.Fx = -s.phi * gmx + (s.rho - Pr.rho_ref) * Pr.gxa;
        s.Fy = -s.phi * gmy + (s.rho - Pr.rho_ref) * Pr.gya;
        s.grx = Pr.drho * gfx;
        s.gry = Pr.drho * gfy;
        s.gpx = gpx;
        s.gpy = gpy;
        const PtInv<T> v = pt_inv_p<T>(Pr, s);
        const T hdt = T(0.5) * Pr.dt;
        PtBar<T> sb = ptbar_zero<T>();
        InvBar<T> vb = invbar_zero<T>();
#pragma unroll
        for (int q = 0; q < Q; q++) {
            const T xf = Ad.xf[q * N + c], xg = Ad.xg[q * N + c];
            eq_src_adj<T>(s, v, q, xf, xg, -hdt * xf, -hdt * xg, sb, vb);
        }
        pt_inv_adj<T>(Pr, s, v, vb, sb, lamb);
        T gmxb = 0, gmyb = 0, gfxb = 0, gfyb = 0;
        force_adj<T>(Pr, s.phi, gmx, gmy, sb, gmxb, gmyb, gfxb, gfyb);
        sb.phi += Pr.drho * sb.rho;
        // u, p and grad p are inputs held fixed
        Ad.phi[c] = sb.phi;
        Ad.mu[c] = sb.mu;
        Ad.lapmu[c] = sb.lapmu;
        Ad.gmx[c] = gmxb;
        Ad.gmy[c] = gmyb;
        Ad.gfx[c] = gfxb;
        Ad.gfy[c] = gfyb;
    }
    slot_add(Ad.lam_cell + sg, lamb);
}

// d/dlambda and d/dkappa of each instance from the slots of its warps, in a fixed
// order; rng = {first face run, face runs, first cell run, cell runs}, trng = {first
// slot of its tiles' warps, slots}.
__global__ void __launch_bounds__(256) ka_params(const int4 *__restrict__ rng, const int2 *__restrict__ trng,
                                                 const double *__restrict__ lam_face, const double *__restrict__ lam_cell,
                                                 const double *__restrict__ kap0, const double *__restrict__ lam_macro,
                                                 const double *__restrict__ kap, double *pk)
{
    __shared__ double s[2][256];
    const int4 r = rng[blockIdx.x];
    double l = 0.0, k = 0.0;
    for (int w = threadIdx.x; w < r.y; w += 256) l += lam_face[r.x + w];
    for (int w = threadIdx.x; w < r.w; w += 256) {
        l += lam_cell[r.z + w];
        k += kap0[r.z + w];
    }
    const int2 u = trng[blockIdx.x];
    for (int w = threadIdx.x; w < u.y; w += 256) {
        l += lam_macro[u.x + w];
        k += kap[u.x + w];
    }
    s[0][threadIdx.x] = l;
    s[1][threadIdx.x] = k;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) {
            s[0][threadIdx.x] += s[0][threadIdx.x + o];
            s[1][threadIdx.x] += s[1][threadIdx.x + o];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        pk[2 * blockIdx.x] = s[0][0];
        pk[2 * blockIdx.x + 1] = s[1][0];
    }
}

// L = sum_cells (phi - phi*)^2: FP64 partial losses, one slot per warp, and the seed
// adjoint of the state (dL/dg~_i = 2 (phi - phi*), dL/df~_i = 0).
template <typename T>
__global__ void __launch_bounds__(TX *TY) ka_seed(const InstDev *__restrict__ insts, const int4 *__restrict__ tiles,
                                                  Planes<T> P, T *xf, T *xg, const double *__restrict__ target,
                                                  const long long *__restrict__ dense0, double *loss)
{
    const int4 t = tiles[blockIdx.x];
    const InstDev &I = insts[t.x];
    const int i = t.y + threadIdx.x, j = t.z + threadIdx.y;
    double l = 0.0;
    if (i < I.nx && j < I.ny) {
        const long long c = cell_of(I, i, j);
        const long long N = P.N;
        double phi = 0.0;
#pragma unroll
        for (int q = 0; q < Q; q++) phi += (double)P.g[q * N + c];
        const double d = phi - target[dense0[t.x] + (long long)j * I.nx + i];
        l = d * d;
#pragma unroll
        for (int q = 0; q < Q; q++) {
            xf[q * N + c] = T(0);
            xg[q * N + c] = T(2.0 * d);
        }
    }
    for (int o = 16; o > 0; o >>= 1) l += __shfl_down_sync(0xffffffffu, l, o);
    if (threadIdx.x == 0) loss[blockIdx.x * TY + threadIdx.y] = l;
}

// The loss of each instance from its tiles' slots, in a fixed order.
__global__ void __launch_bounds__(256) ka_loss(const InstDev *__restrict__ insts, const double *__restrict__ part, double *loss)
{
    __shared__ double s[256];
    const InstDev &I = insts[blockIdx.x];
    double l = 0.0;
    for (int w = threadIdx.x; w < I.ntiles * TY; w += 256) l += part[(long long)I.tile0 * TY + w];
    s[threadIdx.x] = l;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) s[threadIdx.x] += s[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) loss[blockIdx.x] = s[0];
}

}  // namespace dugks
