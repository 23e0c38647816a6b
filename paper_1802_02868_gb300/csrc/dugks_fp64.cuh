// dugks_fp64.cuh -- the arithmetic of the fused step in FP64.
//
// GB300 issues one FP64 warp instruction per 64 cycles and SM sub-partition
// (measured: 19.0 cycles per warp-FMA of an SM with 4 or more warps, 1.06
// TFLOP/s of the device), 1/64 of its FP32 rate: the FP64 step is bound by the
// number of FP64 instructions, and loads, shared memory and integer work are
// free beside them.  These functions therefore form the step with as few as the
// formulas allow:
// - a reconstructed bar distribution is one sum over its six (two for the rest
//   and the normal directions) neighbours, with the products of the stencil and
//   interpolation weights formed once per face;
// - equilibrium and source are added before they are multiplied out: for each
//   kind and opposite pair +-q, b eq + c F is
//       w (A +- B) + s (D +- E),   s = w (a +- b'),
//   with A, D scalars of the point, B = xi.(c F), E = xi.(c (F + c_s^2 grad
//   rho)) for f, both xi.(c fg (F - grad p)) for g (Eqs. feq, geq, F, G with
//   (xi - u).X = xi.X - u.X); the weight of the diagonals is part of b and c;
// - one reciprocal of rho (6K + X) serves 1/rho and the f weights;
// - sums start from their small terms (flux sums, sources, tangential derivatives)
//   and end with the one product as large as the result, so that a value is rounded
//   at its own size once or twice and not after each term;
// - face values are stored without the face area, which the update cancels
//   against the cell volume;
// - grad mu, grad phi, lap mu and u of the p phase are kept for the bar-plus
//   phase instead of being formed again.
// By count of the formulas about 250 instructions per face (373 in the general
// templates), 160 per bar-plus cell (300), 54 for p (70), 93 for the update (130).
// us per step before and after: 64x64 drop 36 and 22.5, four 100x100 drops 200 and
// 132, 512x512 drop 855 and 561, Rayleigh-Taylor 256x1024 892 and 597, 2048x2048
// drop 12050 and 7660 (5.5e8 cells/s).
//
// Every operation is spelled out (fma, add, mul with one rounding each), so that
// the kernels that share these functions give the same bits.
#pragma once
#include "dugks_kernels.cuh"

namespace dugks {
namespace fp64 {

__device__ __forceinline__ double fm(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ double mu(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double ad(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double sb(double a, double b) { return __dsub_rn(a, b); }

// 1 / x for normal x: the hardware's reciprocal estimate and one step of the
// third-order iteration r (1 + e + e^2), e = 1 - x r (Householder).  51 cycles
// per warp against 86 for 1.0 / x; worst |1 - x r| over 1.6e7 random x is
// 1.11e-16, half a unit in the last place of 1.
__device__ __forceinline__ double rcp(double x)
{
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    double e = fm(-x, r, 1.0);
    e = fm(e, e, e);
    return fm(r, e, r);
}

// finite, on the integer pipe
__device__ __forceinline__ bool finite(double v) { return (__double2hiint(v) & 0x7ff00000) != 0x7ff00000; }

__device__ __forceinline__ double rho_of(const InstDev &I, double phi) { return fm(I.drho, sb(phi, I.phiB), I.rhoB); }

// total force F = -phi grad mu + (rho - rho_ref) g
__device__ __forceinline__ double force(double phi, double gm, double drho, double ga) { return fm(-phi, gm, mu(drho, ga)); }

// Sums of the nine values of a distribution and of xi f.
struct Mom { double s, x, y; };
__device__ __forceinline__ Mom moments(const double (&f)[Q])
{
    const double d57 = sb(f[5], f[7]), d68 = sb(f[6], f[8]);
    Mom m;
    m.s = ad(ad(ad(f[0], ad(f[1], f[3])), ad(f[2], f[4])), ad(ad(f[5], f[7]), ad(f[6], f[8])));
    m.x = ad(sb(f[1], f[3]), sb(d57, d68));
    m.y = ad(sb(f[2], f[4]), ad(d57, d68));
    return m;
}

// Chemical potential (Eq. chemicalpotential) from phi and its four differences
// to the neighbours.
__device__ __forceinline__ double chem(const InstDev &I, double p0, double dxm, double dxp, double dym, double dyp,
                                       double cxm, double cxp, double cym, double cyp)
{
    const double lap = ad(fm(cxm, dxm, mu(cxp, dxp)), fm(cym, dym, mu(cyp, dyp)));
    const double d = mu(mu(mu(I.b4, sb(p0, I.cA.d)), sb(p0, I.cB.d)), sb(p0, I.cM.d));
    return fm(-I.kappa, lap, d);
}

// u and p of a point (Eqs. u, P at a cell, Eq. conservedVariable at a face;
// C.kf = c_s^2 times half the time over which the force acts).
__device__ __forceinline__ void velocity(const PtC<double> &C, const Mom &m, double irho, double Fx, double Fy, double &ux, double &uy)
{
    const double r3 = mu(3.0, irho);
    ux = mu(fm(C.kf, Fx, m.x), r3);
    uy = mu(fm(C.kf, Fy, m.y), r3);
}
__device__ __forceinline__ double pressure(const PtC<double> &C, double sf, double ux, double uy, double gfx, double gfy, double rho_lmu)
{
    return fm(C.kp1, fm(ux, gfx, mu(uy, gfy)), fm(-C.kp2, rho_lmu, sf));
}

// What the directions of a point share.  KIND: 1 = f only, 2 = g only, 3 = both.
struct Eq {
    double a, K0, K1, fx, fy, ex, ey;       // f: weight of the distribution; A, D; c F; c (F + c_s^2 grad rho)
    double A2, D2, gx, gy;                  // g: A, D; c fg (F - grad p)
    double s0, ax, bx, ay, by, ap, bp, am, bm;   // s_i / w: rest, x, y, (1,1), (-1,1)
};

// X = h D rho of Eq. (mixvis), see cell_weights
__device__ __forceinline__ double weight_x(const InstDev &I, double phi, double rho)
{
    return mu(fm(sb(phi, I.phiB), I.pd.hmuB, mu(sb(I.phiA, phi), I.pd.hmuA)), rho);
}

template <int KIND>
__device__ __forceinline__ void eq_dirs(double ux, double uy, Eq &E)
{
    const double uxx = mu(ux, ux), uyy = mu(uy, uy);
    const double sA = mu(-1.5, ad(uxx, uyy));
    E.s0 = sA;
    E.ax = fm(4.5, uxx, sA);
    E.bx = mu(3.0, ux);
    E.ay = fm(4.5, uyy, sA);
    E.by = mu(3.0, uy);
    const double up = ad(ux, uy), um = sb(uy, ux);
    E.ap = fm(4.5, mu(up, up), sA);
    E.bp = mu(3.0, up);
    E.am = fm(4.5, mu(um, um), sA);
    E.bm = mu(3.0, um);
}

// f part: r = 1 / (6K + k X), X the weight variable; CELL: Eq. (relations1), else Eq. (original-function)
template <bool CELL>
__device__ __forceinline__ void eq_f(const InstDev &I, const PtC<double> &C, double X, double r, double rho, double rho_lmu, double ux,
                                     double uy, double p, double Fx, double Fy, double gfx, double gfy, Eq &E)
{
    E.a = mu(CELL ? sb(C.k6, X) : C.k6, r);
    const double b = mu(X, mu(C.nb, r)), c = mu(C.nc, r);
    const double FCx = fm(C.cd, gfx, Fx), FCy = fm(C.cd, gfy, Fy);
    const double uF = fm(ux, Fx, mu(uy, Fy)), uFC = fm(ux, FCx, mu(uy, FCy));
    E.K0 = fm(-c, fm(C.cgl, rho_lmu, uF), mu(b, p));
    E.K1 = fm(-c, uFC, mu(b, mu(1.0 / 3.0, rho)));
    E.fx = mu(c, Fx);
    E.fy = mu(c, Fy);
    E.ex = mu(c, FCx);
    E.ey = mu(c, FCy);
}
__device__ __forceinline__ void eq_g(const PtC<double> &C, double phi, double irho, double ux, double uy, double m, double Gx,
                                     double Gy, Eq &E)
{
    const double P = mu(mu(C.gc, phi), irho);
    E.gx = mu(P, Gx);
    E.gy = mu(P, Gy);
    const double u = fm(ux, E.gx, mu(uy, E.gy));
    E.D2 = fm(C.gb, phi, -u);
    E.A2 = fm(C.gbe, m, -u);
}

// b eq + c F (over the diagonals' weight) of direction q in {1, 2, 5, 6} and of
// its opposite, added to a times the distribution's values v0, v1
template <int q>
__device__ __forceinline__ void pair_of(double a, double A, double D, double Bx, double By, double Ex, double Ey, const Eq &E,
                                        double v0, double v1, double &o0, double &o1)
{
    const double s = q == 1 ? E.ax : q == 2 ? E.ay : q == 5 ? E.ap : E.am;
    const double t = q == 1 ? E.bx : q == 2 ? E.by : q == 5 ? E.bp : E.bm;
    const double B = q == 1 ? Bx : q == 2 ? By : q == 5 ? ad(Bx, By) : sb(By, Bx);
    const double X = q == 1 ? Ex : q == 2 ? Ey : q == 5 ? ad(Ex, Ey) : sb(Ey, Ex);
    const double ev = fm(t, X, fm(s, D, A)), od = fm(t, D, fm(s, X, B));
    if (q < 5) {   // the axis weight is four times the diagonals'
        o0 = fm(a, v0, mu(4.0, ad(ev, od)));
        o1 = fm(a, v1, mu(4.0, sb(ev, od)));
    } else {
        o0 = fm(a, v0, ad(ev, od));
        o1 = fm(a, v1, sb(ev, od));
    }
}
template <int q>
__device__ __forceinline__ void pair_f(const Eq &E, double v0, double v1, double &o0, double &o1)
{
    pair_of<q>(E.a, E.K0, E.K1, E.fx, E.fy, E.ex, E.ey, E, v0, v1, o0, o1);
}
template <int q>
__device__ __forceinline__ void pair_g(const PtC<double> &C, const Eq &E, double v0, double v1, double &o0, double &o1)
{
    pair_of<q>(C.ga, E.A2, E.D2, E.gx, E.gy, E.gx, E.gy, E, v0, v1, o0, o1);
}

// bar-plus of f or g at a cell (Eq. relations1), in place of the nine values
__device__ __forceinline__ void bar_plus_f(const Eq &E, double (&v)[Q])
{
    v[0] = fm(E.a, v[0], mu(16.0, fm(E.s0, E.K1, E.K0)));
    pair_f<1>(E, v[1], v[3], v[1], v[3]);
    pair_f<2>(E, v[2], v[4], v[2], v[4]);
    pair_f<5>(E, v[5], v[7], v[5], v[7]);
    pair_f<6>(E, v[6], v[8], v[6], v[8]);
}
__device__ __forceinline__ void bar_plus_g(const PtC<double> &C, const Eq &E, double phi, double m, double (&v)[Q])
{
    // the rest direction's H is phi - (1 - w_0) eta mu
    const double rest = fm(-C.gbe36, m, mu(16.0, fm(E.s0, E.D2, E.A2)));
    v[0] = fm(C.ga, v[0], fm(C.gb36, phi, rest));
    pair_g<1>(C, E, v[1], v[3], v[1], v[3]);
    pair_g<2>(C, E, v[2], v[4], v[2], v[4]);
    pair_g<5>(C, E, v[5], v[7], v[5], v[7]);
    pair_g<6>(C, E, v[6], v[8], v[6], v[8]);
}

// Values that a face interpolates from its cells.
struct Aux { double mu, lmu, gmx, gmy, gfx, gfy, gpx, gpy; };

// Originals (Eq. original-function) of the six flux directions of axis A from
// the nine bar values of each kind; at a wall (side != 0) u = 0 and the incoming
// ones bounce back.  Returned as xi_A phi_i, in fset order.
template <int A>
__device__ __forceinline__ void originals(const InstDev &I, const double (&fb)[Q], const double (&gb)[Q], const Aux &x, int side,
                                          double2 (&o)[6])
{
    const PtC<double> &C = I.face64;
    const Mom m = moments(fb);
    const double phi = ad(ad(ad(gb[0], ad(gb[1], gb[3])), ad(gb[2], gb[4])), ad(ad(gb[5], gb[7]), ad(gb[6], gb[8])));
    const double rho = rho_of(I, phi), dr = sb(rho, I.rho_ref);
    const double Fx = force(phi, x.gmx, dr, I.gxa), Fy = force(phi, x.gmy, dr, I.gya);
    const double X = weight_x(I, phi, rho), den = ad(C.k6, X);
    const double inv = rcp(mu(rho, den)), irho = mu(inv, den), r = mu(inv, rho);
    double ux, uy;
    velocity(C, m, irho, Fx, Fy, ux, uy);
    if (side != 0) ux = uy = 0.0;
    const double rl = mu(rho, x.lmu);
    const double p = pressure(C, m.s, ux, uy, x.gfx, x.gfy, rl);
    Eq E;
    eq_dirs<3>(ux, uy, E);
    eq_f<false>(I, C, X, r, rho, rl, ux, uy, p, Fx, Fy, x.gfx, x.gfy, E);
    eq_g(C, phi, irho, ux, uy, x.mu, sb(Fx, x.gpx), sb(Fy, x.gpy), E);
    constexpr int n = A == 0 ? 1 : 2, n2 = A == 0 ? 3 : 4;
    // fset<A>: +n, -n, 5, 6, 7, 8
    pair_f<n>(E, fb[n], fb[n2], o[0].x, o[1].x);
    pair_g<n>(C, E, gb[n], gb[n2], o[0].y, o[1].y);
    pair_f<5>(E, fb[5], fb[7], o[2].x, o[4].x);
    pair_g<5>(C, E, gb[5], gb[7], o[2].y, o[4].y);
    pair_f<6>(E, fb[6], fb[8], o[3].x, o[5].x);
    pair_g<6>(C, E, gb[6], gb[8], o[3].y, o[5].y);
    if (side != 0) {
#pragma unroll
        for (int k = 0; k < 6; k++) {
            const int r = k < 2 ? 1 - k : k < 4 ? k + 2 : k - 2;   // the place of the opposite
            if (ca(fset<A>(k), A) * side < 0) o[k] = o[r];
        }
    }
}

// mu on the R3 position (x, y)
template <typename TL>
__device__ __forceinline__ void mu_point(const InstDev &I, const TL &S, int x, int y)
{
    double v = 0.0;
    if (S.ok(0, x) && S.ok(1, y)) {
        const double p0 = S.phi[TL::i4(x, y)];
        v = chem(I, p0, sb(S.phi[TL::i4(x + S.om(0, x), y)], p0), sb(S.phi[TL::i4(x + S.op(0, x), y)], p0),
                 sb(S.phi[TL::i4(x, y + S.om(1, y))], p0), sb(S.phi[TL::i4(x, y + S.op(1, y))], p0), S.c(2, 0, x), S.c(3, 0, x),
                 S.c(2, 1, y), S.c(3, 1, y));
    }
    S.mu[TL::i3(x, y)] = v;
}

// p and what the bar-plus phase and the faces reuse (grad mu, lap mu, grad phi,
// u) on the R2 position (x, y); f: its tilde f
template <typename TL>
__device__ __forceinline__ void p_point(const InstDev &I, const TL &S, int x, int y, const double (&f)[Q])
{
    const int k = TL::i2(x, y);
    if (!S.ok(0, x) || !S.ok(1, y)) {
        S.p[k] = 0.0;
        return;
    }
    const double m0 = S.mu[TL::i3(x, y)];
    const double xm = sb(S.mu[TL::i3(x + S.om(0, x), y)], m0), xp = sb(S.mu[TL::i3(x + S.op(0, x), y)], m0);
    const double ym = sb(S.mu[TL::i3(x, y + S.om(1, y))], m0), yp = sb(S.mu[TL::i3(x, y + S.op(1, y))], m0);
    const double gmx = fm(S.c(0, 0, x), xm, mu(S.c(1, 0, x), xp)), gmy = fm(S.c(0, 1, y), ym, mu(S.c(1, 1, y), yp));
    const double lmu = ad(fm(S.c(2, 0, x), xm, mu(S.c(3, 0, x), xp)), fm(S.c(2, 1, y), ym, mu(S.c(3, 1, y), yp)));
    const double phi = S.phi[TL::i4(x, y)];
    const double gfx = fm(S.c(0, 0, x), sb(S.phi[TL::i4(x + S.om(0, x), y)], phi),
                          mu(S.c(1, 0, x), sb(S.phi[TL::i4(x + S.op(0, x), y)], phi)));
    const double gfy = fm(S.c(0, 1, y), sb(S.phi[TL::i4(x, y + S.om(1, y))], phi),
                          mu(S.c(1, 1, y), sb(S.phi[TL::i4(x, y + S.op(1, y))], phi)));
    const double rho = rho_of(I, phi), dr = sb(rho, I.rho_ref);
    const Mom m = moments(f);
    double ux, uy;
    velocity(I.cell64, m, rcp(rho), force(phi, gmx, dr, I.gxa), force(phi, gmy, dr, I.gya), ux, uy);
    S.p[k] = pressure(I.cell64, m.s, ux, uy, gfx, gfy, mu(rho, lmu));
    S.gmx[k] = gmx;
    S.gmy[k] = gmy;
    S.lmu[k] = lmu;
    S.gfx[k] = gfx;
    S.gfy[k] = gfy;
    S.ux[k] = ux;
    S.uy[k] = uy;
}

// bar-plus (Eq. relations1) of f (KIND 1), g and grad p (2) or all (3) on the R1
// position (x, y); f, g: its tilde values
template <int KIND, typename TL>
__device__ __forceinline__ void bar_plus_point(const InstDev &I, const TL &S, int x, int y, double (&f)[Q], double (&g)[Q])
{
    if (!S.ok(0, x) || !S.ok(1, y)) return;   // no face reads it
    const PtC<double> &C = I.cell64;
    const int k1 = TL::i1(x, y), k2 = TL::i2(x, y);
    const double phi = S.phi[TL::i4(x, y)], m = S.mu[TL::i3(x, y)], p = S.p[k2];
    const double rho = rho_of(I, phi), dr = sb(rho, I.rho_ref);
    const double Fx = force(phi, S.gmx[k2], dr, I.gxa), Fy = force(phi, S.gmy[k2], dr, I.gya);
    const double ux = S.ux[k2], uy = S.uy[k2];
    const double X = weight_x(I, phi, rho), den = fm(2.0, X, C.k6);
    const double inv = rcp(mu(rho, den));
    Eq E;
    eq_dirs<KIND>(ux, uy, E);
    if (KIND & 1) {
        eq_f<true>(I, C, X, mu(inv, rho), rho, mu(rho, S.lmu[k2]), ux, uy, p, Fx, Fy, S.gfx[k2], S.gfy[k2], E);
        bar_plus_f(E, f);
#pragma unroll
        for (int q = 0; q < Q; q++) S.bp[q * TL::L::A1 + k1].x = f[q];
    }
    if (KIND & 2) {
        const double gpx = fm(S.c(0, 0, x), sb(S.p[TL::i2(x + S.om(0, x), y)], p), mu(S.c(1, 0, x), sb(S.p[TL::i2(x + S.op(0, x), y)], p)));
        const double gpy = fm(S.c(0, 1, y), sb(S.p[TL::i2(x, y + S.om(1, y))], p), mu(S.c(1, 1, y), sb(S.p[TL::i2(x, y + S.op(1, y))], p)));
        S.gpx[k1] = gpx;
        S.gpy[k1] = gpy;
        eq_g(C, phi, mu(inv, den), ux, uy, m, sb(Fx, gpx), sb(Fy, gpy), E);
        bar_plus_g(C, E, phi, m, g);
#pragma unroll
        for (int q = 0; q < Q; q++) S.bp[q * TL::L::A1 + k1].y = g[q];
    }
}

// Originals of the flux directions at the face between positions a and b = a +
// e_A of a tile, or at the wall face of whichever of the two lies in the domain.
template <int A, bool UNI, typename TL>
__device__ __forceinline__ void face(const InstDev &I, const TL &S, int xa, int ya, double2 (&o)[6])
{
    constexpr int A1 = TL::L::A1;
    const int xb = xa + (A == 0 ? 1 : 0), yb = ya + (A == 1 ? 1 : 0);
    const int pa = A == 0 ? xa : ya, pb = A == 0 ? xb : yb, pt = A == 0 ? ya : xa;
#pragma unroll
    for (int k = 0; k < 6; k++) o[k] = make_double2(0.0, 0.0);
    if (!S.ok(1 - A, pt)) return;
    const bool va = S.ok(A, pa), vb = S.ok(A, pb);
    // tangential neighbours: a row step for x faces, a column step for y faces
    const int tm = A == 0 ? S.rs1(pt, S.om(1, pt)) : S.om(0, pt);
    const int tp = A == 0 ? S.rs1(pt, S.op(1, pt)) : S.op(0, pt);
    const double em = S.c(4, 1 - A, pt), e0 = S.c(5, 1 - A, pt), ep = S.c(6, 1 - A, pt);   // times h
    // the side of a wall face's cell that the wall is on; 0 for any other face.
    // Both kinds meet again before originals(): a warp that holds wall faces and
    // interior ones then runs the longer part of a face once.
    int side = 0;
    const bool inner = UNI || (va && vb);
    if (!inner) {
        if (!va && vb && (S.gf[S.ge(A, pb)] & 4)) side = -1;
        else if (va && !vb && (S.gf[S.ge(A, pa)] & 8)) side = +1;
        else return;
    }
    double fb[Q], gb[Q];
    Aux x;
    if (inner) {
        const int ia = S.i1(xa, ya), ib = S.i1(xb, yb), ja = S.i2(xa, ya), jb = S.i2(xb, yb);
        const double wL = S.c(7, A, pa), wR = S.c(8, A, pa), k = S.c(9, A, pa);   // k = h / distance
        // weights of the two cells for xi_A = 0, +1, -1, and of their tangential
        // neighbours (the two cells' agree on a uniform mesh, and the centre
        // weight of the tangential derivative is zero)
        const double Lp = ad(wL, k), Rp = sb(wR, k), Lm = UNI ? Rp : sb(wL, k), Rm = UNI ? Lp : ad(wR, k);
        const double Lmt = mu(wL, em), Lpt = mu(wL, ep), Rmt = UNI ? Lmt : mu(wR, em), Rpt = UNI ? Lpt : mu(wR, ep);
        const double L0 = UNI ? 0.0 : mu(wL, e0), R0 = UNI ? 0.0 : mu(wR, e0);
#pragma unroll
        for (int q = 0; q < Q; q++) {
            const int n = ca(q, A), t = ca(q, 1 - A);
            const double2 *B = S.bp + q * A1;
            const double2 bL = B[ia], bR = B[ib];
            double cL = n == 0 ? wL : n > 0 ? Lp : Lm, cR = n == 0 ? wR : n > 0 ? Rp : Rm;
            if (t && !UNI) {
                cL = t > 0 ? sb(cL, L0) : ad(cL, L0);
                cR = t > 0 ? sb(cR, R0) : ad(cR, R0);
            }
            if (t) {
                const double2 a0 = B[ia + tm], a1 = B[ia + tp], b0 = B[ib + tm], b1 = B[ib + tp];
                const double l0 = t > 0 ? -Lmt : Lmt, l1 = t > 0 ? -Lpt : Lpt, r0 = t > 0 ? -Rmt : Rmt, r1 = t > 0 ? -Rpt : Rpt;
                const double df = fm(l0, a0.x, fm(l1, a1.x, fm(r0, b0.x, mu(r1, b1.x))));
                const double dg = fm(l0, a0.y, fm(l1, a1.y, fm(r0, b0.y, mu(r1, b1.y))));
                fb[q] = fm(cL, bL.x, fm(cR, bR.x, df));
                gb[q] = fm(cL, bL.y, fm(cR, bR.y, dg));
            } else {
                fb[q] = fm(cL, bL.x, mu(cR, bR.x));
                gb[q] = fm(cL, bL.y, mu(cR, bR.y));
            }
        }
        const int ma = S.i3(xa, ya), mb = S.i3(xb, yb);
        x.mu = fm(wL, S.mu[ma], mu(wR, S.mu[mb]));
        x.lmu = fm(wL, S.lmu[ja], mu(wR, S.lmu[jb]));
        x.gmx = fm(wL, S.gmx[ja], mu(wR, S.gmx[jb]));
        x.gmy = fm(wL, S.gmy[ja], mu(wR, S.gmy[jb]));
        x.gfx = fm(wL, S.gfx[ja], mu(wR, S.gfx[jb]));
        x.gfy = fm(wL, S.gfy[ja], mu(wR, S.gfy[jb]));
        x.gpx = fm(wL, S.gpx[ia], mu(wR, S.gpx[ib]));
        x.gpy = fm(wL, S.gpy[ia], mu(wR, S.gpy[ib]));
    } else {
        const int xc = side < 0 ? xb : xa, yc = side < 0 ? yb : ya, pc = side < 0 ? pb : pa;
        // wall face of cell c: Taylor reconstruction from the cell centre for the
        // outgoing and parallel directions, bounce-back for the incoming ones
        const int ic = S.i1(xc, yc), jc = S.i2(xc, yc);
        const int nm = A == 0 ? S.om(0, pc) : S.rs1(yc, S.om(1, pc));
        const int np = A == 0 ? S.op(0, pc) : S.rs1(yc, S.op(1, pc));
        const double fm_ = S.c(4, A, pc), f0 = S.c(5, A, pc), fp = S.c(6, A, pc);   // times h
        const double half = mu(mu(0.5, S.c(10, A, pc)), I.rh64);                      // half width over h
#pragma unroll
        for (int q = 0; q < Q; q++) {
            if (ca(q, A) * side < 0) continue;
            const double off = sb(side > 0 ? half : -half, (double)ca(q, A));
            const double s = -(double)ca(q, 1 - A);
            const double2 *B = S.bp + q * A1;
            const double2 b = B[ic], b0 = B[ic + nm], b1 = B[ic + np], t0 = B[ic + tm], t1 = B[ic + tp];
            const double nf = fm(fm_, b0.x, fm(f0, b.x, mu(fp, b1.x))), ng = fm(fm_, b0.y, fm(f0, b.y, mu(fp, b1.y)));
            if (ca(q, 1 - A)) {
                fb[q] = ad(b.x, fm(off, nf, mu(s, fm(em, t0.x, fm(e0, b.x, mu(ep, t1.x))))));
                gb[q] = ad(b.y, fm(off, ng, mu(s, fm(em, t0.y, fm(e0, b.y, mu(ep, t1.y))))));
            } else {
                fb[q] = fm(off, nf, b.x);
                gb[q] = fm(off, ng, b.y);
            }
        }
#pragma unroll
        for (int q = 0; q < Q; q++) {
            if (ca(q, A) * side < 0) {
                fb[q] = fb[opp(q)];
                gb[q] = gb[opp(q)];
            }
        }
        x.mu = S.mu[S.i3(xc, yc)];
        x.lmu = S.lmu[jc];
        x.gmx = A == 0 ? 0.0 : S.gmx[jc];
        x.gmy = A == 1 ? 0.0 : S.gmy[jc];
        x.gfx = A == 0 ? 0.0 : S.gfx[jc];
        x.gfy = A == 1 ? 0.0 : S.gfy[jc];
        x.gpx = A == 0 ? 0.0 : S.gpx[ic];
        x.gpy = A == 1 ? 0.0 : S.gpy[ic];
    }
    originals<A>(I, fb, gb, x, side, o);
}

// Update of one kind (Eqs. relations2, updatef) at a cell: east, west, north and
// south face values by flux direction, kx = dt / dx, ky = dt / dy (the face
// areas against the volume), old and bar-plus values by direction.
template <typename FE, typename FW, typename FN, typename FS, typename FO, typename FB>
__device__ __forceinline__ void update(double kx, double ky, FE e, FW w, FN n, FS s, FO old, FB bp, double (&nw)[Q])
{
    double J[Q];   // -dt / |V| times the flux sum
    J[0] = 0.0;
#pragma unroll
    for (int m = 0; m < 6; m++) J[xset(m)] = mu(cx(xset(m)) > 0 ? -kx : kx, sb(e(m), w(m)));
#pragma unroll
    for (int m = 0; m < 6; m++) {
        const int q = yset(m);
        const double k = cy(q) > 0 ? -ky : ky, d = sb(n(m), s(m));
        J[q] = cx(q) ? fm(k, d, J[q]) : mu(k, d);
    }
#pragma unroll
    for (int q = 0; q < Q; q++) nw[q] = fm(4.0 / 3.0, bp(q), fm(-1.0 / 3.0, old(q), J[q]));
}

// The update's KIND (1 f, 2 g, 3 both) at cell c: writes the new state; false if
// a value is not finite.
template <int KIND, typename IO, typename FE, typename FW, typename FN, typename FS, typename TL>
__device__ __forceinline__ bool update_cell(const IO &io, const TL &S, int x, int y, long long c, FE e, FW w, FN n, FS s)
{
    const double kx = S.c(11, 0, x), ky = S.c(11, 1, y);
    const int r1 = TL::i1(x, y);
    const long long N = io.N;
    bool ok = true;
    double v[Q];
    if (KIND & 1) {
        update(kx, ky, [&](int m) { return e(m).x; }, [&](int m) { return w(m).x; }, [&](int m) { return n(m).x; },
               [&](int m) { return s(m).x; }, [&](int q) { return io.f_in[q * N + c]; },
               [&](int q) { return S.bp[q * TL::L::A1 + r1].x; }, v);
#pragma unroll
        for (int q = 0; q < Q; q++) {
            io.f_out[q * N + c] = v[q];
            ok = ok && finite(v[q]);
        }
    }
    if (KIND & 2) {
        update(kx, ky, [&](int m) { return e(m).y; }, [&](int m) { return w(m).y; }, [&](int m) { return n(m).y; },
               [&](int m) { return s(m).y; }, [&](int q) { return io.g_in[q * N + c]; },
               [&](int q) { return S.bp[q * TL::L::A1 + r1].y; }, v);
        double phi = v[0];
#pragma unroll
        for (int q = 0; q < Q; q++) {
            io.g_out[q * N + c] = v[q];
            if (q > 0) phi = ad(phi, v[q]);
            ok = ok && finite(v[q]);
        }
        io.phi_out[c] = phi;
    }
    return ok;
}

}  // namespace fp64
}  // namespace dugks
