"""The algebra of the FP64 step's point functions (dugks_fp64.cuh), restated in
extended precision on the CPU: b eq + c F of every direction equals the sum of
the separate equilibria and sources (Eqs. feq, geq, F, G)."""
import numpy as np

CX = [0, 1, 0, -1, 0, 1, -1, -1, 1]
CY = [0, 0, 1, 0, -1, 1, 1, -1, -1]
L = np.longdouble
W = [L(4) / 9] + [L(1) / 9] * 4 + [L(1) / 36] * 4


def test_combined_equilibria_and_sources():
    rng = np.random.default_rng(5)
    for _ in range(50):
        phi, rho, ux, uy, p, mu, lmu, Fx, Fy, gfx, gfy, gpx, gpy = (L(v) for v in rng.uniform(-1, 1, 13))
        rho = rho + 2
        drho, gam, lam, eta, a, b, c, a2, b2, c2 = (L(v) for v in rng.uniform(0.1, 1, 10))
        w = W[5]
        # the point's scalars and vectors, the diagonals' weight folded in
        cs2 = L(1) / 3
        FC = (Fx + cs2 * drho * gfx, Fy + cs2 * drho * gfy)
        uF, uFC = ux * Fx + uy * Fy, ux * FC[0] + uy * FC[1]
        K0 = w * (b * p - c * (cs2 * gam * lam * rho * lmu + uF))
        K1 = w * (b * rho / 3 - c * uFC)
        P = 3 * w * c2 * phi / rho
        g = (P * (Fx - gpx), P * (Fy - gpy))
        ug = ux * g[0] + uy * g[1]
        D2, A2 = w * b2 * phi - ug, w * b2 * eta * mu - ug
        uu = ux * ux + uy * uy
        for q in range(9):
            xu = CX[q] * ux + CY[q] * uy
            s = 3 * xu + L(4.5) * xu * xu - L(1.5) * uu
            ex, ey = CX[q] - ux, CY[q] - uy
            feq = W[q] * p + rho / 3 * W[q] * s
            H = phi - (1 - W[0]) * eta * mu if q == 0 else W[q] * eta * mu
            geq = H + phi * W[q] * s
            G = W[q] * (1 + s)
            Ff = G * (ex * Fx + ey * Fy) + W[q] * s * cs2 * drho * (ex * gfx + ey * gfy) - W[q] * cs2 * rho * gam * lam * lmu
            Fg = 3 * phi / rho * (ex * (Fx - gpx) + ey * (Fy - gpy)) * G
            ratio = W[q] / w
            f_new = ratio * (K0 + w * c * (CX[q] * Fx + CY[q] * Fy) + s * (K1 + w * c * (CX[q] * FC[0] + CY[q] * FC[1])))
            g_new = ratio * (A2 + CX[q] * g[0] + CY[q] * g[1] + s * (D2 + CX[q] * g[0] + CY[q] * g[1]))
            if q == 0:
                g_new += b2 * (phi - eta * mu)
            # the terms are O(10): 1e-16 of them in extended precision
            assert abs(f_new - (b * feq + c * Ff)) < 1e-15 and abs(g_new - (b2 * geq + c2 * Fg)) < 1e-15
