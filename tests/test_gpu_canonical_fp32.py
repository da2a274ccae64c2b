"""The canonical step in single precision with walls, both wetting rules, both
equations of state and separate rates, and the fields and the largest speed of the
same kernel: bit for bit against the expressions evaluated operation by operation
in float32, at the edges of its tiles (64 columns in lane pairs 32 apart, 4 rows)."""
import math

import numpy as np
import pytest

from paper_1501_05430_gb300 import inputs as I
from paper_1501_05430_gb300 import lbm as L

pytestmark = pytest.mark.gpu

R = np.float32
EX, EY, OPP = (0, 1, 0, -1, 0, 1, -1, -1, 1), (0, 0, 1, 0, -1, 1, 1, -1, -1), (0, 3, 4, 1, 2, 7, 8, 5, 6)
M = [[1] * 9, [-4, -1, -1, -1, -1, 2, 2, 2, 2], [4, -2, -2, -2, -2, 1, 1, 1, 1], [0, 1, 0, -1, 0, 1, -1, -1, 1],
     [0, -2, 0, 2, 0, 1, -1, -1, 1], [0, 0, 1, 0, -1, 1, 1, -1, -1], [0, 0, -2, 0, 2, 1, 1, -1, -1],
     [0, 1, -1, 1, -1, 0, 0, 0, 0], [0, 0, 0, 0, 0, 1, -1, 1, -1]]
PW10 = (0.25, -0.02, 0.3, 1.1216073327407194, 9.540106186999981)
MODELS = {
    "geometric": dict(),
    "eq19": dict(n_iter=0, tau=0.8),
    "eight_iterations_rates": dict(n_iter=8, tau=0.8, s_e=0.8, s_eps=0.9, s_j=1.0, s_q=1.1),
    "martys_chen": dict(wetting=1, G_w=-0.2, tau=0.9),
    "piecewise": dict(pw=PW10, tau=0.9),
    "piecewise_martys_chen": dict(pw=PW10, wetting=1, G_w=-0.1),
    "periodic_piecewise": dict(pw=PW10, walls=False, tau=0.8),
    "periodic": dict(walls=False, tau=0.8),
}
SIZES = [(33, 5), (63, 6), (64, 7), (65, 8), (66, 9), (67, 10), (129, 7), (130, 6), (4, 5)]


class Model:
    def __init__(self, nx, ny, seed, walls=True, pw=None, tau=1.0, n_iter=4, wetting=0, G_w=0.0, **rates):
        rng = np.random.default_rng(seed)
        self.nx, self.ny, self.walls, self.pw, self.n_iter, self.wetting, self.tau = nx, ny, walls, pw, n_iter, wetting, tau
        self.eos = L.piecewise(*pw) if pw else L.carnahan_starling()  # a = 1, b = 4, R = 1
        self.T = 0.0 if pw else 0.7 * L.lbm_eos_critical(self.eos)[0]
        self.rho_v, self.rho_l, self.rho_max, _ = L.lbm_eos_bounds(self.eos, self.T)
        self.theta = rng.uniform(np.deg2rad(20), np.deg2rad(160), (ny, nx))
        self.G_w, inv = G_w, 1.0 / tau
        self.s = [0.0] + [rates.get(k, inv) for k in ("s_e", "s_eps", "s_j", "s_q", "s_j", "s_q")] + [inv, inv]
        self.params = L.lbm_params_default(precision=32, kernel=L.LBM_KERNEL_REFERENCE, check_every=0, n_iter=n_iter,
                                           wetting=wetting, G_w=G_w, **rates)

    def context(self):
        return L.Lbm(self.nx, self.ny, self.eos, self.T, self.tau, theta=self.theta, walls=self.walls, params=self.params,
                     torch_state=False)

    def psi_U(self, rho):
        if self.pw:
            tv, tm, tl, r1, r2 = (R(v) for v in self.pw)
            p = np.where(rho <= r1, rho * tv,
                         np.where(rho <= r2, r1 * tv + (rho - r1) * tm, (r1 * tv + (r2 - r1) * tm) + (rho - r2) * tl))
        else:
            eta = (R(4) * rho) * R(0.25)
            om = R(1) - eta
            num = ((R(1) + eta) + eta * eta) - (eta * eta) * eta
            p = ((rho * R(self.T)) * num) / ((om * om) * om) - rho * rho
        U = p - rho / R(3)
        return np.sqrt(np.fmax(R(0), R(-2) * U)), U

    def ghost(self, y1, y2, wall):
        """Densities of the solid row of the wall whose first two fluid rows are y1, y2."""
        th = self.theta[0 if wall == 0 else -1]
        fn = math.sin if self.n_iter > 0 else math.tan
        c = np.array([fn(math.pi / 2 - t) for t in th]).astype(R)
        a = np.roll(y1, -1) - np.roll(y1, 1)
        g = y2
        if self.n_iter <= 0:
            g = y2 + c * np.abs(a)
        else:
            d = R(2) * (y2 - y1)
            for _ in range(self.n_iter):
                g = y2 + c * np.sqrt(a * a + d * d)
                d = y2 - g
        return np.fmin(np.fmax(g, R(0)), R(min(self.rho_max, 3.4e38)))

    def evaluate(self, f):
        """Fields of the state f and the state after a step."""
        s, A, kappa = [R(v) for v in self.s], R(-0.6), R(0.5)
        solid = np.zeros((self.ny, self.nx), bool)
        rho = f[0]
        for a in range(1, 9):
            rho = rho + f[a]
        rho = rho.copy()
        psi, U = self.psi_U(rho)
        if self.walls:
            solid[0] = solid[-1] = True
            for row, y1, y2, w in ((0, 1, 2, 0), (-1, -2, -3, 1)):
                rho[row] = psi[row] = U[row] = 0
                if self.wetting == 0:
                    g = self.ghost(rho[y1], rho[y2], w)
                    p, u = self.psi_U(g)
                    rho[row] = g
                    psi[row], U[row] = (np.where(g < R(self.rho_max), v, R(0)) for v in (p, u))
        z = np.zeros_like(rho)
        sp, sU, ss, q1, q2 = [z, z], [z, z], [z, z], [z, z, z], [z, z, z]
        for a in range(1, 9):
            w = R(1) / R(3) if a < 5 else R(1) / R(12)
            pn, un, sn = (np.roll(v, (-EY[a], -EX[a]), (0, 1)) for v in (psi, U, solid.astype(R)))
            t1, t2 = w * (pn - psi), w * (pn * pn - psi * psi)
            for d, e in enumerate((EX[a], EY[a])):
                if e:
                    sp[d], sU[d], ss[d] = sp[d] + R(e) * (w * pn), sU[d] + R(e) * (w * un), ss[d] + R(e) * (w * sn)
            for d, e in enumerate((EX[a] ** 2, EY[a] ** 2, EX[a] * EY[a])):
                if e:
                    q1[d], q2[d] = q1[d] + R(e) * t1, q2[d] + R(e) * t2
        c1, c2, pre = (R(1) - A) * psi, A * R(0.5), kappa * R(-0.5)
        F = [c1 * sp[d] - A * sU[d] for d in (0, 1)]
        if self.wetting:
            F = [F[d] - (R(self.G_w) * psi) * ss[d] for d in (0, 1)]
        Q = [pre * (c1 * q1[d] + c2 * q2[d]) for d in (0, 1, 2)]
        m = []
        for k in range(9):
            acc = z
            for a in range(9):
                if M[k][a]:
                    acc = acc + R(M[k][a]) * f[a]
            m.append(acc)
        Fx, Fy = F
        vx, vy = (m[3] + R(0.5) * Fx) / rho, (m[5] + R(0.5) * Fy) / rho
        v2, vF = vx * vx + vy * vy, vx * Fx + vy * Fy
        eq = [rho, rho * (R(-2) + R(3) * v2), rho * (R(1) - R(3) * v2), rho * vx, -(rho * vx), rho * vy, -(rho * vy),
              rho * (vx * vx - vy * vy), rho * (vx * vy)]
        S = [z, R(6) * vF, -(R(6) * vF), Fx, -Fx, Fy, -Fy, R(2) * (vx * Fx - vy * Fy), vx * Fy + vy * Fx]
        C = [z, (R(1.5) * s[1]) * (Q[0] + Q[1]), z, z, z, z, z, -(s[7] * (Q[0] - Q[1])), -(s[8] * Q[2])]
        r = []
        for k, n in enumerate((9, 36, 36, 6, 12, 6, 12, 4, 4)):
            r.append((((m[k] - s[k] * (m[k] - eq[k])) + (R(1) - R(0.5) * s[k]) * S[k]) + C[k]) / R(n))
        out = np.zeros_like(f)
        for a in range(9):
            acc = z
            for k in range(9):
                if M[k][a]:
                    acc = acc + R(M[k][a]) * r[k]
            into = np.roll(solid, (-EY[a], -EX[a]), (0, 1))  # the node it streams to is solid
            moved = np.roll(np.where(solid | into, R(0), acc), (EY[a], EX[a]), (0, 1))
            came = np.roll(~(solid | into), (EY[a], EX[a]), (0, 1))
            out[a] = np.where(came, moved, out[a])
            out[OPP[a]] = np.where(into & ~solid, acc, out[OPP[a]])
        inside = lambda v: np.where(solid, R(0), v)  # noqa: E731
        return dict(rho=rho, psi=psi, U=U, Fx=inside(Fx), Fy=inside(Fy), Qxx=inside(Q[0]), Qyy=inside(Q[1]),
                    Qxy=inside(Q[2]), ux=inside(vx), uy=inside(vy), f=out)


def _state(m, seed):
    rho = I.droplet_field(m.nx, m.ny, [(m.nx * 0.3, m.ny * 0.35, 0), (m.nx * 0.75, m.ny * 0.3, 1)], m.rho_v, m.rho_l)
    return I.random_distributions(rho, seed, walls=m.walls).astype(R)


def _check(m, f):
    with np.errstate(all="ignore"):
        want = m.evaluate(f)
    with m.context() as s:
        assert s.info.kernel_in_use == L.LBM_KERNEL_REFERENCE
        s.set_f(f.astype(np.float64))
        got = dict(s.fields())
        got["ux"], got["uy"] = s.u()
        speed = s.max_speed()
        s.step(1)
        got["f"] = s.f()
    for k, v in want.items():
        assert np.array_equal(got[k], v.astype(np.float64), equal_nan=True), k
    with np.errstate(all="ignore"):
        assert speed == np.sqrt(np.fmax.reduce((got["ux"] ** 2 + got["uy"] ** 2).ravel()))


@pytest.mark.parametrize("nx,ny", SIZES)
@pytest.mark.parametrize("name", list(MODELS))
def test_step_and_fields_are_the_float32_evaluation(name, nx, ny):
    m = Model(nx, ny, nx + ny, **MODELS[name])
    _check(m, _state(m, nx))


@pytest.mark.parametrize("name", ["periodic", "martys_chen", "periodic_piecewise", "geometric"])
def test_densities_out_of_the_ordinary(name):
    """Nodes of very small, zero, negative and very large density among ordinary ones:
    their quotients and roots are taken plainly, and so are their neighbours'."""
    m = Model(130, 30, 7, **MODELS[name])
    f = _state(m, 3)
    rng = np.random.default_rng(5)
    for scale in (1e-13, 1e-11, 0.0, -1.0, 1e-8, 4.0, 50.0, 1e4):
        for _ in range(4):
            f[:, rng.integers(4, 26), rng.integers(0, 130)] *= R(scale)
    _check(m, f)
