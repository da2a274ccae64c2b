"""The canonical step (one kernel, lbm_canon.cu) at the edges of its tiles:
FP64 bit for bit against the oracle, FP32 bit for bit against the same
expressions evaluated operation by operation in float32."""
import numpy as np
import pytest

from paper_1501_05430_gb300 import inputs as I
from paper_1501_05430_gb300 import lbm as L

from helpers import Pair

pytestmark = pytest.mark.gpu

MODELS = {
    "geometric": dict(),
    "martys_chen": dict(wetting=1, G_w=-0.2, tau=0.9),
    "piecewise": dict(eos="pw", pw=(0.25, -0.02, 0.3, 1.1216073327407194, 9.540106186999981)),
    "periodic_mrt": dict(walls=False, rates=dict(s_e=0.8, s_eps=0.9, s_j=1.0, s_q=1.1)),
}


# tiles of 2 rows (odd and even row counts, one to three strips of 32 columns or
# less), and of 8 rows (80,000 nodes and more; remainders 1 and 0)
@pytest.mark.parametrize("nx,ny", [(33, 7), (32, 6), (65, 9), (403, 203), (1003, 82)])
@pytest.mark.parametrize("name", list(MODELS))
def test_fp64_step_is_the_oracles(name, nx, ny):
    kw = dict(MODELS[name])
    rng = np.random.default_rng(nx)
    p = Pair(nx, ny, theta=rng.uniform(np.deg2rad(20), np.deg2rad(160), (ny, nx)), precision=64,
             kernel=L.LBM_KERNEL_REFERENCE, **kw)
    rho = I.droplet_field(nx, ny, [(nx * 0.3, ny * 0.35, 0), (nx * 0.75, ny * 0.3, 1)], p.rho_v, p.rho_l)
    p.set_f(I.random_distributions(rho, 1, walls=p.walls))
    assert p.step(3) == 0
    assert np.array_equal(p.gpu.f(), p.orc.get_f())
    p.close()


EX, EY = (0, 1, 0, -1, 0, 1, -1, -1, 1), (0, 0, 1, 0, -1, 1, 1, -1, -1)
M = [[1] * 9, [-4, -1, -1, -1, -1, 2, 2, 2, 2], [4, -2, -2, -2, -2, 1, 1, 1, 1], [0, 1, 0, -1, 0, 1, -1, -1, 1],
     [0, -2, 0, 2, 0, 1, -1, -1, 1], [0, 0, 1, 0, -1, 1, 1, -1, -1], [0, 0, -2, 0, 2, 1, 1, -1, -1],
     [0, 1, -1, 1, -1, 0, 0, 0, 0], [0, 0, 0, 0, 0, 1, -1, 1, -1]]


def _float32_step(f, T, A, kappa, s):
    """One step of a periodic Carnahan-Starling (a = 1, b = 4, R = 1) box."""
    R = np.float32
    T, A, kappa, s = R(T), R(A), R(kappa), R(s)
    rho = f[0]
    for a in range(1, 9):
        rho = rho + f[a]
    eta = (R(4) * rho) * R(0.25)
    om = R(1) - eta
    num = ((R(1) + eta) + eta * eta) - (eta * eta) * eta
    p = ((rho * T) * num) / ((om * om) * om) - rho * rho
    U = p - rho / R(3)
    psi = np.sqrt(np.maximum(R(0), R(-2) * U))
    z = np.zeros_like(rho)
    sp, sU, q1, q2 = [z, z], [z, z], [z, z, z], [z, z, z]
    for a in range(1, 9):
        w = R(1) / R(3) if a < 5 else R(1) / R(12)
        pn, un = (np.roll(v, (-EY[a], -EX[a]), (0, 1)) for v in (psi, U))
        t1, t2 = w * (pn - psi), w * (pn * pn - psi * psi)
        for d, e in enumerate((EX[a], EY[a])):
            if e:
                sp[d] = sp[d] + R(e) * (w * pn)
                sU[d] = sU[d] + R(e) * (w * un)
        for d, e in enumerate((EX[a] ** 2, EY[a] ** 2, EX[a] * EY[a])):
            if e:
                q1[d], q2[d] = q1[d] + R(e) * t1, q2[d] + R(e) * t2
    c1, c2, pre = (R(1) - A) * psi, A * R(0.5), kappa * R(-0.5)
    Fx, Fy = (c1 * sp[d] - A * sU[d] for d in (0, 1))
    Qxx, Qyy, Qxy = (pre * (c1 * q1[d] + c2 * q2[d]) for d in (0, 1, 2))
    m = []
    for k in range(9):
        acc = z
        for a in range(9):
            if M[k][a]:
                acc = acc + R(M[k][a]) * f[a]
        m.append(acc)
    vx, vy = (m[3] + R(0.5) * Fx) / rho, (m[5] + R(0.5) * Fy) / rho
    v2, vF = vx * vx + vy * vy, vx * Fx + vy * Fy
    eq = [rho, rho * (R(-2) + R(3) * v2), rho * (R(1) - R(3) * v2), rho * vx, -(rho * vx), rho * vy, -(rho * vy),
          rho * (vx * vx - vy * vy), rho * (vx * vy)]
    S = [z, R(6) * vF, -(R(6) * vF), Fx, -Fx, Fy, -Fy, R(2) * (vx * Fx - vy * Fy), vx * Fy + vy * Fx]
    C = [z, (R(1.5) * s) * (Qxx + Qyy), z, z, z, z, z, -(s * (Qxx - Qyy)), -(s * Qxy)]
    r = []
    for k, n in enumerate((9, 36, 36, 6, 12, 6, 12, 4, 4)):
        sk = s if k else R(0)
        r.append((((m[k] - sk * (m[k] - eq[k])) + (R(1) - R(0.5) * sk) * S[k]) + C[k]) / R(n))
    out = np.empty_like(f)
    for a in range(9):
        acc = z
        for k in range(9):
            if M[k][a]:
                acc = acc + R(M[k][a]) * r[k]
        out[a] = np.roll(acc, (EY[a], EX[a]), (0, 1))
    return out


@pytest.mark.parametrize("nx,ny", [(33, 7), (64, 8), (130, 9), (67, 6), (5, 5)])
@pytest.mark.parametrize("tau", [1.0, 0.8])
def test_fp32_step_is_the_float32_evaluation(nx, ny, tau):
    eos = L.carnahan_starling()
    T = 0.7 * L.lbm_eos_critical(eos)[0]
    rv, rl = L.lbm_coexistence(eos, T)
    f = I.random_distributions(I.droplet_field(nx, ny, [(nx * 0.4, ny * 0.25, ny * 0.5)], rv, rl), 1, walls=False)
    params = L.lbm_params_default(precision=32, kernel=L.LBM_KERNEL_REFERENCE, check_every=0)
    with L.Lbm(nx, ny, eos, T, tau, walls=False, params=params, torch_state=False) as s:
        s.set_f(f)
        s.step(1)
        got = s.f()
    want = _float32_step(f.astype(np.float32), T, -0.6, 0.5, 1.0 / tau)
    assert np.array_equal(got, want.astype(np.float64))
