"""The contact-angle measurement (parallel column sums that narrow the centre
column down, sequential sums where columns tie) and the mass, against the
oracle's sequential measurement of the library's own density field."""
import math

import numpy as np
import pytest

import oracle as O
from paper_1501_05430_gb300 import inputs as I
from paper_1501_05430_gb300 import lbm as L

pytestmark = pytest.mark.gpu


def _sim(nx, ny, precision):
    eos = L.carnahan_starling()
    T = 0.7 * L.lbm_eos_critical(eos)[0]
    p = L.lbm_params_default(precision=precision, check_every=0)
    return L.Lbm(nx, ny, eos, T, 1.0, params=p, torch_state=False), L.lbm_coexistence(eos, T)


def _block(nx, ny, rv, rl, seed, columns, wall):
    """A liquid block whose columns hold the same densities in different orders:
    sums equal up to their rounding, different heights of the first vapour node."""
    rng = np.random.default_rng(seed)
    rho = np.full((ny, nx), rv)
    values = np.concatenate([rng.uniform(0.9, 1.1, 12) * rl, rng.uniform(0.9, 1.1, 8) * rv])
    x0 = nx // 3
    for x in range(x0, x0 + columns):
        col = np.concatenate([[rl], rng.permutation(values)])
        if wall == 0:
            rho[1:22, x] = col
        else:
            rho[ny - 22:ny - 1, x] = col[::-1]
    return rho


@pytest.mark.parametrize("wall", [0, 1])
@pytest.mark.parametrize("precision", [32, 64])
@pytest.mark.parametrize("nx,ny,columns", [(64, 140, 1), (96, 300, 2), (131, 64, 16), (131, 133, 17), (300, 50, 90)])
def test_ties_are_broken_like_the_sequential_measurement(nx, ny, columns, precision, wall):
    sim, (rv, rl) = _sim(nx, ny, precision)
    with sim:
        sim.set_rho(_block(nx, ny, rv, rl, nx + ny, columns, wall))
        th, H, Lb = sim.contact_angle(wall, 2, nx - 1)
        mid = sim.info.rho_mid
        ot, oH, oL, _ = O.contact_angle_field(sim.rho(), wall, 2, nx - 1, mid)
        assert H == oH and Lb == oL and th == pytest.approx(ot, rel=1e-15)


# low halves (200 rows) and higher ones, with up to four and more columns to tell apart
@pytest.mark.parametrize("wall", [0, 1])
@pytest.mark.parametrize("precision", [32, 64])
@pytest.mark.parametrize("nx,ny,columns", [(513, 400, 2), (60, 404, 2), (70, 405, 40), (700, 200, 40), (100, 502, 4), (100, 502, 5), (500, 602, 90), (3000, 66, 1500)])
def test_ties_in_large_domains(nx, ny, columns, precision, wall):
    sim, (rv, rl) = _sim(nx, ny, precision)
    with sim:
        sim.set_rho(_block(nx, ny, rv, rl, nx + ny, columns, wall)[:, :nx])
        mid = sim.info.rho_mid
        for x0, x1 in ((0, nx), (1, nx - 3)):
            ot, oH, oL, _ = O.contact_angle_field(sim.rho(), wall, x0, x1, mid)
            if math.isnan(ot):
                with pytest.raises(L.LbmError):
                    sim.contact_angle(wall, x0, x1)
                continue
            th, H, Lb = sim.contact_angle(wall, x0, x1)
            assert H == oH and Lb == oL and th == pytest.approx(ot, rel=1e-15)


@pytest.mark.parametrize("precision", [32, 64])
@pytest.mark.parametrize("nx,ny", [(131, 140), (200, 500)])
def test_angle_over_columns_with_negative_densities(nx, ny, precision):
    """Sums with negative terms have no bound from the parallel ones: such columns are
    always summed in order.  They may hold the largest sum (a large positive density
    beside the negative one) or not."""
    sim, (rv, rl) = _sim(nx, ny, precision)
    with sim:
        rho = _block(nx, ny, rv, rl, 3, 9, 0)
        for boost in (False, True):
            f = I.random_distributions(rho, 1)
            x = nx // 3 + 4
            f[:, ny // 2 - 2, x] *= -0.5
            f[:, 30, 5] *= -3.0
            if boost:
                f[:, 24, x] *= 50.0 * rl / rv
            sim.set_f(f)
            ot, oH, oL, oxc = O.contact_angle_field(sim.rho(), 0, 0, nx, sim.info.rho_mid)
            th, H, Lb = sim.contact_angle(0, 0, nx)
            assert H == oH and Lb == oL and th == pytest.approx(ot, rel=1e-15)


def test_a_wall_without_droplets_takes_no_longer_than_a_few_angles():
    """All columns tie there: their sums are taken in parallel (one block alone took
    a hundred times as long as the angle of a droplet)."""
    import time

    nx, ny = 4096, 1024
    sim, (rv, rl) = _sim(nx, ny, 32)
    with sim:
        sim.set_rho(I.droplet_field(nx, ny, [(nx * 0.3, ny * 0.3, 0)], rv, rl))

        def best(wall):
            t = []
            for _ in range(8):
                t0 = time.perf_counter()
                try:
                    sim.contact_angle(wall, 0, nx)
                except L.LbmError as e:
                    assert e.status == L.LBM_ENOCONTACT
                t.append(time.perf_counter() - t0)
            return min(t)

        assert best(1) < 5 * best(0)


@pytest.mark.parametrize("precision", [32, 64])
def test_no_contact_line(precision):
    sim, (rv, rl) = _sim(40, 30, precision)
    with sim:
        for rho in (np.full((30, 40), rv), np.full((30, 40), rl)):
            sim.set_rho(rho)
            with pytest.raises(L.LbmError) as e:
                sim.contact_angle(0, 0, 40)
            assert e.value.status == L.LBM_ENOCONTACT
        sim.set_f(np.full((9, 30, 40), np.nan))
        with pytest.raises(L.LbmError) as e:
            sim.contact_angle(1, 3, 20)
        assert e.value.status == L.LBM_ENOCONTACT


def test_batch_angles_are_the_instances_own():
    ws = I.batched(count=9)
    eos = L.carnahan_starling(0.25, 4.0, 1.0)
    tc = L.lbm_eos_critical(eos)[0]
    descs = [dict(nx=w.nx, ny=w.ny, eos=eos, T=w.t_over_tc * tc, tau=w.tau, theta=w.theta) for w in ws]
    with L.LbmBatch(descs) as b:
        for w, d, inst in zip(ws, descs, b.instances):
            rv, rl = L.lbm_coexistence(eos, d["T"])
            inst.set_rho(I.droplet_field(w.nx, w.ny, w.droplets, rv, rl, w.width))
        b[4].set_rho(np.full((ws[4].ny, ws[4].nx), rv))
        th, H, Lb, st = b.contact_angles(0)
        assert st[4] == L.LBM_ENOCONTACT and (st == 0).any()
        for k, inst in enumerate(b.instances):
            try:
                own = inst.contact_angle(0, 0, inst.nx)
            except L.LbmError as e:  # (a wide cap may reach the region's edge too)
                assert st[k] == e.status == L.LBM_ENOCONTACT and math.isnan(th[k])
            else:
                assert st[k] == 0 and (th[k], H[k], Lb[k]) == own


def test_batch_angles_of_large_instances_with_ties():
    """Instances that the batch's pass leaves undecided, among others."""
    eos = L.carnahan_starling()
    T = 0.7 * L.lbm_eos_critical(eos)[0]
    rv, rl = L.lbm_coexistence(eos, T)
    sizes = [(512, 500), (64, 60), (512, 430), (508, 470)]
    with L.LbmBatch([dict(nx=nx, ny=ny, eos=eos, T=T, tau=1.0, theta=None) for nx, ny in sizes]) as b:
        for k, ((nx, ny), inst) in enumerate(zip(sizes, b.instances)):
            inst.set_rho(_block(nx, ny, rv, rl, k, (2, 3, 1, 200)[k], 0))
        for wall in (0, 1):
            th, H, Lb, st = b.contact_angles(wall)
            assert (st == (L.LBM_OK if wall == 0 else L.LBM_ENOCONTACT)).all()
            if wall == 0:
                for k, inst in enumerate(b.instances):
                    ot, oH, oL, _ = O.contact_angle_field(inst.rho(), 0, 0, inst.nx, inst.info.rho_mid)
                    assert (H[k], Lb[k]) == (oH, oL) == inst.contact_angle(0, 0, inst.nx)[1:]


@pytest.mark.parametrize("nx,ny,walls", [(4, 5, True), (64, 33, True), (30, 17, False), (1024, 300, True)])
def test_fp32_mass_is_the_exact_sum(nx, ny, walls):
    """Against the correctly rounded sum of the populations: 48 bits a term and
    fixed-order FP64 sums of up to 3e5 of them stay within 1e-13."""
    eos = L.carnahan_starling()
    T = 0.7 * L.lbm_eos_critical(eos)[0]
    rng = np.random.default_rng(nx)
    f = rng.uniform(0.01, 2.0, (9, ny, nx)) * 10.0 ** rng.uniform(-3, 3, (9, ny, nx))
    if walls:
        f[:, 0] = f[:, -1] = 0.0
    p = L.lbm_params_default(precision=32, check_every=0)
    with L.Lbm(nx, ny, eos, T, 1.0, walls=walls, params=p, torch_state=False) as s:
        s.set_f(f)
        want = math.fsum(f.astype(np.float32).astype(float).ravel())
        assert s.mass() == pytest.approx(want, rel=1e-13)
        f[3, 2, 1] = np.inf
        s.set_f(f)
        assert s.mass() == math.inf


@pytest.mark.parametrize("nx,ny,walls", [(4, 5, True), (8, 6, False), (64, 9, True), (33, 7, True)])
def test_fp32_mass_in_double_precision(nx, ny, walls):
    """Populations added in double: a term passes through at most 9 roundings in
    its density (none where their span allows an exact sum), 4 in a group of four
    nodes, 10 in the block and 10 over the blocks.  The sum may exceed the
    largest float; zeros, negative and subnormal populations count."""
    eos = L.carnahan_starling()
    T = 0.7 * L.lbm_eos_critical(eos)[0]
    p = L.lbm_params_default(precision=32, check_every=0)
    with L.Lbm(nx, ny, eos, T, 1.0, walls=walls, params=p, torch_state=False) as s:
        for seed in range(7):
            rng = np.random.default_rng(seed)
            f = (rng.uniform(0.01, 2.0, (9, ny, nx)) * 10.0 ** rng.uniform(-3, 3, (9, ny, nx))).astype(np.float32)
            if seed == 4:
                f *= rng.choice(np.array([-1.0, 0.0, 1e-40, 1.0], np.float32), f.shape)
            if seed == 5:
                f *= np.float32(1e35)
            if seed == 6:
                f *= np.where(rng.random(f.shape) < 0.05, np.float32(-1e-6), np.float32(1))
            if walls:
                f[:, 0] = f[:, -1] = 0.0
            s.set_f(f.astype(float))
            g = f.astype(float).ravel()
            want, size = math.fsum(g), math.fsum(abs(g))
            assert size < 3.4e38 or seed == 5
            assert abs(s.mass() - want) <= 33 * 2.0**-53 * size


@pytest.mark.parametrize("nx,ny", [(33, 7), (64, 40)])
def test_populations_through_doubles(nx, ny):
    """lbm_set_f rounds to nearest, lbm_get_f is exact, through either buffer
    (the field queries' is there after the first of them)."""
    sim, (rv, rl) = _sim(nx, ny, 32)
    with sim as s:
        for seed in (1, 2):
            f = np.random.default_rng(seed).uniform(1e-3, 1.0, (9, ny, nx))
            f[:, 3, 3] = (1e-42, 1e-46, 3e38, 0.0, -0.0, -1.5, 1 / 3, 2.0**-127, 1 + 2.0**-24)
            s.set_f(f)
            assert np.array_equal(s.f(), f.astype(np.float32).astype(np.float64))
            s.set_f(I.random_distributions(np.full((ny, nx), rv), seed))
            s.u()
