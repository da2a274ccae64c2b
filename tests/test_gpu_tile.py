"""The small-domain kernel of the FP32 step (one tile per CTA) against the ring
kernel: the same per-node operations on the same values, so the same bits, and
the same verdict on an unstable state.  (Both are compared with the oracle in
test_gpu_parity.py.)"""
import numpy as np
import pytest

from paper_1501_05430_gb300 import inputs as I
from paper_1501_05430_gb300 import lbm as L

from helpers import Case

pytestmark = pytest.mark.gpu

PW10 = (0.25, -0.02, 0.3, 1.1216073327407194, 9.540106186999981)
MODELS = {
    "geometric": dict(),
    "eq19": dict(n_iter=0),
    "general_rates": dict(rates=dict(s_e=0.8, s_eps=0.9, s_j=1.0, s_q=1.1), tau=0.8),
    "martys_chen": dict(wetting=1, G_w=-0.2),
    "martys_chen_general": dict(wetting=1, G_w=-0.2, tau=0.9),
    "piecewise": dict(eos="pw", pw=PW10),
    "piecewise_martys_chen_general": dict(eos="pw", pw=PW10, wetting=1, G_w=-0.1, tau=0.8),
    "periodic": dict(walls=False),
}
# one and several strips with a ragged last one (64 columns a tile, 58 with two
# steps per launch, which 4 columns are too few for), bands with every remainder
# (walled: ny - 2 rows), the smallest grids, seven strips of the ring kernel (whose
# CTAs are then a multiple of seven)
SIZES = [(4, 5), (8, 5), (8, 6), (56, 6), (60, 7), (64, 6), (68, 8), (116, 10), (132, 9), (260, 24), (128, 13), (1700, 100)]


def _context(c, f, monkeypatch, ring):
    if ring:
        monkeypatch.setenv("LBM_FUSED_STAGES", "3")
    else:
        monkeypatch.delenv("LBM_FUSED_STAGES", raising=False)
    g = L.Lbm(c.nx, c.ny, c.geos, c.T, c.tau, theta=c.theta, walls=c.walls, params=c.params, torch_state=False)
    assert g.info.kernel_in_use == L.LBM_KERNEL_FUSED
    assert (g.info.tile_stages > 0) == ring
    g.set_f(f)
    return g


def _case(nx, ny, seed, **kw):
    rng = np.random.default_rng(seed)
    c = Case(nx, ny, theta=rng.uniform(np.deg2rad(20), np.deg2rad(160), (ny, nx)), precision=32, **kw)
    rho = I.droplet_field(nx, ny, [(nx * 0.3, ny * 0.35, 0), (nx * 0.75, ny * 0.3, 1)], c.rho_v, c.rho_l)
    return c, I.random_distributions(rho, seed, walls=c.walls)


@pytest.mark.parametrize("nx,ny", SIZES)
@pytest.mark.parametrize("name", list(MODELS))
def test_tile_and_ring_kernels_give_the_same_bits(name, nx, ny, monkeypatch):
    c, f = _case(nx, ny, nx + ny, **MODELS[name])
    out = []
    for ring in (False, True):
        with _context(c, f, monkeypatch, ring) as g:
            g.step(7)  # two launches of two steps and three of one where both forms exist
            out.append((g.f(), g.status()))
    c.orc.close()
    assert np.array_equal(out[0][0], out[1][0])
    assert out[0][1] == out[1][1] == 0


@pytest.mark.parametrize("nx,ny", [(128, 8300), (72, 30001)])
def test_narrow_domains_above_2_20_nodes(nx, ny, monkeypatch):
    """Tiles of six rows (the second: a size at which wide domains take the ring)."""
    c, f = _case(nx, ny, 3, tau=0.8)
    out = []
    for ring in (False, True):
        with _context(c, f, monkeypatch, ring) as g:
            g.step(3)
            out.append(g.f())
    c.orc.close()
    assert np.array_equal(out[0], out[1])


@pytest.mark.parametrize("rho", [2.0**-125, 2.0**-126, 0.9 * 2.0**-126, 2.0**-127, 1.001 * 2.0**-128])
@pytest.mark.parametrize("nx,ny", [(64, 12), (400, 200), (1024, 1030)])
def test_subnormal_densities(nx, ny, rho, monkeypatch):
    """A uniform vapour of a density whose reciprocal is finite stays at rest (the
    three sizes: two steps per launch, tiles of four and of six rows)."""
    c, _ = _case(nx, ny, 1, walls=False, tau=0.9)
    f = rho * np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)[:, None, None] * np.ones((9, ny, nx))
    out = []
    for ring in (False, True):
        with _context(c, f, monkeypatch, ring) as g:
            g.step(5)
            out.append((g.f(), g.status()))
    c.orc.close()
    assert np.array_equal(out[0][0], out[1][0]) and out[0][0].min() > 0
    assert out[0][1] == out[1][1] == 0


@pytest.mark.parametrize("y,x", [(1, 0), (3, 63), (4, 64), (8, 67)])
def test_tile_kernel_flags_an_unstable_node(y, x, monkeypatch):
    """A density of 0 in the first and last row and column of tiles."""
    c, f = _case(68, 10, 5)
    f[:, y, x] = 0.0
    with _context(c, f, monkeypatch, False) as g:
        g.step(1)
        assert g.status() == L.LBM_EUNSTABLE
    c.orc.close()


def test_state_alternates_between_the_two_arrays():
    """n steps leave the state in array n % 2, however many a launch makes, and
    stability checks fall due after every check_every-th step."""
    torch = pytest.importorskip("torch")
    c, f = _case(72, 20, 9)
    c.params.check_every = 6
    nbytes = L.lbm_required_state_bytes(c.nx, c.ny, 32)
    for stream in (None, torch.cuda.Stream()):
        buf = torch.zeros((2, 9, c.ny, c.nx), dtype=torch.float32, device="cuda")
        ctx = L.lbm_create_with_buffer(c.nx, c.ny, c.geos, c.T, c.tau, buf.data_ptr(), nbytes, c.theta, True, c.params,
                                       stream)
        L.lbm_set_f(ctx, f)
        done = 0
        for n in (1, 2, 3, 4, 5, 8, 13, 70):
            L.lbm_step(ctx, n)
            done += n
            got = L.lbm_get_f(ctx)
            assert np.array_equal(buf[done % 2].cpu().numpy(), got.astype(np.float32))
        assert L.lbm_get_info(ctx).steps_done == done
        bad = f.copy()
        bad[:, 9, 9] = np.nan
        L.lbm_set_f(ctx, bad)
        with pytest.raises(L.LbmError) as e:
            L.lbm_step(ctx, 20)
        assert e.value.status == L.LBM_EUNSTABLE
        if stream is None:
            assert L.lbm_get_info(ctx).steps_done == done + 6 - done % 6
        L.lbm_destroy(ctx)
    c.orc.close()
