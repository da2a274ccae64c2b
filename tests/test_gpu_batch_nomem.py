"""A batch whose list of tiles gets no device memory runs the persistent kernel
instead, and one without memory for its table of angles measures one by one: the
library linked anew from its objects, with a cudaMalloc that refuses allocations of
one size."""
import os
import subprocess

import numpy as np
import pytest

from paper_1501_05430_gb300 import build as B
from paper_1501_05430_gb300 import lbm as L

pytestmark = pytest.mark.gpu

FAKE = """
#include <stddef.h>
static size_t refused;
int __real_cudaMalloc(void **p, size_t n);
int __wrap_cudaMalloc(void **p, size_t n) { return n == refused ? 2 : __real_cudaMalloc(p, n); }
void refuse_allocations_of(size_t n) { refused = n; }
"""


@pytest.fixture
def refuse(tmp_path, monkeypatch):
    src, obj, lib = (str(tmp_path / n) for n in ("fake.c", "fake.o", "liblbm_fake.so"))
    L.load()  # (builds the objects)
    with open(src, "w") as h:
        h.write(FAKE)
    subprocess.run(["gcc", "-O1", "-fPIC", "-c", src, "-o", obj], check=True)
    objs = [os.path.join(B.OUT_DIR, u.replace(".cu", ".o")) for u in B.UNITS]
    subprocess.run([B._nvcc()] + B.ARCH + ["-shared", "-Xlinker", "--wrap=cudaMalloc", "-o", lib, obj] + objs, check=True)
    monkeypatch.setattr(L, "_lib", None)
    monkeypatch.setattr(L._build, "LIB", lib)
    import ctypes

    fn = L.load(rebuild=False).refuse_allocations_of
    fn.argtypes = [ctypes.c_size_t]
    return fn


def _batch(**cfg):
    nx, ny = 64, 32
    eos = L.carnahan_starling()
    T = 0.8 * L.lbm_eos_critical(eos)[0]
    rv, rl = L.lbm_coexistence(eos, T)
    rho = np.full((ny, nx), rv)
    rho[1:8, 20:40] = rl
    d = dict(nx=nx, ny=ny, eos=eos, T=T, tau=1.0, theta=np.full((ny, nx), 1.2))
    b = L.LbmBatch([d, d], L.lbm_batch_config_default(**cfg))
    for inst in b.instances:
        inst.set_rho(rho)
    return b


def test_no_memory_for_the_tiles(refuse):
    with _batch() as b:
        plan = b.plan()
        assert plan["smem_bytes"] == 0  # tiles
        b.step(6)
        want = b[1].f()
    refuse(plan["items"] * 16)
    with _batch() as made, _batch(stages=3) as switched, _batch(stages=3) as tuned:
        switched.set_config(L.lbm_batch_config_default())
        tuned.autotune(trial_steps=2)
        for b in (made, switched, tuned):
            assert b.plan()["smem_bytes"] > 0
            b.step(6)
            assert b.status()[0] == 0 and np.array_equal(b[1].f(), want)


def test_no_memory_for_the_table_of_angles(refuse):
    with _batch() as b, _batch() as c:
        b.step(6)
        c.step(6)
        want = b.contact_angles(0)
        refuse(2 * 128)  # (two entries of 64 bytes an instance)
        got = c.contact_angles(0)
        assert all(np.array_equal(x, y, equal_nan=True) for x, y in zip(want, got))
