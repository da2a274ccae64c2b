"""lbm_round.cuh against IEEE division and square root, bit for bit (numpy's float32
operations round correctly): every significand of divisors and arguments, the
divisors for which the corrected reciprocal is not the rounded one, and operands
over the whole range of single precision."""
import ctypes
import subprocess

import numpy as np
import pytest

from paper_1501_05430_gb300 import build as B

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SRC = r"""
#include "lbm_round.cuh"
using namespace lbm_round;
struct Split { float h, l; };
__device__ bool plain(F2 b) { return b.v.x >= 0x1p-40f && b.v.x <= 0x1p40f && b.v.y >= 0x1p-40f && b.v.y <= 0x1p40f; }
__global__ void k(int what, const float2 *a, const float2 *b, float2 *q, size_t n, Split z) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const F2 u = {a[i]}, w = {make_float2(a[i].y, a[i].x)}, d = {b[i]};
  F2 x = u, y = u;
  if (what == 0) q[i] = plain(d) && in_range(u, u) ? Reciprocal(d).under(u).v : (u / d).v;
  if (what == 1) quotients(u, w, d, plain(d), x, y), q[i] = x.v;
  if (what == 2) quotients(w, u, d, plain(d), x, y), q[i] = y.v;
  if (what == 3) q[i] = u.v.x >= 0.0f && u.v.y >= 0.0f && in_range(u, u) ? root0_in_range(u).v : root0(u).v;
  if (what == 4) q[i] = div_const(u, z.h, z.l).v;
  if (what == 5) q[i] = make_float2(quot(u.v.x, d.v.x, 1.0f / d.v.x), quot(u.v.y, d.v.y, 1.0f / d.v.y));
  if (what == 103) q[i] = make_float2(over<3>(u.v.x), over<3>(u.v.y));
  if (what == 106) q[i] = make_float2(over<6>(u.v.x), over<6>(u.v.y));
  if (what == 109) q[i] = make_float2(over<9>(u.v.x), over<9>(u.v.y));
  if (what == 112) q[i] = make_float2(over<12>(u.v.x), over<12>(u.v.y));
  if (what == 136) q[i] = make_float2(over<36>(u.v.x), over<36>(u.v.y));
}
// numbers of the bit patterns [u0, u1) whose corrected reciprocal or root is not the rounded one
__global__ void k_count(unsigned u0, unsigned u1, unsigned *bad) {
  for (unsigned u = u0 + blockIdx.x * blockDim.x + threadIdx.x; u < u1; u += gridDim.x * blockDim.x) {
    const float b = __uint_as_float(u), s = __uint_as_float(u - (40u << 23));
    if (Reciprocal(both(b)).y.v.x != 1.0f / b) atomicAdd(bad, 1u);
    if (root0_in_range(both(b)).v.x != sqrtf(b)) atomicAdd(bad + 1, 1u);
    if (root0_in_range(both(s)).v.y != sqrtf(s)) atomicAdd(bad + 2, 1u);
  }
}
extern "C" int count(unsigned u0, unsigned u1, void *bad) {
  k_count<<<1520, 256>>>(u0, u1, (unsigned *)bad);
  return cudaDeviceSynchronize();
}
extern "C" int run(int what, const void *a, const void *b, void *q, size_t n, float d) {
  Split z = {1.0f, 0.0f};
  const_reciprocal(d, &z.h, &z.l);
  k<<<(unsigned)((n + 255) / 256), 256>>>(what, (const float2 *)a, (const float2 *)b, (float2 *)q, n, z);
  return cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    d = tmp_path_factory.mktemp("rounding")
    src, lib = str(d / "r.cu"), str(d / "r.so")
    with open(src, "w") as h:
        h.write(SRC)
    subprocess.run([B._nvcc()] + B.ARCH + ["-O3", "-std=c++17", "-fmad=false", "-shared", "-Xcompiler", "-fPIC", "-I", B.CSRC,
                                           src, "-o", lib], check=True)
    so = ctypes.CDLL(lib)
    fn = so.run
    so.count.argtypes = [ctypes.c_uint, ctypes.c_uint, ctypes.c_void_p]
    fn.argtypes = [ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_size_t, ctypes.c_float]

    def call(what, a, b=None, d=1.0):
        ta = torch.from_numpy(a).cuda()
        tb = ta if b is None else torch.from_numpy(b).cuda()
        tq = torch.empty_like(ta)
        torch.cuda.synchronize()
        assert a.size % 2 == 0
        assert fn(what, ta.data_ptr(), tb.data_ptr(), tq.data_ptr(), a.size // 2, d) == 0
        return tq.cpu().numpy()

    call.count = so.count
    return call


def _same(got, want):
    nan = np.isnan(want)
    assert np.array_equal(np.isnan(got), nan)
    bad = (got != want) & ~nan
    assert not bad.any(), (np.flatnonzero(bad)[:4], got[bad][:4], want[bad][:4])


def test_every_reciprocal_and_square_root_in_range(run):
    """All numbers of [2^-40, 2^40], and for the root those of [2^-80, 2^40]."""
    bad = torch.zeros(3, dtype=torch.int32, device="cuda")
    lo, hi = ((127 + e) << 23 for e in (-40, 40))
    torch.cuda.synchronize()
    assert run.count(lo, hi + 1, bad.data_ptr()) == 0
    assert bad.tolist() == [0, 0, 0]


SIGNIFICANDS = (np.arange(1 << 23, dtype=np.uint32) | np.uint32(0x3F800000)).view(np.float32)  # [1, 2)
ALL_ONES = SIGNIFICANDS[-1:]


def _quotients(run, a, b):
    with np.errstate(all="ignore"):
        want = a / b
    for what in (0, 1, 2):
        _same(run(what, a, b), want)


@pytest.mark.parametrize("scale", [1.0, 2.0**-13, 2.0**9])
def test_every_divisor(run, scale):
    b = (SIGNIFICANDS * np.float32(scale)).astype(np.float32)
    rng = np.random.default_rng(1)
    for a in (np.ones_like(b), rng.permutation(SIGNIFICANDS), -rng.permutation(SIGNIFICANDS) * np.float32(3e-5),
              np.zeros_like(b), -np.zeros_like(b)):
        _quotients(run, a.astype(np.float32), b)


@pytest.mark.parametrize("power", [0, -7, 11])
def test_every_dividend_of_the_divisor_with_all_bits_set(run, power):
    b = np.repeat(ALL_ONES * np.float32(2.0**power), SIGNIFICANDS.size)
    _quotients(run, SIGNIFICANDS.copy(), b)


def _any_float(rng, n):
    return rng.integers(0, 1 << 32, n, dtype=np.uint32).view(np.float32)


EDGES = np.array([0.0, -0.0, 1e-45, -1e-45, 1e-40, 2.0**-126, 2.0**-125, 2.0**-102, 2.0**-80, 2.0**-79, -2.0**-81, 2.0**-41,
                  2.0**-40, 2.0**40, 2.0**41, -2.0**40, 2.0**126, 2.0**127, 3.4e38, np.inf, -np.inf, np.nan, 1.0, -1.0, 3.0,
                  np.nextafter(np.float32(2.0**-80), np.float32(0)), np.nextafter(np.float32(2.0**40), np.float32(np.inf))],
                 dtype=np.float32)


def test_quotients_over_the_whole_range(run):
    rng = np.random.default_rng(2)
    a, b = (v.ravel() for v in np.meshgrid(EDGES, EDGES))
    n = a.size // 2 * 2
    _quotients(run, a[:n].copy(), b[:n].copy())
    _quotients(run, a[1:n - 1].copy(), b[1:n - 1].copy())  # (other neighbours in the pair)
    _quotients(run, _any_float(rng, 1 << 22), _any_float(rng, 1 << 22))
    near = lambda: (rng.permutation(SIGNIFICANDS)[:1 << 22] * 2.0 ** rng.integers(-24, 24, 1 << 22)).astype(np.float32)  # noqa: E731
    for _ in range(8):
        _quotients(run, near() * rng.choice(np.array([-1, 1], np.float32), 1 << 22), near())


def test_every_square_root(run):
    for scale in (1.0, 2.0, 2.0**-20, 2.0**-31, 2.0**38):
        x = (SIGNIFICANDS * np.float32(scale)).astype(np.float32)
        _same(run(3, x), np.sqrt(x))
    rng = np.random.default_rng(3)
    for x in (EDGES[: EDGES.size // 2 * 2].copy(), EDGES[1:EDGES.size // 2 * 2 - 1].copy(), _any_float(rng, 1 << 22)):
        _same(run(3, x), np.sqrt(np.where(x > 0, x, np.float32(0))))


@pytest.mark.parametrize("d", [3, 6, 9, 12, 36])
def test_every_quotient_by_a_small_integer(run, d):
    for scale in (1.0, -(2.0**-60), 2.0**-94, 2.0**120):
        x = (SIGNIFICANDS * np.float32(scale)).astype(np.float32)
        _same(run(4, x, d=float(d)), x / np.float32(d))
        _same(run(100 + d, x), x / np.float32(d))


def test_quotients_that_share_a_rounded_reciprocal(run):
    rng = np.random.default_rng(4)
    for scale in (1.0, 2.0**-11, 2.0**6):
        b = (SIGNIFICANDS * np.float32(scale)).astype(np.float32)
        for a in (np.ones_like(b), rng.permutation(SIGNIFICANDS), -rng.permutation(SIGNIFICANDS) * np.float32(1e-29)):
            _same(run(5, a, b), a / b)
    _same(run(5, SIGNIFICANDS.copy(), np.repeat(ALL_ONES, SIGNIFICANDS.size)), SIGNIFICANDS / ALL_ONES)
