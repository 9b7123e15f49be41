"""Every transform length on every axis, against numpy's FP64 transform.

The shapes put each supported length on the x (row), y and tau (column) plans,
with the other axes short.  Tolerance of one transform: an FP32 transform of
N points loses at most a few units of roundoff (6e-8) per radix-2 level in the
mean square, so 4 x 6e-8 x sqrt(log2 N) relative L2.  Twenty round trips may
change the energy by 1e-8 each (a rounding bias in the moduli of single-float
twiddles changes it by 1e-7 each).
"""
import math

import numpy as np
import pytest

from paper_2609_08384_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

LENGTHS = [2, 4, 8, 16, 32, 64, 128, 256, 512, 1024, 2048, 4096, 6, 12, 24, 48, 96, 192, 384, 768]


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_08384_gb300 import build
    build.build()


def _solver(nx, ny, nt):
    import paper_2609_08384_gb300 as br
    g = wl.Grid(nx, ny, nt, 3e-6, 3e-6, 3e-14)
    return br.Solver(g, wl.shg_fields(), wl.D_EFF, 0.0)


@pytest.mark.parametrize("n", LENGTHS)
@pytest.mark.parametrize("axis", ["x", "y", "tau"])
def test_transform_of_every_length(n, axis):
    nx, ny, nt = {"x": (n, 6, 4), "y": (24, n, 4), "tau": (24, 6, n)}[axis]
    rng = np.random.default_rng(wl.SEED_BASE + n)
    a = [(rng.standard_normal((nt, ny, nx)) + 1j * rng.standard_normal((nt, ny, nx))).astype(np.complex64)
         for _ in range(2)]
    a[1][:] = 0
    a[1][nt // 2, ny - 1, (3 * nx) // 4] = 1.0  # an impulse: every output position and phase
    s = _solver(nx, ny, nt)
    s.set_fields(a)
    s.transform(-1)
    got = s.get_fields()
    tol = 4 * 6e-8 * math.sqrt(math.log2(nx * ny * nt))
    for f in range(2):
        ref = np.fft.fftn(a[f].astype(np.complex128))
        assert np.linalg.norm(got[f] - ref) / np.linalg.norm(ref) < tol
    s.transform(1)
    back = s.get_fields()
    for f in range(2):
        assert np.linalg.norm(back[f] - a[f]) / np.linalg.norm(a[f]) < 2 * tol
    s.close()


@pytest.mark.parametrize("shape", [(512, 24, 16), (32, 384, 8), (16, 64, 256), (96, 32, 192), (128, 48, 32)],
                         ids=lambda s: "x".join(map(str, s)))
def test_round_trips_keep_the_energy(shape):
    rng = np.random.default_rng(wl.SEED_BASE + 1)
    nx, ny, nt = shape
    z = (rng.standard_normal((nt, ny, nx)) + 1j * rng.standard_normal((nt, ny, nx))).astype(np.complex64)
    s = _solver(nx, ny, nt)
    s.set_fields([z, np.conj(z)])
    e0, _ = s.energy()
    for _ in range(20):
        s.transform(-1)
        s.transform(1)
    e1, _ = s.energy()
    assert np.all(np.abs(e1 / e0 - 1) < 20 * 1e-8)
    s.close()
