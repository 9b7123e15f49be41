"""Turns of a transform that nothing takes back (brahms_transform).

The transform of an impulse multiplies its amplitude by a product of the transform's
constants.  Over 4096 random amplitudes (the other axis) the roundings average out and
that product shows: held as hi + lo floats it is e^{-/+ 2 pi i p k / n} to FP64's eye,
held as single floats it is off by up to 6e-8 per turn.  Bound: a turn rounds by less
than 2^-24 rms, the other axis's transform by less than 3 * 2^-24, so their mean over
4096 amplitudes lies within 5 (turns + 4) 2^-24 / sqrt(4096).
"""
import numpy as np
import pytest

from paper_2609_08384_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
MANY = 4096
# turns on a path: between the passes, and inside radix 8, 16 (one), 32 and 24 (two)
# and 6 and 12 (the three-point butterfly)
TURNS = {8: 1, 16: 1, 32: 2, 64: 3, 128: 3, 256: 3, 512: 4, 1024: 5, 2048: 5, 4096: 5, 6: 1, 12: 1, 24: 2, 48: 2, 96: 3, 192: 4,
         384: 4, 768: 5}


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_08384_gb300 import build
    build.build()


@pytest.mark.parametrize("n", sorted(TURNS))
@pytest.mark.parametrize("axis", ["x", "y", "tau"])
def test_the_constants_of_a_single_transform(n, axis):
    import paper_2609_08384_gb300 as br
    nx, ny, nt = {"x": (n, MANY, 1), "y": (MANY, n, 1), "tau": (MANY, 1, n)}[axis]
    s = br.Solver(wl.Grid(nx, ny, nt, 1e-6, 1e-6, 1e-14), [wl.FieldParams(532e-9, 2.2), wl.FieldParams(1064e-9, 2.15)], wl.D_EFF, 0.0)
    g = torch.Generator("cuda").manual_seed(wl.SEED_BASE + n)
    k = torch.arange(n, dtype=torch.float64, device="cuda")
    bound = 5 * (TURNS[n] + 4) * 2.0 ** -24 / np.sqrt(MANY)

    def lines(a):  # [n, MANY]
        return a.view(MANY, n).T if axis == "x" else a.view(n, MANY)

    for direction in (-1, 1):
        where = [1, n // 2 + 1 if n > 2 else 1, n - 1]
        for p in where:
            f = [torch.zeros(nt, ny, nx, dtype=torch.complex64, device="cuda") for _ in range(2)]
            for a in f:
                lines(a)[p] = torch.randn(MANY, dtype=torch.complex64, device="cuda", generator=g)
            s.set_fields(f)
            s.transform(direction)
            for a in s.get_fields(on_device=True):
                v = lines(a).to(torch.complex128)
                ratio = (v @ v[0].conj()) / v[0].abs().square().sum()
                exact = torch.polar(torch.ones_like(k), direction * 2 * np.pi * ((k * p) % n) / n)
                assert float((ratio * exact.conj() - 1).abs().max()) < bound
    s.close()
