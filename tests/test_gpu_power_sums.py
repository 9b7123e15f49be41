"""Sums of many terms: the power of a uniform field on the largest plane,
32768 pairs of points to a thread, are the number of pairs times the float that one
pair's squares come to, to 2^-40."""
import numpy as np
import pytest

from paper_2609_08384_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_08384_gb300 import build
    build.build()


@pytest.mark.parametrize("value", [1.07551908493042, 1.2352615594863892, 1.507469892501831, 0.75])
def test_power_of_a_uniform_plane(value):
    import paper_2609_08384_gb300 as br
    n, index = 4096, 2.156
    s = br.Solver(wl.Grid(n, n, 1, 1e-6, 1e-6, 1e-14), [wl.FieldParams(532e-9, 2.234), wl.FieldParams(1064e-9, index)], wl.D_EFF, 0.0)
    a = torch.full((1, n, n), value, dtype=torch.complex64, device="cuda")
    s.set_fields([a, a])
    power, _ = s.diagnostics()
    v = np.float64(np.float32(value))
    one = np.float64(np.float32(v * v + np.float64(np.float32(v * v))))  # fma(v, v, v * v), real fields
    expected = 0.5 * wl.C0 * wl.EPS0 * index * 1e-6 * 1e-6 * one * (n * n // 2)
    assert abs(power[1, 0] / expected - 1) < 2.0 ** -40
    s.close()
