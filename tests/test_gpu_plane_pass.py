"""The plane pass (y-inverse, x-pass and y-forward of a step in one kernel, small
planes) against the separate passes, which the per-field streams keep to: the
arithmetic is the same, so the fields agree bit for bit.  Planes whose rows or
columns do not fill the CTA's 256 threads, one or several rounds of rows and
columns, single-pass transforms, one plane and many.  And grids
without a time axis, whose linear step is one pass along y, against the oracle."""
import numpy as np
import pytest

import oracle
from paper_2609_08384_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PLANES = [(16, 8), (16, 64), (24, 12), (24, 64), (32, 32), (32, 48), (48, 8), (48, 32), (64, 16), (64, 24)]


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_08384_gb300 import build
    build.build()


def _problem(nx, ny, nt, nf):
    g = wl.Grid(nx, ny, nt, 6e-6, 5e-6, 4e-14)
    fields = [wl.FieldParams(1064e-9, 2.15, delta=1e-10, k2=2e-25, rho=2e-3, alpha=10.0),
              wl.FieldParams(1450e-9, 2.14, k2=1e-25), wl.FieldParams(3997e-9, 2.08, delta=-1e-10, rho=1e-3)][:nf]
    rng = np.random.default_rng(wl.SEED_BASE + nx + 7 * ny + nt)
    a = [(4e7 * (rng.standard_normal((nt, ny, nx)) + 1j * rng.standard_normal((nt, ny, nx)))).astype(np.complex64)
         for _ in range(nf)]
    return g, fields, a


@pytest.mark.parametrize("nt,nf", [(2, 3), (6, 2), (48, 3), (256, 2)])
@pytest.mark.parametrize("plane", PLANES, ids=lambda s: "x".join(map(str, s)))
def test_plane_pass_gives_the_bits_of_the_separate_passes(plane, nt, nf):
    import paper_2609_08384_gb300 as br
    g, fields, a = _problem(*plane, nt, nf)
    profile = np.linspace(-300.0, 200.0, 7)
    got = []
    for streams in (0, 1):
        s = br.Solver(g, fields, wl.D_EFF, 40.0)
        s.set_option(br.BRAHMS_OPT_FIELD_STREAMS, streams)
        s.set_fields(a)
        s.set_dk_profile(profile)
        s.propagate(4, 1e-5)
        s.propagate(1, 1e-5)  # a call whose first and last x-pass belong to one step
        s.propagate(5, 1e-5)
        got.append(s.get_fields())
        s.close()
    for x, y in zip(*got):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("plane,nf", [((32, 24), 2), ((48, 16), 3), ((6, 64), 2), ((2, 512), 3), ((128, 96), 2), ((12, 768), 2), ((4, 2048), 2), ((24, 2), 3)])
def test_grid_without_a_time_axis_matches_the_oracle(plane, nf):
    import paper_2609_08384_gb300 as br
    g, fields, a = _problem(*plane, 1, nf)
    s = br.Solver(g, fields, wl.D_EFF, 40.0)
    s.set_fields(a)
    s.propagate(6, 1e-5)
    got = s.get_fields()
    ref, _ = oracle.propagate(oracle.make_problem(g, fields, wl.D_EFF), [x.astype(np.complex128) for x in a], 6, 1e-5, 40.0)
    for x, r in zip(got, ref):
        assert np.linalg.norm(x - r) / np.linalg.norm(r) < 1e-4  # FP32 fields against FP64, the bar of the parity tests
    s.close()
