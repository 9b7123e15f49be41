"""The linear step's 1/(nx ny nt) on grids whose point count is no power of two.

A field uniform along the axes whose length changes goes through the same modes and
the same table entries of the propagator on a grid of 3 2^k points as on one of 2^k
points, so its energy has to change alike on both.  1/3 as a float is 3.0e-8 off; left
in the constants of P = 1 + E it makes the energy of the first grid grow by 2 * 3.0e-8
(1 - cos phi), 6e-8 on average over phases of the whole circle, in every step.  The
bound is a quarter of that, 2^-26 per step; the transforms' roundings differ from
step to step and mode to mode.
"""
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


def _growth(shape, line):
    import paper_2609_08384_gb300 as br
    nx, ny, nt = shape
    a = line[:, None, None] if nt > 1 else line[None, :, None]
    a = a.expand(nt, ny, nx).contiguous()
    # 1 um cells and 10 fs samples: phases of several turns per 20 um step
    f = [wl.FieldParams(532e-9, 2.2), wl.FieldParams(1064e-9, 2.15, k2=1e-23)]
    s = br.Solver(wl.Grid(nx, ny, nt, 1e-6, 1e-6, 1e-14), f, wl.D_EFF, 0.0)
    s.set_fields([torch.zeros_like(a), a])  # 1 V/m: the coupling does not reach single precision
    e0 = s.energy()[0][1]
    s.propagate(200, 20e-6)
    e1 = s.energy()[0][1]
    s.close()
    return e1 / e0


# pipelined and plain tau-pass, plane pass, cw, a single row of planes
@pytest.mark.parametrize("shape, plain", [((6, 8, 512), (8, 8, 512)), ((96, 64, 128), (64, 64, 128)), ((6, 8, 2048), (8, 8, 2048)),
                                          ((128, 6, 32), (128, 8, 32)), ((24, 16, 256), (32, 16, 256)),
                                          ((6, 1024, 1), (8, 1024, 1)), ((6, 1, 512), (8, 1, 512))], ids=str)
def test_energy_changes_as_on_a_grid_of_a_power_of_two(shape, plain):
    n = shape[2] if shape[2] > 1 else shape[1]
    line = torch.randn(n, dtype=torch.complex64, device="cuda", generator=torch.Generator("cuda").manual_seed(wl.SEED_BASE))
    assert abs(_growth(shape, line) - _growth(plain, line)) < 200 * 2.0 ** -26
