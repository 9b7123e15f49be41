"""The linear step by itself (no coupling) against numpy in FP64, on grids whose
x extent is not a whole number of tau-pass tiles, whose tiles are fewer or more
than one wave of CTAs, and for every tau length that has a kernel of its own.

Tolerance: a step is a forward and an inverse transform, each losing at most
4 x 6e-8 x sqrt(log2 N) relative L2 in FP32 (a few units of roundoff per
radix-2 level in the mean square)."""
import math

import numpy as np
import pytest

from paper_2609_08384_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPES = [(6, 2, 64), (2, 4, 128), (12, 6, 256), (4, 2, 512), (6, 8, 768), (24, 12, 64), (48, 96, 256), (96, 48, 512),
          (24, 64, 128), (16, 6, 384), (12, 8, 192), (24, 4, 96), (32, 128, 64), (64, 24, 768)]


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_08384_gb300 import build
    build.build()


def _reference(g, fields, a, dz, nz):
    kx = 2 * np.pi * np.fft.fftfreq(g.nx, g.dx)
    ky = 2 * np.pi * np.fft.fftfreq(g.ny, g.dy)
    om = 2 * np.pi * np.fft.fftfreq(g.nt, g.dt)
    out = []
    for f, x in zip(fields, a):
        k = 2 * np.pi * f.n / f.lambda_
        p = (np.exp(-1j * dz * (kx**2 / (2 * k) + math.tan(f.rho) * kx))[None, None, :] *
             np.exp(-1j * dz * ky**2 / (2 * k))[None, :, None] *
             np.exp(dz * (-0.5 * f.alpha - 1j * f.delta * om + 0.5j * f.k2 * om**2 - 1j * f.k3 / 6 * om**3))[:, None, None])
        out.append(np.fft.ifftn(np.fft.fftn(x.astype(np.complex128)) * p**nz))
    return out


@pytest.mark.parametrize("nf", [2, 3])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_linear_step_matches_fp64(shape, nf):
    import paper_2609_08384_gb300 as br
    g = wl.Grid(*shape, 5e-6, 7e-6, 4e-14)
    fields = [wl.FieldParams(1064e-9, 2.15, delta=1e-10, k2=2e-25, k3=3e-38, rho=2e-3, alpha=20.0),
              wl.FieldParams(1450e-9, 2.14, k2=1e-25), wl.FieldParams(3997e-9, 2.08, delta=-1e-10, rho=1e-3)][:nf]
    rng = np.random.default_rng(wl.SEED_BASE + shape[0] + shape[2])
    a = [(rng.standard_normal((g.nt, g.ny, g.nx)) + 1j * rng.standard_normal((g.nt, g.ny, g.nx))).astype(np.complex64)
         for _ in range(nf)]
    nz, dz = 2, 2e-5
    s = br.Solver(g, fields, 0.0, 0.0)
    s.set_fields(a)
    s.propagate(nz, dz)
    got = s.get_fields()
    tol = 2 * nz * 4 * 6e-8 * math.sqrt(math.log2(g.npoints))
    for x, r in zip(got, _reference(g, fields, a, dz, nz)):
        assert np.linalg.norm(x - r) / np.linalg.norm(r) < tol
    s.close()


@pytest.mark.parametrize("ny", [2, 4, 6, 8, 12, 16, 24, 32, 48, 64, 96, 128, 192, 256, 384, 512, 768, 1024, 2048, 4096])
def test_cw_linear_step_of_every_y_length(ny):
    """nt = 1: the linear step is one pass along y, whose kernel and twiddle table
    are the tau-pass's."""
    test_linear_step_matches_fp64((24, ny, 1), 3)
