"""Bringing fields in and handing them out: device buffers at any alignment, one
buffer for several fields, and buffers that overlap give exactly what copies one
after another give, and the non-finite check sees every point."""
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


def _solver(shape):
    import paper_2609_08384_gb300 as br
    nx, ny, nt = shape
    g = wl.Grid(nx, ny, nt, 3e-6, 3e-6, 3e-14)
    f = [wl.FieldParams(1064e-9, 2.15), wl.FieldParams(1450e-9, 2.14), wl.FieldParams(3997e-9, 2.08)]
    return br.Solver(g, f, wl.D_EFF, 0.0)


@pytest.mark.parametrize("shape", [(2, 1, 1), (6, 2, 2), (24, 6, 8), (64, 48, 96), (2, 512, 384)],
                         ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("shift", [0, 1])
def test_device_buffers_at_any_alignment(shape, shift):
    nx, ny, nt = shape
    n = nx * ny * nt
    s = _solver(shape)
    g = torch.Generator(device="cuda").manual_seed(wl.SEED_BASE)
    raw = [torch.randn(n + 2, dtype=torch.complex64, device="cuda", generator=g) for _ in range(3)]
    a = [r[shift:shift + n].view(nt, ny, nx) for r in raw]  # shift 1: 8 bytes off a 16-byte boundary
    s.set_fields(a)
    out = [torch.zeros(n + 2, dtype=torch.complex64, device="cuda") for _ in range(3)]
    s.get_fields(out=[o[shift:shift + n].view(nt, ny, nx) for o in out], on_device=True)
    for x, o in zip(a, out):
        assert torch.equal(o[shift:shift + n].view(nt, ny, nx), x)
        assert not o[:shift].any() and not o[shift + n:].any()  # nothing beside the field is written
    e, _ = s.energy()
    for f, x in enumerate(a):  # FP32 squares of eight points at a time: within a few roundoffs of the FP64 sum
        ref = float(x.to(torch.complex128).abs().square().sum())
        c = 0.5 * wl.C0 * wl.EPS0 * (2.15, 2.14, 2.08)[f] * 3e-6 * 3e-6 * 3e-14
        assert abs(e[f] / (c * ref) - 1) < 8 * 6e-8
    s.close()


def test_one_buffer_for_all_fields_and_overlapping_outputs():
    shape = (24, 6, 8)
    nx, ny, nt = shape
    n = nx * ny * nt
    s = _solver(shape)
    x = torch.randn(nt, ny, nx, dtype=torch.complex64, device="cuda")
    s.set_fields([x, x, x])
    got = s.get_fields()
    for a in got:
        assert np.array_equal(a, x.cpu().numpy())
    y = [torch.randn(nt, ny, nx, dtype=torch.complex64, device="cuda") for _ in range(3)]
    s.set_fields(y)
    one = torch.zeros(nt, ny, nx, dtype=torch.complex64, device="cuda")
    s.get_fields(out=[one, one, one], on_device=True)
    assert torch.equal(one, y[2])  # the fields go out in order
    s.close()


@pytest.mark.parametrize("where", [0, 1, 2303, 2304 * 2 - 1])
@pytest.mark.parametrize("value", [float("nan"), float("inf")])
def test_non_finite_points_are_seen_wherever_they_are(where, value):
    import paper_2609_08384_gb300 as br
    shape = (24, 24, 8)
    s = _solver(shape)
    x = torch.ones(8, 24, 24, dtype=torch.complex64, device="cuda")
    bad = x.clone()
    bad.view(-1)[where] = value
    with pytest.raises(br.BrahmsError) as e:
        s.set_fields([x, x, bad])
    assert e.value.status == br.BRAHMS_E_ARG
    s.set_fields([x, x, x])  # the context stays usable
    s.close()


@pytest.mark.parametrize("shift", [0, 1])
def test_batch_fields_at_any_alignment(shift):
    import paper_2609_08384_gb300 as br
    b = br.Batch()
    shapes = [(32, 32, 64), (24, 48, 12)]
    f = [wl.FieldParams(532e-9, 2.234), wl.FieldParams(1064e-9, 2.156)]
    a = []
    for i, (nx, ny, nt) in enumerate(shapes):
        b.add(wl.Grid(nx, ny, nt, 3e-6, 3e-6, 3e-14), f, wl.D_EFF, 0.0, 1, 1e-5)
        raw = torch.randn(2, nx * ny * nt + 2, dtype=torch.complex64, device="cuda")
        a.append([raw[k, shift:shift + nx * ny * nt].clone() if not shift else raw[k, 1:1 + nx * ny * nt]
                  for k in range(2)])
        b.set_fields(i, [x.view(nt, ny, nx) for x in a[-1]])
    for i, (nx, ny, nt) in enumerate(shapes):
        for got, x in zip(b.get_fields(i, on_device=True), a[i]):
            assert torch.equal(got.view(-1), x)
        for got, x in zip(b.get_fields(i), a[i]):
            assert np.array_equal(got.reshape(-1), x.cpu().numpy())
    b.close()


@pytest.mark.parametrize("size", [1e-15, 1.0, 3e17])
def test_energy_and_power_of_tiny_and_huge_fields(size):
    """Sums of squares across FP32's range: at 3e17 a point's square fits a float
    and the sums of a thread's points do not."""
    shape = (96, 96, 64)
    nx, ny, nt = shape
    s = _solver(shape)
    x = [size * torch.randn(nt, ny, nx, dtype=torch.complex64, device="cuda") for _ in range(3)]
    s.set_fields(x)
    e, _ = s.energy()
    p, _ = s.diagnostics()
    for f in range(3):
        c = 0.5 * wl.C0 * wl.EPS0 * (2.15, 2.14, 2.08)[f] * 3e-6 * 3e-6
        ref = c * x[f].to(torch.complex128).abs().square().sum((1, 2)).cpu().numpy()
        assert np.allclose(p[f], ref, rtol=4 * 6e-8, atol=0)  # FP32 squares of pairs of points
        assert abs(e[f] / (ref.sum() * 3e-14) - 1) < 8 * 6e-8
    s.close()
