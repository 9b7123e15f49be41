"""A device buffer that ends before its last point, or runs on into another
allocation, is refused by the host before any kernel or copy touches it, and the
context stays usable."""
import ctypes

import pytest

from paper_2609_08384_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
NX, NY, NT = 64, 64, 64
HALF = 1 << 20  # bytes; a field of complex64 takes 2 << 20


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_08384_gb300 import build
    build.build()


@pytest.fixture
def short():
    """A function that gives the address of HALF bytes at the end of an allocation:
    alone (no memory behind it) or followed by another allocation."""
    torch.zeros(1, device="cuda")
    cu = ctypes.CDLL("libcuda.so.1")
    u64, size_t = ctypes.c_uint64, ctypes.c_size_t
    held = []

    def find(alone):
        for size in (2 << 20, 2 << 20, 6 << 20, 6 << 20, 34 << 20, 130 << 20):
            p, base, length = u64(), u64(), size_t()
            assert cu.cuMemAlloc_v2(ctypes.byref(p), size_t(size)) == 0
            held.append(p)
        for p in reversed(held):
            assert cu.cuMemGetAddressRange_v2(ctypes.byref(base), ctypes.byref(length), p) == 0
            end = base.value + length.value
            if (cu.cuMemGetAddressRange_v2(ctypes.byref(base), ctypes.byref(length), u64(end)) != 0) == alone:
                return end - HALF
        pytest.skip("no such allocation")

    yield find
    torch.cuda.synchronize()
    for p in held:
        assert cu.cuMemFree_v2(p) == 0


@pytest.mark.parametrize("dtype", ["complex64", "complex128"])
@pytest.mark.parametrize("which", [0, 2])
@pytest.mark.parametrize("alone", [True, False])
def test_solver_refuses_a_short_buffer(short, dtype, which, alone):
    import paper_2609_08384_gb300 as br
    lib = br.load()
    s = br.Solver(wl.Grid(NX, NY, NT, 3e-6, 3e-6, 3e-14),
                  [wl.FieldParams(1064e-9, 2.15), wl.FieldParams(1450e-9, 2.14), wl.FieldParams(3997e-9, 2.08)], wl.D_EFF, 0.0)
    dt = getattr(torch, dtype)
    code = br.BRAHMS_C64 if dtype == "complex64" else br.BRAHMS_C128
    good = [torch.full((NT, NY, NX), 1.0 + f, dtype=dt, device="cuda") for f in range(3)]
    out = [torch.zeros_like(t) for t in good]
    s.set_fields(good)
    ptrs = [t.data_ptr() for t in good]
    ptrs[which] = end = short(alone)
    assert lib.brahms_set_fields(s.ctx, br._ptr_array(ptrs), code, 1) == br.BRAHMS_E_CUDA
    ptrs = [t.data_ptr() for t in out]
    ptrs[which] = end
    assert lib.brahms_get_fields(s.ctx, br._ptr_array(ptrs), code, 1) == br.BRAHMS_E_CUDA
    for a, b in zip(s.get_fields(out=out, on_device=True), good):  # the fields set before are still there
        assert torch.equal(a, b)
    s.close()


@pytest.mark.parametrize("alone", [True, False])
def test_batch_refuses_a_short_buffer(short, alone):
    import paper_2609_08384_gb300 as br
    lib = br.load()
    b = br.Batch()
    b.add(wl.Grid(NX, NY, NT, 3e-6, 3e-6, 3e-14), [wl.FieldParams(532e-9, 2.234), wl.FieldParams(1064e-9, 2.156)], wl.D_EFF, 0.0,
          1, 1e-5)
    good = [torch.full((NT, NY, NX), 1.0 + f, dtype=torch.complex64, device="cuda") for f in range(2)]
    b.set_fields(0, good)
    end = short(alone)
    for which in range(2):
        ptrs = [t.data_ptr() for t in good]
        ptrs[which] = end
        assert lib.brahms_batch_set_fields(b.h, 0, br._ptr_array(ptrs), br.BRAHMS_C64, 1) == br.BRAHMS_E_CUDA
        assert lib.brahms_batch_get_fields(b.h, 0, br._ptr_array(ptrs), br.BRAHMS_C64, 1) == br.BRAHMS_E_CUDA
    for x, y in zip(b.get_fields(0, on_device=True), good):
        assert torch.equal(x, y)
    b.close()
