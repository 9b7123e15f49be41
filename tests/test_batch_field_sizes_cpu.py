"""Batch.set_fields looks at the number of points before it hands a pointer on: a
field shorter than the instance's grid is refused, on the host, whatever its shape."""
import numpy as np
import pytest

import paper_2609_08384_gb300 as br

torch = pytest.importorskip("torch")


class _Calls:
    def __init__(self):
        self.made = 0

    def brahms_batch_set_fields(self, *a):
        self.made += 1
        return br.BRAHMS_OK


@pytest.fixture
def batch(monkeypatch):
    calls = _Calls()
    monkeypatch.setattr(br, "load", lambda path=None: calls)
    b = object.__new__(br.Batch)
    b.h = None
    b.shapes = [(4, 6, 8), (2, 2, 2)]
    return b, calls


@pytest.mark.parametrize("make", [lambda n: np.zeros(n, np.complex64), lambda n: torch.zeros(n, dtype=torch.complex64)],
                         ids=["numpy", "torch"])
def test_short_fields_are_refused(batch, make):
    b, calls = batch
    for which in range(2):
        sizes = [192, 192]
        sizes[which] = 191
        with pytest.raises(ValueError):
            b.set_fields(0, [make(n) for n in sizes])
    assert calls.made == 0
    b.set_fields(0, [make(192), make(192)])
    b.set_fields(1, [make(192), make(8)])  # more than the grid needs is taken, as before
    b.set_fields(0, [make(192).reshape(4, 6, 8), make(192).reshape(4, 6, 8)])
    assert calls.made == 3
