"""The stage factors that the host hands to a map-free x-pass: e^{i Phi} at the start,
middle and end of both half steps, each phase formed and reduced in FP64 and evaluated
in FP64, so that a factor is the nearest float of the exact value."""
import ctypes
import math
import os
import subprocess

import numpy as np
import pytest

SOURCE = r"""
#include "kernels.cuh"
extern "C" int stage_factors(double phiB, double dkB, double phiA, double dkA, double dz, float* out) {
  brahms::XPassArgs a{};
  a.phiB = phiB;
  a.dkB = dkB;
  a.phiA = phiA;
  a.dkA = dkA;
  a.dz = dz;
  brahms::fill_stage_factors(a);
  for (int k = 0; k < brahms::kStageFactors; ++k) {
    out[2 * k] = a.ecoef[k].x;
    out[2 * k + 1] = a.ecoef[k].y;
  }
  return brahms::kStageFactors;
}
"""


@pytest.fixture(scope="module")
def stage_factors(tmp_path_factory):
    from paper_2609_08384_gb300 import build
    lib = build.build()
    d = tmp_path_factory.mktemp("factors")
    (d / "factors.cu").write_text(SOURCE)
    out = os.path.dirname(lib)
    subprocess.run([build._nvcc(), *build.FLAGS, *build.ARCH, "-shared", str(d / "factors.cu"), "-o", str(d / "factors.so"),
                    "-L" + out, "-lbrahms", "-Xlinker", "-rpath=" + out], check=True)
    fn = ctypes.CDLL(str(d / "factors.so")).stage_factors
    fn.argtypes = [ctypes.c_double] * 5 + [ctypes.POINTER(ctypes.c_float)]

    def call(*a):
        v = np.zeros(64, np.float32)
        n = fn(*a, v.ctypes.data_as(ctypes.POINTER(ctypes.c_float)))
        return v[:2 * n:2] + 1j * v[1:2 * n:2]

    return call


@pytest.mark.parametrize("phi_b, dk_b, phi_a, dk_a, dz", [(0.0, 0.0, 0.0, 0.0, 1e-5), (0.3, 20.0, 0.4, -35.0, 1e-5),
                                                          (1234.5, 2e5, -987.25, 1e5, 2e-5), (-3.1, -4.2, -3.1, 7.5, 1.3e-5)])
def test_every_stage_factor_is_the_nearest_float(stage_factors, phi_b, dk_b, phi_a, dk_a, dz):
    phases = [phi_b + dk_b * (0.5 + 0.25 * s) * dz for s in range(3)] + [phi_a + dk_a * 0.25 * s * dz for s in range(3)]
    got = stage_factors(phi_b, dk_b, phi_a, dk_a, dz)
    assert len(got) == 6
    for g, phi in zip(got, phases):
        # half a float's spacing, and FP64's roundings of a phase of this size
        tol = 2.0 ** -25 + 8 * 2.0 ** -52 * (1 + abs(phi))
        assert abs(g.real - math.cos(phi)) <= tol and abs(g.imag - math.sin(phi)) <= tol
