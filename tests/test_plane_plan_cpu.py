"""The plane pass transforms its columns with the plan that the y axis's twiddle table is
built for, also where that plan is not the rows': with another plan put in for a length,
its columns follow, or the fields would come out wrong without an error."""
import subprocess

SOURCE = r"""
#include "fft_core.cuh"
namespace brahms {
template <>
struct ColPlan<48> : Plan<48, 24, 2, 24, 2> {};
}
#include "plane.cuh"
using P = brahms::PlaneColumnPlan<48>;
static_assert(P::N == 48 && P::E == 24 && P::NP == 2 && P::r(0) == 24 && P::r(1) == 2, "the y axis's plan");
static_assert(brahms::PlaneColumnPlan<32>::E == brahms::AxisPlan<32, 1>::E, "the y axis's plan");
"""


def test_columns_take_the_plan_of_the_y_axis(tmp_path):
    from paper_2609_08384_gb300 import build
    (tmp_path / "plan.cu").write_text(SOURCE)
    r = subprocess.run([build._nvcc(), *build.FLAGS, *build.ARCH, "-c", str(tmp_path / "plan.cu"), "-o", str(tmp_path / "plan.o")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
