"""The kernels compiled for two CTAs an SM (M = 256 at d2 = 8) around the most groups that run as one-warp
CTAs: the first step's groups depend on their index alone, and later steps match the oracle."""
import numpy as np
import pytest

from paper_1203_2394_gb300 import workloads
from tests import test_gpu_step

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

FEW = 8 * 152


@pytest.mark.parametrize("kind", ["la", "std"])
def test_first_step_on_both_sides(kind):
    from paper_1203_2394_gb300 import dpf
    spec = workloads.make_model("growth_clg10", 0)
    model = dpf.Model.from_spec(spec, dpf.DPF_F32)
    y = workloads.simulate(spec, 1, 0)[1][0].astype(np.float32)
    fs = []
    for n in (FEW, FEW + 1):
        f = (dpf.Filter(model, spec.d1, spec.d2, n, 256, 4, 3) if kind == "la" else
             dpf.StandardDPF(model, spec.d1, spec.d2, n, 256, 3))
        f.step(y)
        fs.append(f)
    for name in ("lw", "lwhat", "xbb") if kind == "la" else ("lw", "x", "lq"):
        np.testing.assert_array_equal(fs[0].read(name), fs[1].read(name)[:FEW], err_msg=name)


def test_steps_of_full_ctas():
    test_gpu_step.test_fp32_teacher_forced(("growth_clg10", 2, FEW + 1, 256, 4, 3))
