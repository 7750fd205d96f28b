"""Wide filters (d2 = 56) of different models stepped at once on streams of their own.

Their block kernels and the learned wide pass read the model from one constant bank, which is
filled before the launches that read it: each filter's results must be those of its run alone,
bit for bit, whichever form the step takes (two threads a particle, the block form on the CUDA
cores, the learned pass), and so must a captured run of a batch beside them.
"""
import numpy as np
import pytest

from paper_1203_2394_gb300 import workloads
from tests.test_gpu_amortised_wide import _prop

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

N, M, L, T = 608, 128, 8, 6


def _filter(seed, form, stream=None):
    from paper_1203_2394_gb300 import dpf
    spec = workloads.make_model("growth_clg64", seed)
    f = dpf.Filter(dpf.Model.from_spec(spec, dpf.DPF_F32), spec.d1, spec.d2, N, M, L, 5 + seed, stream=stream)
    f.set_tensor_cores(form != "block")
    p = None
    if form == "learned":
        p, _ = _prop(spec, 0.1)
        f.set_proposal(p)
    ys = torch.from_numpy(workloads.simulate(spec, T, seed)[1].astype(np.float32)).cuda()
    out = torch.zeros((T, f.d + 1), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    return f, p, ys, out


def _step(run, t):
    f, _, ys, out = run
    f.step_device(ys[t].data_ptr(), out[t].data_ptr(), out[t].data_ptr() + 8 * f.d)


@pytest.mark.parametrize("form", ["pair", "block", "learned"])
def test_filters_of_different_models_on_two_streams(form):
    alone = []
    for seed in (0, 3):
        run = _filter(seed, form)
        for t in range(T):
            _step(run, t)
        run[0].sync()
        alone.append(run[3].cpu().numpy())
    assert not np.array_equal(alone[0], alone[1])
    streams = [torch.cuda.Stream() for _ in range(2)]
    runs = [_filter(seed, form, s.cuda_stream) for seed, s in zip((0, 3), streams)]
    for t in range(T):
        for run in runs:
            _step(run, t)
    for run, ref in zip(runs, alone):
        run[0].sync()
        np.testing.assert_array_equal(run[3].cpu().numpy(), ref)


def test_captured_batch_beside_a_filter():
    from paper_1203_2394_gb300 import dpf
    specs = [workloads.make_model("growth_clg64", s) for s in (1, 2)]
    ys = np.stack([workloads.simulate(s, T, 4)[1] for s in specs], 1).astype(np.float32)
    ysd = torch.from_numpy(ys).cuda()

    def batch(stream):
        b = dpf.Batch([dpf.Model.from_spec(s, dpf.DPF_F32) for s in specs], [8, 8], [N, N], [100, M], L, [3, 4],
                      stream=stream)
        means = torch.zeros((T, 2, 64), dtype=torch.float64, device="cuda")
        logz = torch.zeros((T, 2), dtype=torch.float64, device="cuda")
        return b, means, logz

    b, means, logz = batch(None)
    b.run_device(ysd.data_ptr(), T, means.data_ptr(), logz.data_ptr())
    ref = means.cpu().numpy(), logz.cpu().numpy()
    run = _filter(0, "block")
    for t in range(T):
        _step(run, t)
    run[0].sync()
    alone = run[3].cpu().numpy()
    streams = [torch.cuda.Stream() for _ in range(2)]
    b, means, logz = batch(streams[0].cuda_stream)
    run = _filter(0, "block", streams[1].cuda_stream)
    for t in range(T):
        _step(run, t)
    b.run_device(ysd.data_ptr(), T, means.data_ptr(), logz.data_ptr())
    run[0].sync()
    np.testing.assert_array_equal(means.cpu().numpy(), ref[0])
    np.testing.assert_array_equal(logz.cpu().numpy(), ref[1])
    np.testing.assert_array_equal(run[3].cpu().numpy(), alone)
