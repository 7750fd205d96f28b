"""The bootstrap particle filter's own parts: a particle is its own mean, so "xm" and "zm" are the
particles by coordinate at any time (a fresh handle, after steps, after a restored state), and no
buffer of means is held for them. The paper models' particle filter keeps its means apart.
"""
import numpy as np
import pytest

from paper_1203_2394_gb300 import workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _pf(N, prec):
    from paper_1203_2394_gb300 import dpf
    spec = workloads.make_model("growth_clg10" if prec == dpf.DPF_F32 else "lg4", 0)
    return spec, dpf.ParticleFilter(dpf.Model.from_spec(spec, prec), spec.d1, spec.d2, N, 7)


def _own(f):
    np.testing.assert_array_equal(f.read("xm"), f.read("x").T)
    np.testing.assert_array_equal(f.read("zm"), f.read("z")[:, :, 0])
    assert np.isfinite(f.read("xm")).all()


# the rows cross in blocks of 8 MB: one ragged block, and several with a ragged last one
@pytest.mark.parametrize("N,prec", [(3001, 0), (3001, 1), (1_200_001, 0)])
def test_parts_of_a_fresh_a_stepped_and_a_restored_filter(N, prec):
    from paper_1203_2394_gb300 import dpf
    prec = dpf.DPF_F64 if prec else dpf.DPF_F32
    spec, f = _pf(N, prec)
    _own(f)
    _, ys = workloads.simulate(spec, 2, 0)
    for y in ys:
        f.step(y.astype(f.dtype))
    _own(f)
    state = f.get_state()
    _, g = _pf(N, prec)
    g.set_state(state)
    _own(g)
    for k in ("xm", "zm"):
        np.testing.assert_array_equal(g.read(k), f.read(k))


def test_no_buffer_of_means_is_held():
    from paper_1203_2394_gb300 import dpf
    N = 100_000
    spec, f = _pf(N, dpf.DPF_F32)
    # a particle's rows at d = 10, in FP32: two of x padded to 16 bytes, of z, of lq, of the weights and
    # draw of one look-ahead, then its log-weight, weight, ancestor and choice: 144 bytes; the means
    # would be 40 more
    per = 2 * (16 + 32 + 4 + 4 + 8) + 4 * 4
    assert f.memory() < N * (per + 20), f.memory() / N
