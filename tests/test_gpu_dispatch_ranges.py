"""Dispatch branches beyond the sizes of the other edge tests, each against the oracle or an equality.

* the particle filter's weighted sums in double precision, taken with the step and, when every
  weight lies too far below their reference, from the particles;
* a BF16 gradient whose slices of the minibatch hold several chunks of rows;
* global resampling from 16-byte-aligned weights (vector loads) at the partition's edges, beyond the
  2^24 weights up to which the point count's estimate is in single precision, and from two streams
  and threads at once (their scratch comes from one pool).
"""
import threading

import numpy as np
import pytest

from oracle import learned, oracle
from paper_1203_2394_gb300 import workloads
from tests import test_gpu_learned as tl
from tests.gpu_util import rel

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def lib():
    return oracle.load()


@pytest.mark.parametrize("far", [0.0, 40.0])
@pytest.mark.parametrize("N", [257, 512 * 40 + 3])
def test_pf_weighted_sums_in_double(N, far):
    """Sums of N terms of one sign or of order one in double precision, in different orders: N 2^-52."""
    from paper_1203_2394_gb300 import dpf
    spec = workloads.make_model("lg4", 0)
    f = dpf.ParticleFilter(dpf.Model.from_spec(spec, dpf.DPF_F64), spec.d1, spec.d2, N, 5)
    ref = -0.5 * (len(spec.R) * np.log(2 * np.pi) + np.linalg.slogdet(spec.R)[1])
    _, ys = workloads.simulate(spec, 2, 1)
    tol = 4 * N * 2.0 ** -52 + 1e-13
    logz = 0.0
    for t in range(2):
        mean, lz = f.step(ys[t] + far * (t == 1))
        lw = f.read("lw")
        if t == 1 and far:
            assert lw.max() < ref - 20
        x, z = f.read("x"), f.read("z")[:, :, 0].T
        W = np.exp(lw - lw.max())
        em = np.concatenate([W @ x, W @ z]) / W.sum()
        assert np.max(rel(mean, em[np.argsort(spec.perm())])) <= tol
        logz += lw.max() + np.log(W.mean())
        assert abs(lz - logz) <= tol * max(1.0, abs(logz))


def test_bf16_gradient_of_many_rows():
    """5000 rows: slices of 640 rows, three chunks each. The bounds are those of the 600-row test."""
    p = tl._prop()
    W = workloads.init_mlp_weights(tl.DIN, tl.H, tl.DOUT, seed=5)
    W["b4"] = 0.3 * np.random.default_rng(6).standard_normal(tl.DOUT)
    p.set_weights(W)
    F, Z, w = (a.astype(np.float32).astype(np.float64) for a in tl._data(5000, 8))
    loss, g = p.loss_grad(*tl._dev(F, Z, w))
    ref_loss, ref_g = learned.nll_and_grad(p.get_weights(), F, Z, w, tl.D2, tl.C, bf16_mode=True)
    assert loss == pytest.approx(ref_loss, rel=1e-3)
    G = p.unflatten(g.cpu().numpy().astype(np.float64))
    for k in G:
        a, b = G[k].ravel(), ref_g[k].ravel()
        assert a @ b / (np.linalg.norm(a) * np.linalg.norm(b) + 1e-30) >= 0.999, k
        assert np.max(np.abs(a - b)) <= 2e-2 * np.max(np.abs(b)) + 1e-7, k


def _weights(n, dtype, spike, seed):
    rng = np.random.default_rng(seed)
    w = (rng.exponential(size=n) ** 3).astype(dtype)
    if spike:
        w[rng.integers(0, n, 2)] = 1e12
    return w, rng.integers(0, 2**32, 1, dtype=np.uint64).astype(np.uint32)


def _resample(w, u):
    from paper_1203_2394_gb300 import dpf
    return dpf.resample(w, torch.tensor(u.view(np.int32), device="cuda"), dpf.DPF_SYS_GLOBAL).cpu().numpy()


@pytest.mark.parametrize("n,dtype", [(513, "float32"), (513, "float64"), ((1 << 17) + 1, "float32"),
                                     (512 * 1216 + 1, "float64"), (2 * 512 * 1216 + 7, "float32"),
                                     (1 << 24, "float32"), ((1 << 24) + 1, "float32")])
@pytest.mark.parametrize("spike", [False, True])
def test_resample_aligned_and_large(n, dtype, spike, lib):
    w, u = _weights(n, dtype, spike, n)
    t = torch.tensor(w, device="cuda")
    assert t.data_ptr() % 16 == 0
    np.testing.assert_array_equal(_resample(t, u), oracle.sys_global(w.astype(np.float64), int(u[0]), lib))


def test_resample_from_two_streams_at_once(lib):
    sets = [_weights(n, "float32", False, n) for n in (300_007, 90_001)]
    refs = [oracle.sys_global(w.astype(np.float64), int(u[0]), lib) for w, u in sets]
    bad = []

    def work(k):
        with torch.cuda.stream(torch.cuda.Stream()):
            w, u = sets[k]
            t = torch.tensor(w, device="cuda")
            for _ in range(30):
                if not np.array_equal(_resample(t, u), refs[k]):
                    bad.append(k)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    assert bad == []
