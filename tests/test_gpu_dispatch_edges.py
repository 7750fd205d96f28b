"""The kernels of the hot paths at the edges of their dispatch rules and tiles.

Every check is one of the oracle comparisons of the component's own test file, with that
file's tolerances, or an equality that the rule itself requires:

* the DPF without look-ahead and the paper models' step, one warp a group: every class of
  particles a lane, a ragged last lane, one-warp CTAs and full ones, and the size next to a
  class that the block form serves;
* two filters of one kernel whose shared-memory needs differ, stepped in turn;
* the look-ahead step at more groups than run as one-warp CTAs;
* the wide step's two threads a particle at small, odd and large L and an odd count of groups;
* the bootstrap filter when the step's own weighted sums serve and when every weight lies too
  far below their reference;
* the network's forward pass around its tiles and clusters, on rows off 16 bytes, and a
  minibatch's gradient around its tiles;
* global resampling around the chunk, the CTA partition and the scaled count's threshold, from
  a pointer off 16 bytes.
"""
import numpy as np
import pytest

from oracle import learned, oracle
from paper_1203_2394_gb300 import workloads
from tests import test_gpu_learned, test_gpu_paper, test_gpu_std, test_gpu_step, test_gpu_wide
from tests.gpu_util import rel, state_from_gpu, word

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

FEW = 16 * 152  # most groups that run as one-warp CTAs


@pytest.fixture(scope="module")
def lib():
    return oracle.load()


def _std_calls(name, N, M, lib, calls=3):
    spec, f = test_gpu_std._filter(name, "f32", N, M, 9)
    f.set_debug(True)
    om = oracle.OracleModel.from_spec(spec)
    _, ys = workloads.simulate(spec, calls, 1)
    x, z, lq = state_from_gpu(f)
    anc = None
    idx = np.unique(np.linspace(0, N - 1, 60).astype(int))
    for t in range(1, calls + 1):
        y = ys[t - 1].astype(np.float32)
        f.step(y)
        gx, gz, glq = state_from_gpu(f)
        glw = f.read("lw").astype(np.float64)
        test_gpu_std._check_call(om, 9, t, y.astype(np.float64), x, z, lq, idx if anc is None else anc[idx], lib,
                                 gx[idx], gz[idx], glq[idx], glw[idx], f.read("jla")[idx, 0], f.read("bidx")[idx],
                                 1e-5, dest=idx)
        anc = f.read("anc")
        wout = f.read("wout").astype(np.float64)
        np.testing.assert_array_equal(anc, oracle.sys_global(wout, word(9, t, 0, oracle.P_OUTER), lib))
        x, z, lq = gx, gz, glq


@pytest.mark.parametrize("name,N,M", [("lg4", 90, 4), ("lg4", 90, 32), ("growth_clg10", 90, 36), ("lg4", 90, 64),
                                      ("growth_clg10", 90, 68), ("lg4", 90, 132), ("growth_clg10", 90, 136),
                                      ("growth_clg10", 90, 256), ("growth_clg10", FEW, 20),
                                      ("growth_clg10", FEW + 1, 20), ("lg4", 3 * FEW + 5, 32)])
def test_std_classes(name, N, M, lib):
    _std_calls(name, N, M, lib)


@pytest.mark.parametrize("case", [(1, 90, 4, 4, 3), (1, 90, 32, 8, 3), (2, 90, 36, 16, 3), (1, 90, 128, 32, 3),
                                  (2, 90, 136, 8, 3), (2, 90, 256, 32, 3), (-1, 90, 132, 8, 3)],
                         ids=lambda c: f"model{c[0]}-N{c[1]}-M{c[2]}-L{c[3]}")
def test_paper_step_classes(case, lib):
    test_gpu_paper.test_paper_la_dpf_teacher_forced(case, lib)


@pytest.mark.parametrize("kind", [1, 2])
def test_paper_step_few_groups(kind):
    """One-warp CTAs and full ones: the first step's groups depend on their index alone."""
    y = workloads.simulate_paper(kind, 1, 0)[1][0].astype(np.float32)
    a, b = (test_gpu_paper._la(kind, n, 8, 4, 3) for n in (FEW, FEW + 1))
    a.step(y)
    b.step(y)
    for name in ("lw", "lwhat", "xbb"):
        np.testing.assert_array_equal(a.read(name), b.read(name)[:FEW], err_msg=name)


def _interleaved(make_big, make_small, ys):
    alone = make_big()
    ref = [alone.step(y) for y in ys]
    big, small = make_big(), make_small()
    for y, (mean, logz) in zip(ys, ref):
        m, lz = big.step(y)
        np.testing.assert_array_equal(m, mean)
        assert lz == logz
        small.step(y)


def test_filters_of_different_shared_memory_in_turn():
    """Two filters that share a kernel: the smaller one's first step leaves the larger one's
    shared memory as it was (73 KB a CTA against 39 KB; 117 KB against 37 KB)."""
    from paper_1203_2394_gb300 import dpf
    spec = workloads.make_model("lg16", 0, 1)
    model = dpf.Model.from_spec(spec, dpf.DPF_F32)
    ys = workloads.simulate(spec, 3, 0)[1].astype(np.float32)
    _interleaved(lambda: dpf.StandardDPF(model, 1, 15, FEW + 8, 256, 3),
                 lambda: dpf.StandardDPF(model, 1, 15, FEW + 8, 136, 4), ys)
    ys = workloads.simulate_paper(1, 3, 0)[1].astype(np.float32)
    _interleaved(lambda: test_gpu_paper._la(1, FEW + 8, 256, 32, 3), lambda: test_gpu_paper._la(1, FEW + 8, 136, 4, 4),
                 ys)


@pytest.mark.parametrize("case", [("growth_clg10", 2, FEW + 1, 32, 4, 3), ("lg4", 2, FEW + 1, 32, 8, 3),
                                  ("lg4", 2, 90, 256, 16, 3), ("lg4", 2, 90, 64, 12, 3),
                                  ("growth_clg10", 2, 90, 256, 32, 3), ("growth_clg10", 2, 90, 136, 4, 3)],
                         ids=lambda c: f"{c[0]}-N{c[2]}-M{c[3]}-L{c[4]}")
def test_lookahead_step_classes(case):
    test_gpu_step.test_fp32_teacher_forced(case)


@pytest.mark.parametrize("case", [(157, 256, 4, 3, True), (41, 128, 12, 3, True), (305, 128, 40, 3, True),
                                  (33, 256, 1, 3, True), (41, 128, 5, 3, True)],
                         ids=lambda c: f"N{c[0]}-M{c[1]}-L{c[2]}")
def test_wide_pair_edges(case):
    """(L of no multiple of 4: the look-ahead weights' rows are not whole 16-byte units, and the
    step takes its CUDA-core form.)"""
    test_gpu_wide.test_wide_teacher_forced(case)


@pytest.mark.parametrize("far", [0.0, 30.0])
@pytest.mark.parametrize("N", [1, 31, 257, 512 * 40 + 3])
def test_pf_weighted_sums(N, far):
    """far: the observation lies so many units off that every log-weight is more than 20 below
    the reference (the sums are then taken from the particles, as the check states)."""
    from paper_1203_2394_gb300 import dpf
    spec = workloads.make_model("lg4", 0)
    f = dpf.ParticleFilter(dpf.Model.from_spec(spec, dpf.DPF_F32), spec.d1, spec.d2, N, 5)
    ref = -0.5 * (len(spec.R) * np.log(2 * np.pi) + np.linalg.slogdet(spec.R)[1])
    _, ys = workloads.simulate(spec, 3, 1)
    logz = 0.0
    for t in range(3):
        mean, lz = f.step((ys[t] + far * (t == 1)).astype(np.float32))
        lw = f.read("lw").astype(np.float64)
        if t == 1 and far:
            assert lw.max() < ref - 20
        x, z = f.read("x").astype(np.float64), f.read("z")[:, :, 0].T.astype(np.float64)
        W = np.exp(lw - lw.max())
        em = np.concatenate([W @ x, W @ z]) / W.sum()
        assert np.max(rel(mean, em[np.argsort(spec.perm())])) <= 1e-5
        logz += lw.max() + np.log(W.mean())
        assert lz == pytest.approx(logz, rel=1e-5, abs=1e-5)
        np.testing.assert_array_equal(f.read("xm").T, f.read("x"))
        np.testing.assert_array_equal(f.read("zm"), f.read("z")[:, :, 0])


def _off16(a):
    """The array on the device, starting 4 bytes past a 16-byte boundary."""
    t = torch.empty(a.size + 1, dtype=torch.float32, device="cuda")
    v = t[1:].view(a.shape)
    v.copy_(torch.tensor(a, dtype=torch.float32))
    return v


@pytest.mark.parametrize("off", [False, True])
@pytest.mark.parametrize("n", [1, 127, 129, 256, 257, 513, 256 * 152 + 257])
def test_forward_tiles(n, off):
    p = test_gpu_learned._prop()
    W = test_gpu_learned._integer_net(0)
    p.set_weights(W)
    F = np.random.default_rng(n).integers(0, 2, (n, test_gpu_learned.DIN)).astype(np.float64)
    rows = _off16(F) if off else torch.tensor(F, dtype=torch.float32, device="cuda")
    got = p.forward(rows).double().cpu().numpy()
    ref, _ = learned.forward(W, F, bf16_mode=True)
    np.testing.assert_array_equal(got, ref)


@pytest.mark.parametrize("n,off", [(1, False), (31, True), (128, False), (129, False), (300, True)])
def test_gradient_tiles(n, off):
    """The FP32 form against the oracle's backpropagation, as at the training file's size."""
    p = test_gpu_learned._prop()
    W = workloads.init_mlp_weights(test_gpu_learned.DIN, test_gpu_learned.H, test_gpu_learned.DOUT, seed=5)
    p.set_weights(W)
    p.set_bf16(False)
    F, Z, w = (a.astype(np.float32).astype(np.float64) for a in test_gpu_learned._data(n, n))
    loss, g = p.loss_grad(*(_off16(a) for a in (F, Z, w))) if off else p.loss_grad(*test_gpu_learned._dev(F, Z, w))
    ref_loss, ref_g = learned.nll_and_grad(p.get_weights(), F, Z, w, test_gpu_learned.D2, test_gpu_learned.C,
                                           bf16_mode=False)
    assert loss == pytest.approx(ref_loss, rel=1e-5)
    G = p.unflatten(g.cpu().numpy().astype(np.float64))
    for k in G:
        assert np.max(np.abs(G[k] - ref_g[k])) <= 1e-4 * np.max(np.abs(ref_g[k])) + 1e-7, k


@pytest.mark.parametrize("dtype", ["float32", "float64"])
@pytest.mark.parametrize("n", [511, 512, 513, (1 << 17) - 1, 1 << 17, (1 << 17) + 1, 512 * 1216 + 1, 2 * 512 * 1216 + 7])
def test_resample_partition_edges(n, dtype, lib):
    from paper_1203_2394_gb300 import dpf
    rng = np.random.default_rng(n)
    for spike in (False, True):
        w = (rng.exponential(size=n) ** 3).astype(dtype)
        if spike:
            w[rng.integers(0, n, 2)] = 1e12
        u = rng.integers(0, 2**32, 1, dtype=np.uint64).astype(np.uint32)
        t = torch.empty(n + 1, dtype=getattr(torch, dtype), device="cuda")[1:]  # off 16 bytes
        t.copy_(torch.tensor(w))
        got = dpf.resample(t, torch.tensor(u.view(np.int32), device="cuda"), dpf.DPF_SYS_GLOBAL).cpu().numpy()
        np.testing.assert_array_equal(got, oracle.sys_global(w.astype(np.float64), int(u[0]), lib))
