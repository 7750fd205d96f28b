"""A minibatch's gradient from run to run: the bias gradients repeat bit for bit at every size, the
whole gradient below 1024 rows (two slices of the minibatch a product at most), and with it training.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

H, DIN, DOUT = 256, 8, 20
OFF_B = [H * DIN, H * DIN + H + H * H, H * DIN + 2 * (H + H * H), H * DIN + 2 * (H + H * H) + H + DOUT * H]


def _rows(n):
    g = torch.Generator(device="cuda").manual_seed(n)
    F = torch.randn((n, DIN), generator=g, device="cuda")
    Z = torch.randn((n, 2), generator=g, device="cuda")
    return F, Z, torch.rand((n,), generator=g, device="cuda") + 0.1


def _proposal(bf16=True):
    from paper_1203_2394_gb300 import dpf, workloads
    p = dpf.Proposal(2, 2, 2, hidden=H, components=4)
    p.set_weights(workloads.init_mlp_weights(DIN, H, DOUT, seed=3))
    if not bf16:
        p.set_bf16(False)
    return p


# one slice, two (even, and with a ragged last one), the last size before more, and many
@pytest.mark.parametrize("bf16", [True, False])
@pytest.mark.parametrize("n", [100, 256, 600, 1023, 1024, 5000])
def test_gradient_repeats(n, bf16):
    p, rows = _proposal(bf16), _rows(n)
    ref = p.loss_grad(*rows)[1].cpu().numpy()
    assert np.isfinite(ref).all() and ref[OFF_B[0]:OFF_B[0] + H].any()
    for _ in range(8):
        g = p.loss_grad(*rows)[1].cpu().numpy()
        for o, c in zip(OFF_B, (H, H, H, DOUT)):
            np.testing.assert_array_equal(g[o:o + c], ref[o:o + c])
        if n < 1024:
            np.testing.assert_array_equal(g, ref)


@pytest.mark.parametrize("n", [600, 5000])
def test_gradient_repeats_with_an_odd_head(n):
    """One component of one coordinate: a head of three outputs, so no whole 16-byte units in its rows
    or in the parameters."""
    from paper_1203_2394_gb300 import dpf, workloads
    p = dpf.Proposal(1, 1, 1, hidden=64, components=1)
    p.set_weights(workloads.init_mlp_weights(4, 64, 3, seed=3))
    F, Z, w = _rows(n)
    rows = F[:, :4].contiguous(), Z[:, :1].contiguous(), w
    ref = p.loss_grad(*rows)[1].cpu().numpy()
    assert ref[-3:].any()
    for _ in range(4):
        g = p.loss_grad(*rows)[1].cpu().numpy()
        np.testing.assert_array_equal(g[-3:], ref[-3:])
        if n < 1024:
            np.testing.assert_array_equal(g, ref)


def test_training_repeats():
    rows = _rows(3000)
    runs = []
    for _ in range(2):
        p = _proposal()
        p.train(*rows, batch=512, epochs=3, lr=1e-3, seed=5)
        runs.append(p.get_weights())
    for k in runs[0]:
        np.testing.assert_array_equal(runs[0][k], runs[1][k])
