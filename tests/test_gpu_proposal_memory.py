"""Device memory of a proposal's minibatches: one workspace of the largest minibatch so far, and no
room for gathered rows where a call reads its rows in place.
"""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_a_growing_minibatch_holds_one_workspace():
    from paper_1203_2394_gb300 import dpf
    p = dpf.Proposal(2, 2, 2, hidden=256, components=4)
    sizes = (65536, 131072, 262144)
    g = torch.Generator(device="cuda").manual_seed(1)
    n = sizes[-1]
    F = torch.randn((n, 8), generator=g, device="cuda")
    Z = torch.randn((n, 2), generator=g, device="cuda")
    w = torch.rand((n,), generator=g, device="cuda")
    grads = [p.loss_grad(F[:257], Z[:257], w[:257])[1]]
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    res0 = torch.cuda.memory_reserved()
    for k in sizes:
        p.loss_grad(F[:k], Z[:k], w[:k])
    torch.cuda.synchronize()
    held = free0 - torch.cuda.mem_get_info()[0] - (torch.cuda.memory_reserved() - res0)
    # the largest minibatch's layers: five of 256 values a row and two of the head's 20
    one = 4 * n * (5 * 256 + 2 * 20)
    assert held < 1.1 * one, (held, one)
    # training gathers its rows: their buffers come with it. The first layer's weight gradient of 257
    # rows is one sum or two slices, so it repeats bit for bit
    grads.append(p.loss_grad(F[:257], Z[:257], w[:257])[1])
    assert torch.equal(grads[0][:2048], grads[1][:2048])
    losses = p.train(F[:1000], Z[:1000], w[:1000], batch=256, epochs=1)
    assert len(losses) == 1 and losses[0] == losses[0]
