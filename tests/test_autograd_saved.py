"""What the autograd Function keeps for the backward pass: grad f only where the
first-order point gradient can use it, and a copy of its own of a single point's,
whose outputs are views.  CPU only: the library's calls are replaced."""

import pytest
import torch


@pytest.fixture
def query(monkeypatch):
    import paper_2110_01614_gb300.autograd as ag

    def fake_query(ctx, pts, out, flags):
        out.copy_(2.0 * pts)                       # f = |p|^2, grad f = 2 p
        out[:, 3] = (pts[:, :3] ** 2).sum(1)

    def fake_backward(ctx, pts, g_f, g_grad, g_w, g_p):
        if g_p is not None:
            g_p.zero_()
            g_p[:, :3] = 2.0 * g_f[:, None] * pts[:, :3]
        if g_w is not None:
            g_w.fill_(1.0)

    class Net:
        ctx, arch, precision = None, None, ag.NSDF_FP32

        def load(self, blob):
            return self

    monkeypatch.setattr(ag, "nsdf_query", fake_query)
    monkeypatch.setattr(ag, "nsdf_backward", fake_backward)
    monkeypatch.setattr("paper_2110_01614_gb300.nsdf_num_params", lambda arch: 5)
    return ag, Net()


@pytest.mark.parametrize("points,blob,kept", [(True, False, 2), (True, True, 1), (False, True, 1)])
def test_kept_bytes(query, points, blob, kept):
    ag, net = query
    p = torch.rand(7, 4, requires_grad=points)
    w = torch.rand(5, requires_grad=blob)
    sizes = []
    with torch.autograd.graph.saved_tensors_hooks(lambda t: sizes.append(t.numel()) or t, lambda t: t):
        f, g = ag.sdf_query(p, w, net)
    assert sizes == [28] * kept
    f.sum().backward()
    if points:
        assert torch.equal(p.grad[:, :3], 2.0 * p.detach()[:, :3]) and not p.grad[:, 3].any()
    if blob:
        assert torch.equal(w.grad, torch.ones(5))


def test_other_precisions_keep_the_points_only(query):
    ag, net = query
    net.precision = ag.NSDF_FP32 + 1
    sizes = []
    with torch.autograd.graph.saved_tensors_hooks(lambda t: sizes.append(t.numel()) or t, lambda t: t):
        ag.sdf_query(torch.rand(7, 4, requires_grad=True), torch.rand(5), net)
    assert sizes == [28]


@pytest.mark.parametrize("n", [1, 2])
def test_changed_outputs_do_not_reach_the_gradient(query, n):
    """grad f belongs to the caller, also where it is a view."""
    ag, net = query
    p = torch.rand(n, 4, requires_grad=True)
    f, g = ag.sdf_query(p, torch.rand(5), net)
    g.data.zero_()
    f.sum().backward()
    assert torch.equal(p.grad[:, :3], 2.0 * p.detach()[:, :3])
