"""Backward pass of the batched objective under autograd's own transforms (on the
GPU autograd runs it in another thread): the evaluation is replaced by f_k = |D_k|^2 (gradient 2 D_k, exact in
binary), so only the scaling by the incoming gradient is under test.  All
values are products of two float64 numbers, compared exactly."""
import pytest

torch = pytest.importorskip("torch")
import paper_2010_06931_gb300 as octmc  # noqa: E402
from paper_2010_06931_gb300 import autograd  # noqa: E402

SHAPES = [(2, 3, 4, 5), (2, 3, 1, 1), (2, 3, 7, 2)]  # one plane size per pair


@pytest.fixture(params=["cpu", pytest.param("cuda", marks=pytest.mark.gpu)])
def disps(request, monkeypatch):
    def evaluate(problems, levels, disps, grads=None):
        for D, g in zip(disps, grads or []):
            g.copy_(2.0 * D)
        return [float((D * D).sum()) for D in disps]

    monkeypatch.setattr(octmc, "eval_batch", evaluate)
    gen = torch.Generator().manual_seed(3)
    return [torch.randn(s, generator=gen, dtype=torch.float64).to(request.param).requires_grad_() for s in SHAPES]


def objective(disps, mode):
    return autograd.batch_objective([None] * len(disps), 0, disps, mode=mode)


MODES = pytest.mark.parametrize("mode", ["save", "recompute"])


@MODES
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_backward(disps, mode, dtype):
    (objective(disps, mode).to(dtype) * 3.0).backward()
    for D in disps:
        assert torch.equal(D.grad, 3.0 * (2.0 * D.detach()))


@MODES
def test_several_incoming_gradients_at_once(disps, mode):
    v = torch.tensor([1.0, -0.5, 3.0, 0.0], dtype=torch.float64, device=disps[0].device)
    got = torch.autograd.grad(objective(disps, mode), disps, grad_outputs=v, is_grads_batched=True)
    for D, g in zip(disps, got):
        assert torch.equal(g, v.view(-1, 1, 1, 1, 1) * (2.0 * D.detach()))


@MODES
def test_vectorized_jacobian(disps, mode):
    got = torch.autograd.functional.jacobian(lambda *D: objective(list(D), mode), tuple(disps), vectorize=True)
    for D, g in zip(disps, got):
        assert torch.equal(g, 2.0 * D.detach())


@MODES
def test_create_graph_tracks_the_incoming_gradient(disps, mode):
    s = torch.tensor(3.0, dtype=torch.float64, device=disps[0].device, requires_grad=True)
    got = torch.autograd.grad(objective(disps, mode), disps, grad_outputs=s, create_graph=True)
    for D, g in zip(disps, got):
        assert torch.equal(g.detach(), 3.0 * (2.0 * D.detach()))
    # d/ds sum_k sum(g_k) = sum_k sum(2 D_k): one addition per element and pair
    (ds,) = torch.autograd.grad(sum(g.sum() for g in got), s)
    want = sum((2.0 * D.detach()).sum() for D in disps)
    n = sum(D.numel() for D in disps)
    assert abs(float(ds - want)) <= n * 2.0 ** -52 * float(sum((2.0 * D.detach()).abs().sum() for D in disps))
