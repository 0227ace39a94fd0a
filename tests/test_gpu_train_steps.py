"""mlp_train runs many Adam steps in one launch whose CTAs meet on the device. One step against the
gradient of mlp_loss_grad (a launch of its own) and Adam in numpy, at the edges of the 128-sample tiles
and at the smallest and largest batches; runs across the 256 steps a launch holds against the same steps
taken one call at a time; and a captured run replayed."""

import numpy as np
import pytest

import paper_2505_22822_gb300 as tkf

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
LR = 2e-3


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return tkf.Context(0)


def _records(n, seed=1):
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn(n, 12, generator=g, device="cuda")
    y = torch.sin(x[:, :1]) + 0.3 * x[:, 1:2] * x[:, 2:3]
    return torch.cat([x, y], 1).contiguous()


def _start(ctx):
    p = torch.empty(tkf.MLP_PARAMS, device="cuda")
    tkf.mlp_init(ctx, p, 3)
    return p, torch.zeros(2, tkf.MLP_PARAMS, device="cuda")


@pytest.mark.parametrize("batch", [1, 2, 127, 128, 129, 1000, 1024, 4097, 8192])
def test_one_step_is_adam_on_the_gradient(ctx, batch):
    rec = _records(batch)
    p, mom = _start(ctx)
    loss, grad = tkf.mlp_loss_grad(ctx, p, rec[:, :12].contiguous(), rec[:, 12].contiguous())
    p0, g = p.cpu().numpy(), grad.cpu().numpy()
    el, t = tkf.mlp_train(ctx, rec, p, mom, 0, batch=batch, epochs=1, lr=LR)
    assert t == 1
    # the first step moves every parameter by lr g / (|g| + 1e-8): a few units in the last place
    want = p0.astype(np.float64) - LR * g / (np.abs(g) + 1e-8)
    np.testing.assert_allclose(p.cpu().numpy(), want, rtol=3e-7, atol=LR * 1e-6)
    np.testing.assert_allclose(mom[0].cpu().numpy(), 0.1 * g, rtol=1e-6)
    np.testing.assert_allclose(el.cpu().numpy(), loss.cpu().numpy(), rtol=1e-6)


@pytest.mark.parametrize("batch,steps", [(64, 1), (200, 255), (64, 256), (300, 257), (64, 600)])
def test_steps_of_one_call_are_the_steps_of_many(ctx, batch, steps):
    rec = _records(batch * steps + batch // 2, seed=batch)  # the last partial batch is dropped
    p, mom = _start(ctx)
    el, t = tkf.mlp_train(ctx, rec, p, mom, 0, batch=batch, epochs=2, lr=LR)
    q, mom2 = _start(ctx)
    u, means = 0, []
    for _ in range(2):
        losses = []
        for b in range(steps):
            one, u = tkf.mlp_train(ctx, rec[b * batch:(b + 1) * batch], q, mom2, u, batch=batch, epochs=1, lr=LR)
            losses.append(one)
        means.append(torch.cat(losses).mean())
    assert t == u == 2 * steps
    assert torch.equal(p, q) and torch.equal(mom, mom2)
    # the mean of `steps` FP32 losses, summed in another order
    np.testing.assert_allclose(el.cpu().numpy(), torch.stack(means).cpu().numpy(), rtol=2e-6 * max(1, steps / 16))


def test_captured_training_replays(ctx):
    rec = _records(1024 * 20, seed=4)
    p, mom = _start(ctx)
    tkf.mlp_train(ctx, rec, p, mom, 0, batch=1024, epochs=1, lr=LR)  # grows the scratch
    want = (p.clone(), mom.clone())
    q, mom2 = _start(ctx)
    q0 = q.clone()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        tkf.mlp_train(ctx, rec, q, mom2, 0, batch=1024, epochs=1, lr=LR)
    for _ in range(2):
        q.copy_(q0)
        mom2.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(q, want[0]) and torch.equal(mom2, want[1])
