"""Bits of the network's training that do not depend on scheduling: with at
most 16 rows every sum of the gradient has one order, so gradients and whole
training runs have one result."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

B3, W4, B4 = 8832, 8896, 9152          # parameter offsets of b3, W4, b4


@pytest.fixture(scope="module")
def Q():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2304_02731_gb300 import qcams
    return qcams


def _row_sum(d, bits):
    """FP32 sum of 16 rows: r and r + 8, then the partners r ^ bit."""
    s = d[:8] + d[8:]
    for b in bits:
        s = s + s[np.arange(8) ^ b]
    return s[0]


def test_bias_gradient_row_order(Q):
    """b3's gradient over 16 rows, from a network whose hidden layers are zero
    (SiLU' = 1/2, logits = b4) and whose W4 hands one output's error to each
    unit.  Output 0 has probability 2^-23, so errors of -1/16 and of about
    2^-27 meet in a column and the order of its sum shows."""
    import torch
    mlp = Q.MLP()
    p = np.zeros(Q.MLP_NPARAMS, np.float32)
    k = (np.arange(64) + np.arange(64) // 8) % 4          # the output behind each unit
    w = (2.0 ** -(np.arange(64) % 3)).astype(np.float32)
    p[W4 + 64 * k + np.arange(64)] = w
    p[B4:B4 + 4] = [-14.7, 0.0, 0.3, -0.5]
    mlp.set_params(p)
    x = torch.zeros(16, 8, device="cuda")
    prob = mlp.infer(x)[0].cpu().numpy()
    differ = 0
    for seed in range(40):
        label = np.random.default_rng(seed).integers(0, 5, 16)
        mlp.compute_grad(x, torch.as_tensor(label, dtype=torch.uint8, device="cuda"))
        got = mlp.grad[B3:B3 + 64].cpu().numpy()
        hit = (label[:, None] == np.arange(4)).astype(np.float32)
        d = (prob - hit) * np.float32(1 / 16) * (label < 4)[:, None].astype(np.float32)
        d = torch.from_numpy(d).bfloat16().float().numpy()[:, k] * w * np.float32(0.5)
        want = _row_sum(d, (1, 2, 4))
        differ += int((want != _row_sum(d, (4, 2, 1))).sum())
        assert np.array_equal(got, want), (seed, np.flatnonzero(got != want))
    assert differ > 0                  # the rows chosen do show the order


def _values(m):
    return [t.cpu().numpy() for t in (m.params, m.m, m.v, m.grad, m.params_bf16)]


@pytest.mark.parametrize("how", ["eager", "stream", "graph"])
@pytest.mark.parametrize("batch,steps", [(1, 1), (16, 9), (7, 40)])
def test_training_is_its_single_steps(Q, how, batch, steps):
    """qcams_mlp_train against the same rows one qcams_mlp_train_step at a
    time, bit for bit: losses, last indices, last gradient, parameters,
    moments and the step count; as a plain call, on a stream of its own beside
    other work, and replayed from a graph."""
    import torch
    gen = torch.Generator(device="cuda").manual_seed(batch)
    x = torch.randn(500, 8, device="cuda", generator=gen)
    cls = torch.randint(0, 6, (500,), device="cuda", generator=gen).to(torch.uint8)
    a, b, one = Q.MLP(seed=2), Q.MLP(seed=2), Q.MLP(seed=1)
    for m in (a, b):
        m.train_step(x[:3].contiguous(), cls[:3].contiguous(), 1e-3)     # training goes on from step 1
    want = []
    for s in range(steps):
        one.c.step = 1 + s                                               # the rows of step 1 + s
        rows = one.train(x, cls, 1, batch, 1e-3, seed=21)[1]
        want.append(b.train_step(x[rows].contiguous(), cls[rows].contiguous(), 2e-3).clone())
    side, busy = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    if how == "eager":
        losses, idx = a.train(x, cls, steps, batch, 2e-3, seed=21)
    elif how == "stream":
        big = torch.randn(4096, 4096, device="cuda")
        torch.cuda.synchronize()
        with torch.cuda.stream(busy):
            for _ in range(20):
                big = big @ big * 1e-3
        with torch.cuda.stream(side):
            losses, idx = a.train(x, cls, steps, batch, 2e-3, seed=21)
    else:
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side):
            losses, idx = a.train(x, cls, steps, batch, 2e-3, seed=21)
        graph.replay()
    torch.cuda.synchronize()
    assert a.step == b.step == 1 + steps
    assert np.array_equal(idx.cpu().numpy(), rows.cpu().numpy())
    assert np.array_equal(losses.cpu().numpy(), torch.cat(want).cpu().numpy())
    for u, v in zip(_values(a), _values(b)):
        assert np.array_equal(u, v)
