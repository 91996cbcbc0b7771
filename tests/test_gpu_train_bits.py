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
