"""Every form of the pair force in the lane-group stages against the one-thread
kernel, bit for bit: one adaptive attempt with a given step (modes 0 and 1)
and one step of the fixed-step mode from the same states, for systems whose
three pairs are of all kinds."""
import numpy as np
import pytest

from paper_2304_02731_gb300 import workloads as W

KINDS = [W.HH_MORSE, ("buck", 300.0, 1.4, 200.0, 2.0), ("lj_fit", 12, 6, 0.06, 2.6),
         ("lj_fit", 8, 6, 0.06, 2.6), ("lj_fit", 10, 6, 0.06, 2.6), ("lj_fit", 12, 5, 0.06, 2.6),
         ("lj_fit", 9, 4, 0.1, 2.5), ("lj_fit", 4, 3, 0.02, 3.0), ("lj_fit", 32, 3, 0.02, 3.0)]


@pytest.mark.gpu
@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("n", [60, 400, 4000])       # six lanes; six; three lanes
@pytest.mark.parametrize("first", range(len(KINDS)))
def test_one_attempt_equals_one_step(first, n, mode):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2304_02731_gb300 import qcams as Q
    rng = np.random.default_rng(100 * first + n)
    kinds = [[first, *rng.integers(0, len(KINDS), 2)] for _ in range(4)]
    for k in kinds[1:3]:
        rng.shuffle(k)
    systems = [dict(mass_u=tuple(rng.uniform(1, 40, 3)), pairs=tuple(KINDS[i] for i in k))
               for k in kinds]
    y = np.concatenate([rng.uniform(1.0, 3.0, (6, n)) * rng.choice([-1, 1], (6, n)),
                        rng.normal(0, 10.0, (6, n))])
    sid = rng.integers(0, 4, n).astype(np.int32)
    h = 0.125
    out = []
    for integ in (Q.make_integ(rtol=1e-2, atol=1e-2, r_stop=1e6, t_stop=1e6, max_steps=1,
                               persistent=mode),
                  Q.make_integ(fixed_step=True, h_fixed=h, max_steps=1)):
        b = Q.Batch.empty(n, "cuda", sys_id=sid, keep_u=False)
        b.y.copy_(torch.as_tensor(y))
        b.f64["t_scale"].fill_(1.0)
        for k, x in (("t", 0.0), ("h", h), ("E0", 0.0), ("Ecol", 0.1)):
            b.f64[k].fill_(x)
        for t in (b.status, b.nsteps, b.nrej):
            t.zero_()
        Q.run_batch(systems, b, integ)
        out.append((b.y.cpu().numpy(), b.nsteps.cpu().numpy()))
    (got, steps), (want, _) = out
    taken = steps == 1
    assert taken.mean() > 0.9
    for s in range(4):
        at = taken & (sid == s)
        assert np.array_equal(got[:, at], want[:, at]), [KINDS[i] for i in kinds[s]]
