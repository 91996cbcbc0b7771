"""The autotuner's choice against the runs themselves: on samples of up to one
warp per SM sub-partition, and for systems that are not all-Morse, the mode it
returns is the fastest that qcams_run_batch has, to within 5 % of its time."""
import numpy as np
import pytest

from paper_2304_02731_gb300 import workloads as W


@pytest.fixture(scope="module")
def Q():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2304_02731_gb300 import qcams
    return qcams


def _sample(Q, w):
    import torch
    b = Q.Batch.empty(w.n, "cuda", sys_id=w.sys_id, keep_u=False)
    Q.init_states(w.systems, b, w.E, w.b, w.v, w.j, w.R0, w.seed)
    torch.cuda.synchronize()
    return b


def _run_ms(Q, w, integ, start):
    b = Q.Batch.empty(w.n, "cuda", sys_id=w.sys_id, keep_u=False)
    best = float("inf")
    for _ in range(2):
        b.y.copy_(start.y)
        for k in ("t", "h", "t_scale", "E0", "Ecol"):
            b.f64[k].copy_(start.f64[k])
        for k in ("status", "nsteps", "nrej"):
            getattr(b, k).copy_(getattr(start, k))
        Q.run_batch(w.systems, b, integ)
        best = min(best, Q.last_run_stats()["integrate_ms"])
    return best


def _morse(n):
    w = W.sweep_h2_ca(per_cell=n // 384 + 1)
    return w.take(np.linspace(0, w.n - 1, n).astype(int))


def _mixed(n):
    return W.mixed_ca_h(n=n, seed=6)


@pytest.mark.gpu
@pytest.mark.parametrize("study,n,cap", [(_morse, 12_288, 6000), (_morse, 500, 3000),
                                         (_mixed, 900, 3000), (_mixed, 15_000, 3000)])
def test_choice_is_the_fastest_run(Q, study, n, cap):
    w = study(n)
    start = _sample(Q, w)
    for k in ("vprime", "jprime"):
        start.f64[k].fill_(2.5)
    before = {k: start.f64[k].clone() for k in ("t", "h", "vprime", "jprime")}
    integ = Q.make_integ(**w.integ, persistent=1, max_steps=cap)
    best, table = Q.autotune(w.systems, start, integ, max_attempts=cap)
    for k, x in before.items():
        assert np.array_equal(start.f64[k].cpu().numpy(), x.cpu().numpy()), k
    ms = {m: _run_ms(Q, w, Q.make_integ(**w.integ, persistent=m, max_steps=cap), start)
          for m in (1, 2, 3)}
    print(f"\n{n} lanes: mode 1 {ms[1]:.2f} ms, 2 {ms[2]:.2f}, 3 {ms[3]:.2f}; chosen "
          f"{best.persistent}")
    assert ms[best.persistent] <= 1.05 * min(ms.values())
    if study is _mixed:               # the shapes are not used: one run, listed for each
        assert len({r["ms"] for r in table[:6]}) == 1
        assert abs(table[0]["ms"] - ms[1]) <= 0.1 * ms[1]
