"""FP32 launch mode 1: below several times what the GPU holds it is the launch
of mode 0, in the same time; above, a refill queue with the same bits."""
import numpy as np
import pytest

from paper_2304_02731_gb300 import workloads as W

FIELDS = ["t", "h", "dE", "vprime", "jprime", "gbw"]


@pytest.fixture(scope="module")
def Q():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2304_02731_gb300 import qcams
    return qcams


def _lanes(study, n):
    if study in ("mixed", "lj12"):
        w = W.mixed_ca_h(n=n if study == "mixed" else 4 * n, seed=4)
        if study == "lj12":
            w = w.take(np.flatnonzero(w.sys_id == 1)[:n])
            w.systems, w.sys_id = [w.systems[1]], np.zeros(n, np.int32)
        return w
    per = n // 144 + 1
    w = W.sweep_h2_ca(per_cell=per)
    w = w.slice(10 * 24 * per, w.n)              # the upper energies
    w = w.take(np.linspace(0, w.n - 1, n).astype(int))
    if study == "two":
        w.systems, w.sys_id = w.systems * 2, (np.arange(n) % 2).astype(np.int32)
    return w


def _run(Q, w, mode, repeat):
    import torch
    integ = Q.make_integ(**W.INTEG_FP32, precision=32, persistent=mode)
    b = Q.Batch.empty(w.n, "cuda", sys_id=w.sys_id)
    d = [torch.as_tensor(a, device="cuda") for a in (w.E, w.b, w.v, w.j)]
    best = float("inf")
    for _ in range(repeat):
        Q.init_states(w.systems, b, *d, w.R0, w.seed)
        Q.run_batch(w.systems, b, integ)
        best = min(best, Q.last_run_stats()["integrate_ms"])
    return best, ([b.y.cpu().numpy()] + [b.f64[k].cpu().numpy() for k in FIELDS]
                  + [t.cpu().numpy() for t in (b.status, b.cls, b.nsteps, b.nrej, b.vt, b.jt)])


@pytest.mark.gpu
@pytest.mark.parametrize("study,n", [("morse", 31), ("morse", 512), ("morse", 20_000),
                                     ("two", 20_000), ("mixed", 20_000), ("morse", 150_000)])
def test_mode_1_costs_no_more(Q, study, n):
    w = _lanes(study, n)
    (t0, x0), (t1, x1) = (_run(Q, w, mode, 5) for mode in (0, 1))
    for x, y in zip(x0, x1):
        assert np.array_equal(x, y, equal_nan=x.dtype.kind == "f")
    print(f"\n{study} {n}: mode 0 {t0:.3f} ms, mode 1 {t1:.3f} ms")
    if n >= 512:                  # a shorter run is as long as its launch
        assert t1 < 1.08 * t0


@pytest.mark.gpu
@pytest.mark.parametrize("study,per_sm", [("morse", 1792), ("two", 1792), ("mixed", 1792),
                                          ("lj12", 1024)])
def test_queue_above_its_line(Q, study, per_sm):
    w = _lanes(study, per_sm * Q.device_info()[0] + 1)
    x0, x1 = (_run(Q, w, mode, 1)[1] for mode in (0, 1))
    for x, y in zip(x0, x1):
        assert np.array_equal(x, y, equal_nan=x.dtype.kind == "f")
