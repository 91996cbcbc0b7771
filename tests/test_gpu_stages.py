"""The FP64 run's stages (one thread, then three and six lanes per trajectory,
handing unfinished trajectories on) give every lane the same bits whichever
stages it passes, so a lane of a large batch equals the same lane of a small
one.  Also the outputs that hold the hand-on lists pointed at one buffer."""
import numpy as np
import pytest

from paper_2304_02731_gb300 import workloads as W

FIELDS = ["y", "t", "h", "dE", "vprime", "jprime", "gbw", "status", "cls", "nsteps", "nrej", "vt",
          "jt"]


@pytest.fixture(scope="module")
def Q():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2304_02731_gb300 import qcams
    return qcams


def _subset(Q, b, idx):
    """A batch of lanes idx of the initialised batch b."""
    out = Q.Batch.empty(len(idx), "cuda", sys_id=b.sys_id[idx], keep_u=False)
    out.y.copy_(b.y[:, idx])
    for k in ("t", "h", "t_scale", "E0", "Ecol"):
        out.f64[k].copy_(b.f64[k][idx])
    for k in ("status", "nsteps", "nrej"):
        getattr(out, k).copy_(getattr(b, k)[idx])
    return out


def _values(b):
    import torch
    torch.cuda.synchronize()
    get = lambda k: b.y if k == "y" else b.f64[k] if k in b.f64 else getattr(b, k)  # noqa: E731
    return {k: get(k).cpu().numpy() for k in FIELDS}


def _morse():
    w = W.sweep_h2_ca(per_cell=560)
    return w.slice(10 * 24 * 560, w.n)           # 80,640 lanes, the upper energies


def _generic():
    w = W.mixed_ca_h(n=20_001, seed=3)
    # (10, 6) takes the general Lennard-Jones form
    lj = ("lj_fit", 10, 6, 0.0630, 3.79)
    w.systems = w.systems[:2] + [dict(w.systems[2], pairs=(W.HH_MORSE, lj, lj))]
    return w


@pytest.mark.gpu
@pytest.mark.parametrize("study,sizes", [(_morse, (1, 11, 3041, 12_167)),
                                         (_generic, (5, 610, 3040, 12_161))])
def test_stages_agree_bit_for_bit(Q, study, sizes):
    import torch
    w = study()
    integ = Q.make_integ(**w.integ, persistent=True)
    start = Q.Batch.empty(w.n, "cuda", sys_id=w.sys_id)
    Q.init_states(w.systems, start, w.E, w.b, w.v, w.j, w.R0, w.seed)
    start.sys_id[7] = 9                          # no such system
    start.status[8] = 0x40                       # not a runnable status
    start.status[9] = Q.LANE["RUNNING"]
    big = _subset(Q, start, torch.arange(w.n, device="cuda"))
    Q.run_batch(w.systems, big, integ)
    whole = _values(big)
    assert whole["status"][7] == Q.LANE["INVALID"] and whole["status"][8] == 0x40
    assert np.isin(whole["status"][10:], [2, 3, 4, 8]).all()
    rng = np.random.default_rng(1)
    for n in sizes:
        idx = torch.as_tensor(np.sort(rng.choice(w.n, n, replace=False)), device="cuda")
        if n > 100:
            idx[:5] = torch.arange(6, 11, device="cuda")
        part = _subset(Q, start, idx)
        Q.run_batch(w.systems, part, integ)
        got = _values(part)
        for k in FIELDS:
            want = whole[k][..., idx.cpu().numpy()]
            assert np.array_equal(got[k], want, equal_nan=got[k].dtype.kind == "f"), (n, k)


@pytest.mark.gpu
def test_one_buffer_for_several_outputs(Q):
    w = W.plain_h2_ca(per_b=650)                 # 3,250 lanes: two stages
    integ = Q.make_integ(**w.integ, persistent=True)
    runs = []
    for shared in (False, True):
        b = Q.Batch.empty(w.n, "cuda", sys_id=w.sys_id)
        Q.init_states(w.systems, b, w.E, w.b, w.v, w.j, w.R0, w.seed)
        if shared:
            b.c.jprime = b.c.vprime
        Q.run_batch(w.systems, b, integ)
        runs.append(_values(b))
    for k in ("y", "t", "h", "dE", "status", "cls", "nsteps", "nrej", "vt", "jt"):
        assert np.array_equal(runs[0][k], runs[1][k]), k


@pytest.mark.gpu
@pytest.mark.parametrize("study", ["morse", "mixed"])
def test_fp32_queue_order(Q, study):
    """FP32 batches beyond what the GPU holds at once are taken slowest
    collisions first: each lane as in a batch that is taken as it comes."""
    import torch
    w = _morse() if study == "morse" else W.mixed_ca_h(n=98_304 + 1, seed=5)
    integ = Q.make_integ(**W.INTEG_FP32, precision=32, persistent=True)
    start = Q.Batch.empty(w.n, "cuda", sys_id=w.sys_id)
    Q.init_states(w.systems, start, w.E, w.b, w.v, w.j, w.R0, w.seed)
    start.f64["t_scale"][3] = 0.0                # ends at its first step
    big = _subset(Q, start, torch.arange(w.n, device="cuda"))
    Q.run_batch(w.systems, big, integ)
    whole = _values(big)
    idx = torch.as_tensor(np.r_[0:7, 40_000:42_001, w.n - 5:w.n], device="cuda")
    part = _subset(Q, start, idx)
    Q.run_batch(w.systems, part, integ)
    got = _values(part)
    for k in FIELDS:
        want = whole[k][..., idx.cpu().numpy()]
        assert np.array_equal(got[k], want, equal_nan=got[k].dtype.kind == "f"), k
