"""The one-thread FP64 kernel in each of its launch shapes, on a batch large
enough to be run by it (512 all-Morse lanes per SM), and the FP32 refill queue
above its line: every lane has the bits that the same lane has in a batch of a
few thousand (FP64: the lane-group kernels) or in launch mode 0 (FP32), with
lanes among them that fail, and with a step cap that ends them all."""
import numpy as np
import pytest

from paper_2304_02731_gb300 import workloads as W

F64 = ["t", "h", "dE", "vprime", "jprime", "gbw"]
U8 = ["status", "cls", "nsteps", "nrej", "vt", "jt"]
NAN_LANES, HMIN_LANES = (3, 40_000), (5, 41_111)


@pytest.fixture(scope="module")
def Q():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2304_02731_gb300 import qcams
    return qcams


def _start(Q, n):
    """n lanes of the sweep's upper energies, initialised; some will fail."""
    per = n // 144 + 1
    w = W.sweep_h2_ca(per_cell=per)
    w = w.slice(10 * 24 * per, 10 * 24 * per + n)
    b = Q.Batch.empty(n, "cuda", sys_id=w.sys_id, keep_u=False)
    Q.init_states(w.systems, b, w.E, w.b, w.v, w.j, w.R0, w.seed)
    for k in NAN_LANES:
        b.y[0][k] = float("nan")
    for k in HMIN_LANES:
        b.f64["t"][k], b.f64["h"][k] = 1e15, 1e-3
    return w, b


def _run(Q, w, start, integ, idx=None):
    """Results of the lanes idx (all: None) of the initialised batch."""
    import torch
    if idx is None:
        idx = slice(None)
    b = Q.Batch.empty(start.status[idx].numel(), "cuda", sys_id=start.sys_id[idx], keep_u=False)
    b.y.copy_(start.y[:, idx])
    for k in ("t", "h", "t_scale", "E0", "Ecol"):
        b.f64[k].copy_(start.f64[k][idx])
    for k in ("status", "nsteps", "nrej"):
        getattr(b, k).copy_(getattr(start, k)[idx])
    Q.run_batch(w.systems, b, integ)
    torch.cuda.synchronize()
    out = {k: b.f64[k].cpu().numpy() for k in F64}
    out.update({k: getattr(b, k).cpu().numpy() for k in U8}, y=b.y.cpu().numpy())
    return out


def _same(got, want, idx):
    for k, x in want.items():
        assert np.array_equal(got[k][..., idx], x, equal_nan=x.dtype.kind == "f"), k


def _failures(Q, got, cap):
    assert (got["status"][list(NAN_LANES)] == Q.LANE["FAIL_NAN"]).all()
    assert (got["status"][list(HMIN_LANES)] == Q.LANE["FAIL_HMIN"]).all()
    if cap:
        rest = np.ones(got["status"].size, bool)
        rest[list(NAN_LANES + HMIN_LANES)] = False
        assert (got["status"][rest] == Q.LANE["FAIL_MAXSTEPS"]).all()
        assert (got["nsteps"][rest] + got["nrej"][rest] == cap).all()


@pytest.fixture(scope="module")
def fp64(Q):
    """The batch and the results of 3,000 of its lanes by the lane groups."""
    import torch
    n = 512 * Q.device_info()[0] + 777
    w, start = _start(Q, n)
    idx = np.unique(np.r_[NAN_LANES, HMIN_LANES, np.linspace(0, n - 1, 3000).astype(int)])
    dev = torch.as_tensor(idx, device="cuda")
    want = {cap: _run(Q, w, start, Q.make_integ(**w.integ, persistent=1, max_steps=cap or 10 ** 6),
                      dev) for cap in (0, 20)}
    return w, start, idx, want


@pytest.mark.gpu
@pytest.mark.parametrize("cap", [0, 20])
@pytest.mark.parametrize("block,per_sm", [(128, 1), (64, 1), (128, 3), (64, 6), (64, 7), (256, 1)])
def test_one_thread_shapes(Q, fp64, block, per_sm, cap):
    w, start, idx, want = fp64
    integ = Q.make_integ(**w.integ, persistent=1, block=block, blocks_per_sm=per_sm,
                         max_steps=cap or 10 ** 6)
    got = _run(Q, w, start, integ)
    _failures(Q, got, cap)
    _same(got, want[cap], idx)


@pytest.mark.gpu
@pytest.mark.parametrize("cap", [0, 20])
def test_fp32_queue(Q, cap):
    w, start = _start(Q, 1792 * Q.device_info()[0] + 777)
    got, want = (_run(Q, w, start, Q.make_integ(**W.INTEG_FP32, precision=32, persistent=mode,
                                                max_steps=cap or 10 ** 6)) for mode in (1, 0))
    _failures(Q, got, cap)
    _same(got, want, slice(None))
