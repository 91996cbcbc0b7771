"""Reduction and proposal kernels at the edges of their tiles, against plain
integer / FP64 numpy: chunks and cells of one, odd and large sizes, lanes with
classes, bins and cells out of range; grids below, at and above the run and
scan blocks."""
import numpy as np
import pytest


@pytest.fixture(scope="module")
def Q():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2304_02731_gb300 import qcams
    return qcams


@pytest.mark.gpu
@pytest.mark.parametrize("n,n_cells,weighted,sort", [
    (1, 1, False, False), (37, 3, True, False), (4096, 5, False, True), (4097, 400, True, False),
    (30_011, 9000, False, False), (50_001, 2, True, True)])
def test_reduce_matches_counts(Q, n, n_cells, weighted, sort):
    rng = np.random.default_rng(n)
    cell = rng.integers(-1, n_cells + 1, n).astype(np.int32)
    if sort:
        cell.sort()
    cls, vt, jt = rng.integers(0, 8, n), rng.integers(-3, 90, n), rng.integers(-3, 400, n)
    gbw = rng.uniform(0, 9, n)
    w = rng.uniform(0, 3, n) if weighted else np.ones(n)
    b = Q.Batch.empty(n, "cuda", cell=cell, isw=w if weighted else None)
    import torch
    for dst, src in ((b.cls, cls), (b.vt, vt), (b.jt, jt), (b.f64["gbw"], gbw)):
        dst.copy_(torch.as_tensor(src))
    hist, cells, _ = Q.reduce_xsec(b, n_cells, np.ones(n_cells), np.ones(n_cells),
                                   np.zeros(n_cells), 1, weighted=weighted)
    want = np.zeros((n_cells, Q.H_STRIDE), np.int64)
    fix = lambda x: np.rint(x * 2.0 ** 32).astype(np.int64)  # noqa: E731
    keep = (cell >= 0) & (cell < n_cells)
    c, k = cell[keep], np.where(cls < 6, cls, 5)[keep]
    v, j = np.clip(vt[keep], 0, 63), np.clip(jt[keep], 0, 255)
    np.add.at(want, (c, Q.H_COUNT + k), 1)
    np.add.at(want, (c, np.full(c.size, Q.H_COUNT + 6)), 1)
    np.add.at(want, (c, Q.H_W + k), fix(w[keep]))
    np.add.at(want, (c, Q.H_W2 + k), fix(w[keep] * w[keep]))
    p = k <= 2
    np.add.at(want, (c[p], Q.H_VT + 64 * k[p] + v[p]), 1)
    np.add.at(want, (c[p], Q.H_JT + 256 * k[p] + j[p]), 1)
    np.add.at(want, (c[p], Q.H_GB + 64 * k[p] + v[p]), fix(gbw[keep][p]))
    assert np.array_equal(hist.cpu().numpy(), want)
    host, _ = Q.xsec_from_hist(want, np.ones(n_cells), np.ones(n_cells), np.zeros(n_cells), 1,
                               weighted=weighted)
    # a cell with more failures than outcomes has no error estimate (NaN) in class 5
    assert np.array_equal(cells, host, equal_nan=True)


@pytest.mark.gpu
@pytest.mark.parametrize("n", [0, 1, 513, 1024, 1025, 131_072, 131_073])
@pytest.mark.parametrize("n_cells,weighted", [(1, False), (2, True), (9, False), (9, True)])
def test_histograms_without_cross_sections(Q, n, n_cells, weighted):
    """A call of up to 1,024 lanes that wants no cross sections adds every entry
    in one launch, one of up to 131,072 gives a block 512 lanes: the records
    are those of the lanes taken in halves with cross sections, added up."""
    import torch
    weighted = weighted and n > 0        # without lanes there is no weight array to pass
    rng = np.random.default_rng(n)
    cell = rng.integers(-1, n_cells + 1, n).astype(np.int32)
    b = Q.Batch.empty(n, "cuda", cell=cell, isw=rng.uniform(0, 3000, n) if weighted else None)
    for dst, lo, hi in ((b.cls, 0, 8), (b.vt, -3, 90), (b.jt, -3, 400)):
        dst.copy_(torch.as_tensor(rng.integers(lo, hi, n)))
    b.f64["gbw"].copy_(torch.as_tensor(rng.uniform(0, 9, n)))
    one = np.ones(n_cells)
    got, _, _ = Q.reduce_xsec(b, n_cells, weighted=weighted, finalize=False)
    want = torch.zeros_like(got)
    for lo, hi in ((0, n // 2), (n // 2, n)):
        h = Q.Batch.empty(hi - lo, "cuda", cell=cell[lo:hi],
                          isw=b.isw[lo:hi].cpu().numpy() if weighted else None)
        for k in ("cls", "vt", "jt"):
            getattr(h, k).copy_(getattr(b, k)[lo:hi])
        h.f64["gbw"].copy_(b.f64["gbw"][lo:hi])
        want += Q.reduce_xsec(h, n_cells, one, one, 0 * one, 1, weighted=weighted and hi > lo)[0]
    assert torch.equal(got, want)


@pytest.mark.gpu
@pytest.mark.parametrize("n,most", [(1, 6.0), (2000, 14.0)])
def test_small_reductions_take_few_passes(Q, n, most):
    """Time of small calls without cross sections, in microseconds: a memset and
    one kernel for one lane (two kernels take 1.2 us more), and for 2,000 lanes
    about ten atomics one after the other at 0.7 us and two launches."""
    cell = np.arange(n) % 5
    b = Q.Batch.empty(n, "cuda", cell=cell, isw=np.ones(n))
    import torch
    hist = torch.empty(5 * Q.H_STRIDE, dtype=torch.int64, device="cuda")
    us = _graph_us(lambda: Q.reduce_xsec(b, 5, hist_out=hist, finalize=False))
    print(f"\nreduce of {n} lanes: {us:.2f} us")
    assert us < most


def _graph_us(f, reps=20):
    """Device time of one call, from a graph of `reps`."""
    import torch
    f()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for _ in range(reps):
            f()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    best = float("inf")
    for _ in range(5):
        a.record()
        graph.replay()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) * 1e3 / reps)
    return best


@pytest.mark.gpu
def test_weight_sums_do_not_serialise(Q):
    """Weights add two sums per lane to the three of a lane without them, and 8
    bytes to its 25: 2 M lanes of sorted cells take less than 3.5 times as long
    (2.2 with adds the hardware has, 5 where they are compare-and-swap loops).
    The sums wrap and carry at 32 bits."""
    import torch
    n, n_cells = 2_000_000, 8
    cell = (np.arange(n) * n_cells // n).astype(np.int32)
    w = np.random.default_rng(2).uniform(0, 4000, n)
    us = []
    for isw in (None, w):
        b = Q.Batch.empty(n, "cuda", cell=cell, isw=isw)
        gen = torch.Generator(device="cuda").manual_seed(1)
        for dst, hi in ((b.cls, 6), (b.vt, 12), (b.jt, 40)):
            dst.copy_(torch.randint(0, hi, (n,), device="cuda", generator=gen))
        b.f64["gbw"].copy_(torch.rand(n, dtype=torch.float64, device="cuda", generator=gen))
        hist = torch.empty(n_cells * Q.H_STRIDE, dtype=torch.int64, device="cuda")
        us.append(_graph_us(lambda: Q.reduce_xsec(b, n_cells, hist_out=hist, finalize=False)))
    got = hist.view(n_cells, Q.H_STRIDE).cpu().numpy()
    cls = b.cls.cpu().numpy()
    for at, x in ((Q.H_W, w), (Q.H_W2, w * w)):
        want = np.zeros((n_cells, 6), np.int64)
        np.add.at(want, (cell, cls), np.rint(x * 2.0 ** 32).astype(np.int64))
        assert np.array_equal(got[:, at:at + 6], want)
    print(f"\nreduce of {n} lanes: {us[0]:.1f} us, weighted {us[1]:.1f} us")
    assert us[1] < 3.5 * us[0]


@pytest.mark.gpu
@pytest.mark.parametrize("dims", [(1, 1, 1, 1, 1), (3, 1, 2, 1, 1), (1023, 1, 1, 1, 1),
                                  (2048, 1, 1, 1, 1), (2049, 1, 1, 1, 1), (31, 17, 13, 11, 7),
                                  (1, 1, 1, 1 << 20, 3)])
def test_proposal_cdf_and_draws(Q, dims):
    import torch
    mlp = Q.MLP("cuda", seed=3)
    spec = Q.proposal_spec(0.1, 3, 5, dims=dims, b2_max=77.0)
    q, qfix, cdf = (t.cpu().numpy() for t in mlp.build_proposal(spec))
    N = int(np.prod(dims))
    assert abs(q.sum() - 1.0) < 1e-12
    assert np.array_equal(qfix, np.rint(q * 2.0 ** 40).astype(np.int64))
    assert np.array_equal(cdf, np.cumsum(qfix))
    n = 3001
    b, u, w, cell = (t.cpu().numpy() for t in Q.sample_proposal(
        spec, torch.as_tensor(qfix).cuda(), torch.as_tensor(cdf).cuda(), n, 9, 12345678901))
    idx = np.stack(np.unravel_index(cell, dims))
    pos = np.stack([b * b / 77.0, *u])
    d = np.array(dims, np.float64)[:, None]
    # a coordinate lies in its cell to the rounding of sqrt and its square
    assert np.all(pos * d >= idx * (1 - 1e-15)) and np.all(pos * d <= (idx + 1) * (1 + 1e-15))
    assert np.array_equal(w, (cdf[-1] / N) / qfix[cell])
