"""Float instances of a batch whose records overflow the shared buffer or whose magnitudes leave the
candidate margin no room: solved again alone, with the results of the CPU oracle (FP64)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def q():
    import paper_2607_04857_gb300 as q

    q.load_library()
    return q


def twins(n, pairs, scale, seed):
    """A float matrix of whole numbers in which variables v and v + n/2 (v < pairs) couple alike to all
    others and exclude each other: exact ties in FP64 whose FP32 energies differ by their rounding."""
    rng = np.random.default_rng(seed)
    A = np.triu(rng.integers(-scale, scale + 1, size=(n, n)), 1)
    A = A + A.T
    d = rng.integers(-scale, scale + 1, size=n)
    of = np.arange(n)
    of[n // 2:n // 2 + pairs] -= n // 2  # a twin has its original's row
    A, d = A[np.ix_(of, of)], d[of]
    for v in range(pairs):
        t = v + n // 2
        A[v, t] = A[t, v] = 4 * scale
        d[v] = d[t] = d[v] - 3 * scale
    return (np.triu(A, 1) + np.diag(d)).astype(np.float64)


def check(r, o):
    assert r.min == o.min and r.n_ties == o.n_ties
    assert np.array_equal(r.ties, o.ties) and np.array_equal(r.topk, o.topk) and np.array_equal(r.topk_E, o.topk_E)


@pytest.mark.parametrize("scale", [10, 10**4, 10**7])
@pytest.mark.parametrize("graph", [False, True])
def test_overflow_beside_large_magnitudes(q, scale, graph, monkeypatch):
    """One instance of nothing but ties fills the buffer; the others lose records and are solved again,
    with FP32's rounding at scale 10^7 a thousand times the default margin."""
    Qs = [np.zeros((16, 16))] + [twins(22, 5, scale, seed) for seed in range(6)]
    monkeypatch.setenv("QUBO_MAX_RECORDS", "2000")
    if graph:
        b = q.Batch(Qs, topk=20, states_cap=64)
        b.run()
        rs = b.fetch()
    else:
        rs = q.solve_batched(Qs, topk=20, states_cap=64)
    assert max(r.info["passes"] for r in rs) > 1
    for Q, r in zip(Qs, rs):
        check(r, oracle.solve(Q, topk=20, cap=64))
    if graph:
        b.close()


def test_every_part_of_a_split_range_keeps_to_the_margin(q, monkeypatch):
    """Eight low variables whose fields the six top ones cancel when all are set: the sub-cube of the
    top ones set holds the minimum 2^8 times, overflows and is split down to direct evaluation (FP64),
    while the other parts are scanned in FP32 (factored), whose rounding at 10^6 is beyond the margin."""
    scale, rng = 10**6, np.random.default_rng(0)
    Q = np.zeros((20, 20))
    Q[np.arange(8), np.arange(8)] = 6 * scale
    Q[:8, 14:] = -scale
    Q[8:, 8:] = np.triu(rng.integers(-scale, scale + 1, size=(12, 12)))
    Q[np.arange(14, 20), np.arange(14, 20)] -= 4 * scale
    assert oracle.solve(Q).n_ties == 256 and q.plan_query(Q)["acc"] == "f32z"
    monkeypatch.setenv("QUBO_MAX_RECORDS", "64")
    p = q.Problem(Q, topk=8)
    p.run()
    r = p.fetch()
    p.close()
    check(r, oracle.solve(Q, topk=8))
    assert r.info["acc"] == "f64", r.info


@pytest.mark.parametrize("n", [1, 6, 11, 12, 16])
def test_entries_beyond_fp32(q, n):
    """Entries of 10^39 on every path, directly evaluated sizes among them: FP64 decides, and no
    infinite energy enters the records or the reported rounding error."""
    Q = np.random.default_rng(n).uniform(-1e39, 1e39, (n, n))
    o = oracle.solve(Q, topk=2, cap=64)
    b, p = q.Batch([Q, Q], topk=2), q.Problem(Q, topk=2)
    b.run()
    p.run()
    rs = [q.solve(Q, topk=2), q.solve(Q, topk=2, rigorous=True), *q.solve_batched([Q, Q], topk=2), *b.fetch(), p.fetch()]
    for r in rs:
        check(r, o)
        assert r.info["fp32_max_abs_err"] <= 1e-9 * abs(o.min), r.info
    b.close()
    p.close()


@pytest.mark.parametrize("scale", [1.0, 100.0])
def test_window_is_part_of_the_rounding_bound(q, scale):
    """A float window's width is added to the threshold in FP32, and the bound counts the rounding of the
    sum: reported with the run, and every state of wide and narrow windows returned."""
    from plan_checks import fp32_bound

    Q = np.random.default_rng(7).uniform(-scale, scale, (19, 19))
    o = oracle.solve(Q, topk=4096, cap=1)
    for k in (1, 20, 3000):
        width = float(np.nextafter(o.topk_E[k] - o.min, np.inf))
        sel = o.topk_E <= o.min + width
        cnt, codes, E, info = q.solve_window(Q, width)
        assert info["acc"] == "f32" and cnt == int(sel.sum())
        assert np.array_equal(codes, o.topk[sel]) and np.array_equal(E, o.topk_E[sel])
        ref = fp32_bound(Q, info["suffix_bits"], info["walk_bits"], info["reg_rows"], info["anchor_bits"], window=width)
        assert info["fp32_err_bound"] == pytest.approx(ref, rel=1e-9)


def test_a_long_list_costs_a_batch_what_it_costs_alone(q):
    """2^20 ties in a small batch: rescored and sorted once, by the whole GPU (0.8 times the device time of
    the instance alone; 3.8 times when the batch's own pass rescored them first, on one block)."""
    from paper_2607_04857_gb300 import workloads as wl

    Q = wl.diagonal(22, seed=3, zeros=20).astype(np.float32)
    few = [wl.upper_int(17, -50, 50, seed=9 + k).astype(np.float32) for k in range(3)]
    alone = min(q.solve(Q, topk=4, states_cap=64).info["seconds_gpu"] for _ in range(3))
    batch = [q.solve_batched([Q] + few, topk=4, states_cap=64) for _ in range(3)]
    assert min(rs[0].info["seconds_gpu"] for rs in batch) < 2 * alone
    for M, r in zip([Q] + few, batch[0]):
        check(r, oracle.solve(M, topk=4, cap=64))
