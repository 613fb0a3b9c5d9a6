"""The grouped step form of the int32 and packed 16-bit scans against the CPU oracle, at the sizes
where it can go wrong: the shortest walks (one group per body, one body per unit), walks across
several memory rows, entries at the limits its arithmetic admits (packed columns up to the cap of
its adds, int32 energies near 2^30), and instances whose groups mostly or always reach the threshold
(small integers, ties everywhere, a wide energy window)."""
import os

import numpy as np
import pytest

import oracle
from paper_2607_04857_gb300 import workloads as wl
from plan_checks import column_range

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def q():
    import paper_2607_04857_gb300 as q

    q.load_library()
    return q


@pytest.fixture(autouse=True)
def dense(monkeypatch):
    monkeypatch.setenv("QUBO_NO_I32Z", "1")


def check(r, o):
    assert r.min == o.min and r.n_ties == o.n_ties
    assert np.array_equal(r.ties, o.ties) and np.array_equal(r.topk, o.topk) and np.array_equal(r.topk_E, o.topk_E)


@pytest.mark.parametrize("acc,variant", [("i16p", 20), ("i16p", 21), ("i32", 20), ("i32", 21)])
@pytest.mark.parametrize("walk", [5, 6, 7, 11, 14])
def test_walks(q, acc, variant, walk, monkeypatch):
    if walk == 5 and variant == 20:
        pytest.skip("five register rows need six walked bits")
    monkeypatch.setenv("QUBO_SCAN_VARIANT", str(variant))
    Q = wl.upper_int(26, -90, 90, seed=walk + variant)
    o = oracle.solve(Q, topk=12)
    r = q.solve(Q, topk=12, walk_bits=walk, int32=acc == "i32")
    assert (r.info["acc"], r.info["grouped"], r.info["walk_bits"]) == (acc, 1, walk), r.info
    check(r, o)
    check(q.solve(Q, walk_bits=walk, int32=acc == "i32"), oracle.solve(Q))


@pytest.mark.parametrize("scale", [1.0, 1.0005, 1.01, 1.3])
def test_packed_limits(q, scale):
    """Columns scaled up to 32767: the grouped form runs while none reaches 32767 and the rows' moves
    fit 16 bits, its interleaved twin beyond (both exact), other accumulators past 16 bits."""
    Q = wl.upper_int(24, -1000, 1000, seed=31)
    hi = max(column_range(Q, 10, 6, 5)[1], -column_range(Q, 10, 6, 5)[0])
    Q = (Q * (32766.0 / hi * scale)).astype(np.int32)
    r = q.solve(Q, topk=8, walk_bits=6)
    lo, hi = column_range(Q, 10, 6, 5)
    assert (r.info["acc"] == "i16p") == (lo >= -32768 and hi <= 32767)
    if r.info["grouped"] and r.info["acc"] == "i16p":
        assert hi < 32767
    check(r, oracle.solve(Q, topk=8))


@pytest.mark.parametrize("sign", [-1, 0, 1])
def test_int32_limits(q, sign):
    """Energies up to the int32 bound (sum of |U| just below 2^30), of both signs and of one."""
    Q = wl.upper_int(23, 1, 1 << 20, seed=40)
    Q = Q * np.where((sign > 0) | ((sign == 0) & (np.arange(23 * 23).reshape(23, 23) % 2 == 1)), 1, -1)
    Q = (Q.astype(np.float64) * ((2.0**30 - 600) / np.abs(np.triu(Q)).astype(np.float64).sum())).astype(np.int32)
    assert np.abs(Q.astype(np.int64)).sum() < 1 << 30
    r = q.solve(Q, topk=8)
    assert r.info["acc"] == "i32" and r.info["grouped"] == 1, r.info
    check(r, oracle.solve(Q, topk=8))


@pytest.mark.parametrize("acc", ["i16p", "i32"])
def test_every_group_reaches_the_threshold(q, acc):
    """Ties in every group (10 diagonal entries of -1, the other variables free), and +-1 couplings."""
    Q = np.zeros((24, 24), dtype=np.int32)
    Q[np.arange(10), np.arange(10)] = -1
    kw = dict(int32=acc == "i32", walk_bits=9)
    check(q.solve(Q, states_cap=1 << 14, **kw), oracle.solve(Q, cap=1 << 14))
    Q = wl.upper_int(24, -1, 1, seed=2)
    r = q.solve(Q, topk=40, states_cap=4096, **kw)
    assert r.info["acc"] == acc and r.info["grouped"] == 1
    check(r, oracle.solve(Q, topk=40, cap=4096))


def test_window_and_sub_cubes(q):
    Q = wl.upper_int(30, -120, 120, seed=5)
    o = oracle.solve(Q, topk=4096, cap=1, fix_bits=6, fix_value=11)
    width = int(o.topk_E[1500] - o.min)
    sel = o.topk_E <= o.min + width
    assert not sel.all()
    cnt, codes, E, info = q.solve_window(Q, width, fix_bits=6, fix_value=11)
    assert info["acc"] == "i16p" and cnt == int(sel.sum())
    assert np.array_equal(codes, o.topk[sel]) and np.array_equal(E, o.topk_E[sel])
    for v in (0, 63):
        check(q.solve(Q, topk=5, fix_bits=6, fix_value=v), oracle.solve(Q, topk=5, fix_bits=6, fix_value=v))


@pytest.mark.parametrize("count", [1, 3, 40])
def test_small_batches(q, count):
    """A small batch's walk is shortened to occupy the GPU; sizes from direct evaluation to 24."""
    insts = [wl.upper_int(int(n), -100, 100, seed=int(n), dtype=np.int16) for n in np.linspace(24, 11, count)]
    for Q, r in zip(insts, q.solve_batched(insts, topk=3, states_cap=16)):
        check(r, oracle.solve(Q.astype(np.int32), topk=3, cap=16))


# --- direct evaluation (sub-cubes too small to split) ------------------------------------------

@pytest.mark.parametrize("free", [0, 1, 4, 5, 6, 9, 10, 11, 12, 13])
def test_direct_evaluation(q, free):
    """Items of 2^10 states: fewer states than lanes, one partial item, several; variables above the
    sub-cube fixed to patterns with both values, up to variable 63; every accumulator."""
    for n, fix in ((free, 0), (40, 0x15555), (64, (1 << 40) + 12345)):
        if n < max(free, 1):
            continue
        fb = n - free
        fv = fix & ((1 << fb) - 1)
        K = min(1 << free, 20)
        Q = wl.upper_int(n, -1000, 1000, seed=free + n)
        wide = wl.upper_int(n, -(1 << 30), 1 << 30, seed=free + n)
        for M in (Q, wide, Q.astype(np.int16)):
            check(q.solve(M, topk=K, fix_bits=fb, fix_value=fv),
                  oracle.solve(M.astype(np.int32), topk=K, fix_bits=fb, fix_value=fv))
        F = wl.sk_float32(n, seed=free + n)
        for kw in ({}, {"plain": True}):
            r, o = q.solve(F, topk=K, fix_bits=fb, fix_value=fv, **kw), oracle.solve(F, topk=K, fix_bits=fb, fix_value=fv)
            assert r.min == o.min and np.array_equal(r.topk, o.topk) and np.array_equal(r.ties, o.ties)


# --- record lists: sorted and extracted on the device, short and long --------------------------

@pytest.mark.parametrize("zeros", [0, 5, 10, 11, 12, 16])
def test_record_list_lengths(q, zeros):
    """2^zeros minimisers: lists of one record, up to the short list's 2048 and beyond, alone and in a
    batch beside short ones (single calls and graph replays), integer and float."""
    Q = wl.diagonal(18, seed=3, zeros=zeros)
    o = oracle.solve(Q, topk=30, cap=5000)
    check(q.solve(Q, topk=30, states_cap=5000), o)
    few = wl.upper_int(17, -50, 50, seed=9)
    of = oracle.solve(few, topk=30, cap=5000)
    b = q.Batch([few, Q, few, Q], topk=30, states_cap=5000)
    for _ in range(2):
        b.run()
        for rs in (q.solve_batched([few, Q, few, Q], topk=30, states_cap=5000), b.fetch()):
            for r, e in zip(rs, (of, o, of, o)):
                check(r, e)
        b.run()
    b.fetch()
    b.close()
    F = Q.astype(np.float32)
    r = q.solve(F, topk=30, states_cap=5000)
    assert r.min == o.min and r.n_ties == o.n_ties and np.array_equal(r.ties, o.ties) and np.array_equal(r.topk, o.topk)
    for r, e in zip(q.solve_batched([few.astype(np.float32), F], topk=30, states_cap=5000), (of, o)):
        assert r.min == e.min and r.n_ties == e.n_ties and np.array_equal(r.ties, e.ties)


# --- float magnitudes beyond the caller's margin -------------------------------------------------

def check_exact_float(r, o):
    assert r.min == o.min and r.n_ties == o.n_ties
    assert np.array_equal(r.ties, o.ties) and np.array_equal(r.topk, o.topk) and np.array_equal(r.topk_E, o.topk_E)


@pytest.mark.parametrize("scale", [1.0, 30.0, 100.0, 1e6, 1e20, 1e35])
@pytest.mark.parametrize("n", [14, 20, 26])
def test_float_proven_margin(q, n, scale):
    """Entries from where the default margin holds to where no FP32 scan can run: FP32 with a proven
    margin up to FP32's range (every returned energy the FP64 sum), FP64 beyond it."""
    rng = np.random.default_rng(n)
    Q = rng.uniform(-scale, scale, (n, n))
    r, o = q.solve(Q, topk=10), oracle.solve(Q, topk=10)
    check_exact_float(r, o)
    assert r.info["acc"] == ("f64" if scale > 1e30 else "f32"), r.info
    if r.info["acc"] == "f32" and scale >= 100 and n > 14:
        assert r.info["passes"] == 1
    rs = q.solve_batched([Q, Q / scale], topk=10)
    check_exact_float(rs[0], o)


def test_float_proven_margin_gives_up(q):
    """A penalty encoding: 2^16 and more states within the proven margin of the minimum; the attempt
    ends early and the FP64 scan decides."""
    n = 22
    Q = np.zeros((n, n))
    Q[0, 0] = 1e7
    Q[np.arange(1, n), np.arange(1, n)] = np.random.default_rng(1).uniform(-1e-3, 1e-3, n - 1)
    Q[1, 2] = 1e-4
    r = q.solve(Q, topk=16)
    assert r.info["acc"] == "f64" and r.info["passes"] >= 2, r.info
    check_exact_float(r, oracle.solve(Q, topk=16))
    cnt, codes, E, _ = q.solve_window(Q, 2e-4)
    o = oracle.solve(Q, topk=4096, cap=1)
    sel = o.topk_E <= o.min + 2e-4
    assert not sel.all() and cnt == int(sel.sum()) and np.array_equal(codes, o.topk[sel])


# --- int64 energies on two limbs -----------------------------------------------------------------

@pytest.mark.parametrize("walk", [0, 5, 6, 9, 14])
@pytest.mark.parametrize("scale", [1 << 22, 1 << 26, (1 << 31) - 1])
def test_two_limbs(q, walk, scale):
    """Energies from just beyond int32 to the largest an int32 matrix gives, on random entries and on
    entries whose low halves all lie at the split's extremes."""
    n = 25
    Q = wl.upper_int(n, -scale, scale, seed=walk + 3).astype(np.int64)
    iu = np.triu_indices(n)
    for low in (None, 0x2aaaaa, -1):
        M = Q.copy()
        if low is not None:
            M[iu] = (M[iu] >> 23 << 23) + (low & 0x3fffff) if scale > 1 << 24 else M[iu] | 1
        M = np.clip(M, -(2**31), 2**31 - 1).astype(np.int32)
        M[0, 0] = 2**31 - 1  # the sum of |U| above 2^30
        r, o = q.solve(M, topk=9, walk_bits=walk), oracle.solve(M, topk=9)
        assert r.info["acc"] == "i64" and r.info["grouped"] == 1, r.info
        check(r, o)
        check(q.solve(M, walk_bits=walk), oracle.solve(M))
    p = q.solve(M, topk=9, plain=True)
    assert p.info["acc"] == "i64" and p.info["grouped"] == 0
    check(p, oracle.solve(M, topk=9))


def test_two_limbs_ties_window_batch(q):
    """Ties in every group, every state of a window, and a batch with direct evaluation beside it."""
    Q = np.zeros((24, 24), dtype=np.int32)
    Q[np.arange(10), np.arange(10)] = -(1 << 30)
    check(q.solve(Q, states_cap=1 << 14), oracle.solve(Q, cap=1 << 14))
    W = wl.upper_int(24, -(1 << 27), 1 << 27, seed=8)
    o = oracle.solve(W, topk=4096, cap=1)
    width = int(o.topk_E[900] - o.min)
    sel = o.topk_E <= o.min + width
    if width < 1 << 30:
        cnt, codes, E, info = q.solve_window(W, width)
        assert info["acc"] == "i64" and cnt == int(sel.sum())
        assert np.array_equal(codes, o.topk[sel]) and np.array_equal(E, o.topk_E[sel])
    insts = [wl.upper_int(n, -(1 << 28), 1 << 28, seed=n) for n in (9, 13, 14, 15, 19, 22)]
    for M, r in zip(insts, q.solve_batched(insts, topk=4)):
        assert r.info["acc"] == "i64"
        check(r, oracle.solve(M, topk=4, cap=64))


@pytest.mark.parametrize("walk", [13, 14, 15, 16])
def test_two_limbs_longest_walk(q, walk, tmp_path):
    """A minimum whose base and walked rows all have the lowest low limb: the sum of `walk` of them and
    the base's.  A batch takes an installed plan's walk up to the 14 rows the group test allows for."""
    n = 9 + walk + 2
    Q = np.zeros((n, n), dtype=np.int32)
    Q[0, 0] = Q[0, 9:9 + walk] = -(1 << 30) + 32
    Q[1, 1], Q[9 + walk, 9 + walk], Q[10 + walk, 10 + walk] = 5, 77, 1000
    path = str(tmp_path / "plans")
    q.autotune_batched([wl.upper_int(16, -90, 90, seed=k, dtype=np.int16) for k in range(2)])
    q.autotune_save(path)
    device = open(path).read().split("\n")[1].split("\t")[:2]
    q.autotune_clear()
    with open(path, "w") as f:
        f.write("qubo-autotune 1\n" + "\t".join(device + ["2", str(-n), "1", str(walk)]) + "\n")
    assert q.autotune_load(path) == 1
    try:
        rs = q.solve_batched([Q, Q], topk=3)
    finally:
        q.autotune_clear()
    for r in rs:
        assert r.info["acc"] == "i64" and r.info["grouped"] == 1, r.info
        assert r.info["walk_bits"] == walk if walk <= 14 else r.info["walk_bits"] <= 14, r.info
        check(r, oracle.solve(Q, topk=3, cap=64))


def test_a_batch_has_the_whole_record_buffer(q):
    """2^21 minimisers and a little more in one batch, half of what the buffer of a call holds: no
    instance is solved a second time."""
    Qs = [wl.diagonal(22, seed=3, zeros=21)] + [wl.upper_int(17, -50, 50, seed=9 + k) for k in range(3)]
    rs = q.solve_batched(Qs, topk=4)
    assert rs[0].n_ties == 1 << 21 and rs[0].info["passes"] == 1, rs[0].info
    for Q, r in list(zip(Qs, rs))[1:]:
        check(r, oracle.solve(Q, topk=4, cap=64))
