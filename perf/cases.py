"""Measured workloads of the exhaustive QUBO solver, through its public Python entry points.

Each case is one call a user makes on host matrices (or, for a device-resident problem or batch,
on the handle such a program keeps): the exact minimum, the tie set, the K lowest states or an
energy window, over all 2^n states or one sub-cube.  Sizes and value ranges are those of the
repository's configurations, benchmark and tests.  Rates are states per second; ``work`` counts
one addition and one comparison per state, and the bytes of the matrix and the results.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

import paper_2607_04857_gb300 as q
from paper_2607_04857_gb300 import workloads as wl

# ---- instances ---------------------------------------------------------------------------------


def _matrix(case: dict, seed: int) -> np.ndarray:
    """The instance of a single-matrix case."""
    n, kind, s = case["n"], case["values"], seed
    if kind == "int":  # upper-triangular, uniform in [-hi, hi]
        return wl.upper_int(n, -case["hi"], case["hi"], seed=s)
    if kind == "int16":
        return wl.upper_int(n, -case["hi"], case["hi"], seed=s, dtype=np.int16)
    if kind == "sk32":
        return wl.sk_float32(n, seed=s)
    if kind == "float64":  # symmetric, uniform in [-hi, hi]
        a = np.random.Generator(np.random.PCG64(s)).uniform(-case["hi"], case["hi"], (n, n))
        return np.ascontiguousarray((a + a.T) / 2)
    if kind == "maxcut":
        return wl.maxcut_qubo(n, case["density"], seed=s)
    if kind == "sparse":
        return wl.sparse_int(n, case["density"], -1000, 1000, seed=s)
    raise ValueError(kind)


def _batch(case: dict, seed: int) -> list:
    """The instances of a batch case: n uniform in [n_lo, n_hi]."""
    count, lo, hi = case["count"], case["n_lo"], case["n_hi"]
    rng = np.random.Generator(np.random.PCG64(seed))
    ns = rng.integers(lo, hi, size=count, endpoint=True)
    # the total work is the same for every seed: the sizes are dealt out evenly
    ns = lo + (np.argsort(np.argsort(ns + rng.random(count))) * (hi - lo + 1)) // count
    ns = rng.permutation(ns)
    sub = rng.integers(0, 2**31 - 1, size=count)
    out = []
    for i in range(count):
        n, s = int(ns[i]), int(sub[i])
        if case["values"] == "sk32":
            out.append(wl.sk_float32(n, seed=s))
        elif i % 2 == 0:
            out.append(wl.upper_int(n, -127, 127, seed=s, dtype=np.int16))
        else:
            out.append(wl.maxcut_qubo(n, 0.5, seed=s, dtype=np.int16))
    return out


# ---- cases -------------------------------------------------------------------------------------


def _solve(name, n, values, hi=0, density=0.0, topk=0, free=0, resident=False):
    """A single solve of 2^free states (free == n: the whole cube)."""
    return {"name": name, "call": "problem" if resident else "solve", "n": n, "values": values, "hi": hi,
            "density": density, "topk": topk, "free": free or n}


def listed() -> list:
    return [
        # the smallest call: a host program solving one small instance after another
        _solve("solve_n16_int16", 16, "int16", hi=100),
        # the 36-variable configuration: small coefficients, minimum, ties and 16 lowest states
        _solve("solve_n36_int32_top16", 36, "int", hi=1000, topk=16),
        # coefficients of six digits: energies need 32 bits
        _solve("solve_n38_int32_large", 38, "int", hi=500_000),
        # coefficients up to 2^30 (scaled or penalty encodings): energies need 64 bits
        _solve("solve_n34_int64", 34, "int", hi=1 << 30, topk=4),
        # one step of the 50-variable configuration on a device-resident problem
        _solve("problem_n50_int32_sub41", 50, "int", hi=32767, topk=16, free=41, resident=True),
        # one step of the 44-variable Sherrington-Kirkpatrick configuration, from host buffers
        _solve("solve_n44_float32_sub39", 44, "sk32", topk=16, free=39),
        # a double-precision matrix with entries of order 100, as exported from a model
        _solve("solve_n31_float64", 31, "float64", hi=100, topk=8),
        # 56 variables at 5% density, one sub-cube
        _solve("solve_n56_sparse_sub45", 56, "sparse", density=0.05, topk=16, free=45),
        # every state near the minimum (a low-energy spectrum)
        {"name": "window_n36_int32", "call": "window", "n": 36, "values": "int", "hi": 1000, "density": 0.0,
         "free": 36, "window": 5000},
        # 72 variables as 32-variable sub-problems of fixed outer variables
        {"name": "wide_n72_inner32", "call": "wide", "n": 72, "values": "int", "hi": 1000, "density": 0.0,
         "n_inner": 32, "outer": 32, "topk": 8},
        # the batched configuration: 4096 instances of 16 to 32 variables from host buffers
        {"name": "batch_4096_n16_32", "call": "batched", "values": "mixed16", "count": 4096, "n_lo": 16, "n_hi": 32,
         "topk": 0},
        # a device-resident batch of small float instances replayed as one graph
        {"name": "graph_512_float32_n8_20", "call": "graph", "values": "sk32", "count": 512, "n_lo": 8, "n_hi": 20,
         "topk": 4},
    ]


def draw(rng) -> dict:
    """One more case of the same ranges."""
    kind = rng.choice(["int16", "int", "int", "int", "sk32", "float64", "sparse", "maxcut", "problem", "window", "wide",
                       "batched", "graph"])

    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    topk = rng.choice([0, 0, 1, 3, 8, 16, 50])
    if kind in ("int", "int16"):
        hi = logint(20, 1 << 30) if kind == "int" else logint(20, 30000)
        n = rng.randint(12, 39 if hi < 20_000 else 37 if hi < 500_000 else 34)
        c = _solve("", n, kind, hi=hi, topk=topk)
    elif kind == "sk32":
        n = rng.randint(12, 46)
        c = _solve("", n, kind, topk=topk, free=min(n, rng.randint(30, 39)))
    elif kind == "float64":
        c = _solve("", rng.randint(12, 31), kind, hi=logint(1, 200), topk=topk)
    elif kind == "sparse":
        n = rng.randint(40, 60)
        c = _solve("", n, kind, density=round(rng.uniform(0.03, 0.08), 3), topk=topk, free=min(n, rng.randint(34, 42)))
    elif kind == "maxcut":
        n = rng.randint(14, 48)
        c = _solve("", n, kind, density=round(rng.uniform(0.4, 1.0), 2), topk=topk, free=min(n, rng.randint(30, 39)))
    elif kind == "problem":
        n = rng.randint(38, 54)
        c = _solve("", n, "int", hi=logint(100, 32767), topk=topk, free=rng.randint(30, 40), resident=True)
    elif kind == "window":
        n = rng.randint(16, 38)
        c = {"call": "window", "n": n, "values": "int", "hi": 1000, "density": 0.0, "free": n,
             "window": rng.randint(50, 6000)}
    elif kind == "wide":
        inner = rng.randint(18, 34)
        c = {"call": "wide", "n": rng.randint(inner + 8, 90), "values": "int", "hi": logint(100, 3000), "density": 0.0,
             "n_inner": inner, "outer": logint(2, 40), "topk": topk}
    elif kind == "batched":
        lo = rng.randint(8, 18)
        c = {"call": "batched", "values": "mixed16", "count": logint(16, 2000), "n_lo": lo,
             "n_hi": lo + rng.randint(4, 12), "topk": rng.choice([0, 0, 4])}
    else:
        lo = rng.randint(6, 12)
        c = {"call": "graph", "values": "sk32", "count": logint(16, 1000), "n_lo": lo, "n_hi": lo + rng.randint(4, 12),
             "topk": rng.choice([0, 4])}
    c.pop("name", None)
    return c


# ---- one pass ----------------------------------------------------------------------------------


def _ptr(a: np.ndarray):
    return ctypes.c_void_p(a.ctypes.data) if a.size else None


class _BatchOutputs:
    """The result arrays a caller of the C ABI hands to a batch call, one row per instance."""

    def __init__(self, count: int, topk: int, cap: int, is_float: bool):
        energy = np.float64 if is_float else np.int64
        self.min = np.zeros(count, dtype=energy)
        self.ties = np.zeros(count * cap, dtype=np.uint64)
        self.topk = np.zeros(count * topk, dtype=np.uint64)
        self.topk_E = np.zeros(count * topk, dtype=energy)
        self.info = (q.ResultInfo * count)()

    def results(self) -> dict:
        info = np.frombuffer(self.info, dtype=np.dtype(q.ResultInfo))
        return {"min": self.min.copy(), "n_ties": info["n_ties"].astype(np.int64), "ties": self.ties.copy(),
                "topk": self.topk.copy(), "topk_E": self.topk_E.copy()}


_CAP = 16  # tie codes kept per batched instance, and returned for a single one
_WINDOW_CAP = 1 << 16  # states of an energy window kept


def _stream():
    return ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)


def _check(status: int, where: str) -> None:
    if status < 0:
        raise q.QuboError(status, where)


class _GraphBatch:
    """A device-resident batch (qubo_batch_*) with the caller's result arrays."""

    def __init__(self, mats, topk: int, is_float: bool):
        self.lib, p = q.load_library(), q.pack_batch(mats)
        self.out, self.handle = _BatchOutputs(len(p), topk, _CAP, is_float), ctypes.c_void_p()
        _check(self.lib.qubo_batch_create(_ptr(p.packed), _ptr(p.ns), _ptr(p.offs), len(p), p.dt, topk, _CAP,
                                          ctypes.byref(self.handle)), "qubo_batch_create")

    def run(self) -> dict:
        o = self.out
        _check(self.lib.qubo_batch_run(self.handle, _stream()), "qubo_batch_run")
        _check(self.lib.qubo_batch_fetch(self.handle, _ptr(o.min), _ptr(o.ties), _ptr(o.topk), _ptr(o.topk_E), o.info),
               "qubo_batch_fetch")
        return o.results()

    def __del__(self):
        if self.handle:
            self.lib.qubo_batch_destroy(self.handle)


def prepare(case: dict, seed: int) -> dict:
    call = case["call"]
    st = {"case": dict(case)}
    if call in ("batched", "graph"):
        mats = _batch(case, seed)
        is_float = case["values"] == "sk32"
        if call == "graph":
            st["batch"] = _GraphBatch(mats, case["topk"], is_float)
        else:
            st["packed"] = q.pack_batch(mats)
            st["out"] = _BatchOutputs(len(mats), case["topk"], _CAP, is_float)
        return st
    st["Q"] = _matrix(case, seed)
    if call in ("solve", "problem"):
        st["fix"] = _sub_cube(case, seed)
    if call == "problem":
        st["problem"] = q.Problem(st["Q"], topk=case["topk"])
    if call == "window":
        st["codes"], st["E"] = np.zeros(_WINDOW_CAP, dtype=np.uint64), np.zeros(_WINDOW_CAP, dtype=np.int64)
    return st


def _sub_cube(case: dict, seed: int) -> tuple:
    """The sub-cube a step scans: how many top bits are fixed, and to what."""
    fix = case["n"] - case["free"]
    return fix, int(np.random.Generator(np.random.PCG64(seed + 77)).integers(0, 1 << fix)) if fix else 0


def _first(ties) -> np.ndarray:
    """The first tie codes, in an array of one size for every instance (n_ties counts them all)."""
    out = np.zeros((_CAP,) + ties.shape[1:], dtype=ties.dtype)
    out[: min(_CAP, len(ties))] = ties[:_CAP]
    return out


def _result(r) -> dict:
    return {"min": r.min, "n_ties": r.n_ties, "ties": _first(r.ties), "topk": r.topk, "topk_E": r.topk_E}


def _words(codes) -> np.ndarray:
    """Codes beyond 64 bits as rows of (low 63 bits, the rest)."""
    return np.array([[k & (2**63 - 1), k >> 63] for k in codes], dtype=np.int64).reshape(-1, 2)


def run(state: dict):
    c = state["case"]
    call = c["call"]
    if call == "solve":
        fb, fv = state["fix"]
        return _result(q.solve(state["Q"], topk=c["topk"], fix_bits=fb, fix_value=fv))
    if call == "problem":
        p = state["problem"]
        p.run(*state["fix"])
        return _result(p.fetch())
    if call == "window":
        Q, count, codes, E = state["Q"], ctypes.c_uint64(), state["codes"], state["E"]
        _check(q.load_library().qubo_solve_window(
            _ptr(Q), c["n"], q.QUBO_I32, float(c["window"]), None, _ptr(codes), _ptr(E), _WINDOW_CAP,
            ctypes.byref(count), None, _stream()), "qubo_solve_window")
        return {"count": count.value, "codes": codes, "E": E}
    if call == "wide":
        r = q.solve_wide(state["Q"], c["n_inner"], outer_begin=_OUTER0, outer_count=c["outer"], topk=c["topk"])
        return {"min": r.min, "n_ties": r.n_ties, "ties": _first(_words(r.ties)), "topk": _words(r.topk),
                "topk_E": r.topk_E}
    if call == "batched":
        # the C ABI on arrays the caller owns (the Python wrapper adds an object per instance)
        p, o = state["packed"], state["out"]
        _check(q.load_library().qubo_solve_batched(
            _ptr(p.packed), _ptr(p.ns), _ptr(p.offs), len(p), p.dt, c["topk"], _ptr(o.min), _ptr(o.ties), _CAP,
            _ptr(o.topk), _ptr(o.topk_E), o.info, _stream()), "qubo_solve_batched")
        return o.results()
    if call == "graph":
        return state["batch"].run()
    raise ValueError(call)


# ---- what a pass cannot do without, and what it is held to ---------------------------------------

_OUTER0 = 5  # first outer value of the wide cases


def _batch_sizes(case: dict) -> list:
    lo, hi, count = case["n_lo"], case["n_hi"], case["count"]
    return [lo + (i * (hi - lo + 1)) // count for i in range(count)]


def _states(case: dict) -> int:
    call = case["call"]
    if call in ("batched", "graph"):
        return sum(1 << n for n in _batch_sizes(case))
    if call == "wide":
        return case["outer"] << case["n_inner"]
    return 1 << case["free"]


def work(case: dict) -> dict:
    call = case["call"]
    elem = 2 if case["values"] in ("int16", "maxcut", "mixed16") else 8 if case["values"] == "float64" else 4
    sizes = _batch_sizes(case) if call in ("batched", "graph") else [case["n"]]
    nbytes = sum(elem * n * n + 16 + 16 * case.get("topk", 0) for n in sizes)
    flops = 2.0 * _states(case)
    if case["values"] == "sparse":
        # variables without couplings between them separate: about 2^11 patterns of one set and 2^14
        # of the other are scored once each instead of once per combination
        flops /= 1024.0
    return {"bytes": float(nbytes), "flops": flops}


def tolerance(case: dict):
    # integer energies, and state codes throughout, are exact; float energies are FP64 sums of at
    # most n(n+1)/2 terms, which another summation order changes in the last digits (measured against
    # exact(): at most 4e-15 relative)
    return {"rel": 2e-14, "max": 2e-14, "differ": 0.0} if case["values"] in ("sk32", "float64") else "exact"


# ---- the same results in 64 bits, by plain enumeration -------------------------------------------


class _Lowest:
    """The lowest states seen so far: every state at the minimum and the K lowest."""

    def __init__(self, K: int, window: float):
        self.K, self.window = max(K, 1), window
        self.E = torch.empty(0, dtype=torch.float64, device="cuda")
        self.code = torch.empty(0, dtype=torch.int64, device="cuda")
        self.limit = float("inf")

    def add(self, E, code_of):
        """E: a block of energies; code_of(flat indices) gives their codes."""
        flat = E.reshape(-1)
        if self.limit == float("inf"):
            k = min(flat.numel(), self.K)
            self.limit = float(torch.kthvalue(flat, k).values) if flat.numel() <= 1 << 20 else \
                float(torch.topk(flat, k, largest=False).values.max())
            if self.window >= 0:
                self.limit = float(flat.min()) + self.window
        lowest = float(flat.min())
        if lowest > self.limit:
            return
        idx = torch.nonzero(flat <= self.limit).reshape(-1)
        self.E = torch.cat([self.E, flat[idx]])
        self.code = torch.cat([self.code, code_of(idx)])
        best = float(self.E.min())
        if self.window >= 0:
            limit = best + self.window
        else:
            limit = float(torch.topk(self.E, self.K, largest=False).values.max()) if len(self.E) >= self.K else \
                self.limit
        keep = self.E <= limit
        self.E, self.code, self.limit = self.E[keep], self.code[keep], limit

    def sorted(self):
        E, code = self.E.cpu().numpy(), self.code.cpu().numpy()
        order = np.lexsort((code, E))
        return E[order], code[order]


def _enumerate(Q: np.ndarray, free: int, fix_value: int, K: int, window: float = -1.0):
    """(energies, codes) of the lowest states of the sub-cube, ascending: every state's energy as
    prefix part + suffix part + their coupling, in FP64 (exact for integers below 2^53)."""
    A = torch.tensor(np.asarray(Q, dtype=np.float64), device="cuda")
    n = A.shape[0]
    U = torch.triu(A) + torch.tril(A, -1).T

    def bits(codes, k):
        return ((codes[:, None] >> torch.arange(k, device="cuda")) & 1).to(torch.float64)

    s = min(free, 13)  # suffix bits
    xs = bits(torch.arange(1 << s, device="cuda"), s)
    es = ((xs @ U[:s, :s]) * xs).sum(1)
    low = _Lowest(K, window)
    rows = 1 << max(0, min(free - s, 13))
    for p0 in range(0, 1 << (free - s), rows):
        p = torch.arange(p0, p0 + rows, device="cuda") + (fix_value << (free - s))
        xp = bits(p, n - s)
        ep = ((xp @ U[s:, s:]) * xp).sum(1)
        E = torch.addmm(ep[:, None], xp @ U[:s, s:].T, xs.T)
        E += es[None, :]
        low.add(E, lambda idx: (p[idx >> s] << s) | (idx & ((1 << s) - 1)))
    return low.sorted()


def _answer(E, code, K: int, energy) -> dict:
    ties = code[E == E[0]]
    return {"min": energy(E[0]), "n_ties": len(ties), "ties": _first(ties), "topk": code[:K],
            "topk_E": np.array([energy(e) for e in E[:K]])}


def exact(case: dict, seed: int):
    call = case["call"]
    if _states(case) > 1 << 36 or not torch.cuda.is_available():
        return None
    is_float = case["values"] in ("sk32", "float64")
    energy = float if is_float else int
    if call in ("batched", "graph"):
        if call == "batched":
            return None  # thousands of instances one by one
        mats, K = _batch(case, seed), case["topk"]
        rs = [_answer(*_enumerate(Q, Q.shape[0], 0, K), K, energy) for Q in mats]
        return {"min": np.array([r["min"] for r in rs]), "n_ties": np.array([r["n_ties"] for r in rs]),
                "ties": np.concatenate([r["ties"] for r in rs]), "topk": np.concatenate([r["topk"] for r in rs]),
                "topk_E": np.concatenate([r["topk_E"] for r in rs])}
    Q = _matrix(case, seed)
    if call == "wide":
        n, m, K = case["n"], case["n_inner"], case["topk"]
        U = np.triu(Q.astype(np.int64)) + np.tril(Q.astype(np.int64), -1).T
        found = []
        for v in range(_OUTER0, _OUTER0 + case["outer"]):
            x = np.array([(v >> f) & 1 for f in range(n - m)], dtype=np.int64)
            c = int(x @ U[m:, m:] @ x)
            E, code = _enumerate(U[:m, :m] + np.diag(U[:m, m:] @ x), m, 0, max(K, 1))
            found += [(int(e) + c, int(k) | (v << m)) for e, k in zip(E, code)]
        found.sort()
        ties = [k for e, k in found if e == found[0][0]]
        return {"min": found[0][0], "n_ties": len(ties), "ties": _first(_words(ties)), "topk": _words(k for _, k in found[:K]),
                "topk_E": np.array([e for e, _ in found[:K]], dtype=np.int64)}
    if call == "window":
        E, code = _enumerate(Q, case["free"], 0, 1, float(case["window"]))
        pad = lambda a: np.pad(a[:_WINDOW_CAP].astype(np.int64), (0, max(0, _WINDOW_CAP - len(a))))
        return {"count": len(E), "codes": pad(code), "E": pad(E)}
    K = case["topk"]
    return _answer(*_enumerate(Q, case["free"], _sub_cube(case, seed)[1], K), K, energy)
