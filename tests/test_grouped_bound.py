"""The lower bound behind the grouped step form, restated in numpy and checked by brute force (no
GPU).  A unit's columns are walked in reflected Gray order in groups of 16 states, over which a
column takes its value with the register rows 0-3 clear plus every subset of the four.  First test:
with m the thread's exact column minimum at the group's first state and D the smallest of its
columns' offsets (the rows' negative parts, less row 3 where the group starts with it set), no
column falls below m + D.  Second test: each column with its own offset, the exact minimum.  E_L's
group minimum completes both.  A wrong sign pattern, a dropped coupling to the fixed bits or an
offset of the wrong parity fails these checks."""
import os
import subprocess

import numpy as np
import pytest

from paper_2607_04857_gb300 import workloads as wl

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def columns_over_walk(U, B, L, fixed):
    """Column values col[i, j] (suffix pattern j, walk step i) and E_L(i) of one unit: the state's
    energy is col + E_L + const, col holding every term with a suffix variable."""
    n = U.shape[0]
    S = U + U.T - np.diag(np.diag(U))
    steps = 1 << L
    col = np.zeros((steps, 1 << B), dtype=np.int64)
    el = np.zeros(steps, dtype=np.int64)
    for i in range(steps):
        g = i ^ (i >> 1)
        x = np.zeros(n, dtype=np.int64)
        for r in range(L):
            x[B + r] = (g >> r) & 1
        x[B + L:] = fixed
        base = x @ U @ x
        for j in range(1 << B):
            y = x.copy()
            y[:B] = [(j >> b) & 1 for b in range(B)]
            col[i, j] = y @ U @ y - base
        walked = np.zeros(n, dtype=np.int64)
        walked[B:B + L] = x[B:B + L]
        el[i] = walked @ U @ walked
    return col, el, S


def offsets(M, w, par):
    """A column's group minimum less its value at the group's first state: register rows r = 0..3 move
    column j by +-(M[r, j] + w[r]), and groups of odd index start with row 3 set."""
    rows = M + w[:, None]
    return np.minimum(rows, 0).sum(axis=0) - (rows[3] if par else 0)


@pytest.mark.parametrize("seed", range(4))
def test_group_bound_holds_by_brute_force(seed):
    n, B, L = 12, 3, 6  # 8 columns, 64 walk steps = 4 groups of 16, 3 fixed bits
    U = np.triu(wl.upper_int(n, -50, 50, seed=seed).astype(np.int64))
    rng = np.random.default_rng(seed)
    fixed = rng.integers(0, 2, n - B - L)
    col, el, S = columns_over_walk(U, B, L, fixed)
    # register row r: M[r, j] = sum of U over the suffix bits set in j, w[r] = coupling to the set
    # fixed bits (the kernel folds it into the row)
    M = np.array([[sum(S[b, B + r] for b in range(B) if (j >> b) & 1) for j in range(1 << B)] for r in range(4)])
    w = np.array([S[B + r, B + L:] @ fixed for r in range(4)])
    # the kernel's columns carry the fixed-bit couplings of the set register rows (the rest of the
    # prefix energy, constant within a group, sits in the threshold)
    steps = np.arange(1 << L)
    gray = steps ^ (steps >> 1)
    col = col + sum(((gray >> r) & 1) * w[r] for r in range(4))[:, None]
    # the row moves every column exactly as the walk does
    for i in range(1, 1 << L):
        kk = (i & -i).bit_length() - 1
        if kk < 4:
            sign = -1 if (i >> (kk + 1)) & 1 else 1
            assert np.array_equal(col[i] - col[i - 1], sign * (M[kk] + w[kk]))
    for g in range(col.shape[0] // 16):
        group, off = col[16 * g:16 * g + 16], offsets(M, w, g & 1)
        assert np.array_equal(group[0] + off, group.min(axis=0))  # the second test
        m, D = group[0].min(), off.min()  # the first
        assert m + D <= group.min()
        # the test: no state of the group is at or below u when m + D > u - min E_L
        emin = (group + el[16 * g:16 * g + 16, None]).min()
        assert m + D + el[16 * g:16 * g + 16].min() <= emin


def test_group_bound_is_tight_for_one_column():
    """With a single column m + D is the column's exact minimum over the group, for either sign of
    row 3."""
    M = np.array([[5], [-7], [3], [-2]])
    w = np.array([1, 2, -4, 0])
    for par in (0, 1):
        walk = [0]
        for t in range(1, 16):
            kk = (t & -t).bit_length() - 1
            neg = par if kk == 3 else (t >> (kk + 1)) & 1
            walk.append(walk[-1] + (-1 if neg else 1) * (M[kk, 0] + w[kk]))
        assert offsets(M, w, par).min() == min(walk)


@pytest.mark.parametrize("seed", range(3))
def test_exact_group_minimum(seed):
    """The second test's bound: a column's minimum over a group is its value with rows 0-3 clear plus
    the negative parts of the four rows (rows 0-2 are clear and row 3 follows the group's parity at
    the group's first state)."""
    rng = np.random.default_rng(seed)
    rows, start = rng.integers(-50, 51, size=(4, 8)), rng.integers(-300, 300, size=8)
    for par in (0, 1):
        base = start  # rows 0-3 clear
        first = base + par * rows[3]
        col, least = first.copy(), first.copy()
        for t in range(1, 16):
            kk = (t & -t).bit_length() - 1
            neg = bool(par) if kk == 3 else bool((t >> (kk + 1)) & 1)
            col = col + (-1 if neg else 1) * rows[kk]
            least = np.minimum(least, col)
        assert np.array_equal(least, first - par * rows[3] + np.minimum(rows, 0).sum(axis=0))


@pytest.mark.parametrize("seed", range(3))
def test_smallest_offset_bounds_every_column(seed):
    """The first test's bound: m + D, D the smallest over a thread's columns of the offset between a
    column's group minimum and its value at the group's first state, is at or below every column in the
    group."""
    rng = np.random.default_rng(100 + seed)
    rows, start = rng.integers(-80, 81, size=(4, 16)), rng.integers(-400, 400, size=16)
    for par in (0, 1):
        first = start + par * rows[3]
        D = offsets(rows, np.zeros(4, dtype=np.int64), par).min()
        least = min((start + sum(((p >> r) & 1) * rows[r] for r in range(4))).min() for p in range(16))
        assert first.min() + D <= least


def test_kept_rows_add_without_signed_overflow(tmp_path):
    """A register row kept divided by kMad comes back as the plain row, in arithmetic that is defined for
    every 32-bit word: signed overflow traps here."""
    src = tmp_path / "rows.cpp"
    src.write_text("""
#include "internal.h"
using namespace qubo;
int main()
{
    uint32_t s = 12345;
    for (int i = 0; i < 100000; ++i) {
        s = s * 1664525u + 1013904223u;
        const int32_t row = (int32_t)s >> (2 + i % 28), x = (int32_t)(s * 2654435761u) >> (2 + i % 5);
        const int32_t kept = (int32_t)((uint32_t)row * kMadInverse);
        for (int32_t sign = -1; sign <= 1; ++sign)
            if (add_kept_row<int32_t>(x, sign, (int32_t)kMad, kept) != x + sign * row ||
                add_kept_row<int32_t>(x, sign, 1, row) != x + sign * row)
                return 1;
        if (add_kept_row<float>(0.5f, -1.0f, 1.0f, 3.0f) != -2.5f)
            return 2;
    }
    return 0;
}
""")
    csrc = os.path.join(ROOT, "paper_2607_04857_gb300", "csrc")
    exe = str(tmp_path / "rows")
    subprocess.run(["g++", "-std=c++20", "-O1", "-fsanitize=signed-integer-overflow", "-fsanitize-undefined-trap-on-error",
                    "-I", csrc, "-I", os.path.join(ROOT, "include"), "-I", "/usr/local/cuda/include", str(src), "-o", exe],
                   check=True)
    assert subprocess.run([exe]).returncode == 0
