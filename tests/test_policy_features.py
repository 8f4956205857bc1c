"""The policy's features bit by bit: the engine's warps and the host function
share one formula, whose roundings are those of its printed form in single
precision (a scale by a power of two is exact wherever it stands)."""
import numpy as np
import pytest

import paper_1903_12085_gb300 as sp

F = np.float32


def printed(nF, n, m, k, e, s, f):
    nF, n, m, k, e, s, f = (F(v) for v in (nF, n, m, k, e, s, f))
    log = lambda x: F(np.log2(np.float64(x)))  # (correctly rounded, which the host's log2f is to within an ulp)
    return [log(F(1) + nF) / F(24), nF / n, log(F(1) + e) / F(24), log(F(1) + s) / F(24), log(F(1) + k) / F(16),
            log(n) / F(32), (m / n) / F(32), s / (F(1) + f)]


def test_features_as_printed():
    rng = np.random.default_rng(7)
    for _ in range(2000):
        n = int(2 ** rng.uniform(0, 31)) or 1
        args = [int(2 ** rng.uniform(0, 31)) - 1 for _ in range(6)]
        case = (args[0], n, args[1], *args[2:])
        got, want = sp.policy_features(*case), np.array(printed(*case), np.float32)
        exact = [1, 6, 7]  # no logarithm: one rounding per operation on both sides
        assert (got[exact] == want[exact]).all(), case
        assert (np.abs(got - want) <= 4 * np.spacing(np.abs(want))).all(), case
