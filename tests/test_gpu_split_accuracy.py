"""Accuracy of the FP64 split's factors: singular directions far below the
leading one keep their own relative accuracy."""
import math
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def eng_cls():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1801_00142_gb300.build import build
    build()
    from paper_1801_00142_gb300.engine import XTRG
    return XTRG


def _trace_moments(L, Delta, n):
    """Tr H^q for q = 0..n as exact fractions (H times 16 has integer entries)."""
    from oracle import hamiltonian as oh
    H = oh.dense_xxz(L, 1.0, Delta) * 16
    assert np.array_equal(H, np.rint(H))
    H = H.astype(int).astype(object)   # Python integers: no overflow, no rounding
    P, out = np.eye(len(H), dtype=int).astype(object), []
    for q in range(n + 1):
        out.append(Fraction(int(np.trace(P)), 16 ** q))
        P = P.dot(H)
    return out


@pytest.mark.parametrize("L", [4, 6])
def test_series_energy_at_small_tau(eng_cls, L):
    """The series state at tau0 is the identity plus tau0 H plus ever smaller
    terms, each in bond directions of its own.  Its energy is a ratio of the
    part of weight tau0 to the leading one: an error of 2.2e-16 of the
    norm put into those directions shows as 2.2e-16 / tau0 (1.5e-8 at 2^-26).
    With every direction right to its own rounding the energy is right to the
    rounding of the contractions behind it, fewer than 2^12 operations deep:
    2^12 * 2.2e-16 < 1e-12, whatever tau0."""
    Delta, order = 0.75, 4
    m = _trace_moments(L, Delta, order + 1)
    for k in (8, 14, 20, 26, 32):
        tau = Fraction(1, 2 ** k)
        t = [sum((-tau) ** j / math.factorial(j) * m[j + q] for j in range(order + 1))
             for q in range(2)]
        u = float(t[1] / t[0] / L)
        eng = eng_cls.xxz(L, 1.0, Delta, tau0=2.0 ** -k, dstar=64, sweeps=2, order=order)
        eng.init()
        g = eng.observables()["u"]
        eng.close()
        assert abs(g - u) <= 1e-12 * abs(u), (k, g, u)
