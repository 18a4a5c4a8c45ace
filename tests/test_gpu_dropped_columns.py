"""Columns that the tensor-core truncation drops as numerically dependent."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _random_state(L, D, seed, fall):
    """Random sites whose weight falls along each bond: bases with columns of
    every degree of dependence."""
    r = np.random.default_rng(seed)
    b = [min(D, 4 ** min(i, L - i)) for i in range(L + 1)]
    sites = []
    for i in range(L):
        w = r.standard_normal((b[i], 2, 2, b[i + 1])) * np.exp(-fall * np.arange(b[i + 1]))
        sites.append(w / np.linalg.norm(w))
    return sites


def test_second_pass_drops_no_more_than_rounding():
    """A column dropped in the second orthonormalisation pass is a bond
    direction lost, for good in the last sweep.  The count to meet, 7442 over
    these 100 doublings of one sweep, was taken when Gram-Schmidt still
    completed every basis that failed the second pass, so that only the first
    pass dropped columns.  Two codes with that rule differ by the rounding of
    pivots at the threshold: by 2.6 columns a doubling (standard deviation, 400
    of them), 26 over 100; three times that is the allowance."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1801_00142_gb300.build import build
    build()
    from paper_1801_00142_gb300.engine import XTRG
    dropped = fallbacks = 0
    for D in (90, 128):
        for fall in (0.3, 0.5):
            for seed in range(100, 125):
                # a context of its own each: the noise is drawn from a seed that it counts up
                eng = XTRG.xxz(8, 1.0, 0.7, tau0=2.0 ** -4, dstar=D, sweeps=1, prec="bf16x6")
                eng.set_state(_random_state(8, D, seed, fall), 0.0, 1.0)
                eng.double()
                c = eng.counters()
                dropped += c["orth_deflated_columns"]
                fallbacks += c["exact_split_fallbacks"]
                eng.close()
    print("dropped", dropped, "exact splits", fallbacks)
    assert dropped <= 7442 + 78
    assert fallbacks <= 2
