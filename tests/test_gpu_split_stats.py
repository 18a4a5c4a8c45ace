"""The split's flop count of xtrg_get_stats follows the algorithm that runs:
pivoted QR, Jacobi sweeps over its columns, the projection and its correction."""
import pytest

pytestmark = pytest.mark.gpu


def test_split_flops_of_a_two_site_chain():
    """L = 2 with full-rank sites: one doubling of one sweep splits a 4 x 4
    matrix of rank 4 twice.  Each costs 6 * 4 * (4 * 4 - 10) for the QR, 6 pairs
    * 8 * 4 a sweep, 2 * 4 * 4 * 4 each for the projection and the Gram of the
    isometry and 4 * 4 * 3 for its lower part; only the number of sweeps is not
    known beforehand."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import numpy as np
    from paper_1801_00142_gb300.build import build
    build()
    from paper_1801_00142_gb300.engine import XTRG
    r = np.random.default_rng(5)
    sites = [r.standard_normal((1, 2, 2, 4)),
             np.linalg.qr(r.standard_normal((4, 4)))[0].reshape(4, 2, 2, 1)]
    eng = XTRG.xxz(2, 1.0, 0.7, tau0=2.0 ** -4, dstar=4, sweeps=1)
    eng.set_state(sites, 0.0, 1.0, right_canonical=True)
    before = eng.counters()
    eng.double()
    after = eng.counters()
    assert eng.observables()["max_bond"] == 4
    eng.close()
    assert after["two_site_updates"] - before["two_site_updates"] == 2
    sweeps = (after["split_flops"] - before["split_flops"] - 2 * (144 + 128 + 128 + 48)) / 192.0
    assert sweeps == int(sweeps)
    assert 2 <= sweeps <= 2 * 60
