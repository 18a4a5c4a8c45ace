"""The FP64 kernels at the sizes where they change path, through the C ABI
against the oracle: the singular value split (cluster or grid, columns in
registers or in L2, rank-deficient and tiny matrices) by the entanglement of
random MPOs, and the strided FP64 GEMM (split contraction, exchanged operands,
ragged tiles) by the transfers of xtrg_observables."""
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


def _random_mpo(dims, seed, fall):
    """Identity plus a random part whose weight falls by `fall` decades along a bond."""
    rng = np.random.default_rng(seed)
    sites = []
    for l, r in zip(dims, dims[1:]):
        wl = 10.0 ** (-fall * np.arange(l) / max(1, l - 1) / 2)
        wr = 10.0 ** (-fall * np.arange(r) / max(1, r - 1) / 2)
        w = 0.2 * rng.standard_normal((l, 2, 2, r)) * wl[:, None, None, None] * wr
        w[0, :, :, 0] += np.eye(2)
        sites.append(w)
    return sites


# bonds; decades of weight.  4 x 150 by 150 runs on the grid, 4 x 70 has
# columns longer than the registers hold, the others run in clusters.
SPLITS = [
    ([1, 1, 1], 0.0),
    ([1, 2, 3, 1], 1.0),
    ([1, 4, 5, 4, 1], 3.0),
    ([1, 4, 16, 33, 16, 4, 1], 8.0),
    ([1, 4, 16, 64, 70, 64, 16, 4, 1], 10.0),
    ([1, 4, 16, 64, 150, 150, 64, 16, 4, 1], 6.0),
]


@pytest.mark.parametrize("dims,fall", SPLITS)
@pytest.mark.parametrize("doubled", [False, True])
def test_split_sizes_by_entanglement(eng_cls, dims, fall, doubled):
    """doubled: every bond carries the state twice at half weight (a direct sum
    of the MPO with itself), so every split has half its columns dependent.
    1e-10: the bound of the entanglement tests (FP64 on both sides)."""
    from oracle import xtrg as ox
    sites = _random_mpo(dims, len(dims), fall)
    L = len(sites)
    ref = ox.mpo_entanglement(sites)
    if doubled:
        twice = []
        for i, w in enumerate(sites):
            l, r = w.shape[0], w.shape[3]
            z = np.zeros((l if i == 0 else 2 * l, 2, 2, r if i == L - 1 else 2 * r))
            z[:l, :, :, :r] += w
            z[-l:, :, :, -r:] += w
            if i == 0:
                z[:, :, :, :r], z[:, :, :, r:] = w, w
            if i == L - 1:
                z[:l], z[l:] = w, w
            twice.append(z)
        sites = twice
    eng = eng_cls.xxz(L, 1.0, 1.0, tau0=0.1, dstar=max(w.shape[3] for w in sites), sweeps=1)
    eng.set_state(sites, 0.0, 1.0, right_canonical=False)
    S = eng.entanglement()
    assert max(abs(a - b) for a, b in zip(S, ref)) <= 1e-10 * max(1.0, max(ref))
    eng.close()


@pytest.mark.parametrize("dims", [[1, 1, 1], [1, 4, 7, 1], [1, 4, 31, 33, 4, 1],
                                  [1, 4, 16, 65, 127, 64, 15, 1]])
def test_gemm_sizes_by_observables(eng_cls, dims):
    """Sums of n FP64 products differ between two orders by about n eps times
    the sum of their magnitudes; 1e-11 covers the chains used here."""
    from oracle import hamiltonian as oh
    from oracle import xtrg as ox
    sites = _random_mpo(dims, 7, 3.0)
    L = len(sites)
    H = oh.xxz_chain_mpo(L, 1.0, 0.7)
    tr = ox.trace(sites)
    e1, e2 = ox.trace_H_rho(H, sites) / tr, ox.trace_H2_rho(H, sites) / tr
    eng = eng_cls.xxz(L, 1.0, 0.7, tau0=0.1, dstar=max(dims), sweeps=1)
    eng.set_state(sites, 0.25, 2.0, right_canonical=False)
    o = eng.observables()
    assert abs(o["lnZ"] - 0.25 - np.log(tr)) <= 1e-11
    assert abs(o["u"] - e1 / L) <= 1e-11 * max(1.0, abs(e1))
    assert abs(o["c"] - 4.0 * (e2 - e1 * e1) / L) <= 1e-11 * max(1.0, abs(e2))
    ratio = ox.trace_rho_rho(sites) / ox.frobenius2(sites)
    assert abs(o["herm_defect"] ** 2 - (2.0 - 2.0 * ratio)) <= 1e-11
    eng.close()
