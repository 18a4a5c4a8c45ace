"""The tensor-core truncation at the edges of its tiles and blocks: one
doubling in split-BF16 arithmetic against the same doubling in FP64, from the
same state, for bond dimensions around the 32-wide panels, the 128-wide
product tiles and one column block (256, or 32 with orth_block set, beyond
which the orthonormalisation runs block by block)."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dstar,orth_block", [(7, 0), (31, 0), (33, 0), (64, 32), (65, 0), (127, 0),
                                              (129, 0), (200, 0), (256, 0)])
@pytest.mark.parametrize("keep_parts", [True, False])
def test_doubling_matches_fp64(dstar, orth_block, keep_parts):
    """Bounds: the arithmetic's 2e-6 of ln Z (the smoke bound), and where D*
    cuts the spectrum what the cut discards: each of the L - 1 bonds of either
    path loses at most trunc_err of the weight, which moves ln Z by that much
    and the energy per site by its square root at most."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1801_00142_gb300.build import build
    build()
    from paper_1801_00142_gb300.engine import XTRG
    L = 9
    ref = XTRG.xxz(L, 1.0, 0.7, tau0=2.0 ** -4, dstar=dstar, sweeps=3)
    ref.init()
    for _ in range(3):
        ref.double()
    sites, lnc, beta = ref.get_state()
    mix = XTRG.xxz(L, 1.0, 0.7, tau0=2.0 ** -4, dstar=dstar, sweeps=3, prec="bf16x6",
                   keep_parts=keep_parts, orth_block=orth_block)
    mix.set_state(sites, lnc, beta, right_canonical=True)
    ref.double()
    for _ in range(2):   # the second pass over the same state may replay a graph
        mix.set_state(sites, lnc, beta, right_canonical=True)
        mix.double()
        g, o = mix.observables(), ref.observables()
        cut = (L - 1) * (g["trunc_err"] + o["trunc_err"])
        assert abs(g["lnZ"] - o["lnZ"]) <= 2e-6 * max(1.0, abs(o["lnZ"])) + 2.0 * cut
        assert abs(g["u"] - o["u"]) <= 1e-5 + cut ** 0.5
    ref.close()
    mix.close()


@pytest.mark.parametrize("dstar", [15, 33, 64, 97, 173])
@pytest.mark.parametrize("keep_parts", [True, False])
def test_three_product_doubling_matches_fp64(dstar, keep_parts):
    """The three-product kernels (another division of the tile among the
    epilogue's warps), bonds on either side of their 16- and 32-column pieces.
    Bound: an operand of two BF16 planes is right to 2^-17 and the dropped
    product of the low planes is smaller, so each of the four contractions of a
    site moves ln Z by 2^-17 at most per operand pair, and the energy by twice
    that (numerator and denominator); the cut as above."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1801_00142_gb300.build import build
    build()
    from paper_1801_00142_gb300.engine import XTRG
    L = 9
    arith = 4 * L * 2.0 ** -17 * 2
    ref = XTRG.xxz(L, 1.0, 0.7, tau0=2.0 ** -4, dstar=dstar, sweeps=2)
    ref.init()
    for _ in range(3):
        ref.double()
    sites, lnc, beta = ref.get_state()
    mix = XTRG.xxz(L, 1.0, 0.7, tau0=2.0 ** -4, dstar=dstar, sweeps=2, prec="bf16x3",
                   keep_parts=keep_parts)
    mix.set_state(sites, lnc, beta, right_canonical=True)
    ref.double()
    mix.double()
    g, o = mix.observables(), ref.observables()
    cut = (L - 1) * (g["trunc_err"] + o["trunc_err"])
    assert abs(g["lnZ"] - o["lnZ"]) <= arith + 2.0 * cut
    assert abs(g["u"] - o["u"]) <= 2 * arith + cut ** 0.5
    ref.close()
    mix.close()
