"""xtrg_tc_gemm on large batches of small matrices: their rows share conversion
tiles, and few ragged rows take their FP64 values through partial sums."""
import pytest

pytestmark = pytest.mark.gpu


def _call(torch, lib, A, B, nn, planes, nprod):
    b, M, K = A.shape
    N = B.shape[2] if nn else B.shape[1]
    size = lib.xtrg_tc_gemm_nn_workspace_bytes if nn else lib.xtrg_tc_gemm_workspace_bytes
    n = size(M, N, K, b, planes, 1)
    ws = torch.empty(n + 256, dtype=torch.uint8, device="cuda")
    C = torch.full((b, M, N), float("nan"), dtype=torch.float64, device="cuda")
    f = lib.xtrg_tc_gemm_nn if nn else lib.xtrg_tc_gemm
    f(A.data_ptr(), B.data_ptr(), C.data_ptr(), M, N, K, b, planes, nprod, 1,
      (ws.data_ptr() + 255) // 256 * 256, n, torch.cuda.current_stream().cuda_stream)
    return C


@pytest.mark.parametrize("M,N,K,batch", [(1, 1, 1, 700), (5, 300, 7, 250), (32, 33, 9, 650), (32, 64, 8, 650),
                                         (31, 130, 40, 310), (33, 33, 33, 610), (3, 5, 2049, 620)])
@pytest.mark.parametrize("nn", [False, True])
@pytest.mark.parametrize("planes,nprod,bits", [(3, 6, 22), (2, 3, 15)])
def test_batches_of_small_matrices(M, N, K, batch, nn, planes, nprod, bits):
    """Bounds of the split (24 and 16 bits, a factor of two or four for the
    dropped products), and each matrix's values bit for bit those of a call with
    fewer of them, which takes the other route."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1801_00142_gb300.build import build
    build()
    from paper_1801_00142_gb300 import _lib
    g = torch.Generator(device="cuda").manual_seed(M + 1000 * N + K)
    kw = dict(generator=g, device="cuda", dtype=torch.float64)
    A = torch.randn(batch, M, K, **kw)
    B = torch.randn(batch, K, N, **kw) if nn else torch.randn(batch, N, K, **kw)
    C = _call(torch, _lib, A, B, nn, planes, nprod)
    Bt = B if nn else B.transpose(1, 2)
    assert bool(((C - A @ Bt).abs() <= 2.0 ** -bits * (A.abs() @ Bt.abs())).all())
    few = torch.tensor([0, 1, batch // 2, batch - 1], device="cuda")
    D = _call(torch, _lib, A[few].contiguous(), B[few].contiguous(), nn, planes, nprod)
    assert bool((C[few] == D).all())
