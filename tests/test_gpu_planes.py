"""The conversion of FP64 operands to BF16 planes at the edges of its tiles
(32 rows x 64 columns) and of its integer path (values below 2^-74 convert in
FP64), through xtrg_tc_gemm and xtrg_tc_gemm_nn against FP64 numpy.  The bound
is the one of the contraction's own test for six products."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("power", [-80, -70, 0, 60])
@pytest.mark.parametrize("M,N,K", [(31, 33, 7), (32, 64, 64), (65, 1, 65), (1, 130, 200)])
@pytest.mark.parametrize("nn", [False, True])
def test_planes_of_any_size_and_magnitude(M, N, K, power, nn):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1801_00142_gb300.build import build
    build()
    from paper_1801_00142_gb300 import _lib as lib
    rng = np.random.default_rng(M + 3 * N + 5 * K)
    A = np.ldexp(rng.standard_normal((2, M, K)), power)
    A[:, 0, 0] = 0.0
    B = rng.standard_normal((2, K, N) if nn else (2, N, K))
    ref = np.einsum("bmk,bkn->bmn" if nn else "bmk,bnk->bmn", A, B)
    scale = np.einsum("bmk,bkn->bmn" if nn else "bmk,bnk->bmn", np.abs(A), np.abs(B))
    size = lib.xtrg_tc_gemm_nn_workspace_bytes if nn else lib.xtrg_tc_gemm_workspace_bytes
    call = lib.xtrg_tc_gemm_nn if nn else lib.xtrg_tc_gemm
    dA, dB = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
    dC = torch.zeros((2, M, N), dtype=torch.float64, device="cuda")
    n = size(M, N, K, 2, 3, 1)
    ws = torch.empty(n + 256, dtype=torch.uint8, device="cuda")
    call(dA.data_ptr(), dB.data_ptr(), dC.data_ptr(), M, N, K, 2, 3, 6, 1,
         (ws.data_ptr() + 255) // 256 * 256, n, torch.cuda.current_stream().cuda_stream)
    assert np.all(np.abs(dC.cpu().numpy() - ref) <= 2e-6 * scale)
