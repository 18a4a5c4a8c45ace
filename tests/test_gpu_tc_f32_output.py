"""FP32 output of the tensor-core GEMM (the products of truncations of bonds of
about 560 and more): 16-byte stores where a row's columns are contiguous and
aligned, single ones otherwise.  The GEMM is an internal function of the
library, reached through a few lines of C++ compiled here."""
import ctypes as C
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_1801_00142_gb300")

ENTRY = r"""
#include <string.h>
#include "mixed_ops.cuh"
#include "tc_gemm.cuh"
// C = A B^T (row-major FP64 A: M x K, B: N x K), element (m, n) at m * sm + n * sn
extern "C" int gemm_f32(const double* A, const double* B, int M, int N, int K, __nv_bfloat16* pa,
                        __nv_bfloat16* pb, float* C, long long sm, long long sn, int* err) {
  const long long ld = tc_ld(K), psa = M * ld, psb = N * ld;
  cudaError_t e = to_planes(A, idx_plain(K), idx_plain(1), 0, M, K, 1, pa, ld, 0, 3, psa, 0);
  if (e == cudaSuccess) e = to_planes(B, idx_plain(K), idx_plain(1), 0, N, K, 1, pb, ld, 0, 3, psb, 0);
  if (e != cudaSuccess) return (int)e;
  TcOutput o;
  memset(&o, 0, sizeof o);
  o.mode = TC_OUT_F32;
  o.f32 = C;
  o.cm = idx_plain(sm);
  o.cn = idx_plain(sn);
  o.alpha = 1.0;
  const TcOperand a{pa, 3, M, K, ld, 0, psa, 1}, b{pb, 3, N, K, ld, 0, psb, 1};
  e = tc_gemm(a, b, M, N, K, 1, 6, 1, o, err, 0);
  return (int)(e != cudaSuccess ? e : cudaDeviceSynchronize());
}
"""


@pytest.fixture(scope="module")
def gemm(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1801_00142_gb300.build import ARCH, build, nvcc
    lib = build()
    d = tmp_path_factory.mktemp("tcf32")
    src, so = d / "entry.cu", d / "entry.so"
    src.write_text(ENTRY)
    subprocess.run([nvcc(), *ARCH, "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-cudart", "shared",
                    f"-I{PKG}/csrc", str(src), lib, "-o", str(so),
                    "-Xlinker", f"-rpath,{PKG}", "-Xlinker", "-rpath,/usr/local/cuda/lib64"], check=True)
    return C.CDLL(str(so)).gemm_f32


# ldc: rows aligned to 16 bytes or not; start: of the output; columns strided last
@pytest.mark.parametrize("M,N,K,ldc,start,sn", [
    (1, 1, 16, 1, 0, 1), (130, 32, 64, 32, 0, 1), (257, 128, 100, 132, 0, 1), (300, 200, 130, 200, 0, 1),
    (129, 161, 72, 161, 0, 1), (200, 96, 64, 100, 4, 1), (200, 96, 64, 100, 3, 1), (140, 65, 80, 150, 0, 2)])
def test_f32_output_forms(gemm, M, N, K, ldc, start, sn):
    """Six products of three planes each are right to 2^-23 of sum |a b| (24-bit
    operands, FP32 accumulation in steps); entries between the rows stay as they were."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(M * 1000 + N)
    kw = dict(dtype=torch.float64, device="cuda")
    A, B = (torch.randn(r, K, generator=g, **kw) for r in (M, N))
    ld = (K + 7) // 8 * 8
    pa, pb = (torch.empty(3 * r * ld, dtype=torch.bfloat16, device="cuda") for r in (M, N))
    row = max(ldc, N * sn)
    out = torch.full((start + M * row + 8,), -7.0, dtype=torch.float32, device="cuda")
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    P = C.c_void_p
    torch.cuda.synchronize()
    e = gemm(P(A.data_ptr()), P(B.data_ptr()), M, N, K, P(pa.data_ptr()), P(pb.data_ptr()),
             P(out.data_ptr() + 4 * start), C.c_longlong(row), C.c_longlong(sn), P(err.data_ptr()))
    assert e == 0 and int(err[0]) == 0
    body = out[start:start + M * row].reshape(M, row)
    got = body[:, :N * sn:sn].double()
    bound = 2.0 ** -23 * 2 * (A.abs() @ B.abs().T)
    assert bool(((got - A @ B.T).abs() <= bound).all())
    body[:, :N * sn:sn] = -7.0
    assert bool((out == -7.0).all())
