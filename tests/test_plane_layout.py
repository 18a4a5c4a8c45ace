"""Layout of the tensor-core operands' BF16 planes: the strides that the
conversion writes with and the GEMM reads with are formed in 64 bits.  A host
check: the header that forms them is compiled with the host compiler."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1801_00142_gb300", "csrc")

MAIN = r"""
#include <stdio.h>
#include <stdlib.h>
#include "plane_layout.h"
int main(int argc, char** argv) {
  for (int i = 1; i + 2 < argc; i += 3) {
    const PlaneLayout p = plane_layout(atoi(argv[i]), atoi(argv[i + 1]), atoi(argv[i + 2]));
    printf("%lld %lld %lld\n", p.ld, p.batch_stride, p.plane_stride);
  }
}
"""

# rows, columns, batch; the last three pass 2^31 in batch * rows, in the matrix
# and in rows * ld
SIZES = [(1, 1, 1), (60, 52, 1), (250, 201, 33), (7, 8, 5), (32769, 1, 65535), (46341, 46341, 1),
         (2147483647, 8, 1)]


def test_plane_strides_are_formed_in_64_bits(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "layout.cpp", tmp_path / "layout"
    src.write_text(MAIN)
    subprocess.run([cxx, "-std=c++17", "-Wall", "-Werror", "-fsanitize=undefined",
                    "-fno-sanitize-recover", f"-I{CSRC}", str(src), "-o", str(exe)], check=True)
    args = [str(x) for s in SIZES for x in s]
    out = subprocess.run([str(exe), *args], check=True, capture_output=True, text=True).stdout
    got = [tuple(int(x) for x in line.split()) for line in out.splitlines()]
    want = []
    for rows, cols, batch in SIZES:
        ld = (cols + 7) // 8 * 8
        want.append((ld, rows * ld, batch * rows * ld))
    assert got == want


@pytest.mark.parametrize("nn", [False, True])
@pytest.mark.parametrize("M,N,K,batch,planes", [(60, 44, 52, 1, 3), (250, 330, 201, 33, 2),
                                                (32769, 1, 1, 65535, 2), (1, 1, 32769, 65535, 2)])
def test_scratch_holds_the_planes_of_that_layout(nn, M, N, K, batch, planes):
    """The workspace of a call is at least its two operands' planes, partials
    and error flag, at sizes that no 32-bit product can hold too."""
    from paper_1801_00142_gb300.build import build
    build()
    from paper_1801_00142_gb300 import _lib

    def up8(x):
        return (x + 7) // 8 * 8

    a = planes * batch * M * up8(K) * 2
    b = planes * batch * (K * up8(N) if nn else N * up8(K)) * 2
    size = _lib.xtrg_tc_gemm_nn_workspace_bytes if nn else _lib.xtrg_tc_gemm_workspace_bytes
    n = size(M, N, K, batch, planes, 1)
    need = a + b + batch * M * N * 4 + 4
    assert need <= n < need + 4 * 256


REFUSE = r"""
#include <stdio.h>
#include "mixed_ops.cu"
unsigned long long g_xtrg_launches;
thread_local unsigned long long t_xtrg_launches;
int main() {
  struct { size_t out; long long ld, obs, ops; } c[] = {
      {256, 9, 0, 96}, {256, 16, 56, 196}, {256, 16, 60, 192}, {264, 16, 64, 192}};
  const Idx3 u = idx_plain(1), w = idx_plain(9);
  for (auto& x : c) {
    __nv_bfloat16* out = (__nv_bfloat16*)x.out;
    printf("%d %d %d\n",
           (int)to_planes((const double*)256, w, u, 36, 4, 9, 3, out, x.ld, x.obs, 2, x.ops, 0),
           (int)to_planes_f32((const float*)256, w, u, 36, 4, 9, 3, out, x.ld, x.obs, 2, x.ops, 0),
           x.obs ? 1 : (int)to_planes_if((const double*)256, w, u, 4, 9, out, x.ld, 2, x.ops,
                                         (const double*)256, 0.0, 0));
  }
}
"""


def test_unaligned_plane_layouts_are_refused(tmp_path):
    """A thread stores eight columns at a time, so a row stride, batch stride,
    plane stride or start that is no multiple of 16 bytes would write past the
    rows: the host refuses it (cudaErrorInvalidValue = 1), nothing is launched."""
    from paper_1801_00142_gb300.build import ARCH, nvcc
    try:
        cc = nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    src, exe = tmp_path / "refuse.cu", tmp_path / "refuse"
    src.write_text(REFUSE)
    subprocess.run([cc, *ARCH, "-std=c++17", "-cudart", "shared", f"-I{CSRC}", str(src), "-o", str(exe),
                    "-Xlinker", "-rpath,/usr/local/cuda/lib64"], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, check=True)
    assert r.stdout.split() == ["1"] * 12
