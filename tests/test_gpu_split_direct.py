"""The FP64 split called directly, on matrices of chosen spectrum: what is kept
where kcap cuts, against numpy's singular value decomposition.  The entry is an
internal function of the library, reached through a few lines of C++ compiled
here."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_1801_00142_gb300")
EPS = 2.220446049250313e-16

ENTRY = r"""
#include "common.cuh"
// b: W, V, nrm, sig, stats (device doubles); w: perm, counter, kept (device ints)
extern "C" int split_entry(const double* M, int m, int n, int kcap, int mode, double* left,
                           double* right, double* const* b, int* const* w, size_t max_elems,
                           int max_cols, double* out) {
  SvdBuffers s{};
  s.W = b[0]; s.V = b[1]; s.nrm = b[2]; s.sig = b[3]; s.stats = b[4];
  s.perm = w[0]; s.counter = w[1]; s.kept = w[2];
  s.max_elems = max_elems;
  s.max_cols = max_cols;
  SvdResult r{};
  bool ok = false;
  const cudaError_t e = svd_split_f64(M, m, n, kcap, 1e-15, (SplitMode)mode, left, right, s, 0, &r, &ok);
  out[0] = r.k;
  out[1] = r.discarded;
  out[2] = r.sigma_max;
  out[3] = ok;
  return (int)e;
}
"""


@pytest.fixture(scope="module")
def split(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1801_00142_gb300.build import ARCH, build, nvcc
    lib = build()
    d = tmp_path_factory.mktemp("split")
    src, so = d / "entry.cu", d / "entry.so"
    src.write_text(ENTRY)
    subprocess.run([nvcc(), *ARCH, "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-cudart", "shared",
                    f"-I{PKG}/csrc", str(src), lib, "-o", str(so),
                    "-Xlinker", f"-rpath,{PKG}", "-Xlinker", "-rpath,/usr/local/cuda/lib64"], check=True)
    fn = C.CDLL(str(so)).split_entry

    def run(M, kcap, mode):
        """(left, right, discarded fraction, sigma_max); mode 0: left is the isometry."""
        m, n = M.shape
        f = dict(dtype=torch.float64, device="cuda:0")
        i = dict(dtype=torch.int32, device="cuda:0")
        cols, elems = max(m, n), max(m, n) ** 2
        Md = torch.from_numpy(np.ascontiguousarray(M)).cuda()
        left, right = torch.empty(m * kcap, **f), torch.empty(kcap * n, **f)
        bufs = [torch.empty(s, **f) for s in (elems, elems, 2 * cols, cols, 8)]
        words = [torch.empty(s, **i) for s in (cols, 8, 4)]
        P = C.c_void_p
        out = (C.c_double * 4)()
        torch.cuda.synchronize()
        e = fn(P(Md.data_ptr()), m, n, kcap, mode, P(left.data_ptr()), P(right.data_ptr()),
               (P * 5)(*[b.data_ptr() for b in bufs]), (P * 3)(*[w.data_ptr() for w in words]),
               C.c_size_t(elems), cols, out)
        assert e == 0 and out[3] == 1.0
        k = int(out[0])
        return (left[:m * k].reshape(m, k).cpu().numpy(), right[:k * n].reshape(k, n).cpu().numpy(),
                out[1], out[2])

    return run


def _matrix(n, s, seed):
    r = np.random.default_rng(seed)
    U = np.linalg.qr(r.standard_normal((n, n)))[0]
    V = np.linalg.qr(r.standard_normal((n, n)))[0]
    return (U * s) @ V.T


def _check(M, k, mode, split):
    """Kept weight, isometry and kept matrix.  With n rows a backward stable
    split is exact for a matrix n eps sigma_1 away: the kept subspace turns by
    twice that over the gap at the cut, and the kept matrix changes by no more
    than that times sigma_k <= sigma_1."""
    n = M.shape[0]
    u, s, vt = np.linalg.svd(M)
    left, right, disc, smax = split(M, k, mode)
    X = left if mode == 0 else right.T
    assert X.shape == (n, k)
    # cosines below sqrt(n) eps each
    assert np.linalg.norm(X.T @ X - np.eye(k)) <= 2 * k * np.sqrt(n) * EPS
    assert abs(smax - s[0]) <= n * EPS * s[0]
    tail, total = (s[k:] ** 2).sum(), (s ** 2).sum()
    lost = total - np.linalg.norm(left @ right) ** 2
    assert abs(disc - tail / total) <= 2 * n * EPS
    # all but 1e-12 of the weight left after the cut, to rounding
    assert abs(lost - tail) <= 1e-12 * tail + 2 * n * EPS * total
    best = (u[:, :k] * s[:k]) @ vt[:k]
    assert np.linalg.norm(left @ right - best) <= 2 * n * EPS * s[0] ** 2 / (s[k - 1] - s[k])


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("n,k", [(12, 3), (24, 3)])
def test_close_values_at_the_cut_before_a_drop(split, n, k, mode):
    """Values around 1, the k-th and the next 1e-5 apart, one of 9e-7 after
    them: small enough to be left out of the QR by its weight, but not by what
    it turns the kept subspace by."""
    s = np.r_[1 - 0.01 * np.arange(k), 0.0, 9e-7, 1e-14 * np.ones(n - k - 2)]
    s[k] = s[k - 1] * (1 - 1e-5)
    for seed in range(16):
        _check(_matrix(n, s, seed), k, mode, split)


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("n,k,fall", [(64, 20, 0.0), (64, 40, 0.02), (96, 33, 0.1), (200, 77, 0.03)])
def test_slow_spectra(split, n, k, fall, mode):
    """Spectra that fall by `fall` decades a value, the k-th and the next 1e-6 apart."""
    s = 10.0 ** (-fall * np.arange(n)) * (1 - 1e-3 * np.arange(n))
    s[k] = s[k - 1] * (1 - 1e-6)
    _check(_matrix(n, s, n + k), k, mode, split)
