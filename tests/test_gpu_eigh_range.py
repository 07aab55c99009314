"""The dense eigensolver and the closure on input outside the ordinary: entries that are not
finite.  The call must end with the status that include/chfsi.h names, touch no memory but
its own, and leave the context and the workspace usable: a finite matrix on the same
workspace is solved as by LAPACK afterwards."""
import ctypes

import numpy as np
import pytest
import torch

from tests.util import dense_to_csr

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    from paper_2110_15853_gb300 import build
    build.build()
    import paper_2110_15853_gb300 as P
    return P


def _symmetric(n, seed):
    A = np.random.default_rng(seed).standard_normal((n, n))
    return (A + A.T) / 2


class _Solver:
    """chfsi_eigh on one workspace: (status word, w, Q) per call."""

    def __init__(self, P, n):
        self.lib, self.n = P.load(), n
        sz = ctypes.c_size_t(0)
        assert self.lib.chfsi_eigh_workspace_size(n, ctypes.byref(sz)) == 0
        self.ws = torch.full((sz.value,), 0x7f, dtype=torch.uint8, device="cuda")   # ints far out of any range

    def __call__(self, A):
        n, st = self.n, torch.cuda.current_stream().cuda_stream
        Ad = torch.as_tensor(A).cuda()
        w = torch.empty(n, dtype=torch.float64, device="cuda")
        Q = torch.empty(n, n, dtype=torch.float64, device="cuda")
        assert self.lib.chfsi_eigh(Ad.data_ptr(), n, n, w.data_ptr(), Q.data_ptr(), n, self.ws.data_ptr(),
                                   self.ws.numel(), st) == 0
        return self.lib.chfsi_read_status(self.ws.data_ptr(), st), w.cpu().numpy(), Q.cpu().numpy()


def _check(A, w, Q, tol=1e-12):
    ref = np.linalg.eigvalsh(A)
    n = A.shape[0]
    assert np.max(np.abs(w - ref)) <= tol * np.max(np.abs(ref))
    assert np.linalg.norm(A @ Q - Q * w) <= tol * np.linalg.norm(A) * max(1.0, np.sqrt(n) / 10)
    assert np.max(np.abs(Q.T @ Q - np.eye(n))) <= tol


@pytest.mark.parametrize("n", [33, 64, 97, 300, 700])
@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("where", ["first", "last", "all"])
def test_eigh_of_a_matrix_that_is_not_finite(P, n, value, where):
    """Sizes with one merge, two equal halves, merges of several levels, and products on
    either side of the FP64 / Ozaki line."""
    from paper_2110_15853_gb300 import _abi
    A = _symmetric(n, n)
    B = A.copy()
    B[{"first": (0, 0), "last": (n - 1, n - 1), "all": (slice(None), slice(None))}[where]] = value
    solve = _Solver(P, n)
    assert solve(B)[0] == _abi.CHFSI_ERR_NONFINITE
    status, w, Q = solve(A)
    assert status == 0
    _check(A, w, Q)


@pytest.mark.parametrize("n", [40, 96, 300])
@pytest.mark.parametrize("passes", [1, 2])
@pytest.mark.parametrize("value", [np.nan, np.inf])
def test_closure_of_an_operator_or_a_block_that_is_not_finite(P, n, passes, value):
    """An entry of H that is not finite is found after the eigensolve (NONFINITE); one of Y
    makes a Cholesky pivot that is not positive (CHOL)."""
    from paper_2110_15853_gb300 import _abi
    N = 400
    A, Y = _symmetric(N, 3), np.random.default_rng(n).standard_normal((N, n))
    H, bad = dense_to_csr(A), dense_to_csr(A)
    bad["val"][N * 7 + 9] = value
    Yb = Y.copy()
    Yb[5, n // 2] = value
    ws = P.Workspace("cuda")
    dev = lambda h: P.CsrMatrix.from_arrays(h["row_ptr"], h["col"], h["val"], device="cuda")
    for h, y, want in ((bad, Y, _abi.CHFSI_ERR_NONFINITE), (H, Yb, _abi.CHFSI_ERR_CHOL)):
        with pytest.raises(P.ChfsiError) as e:
            P.rayleigh_ritz(dev(h), torch.as_tensor(y).cuda(), passes, workspace=ws)
        assert e.value.code == want
    ritz, psi = P.rayleigh_ritz(dev(H), torch.as_tensor(Y).cuda(), passes, workspace=ws)
    p, th = psi.cpu().numpy(), ritz.cpu().numpy()
    Qy = np.linalg.qr(Y)[0]
    assert np.max(np.abs(th - np.linalg.eigvalsh(Qy.T @ A @ Qy))) <= 1e-10 * np.max(np.abs(th))
    assert np.max(np.abs(p.T @ p - np.eye(n))) <= (1e-12 if passes == 2 else 1e-9)
