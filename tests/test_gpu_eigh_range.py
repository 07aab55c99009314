"""The dense eigensolver and the closure on input outside the ordinary.

Entries that are not finite: the call must end with the status that include/chfsi.h names,
touch no memory but its own, and leave the context and the workspace usable (a finite matrix
on the same workspace is solved as by LAPACK afterwards).  Entries near the ends of the FP64
range, and couplings whose squares vanish: the tolerances of the ordinary matrices
(eigenvalues, residuals and orthogonality to 1e-12), a power of two taken out first."""
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


@pytest.mark.parametrize("n", [3, 12, 32, 40, 97, 300])
@pytest.mark.parametrize("exponent", [-1000, -500, -350, 350, 500, 1000])
def test_eigh_of_any_magnitude(P, n, exponent):
    A = _symmetric(n, n)
    status, w, Q = _Solver(P, n)(np.ldexp(A, exponent))
    assert status == 0
    _check(A, np.ldexp(w, -exponent), Q)


@pytest.mark.parametrize("n", [300, 600, 1500, 2100])
@pytest.mark.parametrize("kind", ["random", "spread", "dominant"])
@pytest.mark.parametrize("scale", [1e-8, 1.0, 13.0])
def test_eigh_panel_updates_of_any_norm(P, n, kind, scale):
    """The trailing updates on the tensor cores (256 rows and more) to the accuracy of FP64 ones,
    whatever A's norm is against its entries: a random matrix (norm sqrt(n) entries), a
    spectrum in [1, 3], and a matrix of ones with a random part of 1e-3 (norm n entries).
    Residual within 4 eps sqrt(n) of |A|_F, the growth of the rounding errors of n
    reflections."""
    if kind == "spread":
        Qr = np.linalg.qr(np.random.default_rng(n).standard_normal((n, n)))[0]
        A = (Qr * np.linspace(1.0, 3.0, n)) @ Qr.T
        A = (A + A.T) / 2
    else:
        A = _symmetric(n, n) if kind == "random" else 1.0 + 1e-3 * _symmetric(n, n)
    status, w, Q = _Solver(P, n)(A * scale)
    assert status == 0
    A, eps = A * scale, np.finfo(float).eps
    assert np.linalg.norm(A @ Q - Q * w) <= 4 * eps * np.sqrt(n) * np.linalg.norm(A)
    assert np.max(np.abs(w - np.linalg.eigvalsh(A))) <= 4 * eps * np.sqrt(n) * np.linalg.norm(A)
    assert np.max(np.abs(Q.T @ Q - np.eye(n))) <= 1e-12


@pytest.mark.parametrize("n", [12, 40, 66, 300])
@pytest.mark.parametrize("coupling", [1e-130, 1e-145, 1e-156, 1e-158, 1e-161, 1e-165, 1e-200, 1e-310])
def test_eigh_of_blocks_that_hardly_couple(P, n, coupling):
    A, h = _symmetric(n, n), n // 2
    A[:h, h:] *= coupling
    A[h:, :h] *= coupling
    status, w, Q = _Solver(P, n)(A)
    assert status == 0
    _check(A, w, Q)


@pytest.mark.parametrize("n", [40, 300])
@pytest.mark.parametrize("exponent", [-400, 400])
def test_closure_of_an_operator_of_any_magnitude(P, n, exponent):
    N = 400
    A, Y = _symmetric(N, 3), np.random.default_rng(n).standard_normal((N, n))
    h = dense_to_csr(np.ldexp(A, exponent))
    Hd = P.CsrMatrix.from_arrays(h["row_ptr"], h["col"], h["val"], device="cuda")
    ritz, psi = P.rayleigh_ritz(Hd, torch.as_tensor(Y).cuda(), 2)
    p, Qy = psi.cpu().numpy(), np.linalg.qr(Y)[0]
    ref = np.linalg.eigvalsh(Qy.T @ A @ Qy)
    assert np.max(np.abs(np.ldexp(ritz.cpu().numpy(), -exponent) - ref)) <= 1e-10 * np.max(np.abs(ref))
    assert np.max(np.abs(p.T @ p - np.eye(n))) <= 1e-12


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


@pytest.mark.parametrize("n", [100, 300, 700])
def test_a_grid_barrier_that_gives_up(P, n):
    """With a limit of a few nanoseconds the first barrier of a panel that is not complete at
    once gives up: the status says so, in chfsi_eigh, in the binding and in the closure,
    and the next call on the same workspace is right."""
    from paper_2110_15853_gb300 import _abi
    A, solve = _symmetric(n, n), _Solver(P, n)
    h = dense_to_csr(_symmetric(800, 1))
    Hd = P.CsrMatrix.from_arrays(h["row_ptr"], h["col"], h["val"], device="cuda")
    Y = torch.as_tensor(np.random.default_rng(n).standard_normal((800, n))).cuda()
    lib = P.load()
    assert lib.chfsi_set_pipeline_wait_limit(4) == 0
    try:
        assert solve(A)[0] == _abi.CHFSI_ERR_TIMEOUT
        for call in (lambda: P.eigh(torch.as_tensor(A).cuda()), lambda: P.rayleigh_ritz(Hd, Y, 2)):
            with pytest.raises(P.ChfsiError) as e:
                call()
            assert e.value.code == _abi.CHFSI_ERR_TIMEOUT
    finally:
        assert lib.chfsi_set_pipeline_wait_limit(0) == 0
    status, w, Q = solve(A)
    assert status == 0
    _check(A, w, Q)
    w, Q = P.eigh(torch.as_tensor(A).cuda())
    _check(A, w.cpu().numpy(), Q.cpu().numpy())


def test_eigh_binding_raises_on_a_matrix_that_is_not_finite(P):
    from paper_2110_15853_gb300 import _abi
    A = _symmetric(20, 0)
    A[3, 4] = A[4, 3] = np.nan
    with pytest.raises(P.ChfsiError) as e:
        P.eigh(torch.as_tensor(A).cuda())
    assert e.value.code == _abi.CHFSI_ERR_NONFINITE


@pytest.fixture(scope="module")
def stream_of_few_sms():
    """A stream of a green context with the smallest share of the SMs that the driver gives."""
    torch.cuda.init()
    torch.zeros(1, device="cuda")
    cu = ctypes.CDLL("libcuda.so.1")
    if not hasattr(cu, "cuGreenCtxStreamCreate"):
        pytest.skip("the driver has no green contexts")
    ok = lambda rc: rc == 0 or pytest.fail(f"driver error {rc}")
    resource = ctypes.c_char * 144                       # CUdevResource
    dev, every, some, rest = ctypes.c_int(), resource(), resource(), resource()
    groups, desc, ctx, stream = ctypes.c_uint(1), ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_void_p()
    ok(cu.cuDeviceGet(ctypes.byref(dev), torch.cuda.current_device()))
    ok(cu.cuDeviceGetDevResource(dev, every, 1))         # CU_DEV_RESOURCE_TYPE_SM
    ok(cu.cuDevSmResourceSplitByCount(some, ctypes.byref(groups), every, rest, 0, 1))
    ok(cu.cuDevResourceGenerateDesc(ctypes.byref(desc), some, 1))
    ok(cu.cuGreenCtxCreate(ctypes.byref(ctx), desc, dev, 1))
    ok(cu.cuGreenCtxStreamCreate(ctypes.byref(stream), ctx, 1, 0))
    yield torch.cuda.ExternalStream(stream.value)
    torch.cuda.synchronize()
    ok(cu.cuStreamDestroy_v2(stream))
    ok(cu.cuGreenCtxDestroy(ctx))


@pytest.mark.parametrize("n", [40, 300, 1500])
def test_eigh_on_a_stream_of_few_sms(P, stream_of_few_sms, n):
    """The grid of the tridiagonalisation's panels shrinks to what can be resident."""
    A = _symmetric(n, n)
    torch.cuda.synchronize()
    with torch.cuda.stream(stream_of_few_sms):
        w, Q = P.eigh(torch.as_tensor(A).cuda())
        w, Q = w.cpu().numpy(), Q.cpu().numpy()
    _check(A, w, Q)
