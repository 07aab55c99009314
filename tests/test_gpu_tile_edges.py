"""Sizes at which the kernels' tiles, panels, leaves and lists end or begin, against the
oracle or LAPACK at the tolerances of the paths they belong to (eigensolver 1e-12 of the
spectral radius; FP64 and FP64-accurate filter 1e-12 relative Frobenius; closure Ritz
values 1e-10; Ozaki products K 2^-50 of the row scales)."""
import numpy as np
import pytest
import torch

import chfsi_workloads as W
from tests.test_gpu_ozaki import _bsr_to_csr
from tests.util import dense_to_csr, rel_fro

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    from paper_2110_15853_gb300 import build
    build.build()
    import paper_2110_15853_gb300 as P
    return P


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a)).to("cuda")


@pytest.mark.parametrize("n", [4, 15, 16, 17, 34, 35, 48, 66, 255, 256, 258, 511, 513, 546])
def test_eigh_leaves_panels_and_merge_products(P, n):
    """Leaves and panels of 32 rows (and the last two rows), merges on either side of
    the FP64 / Ozaki product line, odd leading dimensions, on a random matrix and on one
    with threefold clusters (rotations in the merges)."""
    rng = np.random.default_rng(n)
    A = rng.standard_normal((n, n))
    Qr, _ = np.linalg.qr(rng.standard_normal((n, n)))
    lam = np.repeat(np.linspace(-1.0, 2.0, (n + 2) // 3), 3)[:n] + 1e-14 * rng.standard_normal(n)
    for M in ((A + A.T) / 2, (Qr * lam) @ Qr.T):
        M = (M + M.T) / 2
        w, Q = P.eigh(_dev(M))
        w, Q = w.cpu().numpy(), Q.cpu().numpy()
        ref = np.linalg.eigvalsh(M)
        scale = np.max(np.abs(ref))
        assert np.max(np.abs(w - ref)) <= 1e-12 * scale
        assert np.linalg.norm(M @ Q - Q * w) <= 1e-12 * np.linalg.norm(M) * max(1.0, np.sqrt(n) / 10)
        assert np.max(np.abs(Q.T @ Q - np.eye(n))) <= 1e-12


def _blocked(rng, nbr, keep, diag, drop_diag=()):
    """Symmetric blocked operator with random 8-column chunks zeroed (mirrored), stored zero
    blocks, and no stored diagonal block in the rows `drop_diag`."""
    N = nbr * 64
    A = rng.standard_normal((N, N)) * 0.05
    chunk = rng.random((N, N // 8)) < keep
    A *= np.repeat(np.repeat(chunk[::64], 64, axis=0), 8, axis=1)
    A = np.triu(A, 1)
    A = A + A.T
    A[np.arange(N), np.arange(N)] = diag(np.arange(N))
    bp, bc, val = [0], [], []
    for R in range(nbr):
        for C in range(nbr):
            if R == C and R in drop_diag:
                A[R * 64:(R + 1) * 64, R * 64:(R + 1) * 64] = 0.0
                continue
            if (R + C) % 3 == 2 and abs(R - C) > 1:
                A[R * 64:(R + 1) * 64, C * 64:(C + 1) * 64] = 0.0
                if (R + C) % 2:
                    continue            # not stored; else stored as zeros
            bc.append(C)
            val.append(A[R * 64:(R + 1) * 64, C * 64:(C + 1) * 64].copy())
        bp.append(len(bc))
    return dict(n_block_rows=nbr, bdim=64, brow_ptr=np.array(bp, dtype=np.int32), bcol=np.array(bc, dtype=np.int32),
                val=np.concatenate([v.ravel() for v in val]))


@pytest.mark.parametrize("nbr,n,keep,case", [(5, 1, 0.5, "folded"), (5, 64, 0.1, "folded"), (6, 127, 0.3, "grown"),
                                             (7, 129, 0.02, "mixed"), (3, 257, 1.0, "no_diagonal"), (1, 33, 1.0, "mixed")])
@pytest.mark.parametrize("kind,tol", [("ozaki", 1e-12), ("ozaki40", 1e-9)])
def test_bsr_ozaki_steps_chunk_lists_and_shift(P, oracle_mod, nbr, n, keep, case, kind, tol):
    """Steps on operators whose blocks have zero column chunks (any number left in a block
    row, zero blocks stored), with the shift c in H's digits (diagonal near c), outside them
    (a diagonal far below c would raise the row scale; or no diagonal block), and both in
    one operator; state counts around one and two tiles."""
    rng = np.random.default_rng(7 * nbr + n)
    a, b, a0 = 6.0, 10.0, 4.0          # c = 8
    diag = {"folded": lambda i: 7.5 + 0.3 * np.sin(i), "grown": lambda i: 0.2 + 0.0 * i,
            "mixed": lambda i: np.where((i // 64) % 2 == 0, 7.9, 0.1), "no_diagonal": lambda i: 7.0 + 0.0 * i}[case]
    B = _blocked(rng, nbr, keep, diag, drop_diag=range(0, nbr, 2) if case == "no_diagonal" else ())
    N = nbr * 64
    X = rng.standard_normal((N, n)) / np.sqrt(N)
    m = 4
    ws = P.Workspace("cuda")
    Hd = P.BsrMatrix.from_arrays(B["brow_ptr"], B["bcol"], B["val"], device="cuda")
    Y = P.filter(Hd, _dev(X), m, a, b, a0, schedule=[kind] * m, workspace=ws)
    assert P.read_status(ws) == 0
    assert rel_fro(Y.cpu().numpy(), oracle_mod.filter(_bsr_to_csr(B), X, m, a, b, a0)) <= tol


@pytest.mark.parametrize("K,M", [(33, 1), (40, 65), (130, 129), (9000, 191)])
def test_ozaki_gram_of_one_operand(P, K, M):
    """A^T A with B_hat the halves of A_hat's 128-row tiles."""
    rng = np.random.default_rng(K + M)
    A = rng.standard_normal((K, M))
    C = P.ozaki_gemm(_dev(A), _dev(A), transpose_a=True, symmetric=True).cpu().numpy()
    Ad = _dev(A)
    D = P.ozaki_gemm(Ad, Ad, transpose_a=True, symmetric=True).cpu().numpy()
    bound = K * 2.0 ** -50 * np.outer(np.abs(A).max(0), np.abs(A).max(0)) + 1e-15 * np.abs(A.T @ A)
    assert np.all(np.abs(C - A.T @ A) <= bound) and np.array_equal(C, D)


@pytest.mark.parametrize("n", [1, 15, 31, 32, 33, 63, 65, 96, 97, 129, 193])
@pytest.mark.parametrize("precision", ["f64", "ozaki"])
def test_closure_cholesky_blocks_and_inverse_levels(P, oracle_mod, n, precision):
    """State counts around the 32-column blocks and 64-column panels of the Cholesky
    factorisation, the 64-column leaves of the triangular inverse and its pairs of unequal
    halves, and the 16 x 16 and 64 x 64 product tiles."""
    rng = np.random.default_rng(n)
    N = 640
    A = rng.standard_normal((N, N))
    H = dense_to_csr((A + A.T) / 2)
    Y = rng.standard_normal((N, n)) * np.logspace(0, -2, n)
    theta, _, _ = oracle_mod.rayleigh_ritz(H, Y)
    Hd = P.CsrMatrix.from_arrays(H["row_ptr"], H["col"], H["val"], device="cuda")
    ritz, psi = P.rayleigh_ritz(Hd, _dev(Y), 2, precision=precision)
    p = psi.cpu().numpy()
    assert np.max(np.abs(ritz.cpu().numpy() - theta)) <= 1e-10 * np.max(np.abs(theta))
    assert np.max(np.abs(p.T @ p - np.eye(n))) <= 1e-12


@pytest.mark.parametrize("n", [1, 7, 8, 9, 16, 17, 24, 31, 33, 40, 47, 48, 49, 56, 64, 65, 104, 120, 193, 257, 301, 321])
@pytest.mark.parametrize("schedule", [None, "f32x2"])
def test_csr_steps_last_columns(P, oracle_mod, n, schedule):
    """State counts whose last columns take each width of the FP64 step (64, 32, 16 and 8
    columns, entries shared by groups of lanes) and each number of chunks per pass of the
    two-float step, on rows of 0 to 40 entries (empty and single-entry rows among them)."""
    rng = np.random.default_rng(n)
    N, m = 75, 3
    A = np.where(rng.random((N, N)) < rng.random((N, 1)) * 0.6, rng.standard_normal((N, N)), 0.0)
    A[::13] = 0.0
    A[5, :] = 0.0
    A[5, 70] = 1.5
    H = dense_to_csr(A / 10, keep_zeros=False)
    X = rng.standard_normal((N, n))
    a, b, a0 = 0.5, 2.0, -2.0
    Hd = P.CsrMatrix.from_arrays(H["row_ptr"], H["col"], H["val"], device="cuda")
    ws = P.Workspace("cuda")
    Y = P.filter(Hd, _dev(X), m, a, b, a0, schedule=None if schedule is None else [schedule] * m, workspace=ws)
    assert P.read_status(ws) == 0
    assert rel_fro(Y.cpu().numpy(), oracle_mod.filter(H, X, m, a, b, a0)) <= 1e-12


@pytest.mark.parametrize("N", [2, 3, 5, 31, 33, 63, 130, 511, 513, 1100])
def test_lanczos_rows_per_warp_and_chunks(P, oracle_mod, N):
    """Row counts around the four rows of a warp, the 32 of a block and the 512 of a vector
    chunk, with rows of very different lengths."""
    rng = np.random.default_rng(N)
    A = np.where(rng.random((N, N)) < rng.random((N, 1)), rng.standard_normal((N, N)), 0.0)
    A = (A + A.T) / 2 + np.diag(np.linspace(1.0, 5.0, N))
    H = dense_to_csr(A, keep_zeros=False)
    v0 = rng.standard_normal(N)
    Hd = P.CsrMatrix.from_arrays(H["row_ptr"], H["col"], H["val"], device="cuda")
    got = P.lanczos_bounds(Hd, _dev(v0), 12, 1)
    want = oracle_mod.lanczos_bounds(H, v0, 12, 1)
    scale = max(abs(x) for x in want)
    assert max(abs(g - w) for g, w in zip(got, want)) <= 1e-10 * scale
