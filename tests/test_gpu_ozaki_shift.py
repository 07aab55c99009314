"""The shift c of an Ozaki BSR step: in the digits of H's diagonal only where that costs no
accuracy, else an FP64 multiply-add on the iterate itself."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    from paper_2110_15853_gb300 import build
    build.build()
    import paper_2110_15853_gb300 as P
    return P


@pytest.mark.parametrize("kind", ["ozaki", "ozaki40"])
def test_shift_of_rows_without_a_diagonal(P, kind):
    """Two blocks with large entries between them and zeros on the diagonal: where X vanishes
    on the second block, the first block of one step is -alpha c X, two FP64 roundings of
    each entry, however small beside the largest of its column (2^-30 .. 1 here), and not
    the digits of X times c."""
    rng = np.random.default_rng(5)
    a, b, a0, n = 6.3, 10.1, 4.2, 70
    e, c = (b - a) / 2, (b + a) / 2
    blocks = np.zeros((4, 64, 64))                    # (0,0) (0,1) (1,0) (1,1)
    blocks[1] = 100.0 * rng.standard_normal((64, 64))
    blocks[2] = blocks[1].T
    H = P.BsrMatrix.from_arrays([0, 2, 4], [0, 1, 0, 1], blocks.ravel())
    X = rng.standard_normal((128, n)) * np.exp2(-rng.integers(0, 31, (128, n)))
    X[64:] = 0.0
    ws = P.Workspace("cuda")
    Y = P.filter(H, torch.as_tensor(X).cuda(), 1, a, b, a0, schedule=[kind], workspace=ws).cpu().numpy()
    assert P.read_status(ws) == 0
    exact = -(e / (a0 - c)) / e * c * X[:64]
    # alpha and c are four roundings away from their values here, the result two more
    assert np.all(np.abs(Y[:64] - exact) <= 6 * np.finfo(float).eps * np.abs(exact))
