"""The filter's columns are independent, and the FP64 steps keep that to the bit: a column's
result does not depend on how many columns stand beside it or where it stands, so that column
shards give what the whole block gives."""
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


def _rows_of_many_lengths(P, rng, N, longest):
    """CSR rows of 0 to `longest` entries, empty and single-entry ones among them."""
    counts = rng.integers(0, longest + 1, N)
    counts[::13] = 0
    counts[5::17] = 1
    rp = np.zeros(N + 1, dtype=np.int64)
    np.cumsum(counts, out=rp[1:])
    return P.CsrMatrix.from_arrays(rp, rng.integers(0, N, rp[-1]).astype(np.int32), rng.standard_normal(rp[-1]) / longest)


# 75 and 1700 rows: four rows a CTA; 9800: eight; rows of up to 1500 entries are not staged
@pytest.mark.parametrize("N,longest", [(75, 40), (1700, 30), (301, 1500), (9800, 20)])
@pytest.mark.parametrize("schedule", [None, ["f32", "f32", "f64", "f64", "f64"]])
def test_csr_columns_have_the_same_bits_in_every_block(P, N, longest, schedule):
    rng = np.random.default_rng(N)
    H, m = _rows_of_many_lengths(P, rng, N, longest), 5
    X = torch.as_tensor(rng.standard_normal((N, 256))).cuda()
    bounds = (0.5, 2.0, -2.0)
    whole = P.filter(H, X, m, *bounds, schedule=schedule)
    for n in (1, 7, 8, 9, 16, 17, 24, 32, 33, 40, 48, 49, 56, 64, 65, 80, 104, 200):
        for j in (0, 256 - n):
            part = P.filter(H, X[:, j:j + n].contiguous(), m, *bounds, schedule=schedule)
            assert torch.equal(part, whole[:, j:j + n]), (n, j)


@pytest.mark.parametrize("n", [8, 13, 40, 56])
def test_split_columns_have_the_same_bits_in_every_block(P, n):
    rng = np.random.default_rng(n)
    N = 700
    d = np.abs(np.subtract.outer(np.arange(N), np.arange(N)))
    A = np.where((d < 90) | (rng.random((N, N)) < 0.02), rng.standard_normal((N, N)) / 30, 0.0)
    h = dense_to_csr((A + A.T) / 2, keep_zeros=False)
    H = P.SplitMatrix.from_csr(h["row_ptr"], h["col"], h["val"], block=128)
    X = torch.as_tensor(rng.standard_normal((N, 128))).cuda()
    whole = P.filter(H, X, 4, 0.5, 2.0, -2.0)
    part = P.filter(H, X[:, 128 - n:].contiguous(), 4, 0.5, 2.0, -2.0)
    assert torch.equal(part, whole[:, 128 - n:])
