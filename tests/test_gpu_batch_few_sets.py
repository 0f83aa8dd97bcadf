"""GPU: two to seven sets in the uneven batch: its fills go through working copies of
the tables as the separate calls do, with the results of the separate calls.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SPACE = (3, 3, 4, 0)                             # 17,040 rows: the copy for one to four sets
LARGE = (3, 4, 4, 1)                             # 48,917 rows: for five to seven, too


@pytest.fixture(scope="module")
def cih():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1412_5989_gb300 import cih as mod
    return mod


def tables(B, K):
    g = torch.Generator(device="cuda").manual_seed(11)
    return torch.randn((K, B.tbme_len), generator=g, device="cuda")


@pytest.mark.parametrize("K", [2, 3, 4, 7])
def test_batch_of_few_sets(cih, K):
    B = [cih.Basis(*s) for s in (SPACE, (2, 2, 2, 0), LARGE)]
    T = [tables(b, K) for b in B]
    _, got = cih.solve_batch([(b, t) for b, t in zip(B, T)], 20.0, 1, 200, 1e-8)
    for b, t, r in zip(B, T, got):
        rowptr, nnz = b.count()
        col, val = b.fill(rowptr, nnz, t)
        ev, vec, _ = b.lanczos(rowptr, col, val, 1, 200, 1e-8)
        assert r["nnz"] == nnz and r["status"] == 0
        np.testing.assert_array_equal(np.asarray(r["evals"]), np.asarray(ev))
        assert torch.equal(r["grad"], b.tbme_grad(rowptr, vec))
        b.check()


def test_batch_prepares_few_sets(cih):
    """The batch's fill of three sets is the copy's two kernels, not the row kernel."""
    B = cih.Basis(*SPACE)
    T = tables(B, 3)
    rowptr, nnz = B.count()

    def launches(f):
        n0 = cih.kernel_launches()
        f()
        return cih.kernel_launches() - n0

    col, val = B.fill(rowptr, nnz, T)
    solve = launches(lambda: B.lanczos(rowptr, col, val, 1, 5, 1e-8))
    count = launches(lambda: B.count_into(torch.empty(B.dim + 1, dtype=torch.int64, device="cuda")))
    both = launches(lambda: cih.solve_batch([(B, T)], 20.0, 1, 5, 1e-8, want_grad=False))
    assert both == count + 2 + solve
