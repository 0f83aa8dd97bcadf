"""GPU: the build to host memory of one to seven sets.  Its row chunks share one
working copy of the tables, or take none, and the arrays are those of the fill call.
"""
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


@pytest.mark.parametrize("space,K,copies", [(SPACE, 1, 1), (SPACE, 3, 1), (LARGE, 2, 1), (LARGE, 4, 1), (LARGE, 5, 0),
                                            (LARGE, 7, 0)])
def test_build_to_host(cih, space, K, copies):
    B = cih.Basis(*space)
    rowptr, nnz = B.count()
    T = tables(B, K)
    col, val = B.fill(rowptr, nnz, T)
    rp = torch.empty(B.dim + 1, dtype=torch.int64).pin_memory()
    c = torch.empty(nnz, dtype=torch.int32).pin_memory()
    v = torch.empty((K, nnz), dtype=torch.float32).pin_memory()
    t = T.cpu()
    B.build_to_host(t, rp, c, v)
    n0 = cih.kernel_launches()
    B.count_into(torch.empty(B.dim + 1, dtype=torch.int64, device="cuda"))
    count = cih.kernel_launches() - n0
    n0 = cih.kernel_launches()
    assert B.build_to_host(t, rp, c, v) == nnz
    # eight fills and at most one preparation for all of them
    assert cih.kernel_launches() - n0 == count + 8 + copies
    assert torch.equal(rp, rowptr.cpu()) and torch.equal(c, col.cpu()) and torch.equal(v, val.cpu())
    B.check()
