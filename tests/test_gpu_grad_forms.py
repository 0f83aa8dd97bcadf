"""GPU: the adjoint of one vector in the form large bases take (pairs of one
species summed over their common partners, pn entries in full squares) against
the row kernel's, which two vectors at once take: integer sums, so the same bits.
"""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cih():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1412_5989_gb300 import cih as mod
    return mod


# from 2^19 rows: unequal species, odd 2M, many levels, few protons
@pytest.mark.parametrize("space", [(5, 6, 4, 1), (2, 6, 6, 0), (3, 4, 6, 1), (6, 2, 6, 4), (4, 4, 5, 0)])
def test_one_vector_against_the_row_kernel(cih, space):
    B = cih.Basis(*space)
    assert B.dim >= 1 << 19
    rowptr, _ = B.count()
    g = torch.Generator(device="cuda").manual_seed(5)
    psi = torch.randn((2, B.dim), generator=g, dtype=torch.float64, device="cuda")
    psi /= psi.norm(dim=1, keepdim=True)
    both = B.tbme_grad(rowptr, psi)
    for k in range(2):
        assert torch.equal(B.tbme_grad(rowptr, psi[k])[0], both[k])
    B.check()
    # an eigenvector's few large entries: half the norm in one of them
    psi[0] *= 0.0
    psi[0, 7], psi[0, B.dim // 2], psi[0, B.dim - 1] = 0.8, -0.59, 0.1
    both = B.tbme_grad(rowptr, psi)
    assert torch.equal(B.tbme_grad(rowptr, psi[0])[0], both[0])
    B.check()
