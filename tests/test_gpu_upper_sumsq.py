"""GPU: the sum of squares of the strictly-upper values (the bound of the
product's fixed-point scale) streams the values across the ends of the rows; it
is compared with FP64 over whole matrices, single rows and ranges of rows, set
counts around the strides of its loads, and values off a 16-byte boundary.

Each value's square is an exact FP32 pair; a double-float add of positive numbers
errs by at most 2^-44 relative.  A lane adds fewer than 2^4 values to each of its
sums here between two rows' ends and fewer than 2^9 in all: 2^-35 is allowed."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cih():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1412_5989_gb300 import cih as mod
    return mod


@pytest.mark.parametrize("space", [(1, 1, 2, 0), (2, 3, 2, 1), (2, 2, 6, 0), (3, 4, 4, 1)])
@pytest.mark.parametrize("K", [1, 2, 3, 8, 9, 64])
def test_against_fp64(cih, space, K):
    B = cih.Basis(*space)
    rowptr, nnz = B.count()
    if nnz * K > 10 ** 8:
        pytest.skip("enough with fewer sets")
    t = torch.randn(K, B.tbme_len, device="cuda", generator=torch.Generator("cuda").manual_seed(3))
    if K == 1:
        col, val = B.fill(rowptr, nnz, t)
        V = val.reshape(nnz, 1)
    else:
        col, V = B.fill_batched(rowptr, nnz, cih.tbme_interleave(t), K)
    i = torch.repeat_interleave(torch.arange(B.dim, device="cuda"), rowptr[1:] - rowptr[:-1])
    sq = (V.double() ** 2).sum(1) * (col.long() != i)
    for r0, r1 in [(0, B.dim), (B.dim // 3, B.dim // 2), (B.dim // 2, B.dim // 2 + 1), (B.dim - 1, B.dim)]:
        a, b = int(rowptr[r0]), int(rowptr[r1])
        want = float(sq[a:b].sum())
        buf = torch.full(((b - a) * K + 3,), float("nan"), device="cuda")
        for shift in range(4):
            part = buf[shift:shift + (b - a) * K].view((b - a, K) if K > 1 else (1, b - a))
            part.copy_(V[a:b].reshape(part.shape))
            got = B.upper_sumsq(rowptr, r0, r1, part, element_major=K > 1)
            assert abs(got - want) <= 2.0 ** -35 * want
