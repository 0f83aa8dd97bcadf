"""GPU: the default budget of the uneven batch counts the library pool's idle blocks.
A Lanczos call leaves freed blocks in the pool; a batch that fits the device's free
memory before it must fit after it.
"""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_default_budget_counts_idle_blocks():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1412_5989_gb300 import cih
    B = cih.Basis(4, 4, 4, 0)
    K, GiB = 4, 1 << 30
    T = torch.randn((K, B.tbme_len), generator=torch.Generator(device="cuda").manual_seed(3), device="cuda")
    rowptr, nnz = B.count()
    col, val = B.fill(rowptr, nnz, T)
    B.lanczos(rowptr, col, val, 1, 300, 1e-6, want_vectors=False)         # 1.4 GB of vectors: 1 GiB stays in the pool
    del col, val
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    left = 5 * GiB
    hold = torch.empty(free - left, dtype=torch.uint8, device="cuda")     # (reserved, not written)
    try:
        free = torch.cuda.mem_get_info()[0]
        # an instance between 0.9 of the free memory and 0.9 of it with the idle GiB
        want = int(0.9 * (free + 0.55 * GiB))
        per = 8 * B.dim * K                                               # bytes a Lanczos step adds
        _, got = cih.solve_batch([(B, T)], 20.0, 1, 300, 1e-6, want_grad=False)
        steps = 300 + (want - got[0]["bytes"]) // (per + 8 * K * 257)
        assert 300 < steps <= 2048
        _, got = cih.solve_batch([(B, T)], 20.0, 1, int(steps), 1e-6, want_grad=False)
        assert 0.9 * free < got[0]["bytes"] < 0.9 * (free + GiB)
        assert got[0]["status"] == 0 and got[0]["wave"] == 0
    finally:
        del hold
        torch.cuda.empty_cache()
