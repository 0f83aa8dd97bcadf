"""GPU: a captured fill is one kernel without scratch of its own: its graph can be
instantiated twice and be a child graph, and replays give the bits of the call.
"""
import ctypes as C

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cih():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1412_5989_gb300 import cih as mod
    return mod


def capture(drv, stream, call):
    g = C.c_void_p()
    assert drv.cuStreamBeginCapture_v2(C.c_void_p(stream.cuda_stream), 1) == 0           # thread-local
    call()
    assert drv.cuStreamEndCapture(C.c_void_p(stream.cuda_stream), C.byref(g)) == 0
    return g


@pytest.mark.parametrize("K", [1, 3])
@pytest.mark.parametrize("onebody", [False, True])
def test_captured_fill(cih, K, onebody):
    drv = C.CDLL("libcuda.so.1")
    B = cih.Basis(3, 3, 4, 0)                    # 17,040 rows: the call itself goes through the working copy
    rowptr, nnz = B.count()
    g = torch.Generator(device="cuda").manual_seed(5)
    # sums of ones and half last bits, decided by one-body terms of 2^-46: the order of a sum shows
    t = 1.0 + torch.randint(-(1 << 20), 1 << 20, (2, K, B.tbme_len), generator=g, device="cuda") * 2.0 ** -23
    T = t.to(torch.float32).contiguous()
    n1 = B.onebody_len if onebody else sum(B.n_orb)
    t1 = torch.randn(n1, generator=g, device="cuda", dtype=torch.float64) * 2.0 ** -46
    now = T[0].clone()
    col = torch.empty(nnz, dtype=torch.int32, device="cuda")
    val = torch.empty((K, nnz), dtype=torch.float32, device="cuda")

    def fill(t, stream=None, **out):
        if onebody:
            return B.fill_onebody(rowptr, nnz, t, t1, stream=stream, **out)
        return B.fill(rowptr, nnz, t, e_sp=t1, stream=stream, **out)

    want = [fill(T[i]) for i in (0, 1)]
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    graph = capture(drv, s, lambda: fill(now, stream=s, col=col, val=val))
    execs = [C.c_void_p(), C.c_void_p(), C.c_void_p()]
    for x in execs[:2]:
        assert drv.cuGraphInstantiateWithFlags(C.byref(x), graph, C.c_uint64(0)) == 0
    parent, node = C.c_void_p(), C.c_void_p()
    assert drv.cuGraphCreate(C.byref(parent), 0) == 0
    assert drv.cuGraphAddChildGraphNode(C.byref(node), parent, None, C.c_size_t(0), graph) == 0
    assert drv.cuGraphInstantiateWithFlags(C.byref(execs[2]), parent, C.c_uint64(0)) == 0
    for i, x in enumerate(execs):
        now.copy_(T[i % 2])                      # a replay reads the tables anew
        col.zero_()
        val.zero_()
        torch.cuda.synchronize()
        assert drv.cuGraphLaunch(x, C.c_void_p(s.cuda_stream)) == 0
        s.synchronize()
        assert torch.equal(col, want[i % 2][0]) and torch.equal(val, want[i % 2][1])
    for x in execs:
        assert drv.cuGraphExecDestroy(x) == 0
    assert drv.cuGraphDestroy(parent) == 0 and drv.cuGraphDestroy(graph) == 0
    B.check()
