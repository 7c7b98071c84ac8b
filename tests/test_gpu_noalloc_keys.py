"""kc_lower_bounds_noalloc after a call whose last launch never ran: the bound
kernel has left its keys, the kernel that reads them out did not follow.  Made
here by capturing a call into a graph and launching the graph without its last
node; the next call has to start from cleared keys."""
import ctypes as C

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2301_00061_gb300 as kcm  # noqa: E402

DEV = torch.device("cuda:0")


# few nodes (streaming kernel), a batch (pruning kernel), wide data
@pytest.mark.parametrize("n,d,k,b", [(5_000, 2, 3, 4), (20_000, 4, 3, 100), (3_000, 29, 2, 40)])
def test_keys_of_an_unfinished_call(n, d, k, b):
    cu = C.CDLL("libcuda.so.1")

    def ok(st):
        assert st == 0, st

    rng = np.random.default_rng(n)
    X = torch.from_numpy(rng.normal(size=(d, n)).astype(np.float32)).to(DEV)
    c = torch.from_numpy(rng.normal(size=(b, k, d)).astype(np.float32)).to(DEV)
    far = c + 50.0                        # larger values than c's
    lb = torch.full((b,), -1.0, dtype=torch.float64, device=DEV)
    raw, arg = torch.full_like(lb, -1.0), torch.full((b,), -7, dtype=torch.int64, device=DEV)
    stream = torch.cuda.Stream()
    sp = C.c_void_p(stream.cuda_stream)
    torch.cuda.synchronize()

    def call(box, out=(lb, raw, arg)):
        kcm.kc_lower_bounds_noalloc(X, n, n, d, k, box, box, *out, stream=stream.cuda_stream)

    call(c)
    stream.synchronize()
    want = [t.clone() for t in (lb, raw, arg)]
    for t in (lb, raw):
        t.fill_(-1.0)
    torch.cuda.synchronize()

    graph, execu = C.c_void_p(), C.c_void_p()
    ok(cu.cuStreamBeginCapture_v2(sp, 2))   # relaxed
    call(far)
    ok(cu.cuStreamEndCapture(sp, C.byref(graph)))
    num = C.c_size_t(0)
    ok(cu.cuGraphGetNodes(graph, None, C.byref(num)))
    nodes = (C.c_void_p * num.value)()
    ok(cu.cuGraphGetNodes(graph, nodes, C.byref(num)))
    ok(cu.cuGraphDestroyNode(C.c_void_p(nodes[num.value - 1])))
    ok(cu.cuGraphInstantiateWithFlags(C.byref(execu), graph, C.c_ulonglong(0)))
    ok(cu.cuGraphLaunch(execu, sp))
    stream.synchronize()
    assert torch.all(lb == -1.0)            # the outputs were not written
    ok(cu.cuGraphExecDestroy(execu))
    ok(cu.cuGraphDestroy(graph))

    call(c)
    stream.synchronize()
    for a, w in zip((lb, raw, arg), want):
        assert torch.equal(a, w)
