"""Calls that would split a small batch's bins over the GPU, and then find no
scratch to add the splits up in.  The failure is injected as a request that
the runtime itself refuses, so the thread is left as a real failure leaves it."""
import ctypes
import os
import subprocess
import sys

import numpy as np
import pytest

import datagen
import oracle
import paper_1806_07300_gb300 as fp

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


@pytest.fixture(autouse=True)
def _clear_injection():
    yield
    fp.fp_inject_fault(None, fp.FP_FAULT_ALLOC, 0)


def _upload_meets_no_injection(pf):
    fp.fp_upload(pf).release()  # raises FP_ENOMEM if the injection was not used up


@pytest.mark.parametrize("n", [1, 33, 700])
def test_votes_without_scratch(tiny_forest, tiny_rows, n):
    X = np.ascontiguousarray(tiny_rows[0][:n])
    pf = fp.fp_pack_forest(tiny_forest, bin_size=1, interleave_depth=3, pass_bytes=-1)
    df = fp.fp_upload(pf)
    Xd = torch.from_numpy(X).cuda()
    ref = oracle.predict(tiny_forest, X)
    for _ in range(2):
        fp.fp_inject_fault(None, fp.FP_FAULT_ALLOC, 1)
        v, c = df.predict(Xd)
        _upload_meets_no_injection(pf)
        assert df.sync_status() == fp.FP_OK
        np.testing.assert_array_equal(v.cpu().numpy().astype(np.uint32), ref["votes"])
        np.testing.assert_array_equal(c.cpu().numpy(), ref["cls"])
    df.release()


@pytest.mark.parametrize("n", [1, 33, 700])
def test_values_without_scratch(n):
    Xt, yt = datagen.gen_regression(53, 2000, 0, 1.0, 1.0)
    F = datagen.train_regression(Xt, yt, 24, mtry=9, min_leaf=3, seed=53)
    pf = fp.fp_pack_forest(F, bin_size=1, interleave_depth=3, pass_bytes=-1)
    df = fp.fp_upload(pf)
    X, _ = datagen.gen_regression(53, n, 1, 1.0, 1.0)
    Xd = torch.from_numpy(X).cuda()
    ref = oracle.predict_values(F, X)
    fp.fp_inject_fault(None, fp.FP_FAULT_ALLOC, 1)
    out = df.predict_values(Xd)
    _upload_meets_no_injection(pf)
    assert df.sync_status() == fp.FP_OK
    err = np.abs(out.cpu().numpy().astype(np.float64) - ref["out"])
    assert np.all(err <= oracle.value_tolerance(F, ref["abs"]))
    df.release()


def _multi_pass(tiny_forest):
    pf = fp.fp_pack_forest(tiny_forest, bin_size=2, interleave_depth=2, pass_bytes=2048)
    assert pf.info()["passes"] > 1
    return fp.fp_upload(pf)


def _node_types(graph):
    """Types of the nodes of a captured graph that was kept (CUgraphNodeType)."""
    drv, g = ctypes.CDLL("libcuda.so.1"), ctypes.c_void_p(graph.raw_cuda_graph())
    n = ctypes.c_size_t(0)
    assert drv.cuGraphGetNodes(g, None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert drv.cuGraphGetNodes(g, nodes, ctypes.byref(n)) == 0
    types = []
    for node in nodes:
        t = ctypes.c_int(-1)
        assert drv.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(t)) == 0
        types.append(t.value)
    return types


MEMORY_NODES = {10, 11}  # CU_GRAPH_NODE_TYPE_MEM_ALLOC, CU_GRAPH_NODE_TYPE_MEM_FREE


@pytest.mark.parametrize("n", [1, 33, 3000])
def test_votes_alone_need_no_scratch(tiny_forest, tiny_rows, n):
    """A forest of several passes, votes without classes: no allocation is
    made (an injected failure waits for the next one)."""
    X = np.ascontiguousarray(tiny_rows[0][:n])
    df = _multi_pass(tiny_forest)
    Xd = torch.from_numpy(X).cuda()
    want = oracle.predict(tiny_forest, X)["votes"]
    fp.fp_inject_fault(None, fp.FP_FAULT_ALLOC, 1)
    v, _ = df.predict(Xd, classes=False)
    with pytest.raises(fp.FPError):
        fp.fp_upload(fp.fp_pack_forest(tiny_forest))
    w = torch.full((n, tiny_forest.n_classes), -1, dtype=torch.int32, device="cuda")
    fp.fp_predict_noalloc(df, Xd, w, None)
    assert df.sync_status() == fp.FP_OK
    np.testing.assert_array_equal(v.cpu().numpy().astype(np.uint32), want)
    np.testing.assert_array_equal(w.cpu().numpy().astype(np.uint32), want)
    df.release()


@pytest.mark.parametrize("several_passes", [False, True])
@pytest.mark.parametrize("classes", [False, True])
def test_memory_nodes_under_capture(tiny_forest, tiny_rows, several_passes, classes):
    """Under capture a small batch makes memory nodes only for the classes of
    a forest of several passes."""
    X = np.ascontiguousarray(tiny_rows[0][:64])
    df = _multi_pass(tiny_forest) if several_passes else fp.fp_upload(
        fp.fp_pack_forest(tiny_forest, bin_size=1, interleave_depth=3, pass_bytes=-1))
    Xd = torch.from_numpy(X).cuda()
    v = torch.empty((64, tiny_forest.n_classes), dtype=torch.int32, device="cuda")
    c = torch.empty((64,), dtype=torch.int32, device="cuda") if classes else None
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    fp.fp_predict(df, Xd, v, c, stream=s)
    s.synchronize()
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g, stream=s):
        fp.fp_predict(df, Xd, v, c, stream=torch.cuda.current_stream())
    assert bool(MEMORY_NODES & set(_node_types(g))) == (several_passes and classes)
    g.instantiate()
    v.fill_(-1)
    g.replay()
    torch.cuda.synchronize()
    ref = oracle.predict(tiny_forest, X)
    np.testing.assert_array_equal(v.cpu().numpy().astype(np.uint32), ref["votes"])
    if classes:
        np.testing.assert_array_equal(c.cpu().numpy(), ref["cls"])
    df.release()


def test_noalloc_votes_alone_overlap(tiny_forest, tiny_rows):
    """fp_predict_noalloc for votes alone leaves the shared array alone, so
    calls on two streams do not meet in it."""
    df = _multi_pass(tiny_forest)
    streams = [torch.cuda.Stream() for _ in range(2)]
    Xs = [np.ascontiguousarray(tiny_rows[0][k * 500:k * 500 + 500]) for k in range(2)]
    Xd = [torch.from_numpy(x).cuda() for x in Xs]
    vs = [[torch.full((500, tiny_forest.n_classes), -1, dtype=torch.int32, device="cuda") for _ in range(20)]
          for _ in range(2)]
    torch.cuda.synchronize()
    for i in range(20):
        for k, s in enumerate(streams):
            fp.fp_predict_noalloc(df, Xd[k], vs[k][i], None, stream=s)
    torch.cuda.synchronize()
    assert df.sync_status() == fp.FP_OK
    for k in range(2):
        want = oracle.predict(tiny_forest, Xs[k])["votes"]
        for v in vs[k]:
            np.testing.assert_array_equal(v.cpu().numpy().astype(np.uint32), want)
    df.release()


def test_noalloc_small_call_captured_after_a_large_one(tiny_forest, tiny_rows):
    """The first call on a device looks up the array, also when it is large
    enough to need none; a small classes-only call can then be captured.  A
    process of its own, since the address is kept."""
    code = """
import numpy as np, torch, datagen, oracle
import paper_1806_07300_gb300 as fp
F, X = datagen.forest("tiny"), datagen.test_rows("tiny")[0]
df = fp.fp_upload(fp.fp_pack_forest(F, bin_size=2, interleave_depth=2, pass_bytes=2048))
Xd = torch.from_numpy(np.tile(X, (16, 1))).cuda()
n = Xd.shape[0]
v, c = (torch.empty(s, dtype=torch.int32, device="cuda") for s in ((n, F.n_classes), (n,)))
fp.fp_predict_noalloc(df, Xd, v, c)
torch.cuda.synchronize()
s, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
with torch.cuda.graph(g, stream=s):
    fp.fp_predict_noalloc(df, Xd[:64], None, c[:64], stream=torch.cuda.current_stream())
c.fill_(-1)
g.replay()
torch.cuda.synchronize()
assert np.array_equal(c[:64].cpu().numpy(), oracle.predict(F, X[:64])["cls"])
"""
    subprocess.run([sys.executable, "-c", code], check=True, cwd=ROOT, timeout=600)
