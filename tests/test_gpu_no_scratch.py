"""Calls that would split a small batch's bins over the GPU, and then find no
scratch to add the splits up in.  The failure is injected as a request that
the runtime itself refuses, so the thread is left as a real failure leaves it."""
import numpy as np
import pytest

import datagen
import oracle
import paper_1806_07300_gb300 as fp

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


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
