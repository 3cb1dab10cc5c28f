"""An upload that finds no memory for the second, one-word form of the trees'
heads keeps the packed heads, and every call walks those."""
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


def _upload_without_one_word_heads(pf):
    fp.fp_inject_fault(None, fp.FP_FAULT_ALLOC_AFTER, 1)  # the image itself
    fp.fp_inject_fault(None, fp.FP_FAULT_ALLOC, 1)
    df = fp.fp_upload(pf)
    fp.fp_upload(pf).release()  # the injection was used up
    return df


@pytest.mark.parametrize("sel,depth", [(1, 4), (2, 3), (2, 5)])
@pytest.mark.parametrize("fmt", [1, 2])
@pytest.mark.parametrize("warps", [16, 32])
def test_classification(tiny_forest, tiny_rows, sel, depth, fmt, warps):
    X = np.ascontiguousarray(tiny_rows[0][:5003])
    ref = oracle.predict(tiny_forest, X)
    pf = fp.fp_pack_forest(tiny_forest, bin_size=3, interleave_depth=depth, head_select=sel, deep_format=fmt,
                           warps_per_cta=warps)
    df, full = _upload_without_one_word_heads(pf), fp.fp_upload(pf)
    Xd = torch.from_numpy(X).cuda()
    v, c = df.predict(Xd)
    np.testing.assert_array_equal(v.cpu().numpy().astype(np.uint32), ref["votes"])
    np.testing.assert_array_equal(c.cpu().numpy(), ref["cls"])
    np.testing.assert_array_equal(df.predict_leaves(Xd).cpu().numpy(), ref["leaf"])
    cs = [torch.full((5003,), -1, dtype=torch.int32, device="cuda") for _ in range(2)]
    for other in (df, full):  # one kind of head in the launch, and two
        fp.fp_predict_batched([df, other], [Xd, Xd], None, cs)
        for c in cs:
            np.testing.assert_array_equal(c.cpu().numpy(), ref["cls"])
    assert df.sync_status() == fp.FP_OK
    df.release()
    full.release()


@pytest.mark.parametrize("sel,depth", [(1, 4), (2, 5)])
def test_values(sel, depth):
    Xt, yt = datagen.gen_regression(53, 2000, 0, 1.0, 1.0)
    F = datagen.train_regression(Xt, yt, 24, mtry=9, min_leaf=3, seed=53)
    df = _upload_without_one_word_heads(fp.fp_pack_forest(F, bin_size=3, interleave_depth=depth, head_select=sel))
    X, _ = datagen.gen_regression(53, 4099, 1, 1.0, 1.0)
    ref = oracle.predict_values(F, X)
    out = df.predict_values(torch.from_numpy(X).cuda())
    assert df.sync_status() == fp.FP_OK
    err = np.abs(out.cpu().numpy().astype(np.float64) - ref["out"])
    assert np.all(err <= oracle.value_tolerance(F, ref["abs"]))
    df.release()
