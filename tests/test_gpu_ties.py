"""Rows whose values are the thresholds themselves: every walk through a head
of one-word nodes meets equal top bits, where the word's low bits are no part
of the threshold.  Whole numbers of either sign (keys whose low bits are all
zero or all one), binary features beside continuous ones, and the float
neighbours of the thresholds, for both level heads, depths and formats."""
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


def _rows(kind, n, F, seed):
    rng = np.random.default_rng(seed)
    if kind == "binary":
        X = rng.integers(0, 2, (n, F)).astype(np.float32)
    else:
        X = rng.integers(-4, 5, (n, F)).astype(np.float32)
    if kind == "mixed":
        X[:, ::2] = rng.normal(size=(n, (F + 1) // 2)).astype(np.float32)
    return X


@pytest.mark.parametrize("kind", ["binary", "whole", "mixed"])
@pytest.mark.parametrize("n_features", [3, 28])
@pytest.mark.parametrize("sel,depth", [(1, 3), (1, 6), (2, 5), (2, 7)])
@pytest.mark.parametrize("fmt", [1, 2])
def test_thresholds_on_values(kind, n_features, sel, depth, fmt):
    X = _rows(kind, 3000, n_features, 1)
    y = np.random.default_rng(2).integers(0, 3, 3000).astype(np.int32)
    F = datagen.train_forest(X, y, 3, 12, 3, seed=4)
    thr = np.floor(F.threshold).astype(np.float32)
    if kind == "mixed":  # continuous features keep theirs
        thr = np.where(F.feature % 2 == 0, F.threshold, thr).astype(np.float32)
    G = datagen.Forest(F.n_features, F.n_classes, F.node_begin, F.left, F.right, F.feature, thr, F.leaf_class,
                       F.cardinality, F.tree_depth)
    df = fp.fp_upload(fp.fp_pack_forest(G, bin_size=5, interleave_depth=depth, head_select=sel, deep_format=fmt))
    Xt = _rows(kind, 2011, n_features, 3)
    Xt[1000:] = np.nextafter(Xt[1000:], np.where(np.arange(1011) % 2, np.inf, -np.inf)[:, None].astype(np.float32))
    ref = oracle.predict(G, Xt)
    Xd = torch.from_numpy(Xt).cuda()
    v, c = df.predict(Xd)
    np.testing.assert_array_equal(v.cpu().numpy().astype(np.uint32), ref["votes"])
    np.testing.assert_array_equal(c.cpu().numpy(), ref["cls"])
    np.testing.assert_array_equal(df.predict_leaves(Xd).cpu().numpy(), ref["leaf"])
    assert df.sync_status() == fp.FP_OK
    df.release()
