"""Forests whose trees end inside the interleaved heads (no super-nodes) have
a walk of their own: runs of a bin's trees for a slab of 32 rows.  Every head
kind, super-node kind and mode, at the sizes where runs and slabs end: one
row, a slab less and more than one, bins narrower and wider than a run, more
warps than units, two classes (counted in a register) and more."""
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


def shallow_forest(seed: int, n_trees: int, n_features: int, n_classes: int, depth: int) -> datagen.Forest:
    """Random trees of at most `depth` levels, some of them a single leaf."""
    rng = np.random.default_rng(seed)
    nb, L, R, Fe, Th, Cl = [0], [], [], [], [], []
    for t in range(n_trees):
        left, right, feat, thr, cls = [], [], [], [], []

        def node(level):
            i = len(left)
            left.append(-1); right.append(-1); feat.append(-1); thr.append(0.0); cls.append(-1)
            if level == depth or t % 7 == 3 or (level > 0 and rng.random() < 0.15):
                cls[i] = int(rng.integers(n_classes))
                return i
            feat[i] = int(rng.integers(n_features))
            thr[i] = float(np.float32(rng.normal()))
            left[i] = node(level + 1)
            right[i] = node(level + 1)
            return i

        node(0)
        L += left; R += right; Fe += feat; Th += thr; Cl += cls
        nb.append(nb[-1] + len(left))
    return datagen.Forest(n_features, n_classes, nb, L, R, Fe, np.array(Th, np.float32), Cl, np.ones(len(L), np.int64))


@pytest.mark.parametrize("n_trees,bin_size,n_features,n_classes", [(1, 1, 5, 1), (7, 3, 16, 2), (40, 40, 9, 2),
                                                                   (33, 16, 28, 7)])
@pytest.mark.parametrize("sel,depth", [(1, 4), (2, 5), (3, 6)])
@pytest.mark.parametrize("levels,fmt,warps", [(2, 0, 32), (3, 1, 16), (3, 2, 32)])
def test_votes_classes_and_leaves(n_trees, bin_size, n_features, n_classes, sel, depth, levels, fmt, warps):
    F = shallow_forest(n_trees, n_trees, n_features, n_classes, 4)
    df = fp.fp_upload(fp.fp_pack_forest(F, bin_size=bin_size, interleave_depth=depth, head_select=sel,
                                        deep_levels=levels, deep_format=fmt, warps_per_cta=warps))
    X = np.random.default_rng(1).normal(size=(5003, n_features)).astype(np.float32)
    for n in (1, 31, 33, 5003):
        ref = oracle.predict(F, X[:n])
        Xd = torch.from_numpy(X[:n].copy()).cuda()
        votes, cls = df.predict(Xd)
        leaves = df.predict_leaves(Xd)
        torch.cuda.synchronize()
        assert df.sync_status() == fp.FP_OK
        np.testing.assert_array_equal(votes.cpu().numpy().astype(np.uint32), ref["votes"])
        np.testing.assert_array_equal(cls.cpu().numpy(), ref["cls"])
        np.testing.assert_array_equal(leaves.cpu().numpy(), ref["leaf"])
    df.release()


@pytest.mark.parametrize("sel,depth,bin_size", [(1, 3, 5), (2, 3, 64), (3, 5, 8), (2, 9, 3)])
@pytest.mark.parametrize("levels", [2, 3])
def test_values(sel, depth, bin_size, levels):
    """Leaf values kept in the heads' exits; leaf ids still from the table."""
    Xt, yt = datagen.gen_regression(47, 2000, 0, 1.0, 1.0)
    F = datagen.train_regression(Xt, yt, 37, mtry=28, max_depth=4, eta=0.1, seed=47)
    df = fp.fp_upload(fp.fp_pack_forest(F, bin_size=bin_size, interleave_depth=depth, head_select=sel,
                                        deep_levels=levels))
    X, _ = datagen.gen_regression(47, 4099, 1, 1.0, 1.0)
    for n in (1, 33, 4099):
        ref = oracle.predict_values(F, X[:n])
        Xd = torch.from_numpy(X[:n].copy()).cuda()
        out = df.predict_values(Xd)
        leaves = df.predict_leaves(Xd)
        torch.cuda.synchronize()
        assert df.sync_status() == fp.FP_OK
        np.testing.assert_array_equal(leaves.cpu().numpy(), ref["leaf"])
        err = np.abs(out.cpu().numpy().astype(np.float64) - ref["out"])
        assert np.all(err <= oracle.value_tolerance(F, ref["abs"]))
    df.release()
