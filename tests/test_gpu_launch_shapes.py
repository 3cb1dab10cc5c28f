"""A call's rows are launched in tiles whose bins may be split over CTAs, and a
batch of a few waves in two parts.  Batches at the edges of those choices: one
row, a slab more and less, fewer tiles than SMs (bins split, one per CTA or
several), whole waves of the smallest tile and a few rows more (two parts), for
forests of one pass and of several, each combination of outputs, and every
mode; all equal to the oracle's.  Batched launches choose their shapes too."""
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


def _slots():
    return torch.cuda.get_device_properties(0).multi_processor_count


def _sizes():
    wave = 32 * _slots()  # rows of one wave of 32-row tiles, one CTA per SM
    return [1, 31, 33, 700, wave - 1, wave, wave + 5, 2 * wave + 33]


@pytest.fixture(scope="module")
def tiny_ref(tiny_forest, tiny_rows):
    X, _ = tiny_rows
    return X, oracle.predict(tiny_forest, X)


@pytest.mark.parametrize("pass_bytes", [-1, 2048])
@pytest.mark.parametrize("bin_size,tile,fmt", [(1, 32, 1), (3, 1024, 2), (16, 64, 1), (2, 32, 0)])
def test_votes_classes_leaves(tiny_forest, tiny_ref, pass_bytes, bin_size, tile, fmt):
    X, ref = tiny_ref
    df = fp.fp_upload(fp.fp_pack_forest(tiny_forest, bin_size=bin_size, interleave_depth=3, obs_tile=tile,
                                        pass_bytes=pass_bytes, deep_format=fmt, deep_levels=3 if fmt else 2))
    for n in _sizes():
        n = min(n, X.shape[0])
        Xd = torch.from_numpy(np.ascontiguousarray(X[:n])).cuda()
        for votes, classes in [(True, True), (True, False), (False, True)]:
            v, c = df.predict(Xd, votes=votes, classes=classes)
            if votes:
                np.testing.assert_array_equal(v.cpu().numpy().astype(np.uint32), ref["votes"][:n])
            if classes:
                np.testing.assert_array_equal(c.cpu().numpy(), ref["cls"][:n])
        np.testing.assert_array_equal(df.predict_leaves(Xd).cpu().numpy(), ref["leaf"][:n])
        v = torch.full((n, 4), -1, dtype=torch.int32, device="cuda")
        c = torch.full((n,), -1, dtype=torch.int32, device="cuda")
        fp.fp_predict_noalloc(df, Xd, v, c)
        np.testing.assert_array_equal(v.cpu().numpy().astype(np.uint32), ref["votes"][:n])
        np.testing.assert_array_equal(c.cpu().numpy(), ref["cls"][:n])
    assert df.sync_status() == fp.FP_OK
    df.release()


@pytest.mark.parametrize("n_classes", [1, 3, 50])
def test_many_classes_split(n_classes):
    """The last CTA of a split tile spreads a row's classes over lanes."""
    X, _ = datagen.gen_mixture(61, max(2, n_classes), 7, 1500, 0)
    y = np.random.default_rng(2).integers(0, n_classes, 1500).astype(np.int32)
    F = datagen.train_forest(X, y, n_classes, 23, 3, seed=5)
    df = fp.fp_upload(fp.fp_pack_forest(F, bin_size=2, interleave_depth=2, head_select=1))
    Xt, _ = datagen.gen_mixture(61, max(2, n_classes), 7, 1501, 1)
    for n in (1, 40, 1501):
        ref = oracle.predict(F, Xt[:n])
        v, c = df.predict(torch.from_numpy(Xt[:n].copy()).cuda())
        np.testing.assert_array_equal(v.cpu().numpy().astype(np.uint32), ref["votes"])
        np.testing.assert_array_equal(c.cpu().numpy(), ref["cls"])
    assert df.sync_status() == fp.FP_OK
    df.release()


@pytest.mark.parametrize("pass_bytes", [-1, 4096])
def test_values_split(pass_bytes):
    Xt, yt = datagen.gen_regression(53, 2000, 0, 1.0, 1.0)
    F = datagen.train_regression(Xt, yt, 24, mtry=9, min_leaf=3, seed=53)
    df = fp.fp_upload(fp.fp_pack_forest(F, bin_size=2, interleave_depth=3, obs_tile=32, pass_bytes=pass_bytes))
    X, _ = datagen.gen_regression(53, max(_sizes()), 1, 1.0, 1.0)
    ref = oracle.predict_values(F, X, threads=oracle.default_threads())
    tol = oracle.value_tolerance(F, ref["abs"])
    for n in _sizes():
        out = df.predict_values(torch.from_numpy(X[:n].copy()).cuda())
        err = np.abs(out.cpu().numpy().astype(np.float64) - ref["out"][:n])
        assert np.all(err <= tol[:n])
    assert df.sync_status() == fp.FP_OK
    df.release()


def test_small_batch_under_capture(tiny_forest, tiny_ref):
    """While a stream is captured a forest of one pass takes no scratch, so
    the graph holds no memory nodes and can be instantiated again."""
    X, ref = tiny_ref
    df = fp.fp_upload(fp.fp_pack_forest(tiny_forest, bin_size=1, interleave_depth=3))
    Xd = torch.zeros((64, tiny_forest.n_features), device="cuda")
    c = torch.empty((64,), dtype=torch.int32, device="cuda")
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    fp.fp_predict(df, Xd, None, c, stream=s)
    s.synchronize()
    graphs = [torch.cuda.CUDAGraph() for _ in range(2)]
    for g in graphs:
        with torch.cuda.graph(g, stream=s):
            fp.fp_predict(df, Xd, None, c, stream=torch.cuda.current_stream())
    for k, g in enumerate(graphs + graphs):
        Xd.copy_(torch.from_numpy(np.ascontiguousarray(X[64 * k:64 * k + 64])))
        g.replay()
        torch.cuda.synchronize()
        np.testing.assert_array_equal(c.cpu().numpy(), ref["cls"][64 * k:64 * k + 64])
    df.release()


@pytest.mark.parametrize("sizes", [(1, 5, 33), (9000, 2, 64), (10000, 10000, 10000)])
@pytest.mark.parametrize("votes", [True, False])
def test_batched_shapes(tiny_forest, tiny_ref, sizes, votes):
    X, ref = tiny_ref
    params = [dict(bin_size=1, interleave_depth=2), dict(bin_size=2, interleave_depth=3, pass_bytes=2048),
              dict(bin_size=4, interleave_depth=1, deep_format=2)]
    dfs = [fp.fp_upload(fp.fp_pack_forest(tiny_forest, **p)) for p in params]
    Xs = [torch.from_numpy(np.ascontiguousarray(X[:n])).cuda() for n in sizes]
    vs = [torch.full((n, 4), -1, dtype=torch.int32, device="cuda") for n in sizes] if votes else None
    cs = [torch.full((n,), -1, dtype=torch.int32, device="cuda") for n in sizes]
    fp.fp_predict_batched(dfs, Xs, vs, cs)
    torch.cuda.synchronize()
    for i, n in enumerate(sizes):
        assert dfs[i].sync_status() == fp.FP_OK
        if votes:
            np.testing.assert_array_equal(vs[i].cpu().numpy().astype(np.uint32), ref["votes"][:n])
        np.testing.assert_array_equal(cs[i].cpu().numpy(), ref["cls"][:n])
        dfs[i].release()
