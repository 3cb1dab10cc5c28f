"""Votes and classes of tiles whose bins are not split, by the number of
classes: below and at the numbers from which a slab's classes are spread over
the warps (32 with votes, 128 without), with parts that end unevenly, and the most there can be; tiles of
one slab to several, fewer and more warps than slabs, and ties."""
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


@pytest.mark.parametrize("n_classes", [31, 32, 33, 127, 128, 511, 512])
@pytest.mark.parametrize("tile,warps", [(32, 32), (96, 1), (128, 6)])
def test_unsplit_tiles(n_classes, tile, warps):
    X, _ = datagen.gen_mixture(61, n_classes, 7, 2000, 0)
    y = np.random.default_rng(2).integers(0, n_classes, 2000).astype(np.int32)
    F = datagen.train_forest(X, y, n_classes, 5, 3, seed=5)  # few trees: most classes tie
    df = fp.fp_upload(fp.fp_pack_forest(F, bin_size=3, interleave_depth=2, obs_tile=tile, warps_per_cta=warps,
                                        pass_bytes=-1))
    Xt, _ = datagen.gen_mixture(61, n_classes, 7, 1001, 1)
    for n in (1, 31, 97, 1001):
        ref = oracle.predict(F, Xt[:n])
        Xd = torch.from_numpy(Xt[:n].copy()).cuda()
        v = torch.full((n, n_classes), -1, dtype=torch.int32, device="cuda")
        c = torch.full((n,), -1, dtype=torch.int32, device="cuda")
        for votes, classes in ((v, c), (v, None), (None, c)):
            v.fill_(-1)
            c.fill_(-1)
            fp.fp_predict_noalloc(df, Xd, votes, classes)  # a forest of one pass: never split
            if votes is not None:
                np.testing.assert_array_equal(v.cpu().numpy().astype(np.uint32), ref["votes"])
            if classes is not None:
                np.testing.assert_array_equal(c.cpu().numpy(), ref["cls"])
    assert df.sync_status() == fp.FP_OK
    df.release()
