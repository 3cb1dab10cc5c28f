"""Rows are staged 8 features at a time: one 32-byte load where the address
allows it, two of 16 bytes or single words elsewhere.  Feature counts on both
sides of each of these, with rows that start 0, 16 or 4 bytes past a 32-byte
boundary, all equal to the oracle's."""
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


@pytest.mark.parametrize("n_features", [1, 4, 7, 8, 9, 12, 16, 20, 36, 40, 65])
@pytest.mark.parametrize("tile,fmt", [(32, 1), (64, 2), (1024, 0)])
def test_row_alignment(n_features, tile, fmt):
    rng = np.random.default_rng(n_features)
    X = rng.standard_normal((600, n_features)).astype(np.float32)
    y = ((X * np.arange(1, n_features + 1, dtype=np.float32)).sum(1) > 0).astype(np.int32)
    F = datagen.train_forest(X, y, 2, 9, seed=3, mtry=n_features)
    df = fp.fp_upload(fp.fp_pack_forest(F, bin_size=4, interleave_depth=2, obs_tile=tile, deep_format=fmt,
                                        deep_levels=3 if fmt else 2))
    Xt = rng.standard_normal((n_rows := 161, n_features)).astype(np.float32)
    Xt[5, 0], Xt[6, -1], Xt[7, 0] = np.inf, -np.inf, -0.0
    ref = oracle.predict(F, Xt)
    room = torch.empty(n_rows * n_features + 8, dtype=torch.float32, device="cuda")
    for skip in (0, 4, 1):
        Xd = room[skip:skip + n_rows * n_features].view(n_rows, n_features)
        assert Xd.data_ptr() % 32 == 4 * skip
        Xd.copy_(torch.from_numpy(Xt))
        v, c = df.predict(Xd)
        np.testing.assert_array_equal(v.cpu().numpy().astype(np.uint32), ref["votes"])
        np.testing.assert_array_equal(c.cpu().numpy(), ref["cls"])
        np.testing.assert_array_equal(df.predict_leaves(Xd).cpu().numpy(), ref["leaf"])
    assert df.sync_status() == fp.FP_OK
    df.release()
