"""The sweep pass by pass of a forest larger than L2 by tiles of 32 rows, in
batches of many waves (at, below and above the number of rows from which it
is taken): votes, classes and leaf ids equal those of the default tiles, and
the oracle's on a sample."""
import numpy as np
import pytest

import datagen
import oracle
import paper_1806_07300_gb300 as fp

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_small_tiles_on_the_large_forest():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    F = datagen.forest("hbm")
    small = fp.fp_upload(fp.fp_pack_forest(F, obs_tile=32, warps_per_cta=32))
    default = fp.fp_upload(fp.fp_pack_forest(F))
    assert small.info["passes"] > 1
    assert 32 * small.info["n_super"] > 0.75 * torch.cuda.get_device_properties(0).L2_cache_size
    edge = 8 * 32 * torch.cuda.get_device_properties(0).multi_processor_count  # one CTA to an SM
    X, _ = datagen.test_rows("hbm", edge + 33)
    Xd = torch.from_numpy(X).cuda()
    want_v, want_c = default.predict(Xd)
    want_l = default.predict_leaves(Xd)
    ref = oracle.predict(F, X[-500:])
    np.testing.assert_array_equal(want_c[-500:].cpu().numpy(), ref["cls"])
    np.testing.assert_array_equal(want_l[-500:].cpu().numpy(), ref["leaf"])
    for n in (edge - 1, edge, edge + 33):
        v, c = small.predict(Xd[:n])
        assert torch.equal(v, want_v[:n]) and torch.equal(c, want_c[:n])
        v.fill_(-1)
        fp.fp_predict(small, Xd[:n], v, None)
        assert torch.equal(v, want_v[:n])
        c.fill_(-1)
        fp.fp_predict_noalloc(small, Xd[:n], v, c)
        assert torch.equal(v, want_v[:n]) and torch.equal(c, want_c[:n])
        assert torch.equal(small.predict_leaves(Xd[:n]), want_l[:n])
    assert small.sync_status() == fp.FP_OK
    small.release()
    default.release()
