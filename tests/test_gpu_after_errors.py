"""Calls that follow a failed one: what they return, and the window they see."""
import numpy as np
import pytest

from paper_1803_11449_gb300 import traffic as T

pytestmark = pytest.mark.gpu
SEED = 0xAF7E


@pytest.fixture(scope="module")
def mods():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import oracle as O
    from paper_1803_11449_gb300 import sd
    sd.lib()
    O.build()
    return torch, sd, O


def _dev(torch, pairs):
    return torch.from_numpy(np.ascontiguousarray(pairs).reshape(-1).view(np.int32)).cuda()


def _same(O, op, grid, rep):
    ref = O.close_window(op, grid)
    assert [rep.dir_flags(d) for d in range(op.dirs)] == ref["flags"]
    assert np.array_equal(rep.zr, ref["zr"]) and np.array_equal(rep.n_hot, ref["n_hot"])
    assert rep.n_cand == ref["n_cand"]
    for f in ("ip", "sz", "dir", "est"):
        assert np.array_equal(rep.hits[f], ref[f]), f


@pytest.mark.parametrize("mode", [1, 5, 6])
def test_out_of_memory_is_reported_once(mods, mode):
    """An allocation that fails in one call is not reported again by the
    launches of the next one, on the same or another handle."""
    torch, sd, O = mods
    w = T.WORKLOADS["core"].with_(n=1 << 17, src_pool=1 << 14, dst_pool=1 << 14, planted=4,
                                  planted_c=("uniform", 1500, 4000))
    pairs = T.make_window(w, 1).pairs
    op = O.params_from(w.sketch(), seed=SEED)
    og = O.new_grid(op)
    O.update(op, og, pairs)
    h = sd.sd_create(sd.params_for(w, SEED))
    try:
        with pytest.raises(sd.SdError):  # 2^40 candidates: 4 TiB
            sd.sd_create(sd.params_for(w, SEED, cand_cap=1 << 40))
        sd.sd_set_tuning(h, mode=5, bin_chunk_log2=28, bin_slack_pct=40000)  # bins of terabytes
        with pytest.raises(sd.SdError):
            sd.sd_update(h, _dev(torch, pairs))
        sd.sd_set_tuning(h, mode=mode, bin_chunk_log2=20, bin_slack_pct=100)
        sd.sd_update(h, _dev(torch, pairs))
        _same(O, op, og, sd.sd_close_window(h))
    finally:
        sd.sd_destroy(h)
