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
    dev = _dev(torch, pairs)
    h = sd.sd_create(sd.params_for(w, SEED))
    try:
        with pytest.raises(sd.SdError):  # 2^40 candidates: 4 TiB
            sd.sd_create(sd.params_for(w, SEED, cand_cap=1 << 40))
        sd.sd_set_tuning(h, mode=5, bin_chunk_log2=28, bin_slack_pct=40000)  # bins of terabytes
        with pytest.raises(sd.SdError):
            sd.sd_update(h, dev)
        sd.sd_set_tuning(h, mode=mode, bin_chunk_log2=20, bin_slack_pct=100)
        sd.sd_update(h, dev)
        _same(O, op, og, sd.sd_close_window(h))
    finally:
        sd.sd_destroy(h)


def test_a_close_without_memory_for_the_join_keeps_the_window(mods):
    """2^31 candidates: the handle's lists take 86 GB, the staged join's 275 GB.
    The close that cannot have them leaves the window as it was, alone and
    among others."""
    torch, sd, O = mods
    torch.cuda.empty_cache()
    w = T.WORKLOADS["core"].with_(n=1 << 17, src_pool=1 << 14, dst_pool=1 << 14, planted=4,
                                  planted_c=("uniform", 1500, 4000))
    wins = [T.make_window(w, s).pairs for s in (1, 2)]
    op = O.params_from(w.sketch(), seed=SEED)
    grids = [O.new_grid(op) for _ in wins]
    for og, pairs in zip(grids, wins):
        O.update(op, og, pairs)
    dev = [_dev(torch, pairs) for pairs in wins]  # (kept until their updates are done)
    h, h2 = sd.sd_create(sd.params_for(w, SEED, cand_cap=1 << 31)), sd.sd_create(sd.params_for(w, SEED))
    try:
        for window in range(2):
            sd.sd_set_tuning(h, mode=6, restore=1)
            sd.sd_update(h, dev[0])
            with pytest.raises(sd.SdError) as e:
                sd.sd_close_window(h)
            assert e.value.code == -2  # SD_ERR_NOMEM
            sd.sd_update(h2, dev[1])
            with pytest.raises(sd.SdError):
                sd.sd_close_many([h, h2])
            sd.sd_set_tuning(h, mode=6, restore=0)
            _same(O, op, grids[0], sd.sd_close_window(h))
            rep = sd.sd_close_window(h2)  # closed above, beside the one that failed
            assert rep.n_hits_total == 0 and rep.psi == [0.0, 0.0]
    finally:
        sd.sd_destroy(h)
        sd.sd_destroy(h2)
