"""The staged join on windows that were counted in the plane copy, and switches
of the restore between windows of one handle."""
import numpy as np
import pytest

from paper_1803_11449_gb300 import traffic as T

pytestmark = pytest.mark.gpu
SEED = 0x701A


@pytest.mark.parametrize("restores", [(1, 1, 1), (1, 0, 1, 0), (0, 1, 1, 0)])
@pytest.mark.parametrize("together", [False, True])
def test_join_behind_the_plane_scan(restores, together, O):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1803_11449_gb300 import sd
    sd.lib()
    w = T.WORKLOADS["tiny"].with_(dirs=2, n=1 << 18, planted=8)
    wins = [T.make_window(w, s).pairs for s in (1, 2, 3, 4)]
    op = O.params_from(w.sketch(), seed=SEED)
    dev = [torch.from_numpy(p.reshape(-1).view(np.int32)).cuda() for p in wins]
    torch.cuda.synchronize()
    hs = [sd.sd_create(sd.params_for(w, SEED)) for _ in range(2 if together else 1)]
    try:
        for i, restore in enumerate(restores):
            feeds = [i, (i + 1) % 4][:len(hs)]
            for h, f in zip(hs, feeds):
                sd.sd_set_tuning(h, mode=6, restore=restore)
                sd.sd_update(h, dev[f])
            reps = sd.sd_close_many(hs) if together else [sd.sd_close_window(hs[0])]
            for h, f, rep in zip(hs, feeds, reps):
                og = O.new_grid(op)
                O.update(op, og, wins[f])
                ref = O.close_window(op, og, want_cands=True)
                assert rep.flags == 0 and rep.n_cand == ref["n_cand"] and rep.psi == ref["psi"]
                assert np.array_equal(rep.n_hot, ref["n_hot"]) and np.array_equal(rep.zr, ref["zr"])
                for k in ("ip", "sz", "dir", "est"):
                    assert np.array_equal(rep.hits[k], ref[k]), k
                for d in range(2):
                    assert np.array_equal(np.sort(sd.sd_get_candidates(h, d)[1]), ref["cands"][d])
                assert len(rep.hits) > 5
        # an empty window behind them, and the DHLA it leaves
        assert all(r.n_hits_total == 0 for r in (sd.sd_close_many(hs) if together else [sd.sd_close_window(hs[0])]))
        assert not any(sd.sd_get_grid(h, d).any() for h in hs for d in range(2))
    finally:
        for h in hs:
            sd.sd_destroy(h)
