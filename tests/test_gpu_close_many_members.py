"""Batched closes (sd_close_many) whose members do not all restore: the first
one overloaded, saturated or empty, the others with full hit lists."""
import numpy as np
import pytest

from paper_1803_11449_gb300 import traffic as T

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("first", ["overloaded", "saturated", "empty"])
def test_members_behind_one_that_does_not_restore(first, O):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1803_11449_gb300 import sd
    sd.lib()
    # rows 2 and 3 of the hot bitmap: 16 KiB of shared memory in each block
    w = T.WORKLOADS["core"].with_(n=1 << 20, planted=20, planted_c=("loguniform", 1024, 20000),
                                  src_pool=1 << 18, dst_pool=1 << 20)
    wins = [T.make_window(w, s).pairs for s in (21, 22, 23)]
    seeds = [210, 220, 230]
    caps = [dict(pair_cap=1) if first == "overloaded" else {}, {}, {}]
    dev = [torch.from_numpy(p.reshape(-1).view(np.int32)).cuda() for p in wins]  # (kept until the closes)
    hs = [sd.sd_create(sd.params_for(w, s, **c)) for s, c in zip(seeds, caps)]
    ops = [O.params_from(w.sketch(), seed=s, **c) for s, c in zip(seeds, caps)]
    try:
        for window in range(2):
            grids = []
            for i, (h, op, pairs, on) in enumerate(zip(hs, ops, wins, dev)):
                og = O.new_grid(op)
                if i or first != "empty":
                    sd.sd_update(h, on)
                    O.update(op, og, pairs)
                if i == 0 and first == "saturated":
                    full = np.full(og.size // 2, 0xFFFFFFFF, np.uint32)
                    for d in range(2):
                        sd.sd_set_grid(h, d, full)
                    og[:] = 0xFFFFFFFF
                grids.append(og)
            for h, op, og, rep in zip(hs, ops, grids, sd.sd_close_many(hs)):
                ref = O.close_window(op, og)
                assert [rep.dir_flags(d) for d in range(2)] == ref["flags"]
                assert rep.n_cand == ref["n_cand"] and rep.psi == ref["psi"]
                for f in ("ip", "sz", "dir", "est"):
                    assert np.array_equal(rep.hits[f], ref[f]), f
                assert h is hs[0] or len(rep.hits) > 10
            assert first == "empty" or any(O.close_window(ops[0], grids[0])["flags"])
    finally:
        for h in hs:
            sd.sd_destroy(h)
