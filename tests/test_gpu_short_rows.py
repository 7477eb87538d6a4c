"""Sketches whose rows take one or two words of a bit plane (k = 5 and 6): the
fold of the plane copy, the merge of DHLAs that hold bits and the close, for
every estimator width, against the oracle."""
import numpy as np
import pytest

from paper_1803_11449_gb300 import traffic as T

pytestmark = pytest.mark.gpu
SEED = 0x5407


@pytest.mark.parametrize("k,r,alpha", [(5, 8, 5), (6, 7, 6), (6, 8, 5), (7, 8, 5)])
@pytest.mark.parametrize("g", [32, 64, 256, 512, 1024, 4096])
def test_fold_and_close(g, k, r, alpha, O):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1803_11449_gb300 import sd
    sd.lib()
    # few enough pairs that few estimators are hot (2^(32-2k) preimages each)
    w = T.WORKLOADS["tiny"].with_(g=g, r=r, k=k, alpha=alpha, theta=g, dirs=2, n=g * 4, src_pool=1 << 10,
                                  dst_pool=1 << 10, planted=1, planted_c=("uniform", 2 * g, 3 * g))
    wins = [T.make_window(w, s).pairs for s in (1, 2, 3)]
    op = O.params_from(w.sketch(), seed=SEED)
    dev = [torch.from_numpy(x.reshape(-1).view(np.int32)).cuda() for x in wins]

    def grid(h):
        return np.concatenate([sd.sd_get_grid(h, d) for d in range(2)])

    def same(h, og):
        rep, ref = sd.sd_close_window(h), O.close_window(op, og)
        assert [rep.dir_flags(d) for d in range(2)] == ref["flags"]
        assert np.array_equal(rep.zr, ref["zr"]) and rep.n_cand == ref["n_cand"]
        for f in ("ip", "sz", "dir", "est"):
            assert np.array_equal(rep.hits[f], ref[f]), f

    a, b = (sd.sd_create(sd.params_for(w, SEED)) for _ in range(2))
    try:
        og = O.new_grid(op)
        O.update(op, og, wins[0])
        sd.sd_update(a, dev[0])
        same(a, og)                                   # a close from the plane copy
        sd.sd_update(a, dev[1])
        og = O.new_grid(op)
        O.update(op, og, wins[1])
        assert np.array_equal(grid(a), np.asarray(og).reshape(-1))
        sd.sd_update(a, dev[2])                       # on a DHLA that holds bits
        sd.sd_update(b, dev[0])
        sd.sd_merge(a, b)                             # by words
        O.update(op, og, wins[2])
        O.update(op, og, wins[0])
        sd.sd_update(a, dev[0])
        same(a, og)
    finally:
        sd.sd_destroy(a)
        sd.sd_destroy(b)
