"""The close that counts the plane copy as it is, against the oracle: shapes
at the edges of its tiles (words per row below and above a block's, 8, 16 and
32 words per estimator), windows after windows on one handle, and every other
reader of the DHLA in between."""
import numpy as np
import pytest

from paper_1803_11449_gb300 import traffic as T

pytestmark = pytest.mark.gpu
SEED = 0xD1A0


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


def _window(g, r, k, alpha, theta, n, pool, planted, c, dirs, seed):
    w = T.WORKLOADS["tiny"].with_(g=g, r=r, k=k, alpha=alpha, theta=theta, dirs=dirs, n=n, src_pool=pool,
                                  dst_pool=pool, planted=planted, planted_c=("uniform",) + c)
    return w, T.make_window(w, seed).pairs


def _same(O, op, pairs, rep, grid=None):
    og = O.new_grid(op) if grid is None else grid
    if grid is None:
        O.update(op, og, pairs)
    ref = O.close_window(op, og)
    assert np.array_equal(rep.zr, np.asarray(ref["zr"])[: rep.zr.shape[0], : rep.zr.shape[1]])
    assert np.array_equal(rep.n_hot, np.asarray(ref["n_hot"])[: rep.n_hot.shape[0], : rep.n_hot.shape[1]])
    assert rep.n_cand == list(ref["n_cand"]) and rep.psi == list(ref["psi"])
    for f in ("ip", "sz", "dir", "est"):
        assert np.array_equal(rep.hits[f], ref[f]), f


SHAPES = [
    (256, 4, 12, 10, 300, 1 << 17, 1 << 12, 8, (400, 900), 1),    # 128 words a row, 32 a block
    (256, 7, 8, 5, 300, 30_000, 1 << 9, 3, (400, 900), 2),        # 8 words a row, 32 a block
    (512, 6, 9, 6, 500, 60_000, 1 << 10, 4, (700, 1500), 2),      # 16 and 16
    (1024, 5, 11, 7, 1024, 1 << 18, 1 << 12, 6, (1500, 3000), 2),  # 64 and 8
    (1024, 3, 17, 16, 1024, 1 << 18, 1 << 14, 6, (1500, 3000), 1),
]


@pytest.mark.parametrize("g,r,k,alpha,theta,n,pool,planted,c,dirs", SHAPES)
def test_scan_matches_oracle_window_after_window(mods, g, r, k, alpha, theta, n, pool, planted, c, dirs):
    torch, sd, O = mods
    w, a = _window(g, r, k, alpha, theta, n, pool, planted, c, dirs, 5)
    _, b = _window(g, r, k, alpha, theta, n // 3 | 1, pool, planted, c, dirs, 6)
    op = O.params_from(w.sketch(), seed=SEED)
    h = sd.sd_create(sd.params_for(w, SEED))
    try:
        for pairs in (a, b, a):
            sd.sd_update(h, torch.from_numpy(pairs.reshape(-1).view(np.int32)).cuda())
            _same(O, op, pairs, sd.sd_close_window(h))
        rep = sd.sd_close_window(h)  # an empty window on the stale DHLA
        assert rep.n_hits_total == 0 and rep.psi == [0.0] * dirs
    finally:
        sd.sd_destroy(h)


def test_every_reader_after_a_scan(mods):
    """After a close the DHLA's words are stale: checkpoint reads and writes,
    merges, exports and the other update modes must all see it empty."""
    torch, sd, O = mods
    g, r, k, alpha, theta, n, pool, planted, c, dirs = SHAPES[2]
    w, a = _window(g, r, k, alpha, theta, n, pool, planted, c, dirs, 5)
    _, b = _window(g, r, k, alpha, theta, n, pool, planted, c, dirs, 7)
    op = O.params_from(w.sketch(), seed=SEED)
    da, db = (torch.from_numpy(x.reshape(-1).view(np.int32)).cuda() for x in (a, b))
    words = sd.sd_grid_words(sd.params_for(w, SEED))
    ob = O.new_grid(op)
    O.update(op, ob, b)
    both = O.new_grid(op)
    O.update(op, both, a)
    O.update(op, both, b)
    flat = np.asarray(ob, np.uint32).reshape(-1)

    def closed():
        h = sd.sd_create(sd.params_for(w, SEED))
        sd.sd_update(h, da)
        sd.sd_close_window(h)
        return h

    def grid(h):
        return np.concatenate([sd.sd_get_grid(h, d) for d in range(dirs)])

    h, h2 = closed(), closed()
    try:
        assert not grid(h).any()                         # read right after the close
        sd.sd_update(h, db)
        assert np.array_equal(grid(h), flat)             # folded into the cleared DHLA
        _same(O, op, b, sd.sd_close_window(h))           # by the fold path: the DHLA held bits
        sd.sd_update(h, da)
        sd.sd_close_window(h)
        for mode in (0, 5):                              # a stale DHLA updated in place
            sd.sd_set_tuning(h, mode=mode, bin_chunk_log2=16)
            sd.sd_update(h, db)
            _same(O, op, b, sd.sd_close_window(h))
            sd.sd_set_tuning(h, mode=6)
            sd.sd_update(h, da)
            sd.sd_close_window(h)
        img = torch.zeros(dirs * words, dtype=torch.int32, device="cuda")
        sd.sd_export_grid(h, img)
        sd.sd_sync(h)
        assert not img.any().item()
        sd.sd_update(h, da)
        sd.sd_update(h2, db)
        sd.sd_merge(h, h2)                               # plane copies merged as such
        sd.sd_update(h, db)
        _same(O, op, None, sd.sd_close_window(h), both)
        _same(O, op, b, sd.sd_close_window(h2))          # the source keeps its window
        sd.sd_update(h, da)
        assert grid(h).any()                             # now the DHLA holds bits: merged by words
        sd.sd_update(h2, db)
        sd.sd_merge(h, h2)
        both = O.new_grid(op)
        O.update(op, both, a)
        O.update(op, both, b)
        _same(O, op, None, sd.sd_close_window(h), both)
        _same(O, op, b, sd.sd_close_window(h2))
        for x in (h, h2):
            sd.sd_update(x, da)
            sd.sd_close_window(x)
        for d in range(dirs):
            sd.sd_set_grid(h, d, flat[d * words:(d + 1) * words])
        sd.sd_update(h2, db)
        ra, rb = sd.sd_close_many([h, h2])               # one by its words, one by its plane copy
        _same(O, op, b, ra)
        _same(O, op, b, rb)
    finally:
        sd.sd_destroy(h)
        sd.sd_destroy(h2)
