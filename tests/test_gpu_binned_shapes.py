"""Binned plane rounds at the edges of the shape space and on every kind of bin
layout.  Rounds short of the tuning's full one may set their bits directly, so
the tests here tune the round to the sizes that they feed."""
import numpy as np
import pytest

from paper_1803_11449_gb300 import traffic as T

pytestmark = pytest.mark.gpu
SEED = 0xB155


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


def _dev(torch, pairs, offset=0):
    buf = torch.zeros(2 * len(pairs) + offset, dtype=torch.int32, device="cuda")
    buf[offset:] = torch.from_numpy(np.ascontiguousarray(pairs).reshape(-1).view(np.int32)).cuda()
    torch.cuda.synchronize()
    return buf[offset:]


def _launches(sd, fn):
    n = sd.sd_kernel_launches()
    fn()
    return sd.sd_kernel_launches() - n


@pytest.mark.parametrize("offset", [0, 1, 2])
@pytest.mark.parametrize("g,r,k,alpha", [
    (32, 3, 16, 16), (64, 6, 10, 6), (128, 7, 9, 6), (256, 8, 8, 4), (512, 5, 14, 6), (1024, 4, 18, 7),
    (2048, 4, 12, 10),   # 4096 planes: more than two per thread of the binning block
    (4096, 3, 17, 16),   # 8192 planes, tiles of 4096 pairs
    (4096, 8, 5, 5),     # planes of eight words
])
def test_full_rounds_of_every_shape(mods, g, r, k, alpha, offset):
    """Two full rounds (the first counted, the second on the layout it left)
    and a tail set directly, by the update of both directions."""
    torch, sd, O = mods
    w = T.WORKLOADS["tiny"].with_(g=g, r=r, k=k, alpha=alpha, theta=2 * g, dirs=2, src_pool=1 << 12, dst_pool=1 << 12,
                                  planted=0)
    pairs = T.make_window(w, 5, n=(1 << 17) + 4097).pairs
    op = O.params_from(w.sketch(), seed=SEED)
    og = O.new_grid(op)
    O.update(op, og, pairs)
    dev = _dev(torch, pairs, offset)
    h = sd.sd_create(sd.params_for(w, SEED))
    try:
        sd.sd_set_tuning(h, mode=6, plane_round_log2=16)
        # count, bin and apply; bin and apply; direct
        assert _launches(sd, lambda: sd.sd_update(h, dev)) == 6
        got = np.concatenate([sd.sd_get_grid(h, d) for d in range(2)])
    finally:
        sd.sd_destroy(h)
    assert np.array_equal(got, np.asarray(og).reshape(-1))


@pytest.mark.parametrize("sketch", ["core", "paper"])
def test_one_direction_rounds(mods, sketch):
    """sd_update_dir through the bins, between updates of both directions."""
    torch, sd, O = mods
    w = T.WORKLOADS[sketch].with_(src_pool=1 << 14, dst_pool=1 << 16, planted=0)
    x = T.make_window(w, 6, n=1 << 18).pairs
    back = np.ascontiguousarray(x[:, ::-1])  # (key, peer) pairs of direction 1
    op = O.params_from(w.sketch(), seed=SEED)
    both, half = O.new_grid(op), O.new_grid(op)
    O.update(op, both, x[:1 << 16])
    O.update(op, half, x)
    both, half = (np.asarray(a).reshape(2, -1) for a in (both, half))
    dev, dev_back = _dev(torch, x), _dev(torch, back)
    h = sd.sd_create(sd.params_for(w, SEED))
    try:
        sd.sd_set_tuning(h, mode=6, plane_round_log2=16)
        n = 2 << 16
        assert _launches(sd, lambda: sd.sd_update_dir(h, 0, dev)) == 9
        assert np.array_equal(sd.sd_get_grid(h, 0), half[0]) and not sd.sd_get_grid(h, 1).any()
        assert _launches(sd, lambda: sd.sd_update(h, dev[:n])) == 3
        assert _launches(sd, lambda: sd.sd_update_dir(h, 1, dev_back[:n])) == 3
        assert np.array_equal(sd.sd_get_grid(h, 0), half[0]) and np.array_equal(sd.sd_get_grid(h, 1), both[1])
        assert _launches(sd, lambda: sd.sd_update_dir(h, 1, dev_back)) == 8
        assert np.array_equal(sd.sd_get_grid(h, 1), half[1])
    finally:
        sd.sd_destroy(h)


def test_scaled_layouts_where_the_bins_are_tight(mods):
    """A full round after one of half its size and a little more: the bins
    have no room for that layout times two, so its counts are scaled."""
    torch, sd, O = mods
    w = T.WORKLOADS["core"].with_(src_pool=1 << 16, dst_pool=1 << 18, planted=0)
    x = T.make_window(w, 7, n=3 << 20).pairs
    y = x[::-1].copy()
    y[::3] = y[0]  # (a third of the second window in one plane: past its bin)
    op = O.params_from(w.sketch(), seed=SEED)
    m = 2 * ((1 << 20) + 77_777)
    for big in (x, y):
        og = O.new_grid(op)
        O.update(op, og, x[:m // 2])
        O.update(op, og, big[:1 << 21])
        dev, dev_big = _dev(torch, x), _dev(torch, big)
        h = sd.sd_create(sd.params_for(w, SEED))
        try:
            sd.sd_set_tuning(h, mode=6, plane_round_log2=21)
            assert _launches(sd, lambda: sd.sd_update(h, dev[:m])) == 3         # counted
            assert _launches(sd, lambda: sd.sd_update(h, dev_big[:2 << 21])) == 3  # scaled
            got = np.concatenate([sd.sd_get_grid(h, d) for d in range(2)])
        finally:
            sd.sd_destroy(h)
        assert np.array_equal(got, np.asarray(og).reshape(-1))


def test_batches_of_full_and_growing_rounds(mods):
    """Members of a batch through the driver's bins: feeds that grow beyond
    the last round's layout, and full rounds of the driver's tuning."""
    torch, sd, O = mods
    w = T.WORKLOADS["tiny"].with_(dirs=2, src_pool=1 << 14, dst_pool=1 << 16, planted=0)
    seeds = [11, 12, 13, 14, 15, 16]
    wins = [T.make_window(w, s, n=700_000).pairs for s in seeds]
    feeds = [[1 << 15, 1 << 16, (1 << 16) + 1], [1 << 17, 1 << 15, 1 << 18], [(1 << 15) + 5, 70_000, 1 << 15],
             [200_000, 1 << 15, 300_000], [1 << 15, 1 << 15, 1 << 15], [40_000, 1 << 17, 1 << 16]]
    ops = [O.params_from(w.sketch(), seed=s) for s in seeds]
    grids = [O.new_grid(op) for op in ops]
    devs = [_dev(torch, x) for x in wins]
    hs = [sd.sd_create(sd.params_for(w, s)) for s in seeds]
    try:
        for h in hs:
            sd.sd_set_tuning(h, mode=6, plane_round_log2=15)
        at = [0] * len(hs)
        for step in range(3):
            parts = []
            for i, f in enumerate(feeds):
                parts.append(devs[i][2 * at[i]:2 * (at[i] + f[step])])
                O.update(ops[i], grids[i], wins[i][at[i]:at[i] + f[step]])
                at[i] += f[step]
            sd.sd_update_many(hs, parts)
        for h, og in zip(hs, grids):
            got = np.concatenate([sd.sd_get_grid(h, d) for d in range(2)])
            assert np.array_equal(got, np.asarray(og).reshape(-1))
    finally:
        for h in hs:
            sd.sd_destroy(h)
