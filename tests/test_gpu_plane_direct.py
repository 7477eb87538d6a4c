"""Short rounds of the plane-binned update set their bits directly, longer ones
go through the bins: the DHLA equals the oracle's on both sides of the line,
for every alignment of the pairs, for repeated pairs, and for windows that mix
both kinds of round."""
import numpy as np
import pytest

from paper_1803_11449_gb300 import traffic as T

pytestmark = pytest.mark.gpu
SEED = 0xD1EC7


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


def _put(torch, pairs, offset):
    buf = torch.zeros(2 * len(pairs) + offset, dtype=torch.int32, device="cuda")
    buf[offset:] = torch.from_numpy(np.ascontiguousarray(pairs).reshape(-1).view(np.int32)).cuda()
    return buf[offset:]


def _check(mods, w, parts, offset, dirs_view=None):
    torch, sd, O = mods
    op = O.params_from(w.sketch(), seed=SEED)
    og = O.new_grid(op)
    h = sd.sd_create(sd.params_for(w, SEED))
    try:
        for p in parts:
            sd.sd_update(h, _put(torch, p, offset))
            O.update(op, og, p)
        got = np.concatenate([sd.sd_get_grid(h, d) for d in range(w.dirs)])
    finally:
        sd.sd_destroy(h)
    assert np.array_equal(got, np.asarray(og).reshape(-1))


@pytest.mark.parametrize("sketch", ["tiny", "core", "paper"])
@pytest.mark.parametrize("offset", [0, 1, 2])
def test_short_rounds(mods, sketch, offset):
    w = T.WORKLOADS[sketch].with_(src_pool=1 << 12, dst_pool=1 << 14, planted=0)
    win = T.make_window(w, 3, n=20_011).pairs
    for n in (1, 2, 31, 32, 33, 255, 257, 20_011):
        _check(mods, w, [win[:n]], offset)
    same = np.repeat(win[:9], 700, axis=0)  # runs of one pair, across warps and blocks
    _check(mods, w, [same, np.ascontiguousarray(same[::-1])], offset)


@pytest.mark.parametrize("sketch,offset", [("core", 0), ("core", 1), ("core", 2), ("tiny", 0), ("paper", 2)])
def test_both_sides_of_the_line_in_one_window(mods, sketch, offset):
    """A binned round without history, a direct one, binned ones that reuse
    and scale the layout, another direct one."""
    w = T.WORKLOADS[sketch].with_(src_pool=1 << 16, dst_pool=1 << 18, planted=0)
    win = T.make_window(w, 4, n=1_700_003).pairs
    # the line lies between 0.47 M (paper) and 0.9 M (tiny) pairs
    _check(mods, w, [win, win[:333], win[5:1_500_002], win[7:1_000_008], win[9:200_010]], offset)


def test_growing_rounds_and_shifted_traffic(mods):
    """Rounds of 0.8 M, 1.7 M, 3.3 M and 1.6 M pairs: bins of the round before
    times 1, 2 and 4, and traffic whose planes they do not fit."""
    w = T.WORKLOADS["core"].with_(src_pool=1 << 16, dst_pool=1 << 18, planted=0)
    win = T.make_window(w, 6, n=3_300_001).pairs
    other = win.copy()
    other[::2] = other[0]  # half of the pairs in one plane of either direction
    _check(mods, w, [win[:800_001], win[5:1_700_000], other, win[: 1_600_000]], 0)
    _check(mods, w, [win[:800_001], other, win], 2)
