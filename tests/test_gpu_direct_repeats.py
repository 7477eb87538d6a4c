"""Short rounds in which flows repeat: the bits are the oracle's wherever the
equal pairs lie, and a flow that makes up half of the packets does not make
the round slower than one without repeats."""
import numpy as np
import pytest

from paper_1803_11449_gb300 import traffic as T

pytestmark = pytest.mark.gpu
SEED = 0xD0B


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


def _mixed(n, share, flows, seed):
    """n distinct pairs, a share of them replaced by a few flows, interleaved"""
    w = T.WORKLOADS["tiny"].with_(src_pool=1 << 16, dst_pool=1 << 20, planted=0)
    x = T.make_window(w, seed, n=n).pairs.copy()
    rng = np.random.default_rng(seed)
    at = rng.random(n) < share
    x[at] = x[rng.integers(0, flows, n)][at]
    return x


@pytest.mark.parametrize("dirs", [1, 2])
@pytest.mark.parametrize("offset", [0, 1])
def test_bits_with_repeats(mods, dirs, offset):
    torch, sd, O = mods
    w = T.WORKLOADS["tiny"].with_(dirs=dirs)
    op = O.params_from(w.sketch(), seed=SEED)
    # below, at and above one block's tile, and above the tiles of one launch
    for n, share, flows in ((200, .5, 1), (255, 1., 1), (256, .9, 2), (257, .5, 3), (5000, .3, 50), (300_001, .6, 7)):
        x = _mixed(n, share, flows, n)
        x[::17] = 0  # pairs of zeros, as in the threads past the end
        og = O.new_grid(op)
        O.update(op, og, x)
        buf = torch.zeros(2 * n + offset, dtype=torch.int32, device="cuda")
        buf[offset:] = torch.from_numpy(x.reshape(-1).view(np.int32)).cuda()
        torch.cuda.synchronize()
        h = sd.sd_create(sd.params_for(w, SEED))
        try:
            sd.sd_update(h, buf[offset:])
            got = np.concatenate([sd.sd_get_grid(h, d) for d in range(dirs)])
        finally:
            sd.sd_destroy(h)
        assert np.array_equal(got, np.asarray(og).reshape(-1)), (n, share, flows)


def test_a_heavy_flow_does_not_serialise(mods):
    """Half of 2^19 packets in one flow, interleaved with the others, took 7
    times as long as none; equal pairs of a block set once, they take less.
    Launch times vary by a third, so the line is at 2.5."""
    torch, sd, O = mods
    st = torch.cuda.Stream()
    w = T.WORKLOADS["tiny"].with_(dirs=1)
    with torch.cuda.stream(st):
        h = sd.sd_create(sd.params_for(w, SEED, cuda_stream=st.cuda_stream))
        try:
            took = []
            for share in (0.0, 0.5):
                d = torch.from_numpy(_mixed(1 << 19, share, 1, 5).reshape(-1).view(np.int32)).cuda()
                us = []
                for _ in range(25):
                    sd.sd_close_window(h)
                    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                    torch.cuda.synchronize()
                    a.record()
                    sd.sd_update(h, d)
                    b.record()
                    torch.cuda.synchronize()
                    us.append(a.elapsed_time(b) * 1e3)
                took.append(float(np.median(us)))
        finally:
            sd.sd_destroy(h)
    assert took[1] < 2.5 * took[0], took
