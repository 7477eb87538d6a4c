"""Where a short round stops setting its bits directly: sketches of narrow
planes go through the bins from fewer pairs on, and no round of either side is
much slower than the binned round of its size."""
import numpy as np
import pytest

from paper_1803_11449_gb300 import traffic as T

pytestmark = pytest.mark.gpu
SEED = 0xD11E


def _window(sketch, n):
    g, r, k, alpha, dirs = sketch
    w = T.WORKLOADS["tiny"].with_(g=g, r=r, k=k, alpha=alpha, theta=2 * g, dirs=dirs, src_pool=1 << 12,
                                  dst_pool=1 << 14, planted=0)
    return w, T.make_window(w, 3, n=n).pairs


@pytest.mark.parametrize("log2_n", [14, 16, 17, 18])
@pytest.mark.parametrize("sketch", [(32, 8, 8, 4, 2), (32, 8, 8, 4, 1), (64, 6, 10, 6, 2), (256, 8, 8, 4, 2),
                                    (256, 4, 12, 10, 2), (512, 4, 14, 9, 2), (512, 4, 16, 8, 2)])
def test_rounds_by_the_line_and_through_the_bins(sketch, log2_n, O):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1803_11449_gb300 import sd
    sd.lib()
    w, pairs = _window(sketch, 1 << log2_n)
    st = torch.cuda.Stream()
    took, grids = [], []
    with torch.cuda.stream(st):
        d = torch.from_numpy(pairs.reshape(-1).view(np.int32)).cuda()
        for binned in (False, True):
            h = sd.sd_create(sd.params_for(w, SEED, cuda_stream=st.cuda_stream, pair_cap=1))
            try:
                if binned:  # a full round of the tuning is always binned
                    sd.sd_set_tuning(h, mode=6, plane_round_log2=log2_n)
                sd.sd_update(h, d)
                grids.append(np.concatenate([sd.sd_get_grid(h, i) for i in range(w.dirs)]))
                us = []
                for _ in range(15):
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
    assert np.array_equal(grids[0], grids[1])
    op = O.params_from(w.sketch(), seed=SEED)
    og = O.new_grid(op)
    O.update(op, og, pairs)
    assert np.array_equal(grids[0], np.asarray(og).reshape(-1))
    # launch times vary by a third; 64-word planes took 2.3 times as long at 2^17 pairs
    assert took[0] < 1.6 * took[1], took
