"""Binned rounds of sketches whose bit planes have few words: a plane's atomics
meet on its words, so each apply block needs an SM to itself."""
import numpy as np
import pytest

from paper_1803_11449_gb300 import traffic as T

pytestmark = pytest.mark.gpu
SEED = 0x9A00


def test_blocks_of_narrow_planes_do_not_share_an_sm(O):
    """700,001 pairs of a sketch with 64-word planes took 2.3 times as long as
    those of the core sketch (8192 words) when several blocks ran on one SM,
    and takes 1.1 times as long now; launch times vary by a third."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1803_11449_gb300 import sd
    sd.lib()
    st = torch.cuda.Stream()
    took = {}
    with torch.cuda.stream(st):
        for g, r, k, alpha in ((32, 8, 8, 4), (512, 4, 16, 8)):
            w = T.WORKLOADS["tiny"].with_(g=g, r=r, k=k, alpha=alpha, theta=2 * g, dirs=2, src_pool=1 << 12,
                                          dst_pool=1 << 14, planted=0)
            pairs = T.make_window(w, 3, n=700_001).pairs
            d = torch.from_numpy(pairs.reshape(-1).view(np.int32)).cuda()
            h = sd.sd_create(sd.params_for(w, SEED, cuda_stream=st.cuda_stream, pair_cap=1))
            try:
                us = []
                for _ in range(25):
                    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                    torch.cuda.synchronize()
                    a.record()
                    sd.sd_update(h, d)
                    b.record()
                    torch.cuda.synchronize()
                    us.append(a.elapsed_time(b) * 1e3)
                got = np.concatenate([sd.sd_get_grid(h, i) for i in range(2)])
            finally:
                sd.sd_destroy(h)
            op = O.params_from(w.sketch(), seed=SEED)
            og = O.new_grid(op)
            O.update(op, og, pairs)
            assert np.array_equal(got, np.asarray(og).reshape(-1))
            took[g] = float(np.median(us))
    assert took[32] < 1.7 * took[512], took
