"""Short rounds whose pairs all share their destination (an attack on one
host): all bits of a direction lie in one plane."""
import numpy as np
import pytest

from paper_1803_11449_gb300 import traffic as T

pytestmark = pytest.mark.gpu
SEED = 0x0A7


@pytest.mark.parametrize("dirs,n", [(1, 1 << 14), (2, 1 << 14), (2, 1 << 17), (2, 1 << 18), (2, 600_000)])
def test_one_victim(dirs, n, O):
    """The DHLA is the oracle's, and the round takes no more than four times
    that of distinct pairs (with the bits of up to 400,000 pairs set directly
    it took more)."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1803_11449_gb300 import sd
    sd.lib()
    w = T.WORKLOADS["tiny"].with_(dirs=dirs)
    rng = np.random.default_rng(n)
    spread = rng.integers(0, 1 << 32, (n, 2), dtype=np.uint32)
    attack = spread.copy()
    attack[:, 1] = 9
    op = O.params_from(w.sketch(), seed=SEED)
    st = torch.cuda.Stream()
    took = []
    with torch.cuda.stream(st):
        for pairs in (spread, attack):
            d = torch.from_numpy(pairs.reshape(-1).view(np.int32)).cuda()
            h = sd.sd_create(sd.params_for(w, SEED, cuda_stream=st.cuda_stream, pair_cap=1))
            try:
                us = []
                for _ in range(17):
                    sd.sd_close_window(h)
                    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                    torch.cuda.synchronize()
                    a.record()
                    sd.sd_update(h, d)
                    b.record()
                    torch.cuda.synchronize()
                    us.append(a.elapsed_time(b) * 1e3)
                got = np.concatenate([sd.sd_get_grid(h, i) for i in range(dirs)])
            finally:
                sd.sd_destroy(h)
            og = O.new_grid(op)
            O.update(op, og, pairs)
            assert np.array_equal(got, np.asarray(og).reshape(-1))
            took.append(float(np.median(us)))
    assert took[1] < 4 * took[0], took
