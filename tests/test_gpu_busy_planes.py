"""Binned rounds of thousands of planes with a few busy hosts: apply units of a
busy plane beside planes of a few keys, for one and for several units a block."""
import numpy as np
import pytest

from paper_1803_11449_gb300 import traffic as T

pytestmark = pytest.mark.gpu
SEED = 0xB057


@pytest.mark.parametrize("g,r,k,alpha", [(2048, 4, 12, 10), (4096, 3, 16, 16), (512, 4, 16, 8)])
@pytest.mark.parametrize("n", [(1 << 18) + 3, 1 << 21, (1 << 23) + 1])
@pytest.mark.parametrize("unit_log2", [8, 14])
def test_units_of_busy_planes(g, r, k, alpha, n, unit_log2, O):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1803_11449_gb300 import sd
    sd.lib()
    w = T.WORKLOADS["tiny"].with_(g=g, r=r, k=k, alpha=alpha, theta=2 * g, dirs=2, src_pool=1 << 12, dst_pool=1 << 14,
                                  planted=0)
    pairs = T.make_window(w, 3, n=n).pairs
    d = torch.from_numpy(pairs.reshape(-1).view(np.int32)).cuda()
    torch.cuda.synchronize()
    op = O.params_from(w.sketch(), seed=SEED)
    og = O.new_grid(op)
    O.update(op, og, pairs)
    h = sd.sd_create(sd.params_for(w, SEED))
    try:
        sd.sd_set_tuning(h, mode=6, plane_unit_log2=unit_log2, plane_round_log2=21)
        sd.sd_update(h, d)
        sd.sd_update(h, d)
        got = np.concatenate([sd.sd_get_grid(h, i) for i in range(2)])
    finally:
        sd.sd_destroy(h)
    assert np.array_equal(got, np.asarray(og).reshape(-1))
