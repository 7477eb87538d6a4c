"""sd_update_noalloc sets bits in place: every alignment of the pairs, sizes
around its launch shapes, and a DHLA that already holds bits."""
import numpy as np
import pytest

from paper_1803_11449_gb300 import traffic as T

pytestmark = pytest.mark.gpu
SEED = 0x0A110C


@pytest.mark.parametrize("sketch", ["tiny", "core"])
@pytest.mark.parametrize("offset", [0, 1, 2, 3])
def test_in_place_sizes_and_alignments(sketch, offset):
    import torch

    import oracle as O
    from paper_1803_11449_gb300 import sd
    sd.lib()
    O.build()
    w = T.WORKLOADS[sketch].with_(src_pool=1 << 12, dst_pool=1 << 14, planted=0)
    # 152 SMs: the short launch ends at 152 * 4096 pairs
    win = T.make_window(w, 9, n=152 * 4096 + 257).pairs
    p = sd.params_for(w, SEED)
    op = O.params_from(w.sketch(), seed=SEED)
    og = O.new_grid(op)
    grid = torch.zeros(p.dirs * sd.sd_grid_words(p), dtype=torch.int32, device="cuda")
    for n in (1, 2, 3, 127, 129, 5001, 152 * 4096 - 1, len(win)):
        part = win[len(win) - n:]
        buf = torch.zeros(2 * n + offset, dtype=torch.int32, device="cuda")
        buf[offset:] = torch.from_numpy(part.reshape(-1).view(np.int32)).cuda()
        assert sd.sd_update_noalloc(p, grid, buf[offset:], torch.cuda.current_stream()) == sd.SD_OK
        O.update(op, og, part)
        assert np.array_equal(grid.cpu().numpy().view(np.uint32), np.asarray(og).reshape(-1)), n
