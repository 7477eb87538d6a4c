"""Plane updates in a CUDA graph: a replay runs on the bin layout that whatever
ran before it left, which may be of one direction only, or of a longer round."""
import numpy as np
import pytest

from paper_1803_11449_gb300 import traffic as T

pytestmark = pytest.mark.gpu
SEED = 0x96AF


def test_replays_between_rounds_of_other_layouts(O):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1803_11449_gb300 import sd
    sd.lib()
    w = T.WORKLOADS["core"].with_(src_pool=1 << 16, dst_pool=1 << 18, planted=0)
    big, mid, other = (T.make_window(w, s, n=n).pairs for s, n in ((1, 3_000_001), (2, 1_000_003), (3, 1_000_003)))
    op = O.params_from(w.sketch(), seed=SEED)
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        on = [torch.from_numpy(x.reshape(-1).view(np.int32)).cuda() for x in (big, mid, other)]
        buf = on[1].clone()
        h = sd.sd_create(sd.params_for(w, SEED, cuda_stream=st.cuda_stream))
        try:
            def check(*parts):
                og = O.new_grid(op)
                half = np.asarray(og).reshape(2, -1)
                for pairs, d in parts:
                    one = O.new_grid(op)
                    O.update(op, one, pairs)
                    one = np.asarray(one).reshape(2, -1)
                    for x in ((0, 1) if d is None else (d,)):
                        half[x] |= one[x]
                for d in range(2):
                    assert np.array_equal(sd.sd_get_grid(h, d), half[d]), d
                sd.sd_close_window(h)

            sd.sd_update(h, buf)                 # the state and the bins exist before the capture
            check((mid, None))
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=st):
                sd.sd_update(h, buf)
            graph.replay()
            check((mid, None))
            graph.replay()                       # the window's only update
            check((mid, None))
            graph.replay()
            rep = sd.sd_close_window(h)
            assert rep.psi[0] > 0 and sd.sd_close_window(h).psi == [0.0, 0.0]
            sd.sd_update_dir(h, 0, on[0])        # a longer layout, of one direction
            graph.replay()
            buf.copy_(on[2])
            graph.replay()
            check((big, 0), (mid, None), (other, None))
            sd.sd_update(h, on[0])               # the host's rounds between replays
            graph.replay()
            sd.sd_update(h, on[0])
            sd.sd_update_dir(h, 1, on[0].view(-1, 2).flip(1).reshape(-1).contiguous())  # (key, peer) order
            graph.replay()
            check((big, None), (other, None))
        finally:
            sd.sd_destroy(h)
