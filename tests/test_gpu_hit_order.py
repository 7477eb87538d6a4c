"""Hit lists of exact lengths through the ordering at the end of a close: one
address range per block, lists beyond the host's buffer, beyond one launch, and
closes after one that made the buffer grow.

A sketch of 2^22 estimators of 32 bits with theta = 0.5 reports every address
that has a peer, so the number of hits is the number of addresses."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
SEED = 77


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


def _window(n0, n1):
    """pairs with n0 sources and n1 destinations, each address at least once"""
    n = max(n0, n1)
    rng = np.random.default_rng([n0, n1])
    a, b = (rng.permutation(np.unique(rng.integers(0, 1 << 32, m + 64, dtype=np.uint32))[:m]) for m in (n0, n1))
    return np.stack([a[np.arange(n) % n0], b[np.arange(n) % n1]], 1)


def _oracle(O, pairs):
    op = O.make_params(32, 4, 22, 8, 0.5, SEED, dirs=2)
    og = O.new_grid(op)
    O.update(op, og, pairs)
    return O.close_window(op, og)


def _handle(sd, restore=0):
    # (the staged join's work bound is the product of three rows' hot estimators)
    h = sd.sd_create(sd.sd_default_params(g=32, r=4, k=22, alpha=8, theta=0.5, seed=SEED, dirs=2, pair_cap=1 << 34))
    t = sd.sd_get_tuning(h)
    sd.sd_set_tuning(h, mode=t.mode, restore=restore)
    return h


def _dev(mods, wins):
    """the windows on the device (kept until their updates are done)"""
    return [mods[0].from_numpy(p.reshape(-1).view(np.int32)).cuda() for p in wins]


def _same(rep, ref):
    assert rep.flags == 0 and rep.n_cand == ref["n_cand"]
    for f in ("ip", "sz", "dir", "est"):
        assert np.array_equal(rep.hits[f], ref[f]), f


LENGTHS = [1, 2, 256, 257, 2047, 2048, 2049, 32_768, 32_769, 50_001, 65_536, 65_537, 140_000]


@pytest.mark.parametrize("n", LENGTHS)
def test_one_list_beside_a_short_one(mods, n):
    """The long list in either direction, twice on one handle (the second time
    into the grown buffer), and a short window behind it."""
    torch, sd, O = mods
    few = min(n, 300)
    wins = [_window(n, few), _window(few, n), _window(few, few)]
    refs = [_oracle(O, p) for p in wins]
    for ref, (n0, n1) in zip(refs, [(n, few), (few, n), (few, few)]):
        assert [int((ref["dir"] == d).sum()) for d in range(2)] == [n0, n1]
    dev = _dev(mods, wins)
    h = _handle(sd)
    try:
        for i in (0, 0, 1, 2, 1):
            sd.sd_update(h, dev[i])
            _same(sd.sd_close_window(h), refs[i])
    finally:
        sd.sd_destroy(h)


def test_both_lists_long(mods):
    """Two lists of 65,536 hits, whose ranges of 512 hits on average now and
    then hold more than a block's shared memory (one close in a hundred)."""
    torch, sd, O = mods
    pairs = _window(65_536, 65_536)
    ref = _oracle(O, pairs)
    dev = _dev(mods, [pairs])
    h = _handle(sd)
    try:
        for _ in range(50):
            sd.sd_update(h, dev[0])
            _same(sd.sd_close_window(h), ref)
    finally:
        sd.sd_destroy(h)


@pytest.mark.parametrize("restore", [0, 1])
def test_closed_together(mods, restore):
    torch, sd, O = mods
    sizes = [(2500, 300), (2048, 2049), (5, 7)] if restore else [(50_001, 300), (300, 70_000), (2048, 2049), (5, 7)]
    wins = [_window(*s) for s in sizes]
    refs = [_oracle(O, p) for p in wins]
    dev = _dev(mods, wins)
    hs = [_handle(sd, restore) for _ in wins]
    try:
        for _ in range(2):
            for h, p in zip(hs, dev):
                sd.sd_update(h, p)
            for rep, ref in zip(sd.sd_close_many(hs), refs):
                _same(rep, ref)
    finally:
        for h in hs:
            sd.sd_destroy(h)
