"""Workloads of the super-point detector, as its users run it.

Every case is a whole piece of work through the Python binding of the C ABI
(``paper_1803_11449_gb300/sd.py``): the pairs of one or more windows are fed
to their handles and the windows are closed, and the outputs are the reports
(hits with their estimates, psi, ZR, |HE(i)|, |K|); ``noalloc`` feeds a
caller-owned DHLA and its output is that DHLA.

Traffic is drawn on the GPU with the recipe of
``paper_1803_11449_gb300/traffic.py``: Zipf-distributed sources over a pool,
uniform destinations, planted super points with distinct peers in one
direction or the other, all positions mixed.

Kinds of case:
  window     one window: sd_update over its pairs, then sd_close_window
  stream     a window that arrives in batches, one sd_update each, then the close
  pipelined  two sketches of a link in turn: both windows are queued, the
             first closes while the second is ingested
  batch      many links' windows of different sizes: sd_update_many, sd_close_many
  merge      monitors with a part of the traffic each: sd_update on every
             handle, sd_merge into the first, one close
  host       a window in pinned host memory (a capture buffer), then the close
  noalloc    sd_update_noalloc into a caller-owned DHLA
"""
import math
import random

import numpy as np
import torch

from paper_1803_11449_gb300 import sd

HASH_SEED = 0x5D5A0002
M32 = 0xFFFFFFFF

# DHLA shapes and the traffic that goes with them: the workloads of traffic.py.
SKETCHES = {
    "tiny": dict(g=256, r=4, k=12, alpha=10, dirs=1, src_pool=1 << 16, zipf=1.1, dst_pool=0,
                 planted=20, c_lo=1500, c_hi=4000, share=0.5, flow=1),
    "core": dict(g=512, r=4, k=16, alpha=8, dirs=2, src_pool=1 << 24, zipf=1.05, dst_pool=1 << 26,
                 planted=500, c_lo=1024, c_hi=200_000, share=0.5, flow=1),
    # the paper's own parameters
    "paper": dict(g=1024, r=5, k=14, alpha=6, dirs=2, src_pool=1 << 24, zipf=1.05, dst_pool=1 << 26,
                  planted=500, c_lo=1024, c_hi=200_000, share=0.5, flow=1),
    # a DHLA of 128 MiB per direction, eight packets per flow
    "stress": dict(g=1024, r=4, k=18, alpha=7, dirs=2, src_pool=1 << 28, zipf=1.0, dst_pool=1 << 30,
                   planted=10_000, c_lo=1024, c_hi=10_000_000, share=0.1, flow=8),
}

# rows of the report that a program keeps per window (of a batch: per link); its report_cap
ROWS, ROWS_BATCH = 1 << 17, 1 << 15
THETA = 1024.0


def listed():
    return [
        # a latency-bound ingest thread hands over one short batch at a time
        dict(name="noalloc_batch", kind="noalloc", sketch="core", n=100_003, offset=0),
        # a quiet link: one short batch in the whole window, so the close decides
        dict(name="quiet_link", kind="window", sketch="core", n=65_537, offset=0),
        # a small one-direction monitor
        dict(name="small_monitor", kind="window", sketch="tiny", n=1 << 20, offset=0),
        # an ordinary link's window, cut out of a ring at an odd place
        dict(name="ragged_link", kind="window", sketch="core", n=3_999_983, offset=2),
        # serving: a window that fills from batches of 64K to 4M pairs
        dict(name="served_window", kind="stream", sketch="core", batches=12, lo=1 << 16, hi=1 << 22, split=4),
        # the paper's own sketch at a load it can resolve
        dict(name="paper_sketch", kind="window", sketch="paper", n=1 << 22, offset=0),
        # four monitors of one network, merged into one report
        dict(name="four_monitors", kind="merge", sketch="core", n=1 << 24, parts=4),
        # a capture buffer in host memory
        dict(name="host_capture", kind="host", sketch="core", n=(1 << 25) + 12_345),
        # the core-link window, the default benchmark's
        dict(name="core_window", kind="window", sketch="core", n=1 << 26, offset=0),
        # the same link without a gap: one window closes while the next is ingested
        dict(name="core_pipelined", kind="pipelined", sketch="core", n=1 << 26),
        # many links on one GPU, lognormal window sizes
        dict(name="many_links", kind="batch", sketch="core", links=64, median=4 << 20, lo=1 << 18, hi=1 << 26,
             split=3),
        # the largest: a backbone's window on a DHLA larger than L2
        dict(name="backbone", kind="window", sketch="stress", n=1 << 30, offset=0),
    ]


def _log_between(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: the same kinds and sketches over the sizes between."""
    kind = rng.choice(["window", "window", "window", "window", "stream", "pipelined", "batch", "merge", "host",
                       "noalloc"])
    if kind == "window":
        s = rng.choice(["tiny", "core", "core", "paper", "stress"])
        lo, hi = {"tiny": (1 << 14, 1 << 22), "core": (1 << 14, 1 << 26), "paper": (1 << 14, 1 << 26),
                  "stress": (1 << 20, 1 << 29)}[s]
        return dict(kind=kind, sketch=s, n=_log_between(rng, lo, hi), offset=rng.choice([0, 0, 2, 1]))
    if kind == "stream":
        return dict(kind=kind, sketch=rng.choice(["core", "core", "paper"]), batches=rng.randint(2, 24),
                    lo=1 << 16, hi=1 << 22, split=rng.randrange(1 << 20))
    if kind == "pipelined":
        return dict(kind=kind, sketch="core", n=_log_between(rng, 1 << 20, 1 << 26))
    if kind == "batch":
        return dict(kind=kind, sketch="core", links=rng.randint(2, 64), median=4 << 20, lo=1 << 18, hi=1 << 25,
                    split=rng.randrange(1 << 20))
    if kind == "merge":
        return dict(kind=kind, sketch="core", n=_log_between(rng, 1 << 18, 1 << 25), parts=rng.randint(2, 6))
    if kind == "host":
        return dict(kind=kind, sketch="core", n=_log_between(rng, 1 << 18, 1 << 25))
    return dict(kind=kind, sketch="core", n=_log_between(rng, 1 << 14, 1 << 22), offset=rng.choice([0, 2]))


# ------------------------------------------------------------------- traffic
def _mix32(x):
    """A bijection of 32-bit values held in int64."""
    x = x ^ (x >> 16)
    x = (x * 0x7FEB352D) & M32
    x = x ^ (x >> 15)
    x = (x * 0x846CA68B) & M32
    return x ^ (x >> 16)


def _zipf(u, pool, s):
    """Zipf(s) ranks 0 .. pool - 1 from uniforms u (inverse of the continuous law)."""
    a, b = 0.5, pool + 0.5
    if abs(s - 1.0) < 1e-9:
        x = a * torch.exp(u * math.log(b / a))
    else:
        e = 1.0 - s
        x = (u * (b ** e - a ** e) + a ** e) ** (1.0 / e)
    return torch.clamp(torch.floor(x + 0.5), 1, pool).to(torch.int64) - 1


def _traffic(sk, n, seed, offset=0):
    """int32 words of n (src, dst) pairs on the GPU, `offset` words into their buffer."""
    dev = "cuda"
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    host = random.Random(seed)
    salt = host.getrandbits(32)
    # planted super points: log-uniform numbers of distinct peers, scaled to their share of the pairs
    lo, hi = math.log(sk["c_lo"]), math.log(sk["c_hi"])
    c = np.array([int(math.exp(host.uniform(lo, hi))) for _ in range(sk["planted"])], dtype=np.float64)
    c = np.maximum(1, np.floor(c * min(1.0, sk["share"] * n / c.sum()))).astype(np.int64)
    ends = torch.from_numpy(np.cumsum(c)).to(dev)
    planted = min(int(c.sum()), n)
    # position p of the window holds pair (p step + start) mod n: pairs below
    # `planted` are planted, the others natural
    step = int(n * 0.6180339887498949) | 1
    while math.gcd(step, n) != 1:
        step += 2
    start = host.randrange(n)
    flows = (n - planted) // sk["flow"] + 1
    buf = torch.empty(2 * n + offset, dtype=torch.int32, device=dev)
    out = buf[offset:].view(n, 2)
    fseed = host.getrandbits(31)
    chunk = 1 << 25
    for p0 in range(0, n, chunk):
        m = min(chunk, n - p0)
        j = (torch.arange(p0, p0 + m, device=dev) * step + start) % n
        if sk["flow"] > 1:
            # the flow's own source and destination, the same for all its packets
            f = torch.where(j < planted, 0, (j - planted) % flows)
            h1 = _mix32((f ^ (fseed & M32)) & M32)
            h2 = _mix32((h1 + 0x9E3779B9) & M32)
            h3 = _mix32((h2 ^ f) & M32)
            u = (h1.double() * 4294967296.0 + h2.double()) / 18446744073709551616.0
            d = h3 & (sk["dst_pool"] - 1)
        else:
            u = torch.rand(m, dtype=torch.float64, device=dev, generator=gen)
            d = torch.randint(0, sk["dst_pool"] or (1 << 32), (m,), device=dev, generator=gen)
        src = _mix32(_zipf(u, sk["src_pool"], sk["zipf"]) ^ salt)
        dst = _mix32(((0x20000000 + d) & M32) ^ salt) if sk["dst_pool"] else d
        owner = torch.clamp(torch.searchsorted(ends, j, right=True), max=sk["planted"] - 1)
        key = _mix32((0x70000000 + owner) ^ salt)
        peer = _mix32(((0x80000000 + j) & M32) ^ salt)
        inbound = (owner & 1 == 1) if sk["dirs"] == 2 else torch.zeros_like(owner, dtype=torch.bool)
        src = torch.where(j < planted, torch.where(inbound, peer, key), src)
        dst = torch.where(j < planted, torch.where(inbound, key, peer), dst)
        for col, v in ((0, src), (1, dst)):
            out[p0:p0 + m, col] = torch.where(v > 0x7FFFFFFF, v - (1 << 32), v).to(torch.int32)
    torch.cuda.synchronize()
    return buf[offset:]


def _sizes(case):
    """Pairs of every batch (stream) or link (batch)."""
    r = random.Random(case["split"])
    if case["kind"] == "stream":
        return [r.randint(case["lo"], case["hi"]) for _ in range(case["batches"])]
    return [int(min(max(case["median"] * math.exp(r.gauss(0.0, 1.0)), case["lo"]), case["hi"]))
            for _ in range(case["links"])]


def _inputs(case, seed):
    """The pair buffers of a case, as the windows they belong to: a list of
    lists of tensors (window by window, the buffers of each)."""
    sk = SKETCHES[case["sketch"]]
    kind = case["kind"]
    if kind == "pipelined":
        return [[_traffic(sk, case["n"], 2 * seed)], [_traffic(sk, case["n"], 2 * seed + 1)]]
    if kind == "batch":
        return [[_traffic(sk, n, 1000 * seed + i)] for i, n in enumerate(_sizes(case))]
    if kind == "stream":
        sizes = _sizes(case)
        w = _traffic(sk, sum(sizes), seed)
        ends = np.cumsum(sizes)
        return [[w[2 * (e - n):2 * e] for n, e in zip(sizes, ends)]]
    if kind == "merge":
        w = _traffic(sk, case["n"], seed)
        cut = [case["n"] * i // case["parts"] for i in range(case["parts"] + 1)]
        return [[w[2 * a:2 * b] for a, b in zip(cut, cut[1:])]]
    return [[_traffic(sk, case["n"], seed, case.get("offset", 0))]]


# --------------------------------------------------------------------- cases
class State:
    """Handles and buffers of one case; the handles go with the object."""

    def __init__(self, kind):
        self.kind = kind
        self.handles = []
        self.pairs = []
        self.params = None
        self.grid = None
        self.out = None

    def __del__(self):
        for h in self.handles:
            sd.sd_destroy(h)


def _params(case, **over):
    sk = SKETCHES[case["sketch"]]
    return sd.sd_default_params(g=sk["g"], r=sk["r"], k=sk["k"], alpha=sk["alpha"], dirs=sk["dirs"], theta=THETA,
                                seed=HASH_SEED, **over)


def prepare(case, seed):
    st = State(case["kind"])
    wins = _inputs(case, seed)
    st.out = _buffers(len(wins), SKETCHES[case["sketch"]], ROWS_BATCH if case["kind"] == "batch" else ROWS)
    if case["kind"] == "noalloc":
        st.params = _params(case)
        st.pairs = wins[0][0]
        words = st.params.dirs * sd.sd_grid_words(st.params)
        st.grid = torch.zeros(words, dtype=torch.int32, device="cuda")
    elif case["kind"] == "batch":
        st.handles = [sd.sd_create(_params(case, cand_cap=1 << 18, report_cap=ROWS_BATCH)) for _ in wins]
        st.pairs = [w[0] for w in wins]
    elif case["kind"] == "pipelined":
        st.handles = [sd.sd_create(_params(case, report_cap=ROWS)) for _ in wins]
        st.pairs = [w[0] for w in wins]
    elif case["kind"] == "merge":
        st.handles = [sd.sd_create(_params(case, report_cap=ROWS)) for _ in wins[0]]
        st.pairs = wins[0]
    else:
        st.handles = [sd.sd_create(_params(case, report_cap=ROWS))]
        st.pairs = wins[0]
        if case["kind"] == "host":
            st.pairs = [wins[0][0].cpu().pin_memory()]
    torch.cuda.synchronize()
    return st


def _buffers(windows, sk, rows):
    """The program's own report store: rows of hits and the scalars, per window."""
    w, d, r = windows, sk["dirs"], sk["r"]
    return {"ip": np.zeros((w, rows), np.uint32), "sz": np.zeros((w, rows), np.uint32),
            "dir": np.zeros((w, rows), np.uint8), "est": np.zeros((w, rows)), "psi": np.zeros((w, d)),
            "zr": np.zeros((w, d, r), np.int64), "n_hot": np.zeros((w, d, r), np.int64),
            "n_cand": np.zeros((w, d), np.int64), "szmax": np.zeros((w, d), np.int64),
            # rc, zhot, flags, pairs, hits
            "window": np.zeros((w, 5), np.int64)}


def _store(out, w, rep):
    n = len(rep.hits)
    for name in ("ip", "sz", "dir", "est"):
        out[name][w, :n] = rep.hits[name]
    out["psi"][w], out["zr"][w], out["n_hot"][w] = rep.psi, rep.zr, rep.n_hot
    out["n_cand"][w], out["szmax"][w] = rep.n_cand, rep.szmax
    out["window"][w] = rep.rc, rep.zhot, rep.flags, rep.n_pairs, rep.n_hits_total


def run(state):
    h, pairs = state.handles, state.pairs
    if state.kind == "noalloc":
        rc = sd.sd_update_noalloc(state.params, state.grid, pairs, torch.cuda.current_stream())
        return {"rc": rc, "grid": state.grid}
    if state.kind == "batch":
        sd.sd_update_many(h, pairs)
        for w, rep in enumerate(sd.sd_close_many(h)):
            _store(state.out, w, rep)
    elif state.kind == "pipelined":
        sd.sd_update(h[0], pairs[0])
        sd.sd_update(h[1], pairs[1])
        for w in range(2):
            _store(state.out, w, sd.sd_close_window(h[w]))
    elif state.kind == "merge":
        for m, p in zip(h, pairs):
            sd.sd_update(m, p)
        for m in h[1:]:
            sd.sd_merge(h[0], m)
        _store(state.out, 0, sd.sd_close_window(h[0]))
        for m in h[1:]:  # the monitors' own windows end as well
            sd.sd_close_window(m)
    else:
        for p in pairs:
            sd.sd_update(h[0], p)
        _store(state.out, 0, sd.sd_close_window(h[0]))
    return state.out


def work(case):
    sk = SKETCHES[case["sketch"]]
    kind = case["kind"]
    n = sum(_sizes(case)) if kind in ("stream", "batch") else case["n"] * (2 if kind == "pipelined" else 1)
    byt = 8 * n  # the pairs, read once (a report is small beside them)
    if kind == "noalloc":  # the words of the caller's DHLA that the pairs touch, read and written
        cells = sk["r"] * sk["dirs"] * (1 << sk["k"]) * (sk["g"] // 32)
        byt += 8 * min(cells, n * sk["r"] * sk["dirs"])
    return {"bytes": byt, "flops": n * sk["r"] * sk["dirs"]}  # one bit-set per pair, row and direction


# ------------------------------------------------------------ exact outputs
def _splitmix(state):
    m = (1 << 64) - 1
    state = (state + 0x9E3779B97F4A7C15) & m
    z = state
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & m
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & m
    return state, z ^ (z >> 31)


def _signed(x):
    return x - (1 << 64) if x >> 63 else x


def _exact_window(sk, bufs, cand_cap):
    """psi and the estimates of one window from the definitions, with plain
    torch (whole numbers in int64, reals in float64); None where the window
    overloads (no hits)."""
    dev = bufs[0].device if bufs[0].is_cuda else "cuda"
    g, r, k, alpha, dirs = sk["g"], sk["r"], sk["k"], sk["alpha"], sk["dirs"]
    lg, cells, km = g.bit_length() - 1, 1 << k, (1 << k) - 1
    psis, ests = [], []
    zmin = g * math.exp(-THETA / g)
    for d in range(dirs):
        s = (HASH_SEED ^ (0x9E3779B97F4A7C15 * (d + 1))) & ((1 << 64) - 1)
        s, z0 = _splitmix(s)
        s, z1 = _splitmix(s)
        s, z2 = _splitmix(s)
        A0, A1, B1 = (z0 & M32) | 1, _signed(z1 | 1), _signed(z2)

        def rows(x):
            c0 = ((A0 * x) & M32) >> (32 - k)
            return [c0] + [((x >> min(63, (i - 1) * alpha)) & km) ^ c0 for i in range(1, r)]

        bits = torch.zeros(r * cells * g, dtype=torch.uint8, device=dev)
        one = torch.ones((), dtype=torch.uint8, device=dev)
        for buf in bufs:
            n = buf.numel() // 2
            for p0 in range(0, n, 1 << 24):
                w = buf[2 * p0:2 * min(n, p0 + (1 << 24))].to(dev).view(-1, 2).to(torch.int64) & M32
                key, peer = w[:, d], w[:, 1 - d]
                b = ((A1 * peer + B1) >> (64 - lg)) & (g - 1)
                for i, c in enumerate(rows(key)):
                    bits[(c + i * cells) * g + b] = one
        bits = bits.view(r, cells, g)
        z = g - bits.sum(dim=2, dtype=torch.int64)
        zr = z.sum(dim=1).tolist()
        if min(zr) == 0:
            psis.append(-1.0)
            continue
        hot = z < zmin
        G = float(g) * cells
        psi = 1.0 - math.exp(-(sum(-G * math.log(v / G) for v in zr) / r) / G)
        psis.append(psi)
        he0, he1 = torch.nonzero(hot[0]).view(-1), torch.nonzero(hot[1]).view(-1)
        if he0.numel() << (32 - k) > 1 << 32:
            continue
        # K: c0 and c1 give the low k bits, DH_0 the 32 - k high ones (all of
        # them tried for k < 16, solved for otherwise through A0^-1)
        inv = pow(A0, -1, 1 << 32)
        ul = max(0, 32 - 2 * k)
        found, total = [], 0
        t = torch.arange(1 << ul, device=dev)
        per = max(1, (1 << 25) // max(1, he1.numel() << ul))
        for q in range(0, he0.numel(), per):
            if he1.numel() == 0:
                break
            c0 = he0[q:q + per].view(-1, 1, 1)
            low = c0 ^ he1.view(1, -1, 1)
            prod = (A0 * low) & M32
            if k >= 16:
                u = c0 >> (2 * k - 32)
                ok = ((prod & km) >> (32 - k)) == (c0 & ((1 << (2 * k - 32)) - 1))
            else:
                u = (c0 << ul) | t.view(1, 1, -1)
                ok = None
            hm = (1 << (32 - k)) - 1
            a = ((inv * ((u - (prod >> k)) & hm)) & hm) << k | low
            a = (a[ok] if ok is not None else a.reshape(-1))
            c = rows(a)
            keep = hot[0][c[0]]
            for i in range(1, r):
                keep = keep & hot[i][c[i]]
            found.append(a[keep])
            total += found[-1].numel()
            if total > cand_cap:
                break
        if total > cand_cap or not found:
            continue
        cand = torch.sort(torch.cat(found)).values
        sz = []
        for q in range(0, cand.numel(), 1 << 17):
            x = cand[q:q + (1 << 17)]
            u = None
            for i, c in enumerate(rows(x)):
                v = bits[i][c]
                u = v if u is None else u & v
            sz.append(g - u.sum(dim=1, dtype=torch.int64))
        sz = torch.cat(sz).cpu().numpy().astype(np.float64)
        with np.errstate(divide="ignore"):
            est = -float(g) * np.log(sz / (g - g * psi ** r))
        ests.append(est[est >= THETA])
    return np.array(psis), np.concatenate(ests) if ests else np.zeros(0)


def exact(case, seed):
    if case["kind"] == "noalloc":
        return None  # bits only
    sk = SKETCHES[case["sketch"]]
    if case["kind"] == "batch":
        # every window on its own, its pairs drawn when it is its turn
        wins = ([_traffic(sk, n, 1000 * seed + i)] for i, n in enumerate(_sizes(case)))
        got = [_exact_window(sk, w, 1 << 18) for w in wins]
    else:
        got = [_exact_window(sk, w, 1 << 20) for w in _inputs(case, seed)]
    out = _buffers(len(got), sk, ROWS_BATCH if case["kind"] == "batch" else ROWS)
    for w, (psi, est) in enumerate(got):
        est = est[:out["est"].shape[1]]
        out["psi"][w], out["est"][w, :len(est)] = psi, est
    return {name: v if name in ("psi", "est") else None for name, v in out.items()}
