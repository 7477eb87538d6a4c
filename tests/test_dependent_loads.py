"""Kernels set up while the kernel before them still runs (they call
wait_for_previous) read what that kernel writes: neither they nor the device
functions they call may use non-coherent loads."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1803_11449_gb300", "csrc")


def _functions(text):
    """name -> (signature, body) of every __global__ and __device__ function"""
    out = {}
    for m in re.finditer(r"(?:__global__|__device__)[^;{}]*?(\w+)\s*\(", text):
        end = _close(text, m.end() - 1)
        if text[end:].lstrip()[:1] != "{":
            continue
        at = text.index("{", end)
        depth, q = 1, at + 1
        while depth:
            depth += {"{": 1, "}": -1}.get(text[q], 0)
            q += 1
        out[m.group(1)] = (text[m.end() - 1:end], text[at:q])
    return out


def _close(text, at):
    """index after the parenthesis that closes the one at `at`"""
    depth, q = 1, at + 1
    while depth:
        depth += {"(": 1, ")": -1}.get(text[q], 0)
        q += 1
    return q


def test_dependents_read_with_coherent_loads():
    read = {f: re.sub(r"//[^\n]*|__launch_bounds__\([^()]*\)", "", open(os.path.join(CSRC, f)).read())
            for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh"))}
    shared = _functions(read["sd_common.cuh"])
    dependents = 0
    for f, text in read.items():
        fns = {**shared, **_functions(text)}
        for name, (sig, body) in fns.items():
            if "wait_for_previous()" not in body or name not in text:
                continue
            dependents += 1
            assert not re.search(r"const\s[^,]*__restrict__", sig), f"{name}: const __restrict__"
            seen, todo = set(), [name]
            while todo:
                fn = todo.pop()
                if fn in seen:
                    continue
                seen.add(fn)
                b = fns[fn][1]
                assert "__ldg(" not in b and "global.nc" not in b, f"{name} reads through {fn}"
                todo += [w for w in set(re.findall(r"\w+", b)) if w in fns]
    assert dependents >= 3  # apply, restore, the close's last kernel
