"""Distributed shared memory: a block's shared memory may be accessed by the other blocks of its cluster
only once every block of the cluster is known to have started, so each function that makes such an
access passes a cluster barrier first.  Read from the kernel sources (nothing runs)."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_12894_gb300", "csrc")

# accesses to a peer's shared memory (the bulk copies and commits of reconstruct_gemm.cu name their own
# block's shared::cluster address) and what waits for the whole cluster
REMOTE = re.compile(r"\b(?:ld|st|red|atom)\.(?:async\.)?shared::cluster")
WAIT = re.compile(r"barrier\.cluster\.wait")


def _functions(text):
    """(name, body) of every device function or kernel at namespace level."""
    text = re.sub(r"//[^\n]*", "", text)
    head = re.compile(r"(?:__global__|__device__)[^;{}=]*?\b(\w+)\s*\((?:[^(){};]|\([^(){};]*\))*\)\s*\{")
    at = 0
    while m := head.search(text, at):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        yield m.group(1), text[m.end():i]
        at = i


def _first(body, direct, helpers):
    at = [m.start() for m in direct.finditer(body)]
    at += [m.start() for h in helpers for m in re.finditer(rf"\b{h}\s*(?:<[^;{{}}()]*>)?\s*\(", body)]
    return min(at, default=None)


def test_no_remote_access_before_the_cluster_has_started():
    funcs = {}
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        for name, body in _functions(open(path).read()):
            funcs[(os.path.basename(path), name)] = body
    # helpers: short functions that are nothing but one access, or a wait
    remote = [n for (_, n), b in funcs.items() if REMOTE.search(b) and b.count(";") <= 6 and not WAIT.search(b)]
    wait = [n for (_, n), b in funcs.items() if WAIT.search(b) and not REMOTE.search(b) and b.count(";") <= 3]
    wait += [n for (_, n), b in funcs.items()
             if b.count(";") <= 3 and any(re.search(rf"\b{w}\(", b) for w in wait)]
    assert remote and wait
    seen = 0
    for (path, name), body in funcs.items():
        if name in remote:
            continue
        r = _first(body, REMOTE, remote)
        if r is None:
            continue
        seen += 1
        w = _first(body, WAIT, wait)
        assert w is not None and w < r, f"{path}: {name} reaches a peer's shared memory before a cluster barrier"
    assert seen >= 3   # the pair tail, the clusters of window peaks and of matched filters
