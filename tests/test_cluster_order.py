"""The shared memory of a cluster's other CTAs may be touched only after a cluster barrier has shown that
they run: in every kernel, the first barrier comes before the first remote access (read off the source,
with the device functions that a kernel calls in place)."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2204_01386_gb300", "csrc")
EVENT = re.compile(r"(?P<sync>\bcluster\.sync\s*\(|this_cluster\(\)\.sync\s*\()|(?P<remote>\bmap_shared_rank\s*\()"
                   r"|(?P<call>\b[A-Za-z_]\w*)\s*(?:<[^;{}()]*>)?\s*\(")


def _functions():
    """name -> (is a kernel, body) of the functions in the CUDA sources, without comments."""
    out = {}
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(path).read(), flags=re.S)
        for m in re.finditer(r"(__global__|__device__)[^;{}=]*?\b(\w+)\s*\([^;{}]*\)\s*\{", text):
            depth, i = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(text[i], 0)
                i += 1
            out[m.group(2)] = (m.group(1) == "__global__", text[m.end():i])
    return out


def _events(funcs, name, stack=()):
    """the cluster barriers and remote accesses of a function in the order of its text"""
    for m in EVENT.finditer(funcs[name][1]):
        if m.group("sync"):
            yield "sync"
        elif m.group("remote"):
            yield "remote"
        elif m.group("call") in funcs and m.group("call") not in stack + (name,):
            yield from _events(funcs, m.group("call"), stack + (name,))


def test_cluster_barrier_before_remote_shared_memory():
    funcs = _functions()
    seen = 0
    for name, (kernel, _) in funcs.items():
        if not kernel:
            continue
        ev = list(_events(funcs, name))
        if "remote" in ev:
            seen += 1
            assert "sync" in ev[:ev.index("remote")], f"{name} touches another CTA's shared memory before a cluster barrier"
    assert seen > 0   # the cluster kernel was found
