"""Tensor-memory instructions are .sync.aligned: all lanes of a warp execute them together or the
result is undefined.  A run does not show a missing reconvergence (the compiler may have predicated
the branch before it), so the rule is read from the source: every function that issues such an
instruction brings its warp, or its block, together first."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1301_0322_gb300", "csrc")


def functions(text):
    """(name, body) of the __device__ functions, by their braces; comments removed."""
    text = re.sub(r"//[^\n]*", "", text)
    for m in re.finditer(r"__device__ __forceinline__ [^;{(]*?(\w+)\([^;{]*\{", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        yield m.group(1), text[m.end():i]


def test_tensor_memory_instructions_follow_a_barrier_of_their_warp():
    issuing = []
    for name in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, name)).read()
        if "tcgen05" not in text:
            continue
        for fn, body in functions(text):
            first = re.search(r"tcgen05\.(alloc|dealloc|st|ld|relinquish)[\w.:]*\.sync\.aligned", body)
            if first:
                issuing.append(fn)
                assert re.search(r"__sync(warp|threads)\(\);", body[:first.start()]), (name, fn)
    assert {"TmemPark", "store", "load", "load16", "close"} <= set(issuing)
