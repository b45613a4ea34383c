"""Kernels that may start while the kernel before them still writes (programmatic dependent launch) read the vectors
that it writes by plain loads after their wait: the read-only path (__ldg, const __restrict__ arguments) is for data
that do not change during the kernel, here the links.  Read from the sources; needs no GPU."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1805_09584_gb300", "csrc")


def _source(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)


def _files():
    """Sources with dependent launches, and the repository's headers that they include."""
    todo = [f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh")) and '#include "launch.cuh"' in open(os.path.join(CSRC, f)).read()]
    out = []
    while todo:
        f = todo.pop()
        if f not in out and f != "launch.cuh":
            out.append(f)
            todo += [h for h in re.findall(r'#include "(\w+\.cuh)"', _source(f))]
    return out


def _kernels(text):
    """(name, parameters, body) of each kernel."""
    starts = [m.start() for m in re.finditer(r"__global__", text)] + [len(text)]
    for a, b in zip(starts, starts[1:]):
        k = text[a:b]
        m = re.search(r"(k_\w+)\s*\(([^{;]*)\)\s*\{(.*)", k, flags=re.S)
        if m:
            yield m.groups()


def test_dependent_kernels_wait_first_and_read_vectors_by_plain_loads():
    files = _files()
    assert {"hop_fx.cu", "dslash_f32.cu", "s16_kernels.cuh"} <= set(files)
    launched, waiting = set(), set()
    for f in files:
        text = _source(f)
        launched |= set(re.findall(r"launch_dependent(?:_if)?\((?:ntile <= nb, )?(k_\w+)", text))
        for arg in re.findall(r"__ldg\(&?(\w+)", text):
            assert arg == "U", (f, arg)  # a link
        for name, params, body in _kernels(text):
            if "dependent_begin();" not in body:
                continue
            waiting.add(name)
            for p in re.findall(r"const \w+ \*__restrict__ (\w+)", params):
                assert p == "links", (f, name, p)
            # nothing but declarations before the wait
            before = body[:body.index("dependent_begin();")]
            assert not re.search(r"[\[*]\w+\]?\s*=|->|\breturn\b", re.sub(r"__shared__[^;]*;|constexpr[^;]*;", "", before)), name
    assert launched and launched <= waiting
