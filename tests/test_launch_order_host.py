"""Kernels that may begin before the one ahead of them has ended read nothing through the read-only path: a
load marked so may be moved above the wait, and the path asks that the data not change while the kernel lives."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2502_01941_b200", "csrc")


def _kernels():
    """(name, parameters, body) of every __global__ function."""
    for f in sorted(os.listdir(CSRC)):
        if f.endswith((".cuh", ".cu")):
            text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read())
            for m in re.finditer(r"__global__[^;{]*?(\w+_kernel)\(", text):
                close, depth = m.end(), 1
                while depth:
                    depth += {"(": 1, ")": -1}.get(text[close], 0)
                    close += 1
                start = end = text.index("{", close) + 1
                depth = 1
                while depth:
                    depth += {"{": 1, "}": -1}.get(text[end], 0)
                    end += 1
                yield m.group(1), text[m.end():close - 1], text[start:end]


def test_nothing_is_read_through_the_read_only_path():
    early = [k for k in _kernels() if "grid_wait()" in k[2]]
    assert len(early) >= 10
    for name, params, body in early:
        assert not re.search(r"const\s+\w+\s*\*\s*__restrict__", params), f"{name}: read-only pointer among the parameters"
        assert "__ldg" not in body, f"{name}: read-only load"


def test_the_ring_of_the_attention_step_is_declared_on_a_line():
    """A warp's 512-byte copies reach one line of shared memory more where the ring does not begin on one."""
    body = {name: body for name, _, body in _kernels()}["decode_attend_kernel"]
    assert re.search(r"extern\s+__shared__\s+__align__\(128\)", body)
    assert re.search(r"ring\s*=\s*dsm;", body), "the ring comes first"
