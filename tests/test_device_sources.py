"""Rules of the CUDA sources that no run can show (breaking them is a race that
a run may win), read from the sources."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1902_07029_gb300", "csrc")


def _code(name):
    src = open(os.path.join(CSRC, name)).read()
    src = re.sub(r"/\*.*?\*/", "", src, flags=re.S)
    return re.sub(r"//[^\n]*", "", src)


def _block(src, at):
    """the braces' block that opens at or after position at"""
    i = src.index("{", at)
    depth = 0
    for j in range(i, len(src)):
        depth += (src[j] == "{") - (src[j] == "}")
        if depth == 0:
            return src[i:j + 1]
    raise AssertionError("unbalanced braces")


def _kernels():
    """(file, name, body) of every kernel"""
    out = []
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith((".cu", ".cuh")):
            continue
        src = _code(f)
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\([^)]*\)\s*)?(\w+)\s*\(", src):
            out.append((f, m.group(1), _block(src, m.end())))
    return out


KERNELS = _kernels()


def test_the_reader_finds_the_kernels():
    names = {n for _, n, _ in KERNELS}
    assert {"k_s_factor", "k_coarsest_factor_cluster", "k_s_coarse", "kb_s_phase", "kb_relax", "k_newton_F"} <= names


@pytest.mark.parametrize("name", ["k_s_factor", "k_coarsest_factor_cluster"])
def test_cluster_meets_before_remote_shared_memory(name):
    """another CTA's shared memory may be accessed only once all CTAs of the
    cluster are known to run and while none has left: a cluster barrier before
    the first access and one after the last"""
    body = next(b for _, n, b in KERNELS if n == name)
    first = body.index("map_shared_rank(")
    assert 0 <= body.find("cl.sync()") < first
    assert body.rindex("cl.sync()") > body.rindex("map_shared_rank(")
