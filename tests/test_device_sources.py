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


def _functions():
    """(file, name, body) of the kernels and of the device functions that pass
    the dependent-launch wait themselves"""
    out = [k for k in KERNELS if any(w in k[2] for w in ("pdl_enter(", "masked(", "s_phase<", "s_outer<"))]
    for f in ("schur.cu",):
        src = _code(f)
        for m in re.finditer(r"__device__\s+__forceinline__\s+void\s+(s_\w+)\s*\(", src):
            body = _block(src, m.end())
            if "pdl_enter(" in body:
                out.append((f, m.group(1), body))
    return out


@pytest.mark.parametrize("f,name,body", _functions(), ids=[n for _, n, _ in _functions()])
def test_no_thread_leaves_before_the_dependent_launch_wait(f, name, body):
    """a grid completes when its CTAs have left; if they can leave without the
    wait it may complete before the grid it depends on, and the grid after it
    then runs beside that one"""
    waits = [body.index(w) for w in ("pdl_enter(", "masked(", "s_phase<", "s_outer<") if w in body]
    head = re.sub(r"if \([^;]*masked\(active, [\w.]+\)\) return;", "", body[:body.find(";", min(waits)) + 1])
    tail = body[len(body[:body.find(";", min(waits)) + 1]):]
    assert "return" not in head
    # a masked instance's CTAs leave in masked(); the others go on to a wait
    if "masked(" in body:
        assert any(w in tail for w in ("pdl_enter(", "s_phase<", "s_outer<"))
        if "pdl_enter(" in tail:
            assert "return" not in tail[:tail.index("pdl_enter(")]


def _allocations():
    """(file, line, pointer, what follows up to the next kernel launch)"""
    out = []
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith(".cu"):
            continue
        lines = _code(f).split("\n")
        for i, l in enumerate(lines):
            m = re.search(r"([\w.>\[\]-]+) = \([^=]*\)\s*[\w>.-]*get(?:_host)?\(", l)
            if not m:
                continue
            rest = []
            for r in lines[i:]:
                if "<<<" in r or "launch_" in r:
                    break
                rest.append(r)
            name = re.sub(r"\[\w+\]", "", m.group(1)).split(".")[-1].split(">")[-1]
            out.append((f, i + 1, name, "\n".join(rest)))
    return out


def test_allocations_are_checked_before_a_kernel_sees_them():
    found = _allocations()
    assert len(found) > 60
    bad = [(f, i, n) for f, i, n, rest in found
           if not re.search(rf"![\w.>-]*\b{n}\b|\b{n} (!=|==|&&)", rest)]
    assert not bad, bad
