"""Lock-step classes whose instances fuse from different levels: the class fuses
from the first level that each of them can, steps as each alone, and builds its
cluster tables once."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu

N = 128
# level 1 holds 2209 nodes of the disk and 1392 of the star
FUSE = 1800
ALONE_TOL, MIXED_TOL = 1e-12, 1e-8  # as in the lock-step tests


def _domains(sulfmg, **solver):
    out = []
    for phi in (workloads.star(N), workloads.disk(N), workloads.star(N, amp=0.1)):
        d = sulfmg.Domain(phi, 2, (-1.0, 1.0), N, 8)
        d.set_model(workloads.PAPER_MODEL)
        d.set_solver(**solver)
        out.append(d)
    return out


def _tables(doms):
    return [d.route()["tables"] for d in doms]


@pytest.mark.parametrize("fuse", [FUSE, 0, -1])
@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "mixed"])
def test_tables_are_built_once(sulfmg, precision, fuse):
    dt = 0.25 * 2.0 / N
    doms = _domains(sulfmg, precision=precision, fuse_below=fuse)
    nodes = [[doms[i].level_info(1)[k] for k in ("nin", "ng")] for i in (0, 1)]
    assert sum(nodes[0]) <= FUSE < sum(nodes[1])
    batch = sulfmg.Batch(doms, nstreams=1, lockstep=True)
    batch.step(dt, 1)
    first = _tables(doms)
    assert all((t > 0) == (fuse != 0) for t in first)
    batch.step(dt, 1)
    assert _tables(doms) == first
    # stepped alone (the finest level may join there) and in the class in turn
    for d in doms:
        d.step(dt, 1)
    both = _tables(doms)
    batch.step(dt, 1)
    for d in doms:
        d.step(dt, 1)
    assert _tables(doms) == both
    batch.close()
    ref = _domains(sulfmg, precision=precision, fuse_below=fuse)
    tol = ALONE_TOL if precision == 0 else MIXED_TOL
    for d, r in zip(doms, ref):
        r.step(dt, 5)
        s, c, t = d.get_state()
        s1, c1, _ = r.get_state()
        act = (t == 1) | (t == 2)
        assert np.abs(s - s1)[act].max() <= tol * np.abs(s1[act]).max()
        assert np.abs(c - c1)[act].max() <= tol * np.abs(c1[act]).max()
        d.close()
        r.close()


def test_tables_follow_the_controls(sulfmg):
    """another threshold, sweep count or boundary condition: built anew, once"""
    dt = 0.25 * 2.0 / N
    doms = _domains(sulfmg, fuse_below=FUSE)
    batch = sulfmg.Batch(doms, nstreams=1, lockstep=True)
    batch.step(dt, 1)
    for change in (dict(fuse_below=200), dict(fuse_below=200, nu1=1), dict(fuse_below=FUSE)):
        for d in doms:
            d.set_solver(**change)
        before = _tables(doms)
        batch.step(dt, 1)
        after = _tables(doms)
        assert all(a > b for a, b in zip(after, before))
        batch.step(dt, 1)
        assert _tables(doms) == after
    ref = _domains(sulfmg, fuse_below=FUSE)
    for d in doms:
        d.set_bc(1)
        d.set_model(workloads.PAPER_MODEL)
    batch.step(0.25 * dt, 1)
    after = _tables(doms)
    batch.step(0.25 * dt, 1)
    assert _tables(doms) == after
    batch.close()
    for d, r in zip(doms, ref):
        r.set_bc(1)
        r.step(0.25 * dt, 2)
        (s, c, _), (s1, c1, _) = d.get_state(), r.get_state()
        assert np.abs(s - s1).max() <= ALONE_TOL * np.abs(s1).max()
        assert np.abs(c - c1).max() <= ALONE_TOL * np.abs(c1).max()
        d.close()
        r.close()
