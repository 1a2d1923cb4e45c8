"""A step that finds no device memory fails with ENOMEM and leaves the handle
usable: the next step gives, bit for bit, what it gives on a handle that never
failed, by the same number of kernel launches.  Each allocation of a first step
is refused in turn (on the host: the request is answered as if the device were
full)."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu

GEOMS = {
    "disk32": lambda: (workloads.disk(32), 2, 32, 8),
    "rbox16": lambda: (workloads.rounded_box(16), 3, 16, 4),
}


def _domain(sulfmg, name, **solver):
    phi, dim, N, cN = GEOMS[name]()
    d = sulfmg.Domain(phi, dim, (-1.0, 1.0), N, cN)
    d.set_model(workloads.PAPER_MODEL)
    d.set_solver(**solver)
    return d, 0.05 * 2.0 / N


def _two_steps(d, dt):
    """the state after two steps and the second one's launches (the first one's
    include set-up)"""
    d.step(dt, 1)
    n = d.stats()["kernel_launches"]
    d.step(dt, 1)
    return d.get_state()[:2], d.stats()["kernel_launches"] - n, d.stats()["loop_graph"]


def _sweep(sulfmg, name, **solver):
    d, dt = _domain(sulfmg, name, **solver)
    (s0, c0), launches, loop = _two_steps(d, dt)
    d.close()
    failed = 0
    for k in range(2000):
        d, dt = _domain(sulfmg, name, **solver)
        d.fail_alloc(k)
        init = d.get_state()[:2]
        try:
            d.step(dt, 1)
        except sulfmg.SulfError as e:
            assert e.code == sulfmg.ENOMEM
            failed += 1
            for a, b in zip(init, d.get_state()[:2]):
                np.testing.assert_array_equal(a, b)
            assert not d.fail_alloc(None)
        else:
            if d.fail_alloc(None):  # never reached: every allocation has been refused once
                d.close()
                return failed, k
            # (a refused buffer of the device-side cycle loop only: this step ran without it)
            d.set_model(workloads.PAPER_MODEL)
        (s, c), n, lp = _two_steps(d, dt)
        np.testing.assert_array_equal(s, s0)
        np.testing.assert_array_equal(c, c0)
        assert (n, lp) == (launches, loop), f"allocation {k}"
        d.close()
    raise AssertionError("a first step of 2000 allocations")


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "mixed"])
@pytest.mark.parametrize("name", list(GEOMS))
def test_two_unknown_path(sulfmg, name, precision):
    """the vectors of the two-unknown kernels, the fused levels' descriptors and
    the buffers of the device-side cycle loop"""
    failed, total = _sweep(sulfmg, name, precision=precision, ghost_compose=0)
    assert 0 < failed < total


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "mixed"])
@pytest.mark.parametrize("name", list(GEOMS))
def test_cycle_on_the_equation_for_s(sulfmg, name, precision):
    """its lists, rows, vectors and cluster tables: a level whose rows were not
    built is not taken for built by the next step"""
    failed, total = _sweep(sulfmg, name, precision=precision)
    assert 0 < failed < total


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "mixed"])
def test_rebuild_for_another_boundary_condition(sulfmg, precision):
    """the rows of a handle that has stepped, rebuilt for the Neumann condition:
    a refused allocation leaves none of the Dirichlet rows in use"""

    def start():
        d, dt = _domain(sulfmg, "disk32", precision=precision)
        d.step(dt, 1)
        d.set_bc(1)
        d.set_model(workloads.PAPER_MODEL)
        return d, dt

    d, dt = start()
    (s0, c0), launches, _ = _two_steps(d, dt)
    d.close()
    for k in range(100):
        d, dt = start()
        d.fail_alloc(k)
        try:
            d.step(dt, 1)
            done = d.fail_alloc(None)
            d.set_model(workloads.PAPER_MODEL)
        except sulfmg.SulfError as e:
            assert e.code == sulfmg.ENOMEM
            done = False
        (s, c), n, _ = _two_steps(d, dt)
        np.testing.assert_array_equal(s, s0)
        np.testing.assert_array_equal(c, c0)
        assert n == launches
        d.close()
        if done:
            return
    raise AssertionError("a rebuild of 100 allocations")


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "mixed"])
def test_lock_step_set_up(sulfmg, precision):
    """the same for a lock-step class: the cluster tables of the instance that
    found no memory are built by the next call"""

    def start():
        doms = [_domain(sulfmg, "disk32", precision=precision)[0] for _ in range(2)]
        return doms, sulfmg.Batch(doms, nstreams=1, lockstep=True), 0.05 * 2.0 / 32

    def run(doms, batch, dt):
        batch.step(dt, 1)
        n = [d.stats()["kernel_launches"] for d in doms]
        batch.step(dt, 1)
        return [d.get_state()[:2] for d in doms], [d.stats()["kernel_launches"] - m for d, m in zip(doms, n)]

    def close(doms, batch):
        batch.close()
        for d in doms:
            d.close()

    doms, batch, dt = start()
    ref, launches = run(doms, batch, dt)
    close(doms, batch)
    for k in range(500):
        doms, batch, dt = start()
        doms[1].fail_alloc(k)
        try:
            batch.step(dt, 1)
            done = doms[1].fail_alloc(None)
            for d in doms:
                d.set_model(workloads.PAPER_MODEL)
        except sulfmg.SulfError as e:
            assert e.code == sulfmg.ENOMEM
            done = False
        out, n = run(doms, batch, dt)
        close(doms, batch)
        for (s, c), (s0, c0) in zip(out, ref):
            np.testing.assert_array_equal(s, s0)
            np.testing.assert_array_equal(c, c0)
        assert n == launches, f"allocation {k}"
        if done:
            return
    raise AssertionError("a lock-step set-up of 500 allocations")
