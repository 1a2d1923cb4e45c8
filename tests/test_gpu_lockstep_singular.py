"""A lock-step instance whose coarsest Jacobian is singular (porosity zero:
alpha = beta = 0, so every inside row of s vanishes) fails with ENOTCONV and
keeps its state bit for bit, as it does when stepped alone; the class goes on."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu

ALONE_TOL = 1e-12  # as in the lock-step tests: the rounding order of a few reductions
MIXED_TOL = 1e-8


def _domain(sulfmg, model, **solver):
    d = sulfmg.Domain(workloads.disk(64), 2, (-1.0, 1.0), 64, 8)
    d.set_model(model)
    d.set_solver(**solver)
    return d


@pytest.mark.parametrize("compose", [1, 0], ids=["scalar", "alone"])
@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "mixed"])
def test_singular_instance_keeps_its_state(sulfmg, precision, compose):
    dt = 0.25 * 2.0 / 64
    good = list(workloads.PAPER_MODEL)
    bad = list(good)
    bad[4] = bad[5] = 0.0
    doms = [_domain(sulfmg, m, precision=precision, ghost_compose=compose) for m in (good, bad, good)]
    s0, c0, _ = doms[1].get_state()
    batch = sulfmg.Batch(doms, nstreams=1, lockstep=True)
    with pytest.raises(sulfmg.SulfError) as e:
        batch.step(dt, 2)
    assert e.value.code == sulfmg.ENOTCONV
    assert list(batch.status()) == [0, sulfmg.ENOTCONV, 0]
    batch.close()
    s, c, t = doms[1].get_state()
    np.testing.assert_array_equal(s, s0)
    np.testing.assert_array_equal(c, c0)
    assert doms[1].stats()["steps_total"] == 0
    alone = _domain(sulfmg, good, precision=precision, ghost_compose=compose)
    alone.step(dt, 2)
    s1, c1, _ = alone.get_state()
    alone.close()
    act = (t == 1) | (t == 2)
    tol = ALONE_TOL if precision == 0 else MIXED_TOL
    for d in (doms[0], doms[2]):
        s, c, _ = d.get_state()
        assert np.abs(s - s1)[act].max() <= tol * np.abs(s1[act]).max()
        assert np.abs(c - c1)[act].max() <= tol * np.abs(c1[act]).max()
    for d in doms:
        d.close()
