"""What the autotuner measures and leaves behind."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


def _domain(sulfmg, dim, N, cN, **solver):
    phi = workloads.star(N) if dim == 2 else workloads.rounded_box(N)
    d = sulfmg.Domain(phi, dim, (-1.0, 1.0), N, cN)
    d.set_model(workloads.PAPER_MODEL)
    d.set_solver(**solver)
    return d


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "mixed"])
def test_no_graph_is_captured_in_a_timed_solve(sulfmg, precision):
    """every candidate is timed on the graphs a step replays, whatever its path:
    a capture inside the timed solve would be charged to some candidates only"""
    d = _domain(sulfmg, 2, 128, 8, precision=precision)
    d.autotune(0.5 * 2.0 / 128, use_cache=False)
    r = d.route()
    assert r["captures"] > 0 and r["captures_timed"] == 0
    d.close()


def test_cached_tiled_sweep_is_used(sulfmg):
    """a fresh domain that takes relax_matrix_free = 2 from the cache runs the
    tiled sweep, as one that is given the control does"""
    N, cN, dt = 72, 9, 0.1 * 2.0 / 72

    def two_steps(d):
        d.step(dt, 1)
        n = d.stats()["kernel_launches"]
        d.step(dt, 1)
        return d.get_state()[:2], d.stats()["kernel_launches"] - n

    a = _domain(sulfmg, 3, N, cN, precision=1, relax_matrix_free=2)
    assert a.level_info(0)["nin"] > 100000  # tiled
    (s0, c0), n0 = two_steps(a)
    a.close()
    b = _domain(sulfmg, 3, N, cN, precision=1)
    b.tune_put(fuse_below=-1, ghost_compose=1, pdl=1, relax_matrix_free=2, candidates=1)
    r = b.autotune(dt)
    assert r["cached"] == 1 and r["relax_matrix_free"] == 2
    (s, c), n = two_steps(b)
    assert n == n0
    np.testing.assert_array_equal(s, s0)
    np.testing.assert_array_equal(c, c0)
    b.close()
