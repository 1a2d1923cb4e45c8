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
    N, cN, dt = 80, 5, 0.1 * 2.0 / 80

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


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "mixed"])
def test_memory_of_one_path(sulfmg, precision):
    """the tuner runs candidates of both paths; afterwards the domain holds what
    a domain given the same controls holds (chunks of 2 MB in three pools)"""
    N, dt = 64, 0.25 * 2.0 / 64
    d = _domain(sulfmg, 3, N, 8, precision=precision)
    d.step(dt, 1)
    r = d.autotune(dt, use_cache=False)
    d.step(dt, 1)
    got = d.stats()["device_bytes"]
    s, c, _ = d.get_state()
    d.close()
    keys = ("fuse_below", "ghost_compose", "pdl", "relax_occupancy", "relax_matrix_free")
    f = _domain(sulfmg, 3, N, 8, precision=precision, **{k: r[k] for k in keys})
    f.step(dt, 2)
    want = f.stats()["device_bytes"]
    s1, c1, _ = f.get_state()
    f.close()
    assert got <= want + 3 * (2 << 20)
    assert got <= sulfmg.estimate_device_bytes(3, N, 8, precision)
    tol = 1e-12 if precision == 0 else 1e-8
    assert np.abs(s - s1).max() <= tol * np.abs(s1).max() and np.abs(c - c1).max() <= tol * np.abs(c1).max()


@pytest.mark.parametrize("base", [dict(relax_matrix_free=2), dict(ghost_compose=0), dict(smoother=1)],
                         ids=["tiled", "pass by pass", "pointwise"])
def test_tuned_from_the_two_unknown_path(sulfmg, base):
    """a domain on the two-unknown kernels: the candidates of the other path take
    its vectors and give them back; the state of the next steps is as before"""
    N, dt = 80, 0.1 * 2.0 / 80
    out = []
    for tune in (False, True):
        d = _domain(sulfmg, 3, N, 5, precision=1, **base)
        d.step(dt, 1)
        if tune:
            d.autotune(dt, use_cache=False)
        d.step(dt, 1)
        out.append(d.get_state()[:2])
        d.close()
    for a, b in zip(*out):
        assert np.abs(a - b).max() <= 1e-8 * np.abs(a).max()
