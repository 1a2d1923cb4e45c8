"""What the autotuner measures and leaves behind."""
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
