"""Which route the cases of test_gpu_scalar_cycle take, from the rules of their
dispatch: a domain that fell back to another route passes those tests all the
same.  The 49^3 box does: the composed ghost map of its coarsest level is over
its bound, so the whole domain runs the two-unknown cycle.  A ragged 3-D box
that has the map on every level is added here."""
import pytest

import test_gpu_scalar_cycle as cycle
import workloads
from test_gpu_scalar_cycle import CASES, GEOMS

pytestmark = pytest.mark.gpu

GEOMS = dict(GEOMS, rbox40=lambda: (workloads.rounded_box(40), 3, 40, 5))
MORE = [("rbox40", {}, 0), ("rbox40", dict(nu1=1, nu2=1), 0), ("rbox40", dict(fuse_below=0), 0)]

CTA_ROWS = 512  # rows of one colour that a CTA sweeps


def _route(sulfmg, name, controls, bc, precision):
    phi, dim, N, cN = GEOMS[name]()
    d = sulfmg.Domain(phi, dim, (-1.0, 1.0), N, cN)
    d.set_model(workloads.PAPER_MODEL)
    d.set_bc(bc)
    d.set_solver(precision=precision, **controls)
    try:
        d.step(0.05 * 2.0 / N, 1)
    except sulfmg.SulfError as e:  # (the route is that of the linear solves either way)
        assert e.code == sulfmg.ENOTCONV
    info = [d.level_info(l) for l in range(d.stats()["levels"])]
    r = d.route()
    d.close()
    return r, info, dim


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "mixed"])
@pytest.mark.parametrize("name,controls,bc", CASES + MORE)
def test_route(sulfmg, name, controls, bc, precision):
    r, info, dim = _route(sulfmg, name, controls, bc, precision)
    assert r["scalar"] == all(i["ghost_map_entries"] >= 0 for i in info)
    assert r["scalar"] == (name != "rbox48")
    if not r["scalar"]:
        assert r["first_fused"] == -1
        return
    below = controls.get("fuse_below", -1)
    if below < 0:
        below = 40000 if dim == 2 and precision == 1 else 10000
    if below == 0 or controls.get("cycle", 1) != 1:
        assert (r["first_fused"], r["ctas"]) == (-1, 0)
        return
    nodes = [i["nin"] + i["ng"] for i in info]
    want = next(l for l, n in enumerate(nodes) if n <= below)
    first = r["first_fused"]
    assert want <= first < len(info) and r["ctas"] in (8, 16)
    if first > want:
        # a level that was passed over does not fit: its rows the threads of the
        # largest cluster (the finest), or its tables the shared memory
        assert nodes[first - 1] > 2000
    if first == 0:
        assert info[0]["nin"] // 2 <= CTA_ROWS * r["ctas"]
    narrow = 300 if dim == 3 else (1200 if precision == 1 else 600)
    if first < len(info) - 1:
        assert r["first_wide"] == (nodes[first] > narrow)


def test_the_cases_cover_the_routes(sulfmg):
    """the finest level in the cluster kernel on one CTA, on 8 and on 16; a
    coarser first level; no level there"""
    seen = set()
    for name, controls, bc in CASES:
        for precision in (0, 1):
            r, _, _ = _route(sulfmg, name, controls, bc, precision)
            f = r["first_fused"]
            seen.add("none" if f < 0 else "coarser" if f else ("one" if not r["first_wide"] else r["ctas"]))
    assert seen == {"none", "coarser", "one", 8, 16}


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "mixed"])
@pytest.mark.parametrize("name,controls,bc", MORE)
def test_more_cycles_match_the_oracle(sulfmg, oracle_mod, monkeypatch, name, controls, bc, precision):
    """the same comparison and bounds for the box added here"""
    monkeypatch.setitem(cycle.GEOMS, name, GEOMS[name])
    cycle.test_cycles_match_the_oracle(sulfmg, oracle_mod, name, controls, bc, precision)
