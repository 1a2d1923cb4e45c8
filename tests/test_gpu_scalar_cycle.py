"""The cycle on the equation for s (schur.cu, coarse.cu) against the oracle's
cycle on both unknowns, at the edges of its routes: the finest level in the
cluster kernel on one CTA, on 8 and on 16, the first level there, no level
there; rows swept in registers or not; ragged grids; one and three sweeps;
W-cycles; Neumann rows; both precisions.

Bounds, from the arithmetic: an FP64 cycle is some 1e3 rounding steps deep on
operators of condition up to 1e3 per level, 1e3 * 1e3 * 2^-53 = 1e-10 relative.
An FP32 cycle solves for the error with a relative error of 1e3 * 2^-24 = 6e-5
at most, and the sum of the corrections is dominated by the first (bound 1e-4).
The cycles' defect norms are compared elsewhere: b - J x cancels, so its rounding
is a share of b and not of the norm."""
import numpy as np
import pytest

import workloads
from test_gpu_parity import _close, _pair, _rand_state, _rand_vec

pytestmark = pytest.mark.gpu

GEOMS = {
    "disk16": lambda: (workloads.disk(16), 2, 16, 8),
    "disk64": lambda: (workloads.disk(64), 2, 64, 8),
    "offdisk80": lambda: (workloads.disk(80, 0.55, (0.13, -0.07)), 2, 80, 10),
    "disk144": lambda: (workloads.disk(144), 2, 144, 9),
    "star256": lambda: (workloads.star(256), 2, 256, 8),
    "rbox32": lambda: (workloads.rounded_box(32), 3, 32, 8),
    "rbox48": lambda: (workloads.rounded_box(48), 3, 48, 6),
}
CASES = [(g, {}, 0) for g in GEOMS]
CASES += [(g, dict(fuse_below=0), 0) for g in ("disk64", "rbox32")]
CASES += [(g, dict(fuse_below=600), 0) for g in ("disk64", "star256")]
CASES += [(g, dict(nu1=1, nu2=1), 0) for g in ("disk64", "star256", "rbox48")]
CASES += [(g, dict(nu1=3, nu2=1), 0) for g in ("disk64", "disk144")]
CASES += [(g, dict(cycle=2), 0) for g in ("disk64", "rbox32")]
CASES += [(g, {}, 1) for g in ("disk64", "star256")]


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "mixed"])
@pytest.mark.parametrize("name,controls,bc", CASES,
                         ids=["-".join([g] + [f"{k}{v}" for k, v in c.items()] + ["neumann"] * b) for g, c, b in CASES])
def test_cycles_match_the_oracle(sulfmg, oracle_mod, name, controls, bc, precision):
    phi, dim, N, cN = GEOMS[name]()
    dom, ref = _pair(sulfmg, oracle_mod, phi, dim, N, cN)
    dom.set_bc(bc)
    ref.set_bc(bc)
    dom.set_solver(precision=precision, **controls)
    ref.set_solver(**{k: v for k, v in controls.items() if k != "fuse_below"})
    rng = np.random.default_rng(17)
    t0 = ref.level_type(0)
    W, rhs = _rand_state(rng, t0), _rand_vec(rng, t0)
    xg, rg = dom.cycles(2.0 / N, W, rhs, 4)
    xo, _ = ref.cycles(2.0 / N, W, rhs, np.zeros_like(rhs), 4)
    _close(xg, xo, 1e-4 if precision else 1e-10)
    # again on the same handle: the tables and graphs of the first call
    xh, rh = dom.cycles(2.0 / N, W, rhs, 4)
    np.testing.assert_array_equal(xh, xg)
    np.testing.assert_array_equal(rh, rg)
