"""Several coarse steps of one call go through graphs of several steps: bit for bit the solve
that takes them one call at a time, for counts around the graphs' sizes and from either level-0
parity, on one level (eight steps a graph) and on an airfoil (two)."""
import numpy as np
import pytest

import paper_2601_18443_gb300 as pkg
from paper_2601_18443_gb300 import workloads as W

pytestmark = pytest.mark.gpu

CASES = {
    "tunnel": lambda: (W.base_config(levels=1, nx0=70, ny0=33, Re=5.0, turbulence=1, solid_walls=0), []),
    "naca0012-4lvl": lambda: W.naca0012_small(levels=4),
}


@pytest.mark.parametrize("name", list(CASES))
def test_steps_in_one_call_equal_single_steps(name):
    pkg.build()
    cfg, loops = CASES[name]()
    a, b = pkg.Solver(cfg), pkg.Solver(cfg)
    for s in (a, b):
        s.set_geometry(loops)
        i0, j0, nx, ny = s.level_box(0)
        s.set_fields(0, ux=0.0577 * (1 + 0.01 * np.random.default_rng(3).standard_normal((ny, nx))))
    for n in (1, 7, 8, 9, 16, 17, 3):
        a.step(n)
        for _ in range(n):
            b.step(1)
        for l in range(cfg["levels"]):
            assert np.array_equal(a.get_populations(l), b.get_populations(l), equal_nan=True), (n, l)
    assert a.coefficients()["step"] == b.coefficients()["step"] == 61
    a.close()
    b.close()
