"""The prolongation launch (Sec 2.2) on its own: after it, the ghost cells of level l + 1 hold the
linear LSQ reconstruction of chi and u about their parent and the parent's rho, restated here in
numpy from the fields of level l.  FP32 rounding of a gradient (six differences of values v) is
within 1e-6 of the values' magnitude."""
import numpy as np
import pytest

import paper_2601_18443_gb300 as pkg
from paper_2601_18443_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("case", ["small", "patch"])
def test_ghosts_hold_the_reconstruction_about_their_parents(case):
    pkg.build()
    if case == "small":
        cfg, loops = W.naca0012_small(levels=4)
    else:       # an L-shaped patch: convex and concave corners, tiles touched by one band cell
        cfg = W.base_config(levels=3, nx0=64, ny0=64, layers=3, periodic=1, solid_walls=0, Re=5.0, turbulence=1)
        loops = [W.l_shape(20, 20, 37, 37, 28, 28)]
    g = pkg.Solver(cfg)
    g.set_geometry(loops)
    rng = np.random.default_rng(9)
    i0, j0, nx, ny = g.level_box(0)
    g.set_fields(0, ux=0.05 + 0.01 * rng.standard_normal((ny, nx)), uy=0.01 * rng.standard_normal((ny, nx)),
                 chi=3.0 + rng.random((ny, nx)))
    g.step(2)
    for l in range(cfg["levels"] - 1):
        P = g.get_fields(l)
        g.step_launch(l, 2)
        F = g.get_fields(l + 1)
        jj, ii = np.nonzero(F["mask"] == 4)
        gi, gj = ii + F["i0"], jj + F["j0"]
        pi, pj = (gi >> 1) - P["i0"], (gj >> 1) - P["j0"]
        near = np.pad((P["mask"] >= 1) & (P["mask"] <= 4), 1)
        ok = np.all([near[pj + 1 + b, pi + 1 + a] for b in (-1, 0, 1) for a in (-1, 0, 1)], axis=0)
        assert ok.sum() > 100
        jj, ii, gi, gj, pi, pj = (v[ok] for v in (jj, ii, gi, gj, pi, pj))
        assert np.array_equal(F["rho"][jj, ii], P["rho"][pj, pi])
        for f in ("ux", "uy", "chi"):
            v = np.pad(P[f], 1)
            at = lambda a, b: v[pj + 1 + b, pi + 1 + a]
            gx = sum(at(1, b) - at(-1, b) for b in (-1, 0, 1)) / 6
            gy = sum(at(a, 1) - at(a, -1) for a in (-1, 0, 1)) / 6
            want = at(0, 0) + 0.5 * ((gi & 1) - 0.5) * gx + 0.5 * ((gj & 1) - 0.5) * gy
            assert np.abs(F[f][jj, ii] - want).max() <= 1e-6 * np.abs(v[np.isfinite(v)]).max(), (l, f)
    g.close()
