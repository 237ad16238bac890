"""The two forms of the level kernel over plain cells: one cell a lane (levels that fit the GPU in
one wave of warps) and pairs of blocks, two cells a lane (larger ones).

A periodic field repeated over a large box evolves as it does alone in the small one, so the
two forms are compared cell by cell; one step and several, every storage, laminar and SA-neg with
both convection schemes and with negative chi.  Same arithmetic up to FP32 rounding: populations
within 1e-6, 16-bit storage within a few units in the last place of the largest stored values.
The restriction of both forms is checked on the c/4096 workload: covered cells hold the means of
their children (u weighted by mass) to FP32 rounding."""
import numpy as np
import pytest

import paper_2601_18443_gb300 as pkg
from paper_2601_18443_gb300 import workloads as W

pytestmark = pytest.mark.gpu

NX, NY, RX, RY = 64, 40, 8, 8           # 80 work warps alone, 5120 repeated (more than one wave)


def _solver(nx, ny, **kw):
    s = pkg.Solver(W.base_config(levels=1, nx0=nx, ny0=ny, Re=5.0, periodic=1, solid_walls=0, **kw))
    s.set_geometry([])
    return s


@pytest.mark.parametrize("kw", [dict(turbulence=0), dict(turbulence=1), dict(turbulence=1, sa_convection=1),
                                dict(turbulence=1, store=1), dict(turbulence=0, store=1), dict(turbulence=1, store=2)])
def test_pairs_of_plain_blocks_compute_what_single_ones_do(kw):
    pkg.build()
    rng = np.random.default_rng(31)
    rho = 1 + 1e-3 * rng.standard_normal((NY, NX))
    ux, uy = 0.05 + 0.01 * rng.standard_normal((NY, NX)), 0.01 * rng.standard_normal((NY, NX))
    chi = 3.0 * rng.random((NY, NX)) - 0.3                    # a tenth of the cells negative
    a, b = _solver(NX, NY, **kw), _solver(NX * RX, NY * RY, **kw)
    a.set_fields(0, rho, ux, uy, chi)
    b.set_fields(0, *(np.tile(f, (RY, RX)) for f in (rho, ux, uy, chi)))
    tol = 1e-6 if kw.get("store", 0) == 0 else (5e-4 if kw["store"] == 1 else 4e-3)
    for n in (1, 1, 9):                                       # an even step, an odd one, more
        a.step(n)
        b.step(n)
        pa, pb = a.get_populations(0), b.get_populations(0)
        assert np.isfinite(pb).all()
        assert np.abs(pb - np.tile(pa, (1, RY, RX))).max() <= tol
        fa, fb = a.get_fields(0), b.get_fields(0)
        if kw["turbulence"]:
            assert np.abs(fb["chi"] - np.tile(fa["chi"], (RY, RX))).max() <= 1e3 * tol
    a.close()
    b.close()


def test_covered_cells_hold_the_means_of_their_children():
    pkg.build()
    cfg, loops = W.naca0012_large()
    g = pkg.Solver(cfg)
    g.set_geometry(loops)
    i0, j0, nx, ny = g.level_box(0)
    g.set_fields(0, ux=0.0866 * (1 + 1e-2 * np.random.default_rng(5).standard_normal((ny, nx))))
    g.step(3)
    for l in range(cfg["levels"] - 1):
        C, F = g.get_fields(l), g.get_fields(l + 1)
        jj, ii = np.nonzero(C["mask"] == 3)
        fj, fi = 2 * (jj + C["j0"]) - F["j0"], 2 * (ii + C["i0"]) - F["i0"]
        ok = (fi >= 0) & (fj >= 0) & (fi + 1 < F["mask"].shape[1]) & (fj + 1 < F["mask"].shape[0])
        jj, ii, fj, fi = jj[ok], ii[ok], fj[ok], fi[ok]
        kids = [(fj + b, fi + a) for b in (0, 1) for a in (0, 1)]
        ok = np.all([np.isin(F["mask"][k], (1, 2)) for k in kids], axis=0)
        assert ok.sum() > 5000
        c = (jj[ok], ii[ok])
        kids = [(k[0][ok], k[1][ok]) for k in kids]
        r = np.array([F["rho"][k] for k in kids])
        assert np.abs(C["rho"][c] - r.mean(0)).max() <= 3e-7
        for f in ("ux", "uy"):
            want = (r * np.array([F[f][k] for k in kids])).sum(0) / r.sum(0)
            assert np.abs(C[f][c] - want).max() <= 1e-7
        want = np.array([F["chi"][k] for k in kids]).mean(0)
        assert np.abs(C["chi"][c] - want).max() <= 1e-6 * np.abs(want).max()
    g.close()
