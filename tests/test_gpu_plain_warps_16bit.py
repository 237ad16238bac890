"""Both forms of the level kernel over plain cells (one cell a lane; pairs of blocks, two cells a lane)
with 16-bit storage, to the last place.

A periodic field repeated over a large box, whose launches take pairs, evolves as it does alone in
the small one, whose launches do not.  Bounds:
- After an even step from the same stored values the two FP32 results differ by their rounding
  (1e-6, the bound of the FP32 comparison), so a stored value differs by one unit in its own last
  place at most.
- The odd step that follows starts from such values.  The collision's sum of magnitudes over the
  nine populations is largest for the one at rest: 4/9 of the density, which nine units shift by 4,
  and 5 with the terms in u.  So a value differs by its own unit and five of the largest value's.
- chi is kept in FP32: 2e-5 by rounding (values up to 3, some tens of operations), and in the second
  step what the first one's difference in u makes of it.  Its derivative by a component of u is at
  most the chi range 3 (an upwind difference; 2.2 with the central ones), by the vorticity
  cb1 chi <= 0.37, which two gradients of a difference du shift by 2 du: 8 du together."""
import numpy as np
import pytest

import paper_2601_18443_gb300 as pkg
from paper_2601_18443_gb300 import workloads as W

pytestmark = pytest.mark.gpu

NX, NY, RX, RY = 64, 40, 8, 8           # 80 work warps alone, 5120 repeated (more than one wave)
MANT = {1: 10, 2: 7}                    # stored mantissa bits: FP16, BF16
CX = np.array([0, 1, -1, 0, 0, 1, -1, 1, -1])
CY = np.array([0, 0, 0, 1, -1, 1, -1, -1, 1])


def _solver(nx, ny, **kw):
    s = pkg.Solver(W.base_config(levels=1, nx0=nx, ny0=ny, Re=5.0, periodic=1, solid_walls=0, **kw))
    s.set_geometry([])
    return s


def _shift(U):
    """What 16-bit storage keeps populations relative to: f_eq(1, U, 0)."""
    h = lambda c, u: np.where(c == 0, 2 / 3 - u * u, 0.5 * (u * u + 1 / 3 + c * u))
    return h(CX, U) * h(CY, 0.0)


def _unit(stored, store):
    """One unit in the last place of the stored values (with room for the shift's own rounding)."""
    m = np.maximum(np.abs(stored) * (1 + 1e-3) + 1e-6, 2.0**-14)
    return 2.0 ** (np.floor(np.log2(m)) - MANT[store])


@pytest.mark.parametrize("kw", [dict(turbulence=1, store=1), dict(turbulence=0, store=1), dict(turbulence=1, store=2),
                                dict(turbulence=0, store=2), dict(turbulence=1, sa_convection=1, store=2)])
def test_pairs_differ_from_single_blocks_by_last_places_only(kw):
    pkg.build()
    rng = np.random.default_rng(59)
    rho = 1 + 1e-3 * rng.standard_normal((NY, NX))
    ux, uy = 0.05 + 0.01 * rng.standard_normal((NY, NX)), 0.01 * rng.standard_normal((NY, NX))
    chi = 3.0 * rng.random((NY, NX)) - 0.3                    # a tenth of the cells negative
    a, b = _solver(NX, NY, **kw), _solver(NX * RX, NY * RY, **kw)
    a.set_fields(0, rho, ux, uy, chi)
    b.set_fields(0, *(np.tile(f, (RY, RX)) for f in (rho, ux, uy, chi)))
    assert np.array_equal(b.get_populations(0), np.tile(a.get_populations(0), (1, RY, RX)))
    shift = _shift(a.cfg["Ma"] / np.sqrt(3.0))[:, None, None]
    du = 0.0
    for step in (1, 2):                                       # an even step, an odd one
        a.step(1)
        b.step(1)
        pa, pb = np.tile(a.get_populations(0), (1, RY, RX)), b.get_populations(0)
        stored = np.maximum(np.abs(pa - shift), np.abs(pb - shift))
        bound = _unit(stored, kw["store"]) + 1e-6
        if step == 2:
            bound = bound + 5 * _unit(stored, kw["store"]).max()
        assert (np.abs(pb - pa) <= bound).all(), step
        fa, fb = ({k: v for k, v in s.get_fields(0).items() if k in ("ux", "uy", "chi")} for s in (a, b))
        fa = {k: np.tile(v, (RY, RX)) for k, v in fa.items()}
        dchi = np.abs(fb["chi"] - fa["chi"]).max()
        assert dchi <= ((2e-5 + 8 * du) if kw["turbulence"] else 0.0), step
        du = max(np.abs(fb[k] - fa[k]).max() for k in ("ux", "uy"))
        assert du <= 1e-6 if step == 1 else True              # the fields come before the storage
    a.close()
    b.close()
