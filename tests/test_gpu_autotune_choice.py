"""Which form lbm_autotune keeps.  Its candidates are two distinct launches a level, of two or four
warps a block, under several names: those of one launch count together, by the median of their
times, and the first of them is reported."""
from statistics import median

import pytest

import paper_2601_18443_gb300 as pkg
from paper_2601_18443_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def warps(sched):
    return 2 if sched == pkg.SCHED_WARPS else 4


@pytest.mark.parametrize("levels", [1, 4])
def test_the_kept_form_is_the_first_name_of_the_fastest_launches(levels):
    pkg.build()
    if levels == 1:
        cfg, loops = W.base_config(levels=1, nx0=64, ny0=40, Re=5.0, periodic=1, solid_walls=0), []
    else:
        cfg, loops = W.naca0012_small(levels=levels)
    for _ in range(4):
        s = pkg.Solver(cfg)
        s.set_geometry(loops)
        rep = s.autotune(steps=4)
        cand = rep["candidates"]
        level_us = list(rep["level_us"].values())                       # [candidate][level]
        forms = {w: [c for c in range(len(cand)) if warps(cand[c][1]) == w] for w in (4, 2)}
        pick = []
        for l in range(levels):
            t = {w: median(level_us[c][l] for c in cs) for w, cs in forms.items()}
            pick.append(2 if t[2] < t[4] else 4)
        variants = [tuple(pick)] * 2 + [(4,) * levels] + [(warps(c[1]),) * levels for c in cand]
        us = list(rep["step_us_confirm"].values())
        times = {f: median(u for u, g in zip(us, variants) if g == f) for f in variants}
        kept = min(times, key=times.get)
        assert rep["confirm_choice"] == variants.index(kept)
        assert tuple(warps(p) for p in rep["sched"]) == kept
        # one name a form, of those that have no effect the first
        assert all(p in (pkg.SCHED_TILE, pkg.SCHED_WARPS) for p in rep["sched"]), rep["sched"]
        assert rep["min_blocks"] == [5] * levels and rep["shape"] == [0] * levels
        s.close()
