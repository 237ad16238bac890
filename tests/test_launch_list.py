"""The list of work warps that the level kernel runs, built on the host (no GPU), against the flag
words and the work warps: every one of them is in it, those with boundary nodes as pairs at the
front, and the plain part, whose code reads no flag word and takes every neighbour tile for present,
holds an even number of warps that are what it assumes."""
import numpy as np
import pytest

import paper_2601_18443_gb300 as pkg
from paper_2601_18443_gb300 import workloads as W

KIND_ACTIVE, FL_SOLID, FL_BNODE, KIND_MASK = 1, 1 << 2, 1 << 4, 0x3


@pytest.fixture(scope="module", autouse=True)
def _built():
    pkg.build()


def _box(nx, ny, periodic):
    return W.base_config(levels=1, nx0=nx, ny0=ny, Re=5.0, periodic=periodic, solid_walls=0, turbulence=1), []


def _polar(levels):
    return W.polar_case(next(q for q in W.polar_requests(64) if q["levels"] == levels))


CASES = {
    "naca-5lvl": lambda: W.naca0012_small(levels=5),
    "naca-1lvl": lambda: W.naca0012_small(levels=1),
    "polar-4lvl": lambda: _polar(4),
    "polar-6lvl": lambda: _polar(6),
    "periodic": lambda: _box(96, 24, 1),
    "ragged": lambda: _box(70, 33, 0),
    "ragged-odd": lambda: _box(131, 45, 0),
    "one-tile": lambda: _box(20, 8, 0),
}


def _level(g, l, finest, periodic):
    """Flag words padded by one tile, and the classes of the level's work warps."""
    i0, j0, nx, ny = g.level_box(l)
    i1, j1 = i0 & ~31, j0 & ~7                                     # whole tiles
    nx1, ny1 = ((i0 + nx + 31) & ~31) - i1, ((j0 + ny + 7) & ~7) - j1
    fl = np.zeros((ny1, nx1), dtype=np.int64)
    fl[j0 - j1:j0 - j1 + ny, i0 - i1:i0 - i1 + nx] = g.flags(l).reshape(ny, nx)
    present = (fl.reshape(ny1 // 8, 8, nx1 // 32, 32) != 0).any(axis=(1, 3))
    present = np.pad(present, 1, mode="wrap" if periodic and l == 0 else "constant")
    plain, pairs = set(), set()
    for i, j, w in g.work_list(l, True).tolist():
        x, y = i - i1 + 16 * (w & 1), j - j1 + 2 * (w >> 1)
        f = fl[y:y + 2, x:x + 16]
        sx, sy = (1 if w & 1 else -1), (-1 if w >> 1 == 0 else 1 if w >> 1 == 3 else 0)
        ty, tx = (j - j1) // 8 + 1, (i - i1) // 32 + 1
        if (f == KIND_ACTIVE).all() and all(present[ty + b, tx + a] for a in {0, sx} for b in {0, sy}):
            plain.add((i, j, w))
        if finest and ((f & (KIND_MASK | FL_SOLID | FL_BNODE)) == (KIND_ACTIVE | FL_BNODE)).any():
            pairs.add((i, j, w))
    return plain, pairs


@pytest.mark.parametrize("name", CASES)
def test_the_launched_list_holds_the_work_as_the_kernel_takes_it(name):
    cfg, loops = CASES[name]()
    g = pkg.Solver(cfg, host_only=True)
    g.set_geometry(loops)
    L, odd = cfg["levels"], 0
    for l in range(L):
        plain, pairs = _level(g, l, l == L - 1, cfg["periodic"])
        work = [tuple(r) for r in g.work_list(l, True).tolist()]
        out, n_pair, n_plain = g.launch_list(l)
        got = [tuple(r) for r in out.tolist()]
        # pairs: both warps in a row, in the order of the work list
        assert n_pair == 2 * len(pairs)
        assert got[0:n_pair:2] == got[1:n_pair:2] == [k for k in work if k in pairs]
        # each other warp once, general ones in the order of the work list
        tail = got[len(got) - n_plain:]
        general = got[n_pair:len(got) - n_plain]
        assert sorted(got[0:n_pair:2] + general + tail) == sorted(work)
        assert general == [k for k in work if k not in pairs and k not in set(tail)]
        # the plain ones, all but one where their number is odd
        assert n_plain == len(plain) & ~1 and set(tail) <= plain
        odd += len(plain) & 1
    if name == "ragged-odd":
        assert odd                                                # the case has that remainder
    g.close()


def test_counts_and_arguments():
    cfg, loops = CASES["ragged"]()
    g = pkg.Solver(cfg, host_only=True)
    with pytest.raises(pkg.LBMError):
        g.launch_list(0)                                          # no geometry
    g.set_geometry(loops)
    with pytest.raises(pkg.LBMError):
        g.launch_list(1)
    g.close()
