"""The wall function inside the level step: a block's records are evaluated by a warp of its own,
four, two or one lanes a record (up to 8, up to 16, more), and reach the warp that updates the
block's cells through shared memory.

One launch of the finest level is compared with the query form of the wall function (one thread a
record) on the same fields: the friction velocities that the step keeps as the next Newton starts,
and the nu_tilde that it sets at the boundary nodes, which is what the partner warp received.
Velocities scaled by position make the iterations of one warp's lanes differ in length.

Bound, per record, on the difference of the two: each sums the velocity at R in FP32 from 16 terms
in its own order, within 16 * 6e-8 of S, the sum of their magnitudes, per component, and takes the
tangential part of it (four roundings of at most S): together 4e-6 S.  The relative error of u_tau
is at most that of u_t; u+ (eq 22) itself is rounded to about 2e-6 on either side (4e-6 / u+), and
the iteration stops within 4.5e-8.  With a factor of two on u+ for its fast logarithms:
4e-6 S / u_t + 8e-6 / u+ + 1e-6."""
from collections import Counter

import numpy as np
import pytest

import paper_2601_18443_gb300 as pkg
from paper_2601_18443_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("store", [0, 1])
@pytest.mark.parametrize("odd", [0, 1])
def test_wall_warps_give_what_the_query_gives(store, odd):
    pkg.build()
    cfg, loops = W.naca0012_small(levels=4)
    cfg = dict(cfg, store=store)
    g = pkg.Solver(cfg)
    g.set_geometry(loops)
    l = cfg["levels"] - 1
    ij, _, _ = g.wall_records()
    per_block = Counter(map(tuple, np.stack([ij[:, 0] // 16, ij[:, 1] // 2], axis=1).tolist()))
    forms = {1 if n <= 8 else 2 if n <= 16 else 3 for n in per_block.values()}
    assert forms == {1, 2, 3}                                  # all three splits of the lanes
    g.step(5)
    F = g.get_fields(l)
    ny, nx = F["ux"].shape
    scale = np.where(np.arange(nx) % 3 == 0, 0.05, 1.0)[None, :] * np.where(np.arange(ny) % 2 == 0, 1.0, 3.0)[:, None]
    g.set_fields(l, ux=np.nan_to_num(F["ux"]) * scale, uy=np.nan_to_num(F["uy"]) * scale)
    if odd:
        g.step_launch(l, 0)
    want, F = g.wall_state(), g.get_fields(l)
    g.step_launch(l, 0)
    blob = g.get_state()
    n, (i0, j0) = len(ij), g.level_box(l)[:2]
    sij, _, wu = g.wall_stencils()
    used = sij[:, :, 0] >= 0
    at = np.where(used, sij[:, :, 1] - j0, 0), np.where(used, sij[:, :, 0] - i0, 0)
    S = sum((np.abs(wu) * np.where(used, np.abs(F[k][at]), 0.0)).sum(1) for k in ("ux", "uy"))
    tail = blob[blob.size - 4 * (10 * n + 12 * cfg["ny0"]):].view(np.float32)
    utau, chi = tail[:n].astype(np.float64), g.get_fields(l)["chi"][ij[:, 1] - j0, ij[:, 0] - i0]
    g.close()
    assert (want[:, 3] > 0).all()
    tol = 4e-6 * S / want[:, 7] + 8e-6 * want[:, 3] / want[:, 7] + 1e-6
    assert (np.abs(utau - want[:, 3]) <= tol * want[:, 3]).all()
    assert (np.abs(chi - want[:, 4]) <= (tol + 1e-6) * want[:, 4]).all()
