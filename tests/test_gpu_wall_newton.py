"""The friction-velocity iteration of the wall function (step 3 of Sec 2.3) from stale starting
values: after a few steps the finest level's velocity is rescaled, so that every record's start
is off by a large factor, and the wall state is compared with the FP64 oracle's steps 1-5.

Bound on u_tau, per record: the library evaluates u+ (eq 22) in FP32 from terms of up to 20,
absolute rounding about 2e-6, and u_tau's relative error is at most that of u+; with 1e-5 for the
gathered velocity at R: 1e-5 + 4e-6 / u+."""
import math

import numpy as np
import pytest

import oracle
import paper_2601_18443_gb300 as pkg
from paper_2601_18443_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1e-3, 0.05, 0.9999, 20.0])
def test_friction_velocity_from_a_stale_start(scale):
    pkg.build()
    oracle.build()
    cfg, loops = W.naca0012_small(levels=4)
    g = pkg.Solver(cfg)
    g.set_geometry(loops)
    g.step(5)
    l = cfg["levels"] - 1
    F = g.get_fields(l)
    g.set_fields(l, ux=np.nan_to_num(F["ux"]) * scale, uy=np.nan_to_num(F["uy"]) * scale)
    F, box = g.get_fields(l), g.level_box(l)
    st = g.wall_state()
    ij, geo, ns = g.wall_records()
    sij, _, _ = g.wall_stencils()
    nu = cfg["Ma"] * math.sqrt(1.0 / 3.0) * (cfg["chord"] / cfg["h0"]) * 2**l / cfg["Re"]
    assert len(st) > 100
    for r in range(len(st)):
        si, sj = sij[r, :ns[r], 0], sij[r, :ns[r], 1]
        dx, dy = si + 0.5 - geo[r, 5], sj + 0.5 - geo[r, 6]
        vals = [F[k][sj - box[1], si - box[0]] for k in ("rho", "ux", "uy")]
        want = oracle.wall_point(cfg, nu, dx, dy, *vals, geo[r, 2:4], geo[r, 4])
        uplus = want[7] / want[3]
        assert abs(st[r, 3] - want[3]) <= (1e-5 + 4e-6 / uplus) * want[3], (r, st[r, 3], want[3])
    g.close()
