"""Batches whose members have the same level count run kernels made for one kind of step, and
grouped prolongations: each member equals its solve alone, for one member, a few, and enough
that the launches take plain blocks in pairs and the prolongations' descriptors overflow one
launch (FP32: rounding, 1e-6 in the populations)."""
import numpy as np
import pytest

import paper_2601_18443_gb300 as pkg
from paper_2601_18443_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("levels,members", [(4, 1), (5, 3), (4, 8), (6, 9)])
def test_uniform_batch_equals_the_solves_alone(levels, members):
    pkg.build()
    cases = [W.polar_case(dict(q, levels=levels, store=0)) for q in W.polar_requests(members, seed=77)]
    alone, batched = [], []
    for cfg, loops in cases:
        for group in (alone, batched):
            s = pkg.Solver(cfg)
            s.set_geometry(loops)
            group.append(s)
    b = pkg.Batch(batched)
    for n in (1, 2, 30):
        b.step(n)
        for a, s in zip(alone, batched):
            a.step(n)
            s.synchronize()
            for l in range(levels):
                x, y = a.get_populations(l), s.get_populations(l)
                assert np.array_equal(np.isnan(x), np.isnan(y)), l
                assert np.nanmax(np.abs(x - y)) <= 1e-6, (n, l)
    b.close()
    for s in alone + batched:
        s.close()
