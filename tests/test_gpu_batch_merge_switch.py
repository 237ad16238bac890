"""lbm_set_prolong_merge on a member holds in a batch too: with one member's prolongations on their
own, those of the batch are, and the values stay those of the grouped ones, bit for bit (the same
kernel over the same cells, in more launches)."""
import numpy as np
import pytest

import paper_2601_18443_gb300 as pkg
from paper_2601_18443_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_a_batch_groups_prolongations_only_where_every_member_does():
    pkg.build()
    levels = 5
    cases = [W.polar_case(dict(q, levels=levels, store=0)) for q in W.polar_requests(3, seed=12)]
    groups = []
    for merge in ((1, 1, 1), (1, 0, 1)):
        members = []
        for (cfg, loops), on in zip(cases, merge):
            s = pkg.Solver(cfg)
            s.set_geometry(loops)
            s.set_prolong_merge(on)
            members.append(s)
        b = pkg.Batch(members)
        # a launch per level step, and per prolongation where they go out on their own
        apart = (2**levels - 1) + (2 ** (levels - 1) - 1)
        if all(merge):
            assert b.info()["kernels_per_step"] < apart
        else:
            assert b.info()["kernels_per_step"] == apart
        b.step(5)
        for s in members:
            s.synchronize()
        groups.append((b, members))
    for x, y in zip(groups[0][1], groups[1][1]):
        for l in range(levels):
            assert np.array_equal(x.get_populations(l), y.get_populations(l), equal_nan=True), l
    for b, members in groups:
        b.close()
        for s in members:
            s.close()
