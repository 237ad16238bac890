"""Field reads of one handle from several threads at once: every call has its own host buffer, so
each returns what a read alone returns, whatever the sizes of the levels read beside it."""
import threading

import numpy as np
import pytest

import paper_2601_18443_gb300 as pkg
from paper_2601_18443_gb300 import workloads as W

pytestmark = pytest.mark.gpu

KEYS = ("rho", "ux", "uy", "chi", "mask")


def test_overlapping_reads_return_what_single_ones_do():
    pkg.build()
    cfg, loops = W.naca0012_small(levels=5)
    cfg = dict(cfg, nx0=256, ny0=128, x0=-11.5, y0=-8.0)         # level 0 far larger than the others
    s = pkg.Solver(cfg)
    s.set_geometry(loops)
    s.step(6)
    L = cfg["levels"]
    want = [s.get_fields(l) for l in range(L)]
    wrong = []

    def read(k):
        for n in range(60):
            l = (k + n * (1 + k % 3)) % L
            f = s.get_fields(l)
            if not all(np.array_equal(f[key], want[l][key], equal_nan=key != "mask") for key in KEYS):
                wrong.append((k, n, l))

    threads = [threading.Thread(target=read, args=(k,)) for k in range(8)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong, wrong[:10]
    # set_fields takes a buffer of its own too: writing a level's own values back changes nothing
    s.set_fields(L - 1)
    f = s.get_fields(L - 1)
    act = np.isin(want[L - 1]["mask"], (1, 2))
    for key in ("rho", "ux", "uy", "chi"):
        assert np.array_equal(f[key][act], want[L - 1][key][act]), key
    s.close()
