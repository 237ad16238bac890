"""What lbm_autotune times: coarse steps through graphs that exist before the clock starts.

On a one-level solve every launch form does the same work a step, and so does a handle that has
stepped before: the times of a fresh handle's forms lie near those of a warm one.  Capturing a
graph of several steps takes the host as long as the ten timed steps of such a solve, so a time
that holds the capture is at least twice the one that does not."""
import pytest

import paper_2601_18443_gb300 as pkg
from paper_2601_18443_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_step_times_hold_no_graph_capture():
    pkg.build()
    cfg = W.base_config(levels=1, nx0=64, ny0=40, Re=5.0, periodic=1, solid_walls=0)
    fresh, warm = [], []
    for _ in range(5):
        a, b = pkg.Solver(cfg), pkg.Solver(cfg)
        a.set_geometry([])
        b.set_geometry([])
        b.step(128)                                # has run its graphs before it is tuned
        ra, rb = a.autotune(steps=10), b.autotune(steps=10)
        warm.append(rb["default_step_us"])
        fresh.append([ra["default_step_us"], *ra["step_us_confirm"].values(), ra["step_us"]["pdl_on"]])
        a.close()
        b.close()
    base = min(warm)
    for times in zip(*fresh):
        assert min(times) <= 1.5 * base, (min(times), base)
