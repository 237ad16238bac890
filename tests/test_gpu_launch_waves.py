"""When the level kernel's launches take plain blocks in pairs: exactly where, one block a warp, they
would not all be resident at once.  The grid of each launch is read from the timeline; the residency
is that of the kernel's register allocation, 4 blocks of 4 warps a SM on levels with a finer one and 5
on the others."""
import pytest
import torch

import paper_2601_18443_gb300 as pkg
from paper_2601_18443_gb300 import workloads as W

pytestmark = pytest.mark.gpu


# 48 and 52 layers: level 2 between the two residencies, with 40 below both; level 3 above
@pytest.mark.parametrize("layers", [40, 48, 52])
def test_launches_of_more_than_one_wave_take_pairs(layers):
    pkg.build()
    cfg, loops = W.naca0012_large(layers=layers)
    s = pkg.Solver(cfg)
    s.set_geometry(loops)
    s.set_timeline(True)
    s.step(2)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    L, seen = cfg["levels"], set()
    lists = [s.launch_list(l) for l in range(L)]
    for t in s.timeline():
        if t["kind"] > 1:
            continue
        l = t["level"]
        rows, _, plain = lists[l]
        singles, pairs = -(-len(rows) // 4), -(-(len(rows) - plain // 2) // 4)
        one_wave = len(rows) <= 4 * sms * (4 if l < L - 1 else 5)
        assert t["blocks"] == (singles if one_wave else pairs), (l, t["blocks"], singles, pairs)
        seen.add((l, one_wave))
    assert {l for l, _ in seen} == set(range(L)) and {w for _, w in seen} == {False, True}
    s.close()
