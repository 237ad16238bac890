"""Aligned barriers of the level kernel, read from the source (no GPU).

`bar.sync` and `bar.arrive` without `.unaligned` must be executed by all lanes of a warp together.
Code with a per-lane branch or a loop of per-lane length stands before each use, and whether the
lanes have met again at its end is the compiler's choice, so every function that issues such an
instruction brings them together itself, before the first one."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2601_18443_gb300", "csrc")


def _functions_with_named_barriers():
    out = []
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith((".cu", ".cuh")):
            continue
        with open(os.path.join(CSRC, name)) as f:
            text = re.sub(r"//[^\n]*", "", f.read())
        # function bodies: a closing brace in the first column ends each
        for body in re.findall(r"^\w[^\n;]*\([^;{]*\)\s*\n\{\n(.*?)^\}", text, re.S | re.M):
            if re.search(r"asm volatile\(\"bar\.", body):
                out.append((name, body))
    return out


def test_lanes_meet_before_every_aligned_barrier():
    bodies = _functions_with_named_barriers()
    assert len(bodies) == 2                                   # the arriving and the waiting side
    for name, body in bodies:
        first = body.index('asm volatile("bar.')
        assert "__syncwarp();" in body[:first], (name, body)
        # ... at the top level of the function, so that no lane can branch around it
        assert re.search(r"^    __syncwarp\(\);", body[:first], re.M), (name, body)
