"""What a handle remembers about its step graphs, read from the source (no GPU: a capture cannot be
made to fail from outside): capture_graphs, which every new grid and every change of the launches
goes through, starts all of it afresh, so that a failed capture of a graph of several steps does
not hold the handle to single steps for good."""
import os
import re

CAPI = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2601_18443_gb300", "csrc",
                    "lbm_capi.cu")


def test_new_graphs_start_without_the_old_ones_state():
    with open(CAPI) as f:
        text = f.read()
    members = re.search(r"cudaGraphExec_t graph\[2\].*?(?=std::vector<void \*> allocs)", text, re.S).group(0)
    names = re.findall(r"^\s*(?:cudaGraphExec_t|bool|long long|int) (\w+)", members, re.M)
    assert names == ["graph", "bulk", "bulk_off", "single_steps"]
    body = re.search(r"^static lbm_status capture_graphs\(.*?^}", text, re.S | re.M).group(0)
    reset = body[:body.index("capture_steps(")]                  # before the first capture
    for name in names:
        assert re.search(r"s->%s(\[b\])? = (nullptr|false|0);" % name, reset), name
