"""The equaliser's two sets of barrier counters take turns: each launch clears the set of the
next one.  A launch that could not be enqueued has cleared nothing, so the sets may change
places only behind a successful launch (host order, read from the source: the launch itself
cannot be made to fail without a broken device)."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2104_06311_gb300", "csrc", "rx_api.cu")


def test_the_sets_change_places_behind_the_launch():
    text = re.sub(r"//[^\n]*", "", open(SRC).read())
    body = text[text.index("rx_status rx_process("):]
    launch = body.index("RX_CUDA(launch_eq(")          # returns from the function where it fails
    toggles = [m.start() for m in re.finditer(r"bar_set = !rx->bar_set", body)]
    assert len(toggles) == 1 and toggles[0] > launch
    between = body[launch:toggles[0]]
    assert between.count(";") == 1 and "{" not in between and "}" not in between
