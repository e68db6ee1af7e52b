"""The bench's headline is timed as users run the library: the events that time single launches also keep the setup's
overlap off, so they belong to a step of their own."""
import inspect
import re

import bench


def test_no_launch_is_timed_within_the_timed_steps():
    src = inspect.getsource(bench.run_ours)
    start, stop = src.index("clocks.start()"), src.index("clocks.stop()")
    assert re.findall(r"hm_profile\(h, (\d)\)", src[:start])[-1] != "1"
    assert "hm_profile" not in src[start:stop]
    assert re.findall(r"hm_profile\(h, (\d)\)", src[stop:])[:3] == ["2", "1", "0"]
