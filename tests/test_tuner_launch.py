"""The tuner of the rows per thread times the pixel kernel as the loop launches it: the
early launch also selects the kernel's variant, so both take it from the plan alike (read
from the source of the two functions; the choice cannot be seen from outside)."""
import os
import re

API = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2207_10940_gb300", "csrc",
                   "api.cpp")


def _early(text, function):
    """The `early` argument (last but one) of each pixel launch in a function of api.cpp."""
    body = text[text.index(f"int {function}("):]
    body = body[:body.index("\n}\n")]
    calls = re.findall(r"launch_track_batch\(([^;]*?),\s*([^,]*),\s*([^,()]*)\)\s*(?:;|!=)", body)
    assert calls, function
    return {c[1].strip() for c in calls}


def test_the_tuner_times_the_variant_that_runs():
    text = open(API).read()
    assert _early(text, "plan_autotune") == _early(text, "plan_enqueue")
