"""Wide full-range passes, host side: a warp's loads of a step's sums stay inside the step."""
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.abspath(__file__)))
import wide_rules  # noqa: E402


def test_a_warp_loads_every_byte_of_a_step_once_and_no_other(tmp_path):
    exe = wide_rules.compile_rules(tmp_path)
    # (cost words per lane, whether the loads are right): odd counts leave 16 lanes without a last one
    assert wide_rules.ask(exe, ["elements"]) == [(nq, 1) for nq in range(3, 9)]
