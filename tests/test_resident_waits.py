"""The bounded waits between the CTAs of a resident march's cluster."""
import os

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0906_5170_gb300", "csrc")


def test_no_wait_is_bounded_by_a_clock():
    # a limit in wall-clock time fails a correct run whose context is switched away for that long
    for f in sorted(os.listdir(CSRC)):
        if f.endswith((".cu", ".cuh")):
            with open(os.path.join(CSRC, f)) as src:
                text = src.read()
            assert not [c for c in ("globaltimer", "clock64", "clock()", "%clock") if c in text], f
