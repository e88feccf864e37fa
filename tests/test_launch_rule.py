"""Programmatic dependent launches of the cycle's kernels follow the documented rule (hn_tuning.pdl: 2, the default:
launches of fewer blocks than SMs only), which stands in one function, hn::pdl_launch."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0904_4152_gb300", "csrc")


def test_every_programmatic_launch_of_the_cycle_takes_the_rule():
    found = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "k_*.cu"))):
        text = open(path).read()
        for m in re.finditer(r"cudaLaunchAttributeProgrammaticStreamSerialization", text):
            found += 1
            assert "pdl_launch(" in text[:m.start()].rsplit("if (", 1)[1].split("{")[0], path
    assert found >= 5
