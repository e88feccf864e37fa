"""A failed index check of the checked build names its source file: every file with checks records its own place."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0904_4152_gb300", "csrc")


def test_checks_record_their_own_file():
    header = open(os.path.join(CSRC, "hn_internal.h")).read()
    names = re.findall(r'"([^"]+)"', header.split("const names[] = {")[1].split("}")[0])
    checked = []
    for path in sorted(glob.glob(os.path.join(CSRC, "k_*.cu"))):
        text = open(path).read()
        if not re.search(r"\bdbg_(item|level)\(", text):
            continue
        checked.append(os.path.basename(path))
        assert names[int(re.search(r"#define HN_SOURCE (\d+)", text).group(1))] == checked[-1]
        assert "__LINE__" not in text
    assert sorted(checked) == sorted(names)
