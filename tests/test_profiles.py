"""The recorded profiler commands stay small: ncu runs the bench with its small-case
options or not at all."""

import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_no_capture_of_the_full_size_bench():
    files = glob.glob(os.path.join(ROOT, "profiles", "*.md"))
    assert files
    for path in files:
        text = open(path).read()
        for block in re.findall(r"```(.*?)```", text, re.S):
            block = block.replace("\\\n", " ")
            if "ncu " not in block:
                continue
            for line in block.splitlines():
                if "bench.py" in line:
                    assert "--reduce-log2" in line and "--store-log2" in line, (path, line)
