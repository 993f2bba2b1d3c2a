"""Every kernel is launched so that it may be set up while its predecessor still runs, and
waits for it in its first statement, grid_begin().  A kernel without that wait would read
its predecessor's output early, and its successor would not be ordered after the
predecessor either: checked on the sources, for every definition and every launch."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2004_14696_gb300", "csrc")


def sources():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        with open(path) as f:
            yield os.path.basename(path), re.sub(r"//[^\n]*", "", f.read())


def test_every_kernel_begins_with_the_wait():
    seen = 0
    for name, text in sources():
        for m in re.finditer(r"__global__", text):
            rest = text[m.end():]
            body, end = rest.find("{"), rest.find(";")
            if end != -1 and end < body:      # a declaration
                continue
            seen += 1
            assert rest[body + 1:].lstrip().startswith("grid_begin();"), (name, rest[:body].split("(")[0].split()[-1])
    assert seen > 30


def test_every_launch_goes_through_the_helper():
    for name, text in sources():
        assert "<<<" not in text, name
