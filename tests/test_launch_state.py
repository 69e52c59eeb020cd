"""Launch state shared by host threads (contexts of several threads run the same launchers):
an occupancy query fills a local variable or a `static const` once and whole, never a
function-static that another thread may read half-made.  Read from the sources, since a
wrong grid size still gives right results."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2502_00152_gb300", "csrc")


def test_occupancy_queries_do_not_write_shared_statics():
    queries = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        with open(path) as f:
            text = re.sub(r"//[^\n]*", "", f.read())
        statics = set(re.findall(r"\bstatic int (\w+)", text)) | set(re.findall(r"\bstatic int \w+ = [^;,]*, (\w+)", text))
        for target in re.findall(r"cudaOccupancyMaxActiveBlocksPerMultiprocessor\(\s*(&?\w+)", text):
            queries += 1
            assert target.startswith("&"), (path, target)  # not through a pointer that may lead to one
            assert target[1:] not in statics, (path, target)
    assert queries >= 4
