"""Properties of the CUDA sources whose breach could fault or corrupt on a GPU: held here by reading them."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2405_09233_gb300", "csrc")
SOURCES = {os.path.basename(f): open(f).read()
           for f in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")))}


def code(text):
    """The text without comments."""
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)


def test_commits_come_from_the_issuing_lane():
    """tcgen05.commit covers the MMAs of the executing thread only, and elect.sync does not say which lane it picks:
    every MMA and every commit is predicated on the elected lane, also on the paths of an expired wait."""
    seen = 0
    for name, text in SOURCES.items():
        text = code(text)
        for m in re.finditer(r"tcgen05\.(mma|commit)\.", text):
            seen += 1
            assert text[:m.start()].endswith("@q "), (name, text[m.start():m.start() + 60])
    assert seen >= 3


def test_host_tables_are_copied_in_stream_order():
    """A plain cudaMemcpy from pageable memory may return before its copy is done, and its stream is not ordered with a
    non-blocking one: whatever kernels read is copied by cudaMemcpyAsync on their stream or one they are ordered after."""
    for name, text in SOURCES.items():
        for m in re.finditer(r"cudaMemcpy\(([^;]*);", code(text)):
            assert "cudaMemcpyHostToDevice" not in m.group(1), (name, m.group(0))
