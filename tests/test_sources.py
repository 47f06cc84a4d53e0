"""Rules that the kernels' sources keep, checked on their text."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1904_11563_gb300", "csrc")


def test_no_tma_load_multicasts():
    """The library also runs as one replica per GPU, where TMA loads stay
    within a CTA's (or a CTA pair's own) shared memory."""
    sources = [p for p in glob.glob(os.path.join(CSRC, "*")) if p.endswith((".cu", ".cuh", ".h"))]
    assert len(sources) > 10
    for path in sources:
        for asm in re.findall(r"asm volatile\((.*?)\);", open(path).read(), re.S):
            assert not ("cp.async.bulk" in asm and "multicast" in asm), (path, asm)
