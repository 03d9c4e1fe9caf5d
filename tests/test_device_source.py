"""Rules of the device sources that no run shows reliably."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2005_08348_gb300", "csrc")


def _code(path):
    """A source without its comments."""
    txt = open(path).read()
    return re.sub(r"/\*.*?\*/", "", re.sub(r"//[^\n]*", "", txt), flags=re.S)


def _sources(*names):
    files = [os.path.join(CSRC, n) for n in names] or glob.glob(os.path.join(CSRC, "*.cu*"))
    assert files
    return {os.path.basename(f): _code(f) for f in files}


def test_no_non_coherent_load():
    """The persistent kernel writes lists, positions and types that it reads
    again in the same launch: a non-coherent load (ld.global.nc, __ldg) may keep
    a line from before a list build, whatever barrier lies between."""
    for name, txt in _sources().items():
        assert not re.search(r"ld\.global(\.\w+|::\w+)*\.nc\b|\b__ldg\s*\(", txt), name


def test_no_aligned_cluster_barrier():
    """k_chain_walk comes to its cluster barriers from code that diverges by
    lane, where an .aligned arrival is undefined (it may wait without end)."""
    for name, txt in _sources().items():
        assert not re.search(r"barrier\.cluster\.(arrive|wait)(\.\w+)*\.aligned", txt), name
