"""Rules of the CUDA sources that no run can show to be kept."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _code(path):
    """The file without its comments and string literals."""
    s = open(path).read()
    s = re.sub(r"/\*.*?\*/", " ", s, flags=re.S)
    s = re.sub(r'"(\\.|[^"\\\n])*"', '""', s)
    return re.sub(r"//[^\n]*", " ", s)


def _sources():
    d = os.path.join(ROOT, "paper_2308_13476_gb300", "csrc")
    files = sorted(f for e in ("*.cu", "*.cuh", "*.h") for f in glob.glob(os.path.join(d, e)))
    assert files
    return {os.path.basename(f): _code(f) for f in files}


def test_warp_exchanges_name_their_lanes():
    """A shuffle or vote names the lanes that must take part; __activemask()
    gives those that happen to have converged, which the language leaves open
    after a divergent branch."""
    assert [f for f, s in _sources().items() if "__activemask" in s] == []


def test_launch_geometry_asks_the_device_for_its_size():
    """No choice of a launch's geometry rests on one chip's number of streaming
    multiprocessors (152, or a small multiple of it) written into the code."""
    sizes = {152 * m + d for m in (1, 2, 3, 4, 6, 8) for d in (-1, 0)}
    found = {f: sorted({int(v) for v in re.findall(r"(?<![\w.])(\d+)(?:[uUlL]*)(?![\w.])", s)} & sizes)
             for f, s in _sources().items()}
    assert {f: v for f, v in found.items() if v} == {}
