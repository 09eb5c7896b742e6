"""Checks of the native sources that need no GPU: rules that every file of csrc/ keeps, and host-side helpers compiled
with the system compiler and run here."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2109_09772_gb300", "csrc")


def _code():
    """file name -> source without comments"""
    out = {}
    for f in sorted(glob.glob(os.path.join(CSRC, "*"))):
        if f.endswith((".cu", ".cuh", ".h")):
            s = re.sub(r"/\*.*?\*/", "", open(f).read(), flags=re.S)
            out[os.path.basename(f)] = re.sub(r"//[^\n]*", "", s)
    return out


def test_every_copy_names_its_stream():
    """A copy or a fill without a stream runs on the legacy stream, which a caller's non-blocking stream does not wait
    for, and one from pageable memory may return before its transfer has ended: a kernel could read a table that is not
    there yet."""
    bad = [f"{name}: {m.group(0)}" for name, s in _code().items()
           for m in re.finditer(r"\bcudaMem(cpy|cpy2D|cpy3D|cpyToSymbol|cpyFromSymbol|set|set2D)\s*\(", s)]
    assert not bad, bad
