"""The stage kernels are launched while the kernel before them still runs and
wait for it inside, so what an earlier kernel of the frame writes is not
constant for their lifetime: it must not be read through the non-coherent
path (__ldg), which is defined for constant data alone."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2604_21749_gb300", "csrc")
# buffers of FrameDev that kernels of the same frame write (meshes and their buffers are older than the frame)
WRITTEN = "hdr|views|pairs|segs|rounds|q1|q2|bits|ctr|err|stamps|tile_cnt|tile_start|tile_fill|units|part_sorted"


def _arguments(text, name):
    """The argument text of every call of `name`, brackets matched."""
    for m in re.finditer(r"\b%s\s*\(" % name, text):
        depth, at = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(text[at], 0)
            at += 1
        yield text[m.end():at - 1]


def test_no_constant_loads_of_what_the_frame_writes():
    seen = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        assert "ld.global.nc" not in text, path
        for arg in _arguments(text, "__ldg"):
            seen += 1
            assert not re.search(r"\bf\.(%s)\b|\bvis\b" % WRITTEN, arg), f"{os.path.basename(path)}: __ldg({arg})"
    assert seen > 20
