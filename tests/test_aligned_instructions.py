"""The tensor-memory instructions of the kernels (tcgen05.ld, .st and their waits) are .aligned: all
lanes of a warp must issue them together, whatever branches the code around them takes.  The helpers
that wrap them bring the warp together themselves, so that no caller has to."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1705_04874_gb300", "csrc")


def functions():
    """(file, name, body) of every device helper whose body holds such an instruction."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = open(path).read()
        for m in re.finditer(r"__device__ (?:__forceinline__|inline) [\w ]+?(\w+)\((?:[^()]|\([^()]*\))*\)\s*\{", text):
            depth, end = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(text[end], 0)
                end += 1
            body = text[m.end():end]
            if re.search(r"tcgen05\.(ld|st|wait::ld|wait::st)\.sync\.aligned", body):
                yield pytest.param(body, id=f"{os.path.basename(path)}:{m.group(1)}")


@pytest.mark.parametrize("body", functions())
def test_the_warp_is_together(body):
    assert "__syncwarp();" in body[:body.index("asm volatile")]


def test_every_use_is_in_a_helper():
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        uses = len(re.findall(r"tcgen05\.(?:ld|st|wait::ld|wait::st)\.sync\.aligned", open(path).read()))
        name = os.path.basename(path)
        held = [p.values[0] for p in functions() if p.id.startswith(name + ":")]
        assert uses == sum(len(re.findall(r"tcgen05\.(?:ld|st|wait::ld|wait::st)\.sync\.aligned", b)) for b in held), name
