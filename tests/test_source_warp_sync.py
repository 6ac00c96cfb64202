"""The warp-collective tensor-memory instructions (tcgen05 ... .sync.aligned) are
undefined unless the whole warp executes them together, and a lane may reach
them out of a branch of its own. Every function that issues one converges the
warp first; read from the sources, since nothing is to run that breaks it."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1710_07041_gb300", "csrc")


def functions(text):
    """(header, body) of every top-level braced block, comments left out."""
    text = re.sub(r"//[^\n]*", "", text)
    for m in re.finditer(r"\b(\w+)\([^;{}]*\)\s*\{", text):
        depth, i = 1, m.end()
        while depth and i < len(text):
            depth += {"{": 1, "}": -1}.get(text[i], 0) if text[i] in "{}" else 0
            i += 1
        yield m.group(1), text[m.end():i]


def test_collective_tensor_memory_instructions_converge_their_warp():
    seen = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = open(path).read()
        if "tcgen05" not in text:
            continue
        for name, body in functions(re.sub(r'"[^"\n]*"', lambda s: s.group(0).replace("{", "<").replace("}", ">"), text)):
            at = body.find(".sync.aligned")
            if at < 0 or "tcgen05" not in body:
                continue
            seen += 1
            assert "__syncwarp();" in body[:at], f"{os.path.basename(path)}: {name}"
    assert seen >= 8, seen
