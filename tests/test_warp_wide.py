"""Warp-wide (.aligned) PTX is undefined in a warp that has not converged, and a block
barrier does not converge one: every such instruction of the CUDA sources follows a
__syncwarp() in the same function, with no branch or wait between."""
import pathlib
import re

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2408_04066_gb300" / "csrc"


def test_every_aligned_instruction_follows_a_syncwarp():
    seen = 0
    for path in sorted(CSRC.glob("*.cu*")):
        text = re.sub(r"//[^\n]*", "", path.read_text())
        for m in re.finditer(r"asm\s+volatile\s*\(", text):
            end = text.index(";\n", text.index(")", m.end()))
            if ".aligned" not in text[m.start():end]:
                continue
            seen += 1
            before = text[:m.start()].rstrip()
            assert before.endswith("__syncwarp();"), (path.name, text[m.start():m.start() + 120])
    assert seen >= 8
