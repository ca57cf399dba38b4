"""The contexts' streams are non-blocking: work on the legacy default stream is not ordered
with them, and cudaMemset or a device-to-device cudaMemcpy there may still run when it
returns.  So the sources issue every copy and clear on a context's own stream."""
import pathlib
import re

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2408_04066_gb300" / "csrc"


def test_no_copies_or_clears_on_the_legacy_stream():
    found = []
    for path in sorted(CSRC.iterdir()):
        if path.suffix in (".cu", ".cpp", ".cuh", ".h"):
            text = re.sub(r"//[^\n]*", "", path.read_text())
            found += [(path.name, m.group(0)) for m in re.finditer(r"\bcuda(?:Memset|Memcpy)(?:2D|3D)?\(", text)]
    assert not found
