"""Every kernel is launched so that it may be set up while the one before it
ends, so each has to wait for it before any other statement."""
import re
from pathlib import Path

CSRC = Path(__file__).resolve().parent.parent / "paper_2507_20441_gb300" / "csrc"


def test_every_kernel_waits_first():
    kernels = 0
    for f in sorted(CSRC.glob("*.cu*")):
        text = f.read_text()
        for m in re.finditer(r"^(?:static )?__global__", text, re.M):
            body = text[text.index("\n{\n", m.start()) + 3:]
            assert body.lstrip().startswith("grid_wait();"), (f.name, text[m.start():m.start() + 100])
            kernels += 1
        assert "<<<" not in text, f.name
    assert kernels >= 30
