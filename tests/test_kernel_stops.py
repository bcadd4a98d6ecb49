"""Kernels that index with what a look-back between tiles has placed ask, before
they do, whether a wait ran out (their input then has holes)."""
import re
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parent.parent / "paper_2507_20441_gb300" / "csrc"

BEHIND = [("csr.cu", k) for k in ("k_rs_sweep", "k_inv_bucket", "k_inv_fill", "k_owners", "k_pairs", "k_cross_rank")] + \
         [("weights.cu", k) for k in ("k_window_totals", "k_guide_fill")]


@pytest.mark.parametrize("name,kernel", BEHIND)
def test_kernel_asks_for_the_status(name, kernel):
    text = (CSRC / name).read_text()
    at = re.search(r"__global__[^;{]*?\b" + kernel + r"\(", text).start()
    body = text[text.index("\n{\n", at):text.index("\n}\n", at)]
    assert "latched(status)" in body
    assert re.search(r"if \((?:s_stop|stop|bits|tile == 0xFFFFFFFFu|latched\(status\) & ST_TIMEOUT)\) (?:return|\{)", body)


def test_build_looks_at_each_copy_of_the_status():
    text = (CSRC / "csr.cu").read_text()
    body = text[text.index("int build_csr("):]
    syncs = [m.start() for m in re.finditer(r'"duplicate scan"', body)]
    assert len(syncs) == 2
    for x in syncs:
        assert "build_status(ctx)" in body[x:x + 120]
