"""Kernels that index with what a look-back between tiles has placed ask, before
they do, whether a wait ran out (their input then has holes), or check their
positions."""
import re
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parent.parent / "paper_2507_20441_gb300" / "csrc"

BEHIND = [("csr.cu", k) for k in ("k_inv_bucket", "k_inv_fill", "k_owners", "k_pairs", "k_cross_rank")] + \
         [("weights.cu", k) for k in ("k_window_totals", "k_guide_fill")]


@pytest.mark.parametrize("name,kernel", BEHIND)
def test_kernel_asks_for_the_status(name, kernel):
    text = (CSRC / name).read_text()
    at = re.search(r"__global__[^;{]*?\b" + kernel + r"\(", text).start()
    body = text[text.index("\n{\n", at):text.index("\n}\n", at)]
    assert "latched(status)" in body
    assert re.search(r"if \((?:s_stop|stop|bits|tile == 0xFFFFFFFFu|latched\(status\) & ST_TIMEOUT)\) (?:return|\{)", body)


def test_radix_pass_checks_its_positions():
    """(Every store of a pass goes through a position in g; the inverse checks the payload that is its place.)"""
    text = (CSRC / "csr.cu").read_text()
    at = text.index("    k_rs_sweep(")
    body = text[at:text.index("\n}\n", at)]
    stores = re.findall(r"^.*(?:J\.kout|pout|J\.inv)\[.*\] = .*$", body, re.M)
    assert len(stores) == 3
    assert all("if (g[j] < n)" in x or "v < n" in x for x in stores), stores


def test_build_looks_at_each_copy_of_the_status():
    text = (CSRC / "csr.cu").read_text()
    body = text[text.index("int build_csr("):]
    syncs = [m.start() for m in re.finditer(r'"duplicate scan"', body)]
    assert len(syncs) == 2
    for x in syncs:
        assert "build_status(ctx)" in body[x:x + 120]
