"""Kernels that may start while the one before them drains (launch_chained) wait
for it in their first statement: a thread that reaches memory before the wait
races with the kernel before.  Read from the sources, as a race need not show."""
import pathlib
import re

import pytest

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2108_00529_gb300" / "csrc"
TEXT = "\n".join(re.sub(r"//[^\n]*", "", p.read_text()) for p in sorted(CSRC.glob("*.cu*")))


def _bodies():
    """Name -> text after the opening brace, of every kernel defined."""
    out = {}
    for m in re.finditer(r"__global__\s+void\b", TEXT):
        brace = TEXT.index("{", m.end())
        head = re.sub(r"__launch_bounds__\([^()]*\)", "", TEXT[m.end():brace])
        name = re.match(r"\s*(k_\w+)\s*\(", head)
        if name and ";" not in head:
            out[name.group(1)] = TEXT[brace + 1:]
    return out


def _chained():
    """Kernels named in the launch_chained calls."""
    names = set()
    for m in re.finditer(r"\blaunch_chained\(", TEXT):
        depth, at = 1, m.end()
        while depth:
            depth += (TEXT[at] in "([{") - (TEXT[at] in ")]}")
            at += 1
        names |= set(re.findall(r"\bk_\w+", TEXT[m.end():at]))
    return sorted(names)


def test_the_chain_is_found():
    assert {"k_hs_rank", "k_hs_count", "k_hs_scatter", "k_hs_bucket", "k_tile", "k_tile_cross", "k_tile_emit",
            "k_repulse"} <= set(_chained())


@pytest.mark.parametrize("kernel", _chained())
def test_the_wait_comes_first(kernel):
    first = _bodies()[kernel].lstrip()
    assert first.startswith("chain_wait();"), first[:80]


def test_waits_stand_nowhere_else():
    waits = len(re.findall(r"\bchain_wait\(\);", TEXT))
    assert waits == sum(b.lstrip().startswith("chain_wait();") for b in _bodies().values())
