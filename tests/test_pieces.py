"""Shares of lists that end near 2^32 (graphs of nearly 2^31 edges), on the CPU: the
pieces that the degree count and the pair sort take cover a list once, whatever the
place at which it ends, as 64-bit arithmetic has it."""
import pathlib
import re
import subprocess

import pytest

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2108_00529_gb300" / "csrc"

MAIN = r"""
#include <cstdio>
#include "%s"
using namespace bgv;
typedef unsigned long long u64;
static int bad(u64 start, u64 end, u64 piece, const char *why) {
    std::printf("%%s: [%%llu, %%llu) by %%llu\n", why, start, end, piece);
    return 1;
}
int main() {
    const u64 starts[] = {0, 1, 5, 7, 8, 40001, 1ull << 31, (1ull << 32) - (1ull << 20), (1ull << 32) - 30000, (1ull << 32) - 40};
    const u64 tails[] = {2, 3, 9, 24576, 24577, 1ull << 18, 300001};
    const u64 pieces[] = {8192, 24576, 1ull << 18};
    for (u64 start : starts)
        for (u64 tail : tails)
            for (u64 piece : pieces) {
                const u64 end = (1ull << 32) - tail;
                if (end <= start || (end - start) / piece > 600000) continue;
                const uint32_t n = pieces_of(uint32_t(end - start), uint32_t(piece));
                if (n != (end - start + piece - 1) / piece) return bad(start, end, piece, "count");
                u64 at = start;
                for (uint32_t q = 0; q < n; ++q) {
                    const uint32_t a = uint32_t(start) + q * uint32_t(piece);
                    const uint32_t len = piece_size(a, uint32_t(end), uint32_t(piece));
                    if (a != at || len == 0 || at + len > end) return bad(start, end, piece, "cover");
                    const uint32_t head = ragged_head(a, a + len, 8u);
                    const u64 up = (at + 7) / 8 * 8;
                    if (at + head != (up < at + len ? up : at + len)) return bad(start, end, piece, "head");
                    at += len;
                }
                if (at != end) return bad(start, end, piece, "end");
            }
    return 0;
}
"""


def test_pieces_near_the_end_of_32_bits(tmp_path):
    src = tmp_path / "pieces.cpp"
    src.write_text(MAIN % (CSRC / "pieces.cuh"))
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-o", tmp_path / "pieces", src], check=True)
    r = subprocess.run([tmp_path / "pieces"], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout


@pytest.mark.parametrize("name,forms", [("sketch.cu", ["pieces_of(c, kDegPiece)", "piece_size(a, start[lo + 1], kDegPiece)",
                                                       "ragged_head(a, b, 8u)"]),
                                        ("pairsort.cu", ["pieces_of(e.count, kPsW)", "piece_size(e.start, end, kPsW)",
                                                         "pieces_of(run_end[t] - run_start[t], kMoveKeys)"])])
def test_they_are_what_the_kernels_take(name, forms):
    text = (CSRC / name).read_text()
    for f in forms:
        assert f in text, f
    # nothing rounded up, and no place moved on by a piece, in 32 bits
    assert not re.search(r"(?<!stage) \+=? k(DegPiece|PsW|MoveKeys)\b( - 1\)|[,;)])", re.sub(r"//[^\n]*", "", text))
