"""What the kernel before writes changes during the life of a kernel that may start
while that one drains (launch_chained), so it may not be read as const __restrict__
or by __ldg, which promise the compiler and the read-only cache the contrary.  Read
from the sources, as a load moved before the wait need not show."""
import pathlib
import re

import pytest

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2108_00529_gb300" / "csrc"
TEXT = "\n".join(re.sub(r"//[^\n]*", "", p.read_text()) for p in sorted(CSRC.glob("*.cu*")))


def _block(at, left, right):
    """From the bracket at or after `at` to its partner, and the place behind it."""
    at = TEXT.index(left, at)
    depth, end = 1, at + 1
    while depth:
        depth += (TEXT[end] == left) - (TEXT[end] == right)
        end += 1
    return TEXT[at + 1:end - 1], end


def _kernel(name):
    """Parameters and body."""
    at = re.search(r"__global__\s+void\s+(__launch_bounds__\([^()]*\)\s+)?%s\b" % name, TEXT).end()
    params, at = _block(at, "(", ")")
    return {re.search(r"(\w+)$", p.strip()).group(1): p for p in params.split(",")}, _block(at, "{", "}")[0]


# kernel -> its parameters that the kernel before it in the chain writes
@pytest.mark.parametrize("kernel,written", [("k_hs_count", ["tmp_key"]), ("k_hs_scatter", ["tmp_key", "tmp_bucket"]),
                                            ("k_hs_bucket", ["slot_key", "slot_id"]), ("k_tile", ["keys", "perm"]),
                                            ("k_repulse", ["geo", "skip", "T"])])
def test_parameters_written_by_the_kernel_before(kernel, written):
    params, body = _kernel(kernel)
    for w in written:
        assert not ("const" in params[w] and "__restrict__" in params[w]), params[w]
        assert not re.search(r"__ldg\(&?%s\b" % w, body), w


def test_splitters_and_samples():
    for struct in ("HsSampled", "HsStored", "HsCounted"):
        body = TEXT[re.search(r"struct %s \{" % struct, TEXT).end():]
        assert "__ldg" not in body[:body.index("\n};")], struct
