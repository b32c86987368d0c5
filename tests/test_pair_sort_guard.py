"""The guard of the pair sort is set by blocks of k_ps_sort while others run: inside
that kernel one thread per block reads it, in the ticket's turn, so that no block
has some of its threads return and others wait for them.  Read from the source: the
moment in which a block could fall apart cannot be made to happen at will."""
import pathlib
import re

SRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2108_00529_gb300" / "csrc" / "pairsort.cu"


def _body(text, name):
    at = text.index("{", re.search(r"\b%s\(" % name, text).end())
    depth, end = 1, at + 1
    while depth:
        depth += (text[end] == "{") - (text[end] == "}")
        end += 1
    return text[at:end]


def test_one_thread_reads_the_guard():
    text = re.sub(r"//[^\n]*", "", SRC.read_text())
    body = _body(text, "k_ps_sort")
    reads = [m.start() for m in re.finditer(r"ctl->guard\b(?!\s*=[^=])", body)]
    assert len(reads) == 1
    owner = body.rindex("if (threadIdx.x == 0) {", 0, reads[0])
    assert "}" not in body[owner:reads[0]]
    assert body.index("__syncthreads();", reads[0]) < body.index("return", reads[0])
