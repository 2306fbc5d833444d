"""Orderings inside the kernels that no run violates on demand, read from the sources."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_05699_b200", "csrc")


def source(name):
    """The file without its comments."""
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*|/\*.*?\*/", "", f.read(), flags=re.S)


def body(text, head):
    """The braces that follow the first occurrence of `head`."""
    at = text.index("{", text.index(head))
    depth = 0
    for i in range(at, len(text)):
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth == 0:
            return text[at:i]
    raise AssertionError("unbalanced braces after " + head)


def test_decode_rebuild_writes_its_reciprocals_after_both_waits():
    """A dequant group's reciprocals in shared memory are read by its four warps until the tile they built for is handed over, and
    row 0 of them by the first build's sixteen warps: both waits (the group's own last tile, the tile before this one) stand
    before the write, the readers of the new row behind it."""
    b = body(source("kvq_umma_decode.cu"), "bool rebuild_b(")
    waits = [m.start() for m in re.finditer(r"wait_or_abort\(", b)]
    post = b.index("post_reciprocals")
    assert len(waits) == 2 and max(waits) < post < b.index("rows.store") < b.index("rows.rest")
