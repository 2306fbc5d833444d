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


def test_non_coherent_loads_read_the_plans_tables_only():
    """The grid ahead on the stream may still be writing x, lambda, codes, scales and positions when a kernel comes up: they are read
    by load_input, behind grid_wait, and never by __ldg."""
    tables = r"(b0|e0|table|brow)\b"
    for name in sorted(os.listdir(CSRC)):
        text = source(name)
        for m in re.finditer(r"__ldg\(", text):
            line = text[m.end():text.index("\n", m.end())]
            assert re.match(r"(reinterpret_cast<const float4 \*>\()?\(?" + tables, line), "%s: __ldg(%s" % (name, line)
        for kernel in re.finditer(r"__global__ void [^;{]*?(kvq_\w+_kernel)\(", text, re.S):
            b = body(text, kernel.group(1) + "(")
            if "load_input" in b:
                assert 0 <= b.find("grid_wait()") < b.index("load_input"), "%s: %s reads an input before grid_wait" % (name, kernel.group(1))


def test_a_warp_is_together_at_the_instructions_that_want_it_so():
    """Cluster barriers and tensor-memory allocation are .aligned: every lane of the warp executes them together.  Callers come out of branches
    that some lanes take (a row maximum sent by the first lanes, a status bit raised or barriers set up by one thread)."""
    text = source("kvq_umma.cuh")
    for helper in ("cluster_arrive", "cluster_wait", "cluster_sync_all", "tmem_alloc", "tmem_alloc_pair"):
        b = body(text, "void %s(" % helper)
        assert re.match(r"\{\s*__syncwarp\(\);\s*asm volatile", b), helper
    for name in sorted(os.listdir(CSRC)):   # and nobody goes past the helpers
        if name != "kvq_umma.cuh":
            assert not re.search(r"barrier\.cluster|tcgen05\.alloc", source(name)), name
