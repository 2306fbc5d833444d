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
    row 0 of them by the first build's warps: both waits (the group's own last tile, the tile before this one) stand
    before the write, the readers of the new row behind it."""
    b = body(source("kvq_umma_decode.cu"), "bool rebuild_b(")
    waits = [m.start() for m in re.finditer(r"wait_or_abort\(", b)]
    post = b.index("post_reciprocals")
    assert len(waits) == 2 and max(waits) < post < b.index("rows.store") < b.index("rows.rest")


def definitions():
    """(file, name, head, body) of every function of the kernels' sources."""
    for name in sorted(os.listdir(CSRC)):
        text = re.sub(r"__launch_bounds__\((?:[^()]|\([^()]*\))*\)", "", source(name))
        for m in re.finditer(r"(__global__|__device__)[^;{}=]*?\b(\w+)\s*\([^;{}]*\)\s*(?:const\s*)?(?::[^;{}]*)?(?=\{)", text):
            yield name, m.group(2), m.group(0), body(text[m.end():], "")


def test_non_coherent_loads_read_the_plans_tables_only():
    """The grid ahead on the stream may still be writing x, lambda, codes, scales and positions when a kernel comes up: they are read
    by load_input and never by __ldg."""
    tables = r"(b0|e0|table|brow)\b"
    for name in sorted(os.listdir(CSRC)):
        text = source(name)
        for m in re.finditer(r"__ldg\(", text):
            line = text[m.end():text.index("\n", m.end())]
            assert re.match(r"(reinterpret_cast<const float4 \*>\()?\(?" + tables, line), "%s: __ldg(%s" % (name, line)


def test_inputs_are_read_behind_the_grid_wait():
    """In a kernel, and in every function that waits for the grid ahead on a kernel's behalf, nothing that reads an input, itself or through what it calls,
    stands in front of grid_wait(); but for a call of a function that waits itself."""
    found = list(definitions())
    kernels = {n for _, n, head, _ in found if "__global__" in head}
    waits = {n for _, n, _, b in found if "grid_wait()" in b}
    readers, grown = {"load_input"}, 0
    while len(readers) > grown:   # the functions (and the types, by their constructors) that read an input at any depth
        grown = len(readers)
        readers |= {n for _, n, _, b in found if re.search(r"\b(%s)\b" % "|".join(readers), b)}
        for name in sorted(os.listdir(CSRC)):
            readers |= {m.group(2) for m in re.finditer(r"typedef (\w+)<[^;]*> (\w+);", source(name)) if m.group(1) in readers}
    assert {"RecipLambda", "Recip", "lift_of", "load_lambda", "load_row_scales", "rebuild_b", "redo_tiles_fp32"} <= readers
    assert {"first_operand", "build_forward", "build_inverse"} <= waits & readers and len(waits & kernels) >= 10
    early = readers - waits
    for name, n, _, b in found:
        if n in waits or n in kernels & readers:
            at, first = b.find("grid_wait()"), re.search(r"\b(%s)\b" % "|".join(early), b)
            assert at >= 0, "%s: %s reads inputs and never waits" % (name, n)
            assert first is None or first.start() > at, "%s: %s reads an input (%s) before grid_wait" % (name, n, first.group(0))


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
