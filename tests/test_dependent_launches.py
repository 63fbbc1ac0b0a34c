"""Kernels launched as programmatic dependents may be resident before their predecessor is
complete. So each begins with the wait, and reads through the read-only path (__ldg: data that
nothing writes during the kernel) only links, clover and tables, never a field that the
predecessor may have produced. Checked on the source text."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1109_2935_gb300", "csrc")

# the functions that read links or clover, and the names by which they hold them (a field
# next to them is `self`, `s`, `src` or `in`)
READERS = {
    "ldg_chunk": r"p", "ld_chunk": r"p",
    "LinkIO": r"plane", "CloverIO": r"b", "clover_block": r"b", "clover_block_raw": r"b",
    "copy_chunk": r"src", "schwarz_kernel": r"clov_g", "apply_clover_site": r"b", "clover_self_h": r"clov",
    "clover_site_n": r"clov", "row64": r"dp|m", "load_link_h": r"plane",
}


def _sources():
    """Text of every file with dependent launches, or included by one, comments removed."""
    text = {}
    for f in sorted(os.listdir(CSRC)):
        s = open(os.path.join(CSRC, f)).read()
        text[f] = re.sub(r"//[^\n]*|/\*.*?\*/", "", s, flags=re.S)
    use = {f for f, s in text.items() if "launch_pdl(" in s}
    todo = list(use)
    while todo:
        for h in re.findall(r'#include "(\w+\.cuh)"', text[todo.pop()]):
            if h not in use:
                use.add(h)
                todo.append(h)
    return {f: text[f] for f in use}


def _definitions(s):
    """(name, body) of the functions and structs that start at the beginning of a line."""
    starts = [m.start() for m in re.finditer(r"^(?=template|__device__|__global__|static|inline|struct)", s, re.M)]
    for a, b in zip(starts, starts[1:] + [len(s)]):
        part = s[a:b]
        if re.fullmatch(r"template <.*>\s*", part):  # its definition is the next part
            continue
        head = part.split("{", 1)[0]
        m = re.search(r"struct (\w+)", head) or re.search(r"(?<!__launch_bounds__)\b(?!__launch_bounds__)(\w+)\((?!\()", head)
        yield (m.group(1) if m else "?"), part


def test_read_only_loads_are_of_links_and_clover():
    seen = set()
    for f, s in _sources().items():
        for name, part in _definitions(s):
            for m in re.finditer(r"(?:__ldg|\bldg_chunk<[^>]*>|\bld_chunk<\w+, \w+>)\(([^;]*)", part):
                arg = re.sub(r"reinterpret_cast<[^>]*>|chunk_at<\d+>", "", m.group(1)).lstrip("( ")
                assert name in READERS, f"{f}: {name} reads `{arg}` through the read-only path"
                got = re.match(r"\w+", arg).group(0)
                assert re.fullmatch(READERS[name], got), f"{f}: {name} reads `{got}` through the read-only path"
                seen.add(name)
    assert {"LinkIO", "CloverIO", "clover_site_n"} <= seen  # the scan does find them
    field = _sources()["field.cuh"]
    spinor_io = field[field.index("struct SpinorIO"):field.index("struct LinkIO")]
    assert "ld_field<" in spinor_io and not re.search(r"__ldg|ldg_chunk|ld_chunk", spinor_io)


def test_dependents_begin_with_the_wait():
    text = "\n".join(_sources().values())
    kernels = set(re.findall(r"launch_pdl\((\w+)", text)) - {"void"}
    kernels = {k if k != "kern" else "schwarz_kernel" for k in kernels}
    assert len(kernels) > 20
    for k in sorted(kernels):
        body = re.search(rf"\b{k}\([^{{;]*\)\s*\{{\s*([^;]*);", text)
        assert body, k
        assert body.group(1).strip() == "pdl_begin()", f"{k} begins with `{body.group(1).strip()}`"


def test_links_and_clover_are_settled_before_a_dependent():
    api = open(os.path.join(CSRC, "api.cu")).read()
    load = api[api.index("int dirac_load_gauge"):]
    load = load[:load.index("\n}\n")]
    last_write = max(load.rindex("launch_pack_links"), load.rindex("launch_build_clover"))
    assert last_write < load.index("launch_settle(st)") < load.index("have_gauge = true")
    for f, s in _sources().items():  # and launched plainly: it waits for the writers' completion
        assert not re.search(r"launch_pdl\(settle_kernel", s), f


def test_no_kernel_lets_its_successor_come_up_beside_it():
    """Blocks that become resident beside a running grid are placed unevenly, which doubles the
    time of grids of a few blocks per SM: successors come up when the blocks have left."""
    for f, s in _sources().items():
        assert "launch_dependents" not in s, f
