"""What every kernel of the library has to keep so that it may be launched before its predecessor has ended: it waits for its
predecessors, and it reads nothing on the read-only path, whose loads may run ahead of that wait and see old data."""
import pathlib
import re

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2510_03246_b200" / "csrc"
SOURCES = sorted(CSRC.glob("*.cu")) + sorted(CSRC.glob("*.cuh"))


def _kernels():
    for path in SOURCES:
        text = path.read_text()
        for m in re.finditer(r"__global__\s+void[^;{]*?(\w+)\s*\([^{;]*\)\s*\{", text):
            depth, end = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(text[end], 0)
                end += 1
            yield path.name, m.group(1), text[m.end():end]


def test_every_kernel_waits_for_its_predecessors():
    kernels = list(_kernels())
    assert len(kernels) > 60
    for name, kernel, body in kernels:
        assert re.search(r"\b(kernel_begin|wait_for_predecessors)\(\)", body), f"{name}: {kernel}"


def test_no_loads_on_the_read_only_path():
    for path in SOURCES:
        code = re.sub(r"//[^\n]*", "", path.read_text())
        for what in (r"__restrict__", r"\b__ldg\s*\(", r"ld\.global\.nc"):
            assert not re.search(what, code), f"{path.name}: {re.search(what, code).group(0)}"
