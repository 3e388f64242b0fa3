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


def test_flags_acquired_by_other_lanes_are_ordered_before_the_loads():
    """The loader of the one-launch solve looks at 32 tiles' flags, a lane each, and lane 0 then issues the loads: between the
    acquires and the proxy fence in front of the loads stands a warp barrier (a vote orders no memory)."""
    text = re.sub(r"//[^\n]*", "", (CSRC / "sp_solve_tc.cu").read_text())
    wait = text[text.index("auto wait_tiles"):text.index("uint32_t kl = kc;")]
    after = wait[wait.rindex("__ballot_sync"):]
    assert re.search(r"__syncwarp\(\);\s*asm volatile\(\"fence\.proxy\.async", after)
