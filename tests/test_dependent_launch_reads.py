"""Kernels that wait for their predecessor (pdl_wait) may start while it still writes
their inputs, and the read-only data path is defined only for memory that stays
unmodified during the whole kernel.  So they read no data through it: no __ldg but of
a constant table, no pointer to const marked __restrict__ (the compiler may turn its
loads into read-only ones) but to the argument tables that the host writes before any
of the kernels is launched.  Kernels without the wait are free to; device functions,
which either may call, are not."""
import pathlib
import re

CSRC = pathlib.Path(__file__).resolve().parents[1] / "paper_2512_03452_gb300" / "csrc"
TABLES = {"FftRun<T>", "FftRun<float>", "BinArgs<T>", "ChunkListArgs", "LayoutArgs"}


def _without_kernels_that_do_not_wait(text):
    """The text less every __global__ function (to the closing brace in the first column) that never waits."""
    def keep(m):
        return m.group(0) if "pdl_wait" in m.group(0) else ""
    return re.sub(r"__global__.*?\n\}\n", keep, text, flags=re.S)


def test_no_read_only_loads_of_data():
    bad = []
    for path in sorted(CSRC.glob("*.cu*")):
        text = _without_kernels_that_do_not_wait(re.sub(r"//[^\n]*", "", path.read_text()))
        for m in re.finditer(r"const\s+([\w<>: ]+?)\s*\*\s*__restrict__", text):
            if m.group(1) not in TABLES:
                bad.append((path.name, m.group(0)))
        for m in re.finditer(r"__ldg\(([^)]*)", text):
            if not m.group(1).startswith("&kLogTable["):
                bad.append((path.name, m.group(0)))
        bad += [(path.name, "ld.global.nc")] * text.count("ld.global.nc")
    assert not bad, bad


def test_kernels_without_the_wait_are_launched_without_overlap():
    """launch_k (and the first kernel of launch_sized) names only kernels that wait."""
    for path in sorted(CSRC.glob("*.cu")):
        text = re.sub(r"//[^\n]*", "", path.read_text())
        waits = {}
        for m in re.finditer(r"__global__[^;{]*?(\w+)\s*\((?:[^;{]*)\)\s*\{.*?\n\}\n", text, flags=re.S):
            name = re.search(r"(k\w*_\w+|k2_\w+)\s*\(", m.group(0)).group(1)
            waits[name] = "pdl_wait" in m.group(0)
        for m in re.finditer(r"launch_k\(\s*(k\w+)", text):
            if m.group(1) in waits:
                assert waits[m.group(1)], (path.name, m.group(1))
