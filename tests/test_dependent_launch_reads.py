"""Kernels that wait for their predecessor (pdl_wait) may start while it still writes
their inputs, and the read-only data path is defined only for memory that stays
unmodified during the whole kernel.  So no device code reads data through it: no
__ldg but of a constant table, no pointer to const marked __restrict__ (the compiler
may turn its loads into read-only ones) but to the argument tables that the host
writes before any of the kernels is launched."""
import pathlib
import re

CSRC = pathlib.Path(__file__).resolve().parents[1] / "paper_2512_03452_gb300" / "csrc"
TABLES = {"FftRun<T>", "FftRun<float>", "BinArgs<T>", "ChunkListArgs", "LayoutArgs"}


def test_no_read_only_loads_of_data():
    bad = []
    for path in sorted(CSRC.glob("*.cu*")):
        text = re.sub(r"//[^\n]*", "", path.read_text())
        for m in re.finditer(r"const\s+([\w<>: ]+?)\s*\*\s*__restrict__", text):
            if m.group(1) not in TABLES:
                bad.append((path.name, m.group(0)))
        for m in re.finditer(r"__ldg\(([^)]*)", text):
            if not m.group(1).startswith("&kLogTable["):
                bad.append((path.name, m.group(0)))
        bad += [(path.name, "ld.global.nc")] * text.count("ld.global.nc")
    assert not bad, bad
