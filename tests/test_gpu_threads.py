"""Contexts of different sizes stepped by two host threads at once: a context is not
thread-safe, two contexts are.  Kernels whose dynamic shared memory depends on a
context's size share one process-wide allowance per kernel, which must never be
lowered under another thread."""
import pathlib
import re
import threading

import numpy as np
import pytest

from paper_2512_03452_gb300 import Batch, Simulation, Simulation2D, make_params

CSRC = pathlib.Path(__file__).resolve().parents[1] / "paper_2512_03452_gb300" / "csrc"


def test_shared_memory_allowance_is_a_constant():
    """Every setting of the allowance names the same maximum, not a launch's own bytes."""
    found = []
    for path in sorted(CSRC.glob("*")):
        found += re.findall(r"cudaFuncAttributeMaxDynamicSharedMemorySize,\s*([^;]*)\)", path.read_text())
    assert found == ["(int)(kMaxSmem - own)"]


def _together(programs, repeats):
    errors = []

    def loop(step):
        try:
            for _ in range(repeats):
                step()
        except Exception as e:   # reported by the main thread
            errors.append(repr(e))

    threads = [threading.Thread(target=loop, args=(p,)) for p in programs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors


@pytest.mark.gpu
@pytest.mark.parametrize("precision", [32, 64])
def test_two_planes(precision):
    P = 8192
    rng = np.random.default_rng(1)
    sims = []
    for H in (64, 256):
        X = rng.uniform(-1, 1, size=(P, 2))
        sims.append(Simulation2D(make_params(P, H, L=10.0, mass=4.0, eps=0.0, k=0.0, dt=1e-5, precision=precision), X))
    _together([lambda s=s: s.step(20) for s in sims], 200)
    for s in sims:
        s.sync()
        d = s.diagnostics()
        assert d["step"] == 4000 and abs(d["mass"] - 4.0) < 1e-3
        s.close()


@pytest.mark.gpu
def test_single_run_and_batch_in_double_precision():
    """The FP64 plane kernels of one run take more warps, and shared memory, than those of many runs."""
    rng = np.random.default_rng(2)
    P, H = 500, 64
    par = [make_params(P, H, dt=1e-5, mass=2.0, seed=i, precision=64) for i in range(9)]
    X = [rng.normal(size=(P, 3)) * 0.1 for _ in par]
    sim, batch = Simulation(par[8], X[8]), Batch(par[:8], X[:8])
    batch.use_graph(False)
    _together([lambda: sim.step(10), lambda: batch.step(10)], 60)
    sim.sync()
    batch.sync()
    assert sim.n == 600 and batch.n == 600
    assert abs(sim.diagnostics()["mass"] - 2.0) < 1e-12 and abs(batch.diagnostics(3)["mass"] - 2.0) < 1e-12
    sim.close()
    batch.close()
