"""Merge windows of a batch's runs: 16 bins below 16 particles a tile, 8 from there on.
Runs on either side of the line, of both grid sizes, compute bit for bit what each
computes alone (whose windows have 8 bins), read-backs and diagnostics included."""
import numpy as np
import pytest

from paper_2512_03452_gb300 import DEPOSIT_DETERMINISTIC, Batch, Simulation, build, make_params

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SIZES = [(32, 1023), (32, 1024), (64, 8191), (64, 8192), (64, 1), (128, 2500)]


@pytest.fixture(scope="module", autouse=True)
def lib():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()


@pytest.mark.parametrize("precision", [32, 64])
def test_runs_around_the_line_match_single_runs(precision):
    rng = np.random.default_rng(5)
    par = [make_params(P, H, mass=8.0, dt=1e-4, seed=i, precision=precision, deposit_mode=DEPOSIT_DETERMINISTIC)
           for i, (H, P) in enumerate(SIZES)]
    X = [rng.normal(size=(P, 3)) * 0.15 for _, P in SIZES]
    with Batch(par, X) as b:
        b.step(20)   # past a capacity rebuild
        b.sync()
        got = [(b.positions(r), b.spectrum(r), b.diagnostics(r)) for r in range(len(par))]
    for r, (p, x) in enumerate(zip(par, X)):
        with Simulation(p, x) as sim:
            sim.step(20)
            sim.sync()
            assert np.array_equal(got[r][0], sim.positions()), SIZES[r]
            assert np.array_equal(got[r][1], sim.spectrum()), SIZES[r]
            assert got[r][2]["peak"] == sim.diagnostics()["peak"], SIZES[r]
