"""Dense bins: their windows are few, however short the work items of the run are.

Four tiles hold 60000 particles each near one cell.  lambda on a lattice and a particle
mass of 1 make the weights' inputs exact, so what is left of a node's error are
independent roundings (u = 2^-24 or 2^-53): the weights (12 of u F), each contribution
to 2^-K, each of the W windows' sums to u, and the W additions to the node, whose sum
grows evenly: u^2 R^2 W / 9 for a total R.  With at most twelve windows to a bin or
windows of 4096, W = 15; items of 512 particles would make it 118 and the sum of squares
seven times larger.  The sample of some 400 nodes that matter may exceed the expected
sum of squares by less than a factor of two."""
import math

import numpy as np
import pytest

from oracle import sipf_oracle as O
from paper_2512_03452_gb300 import Simulation, build, make_params

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

H, TILES, C = 64, [(1, 1, 1), (3, 5, 2), (6, 0, 7), (2, 6, 4)], 60_000


@pytest.fixture(scope="module", autouse=True)
def lib():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()


def positions():
    rng = np.random.default_rng(11)
    X = []
    for t in TILES:
        cell = 4.0 + np.clip(np.round(rng.normal(size=(C, 3)) * 0.5 * 256) / 256, -3.0, 3.0)
        X.append((8 * np.array(t) + cell) / H - 0.5)
    return np.concatenate(X)


def expected(X, precision):
    """Exact node sums and the expected squares of their errors."""
    u = 2.0 ** (-24 if precision == 32 else -53)
    cell, lam = O.cell_and_lambda(X, H, 1.0)
    offs, F = O.stencil(lam, 4)
    idx = O.stencil_indices(cell, offs, H).ravel()
    ref = np.zeros(H ** 3, np.longdouble)
    np.add.at(ref, idx, F.ravel().astype(np.longdouble))
    n = np.bincount(idx, minlength=H ** 3)
    S2 = np.bincount(idx, weights=F.ravel() ** 2, minlength=H ** 3)
    m, W = 4096, math.ceil(C / 4096)
    K = 30 - math.ceil(math.log2(56 * math.ceil(m / 256) + 1)) if precision == 32 else 62 - math.ceil(math.log2(m + 1))
    R2 = np.asarray(ref, np.float64) ** 2
    return ref, u ** 2 * R2 * (W / 9 + 1 / W) + n * 4.0 ** -K / 12 + 12 * S2 * u ** 2


@pytest.mark.parametrize("precision", [32, 64])
def test_error_is_that_of_few_windows(precision):
    X = positions()
    P = X.shape[0]
    ref, var = expected(X, precision)
    with Simulation(make_params(P, H, L=1.0, mass=float(P), dt=1e-4, precision=precision), X) as sim:
        got = sim.density(False).ravel() / float(H) ** 3
    err = np.asarray(got.astype(np.longdouble) - ref, np.float64)
    assert np.sum(err ** 2) <= 2.0 * np.sum(var)
