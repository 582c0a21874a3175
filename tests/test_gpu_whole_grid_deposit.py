"""Deposit of small grids (H <= 16, one window for the whole grid): its sums over
particles are integer sums in units of 2^-K of a weight, added to the grid once per
window, so the grid is far closer to 64 bits than one that rounds at every particle.

The bound, in units of the particle mass w, for a node with n contributions of total
magnitude S: the weights are the same formulas in both (12 roundings of up to u S in
all), each contribution is rounded to 2^-K at most half a unit, K = 30 - ceil(log2(64
ceil(m / 256) + 1)) in single and 62 - ceil(log2(m + 1)) in double precision for the m
particles of a window, and each of the windows' sums is rounded twice when it is added.
Rounding errors are independent of one another, so their root mean square over the
grid is compared with the root mean square of these (a quarter of a unit for each
rounding to nearest is an upper bound of its own 1/sqrt(12))."""
import math

import numpy as np
import pytest

from oracle import sipf_oracle as O
from paper_2512_03452_gb300 import Simulation, build, make_params

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()


def _window_length(P, precision):
    m = 64 if precision == 64 else 512
    while m < 4096 and P // m >= 40:
        m *= 2
    return m


@pytest.mark.parametrize("precision", [32, 64])
@pytest.mark.parametrize("H,P", [(8, 1), (8, 700), (16, 511), (16, 513), (16, 2559), (16, 2560), (16, 10_000),
                                 (16, 30_719), (16, 100_003), (16, 300_000)])
def test_deposit_error_is_that_of_windows(H, P, precision):
    L, M0 = 1.0, 2.0
    rng = np.random.default_rng(P + H)
    # positions on a lattice of 1/256 of a cell: lambda is exact in either precision
    X0 = O.wrap(np.round(rng.normal(size=(P, 3)) * 0.1 * H * 256) / (H * 256), L)
    p = make_params(P, H, L=L, mass=M0, dt=1e-3, precision=precision)
    w, u = M0 / P, 2.0 ** (-24 if precision == 32 else -53)
    with Simulation(p, X0) as sim:
        got = sim.density(False) * (L / H) ** 3
    offs, F = O.stencil(O.cell_and_lambda(X0, H, L)[1], 4)
    idx = O.stencil_indices(O.cell_and_lambda(X0, H, L)[0], offs, H).ravel()
    ref = np.zeros(H ** 3, np.longdouble)
    np.add.at(ref, idx, F.ravel().astype(np.longdouble))
    n = np.bincount(idx, minlength=H ** 3)
    S2 = np.bincount(idx, weights=F.ravel() ** 2, minlength=H ** 3)
    m = min(_window_length(P, precision), P)
    K = 30 - math.ceil(math.log2(64 * math.ceil(m / 256) + 1)) if precision == 32 else 62 - math.ceil(math.log2(m + 1))
    windows = math.ceil(P / m)
    R = np.abs(np.asarray(ref, np.float64))
    var = 12 * S2 * u ** 2 + n * (0.5 * 2.0 ** -K) ** 2 + 2 * windows * (u * R) ** 2 + 4 * (u * R) ** 2
    err = np.asarray(got.ravel().astype(np.longdouble) / np.longdouble(w) - ref, np.float64)
    assert math.sqrt(np.sum(err ** 2)) <= math.sqrt(np.sum(var))
    assert abs(float(np.sum(got)) - M0) <= (1e-5 if precision == 32 else 1e-12) * M0
