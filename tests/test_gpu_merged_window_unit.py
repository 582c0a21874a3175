"""Windows of the small bins that a merged work item holds: their unit and their range.

Unit: lambda on a lattice of 1/256 makes every Gamma_2 weight a multiple of 2^-24, so
windows in units of 2^-24 of a weight give node sums below 1 without any error (a float
holds them too), and a coarser unit does not.  Range: with a bin's particles all at one
point, node sums reach the number of particles, and, beyond the cell of Gamma_4, its
smallest weights, about -0.064 times that number."""
import numpy as np
import pytest

from oracle import sipf_oracle as O
from paper_2512_03452_gb300 import Simulation, build, make_params

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

H, NT = 128, 16 ** 3


@pytest.fixture(scope="module", autouse=True)
def lib():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()


def _tiles(seed, cells, lattice):
    """230 to 255 particles in every tile of 8^3 cells (so that all bins below 240 are merged): cells(rng, count)
    gives their cells in the tile, lattice(rng, count) their lambda in 1/256."""
    rng = np.random.default_rng(seed)
    X = []
    for t in range(NT):
        n = int(rng.integers(230, 256))
        corner = 8 * np.array([t // 256, (t // 16) % 16, t % 16])
        X.append((corner + cells(rng, n) + lattice(rng, n) / 256.0) / H - 0.5)
    return np.concatenate(X)


def _deposited(X, order):
    P = X.shape[0]
    p = make_params(P, H, L=1.0, mass=float(P), dt=1e-4, precision=32, p2g_order=order)
    with Simulation(p, X) as sim:
        return sim.density(False) / float(H) ** 3


def test_sums_below_one_are_exact():
    def cells(rng, n):
        c = rng.permutation(512)[:n]
        return np.stack([c // 64, (c // 8) % 8, c % 8], axis=1)

    X = _tiles(1, cells, lambda rng, n: rng.integers(1, 256, size=(n, 3)))
    got = _deposited(X, 2)
    ref = O.deposit(X, 1.0, H, 1.0, 2)
    low = ref < 1.0
    assert np.count_nonzero(low) > H ** 3 // 4
    assert np.array_equal(got[low], ref[low])


@pytest.mark.parametrize("lam", [1, 148, 255])
def test_range_of_sums(lam):
    def cells(rng, n):
        return np.broadcast_to(rng.integers(0, 8, size=(1, 3)), (n, 3))

    X = _tiles(lam, cells, lambda rng, n: np.full((n, 3), lam))
    got = _deposited(X, 4)
    ref = O.deposit(X, 1.0, H, 1.0, 4)
    assert ref.max() > 100 and ref.min() < (-5 if lam == 148 else 0)
    # 12 roundings a weight, two a sum of at most eight bins, and half a unit of 2^-24 a particle
    assert np.max(np.abs(got - ref)) <= (12 + 16) * 2.0 ** -24 * np.max(np.abs(ref)) + 8 * 256 * 2.0 ** -25
