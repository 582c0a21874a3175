"""Work items of the particle passes at their edges: bins whose particle counts
lie around the item length, the merge threshold, the warp windows' range and the
window threshold, for the item lengths that small, middle and larger runs take.
The deposited grid is compared with the oracle's deposit of the same positions,
node by node: FP32 by the fixed-point and rounding bound of the full-size
deposit test (its K = 19 is the smallest exponent of any window here too), FP64
to 1e-12 of the largest node (fixed-point sums: 1e-11, units of 2^-40 and at most
some thousand contributions to a node); no particle may be lost or doubled by a step."""
import numpy as np
import pytest

from oracle import sipf_oracle as O
from paper_2512_03452_gb300 import Simulation, build, make_params
from test_gpu_parity import _check_deposit

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EDGES = [1, 2, 23, 24, 25, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257, 511, 512, 513, 1023, 1025]


@pytest.fixture(scope="module", autouse=True)
def lib():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()


def _planted(H, L, most, seed):
    """Positions that fill tiles (8^3 cells) of the grid with the EDGES counts in turn, up to `most` particles."""
    rng = np.random.default_rng(seed)
    nt = max(1, H // 8)
    edge = L / nt
    X, total = [], 0
    for i, t in enumerate(rng.permutation(nt ** 3)):
        c = EDGES[i % len(EDGES)]
        if total + c > most:
            break
        # storage tile t covers node indices [8 t, 8 t + 8); fold its coordinates into the box
        corner = np.array([t // (nt * nt), (t // nt) % nt, t % nt]) * edge
        X.append(O.wrap(corner + edge * rng.uniform(1e-3, 1.0 - 1e-3, size=(c, 3)), L))
        total += c
    return np.concatenate(X)


@pytest.mark.parametrize("fixed", [0, 1])
@pytest.mark.parametrize("precision", [32, 64])
@pytest.mark.parametrize("H,most", [(16, 300), (16, 5000), (32, 4000), (64, 60_000), (64, 120_000), (128, 700_000)])
def test_items_deposit_and_keep_every_particle(H, most, precision, fixed):
    L, M0 = 1.0, 3.0
    X0 = _planted(H, L, most, seed=H + most)
    if H == 16:   # one tile: repeat it until the run takes several items
        X0 = np.concatenate([_planted(H, L, most, seed=s) for s in range(3)])
    P = X0.shape[0]
    p = make_params(P, H, L=L, mass=M0, chi=0.5, mu=0.5, dt=1e-4, seed=11, precision=precision, deposit_mode=fixed)
    po = O.Params(P=P, H=H, L=L, mass=M0, chi=0.5, mu=0.5, eps=1.0, k=1.0, dt=1e-4, seed=11)
    h3 = (L / H) ** 3
    with Simulation(p, X0) as sim:
        for n in range(3):
            X = sim.positions()
            assert np.all(np.isfinite(X))
            got = sim.density(False) * h3
            if precision == 32:
                _check_deposit(got, X, po)
            else:
                ref = O.deposit(X, M0 / P, H, L, 4)
                assert np.max(np.abs(got - ref)) <= (1e-11 if fixed else 1e-12) * np.max(np.abs(ref))
            sim.step(1)
            sim.sync()
