"""The 2D deposit through shared-memory windows of the grid: particle numbers
around the line where windows are used, and positions over the whole box, so
that rows inside and outside the window take part.  Node by node against the
oracle's deposit of the same positions: at most 12 roundings a weight and n_j
additions, |got - ref| <= w S_j (12 + n_j) u (Higham's bound for the sums)."""
import numpy as np
import pytest

from oracle import sipf2d_oracle as O2
from paper_2512_03452_gb300 import Simulation2D, build, make_params

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()


@pytest.mark.parametrize("precision", [32, 64])
@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("H,P", [(8, 8192), (64, 8191), (64, 8193), (128, 30_001), (256, 8192), (256, 200_003)])
def test_window_deposit_matches_oracle(H, P, order, precision):
    L, M0 = 3.0, 5.0
    X0 = np.random.default_rng(H + P).uniform(-L / 2, L / 2, size=(P, 2))
    p = make_params(P, H, L=L, mass=M0, mu=1.0, dt=1e-3, precision=precision, p2g_order=order)
    with Simulation2D(p, X0) as sim:
        for _ in range(2):
            X = sim.positions()
            got = sim.density() * (L / H) ** 2
            w = M0 / P
            ref = O2.deposit(X, w, H, L, order)
            cell, lam = O2.cell_and_lambda(X, H, L)
            offs, F = O2.stencil2(lam, order)
            idx = O2.stencil_indices(cell, offs, H).ravel()
            n = np.bincount(idx, minlength=H * H).reshape(H, H)
            S = np.bincount(idx, weights=np.abs(F).ravel(), minlength=H * H).reshape(H, H)
            u = 2.0 ** (-24 if precision == 32 else -53)
            # lambda = H x / L - cell is rounded once at a coordinate of up to H / 2
            slack = 4 * (H / 2) * u * w * n
            assert np.all(np.abs(got - ref) <= w * S * (12 + n) * u + slack + 1e-300)
            sim.step(1)
            sim.sync()
