"""Batches of H = 256 runs: the pencil passes that hand on two spectra (G_x and
Phi alpha, from which the inverse y pass or the cluster kernels form G_y and G_z), for
several runs, every tile the tuner may choose and both precisions: the same bits as
the default shapes and as each run in a context of its own."""
import numpy as np
import pytest

from paper_2512_03452_gb300 import DEPOSIT_DETERMINISTIC, Batch, Simulation, _abi, build, make_params

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

STEPS = 18   # past a capacity rebuild


@pytest.fixture(scope="module", autouse=True)
def lib():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()


def _runs(precision):
    rng = np.random.default_rng(7)
    par, X = [], []
    for i, P in enumerate((3000, 777)):
        par.append(make_params(P, 256, L=1.0 + i, mass=8.0, chi=1.0, mu=1.0, dt=1e-4, seed=i, precision=precision,
                               deposit_mode=DEPOSIT_DETERMINISTIC))
        X.append(rng.normal(size=(P, 3)) * 0.1)
    return par, X


def _tuning(**shape):
    t = _abi.sipf_batch_tuning()
    t.ngroups = 1
    t.H[0] = 256
    t.plane_kernels[0] = 1
    for k, v in shape.items():
        getattr(t, k)[0] = v
    return t


def _advance(par, X, tuning=None):
    with Batch(par, X) as b:
        if tuning is not None:
            _abi.sipf_batch_set_tuning(b.handle, tuning)
        b.step(STEPS)
        b.sync()
        return [(b.positions(r), b.spectrum(r)) for r in range(len(par))]


@pytest.mark.parametrize("precision", [32, 64])
def test_shapes_and_single_runs_give_the_same_bits(precision):
    par, X = _runs(precision)
    ref = []
    for p, x in zip(par, X):
        with Simulation(p, x) as sim:
            sim.step(STEPS)
            sim.sync()
            ref.append((sim.positions(), sim.spectrum()))
    shapes = [None, dict(cols_tile=8), dict(xpass_tile=4), dict(plane_kernels=2)]
    if precision == 32:
        shapes += [dict(cols_tile=32), dict(xpass_tile=16, xpass_warps=16), dict(plane_kernels=2, plane_warps=16),
                   dict(rows_blocks_per_sm=4)]
    for shape in shapes:
        got = _advance(par, X, None if shape is None else _tuning(**shape))
        for r in range(len(par)):
            assert np.array_equal(got[r][0], ref[r][0]), (shape, r)
            assert np.array_equal(got[r][1], ref[r][1]), (shape, r)


def test_tuner_returns_documented_shapes_that_can_be_set():
    par, X = _runs(32)
    with Batch(par, X) as b:
        t = _abi.sipf_batch_autotune(b.handle, 2)
        assert t.ngroups == 1 and t.xpass_warps[0] in (0, 8, 16) and t.plane_warps[0] in (8, 16, 32)
        assert t.cols_tile[0] in (8, 16, 32) and t.xpass_tile[0] in (4, 8, 16)
        assert t.rows_blocks_per_sm[0] == 8   # the default: it has no effect here and is not searched
        _abi.sipf_batch_set_tuning(b.handle, t)
