"""The stateless deposit and gather take grids at any alignment of their element
type: vector paths (16-byte aligned grids) and scalar paths agree to the sums'
rounding, at every offset of a particle's first z layer in its quad and across the
periodic edge."""
import numpy as np
import pytest

from oracle import sipf_oracle as O
from paper_2512_03452_gb300 import _abi, build

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("H", [8, 64])
def test_deposit_and_gather_any_alignment(H, order):
    build.build()
    L, P = 1.0, 4 * H + 3
    rng = np.random.default_rng(H + order)
    X = rng.uniform(-L / 2, L / 2, size=(P, 3))
    X[:H, 2] = (np.arange(H) - H // 2 + 0.25) * (L / H)     # every z cell, the first and last among them
    X = X.astype(np.float32).astype(np.float64)
    t = torch.tensor(np.ascontiguousarray(X.T), dtype=torch.float32, device="cuda")
    xyz = [t[d].data_ptr() for d in range(3)]
    ref = O.deposit(X, 1.0, H, L, order).ravel()
    f = np.random.default_rng(1).normal(size=(2, H, H, H)).astype(np.float32)
    gref = O.gather(f.astype(np.float64), X, H, L, order)
    for off in (0, 1, 2, 3):
        buf = torch.full((H ** 3 + 4,), 9.0, dtype=torch.float32, device="cuda")
        _abi.sipf_deposit_dev(32, *xyz, P, H, L, 1.0, order, buf[off:].data_ptr())
        torch.cuda.synchronize()
        got = buf.cpu().numpy()
        assert np.all(got[:off] == 9.0) and np.all(got[off + H ** 3:] == 9.0)
        assert np.max(np.abs(got[off:off + H ** 3] - ref)) <= 1e-5 * np.max(np.abs(ref))
        fb = torch.empty(2 * H ** 3 + 4, dtype=torch.float32, device="cuda")
        fb[off:off + 2 * H ** 3] = torch.tensor(f.ravel(), device="cuda")
        out = torch.empty((2, P), dtype=torch.float32, device="cuda")
        _abi.sipf_gather_dev(32, *xyz, P, H, L, fb[off:].data_ptr(), 2, order, out.data_ptr())
        torch.cuda.synchronize()
        assert np.max(np.abs(out.cpu().numpy() - gref)) <= 1e-4 * np.max(np.abs(gref))
