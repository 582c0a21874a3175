"""FP64 noise over many counters against the oracle's normals.  |z| <= sqrt(66 ln 2)
< 6.8; the logarithm is within 1.4, its root, the sine or cosine and the product
within 3 units of 2^-52, and the oracle rounds its angle of up to 2 pi (4 units):
8.4 x 6.8 x 2^-52 < 1.3e-14."""
import numpy as np
import pytest

from oracle import sipf_oracle as O
from paper_2512_03452_gb300 import _abi, build

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seed,step,first,P", [(0, 1, 0, 1), (3, 7, 5, 300_001), ((1 << 40) + 9, 2 ** 31, 2 ** 29, 300_000)])
def test_noise64_matches_oracle(seed, step, first, P):
    build.build()
    z = torch.empty((6, P), dtype=torch.float64, device="cuda")
    _abi.sipf_noise_dev(64, seed, step, first, P, z.data_ptr())
    torch.cuda.synchronize()
    ref = O.normals(seed, step, P, first=first).T
    assert np.max(np.abs(z.cpu().numpy() - ref)) < 1.3e-14
