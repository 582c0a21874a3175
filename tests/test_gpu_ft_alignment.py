"""Transforms of spectra at any alignment of their elements' parts: a spectrum that
is only aligned to its real type gives the same bits as an aligned one, and the
memory around it is left alone."""
import pytest

from paper_2512_03452_gb300 import _abi, build

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H", [8, 32, 64])
@pytest.mark.parametrize("precision", [32, 64])
def test_unaligned_spectrum_same_bits(H, precision):
    build.build()
    T = torch.float64 if precision == 64 else torch.float32
    n = H * H * (H // 2 + 1) * 2
    g = torch.randn(H ** 3, dtype=T, device="cuda", generator=torch.Generator("cuda").manual_seed(H))
    res = []
    for off in (0, 1):
        buf = torch.full((n + 2,), 7.0, dtype=T, device="cuda")
        spec = buf[off:off + n]
        _abi.sipf_forward_ft_dev(precision, H, 1.5, g.data_ptr(), spec.data_ptr())
        torch.cuda.synchronize()
        fwd = spec.clone()
        out = torch.empty(H ** 3, dtype=T, device="cuda")
        _abi.sipf_inverse_ft_dev(precision, H, spec.data_ptr(), out.data_ptr())
        torch.cuda.synchronize()
        assert torch.all(buf[:off] == 7.0) and torch.all(buf[off + n:] == 7.0)
        res.append((fwd, out, spec.clone()))
    assert all(torch.equal(a, b) for a, b in zip(*res))
