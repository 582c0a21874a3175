"""The stateless transforms allocate nothing, whatever the spectrum's alignment: the
device's stream-ordered memory pool stays untouched."""
import ctypes

import pytest

from paper_2512_03452_gb300 import _abi, build

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

USED_MEM_HIGH = 8   # CU_MEMPOOL_ATTR_USED_MEM_HIGH


def _pool():
    cuda = ctypes.CDLL("libcuda.so.1")
    pool = ctypes.c_void_p()
    assert cuda.cuDeviceGetDefaultMemPool(ctypes.byref(pool), torch.cuda.current_device()) == 0
    return cuda, pool


@pytest.mark.parametrize("H", [16, 64, 256])
@pytest.mark.parametrize("precision", [32, 64])
def test_transforms_leave_the_pool_alone(H, precision):
    build.build()
    T = torch.float64 if precision == 64 else torch.float32
    n = H * H * (H // 2 + 1) * 2
    grid = torch.randn(H ** 3, dtype=T, device="cuda")
    buf = torch.zeros(n + 2, dtype=T, device="cuda")
    torch.cuda.synchronize()
    cuda, pool = _pool()
    value = ctypes.c_uint64(0)
    assert cuda.cuMemPoolSetAttribute(pool, USED_MEM_HIGH, ctypes.byref(value)) == 0
    for off in (0, 1):
        spec = buf[off:off + n]
        _abi.sipf_forward_ft_dev(precision, H, 1.0, grid.data_ptr(), spec.data_ptr())
        _abi.sipf_inverse_ft_dev(precision, H, spec.data_ptr(), grid.data_ptr())
    torch.cuda.synchronize()
    assert cuda.cuMemPoolGetAttribute(pool, USED_MEM_HIGH, ctypes.byref(value)) == 0
    assert value.value == 0
