"""What lbm_autotune leaves behind when it fails."""
import ctypes

import pytest

import paper_2010_01847_gb300 as plbm

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)


class _PoolProps(ctypes.Structure):            # CUmemPoolProps
    _fields_ = [("alloc_type", ctypes.c_int), ("handle_types", ctypes.c_int),
                ("location_type", ctypes.c_int), ("location_id", ctypes.c_int),
                ("security", ctypes.c_void_p), ("max_size", ctypes.c_size_t),
                ("usage", ctypes.c_ushort), ("reserved", ctypes.c_ubyte * 54)]


@pytest.fixture
def small_pool():
    """The device's stream-ordered allocations from a pool of 32 MB."""
    cu = ctypes.CDLL("libcuda.so.1")
    torch.zeros(1, device="cuda")
    old, pool = ctypes.c_void_p(), ctypes.c_void_p()
    assert cu.cuDeviceGetMemPool(ctypes.byref(old), 0) == 0
    props = _PoolProps(alloc_type=1, location_type=1, location_id=0, max_size=32 << 20)
    assert cu.cuMemPoolCreate(ctypes.byref(pool), ctypes.byref(props)) == 0
    assert cu.cuDeviceSetMemPool(0, pool) == 0
    yield
    torch.cuda.synchronize()
    assert cu.cuDeviceSetMemPool(0, old) == 0
    assert cu.cuMemPoolDestroy(pool) == 0


@pytest.mark.parametrize("kernel", ["vector", "scalar", "auto"])
def test_failing_for_memory_keeps_the_kernel(small_pool, kernel):
    nx, ny = 1024, 1024                       # 64 MB to keep aside
    lat = plbm.Lattice(nx, ny, 0.9, 12.0, kernel=kernel)
    lat.init(torch.ones((ny, nx), dtype=torch.float64, device="cuda"))

    def launches():
        before = lat.kernel_launches
        lat.step(41)
        return lat.kernel_launches - before

    want = launches()
    name = lat.kernel
    with pytest.raises(plbm.LBMError) as ex:
        lat.autotune(4)
    assert ex.value.status == plbm.ENOMEM
    assert lat.kernel == name and launches() == want
