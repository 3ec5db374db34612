"""A set-up that ends with an error gives all its device memory back, its temporaries included."""
import ctypes

import pytest

from paper_2308_11371_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

USED_MEM_CURRENT = 7        # CU_MEMPOOL_ATTR_USED_MEM_CURRENT


def _pool_bytes():
    cu = ctypes.CDLL("libcuda.so.1")
    torch.cuda.synchronize()
    pool, used = ctypes.c_void_p(), ctypes.c_uint64()
    assert cu.cuDeviceGetDefaultMemPool(ctypes.byref(pool), torch.cuda.current_device()) == 0
    assert cu.cuMemPoolGetAttribute(pool, USED_MEM_CURRENT, ctypes.byref(used)) == 0
    return used.value


def test_failed_setup_frees_its_temporaries():
    """Mixed cells of 28^2 elements: the combine kernel has no room for their 1,674 remaining DOF, which
    set-up finds out while it holds the principal K_rp and K_pp blocks."""
    from paper_2308_11371_gb300 import binding
    p = W.lattice_2d(2, 1, 28, r=0.12, n_rb=1)
    used = []
    for _ in range(3):
        with pytest.raises(binding.FetidpError) as e:
            binding.Solver(p, precision=binding.FETIDP_MIXED_BF16)
        assert e.value.status == -1 and "combine kernel" in str(e.value)
        used.append(_pool_bytes())
    assert used[0] == used[1] == used[2]
