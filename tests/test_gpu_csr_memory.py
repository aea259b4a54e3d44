"""The device arrays of a sparse system (lb_csr_arrays; needs an sm_103a GPU)
are ordinary device memory: other devices can be given access to them and other
processes a handle, which memory of a private pool allows neither."""
import ctypes

import pytest

import workloads as wl

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

IPC_CAPABLE, MEMPOOL = 10, 17  # CU_POINTER_ATTRIBUTE_IS_LEGACY_CUDA_IPC_CAPABLE, _MEMPOOL_HANDLE


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1912_01491_gb300 import build
    build.build()


@pytest.mark.parametrize("N", [3, 30, 200])
def test_arrays_are_ordinary_device_memory(N):
    import paper_1912_01491_gb300 as lb
    cu = ctypes.CDLL("libcuda.so.1")
    cu.cuPointerGetAttribute.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_uint64]
    H, L, g = wl.ladder_model(N, 1)
    with lb.Basis(N) as B:
        l = B.expand(torch.tensor(L, device="cuda"))
        nz = torch.nonzero(l.abs() > 0).flatten()
        c = lb.Csr(B, h=B.expand(torch.tensor(H, device="cuda")).real.contiguous(),
                   channels=[(g, nz, l[nz].contiguous())])
        p = [ctypes.c_void_p() for _ in range(4)]
        assert lb.native.load().lb_csr_arrays(c._h, *[ctypes.byref(x) for x in p]) == 0
        for x in p:
            ipc, pool = ctypes.c_uint(0), ctypes.c_void_p()
            assert cu.cuPointerGetAttribute(ctypes.byref(ipc), IPC_CAPABLE, x.value) == 0
            assert cu.cuPointerGetAttribute(ctypes.byref(pool), MEMPOOL, x.value) == 0
            assert ipc.value & 0xff == 1 and not pool.value
        c.close()
