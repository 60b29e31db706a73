"""A batch that the device has memory for with one cell to an SM runs (GPU).

From two cells an SM on, large networks run two CTAs on an SM with a workspace
each. Where the allocator has no room for that, the launch takes one cell to an
SM. The test gives the stream-ordered allocator a pool with a maximum size (a
few hundred MB; the device's memory is not filled).
"""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2511_10558_gb300 import build as _build  # noqa: E402

_build.build()
from paper_2511_10558_gb300 import carbox, synth  # noqa: E402

YR = synth.YEAR


class _PoolProps(ctypes.Structure):  # cudaMemPoolProps
    _fields_ = [("alloc_type", ctypes.c_int), ("handle_types", ctypes.c_int), ("location_type", ctypes.c_int),
                ("location_id", ctypes.c_int), ("security", ctypes.c_void_p), ("max_size", ctypes.c_size_t),
                ("usage", ctypes.c_ushort), ("reserved", ctypes.c_ubyte * 54)]


class _Pool:
    """The current pool of device 0, limited to max_size bytes."""

    def __init__(self, max_size):
        with open("/proc/self/maps") as f:
            self.rt = ctypes.CDLL(next(line.split()[-1] for line in f if "libcudart.so" in line))
        self.old, self.pool = ctypes.c_void_p(), ctypes.c_void_p()
        props = _PoolProps(alloc_type=1, location_type=1, location_id=0, max_size=max_size)  # pinned, on a device
        assert self.rt.cudaDeviceGetMemPool(ctypes.byref(self.old), 0) == 0
        assert self.rt.cudaMemPoolCreate(ctypes.byref(self.pool), ctypes.byref(props)) == 0

    def __enter__(self):
        assert self.rt.cudaDeviceSetMemPool(0, self.pool) == 0

    def __exit__(self, *exc):
        torch.cuda.synchronize()
        assert self.rt.cudaDeviceSetMemPool(0, self.old) == 0
        assert self.rt.cudaMemPoolDestroy(self.pool) == 0


@pytest.mark.parametrize("method", [carbox.CBX_METHOD_BDF, carbox.CBX_METHOD_ESDIRK])
def test_one_cell_to_an_sm_where_two_have_no_memory(method):
    net = synth.make_network(500, 6000)
    N = carbox.Network.from_synth(net)
    dev = torch.device("cuda:0")
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    C = 4 * sms + 7
    phi = torch.tensor(synth.cells(C, seed=8), device=dev)
    x0 = torch.tensor(np.repeat(synth.initial_abundances(net)[:, None], C, axis=1), device=dev).contiguous()
    opt = carbox.options(precision=carbox.CBX_MIXED, method=method)
    want, st, _ = carbox.solve(N, phi, x0, 0.0, 1e5, opt)
    torch.cuda.synchronize()
    cta = 4 * 500 * 500 + 8 * (3 * 6000 + N.info()["nnz_jac"])  # the matrix in FP32, rates and Jacobian
    assert 1.1 * sms * cta < 300 << 20 < 2 * sms * cta  # the premise: one to an SM fits, two do not
    with _Pool(300 << 20):
        x, s, _ = carbox.solve(N, phi, x0, 0.0, 1e5, opt)
        torch.cuda.synchronize()
    assert torch.equal(s, st) and torch.equal(x, want)
    pool = _Pool(64 << 20)  # not even one cell to an SM
    with pool:
        with pytest.raises(carbox.CarboxError) as e:
            carbox.solve(N, phi, x0, 0.0, 1e5, opt)
        pool.rt.cudaGetLastError()  # (PyTorch would report it at its next launch)
    assert e.value.code == carbox.CBX_E_CUDA
