"""An error that the caller has pending with the CUDA runtime is reported by the
calls that prepare and step in one, and by nothing else (needs a GPU)."""
import ctypes

import pytest

from paper_2008_11578_gb300 import api, scenes

pytestmark = pytest.mark.gpu

ORCA_ERR_CUDA = 2


@pytest.mark.parametrize("n", [100, 3000, 21000])
@pytest.mark.parametrize("call", ["noalloc", "capture"])
def test_pending_error_is_reported(call, n):
    rt = ctypes.CDLL("libcudart.so.13")
    ds = api.DeviceScene(scenes.open_square(n, (n / 0.4) ** 0.5, seed=109))

    def status():
        if call == "noalloc":
            return api.orca_step_noalloc(ds.params, ds._agents, 1, synchronize=True)
        try:
            ds.capture(1)
        except api.OrcaError as e:
            return e.status
        return 0

    assert status() == 0
    rt.cudaGetLastError()
    assert rt.cudaSetDevice(9999) != 0     # refused on the host: no such device
    got = status()
    rt.cudaGetLastError()
    assert got == ORCA_ERR_CUDA
    assert status() == 0
    ds.close()
