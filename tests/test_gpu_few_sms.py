"""Cooperative runs on a stream that has a few of the device's SMs (a green context): the same steps and solves as on all
of them."""
import ctypes as ct

import numpy as np
import pytest

from tests.test_gpu_poisson import _gpu_solve, _periodic_problem
from tests.test_gpu_sliced import EPS

pytestmark = pytest.mark.gpu


@pytest.fixture
def small_stream():
    """A stream on at least 8 SMs, by the driver's calls (CUdevResource: 144 bytes)."""
    import torch

    torch.cuda.init()
    torch.zeros(1, device="cuda")
    cu = ct.CDLL("libcuda.so.1")
    if not hasattr(cu, "cuGreenCtxStreamCreate"):
        pytest.skip("the driver has no green contexts")
    device, part, rest = (ct.create_string_buffer(144) for _ in range(3))
    groups, desc, green, stream = ct.c_uint(1), ct.c_void_p(), ct.c_void_p(), ct.c_void_p()
    calls = [lambda: cu.cuDeviceGetDevResource(ct.c_int(0), device, ct.c_int(1)),
             lambda: cu.cuDevSmResourceSplitByCount(part, ct.byref(groups), device, rest, ct.c_uint(0), ct.c_uint(8)),
             lambda: cu.cuDevResourceGenerateDesc(ct.byref(desc), part, ct.c_uint(1)),
             lambda: cu.cuGreenCtxCreate(ct.byref(green), desc, ct.c_int(0), ct.c_uint(1)),
             lambda: cu.cuGreenCtxStreamCreate(ct.byref(stream), green, ct.c_uint(1), ct.c_int(0))]
    for call in calls:
        if call() != 0:
            pytest.skip("the device gives no green context")
    yield torch.cuda.ExternalStream(stream.value)
    torch.cuda.synchronize()
    cu.cuStreamDestroy_v2(stream)
    cu.cuGreenCtxDestroy(green)


def test_runs_on_a_few_sms(small_stream):
    import torch

    def results():
        ns, L, ex, f, dm = _periodic_problem(4, 97)
        phi, _, resid = _gpu_solve(L, f, dm, tol=1e-10)
        u = torch.from_numpy(ex.copy()).to("cuda")
        L.step([1.0], u, 0.015 * float(ns.h[0]) ** 2, 3)
        torch.cuda.synchronize()
        rp = L.get_neighbours()[0].cpu().numpy()
        L.close()
        return u.cpu().numpy(), phi, resid, int(np.diff(rp).max())

    u, phi, _, size = results()
    with torch.cuda.stream(small_stream):
        u2, phi2, resid, _ = results()
    # twice the bound of one run's rounding: dt sum |w| |u_j - u_i| <= 1 a stage (RK4 is stable to dt |lambda| = 2.8)
    assert np.abs(u2 - u).max() <= 2 * 4 * 3 * (size + 8) * EPS
    assert resid <= 1e-10 and np.abs(phi2 - phi).max() <= 1e-6 * np.abs(phi).max()
