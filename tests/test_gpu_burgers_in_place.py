"""Stateless FP64 Burgers forecasts where there is no room for their scratch: the
device's memory pool is replaced by one that is smaller than the scratch.  Grids
of one CTA, and of clusters."""
import ctypes
import math

import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2012_10091_gb300 import mgenkf
    return mgenkf


class _PoolProps(ctypes.Structure):
    # CUmemPoolProps: allocation type, handle types, location (type, id), security
    # attributes, largest size, usage, reserved
    _fields_ = [("alloc", ctypes.c_int), ("handles", ctypes.c_int), ("loc", ctypes.c_int), ("dev", ctypes.c_int),
                ("sec", ctypes.c_void_p), ("max_size", ctypes.c_size_t), ("usage", ctypes.c_ushort),
                ("reserved", ctypes.c_ubyte * 54)]


@pytest.fixture
def small_pool(M):
    import torch
    torch.zeros(1, device="cuda")  # the device's context
    cu = ctypes.CDLL("libcuda.so.1")
    before, pool = ctypes.c_void_p(), ctypes.c_void_p()
    props = _PoolProps(alloc=1, loc=1, dev=0, max_size=2 << 20)
    assert cu.cuDeviceGetMemPool(ctypes.byref(before), 0) == 0
    assert cu.cuMemPoolCreate(ctypes.byref(pool), ctypes.byref(props)) == 0
    assert cu.cuDeviceSetMemPool(0, pool) == 0
    yield
    torch.cuda.synchronize()
    assert cu.cuDeviceSetMemPool(0, before) == 0
    assert cu.cuMemPoolDestroy(pool) == 0


@pytest.mark.parametrize("n,grids", [(4093, 2048), (16384, 512)])
def test_forecast_without_scratch_matches_oracle(M, small_pool, n, grids):
    import torch
    steps, nu, L = 5, 0.01, 2 * math.pi
    dt = 0.3 * (L / n) ** 2 / nu
    x = np.arange(n) / n
    u0 = np.sin(L * x + np.arange(grids)[:, None]) + 0.3
    u = torch.tensor(u0, device="cuda")
    M.mgk_forecast(M.MGENKF_BURGERS1D, M.MGENKF_FP64, u, grids, n, L, dt, nu, nsteps=steps)
    torch.cuda.synchronize()
    ref = O.burgers_rk3(u0, L / n, nu, dt, steps)
    # one rounding of 2^-53 per stage and point over 5 steps: far below 1e-12
    assert np.max(np.abs(u.cpu().numpy() - ref)) <= 1e-12 * np.max(np.abs(ref))
