"""Leaves of the sigma-basis whose CTAs wait for operations that never come: the
call ends with FFSPMV_ERR_TIMEOUT in bounded time, from a single leaf, from the
part of the recursion that runs without the host and from the part that does
not, and the next call is right."""
import ctypes
import time

import numpy as np
import pytest

from oracle import sigma

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,m,n,d,hold", [(65521, 8, 4, 20, 0), (65521, 32, 16, 32, 5), (2**31 - 1, 5, 5, 24, 22), (2, 27, 16, 32, 31),
                                          (65521, 20, 17, 24, 3), (65521, 4, 2, 40, 1), (65521, 3, 2, 450, 2)])
def test_operations_that_never_come(lib, p, m, n, d, hold):
    import torch
    rng = np.random.default_rng(d + hold)
    F = rng.integers(0, p, (d, m, n))
    f = torch.from_numpy(np.ascontiguousarray(F, dtype=np.uint32).view(np.int32)).cuda()
    need = ctypes.c_int64()
    L = lib.lib()
    assert L.sigma_basis_workspace(m, n, d, 0, ctypes.byref(need)) == 0
    work = torch.empty(need.value, dtype=torch.uint8, device="cuda")
    P = torch.empty((d + 1, m, m), dtype=torch.int32, device="cuda")
    delta = np.zeros(m, dtype=np.int32)
    args = (p, m, n, d, 0, f.data_ptr(), None, P.data_ptr(), delta.ctypes.data, None, work.data_ptr(), need.value)
    torch.cuda.synchronize()
    t = time.perf_counter()
    assert L.ffspmv_sigma_basis_hold(*args, hold, lib.stream_ptr()) == 6
    assert time.perf_counter() - t < 2.0
    assert L.sigma_basis(*args, lib.stream_ptr()) == 0
    Po, do = sigma.pmbasis(F.astype(object), d, [0] * m, p, base=8)
    want = np.zeros((d + 1, m, m), dtype=np.int64)
    want[:Po.shape[0]] = np.asarray(Po, dtype=np.int64)
    assert list(delta) == do and np.array_equal(P.cpu().numpy().view(np.uint32).astype(np.int64), want)
