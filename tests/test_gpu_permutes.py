"""Device rows into and out of the internal order, in units of four positions
and by single values, against the host-memory permutes (which go by single
columns): angle counts with and without units, quads and a tail, both
precisions, and caller rows that are not aligned to two values.  Exact."""
import ctypes

import numpy as np
import pytest

from paper_2002_08377_gb300 import build as rtbuild
from paper_2002_08377_gb300 import capi
from tests._problems import make

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    rtbuild.build()
    capi.load()


@pytest.mark.parametrize("offset", [0, 1, 2])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("A", [2, 4, 6, 8, 24, 32, 44, 48, 80, 112])
def test_device_rows_match_host_rows(A, precision, offset):
    import torch
    from paper_2002_08377_gb300.solver import RTSolver
    p = make(n=(5, 6, 7), order=2, seed=4)
    up = np.random.default_rng(A).normal(size=(A // 2, 3))
    up /= np.linalg.norm(up, axis=1, keepdims=True)
    p.dirs = np.ascontiguousarray(np.concatenate([up, -up]))
    p.weights = np.full(A, 1.0 / A)
    p.q0, p.I0 = np.ones(A), np.zeros((1, A))
    s = RTSolver.from_problem(p, precision)
    n = s.N * A
    I = np.random.default_rng(5).random((s.N, A)).astype(s.dtype)
    host = torch.empty((s.N, A), dtype=s.tdtype, pin_memory=True)
    dev = torch.full((n + 4,), -1.0, dtype=s.tdtype, device="cuda")
    view = dev[offset:offset + n]
    p_host, p_dev = ctypes.c_void_p(host.data_ptr()), ctypes.c_void_p(view.data_ptr())
    view.copy_(torch.from_numpy(I).reshape(-1))
    torch.cuda.synchronize()
    s._check(s.lib.rt_set_intensity(s.state, p_dev, 1))
    s._check(s.lib.rt_get_intensity(s.state, p_host, 0))
    assert np.array_equal(host.numpy(), I)
    host.numpy()[:] = I[::-1]
    s._check(s.lib.rt_set_intensity(s.state, p_host, 0))
    view.fill_(0.0)
    torch.cuda.synchronize()
    s._check(s.lib.rt_get_intensity(s.state, p_dev, 1))
    torch.cuda.synchronize()
    assert np.array_equal(view.cpu().numpy().reshape(s.N, A), I[::-1])
    rest = torch.cat([dev[:offset], dev[offset + n:]])
    assert bool((rest == -1.0).all())
    s.close()
