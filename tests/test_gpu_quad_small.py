"""The float step on quad rows on both sides of its line for small meshes (at
most two blocks of 32 cells per SM: 9728 cells) against the oracle: one to four
quads a thread, with and without a tail pair, static and moving mesh, the last
block full and ragged.  Smaller meshes reach the same path in
test_gpu_quad_step.py.

Tolerances as for the other float tests: 1e-5 in L1 of E_r, and of the energy
density of gas and radiation together for the gas."""
import numpy as np
import pytest

import oracle
from paper_2002_08377_gb300 import build as rtbuild
from paper_2002_08377_gb300 import capi
from tests._problems import make, randomise

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    rtbuild.build()
    capi.load()


@pytest.mark.parametrize("n", [(16, 16, 38), (17, 19, 31)])
@pytest.mark.parametrize("w", [None, (0.4, -0.2, 0.1)])
@pytest.mark.parametrize("A", [32, 48, 80, 128])
def test_quad_step_small_and_large(A, w, n):
    from paper_2002_08377_gb300.solver import RTSolver
    rng = np.random.default_rng(A)
    p = make(n=n, order=2, w=w, seed=4)
    up = rng.normal(size=(A // 2, 3))
    up /= np.linalg.norm(up, axis=1, keepdims=True)
    p.dirs = np.ascontiguousarray(np.concatenate([up, -up]))
    wt = rng.uniform(0.5, 1.5, A)
    p.weights = wt / wt.sum()
    p.q0, p.I0 = np.ones(A), np.zeros((1, A))
    p = randomise(p, seed=A)
    o = oracle.Oracle(p)
    dt = 0.5 / o.positivity()
    g = RTSolver.from_problem(p, "fp32")
    assert o.run(2, dt) == oracle.ORC_OK
    g.run(2, dt)
    E_o = o.moments()[0]
    assert np.abs(g.moments()[0] - E_o).sum() < 1e-5 * np.abs(E_o).sum()
    e = g.gas()[0]
    scale = (np.abs(o.e) + E_o).max()
    assert np.abs(e - o.e).max() < 1e-5 * scale
    g.close()
