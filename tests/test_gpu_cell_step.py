"""The float step with two threads per cell (at most 8 angles) against the
oracle: 1 to 4 pairs of angles, unequal weights, static and moving mesh, a
ragged last block, boundary and emitter cells, all orders in v/c, cold cells
that take the double temperature solve; and, with 10 angles, the tile kernel
beside it.

Tolerances as for the other float tests: 1e-5 in L1 of E_r and of the energy
density of gas and radiation together."""
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


@pytest.mark.parametrize("n", [(21, 21, 21), (12, 13, 14)])
@pytest.mark.parametrize("w,boost", [(None, 0), ((0.4, -0.2, 0.1), 1)])
@pytest.mark.parametrize("A", [2, 4, 6, 8, 10])
def test_cell_step_matches_oracle(A, w, boost, n):
    from paper_2002_08377_gb300.solver import RTSolver
    rng = np.random.default_rng(A)
    p = make(n=n, order=2, w=w, seed=4)
    up = rng.normal(size=(A // 2, 3))
    up /= np.linalg.norm(up, axis=1, keepdims=True)
    p.dirs = np.ascontiguousarray(np.concatenate([up, -up]))
    wt = rng.uniform(0.5, 1.5, A)
    p.weights = wt / wt.sum()
    p.q0, p.I0 = np.ones(A), np.zeros((1, A))
    p.boost = boost
    p = randomise(p, seed=A)
    cold = np.nonzero(p.kind == 0)[0][::7]  # transparent cells of cold gas at rest
    p.kappa_P[cold] = p.kappa_J[cold] = p.kappa_s[cold] = 0.0
    p.m[cold] = 0.0
    p.e[cold] = 1e-27
    o = oracle.Oracle(p)
    dt = 0.5 / o.positivity()
    g = RTSolver.from_problem(p, "fp32")
    assert o.run(3, dt) == oracle.ORC_OK
    g.run(3, dt)
    E_o = o.moments()[0]
    assert np.abs(g.moments()[0] - E_o).sum() < 1e-5 * np.abs(E_o).sum()
    I = g.get_intensity()[cold]
    assert np.abs(I - o.I[cold]).max() < 1e-5 * np.abs(o.I[cold]).max()
    e, m, ext = g.gas()
    scale = (np.abs(o.e) + E_o).max()
    assert np.abs(e - o.e).max() < 1e-5 * scale
    assert np.abs(m - o.m).max() < 1e-5 * (np.abs(o.m).max() + E_o.max() / p.cbar)
    assert np.abs(ext - o.ext).max() < 1e-5 * scale
    g.close()
