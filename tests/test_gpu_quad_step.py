"""The float step on rows in the quad layout against the oracle, for every
angle count the layout takes (1 to 4 quads a thread, with and without a tail
pair), equal and unequal weights, static and moving mesh, a ragged last block,
boundary and emitter cells, and cells so cold that the temperature solve
leaves its float range and takes the double one.

Tolerances as for the other float tests: 1e-5 in L1 of E_r.  The gas energy
moves by the exchange alone, so its error is a float error of the exchanged
energy: 1e-5 of the energy density of gas and radiation together."""
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


def _problem(A, equal, w):
    rng = np.random.default_rng(A)
    p = make(n=(5, 6, 7), order=2, w=w, seed=4)
    up = rng.normal(size=(A // 2, 3))
    up /= np.linalg.norm(up, axis=1, keepdims=True)
    p.dirs = np.ascontiguousarray(np.concatenate([up, -up]))
    wt = np.ones(A) if equal else rng.uniform(0.5, 1.5, A)
    p.weights = wt / wt.sum()
    p.q0, p.I0 = np.ones(A), np.zeros((1, A))
    p = randomise(p, seed=A)
    cold = np.nonzero(p.kind == 0)[0][::5]  # transparent cells of cold gas at rest
    p.kappa_P[cold] = p.kappa_J[cold] = p.kappa_s[cold] = 0.0
    p.m[cold] = 0.0
    p.e[cold] = 1e-27
    return p, cold


@pytest.mark.parametrize("float_quartic", [0, 1])
@pytest.mark.parametrize("w", [None, (0.4, -0.2, 0.1)])
@pytest.mark.parametrize("A", [32, 48, 64, 80, 96, 112, 128])
def test_quad_step_matches_oracle(A, w, float_quartic):
    from paper_2002_08377_gb300.solver import RTSolver
    p, cold = _problem(A, A % 32 == 0, w)
    o = oracle.Oracle(p)
    dt = 0.5 / o.positivity()
    g = RTSolver.from_problem(p, "fp32", float_quartic=float_quartic)
    assert o.run(4, dt) == oracle.ORC_OK
    g.run(4, dt)
    E_o = o.moments()[0]
    E_g = g.moments()[0]
    assert np.abs(E_g - E_o).sum() < 1e-5 * np.abs(E_o).sum()
    I = g.get_intensity()[cold]
    assert np.abs(I - o.I[cold]).max() < 1e-5 * np.abs(o.I[cold]).max()
    e, m, ext = g.gas()
    scale = np.abs(o.e) + E_o
    assert np.abs(e - o.e).max() < 1e-5 * scale.max()
    assert np.abs(m - o.m).max() < 1e-5 * (np.abs(o.m).max() + E_o.max() / p.cbar)
    assert np.abs(ext - o.ext).max() < 1e-5 * scale.max()
    g.close()
