"""The float step kernels' rarer branches against the oracle: volumes that follow the
faces, power-law opacities and the plain float temperature root (float_quartic = 1),
on the kernel with two threads per cell (8 angles), the tile kernel (24, 72 and 104)
and the quad kernel (48), each on a mesh with a ragged last block below and above the
quad kernel's line for small meshes (9728 cells).

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


@pytest.mark.parametrize("float_quartic", [0, 1])
@pytest.mark.parametrize("mode", ["plain", "power_law", "gcl"])
@pytest.mark.parametrize("n", [(7, 6, 5), (21, 23, 22)])
@pytest.mark.parametrize("A", [8, 24, 48, 72, 104])
def test_branches_match_oracle(A, n, mode, float_quartic):
    from paper_2002_08377_gb300.solver import RTSolver
    rng = np.random.default_rng(A)
    p = make(n=n, order=2, cbar=10.0, c=100.0, seed=4)
    up = rng.normal(size=(A // 2, 3))
    up /= np.linalg.norm(up, axis=1, keepdims=True)
    p.dirs = np.ascontiguousarray(np.concatenate([up, -up]))
    wt = rng.uniform(0.5, 1.5, A)
    p.weights = wt / wt.sum()
    p.q0, p.I0 = np.ones(A), np.zeros((1, A))
    if mode == "gcl":
        m = p.mesh
        r = m.points - 0.5 * m.box
        m.face_w = m.face_velocity(np.cross([0.4, -0.7, 0.9], r) + 0.15 * r)
        p.gcl = 1
    p = randomise(p, seed=A)
    if mode == "power_law":
        p.beta_P, p.beta_J, p.T_ref = 2.0, -1.0, 1.3
    o = oracle.Oracle(p)
    dt = 0.5 / o.positivity()
    g = RTSolver.from_problem(p, "fp32", float_quartic=float_quartic)
    assert o.run(3, dt) == oracle.ORC_OK
    g.run(3, dt)
    E_o = o.moments()[0]
    assert np.abs(g.moments()[0] - E_o).sum() < 1e-5 * np.abs(E_o).sum()
    e, m, ext = g.gas()
    scale = (np.abs(o.e) + E_o).max()
    assert np.abs(e - o.e).max() < 1e-5 * scale
    assert np.abs(m - o.m).max() < 1e-5 * (np.abs(o.m).max() + E_o.max() / p.cbar)
    assert np.abs(ext - o.ext).max() < 1e-5 * scale
    g.close()
