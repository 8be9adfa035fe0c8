"""The float step on quad rows with every kind of last block: 1 to 31 cells of 32,
so that whole warps (four cells each) and single lanes of it lie past the mesh.
Meshes on both sides of the line for small ones (9728 cells); constant and
power-law opacities, whose temperature solve runs between block barriers; static
mesh and one whose volumes follow its faces.

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


@pytest.mark.parametrize("mode", ["static", "power_law", "gcl"])
@pytest.mark.parametrize("n,tail", [((5, 5, 9), 1), ((5, 5, 4), 4), ((5, 5, 13), 5),
                                    ((5, 5, 16), 16), ((5, 5, 20), 20), ((5, 5, 12), 12),
                                    ((5, 5, 7), 15), ((25, 25, 17), 1), ((25, 25, 20), 20),
                                    ((25, 25, 31), 15)])
def test_ragged_last_block(n, tail, mode):
    from paper_2002_08377_gb300.solver import RTSolver
    assert np.prod(n) % 32 == tail
    p = make(n=n, order=8, cbar=10.0, c=100.0, seed=4)
    if mode == "gcl":
        m = p.mesh
        gen = m.points - 0.5 * m.box
        m.face_w = m.face_velocity(np.cross([0.4, -0.7, 0.9], gen) + 0.15 * gen)
        p.gcl = 1
    p = randomise(p, seed=5)
    if mode == "power_law":
        p.beta_P, p.beta_J, p.T_ref = 2.0, -1.0, 1.3
    o = oracle.Oracle(p)
    dt = 0.5 / o.positivity()
    g = RTSolver.from_problem(p, "fp32")
    assert o.run(3, dt) == oracle.ORC_OK
    g.run(3, dt)
    E_o = o.moments()[0]
    assert np.abs(g.moments()[0] - E_o).sum() < 1e-5 * np.abs(E_o).sum()
    e = g.gas()[0]
    assert np.abs(e - o.e).max() < 1e-5 * (np.abs(o.e) + E_o).max()
    g.close()
