"""The limited gradients of the double van Leer step where intensities fall to the
smallest doubles, as they do ahead of a front in the dark: the Barth-Jespersen
quotients then have subnormal divisors, whose reciprocals are not finite.

Transparent cells, a few of them lit: the step is homogeneous in the intensity,
so parity with the oracle is relative to the largest one.  Tolerance 1e-6: a
subnormal rounds to 5e-324, 5e-14 of the smallest scale here, and the gradient
coefficients amplify that by less than 1e6; a face value left unlimited is off by
1e-2."""
import numpy as np
import pytest

import oracle
from paper_2002_08377_gb300 import build as rtbuild
from paper_2002_08377_gb300 import capi
from tests._problems import make

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    rtbuild.build()
    capi.load()


@pytest.mark.parametrize("scale", [1e-300, 1e-307, 1e-308, 1e-310])
@pytest.mark.parametrize("order", [2, 6, 8])
def test_subnormal_intensities(order, scale):
    from paper_2002_08377_gb300.solver import RTSolver
    p = make(n=(6, 5, 7), order=order, kP=0.0, kJ=0.0, kS=0.0, seed=2)
    rng = np.random.default_rng(order)
    lit = rng.uniform(size=(p.n_cells, 1)) < 0.2
    I = scale * lit * rng.uniform(0.2, 1.0, (p.n_cells, p.n_angles))
    p.initial_intensity = lambda dtype=np.float64: np.ascontiguousarray(I.astype(dtype))
    p.integrator = capi.RT_VAN_LEER
    o = oracle.Oracle(p)
    dt = 0.25 / o.positivity()
    g = RTSolver.from_problem(p, "fp64")
    assert o.run(1, dt) == oracle.ORC_OK
    g.run(1, dt)
    assert np.abs(g.get_intensity() - o.I).max() < 1e-6 * np.abs(o.I).max()
    g.close()
