"""newton_max_iter refuses the same steps in both ways a float state can take its
temperature from the float Newton (float_quartic = 0, refined, and 1, as it is):
the refined solve may stop its float Newton early, but must not accept a step for
which the float Newton itself has not converged within the limit.  24 angles take
the tile kernel, 8 the one with two threads per cell, 80 the quad kernel."""
import pytest

from paper_2002_08377_gb300 import build as rtbuild
from paper_2002_08377_gb300 import capi
from tests._problems import make

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    rtbuild.build()
    capi.load()


def _accepts(prob, limit, float_quartic):
    from paper_2002_08377_gb300.solver import RTSolver
    g = RTSolver.from_problem(prob, "fp32", newton_max_iter=limit, float_quartic=float_quartic)
    try:
        g.step()
        return True
    except capi.RTError as e:
        assert e.code == capi.RT_ERR_NONCONV
        return False
    finally:
        g.close()


@pytest.mark.parametrize("J0", [0.2, 1.0, 5.0, 100.0, 1e4])
@pytest.mark.parametrize("order", [2, 4, 8])
def test_limit_refuses_the_same_steps(order, J0):
    # stiff cells: the root lies far from the temperature before the step
    prob = make(n=(4, 4, 4), order=order, kP=1e6, kJ=1e6, J0=J0)
    limits = list(range(1, 41))
    refined = [_accepts(prob, k, 0) for k in limits]
    plain = [_accepts(prob, k, 1) for k in limits]
    assert refined == plain
    assert not refined[0] and refined[-1]  # the range holds both outcomes
