"""The static outflow coefficients of double states (sum_f max(u, 0) per cell
and angle): where the device has no room for their table the kernels sum them,
in the same order, so a step and its reverse are the same bit for bit."""
import numpy as np
import pytest
import torch

from paper_2002_08377_gb300 import build as rtbuild
from paper_2002_08377_gb300 import capi
from tests._problems import make, randomise

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    rtbuild.build()
    capi.load()


def _results(prob, fill):
    """Step and reverse step of a state created with little free memory (fill)
    or plenty; the state's bytes."""
    from paper_2002_08377_gb300.solver import RTSolver
    hold = None
    if fill:
        torch.cuda.empty_cache()
        N, A, nnz = prob.n_cells, prob.n_angles, 2 * prob.mesh.n_faces
        need = 8 * (nnz * (A // 2 + 8) + 3 * N * (A + 16))  # what the state takes without the table
        hold = torch.empty(torch.cuda.mem_get_info()[0] - need - (16 << 20), dtype=torch.uint8,
                           device="cuda")
    g = RTSolver.from_problem(prob, "fp64")
    size = g.device_bytes()
    del hold
    torch.cuda.empty_cache()
    dt = prob.cfl_dt()
    g.run(2, dt)
    out = [g.get_intensity(), *g.gas()]
    rng = np.random.default_rng(3)
    dev = lambda x: torch.tensor(x, device="cuda")
    N, A = prob.n_cells, prob.n_angles
    gP = torch.zeros(N, dtype=torch.float64, device="cuda")
    gJ = torch.zeros_like(gP)
    out += [t.cpu().numpy() for t in
            g.adjoint_step(dt, dev(out[0]), dev(out[1]), dev(out[2]),
                           dev(rng.standard_normal((N, A))), dev(rng.standard_normal(N)),
                           dev(rng.standard_normal((N, 3))), gP, gJ)]
    g.close()
    return out, size


@pytest.mark.parametrize("order", [4, 8])  # 12 pairs (ragged over 8 threads), 40 pairs
def test_summed_coefficients_equal_the_table(order):
    prob = randomise(make(n=(18, 18, 17), order=order, seed=5))
    a, size_a = _results(prob, False)
    b, size_b = _results(prob, True)
    assert size_a - size_b == 8 * prob.n_cells * prob.n_angles  # the table was left out
    for x, y in zip(a, b):
        assert np.array_equal(x, y)
