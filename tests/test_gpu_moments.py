"""GPU moments (rt_moments) against the sums written out in numpy, on angle
sets with unequal weights, cell counts on both sides of the kernel's two
thread mappings, and angle counts that end inside a staged block of positions.

Tolerance: both sides add A rounded products of at most four factors, so each
result is within (A + 8) 2^-52 of the sum of the terms' magnitudes."""
import numpy as np
import pytest

from paper_2002_08377_gb300 import build as rtbuild
from paper_2002_08377_gb300 import capi
from paper_2002_08377_gb300.inputs import build_mesh

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    rtbuild.build()
    capi.load()


# 19683 cells: one thread per cell, the last block ragged; 80: eight threads
@pytest.mark.parametrize("n", [(27, 27, 27), (4, 4, 5)])
@pytest.mark.parametrize("A", [2, 6, 34, 80, 112])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_moments_match_written_sums(n, A, precision):
    from paper_2002_08377_gb300.solver import RTSolver
    rng = np.random.default_rng(A)
    up = rng.normal(size=(A // 2, 3))
    up /= np.linalg.norm(up, axis=1, keepdims=True)
    dirs = np.ascontiguousarray(np.concatenate([up, -up]))
    w = rng.uniform(0.1, 1.0, A)
    w /= w.sum()
    mesh = build_mesh(n, seed=1)
    g = RTSolver(mesh, dirs, w, cbar=1.0, c=3.0, precision=precision)
    I = rng.uniform(0.0, 2.0, (mesh.n_cells, A)).astype(g.dtype)
    g.set_intensity(I)
    E, F, P = g.moments()
    nn = np.stack([dirs[:, a] * dirs[:, b]
                   for a, b in ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))], 1)
    wI = 4 * np.pi * w * I.astype(np.float64)
    for got, t, f in ((E[:, None], np.ones((A, 1)), 1.0), (F, dirs, 3.0), (P, nn, 1.0)):
        tol = (A + 8) * 2.0 ** -52 * f * (wI @ np.abs(t))
        assert np.all(np.abs(got - f * (wI @ t)) <= tol)
    g.close()
