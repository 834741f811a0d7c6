"""The step's preconditioner on a large mesh of needle triangles. Inside flexible GMRES the
factorised Poisson solves run a fixed number of sweeps; on this mesh (155,000 vertices, a
torus squashed to a tenth of its height) that leaves more than a hundredth of the right-hand
side, and the solves have to go on. The Krylov loop is cut at 20 iterations, so that the
direction shows the preconditioner: each of its two solves is good to a hundredth, hence the
slope dE . x agrees to 2 in a hundred with that of a step whose solves are all CG."""
import numpy as np
import pytest

from oracle import tp_oracle as O
from synth import gaussian_noise, torus

pytestmark = pytest.mark.gpu


def test_needles(lib):
    V, F = torus(620, 250, 1.0, 0.3)
    V = gaussian_noise(V, 1e-3 / 620, 3) * np.array([1.0, 0.1, 1.0])
    c = lib.tp_constraints(flags=1, A0=O.total_area(V, F), V0=0.0)
    slope = []
    with lib.Mesh(V, F) as m:
        for solver in (0, 1):
            m.set_positions(V)
            p = lib.params(theta=0.5, krylov_tol=1e-4, krylov_max=20, cg_tol=1e-4, cg_max=3000, tau0_disp=0.25, ls_max=1,
                           poisson_solver=solver)
            slope.append(lib.precond_step(m, c, p)["slope"])
    assert slope[1] < 0
    assert abs(slope[0] / slope[1] - 1) <= 2e-2, slope
