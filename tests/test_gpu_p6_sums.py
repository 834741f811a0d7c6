"""The FP32 energy and differential at p = 6 (two-sided pair terms over the target
blocks' own and later tiles; equal runs of 32-source units) at the sizes where their
splits change: part of a unit, edges of tiles (128), of target rows (256, 512) and of
the switch between two and four targets a thread (about 3,070 faces), against the
oracle. FP32 terms differ from it by a few 2^-24 each and the sums are compensated;
the parity tolerance of the FP32 path, 1e-5, holds."""
import numpy as np
import pytest

from oracle import tp_oracle as O
from synth import icosphere, small_mesh, torus

pytestmark = pytest.mark.gpu
TOL = 1e-5


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - b) / np.linalg.norm(b))


@pytest.mark.parametrize("a,b", [(4, 4), (9, 7), (16, 4), (13, 5), (8, 16), (43, 3), (64, 4), (37, 7), (48, 32),
                                 (64, 24), (59, 26), (45, 37)])
def test_sizes(lib, a, b):
    # 32, 126, 128, 130, 256, 258, 512, 518, 3072 (both sides of it: 3068) and 3330 faces
    V, F = small_mesh(f"torus{a}x{b}", seed=a)
    with lib.Mesh(V, F) as m:
        p = lib.params()
        E, (g, E2) = lib.tp_energy(m, p), lib.tp_differential(m, p)
        rows = lib.tp_energy_rows(m, np.arange(len(F), dtype=np.int32), p)
    E0 = O.energy(V, F)
    assert abs(E / E0 - 1) <= TOL and abs(E2 / E0 - 1) <= TOL
    assert abs(rows.sum() / E0 - 1) <= TOL
    assert rel(g, O.differential(V, F)) <= TOL


def test_with_an_obstacle(lib):
    # the obstacle adds to the adjoints and to the energy of the step
    V, F = small_mesh("torus16x10", seed=4)
    W, G = icosphere(2, 0.4)
    with lib.Mesh(V, F) as m:
        lib.tp_obstacle_set(m, W, G, weight=2.0)
        c = lib.tp_constraints(flags=0, A0=0.0, V0=0.0)
        rep = lib.precond_step(m, c, lib.params(krylov_tol=1e-6, fixed_tau=1, tau0=1e-3, proj_iters=0))
        f = m.get_positions()
    E0 = O.energy(V, F) + O.obstacle_energy(V, F, W, G, weight=2.0)
    E1 = O.energy(f, F) + O.obstacle_energy(f, F, W, G, weight=2.0)
    assert abs(rep["E_before"] / E0 - 1) <= TOL and abs(rep["E_after"] / E1 - 1) <= TOL
    # slope = dE . x with x the direction moved along; dE within TOL of the oracle's
    x = (f - V) / rep["tau"]
    g = O.differential(V, F) + O.obstacle_differential(V, F, W, G, weight=2.0)
    assert abs(rep["slope"] - float(np.sum(g * x))) <= TOL * np.linalg.norm(g) * np.linalg.norm(x)
