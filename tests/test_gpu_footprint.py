"""tp_mesh_footprint_bytes, by which the server admits requests, against the memory that a
context counts for a mesh after everything that a request runs: energy, differential, the
operators on nine columns and a step with both constraints. Smooth and lightly noisy
surfaces, direct sums and Barnes-Hut at the trees' and lists' extremes, both precisions.
The estimate is not below what is held, and not above three times it (meshes of a few
hundred faces, whose fixed buffers are most of it, aside)."""
import numpy as np
import pytest

from oracle import tp_oracle as O
from synth import gaussian_noise, torus

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("a,b", [(20, 10), (50, 31), (97, 41), (200, 50), (300, 85)])
@pytest.mark.parametrize("kw", [dict(), dict(p=4.5), dict(precision=1), dict(tensor_cores=1), dict(poisson_solver=1),
                                dict(theta=0.5), dict(theta=0.25), dict(theta=0.1), dict(theta=0.5, leaf_size=1),
                                dict(theta=0.5, leaf_size=32), dict(gmres_restart=60)],
                         ids=lambda kw: ",".join(f"{k}={v}" for k, v in kw.items()) or "default")
def test_estimate_covers_what_a_mesh_holds(lib, a, b, kw):
    if kw.get("precision") == 1 and a > 97:
        pytest.skip("FP64 steps of that size take seconds")
    V, F = torus(a, b, 1.0, 0.3)
    V = gaussian_noise(V, 0.002, 1)
    u = np.random.default_rng(2).standard_normal((len(V), 9))
    p = lib.params(krylov_tol=1e-4, krylov_max=30, cg_tol=1e-4, tau0_disp=0.25, **kw)
    c = lib.tp_constraints(flags=3, A0=O.total_area(V, F), V0=O.total_volume(V, F))
    with lib.Context(0) as ctx:
        with lib.Mesh(V, F, ctx=ctx) as m:
            lib.tp_energy(m, p)
            lib.tp_differential(m, p)
            for op in ("A", "B", "B0", "L"):
                lib.fractional_apply(m, op, u, p)
            lib.precond_step(m, c, p)
            _, peak = ctx.memory()
    est = lib.tp_mesh_footprint_bytes(len(V), len(F), p)
    print(f"{a}x{b} {kw}: held {peak / 1e6:.1f} MB, estimate {est / 1e6:.1f} MB, {est / peak:.2f}")
    assert peak <= est
    assert len(F) < 1000 or est <= 3 * peak
