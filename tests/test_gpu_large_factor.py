"""Factorised Poisson solves at the sizes where the factor's paths change: fronts of
one tile and of many, panels of whole and partial blocks of eight columns, chains of
separator supernodes whose update matrices share storage, fronts whose children's
vectors do not fit beside them, and sweeps in three launches (meshes of thousands of
supernodes). A solve promises |b - C z| <= cg_tol |b| per column with the residual in
FP64; the oracle's C differs from the library's by rounding, |C| |z| 2^-50 |b|^-1 at
most here, so the residual by the oracle's C stays below 1.01 cg_tol at 1e-8."""
import numpy as np
import pytest

from oracle import tp_oracle as O
from synth import gaussian_noise, icosphere, linked_tori, torus

pytestmark = pytest.mark.gpu


def mesh_of(kind, a, b):
    if kind == "ico":
        return icosphere(a)
    if kind == "linked":
        return linked_tori(a, b)
    return torus(a, b, 1.0, 0.3)


@pytest.mark.parametrize("kind,a,b", [("torus", 9, 7), ("torus", 12, 11), ("torus", 61, 30), ("linked", 90, 31),
                                      ("ico", 6, 0), ("torus", 700, 143), ("ico", 7, 0)])
@pytest.mark.parametrize("k", [1, 3, 9])
def test_residual(lib, kind, a, b, k):
    import torch
    V, F = mesh_of(kind, a, b)
    V = gaussian_noise(V, 0.2 / max(a, 50) if kind != "ico" else 0.1 / 2 ** a, 7)
    rhs = np.random.default_rng(3).standard_normal((len(V), k))
    with lib.Mesh(V, F) as m:
        assert lib.cotan_factor_info(m)["available"] == 1
        z, it = lib.cotan_solve(m, rhs, lib.params(cg_tol=1e-8))
        # the same factor again, and after new positions a new one
        z2, _ = lib.cotan_solve(m, rhs, lib.params(cg_tol=1e-8))
        m.set_positions(V)
        z3, _ = lib.cotan_solve(m, rhs, lib.params(cg_tol=1e-8))
    assert np.array_equal(z, z2) and np.array_equal(z, z3)
    assert it <= 12
    C = O.cotan_laplacian(V, F)
    comp = O.mesh_components(len(V), F)
    r = O.project_mean_zero(rhs, comp) - C @ z
    res = np.linalg.norm(r, axis=0) / np.linalg.norm(O.project_mean_zero(rhs, comp), axis=0)
    assert res.max() <= 1.01e-8, res
