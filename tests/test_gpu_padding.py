"""Faces next to the bounding box's centre, the origin of the face tables, in meshes
whose face count is no multiple of a tile of 128: the padding of the last tile must
give zero terms there too (a term formed at the origin before it is multiplied by a
zero area would be infinite: |d|^-6 passes FP32's range below |d| = 4e-7). The FP32
path's parity tolerance, 1e-5, holds against the oracle: the padding adds nothing, and
the faces' own pairs are no closer than in the other parity tests."""
import ctypes

import numpy as np
import pytest

from oracle import tp_oracle as O
from synth import icosphere, vertex_vectors

pytestmark = pytest.mark.gpu
TOL = 1e-5


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - b) / np.linalg.norm(b))


def sphere_with_inner_face(h):
    """A sphere and a tetrahedron inside it with a face across the axis at height h."""
    V, F = icosphere(3)
    r = 0.05 * 3.0 ** 0.5
    T = np.array([[0.1, 0.0, h], [-0.05, r, h], [-0.05, -r, h], [0.0, 0.0, -0.1]])
    G = np.array([[0, 1, 2], [0, 3, 1], [1, 3, 2], [2, 3, 0]])
    return np.concatenate([V, T]), np.concatenate([F, G + len(V)]).astype(np.int32)


@pytest.mark.parametrize("h", [1e-7, 1e-8, 1e-9])
@pytest.mark.parametrize("p", [6.0, 4.5])
def test_energy_and_differential(lib, h, p):
    V, F = sphere_with_inner_face(h)
    assert len(F) % 128 == 4
    with lib.Mesh(V, F) as m:
        q = lib.params(p=p)
        E, (g, E2) = lib.tp_energy(m, q), lib.tp_differential(m, q)
        rows = lib.tp_energy_rows(m, np.arange(len(F), dtype=np.int32), q)
    E0 = O.energy(V, F, p)
    assert abs(E / E0 - 1) <= TOL and abs(E2 / E0 - 1) <= TOL
    assert abs(rows.sum() / E0 - 1) <= TOL
    assert rel(g, O.differential(V, F, p)) <= TOL


@pytest.mark.parametrize("h", [1e-7, 1e-8, 1e-9])
@pytest.mark.parametrize("op", ["A", "B", "B0", "L"])
@pytest.mark.parametrize("k", [1, 3, 9])
def test_applies(lib, h, op, k):
    V, F = sphere_with_inner_face(h)
    u = vertex_vectors(len(V), k, 5)
    with lib.Mesh(V, F) as m:
        y = lib.fractional_apply(m, op, u, lib.params())
    assert rel(y, O.apply_operator(V, F, u, op)) <= TOL


@pytest.mark.parametrize("h", [1e-7, 1e-8, 1e-9])
def test_allocation_free_energy(lib, h):
    import torch
    V, F = sphere_with_inner_face(h)
    pos = torch.tensor(V, device="cuda:0")
    faces = torch.tensor(F, device="cuda:0")
    E = torch.zeros(1, dtype=torch.float64, device="cuda:0")
    lib.lib().tp_energy_noalloc(ctypes.c_void_p(pos.data_ptr()), len(V), ctypes.c_void_p(faces.data_ptr()), len(F),
                                ctypes.c_double(6.0), ctypes.c_void_p(E.data_ptr()),
                                ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    torch.cuda.synchronize()
    E0 = O.energy(V, F)
    assert abs(E.item() / E0 - 1) <= TOL
