"""FP64 operator applies: the rational power |d|^{-2s} by a root and a series step
(2 n / p whole for some n <= 16), pow for the other exponents and for distances
outside the root's range, and the combine at every column count and at face counts
around its blocks of 32. Against the FP64 oracle: each of a row's up to 130 terms is
rounded to 2^-53 on both sides and the row sums cancel by less than 10^3 here, so
the difference stays below 130 x 2^-53 x 10^3 = 1.5e-11; the tolerance is 1e-10."""
import numpy as np
import pytest

from oracle import tp_oracle as O
from synth import small_mesh, vertex_vectors

pytestmark = pytest.mark.gpu
TOL = 1e-10


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - b) / np.linalg.norm(b))


@pytest.mark.parametrize("p", [6.0, 4.5, 3.0, 5.0, 4.0, 8.0, 2.5, 32.0 / 13.0, 3.7])
@pytest.mark.parametrize("op", ["A", "B0", "L"])
def test_exponents(lib, p, op):
    V, F = small_mesh("torus13x5", seed=11)          # 130 faces: two source tiles
    u = vertex_vectors(len(V), 3, 5)
    with lib.Mesh(V, F) as m:
        y = lib.fractional_apply(m, op, u, lib.params(p=p, precision=lib.TP_PREC_FP64))
    assert rel(y, O.apply_operator(V, F, u, op, p)) <= TOL


@pytest.mark.parametrize("scale", [1e-17, 1e-14, 1e14, 1e17])
def test_distances_around_the_range_of_the_root(lib, scale):
    V, F = small_mesh("ico1", seed=3)
    V = V * scale                                    # |d|^2 from 1e-36 to 1e35: inside and outside 2^+-100
    u = vertex_vectors(len(V), 3, 6)
    with lib.Mesh(V, F) as m:
        for op in ("A", "L"):
            y = lib.fractional_apply(m, op, u, lib.params(precision=lib.TP_PREC_FP64))
            assert rel(y, O.apply_operator(V, F, u, op)) <= TOL, op


@pytest.mark.parametrize("kind", ["tetra", "octa", "ico0", "torus4x4", "torus11x3", "torus16x4"])
@pytest.mark.parametrize("k", [1, 2, 3, 4, 9])
def test_face_and_column_counts(lib, kind, k):
    V, F = small_mesh(kind, seed=2)                  # 4, 8, 20, 32, 66 and 128 faces
    u = vertex_vectors(len(V), k, 7)
    with lib.Mesh(V, F) as m:
        for op in ("A", "B"):
            y = lib.fractional_apply(m, op, u, lib.params(precision=lib.TP_PREC_FP64))
            assert rel(y, O.apply_operator(V, F, u, op)) <= TOL, op
