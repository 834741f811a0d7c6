"""The Barnes-Hut tree and lists where their construction can go wrong: one leaf, one
full and one partial leaf, leaves of one face, fewer faces than a group of 32 and one
face more, short and long lists in turn, and rebuilds on the same mesh. The tree decides in FP32 as the oracle's does, so E, dE and the applies agree
with the oracle's Barnes-Hut sums over the same tree to the FP32 tolerance, 1e-5."""
import numpy as np
import pytest

from oracle import tp_oracle as O
from synth import small_mesh, vertex_vectors

pytestmark = pytest.mark.gpu
TOL = 1e-5


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - b) / np.linalg.norm(b))


@pytest.mark.parametrize("kind", ["tetra", "octa", "torus3x3", "torus8x4", "torus11x3", "torus13x10", "ico3"])
@pytest.mark.parametrize("leaf", [1, 8, 32])
@pytest.mark.parametrize("theta", [0.05, 0.5])
def test_sums_over_the_tree(lib, kind, leaf, theta):
    V, F = small_mesh(kind, seed=5)
    u = vertex_vectors(len(V), 3, 8)
    p = lib.params(theta=theta, leaf_size=leaf)
    with lib.Mesh(V, F) as m:
        for _ in range(2):                     # the second time on a tree rebuilt in place
            E = lib.tp_energy(m, p)
            g, _ = lib.tp_differential(m, p)
            y = lib.fractional_apply(m, "A", u, p)
            m.set_positions(V)
    assert abs(E / O.bh_energy(V, F, theta, leaf) - 1) <= TOL
    assert rel(g, O.bh_differential(V, F, theta, leaf)) <= TOL
    assert rel(y, O.bh_apply_operator(V, F, u, "A", theta, leaf)) <= TOL


def test_lists_of_different_length_on_one_mesh(lib):
    # the pool of one mesh serves short and long lists in turn; at theta = 0.02 nearly
    # every pair is summed exactly
    V, F = small_mesh("torus61x33", seed=9)
    with lib.Mesh(V, F) as m:
        e = [lib.tp_energy(m, lib.params(theta=t, leaf_size=1)) for t in (1.0, 0.02, 0.5, 0.02)]
    E = O.energy(V, F)
    assert e[1] == e[3]
    assert abs(e[1] / E - 1) <= TOL


@pytest.mark.parametrize("noise,theta,leaf", [(0.3, 0.5, 1), (0.3, 0.25, 1), (0.1, 0.5, 4)])
def test_lists_longer_than_the_first_pool(lib, noise, theta, leaf):
    # a crumpled surface, whose lists are several times those of a smooth one: the first
    # tree's entries are written by a second traversal and the pool is not grown for
    # them, the next tree finds a pool of the size they asked for. The lists are the same,
    # so E and the apply are equal bit by bit; the walks (rows of given targets) sum the
    # same terms in another order
    from synth import gaussian_noise, torus
    V, F = torus(200, 50, 1.0, 0.3)
    V = gaussian_noise(V, noise, 1)
    u = vertex_vectors(len(V), 3, 8)
    p = lib.params(theta=theta, leaf_size=leaf)
    with lib.Context(0) as ctx:
        with lib.Mesh(V, F, ctx=ctx) as m:
            E, y, used = [], [], []
            for _ in range(3):
                E.append(lib.tp_energy(m, p))
                y.append(lib.fractional_apply(m, "A", u, p))
                used.append(ctx.memory()[0])
                m.set_positions(V)
            rows = lib.tp_energy_rows(m, np.arange(len(F), dtype=np.int32), p)
    assert used[0] < used[1] == used[2]
    assert E[0] == E[1] == E[2]
    assert np.array_equal(y[0], y[1]) and np.array_equal(y[0], y[2])
    assert abs(E[0] / rows.sum() - 1) <= TOL


def test_lists_without_room_for_the_pool(lib):
    # an allocator that refuses the pool (43 MB here; nothing else is above 16 MB): two
    # traversals give the same lists, hence E and the apply bit by bit
    import ctypes

    import torch
    from synth import gaussian_noise, torus
    V, F = torus(200, 50, 1.0, 0.3)
    V = gaussian_noise(V, 0.002, 1)
    u = vertex_vectors(len(V), 3, 8)
    p = lib.params(theta=0.25)
    with lib.Mesh(V, F) as m:
        E, y = lib.tp_energy(m, p), lib.fractional_apply(m, "A", u, p)
    refused = []

    @lib._ALLOC_FN
    def alloc(nbytes, device, user):
        if nbytes > 32 << 20:
            refused.append(nbytes)
            return None
        return int(torch.cuda.caching_allocator_alloc(int(nbytes), device, torch.cuda.current_stream(device)))

    @lib._FREE_FN
    def free(ptr, nbytes, device, user):
        torch.cuda.caching_allocator_delete(int(ptr))

    with lib.Context(0) as ctx:
        a = lib.tp_allocator(alloc, free, None)
        lib._check(lib.lib().tp_ctx_set_allocator(ctx.handle, ctypes.byref(a)))
        with lib.Mesh(V, F, ctx=ctx) as m:
            for _ in range(2):
                assert lib.tp_energy(m, p) == E
                assert np.array_equal(lib.fractional_apply(m, "A", u, p), y)
                m.set_positions(V)
    assert len(refused) == 2
