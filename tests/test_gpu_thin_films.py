"""Thin films in the grid kernels, whose rows share words where a launch has rows
enough to fill the GPU, against the CPU oracle.  Integers throughout: every
comparison is exact."""
import numpy as np
import pytest

import paper_1411_5588_gb300 as ig
from oracle import oracle as O

pytestmark = pytest.mark.gpu
SHAPES = pytest.mark.parametrize("shape", [ig.SHAPE_GRID_1, ig.SHAPE_GRID_Q, ig.SHAPE_GRID_2], ids=["one", "two", "four"])


# On both sides of two and a half waves of rows (389120) for four rows per word, of one
# (155648) for two; ragged groups and calls.
@SHAPES
@pytest.mark.parametrize("H", [0.0, 0.2])
@pytest.mark.parametrize("Lx,Ly,Lz", [(379, 1024, 8), (390, 1000, 16), (391, 1004, 10), (152, 1024, 30), (160, 1000, 20),
                                      (157, 1002, 32), (512, 612, 2)])
def test_films(Lx, Ly, Lz, H, shape):
    g = ig.Film(Lx, Ly, Lz, 1.0, 0.5, 2.8, 3, H=H, shape=shape)
    o = O.Film(Lx, Ly, Lz, 1.0, 0.5, 2.8, 3, H=H)
    g.init(ig.INIT_RANDOM)
    o.init(ig.INIT_RANDOM, 0.0)
    g.sweep(2, 1)
    assert np.array_equal(g.read_series(), o.sweep(2, 1))
    assert np.array_equal(g.get_spins(), o.get_spins())
    g.close()


# Small thin films packed by a set's size, and not.
@SHAPES
@pytest.mark.parametrize("big", [True, False], ids=["packed", "rows"])
@pytest.mark.parametrize("H", [0.0, 0.2])
def test_sets(H, big, shape):
    sizes = [(4, 8, 16), (5, 28, 2), (4, 12, 10), (32, 260, 30), (33, 256, 20)] + ([(60, 280, 1600)] if big else [])
    jobs = [dict(Lx=L[0], Ly=L[1], Lz=L[2], T=2.6, H1=0.4, H=H, seed=5, replica=i, init_kind=ig.INIT_RANDOM, measure_every=2)
            for i, L in enumerate(sizes)]
    b = ig.Batch(jobs, lanes=1)
    b.set_shape(shape)
    b.sweep(4, False)
    for i, j in enumerate(jobs):
        o = O.Film(j["Lx"], j["Ly"], j["Lz"], 1.0, j["H1"], j["T"], j["seed"], H=j["H"], replica=i)
        o.init(ig.INIT_RANDOM, 0.0)
        assert np.array_equal(b.read_series(i), o.sweep(4, 2)), i
        assert np.array_equal(b.get_spins(i), o.get_spins()), i
    b.close()


# Sets of short words alone (columns by masks), packed and not, some in a bulk field.
@SHAPES
@pytest.mark.parametrize("sizes", [
    [(391, 1004, 10, 0.0), (5, 28, 2, 0.3), (33, 256, 20, 0.0), (7, 12, 6, -0.2), (32, 260, 30, 0.1)],
    [(24, 61, 40, 0.0), (7, 13, 34, 0.3), (12, 31, 20, 0.0), (3, 2, 2, 0.0), (9, 47, 38, 0.0)]], ids=["packed", "rows"])
def test_sets_of_short_words(sizes, shape):
    jobs = [dict(Lx=L[0], Ly=L[1], Lz=L[2], T=2.6, H1=0.4, H=L[3], seed=5, replica=i, init_kind=ig.INIT_RANDOM,
                 measure_every=1 + i % 2) for i, L in enumerate(sizes)]
    b = ig.Batch(jobs, lanes=1)
    b.set_shape(shape)
    b.sweep(4, False)
    for i, j in enumerate(jobs):
        o = O.Film(j["Lx"], j["Ly"], j["Lz"], 1.0, j["H1"], j["T"], j["seed"], H=j["H"], replica=i)
        o.init(ig.INIT_RANDOM, 0.0)
        assert np.array_equal(b.read_series(i), o.sweep(4, j["measure_every"])), i
        assert np.array_equal(b.get_spins(i), o.get_spins()), i
    b.close()
