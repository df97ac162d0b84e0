"""Kernels that look a site's threshold up by its number of up neighbours,
against the CPU oracle: films in bulk fields and their walls, at the edges of
columns, packed rows, partial words and slabs, and large launches.

Integers throughout: every comparison is exact.
"""
import math

import numpy as np
import pytest

import paper_1411_5588_gb300 as ig
from oracle import oracle as O

pytestmark = pytest.mark.gpu


def _same(Lx, Ly, Lz, shape, calls=((2, 1), (3, 2)), y=ig.Y_GAPBC, x=ig.X_FREE, J=1.0, H1=0.5, H=0.3, T=2.7):
    g = ig.Film(Lx, Ly, Lz, J, H1, T, 31, y_mode=y, x_mode=x, H=H, shape=shape)
    o = O.Film(Lx, Ly, Lz, J, H1, T, 31, y_mode=y, x_mode=x, H=H)
    g.init(ig.INIT_RANDOM)
    o.init(ig.INIT_RANDOM, 0.0)
    for n, every in calls:
        g.sweep(n, every)
        assert np.array_equal(g.read_series(), o.sweep(n, every))
    assert np.array_equal(g.get_spins(), o.get_spins())
    g.close()


# Columns of two and four words: rows from none to one past two columns; words
# that are full, that end in the middle of a call, and the row's only one.
@pytest.mark.parametrize("shape", [ig.SHAPE_GRID_Q, ig.SHAPE_GRID_2], ids=["two", "four"])
@pytest.mark.parametrize("Ly", [2, 3, 5, 6, 10, 11])
@pytest.mark.parametrize("Lx,Lz", [(1, 64), (2, 66), (7, 128), (11, 200), (5, 34), (4, 6)])
def test_columns(Lx, Ly, Lz, shape):
    _same(Lx, Ly, Lz, shape)


@pytest.mark.parametrize("shape", [ig.SHAPE_GRID_2, ig.SHAPE_CLUSTER], ids=["four", "cluster"])
@pytest.mark.parametrize("Lx,Ly,Lz", [(4, 8, 16), (4, 12, 10), (32, 260, 30), (33, 256, 18), (40, 512, 16)])
def test_packed_rows(Lx, Ly, Lz, shape):
    _same(Lx, Ly, Lz, shape)


# Orders of the costly moves (which spin at which k), walls of either sign,
# thresholds that are 0 or always met.
@pytest.mark.parametrize("kw", [dict(H=-0.3), dict(H=-7.5), dict(H=2.0), dict(J=-1.0), dict(J=-0.7, H=0.2),
                                dict(J=0.0, H=0.4), dict(x=ig.X_PBC, H=0.5, H1=-0.5), dict(H1=-5.0, H=0.1),
                                dict(T=1e-3), dict(T=math.inf), dict(T=1e12), dict(y=ig.Y_PBC), dict(y=ig.Y_APBC)], ids=str)
@pytest.mark.parametrize("Lx,Ly,Lz,shape", [(6, 9, 64, ig.SHAPE_GRID_Q), (6, 9, 46, ig.SHAPE_GRID_2),
                                            (8, 200, 66, ig.SHAPE_CLUSTER)])
def test_thresholds(Lx, Ly, Lz, shape, kw):
    _same(Lx, Ly, Lz, shape, **kw)


# One word per thread in launches past a wave, pairs included; packed rows too.
@pytest.mark.parametrize("Lx,Ly,Lz", [(40, 130, 2010), (90, 300, 384), (24, 26000, 10), (13, 12000, 70)])
def test_large_launches_of_one_word(Lx, Ly, Lz):
    _same(Lx, Ly, Lz, ig.SHAPE_GRID_1, calls=((2, 2),))


# Slabs in columns: several turns, two and more CTAs, uneven layers.
@pytest.mark.parametrize("Lx,Ly,Lz,H", [(8, 96, 640, 0.0), (13, 150, 130, 0.3), (16, 384, 64, 0.0), (9, 700, 64, -0.2),
                                        (24, 200, 256, 0.1), (8, 4, 20000, 0.2)])
def test_slab_columns(Lx, Ly, Lz, H):
    _same(Lx, Ly, Lz, ig.SHAPE_CLUSTER, H=H)


# Sets whose films differ in form, in every grid shape.
@pytest.mark.parametrize("shape", [ig.SHAPE_GRID_1, ig.SHAPE_GRID_Q, ig.SHAPE_GRID_2], ids=["one", "two", "four"])
@pytest.mark.parametrize("fields", [(0.0, 0.0, 0.3), (0.3, -0.3, 0.0), (0.2, 0.2, 0.2)], ids=str)
def test_sets_of_both_forms(fields, shape):
    sizes = [(8, 12, 16), (11, 31, 200), (60, 200, 1000)]
    jobs = [dict(Lx=L[0], Ly=L[1], Lz=L[2], T=2.5, H1=0.4, H=H, seed=9, replica=i, init_kind=ig.INIT_RANDOM, measure_every=1 + i)
            for i, (L, H) in enumerate(zip(sizes, fields))]
    b = ig.Batch(jobs, lanes=1)
    b.set_shape(shape)
    b.sweep(5, False)
    b.sweep(40, True)
    for i, j in enumerate(jobs):
        o = O.Film(j["Lx"], j["Ly"], j["Lz"], 1.0, j["H1"], j["T"], j["seed"], H=j["H"], replica=i)
        o.init(ig.INIT_RANDOM, 0.0)
        assert np.array_equal(b.read_series(i), o.sweep(45, j["measure_every"])), i
        assert np.array_equal(b.get_spins(i), o.get_spins()), i
    b.close()
