"""Kernels that draw a half-sweep's masks before its lattice is known, and the
spin packing, against the CPU oracle at the sizes where they can go wrong.

Integers throughout: every comparison is exact.
"""
import math

import numpy as np
import pytest

import paper_1411_5588_gb300 as ig
from oracle import oracle as O

pytestmark = pytest.mark.gpu


def _pair(Lx, Ly, Lz, y=ig.Y_GAPBC, x=ig.X_FREE, J=1.0, H1=0.5, H=0.0, T=3.0, seed=21, shape=ig.SHAPE_AUTO):
    g = ig.Film(Lx, Ly, Lz, J, H1, T, seed, y_mode=y, x_mode=x, H=H, shape=shape)
    o = O.Film(Lx, Ly, Lz, J, H1, T, seed, y_mode=y, x_mode=x, H=H)
    g.init(ig.INIT_RANDOM)
    o.init(ig.INIT_RANDOM, 0.0)
    return g, o


def _same(g, o, calls=((3, 1), (4, 2))):
    for n, every in calls:
        g.sweep(n, every)
        assert np.array_equal(g.read_series(), o.sweep(n, every))
    assert np.array_equal(g.get_spins(), o.get_spins())
    g.close()


# Columns of one, two and four words (GRID_1, GRID_Q, GRID_2): Ly - 2 interior
# rows from none to one past two columns, words that end in the middle of a block.
@pytest.mark.parametrize("shape", [ig.SHAPE_GRID_1, ig.SHAPE_GRID_Q, ig.SHAPE_GRID_2], ids=["one", "two", "four"])
@pytest.mark.parametrize("Ly", [2, 3, 4, 5, 6, 7, 10, 11])
@pytest.mark.parametrize("Lx,Lz", [(3, 70), (11, 200)])
def test_columns_of_every_remainder(Lx, Ly, Lz, shape):
    _same(*_pair(Lx, Ly, Lz, shape=shape))


# Packed rows (four to a word at 8 sites per array, two at 16) with a group
# count around the column length; Lx * Ly past the two-row packing's threshold.
@pytest.mark.parametrize("shape", [ig.SHAPE_GRID_1, ig.SHAPE_GRID_2, ig.SHAPE_CLUSTER], ids=["one", "four", "cluster"])
@pytest.mark.parametrize("Lx,Ly,Lz", [(4, 8, 16), (4, 12, 10), (5, 28, 2), (32, 260, 30), (33, 256, 20)])
def test_packed_rows(Lx, Ly, Lz, shape):
    _same(*_pair(Lx, Ly, Lz, shape=shape), calls=((2, 1), (3, 3)))


# The general seven-threshold form: bulk fields, antiferromagnetic and zero
# couplings, opposite wall kinds under periodic x (one wall's field cancelled by
# the bulk field), T -> 0 and infinity; and the three-mask form beside it.
@pytest.mark.parametrize("shape", [ig.SHAPE_RESIDENT, ig.SHAPE_GRID_1, ig.SHAPE_GRID_2, ig.SHAPE_CLUSTER],
                         ids=["resident", "one", "four", "cluster"])
@pytest.mark.parametrize("kw", [dict(H=0.3), dict(H=-7.5), dict(J=-1.0), dict(J=-0.7, H=0.2), dict(J=0.0, H=0.4),
                                dict(x=ig.X_PBC, H=0.5, H1=-0.5), dict(x=ig.X_PBC, H=0.0, H1=0.0), dict(H1=5.0),
                                dict(T=1e-3), dict(T=1e-3, H=0.3), dict(T=math.inf), dict(T=math.inf, H=0.3),
                                dict(T=1e12)], ids=str)
def test_general_thresholds(kw, shape):
    _same(*_pair(6, 9, 46, shape=shape, **kw))


# Resident and cluster films: four lanes per word, one lane per word, columns
# (slabs past the shared memory of the words and masks), several turns.
@pytest.mark.parametrize("Lx,Ly,Lz,shape", [
    (8, 8, 8, ig.SHAPE_RESIDENT), (5, 25, 64, ig.SHAPE_RESIDENT), (5, 27, 64, ig.SHAPE_RESIDENT),
    (16, 48, 32, ig.SHAPE_CLUSTER), (8, 81, 64, ig.SHAPE_CLUSTER), (16, 150, 130, ig.SHAPE_CLUSTER),
    (9, 700, 64, ig.SHAPE_CLUSTER), (8, 4, 20000, ig.SHAPE_CLUSTER), (24, 200, 256, ig.SHAPE_CLUSTER)])
def test_slabs(Lx, Ly, Lz, shape):
    _same(*_pair(Lx, Ly, Lz, shape=shape), calls=((2, 1), (3, 2)))


# Spins as int8 in device memory: every access width (the address and Lz decide),
# rows that end anywhere in a word pair, values other than +-1.
@pytest.mark.parametrize("offset", [0, 1, 2, 4, 8, 16])
@pytest.mark.parametrize("Lz", [2, 4, 6, 16, 30, 48, 62, 64, 66, 80, 126, 128, 140, 192])
def test_pack_and_unpack(Lz, offset):
    import torch
    Lx, Ly = 3, 5
    n = Lx * Ly * Lz
    rng = np.random.default_rng(100 * Lz + offset)
    s = rng.choice(np.array([-128, -1, 0, 1, 2, 127], dtype=np.int8), n)
    src = torch.zeros(n + 64, dtype=torch.int8, device="cuda")
    src[offset:offset + n] = torch.from_numpy(s).cuda()
    dst = torch.full((n + 64,), 77, dtype=torch.int8, device="cuda")
    torch.cuda.synchronize()
    g = ig.Film(Lx, Ly, Lz, 1.0, 0.5, 3.0, 4)
    g.set_spins_device(src.data_ptr() + offset)
    g.get_spins_device(dst.data_ptr() + offset)
    g.synchronize()
    want = np.where(s > 0, 1, -1).astype(np.int8)
    got = dst.cpu().numpy()
    assert np.array_equal(got[offset:offset + n], want)
    assert (got[:offset] == 77).all() and (got[offset + n:] == 77).all()  # nothing beside the film
    o = O.Film(Lx, Ly, Lz, 1.0, 0.5, 3.0, 4)
    o.set_spins(want)
    assert np.array_equal(g.measure(), o.measure())
    g.close()
