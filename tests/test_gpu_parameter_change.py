"""Films whose coupling or bulk field changes between sweeps, so that their
tables change between the three- and the seven-mask form, against the CPU
oracle.  Integers throughout: every comparison is exact."""
import numpy as np
import pytest

import paper_1411_5588_gb300 as ig
from oracle import oracle as O

pytestmark = pytest.mark.gpu


# Sizes whose slab launches differ between the two forms (shared memory, or the
# kernel's form), and a grid film.
@pytest.mark.parametrize("Lx,Ly,Lz,shape", [
    (8, 8, 8, ig.SHAPE_AUTO), (24, 601, 4, ig.SHAPE_AUTO), (64, 153, 10, ig.SHAPE_AUTO),
    (41, 47, 34, ig.SHAPE_RESIDENT), (96, 192, 64, ig.SHAPE_CLUSTER), (16, 150, 130, ig.SHAPE_CLUSTER),
    (32, 96, 64, ig.SHAPE_GRID_1), (32, 96, 64, ig.SHAPE_GRID_2)])
def test_tables_change_between_sweeps(Lx, Ly, Lz, shape):
    g = ig.Film(Lx, Ly, Lz, 1.0, 0.4, 2.6, 11, shape=shape)
    g.init(ig.INIT_RANDOM)
    o = O.Film(Lx, Ly, Lz, 1.0, 0.4, 2.6, 11)
    o.init(ig.INIT_RANDOM, 0.0)
    spins, count = o.get_spins(), 0
    for J, H, H1 in ((1.0, 0.0, 0.4), (-1.0, 0.0, 0.4), (1.0, 0.0, 0.1), (1.0, 0.3, 0.1), (1.0, 0.0, 0.0)):
        g.set_params(J, H1, 2.6)
        ig.check(ig.lib().ising_set_options(g._h, ig.Y_GAPBC, ig.X_FREE, H, 0), "ising_set_options")
        o = O.Film(Lx, Ly, Lz, J, H1, 2.6, 11, H=H)
        o.set_spins(spins)
        o.sweep_count = count
        g.sweep(3, 1)
        assert np.array_equal(g.read_series(), o.sweep(3, 1)), (J, H, H1)
        spins, count = o.get_spins(), count + 3
        assert np.array_equal(g.get_spins(), spins), (J, H, H1)
    g.close()
