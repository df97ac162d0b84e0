"""Films in shared memory at the edges of the slab kernel's forms (four drawing
lanes per word, one, columns), against the CPU oracle.  Integers throughout:
every comparison is exact."""
import numpy as np
import pytest

import paper_1411_5588_gb300 as ig
from oracle import oracle as O

pytestmark = pytest.mark.gpu


# Words of a CTA: 32 and 128 (five threads each), 129 to 160 (four lanes in one
# turn of 640 threads), 161, 640 and 641 of eight calls; 2544 and 2561 of two;
# packed ones, 288 on two CTAs' layers.
@pytest.mark.parametrize("H", [0.0, 0.2])
@pytest.mark.parametrize("Lx,Ly,Lz,shape", [
    (4, 8, 64, ig.SHAPE_RESIDENT), (8, 16, 64, ig.SHAPE_RESIDENT), (3, 43, 64, ig.SHAPE_RESIDENT),
    (8, 20, 64, ig.SHAPE_RESIDENT), (7, 23, 64, ig.SHAPE_RESIDENT), (16, 40, 64, ig.SHAPE_RESIDENT),
    (1, 641, 64, ig.SHAPE_RESIDENT), (16, 159, 10, ig.SHAPE_RESIDENT), (13, 197, 10, ig.SHAPE_RESIDENT),
    (12, 48, 20, ig.SHAPE_RESIDENT), (64, 96, 64, ig.SHAPE_CLUSTER), (53, 97, 60, ig.SHAPE_CLUSTER)])
def test_forms(Lx, Ly, Lz, shape, H):
    g = ig.Film(Lx, Ly, Lz, 1.0, 0.5, 2.8, 17, H=H, shape=shape)
    o = O.Film(Lx, Ly, Lz, 1.0, 0.5, 2.8, 17, H=H)
    g.init(ig.INIT_RANDOM)
    o.init(ig.INIT_RANDOM, 0.0)
    for n, every in ((3, 1), (4, 2)):
        g.sweep(n, every)
        assert np.array_equal(g.read_series(), o.sweep(n, every))
    assert np.array_equal(g.get_spins(), o.get_spins())
    g.close()
