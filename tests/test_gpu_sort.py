"""The radix sort behind the tree, the tiles and the cell list, through the
tree's particle order (a stable sort of the oracle's keys, bit-exact): one key,
a tile less one, a tile, a tile more one, both tile sizes (the switch is at
2^18), many tiles, and sets where nearly all keys share a digit."""

import numpy as np
import pytest

import gen
from pgtest import need_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pg():
    return need_cuda()


def keys(x):
    lo = x.min(axis=0)
    span = float((x.max(axis=0) - lo).max()) or 1.0
    q = np.minimum(np.floor((x - lo) / span * 1024), 1023).astype(np.int64)
    k = np.zeros(len(x), np.int64)
    for b in range(10):
        for a in range(3):
            k |= ((q[:, a] >> b) & 1) << (3 * b + 2 - a)
    return k


def order(pg, x):
    with pg.Context(0) as c:
        c.set_eps(0.01)
        c.set_self(True)
        c.set_tree(0.75, 256, 8)
        c.set_j(x, np.full(len(x), 1.0 / len(x)))
        c.set_i(x)
        c.run()
        return c.get_tree()["perm"]


@pytest.mark.parametrize("n", [1, 31, 2047, 2048, 2049, 100003, 1 << 18, (1 << 18) + 1, 70 * 8192 + 5])
def test_order_is_the_stable_sort(pg, n):
    x = gen.plummer(n, 50 + n)[0]
    assert np.array_equal(order(pg, x), np.argsort(keys(x), kind="stable"))


@pytest.mark.parametrize("n", [5000, 300000])
def test_crowded_digits(pg, n):
    # all but a few particles in one octant's corner: most digits are equal
    x = gen.uniform_sphere(n, 7, radius=1e-3)[0]
    x[:3] = [[0, 0, 0], [1, 1, 1], [1, 0, 0.5]]
    assert np.array_equal(order(pg, x), np.argsort(keys(x), kind="stable"))


def test_more_cells_than_particles(pg, orc):
    # the cell list sorts its particles (small tiles) and its items (as many
    # as cells, large tiles) in one scratch
    n, nc, E, F = 100000, 70, 3, 5
    x, m = gen.clustered_box(n, 8)
    r_cut = 1.0 / nc * 0.999
    v = orc.table_values(E, F, r_cut, orc.SHAPE_GAUSS_SPLIT, [r_cut / 4.5, r_cut / 16])
    with pg.Context(0) as c:
        c.set_mode(pg.PG_TABLE)
        c.set_table_values(v, r_cut, E, F)
        c.set_self(True)
        c.set_periodic(1.0)
        a, _ = c.forces(x, x, m)
    idx = gen.sample_indices(n, 500, 2)
    G0, G1 = orc.table_from_values(E, F, v)
    ao, amb = orc.table_forces(x[idx], x, m, E, F, r_cut, G0, G1, box=1.0, skip=idx, window=1e-6)
    na = np.linalg.norm(ao, axis=1)
    some = na > 0
    assert np.max((np.maximum(np.linalg.norm(a[idx] - ao, axis=1) - amb, 0))[some] / na[some]) <= 1e-4
    assert np.all(np.linalg.norm(a[idx][~some], axis=1) <= amb[~some])


# a block whose wait for the tiles before it runs out counts their keys
# itself: all blocks do here, with one tile, a remainder, both tile sizes
@pytest.mark.parametrize("n", [1, 2048, 2049, 40001, 1 << 18, (1 << 18) + 1, 70 * 8192 + 5])
def test_order_without_waiting(pg, n):
    with pg.Context(0) as c:
        c.selftest_sort(n)


@pytest.mark.parametrize("other", ["tree", "mesh", "selftest"])
def test_tiles_after_another_sort(pg, other):
    # a tiled run keeps its order between calls in the sort's buffers; other
    # sorts of the context (also larger ones, which move the buffers) use them
    x, m = gen.plummer(20011, 77)
    with pg.Context(0) as c:
        c.set_eps(0.01)
        c.set_self(True)
        c.set_j(x, m)
        c.set_i(x)
        c.run()
        a, p = c.get_force(len(x))
        if other == "tree":
            c.set_tree(0.75, 256, 8)
            c.run()
            c.set_tree(-1.0, 256, 8)
        elif other == "mesh":
            y, w = gen.clustered_box(100003, 5)
            c.set_periodic(1.0)
            c.set_pm(64, pg.PG_SPLIT_GAUSS, 1 / 64)
            c.pm_forces(y, w)
            c.set_pm(0, pg.PG_SPLIT_GAUSS, 1.0)
            c.set_periodic(0.0)
        else:
            c.selftest_sort(1 << 20)
        c.run()
        a2, p2 = c.get_force(len(x))
    assert np.array_equal(a, a2) and np.array_equal(p, p2)
