"""Newton runs of a few i-particles against many j with the differences formed
on the tensor cores (the automatic choice from 48 i on), against the FP64
oracle: the edges of its i tiles (32, 64) and j tiles (128), i spread over the
whole system at 0.5 to 2 eps from j-particles, the self mode, masses of both
signs and many magnitudes, graph replays with new positions, and values that
do not fit its fixed point, where the double-float path stands in (i far
outside the j-set, eps too small or too large for the range, non-finite
records). Tolerances as for the double-float paths (median 2e-6, maximum
1e-4)."""

import numpy as np
import pytest

import gen
from pgtest import assert_parity, need_cuda, rel_scalar, rel_vec

pytestmark = pytest.mark.gpu

EPS = 1e-3


@pytest.fixture(scope="module")
def pg():
    return need_cuda()


def run(pg, xi, xj, mj, eps, self_=False, off=0, path=0):
    with pg.Context(0) as c:
        c.set_allpairs_path(path)
        c.set_eps(eps)
        if self_:
            c.set_self(True)
            if off:
                c.set_self_offset(off)
        c.set_j(xj, mj)
        c.set_i(xi)
        c.run()
        return (*c.get_force(len(xi)), c.info())


def near_j(xj, ni, seed, eps):
    rng = np.random.default_rng(seed)
    u = rng.normal(size=(ni, 3))
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    return xj[rng.choice(len(xj), size=ni, replace=False)] + u * (eps * rng.uniform(0.5, 2.0, ni))[:, None]


def check(orc, a, p, xi, xj, mj, eps, skip=None):
    ao, po = orc.newton(xi, xj, mj, eps, skip=skip)
    assert_parity(rel_vec(a, ao), what="a")
    assert_parity(rel_scalar(p, po), what="phi")


# 349526 j against 48 i: the fewest that take the path (2^24 pairs)
@pytest.mark.parametrize("ni, nj", [(48, 349526), (64, 262144), (65, 262145), (96, 200001), (512, 32769), (1000, 64000),
                                    (4096, 262271)])
def test_spread_sets(pg, orc, ni, nj):
    xj, mj = gen.plummer_cube_mix(nj, 900 + nj % 97)
    xi = near_j(xj, ni, ni, EPS)
    a, p, info = run(pg, xi, xj, mj, EPS)
    assert info["i_per_thread"] in (32, 64) and info["df"] == 1      # the tensor-core tiles
    idx = np.arange(ni) if ni <= 512 else gen.sample_indices(ni, 400, 1)
    check(orc, a[idx], p[idx], xi[idx], xj, mj, EPS)


@pytest.mark.parametrize("off", [0, 777])
def test_self_mode(pg, orc, off):
    x, m = gen.plummer(70000, 31)
    xi = x[off:off + 300]
    a, p, info = run(pg, xi, x, m, 0.01, self_=True, off=off)
    assert info["i_per_thread"] == 64
    check(orc, a, p, xi, x, m, 0.01, skip=np.arange(off, off + 300, dtype=np.int64))


def test_masses(pg, orc):
    x, m = gen.plummer(90001, 5)
    rng = np.random.default_rng(5)
    m = m * 10.0 ** rng.uniform(-12, 3, len(m)) * rng.choice([-1.0, 1.0, 0.0], len(m), p=[0.1, 0.8, 0.1])
    xi = gen.plummer(200, 6)[0]
    a, p, info = run(pg, xi, x, m, 0.01)
    assert info["i_per_thread"] == 64
    ao, po = orc.newton(xi, x, m, 0.01)
    # signs cancel: the error is held against the sums of magnitudes
    aa, pa = orc.newton(xi, x, np.abs(m), 0.01)
    assert np.max(np.abs(p - po) / np.abs(pa)) <= 1e-6
    assert np.max(np.linalg.norm(a - ao, axis=1) / (np.abs(pa) / 0.01)) <= 1e-6


def test_graph_replays_with_new_positions(pg, orc):
    xj, mj = gen.plummer_cube_mix(60000, 12)
    with pg.Context(0) as c:
        c.set_eps(EPS)
        c.set_graph(True)
        for k in range(5):
            y = xj * (1.0 + 0.1 * k)
            xi = near_j(y, 300, k, EPS)
            if k != 3:                  # call 3 keeps the j records of call 2
                c.set_j(y, mj)
                last = y
            c.set_i(xi)
            c.run()
            a, p = c.get_force(300)
            check(orc, a, p, xi, last, mj, EPS)


@pytest.mark.parametrize("what", ["i outside", "eps small", "eps large", "j outlier", "i at the edge"])
def test_values_that_do_not_fit(pg, orc, what):
    xj, mj = gen.plummer(60000, 3)
    xi = gen.plummer(300, 4)[0]
    eps = EPS
    if what == "i outside":
        xi[7] = [500.0, -3.0, 2.0]
    elif what == "i at the edge":
        xi[7] = xj.max(axis=0) * 1.2
    elif what == "eps small":
        eps = 1e-12
    elif what == "eps large":
        eps = 1e8
    else:
        xj[11] = [1e9, 0.0, 0.0]
    a, p, _ = run(pg, xi, xj, mj, eps)
    check(orc, a, p, xi, xj, mj, eps)


@pytest.mark.parametrize("which", ["x", "m", "xi"])
def test_nonfinite_as_on_the_narrow_path(pg, which):
    xj, mj = gen.plummer(60000, 3)
    xi = gen.plummer(300, 4)[0]
    {"x": xj, "m": mj, "xi": xi}[which][5] = np.nan
    a, p, _ = run(pg, xi, xj, mj, EPS)
    a2, p2, _ = run(pg, xi, xj, mj, EPS, path=pg.PG_PATH_NARROW)
    assert np.array_equal(np.isnan(a), np.isnan(a2)) and np.array_equal(np.isnan(p), np.isnan(p2))
    ok = np.isfinite(a2).all(axis=1)
    assert np.array_equal(a[ok], a2[ok])


@pytest.mark.parametrize("ni, nj", [(200, 100003), (2000, 131072)])
def test_no_signed_error(pg, orc, ni, nj):
    # the tensor cores round the differences toward zero; the unit they are
    # read in makes up for the mean (2.6e-8 of a potential without that). A
    # quarter of an FP32 ulp, 1.5e-8, is allowed for what depends on the set.
    # Against the masses as the sums hold them (FP32: 1/100003 rounds by 3.9e-8)
    xj, mj = gen.plummer(nj, ni)
    xi = gen.plummer(ni, nj)[0]
    _, p, info = run(pg, xi, xj, mj, EPS)
    assert info["i_per_thread"] == 64
    _, po = orc.newton(xi, xj, mj.astype(np.float32).astype(np.float64), EPS)
    assert abs(np.mean(p / po - 1)) <= 1.5e-8


def test_double_float_when_asked_for(pg):
    # PG_DIFF_DOUBLE is double-float on the automatic path too: the forced narrow path's bits
    xj, mj = gen.plummer(60000, 3)
    xi = gen.plummer(300, 4)[0]
    out = []
    for path in (pg.PG_PATH_AUTO, pg.PG_PATH_NARROW):
        with pg.Context(0) as c:
            c.set_allpairs_path(path)
            c.set_differencing(pg.PG_DIFF_DOUBLE)
            c.set_eps(EPS)
            c.set_j(xj, mj)
            c.set_i(xi)
            c.run()
            out.append(c.get_force(300))
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])


def both(pg, xi, xj, mj, eps, **kw):
    """The automatic path's (a, phi), and whether the tensor cores made them:
    the stand-in's bits are those of the forced narrow path."""
    a, p, _ = run(pg, xi, xj, mj, eps, **kw)
    a2, p2, _ = run(pg, xi, xj, mj, eps, path=pg.PG_PATH_NARROW, **kw)
    return a, p, not (np.array_equal(a, a2) and np.array_equal(p, p2))


# one far j sets the step of all positions, R 2^-47: just inside the accepted
# range (R = 4096, eps 2^22 times smaller), just outside, and far outside
@pytest.mark.parametrize("far, fits", [(30.0, True), (6000.0, True), (8000.0, False), (1.6e6, False)])
def test_close_pairs_beside_a_far_particle(pg, orc, far, fits):
    xj, mj = gen.plummer(60000, 3)
    xi = near_j(xj, 300, 9, EPS)
    xj[11] = [far, 0.0, 0.0]
    a, p, tc = both(pg, xi, xj, mj, EPS)
    assert tc == fits
    check(orc, a, p, xi, xj, mj, EPS)


# one body 2^k times as heavy as the others: their m / r^3, all of the force
# on the heavy one, has to stay in FP32's range
@pytest.mark.parametrize("k, fits", [(40, True), (110, False)])
def test_one_heavy_body(pg, orc, k, fits):
    x, m = gen.plummer(60000, 8)
    m = np.full(60000, 2.0 ** -k)
    m[5] = 1.0
    a, p, tc = both(pg, x[:300], x, m, 0.01, self_=True)
    assert tc == fits
    # the heavy body's own potential is not compared: its own pair's m / eps is
    # added and taken out in FP32 on every path (2e-3 off at 2^40, all of it from 2^60 on)
    ao, po = orc.newton(x[:300], x, m, 0.01, skip=np.arange(300, dtype=np.int64))
    assert_parity(rel_vec(a, ao), what="a")
    assert_parity(np.delete(rel_scalar(p, po), 5), what="phi")


@pytest.mark.parametrize("graph", [False, True])
def test_a_set_that_does_not_fit_is_remembered(pg, orc, graph):
    # once the host has seen the j-set's geometry, the double-float path runs
    # alone, until the j or eps change
    xj, mj = gen.plummer(60000, 3)
    far = xj.copy()
    far[11] = [1e9, 0.0, 0.0]
    xi = gen.plummer(300, 4)[0]

    def call(c, path):
        c.set_allpairs_path(path)
        c.run()
        a, p = c.get_force(300)
        return a, p, c.info()["launches"]

    with pg.Context(0) as c:
        c.set_graph(graph)
        c.set_eps(EPS)
        c.set_i(xi)
        c.set_j(far, mj)
        first = call(c, pg.PG_PATH_AUTO)
        later = [call(c, pg.PG_PATH_AUTO) for _ in range(3)][-1]
        c.set_graph(False)
        narrow = [call(c, pg.PG_PATH_NARROW) for _ in range(2)][-1]
        assert later[2] == narrow[2]
        for a, p, _ in (first, later):
            assert np.array_equal(a, narrow[0]) and np.array_equal(p, narrow[1])
        # a j-set that fits takes the tensor cores again, and so does an eps that fits
        c.set_graph(graph)
        c.set_j(xj, mj)
        a, p, n = call(c, pg.PG_PATH_AUTO)
        check(orc, a, p, xi, xj, mj, EPS)
        assert not np.array_equal(a, run(pg, xi, xj, mj, EPS, path=pg.PG_PATH_NARROW)[0])
        c.set_eps(1e-9)
        assert np.array_equal(call(c, pg.PG_PATH_AUTO)[0], run(pg, xi, xj, mj, 1e-9, path=pg.PG_PATH_NARROW)[0])
        c.set_eps(EPS)
        assert np.array_equal(call(c, pg.PG_PATH_AUTO)[0], a)


def test_stand_in_after_other_paths(pg, orc):
    # the stand-in's packed records are its own until another path writes the
    # buffer (a tree) or it grows
    xj, mj = gen.plummer(80000, 3)
    xi = gen.plummer(300, 4)[0]
    xi[7] = [500.0, -3.0, 2.0]
    with pg.Context(0) as c:
        c.set_eps(EPS)
        c.set_j(xj, mj)
        c.set_n(60000)

        def stand_in(n):
            c.set_n(n)
            c.set_i(xi)
            out = []
            for _ in range(2):
                c.run()
                out.append(c.get_force(300))
            ref = run(pg, xi, xj[:n], mj[:n], EPS, path=pg.PG_PATH_NARROW)
            for a, p in out:
                assert np.array_equal(a, ref[0]) and np.array_equal(p, ref[1])

        stand_in(60000)
        c.set_i(xj[:60000])
        c.set_self(True)
        c.set_tree(0.75, 256, 8)
        c.run()
        c.set_tree(-1.0, 256, 8)
        c.set_self(False)
        stand_in(60000)
        stand_in(80000)
        stand_in(60000)


@pytest.mark.parametrize("ni", [64, 300])
def test_new_j_records_cost_two_launches_more(pg, ni):
    # a run on new records: their digits and the tensor cores' kernel beside the narrow path's launches
    xj, mj = gen.plummer(349526, 3)
    xi = gen.plummer(ni, 4)[0]
    n = []
    for path in (pg.PG_PATH_AUTO, pg.PG_PATH_NARROW):
        with pg.Context(0) as c:
            c.set_allpairs_path(path)
            c.set_eps(EPS)
            for _ in range(2):
                c.set_j(xj, mj)
                c.set_i(xi)
                c.run()
                a, p = c.get_force(ni)
            n.append(c.info()["launches"])
    assert n[0] <= n[1] + 2


def test_info_of_a_run(pg):
    xj, mj = gen.plummer(60000, 3)
    _, _, info = run(pg, gen.plummer(300, 4)[0], xj, mj, EPS)
    # neither narrow items nor the batched kernel
    assert info["split"] == 0 and info["j_tile"] == 0 and info["block_threads"] == 0
    # the CTAs that share a tile of 64 i, in equal ranges of the (i tile, tile of 128 j) units
    njt = -(-60000 // 128)
    W = 5 * njt

    def owner(u):
        return ((u + 1) * info["grid"] - 1) // W

    assert info["slots"] == max(owner((t + 1) * njt - 1) - owner(t * njt) + 1 for t in range(5))
    assert info["pairs"] == 300 * 60000


def test_more_contexts_than_words_for_their_geometry(pg):
    # 64 contexts of a process can see their geometry; the others ask the
    # device on every call, and closed contexts give their words back
    xj, mj = gen.plummer(32769, 3)
    far = xj.copy()
    far[11] = [1e9, 0.0, 0.0]
    xi = gen.plummer(512, 4)[0]
    ref = [run(pg, xi, y, mj, EPS, path=pg.PG_PATH_NARROW) for y in (xj, far)]
    for _ in range(2):
        cs = [pg.Context(0) for _ in range(66)]
        for k, c in enumerate(cs):
            c.set_eps(EPS)
            c.set_j(far if k % 2 else xj, mj)
            c.set_i(xi)
        for _ in range(2):
            for k, c in enumerate(cs):
                c.run()
                a, p = c.get_force(512)
                same = np.array_equal(a, ref[k % 2][0]) and np.array_equal(p, ref[k % 2][1])
                assert same == bool(k % 2)
        for c in cs:
            c.close()
