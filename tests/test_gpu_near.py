"""The tabulated force's near-pair kernels (sorted i-tiles that leave out the
j-particles beyond r_cut of their box) against the FP64 oracle: the smallest
sorted set and its neighbours, ragged tiles and units, i-sets that are not the
j-set, cutoffs on both sides of the switch to the all-pairs kernel, the
potential's table, single differences, per-thread shapes, non-finite records,
and the gradients. Tolerances as for the all-pairs kernel (per particle,
median 2e-6 and maximum 1e-4 of |a|, pairs within 1e-6 of the cutoff allowed
either side; gradients 1e-4 norm-wise)."""

import numpy as np
import pytest

import gen
from pgtest import assert_parity, need_cuda

pytestmark = pytest.mark.gpu

E, F = 3, 5


@pytest.fixture(scope="module")
def pg():
    return need_cuda()


def table(orc, r_cut):
    # eps resolved by the table's innermost bins (they reach in to r_cut / 16)
    v = orc.table_values(E, F, r_cut, orc.SHAPE_GAUSS_SPLIT, [r_cut / 4.5, max(1 / 64, r_cut / 16)])
    return v, *orc.table_from_values(E, F, v)


def run(pg, xi, xj, mj, v, r_cut, self_, shape=0, diff=0, pot=None):
    with pg.Context(0) as c:
        c.set_mode(pg.PG_TABLE)
        c.set_table_values(v, r_cut, E, F)
        if pot is not None:
            c.set_table_pot_values(pot)
        c.set_self(self_)
        c.set_differencing(diff)
        c.set_allpairs_path(pg.PG_PATH_TILED)
        if shape:
            c.set_shape(shape)
        c.set_j(xj, mj)
        c.set_i(xi)
        c.run()
        return c.get_force(len(xi))


def check(orc, a, xi, xj, mj, r_cut, G0, G1, idx, skip):
    ao, amb = orc.table_forces(xi[idx], xj, mj, E, F, r_cut, G0, G1, skip=idx if skip else None, window=1e-6)
    na = np.linalg.norm(ao, axis=1)
    alone = na == 0
    assert np.all(np.linalg.norm(a[idx][alone], axis=1) <= amb[alone])   # no neighbour: exactly nothing
    err = np.maximum(np.linalg.norm(a[idx] - ao, axis=1) - amb, 0)[~alone] / na[~alone]
    assert_parity(err, what="a vs table semantics")


# 16384 is the smallest sorted set; 513 and 1025 j leave ragged units
@pytest.mark.parametrize("n, r_cut", [(16384, 0.1), (16385, 0.05), (20011, 0.3), (40000, 0.1), (16384, 60.0)])
def test_self_sets(pg, orc, n, r_cut):
    x, m = gen.plummer(n, 300 + n)
    m = m * np.random.default_rng(n).uniform(0.5, 1.5, n)
    v, G0, G1 = table(orc, r_cut)
    a, _ = run(pg, x, x, m, v, r_cut, True)
    check(orc, a, x, x, m, r_cut, G0, G1, gen.sample_indices(n, 1500, n), True)


@pytest.mark.parametrize("nj", [1, 255, 513, 1025, 30000])
def test_other_j_sets(pg, orc, nj):
    xi = gen.plummer(17000, 5)[0]
    xj, mj = gen.plummer(nj, 6)
    v, G0, G1 = table(orc, 0.4)
    a, _ = run(pg, xi, xj, mj, v, 0.4, False)
    check(orc, a, xi, xj, mj, 0.4, G0, G1, gen.sample_indices(17000, 1500, nj), False)


@pytest.mark.parametrize("shape", [1, 2, 4])
@pytest.mark.parametrize("diff", [0, 1])
def test_shapes_and_differences(pg, orc, shape, diff):
    x, m = gen.clustered_box(18003, 77)
    v, G0, G1 = table(orc, 0.04)
    a, _ = run(pg, x, x, m, v, 0.04, True, shape=shape, diff=diff)
    check(orc, a, x, x, m, 0.04, G0, G1, gen.sample_indices(18003, 1500, 3), True)


def test_potential(pg, orc):
    n, r_cut = 17001, 0.3
    x, m = gen.plummer(n, 91)
    v, G0, G1 = table(orc, r_cut)
    pv = -np.linspace(3.0, 0.5, len(v)).astype(np.float32)
    P0, P1 = orc.table_from_values(E, F, pv)
    a, phi = run(pg, x, x, m, v, r_cut, True, pot=pv)
    idx = gen.sample_indices(n, 1000, 4)
    check(orc, a, x, x, m, r_cut, G0, G1, idx, True)
    po, amb = orc.table_potential(x[idx], x, m, E, F, r_cut, P0, P1, skip=idx, window=1e-6)
    scale = np.abs(po) + 3.0 * m[idx]        # the loop also adds and removes the own pair's m psi(0)
    assert_parity(np.maximum(np.abs(phi[idx] - po) - amb, 0) / scale, what="phi")


# a record with a NaN makes every pair NaN, near or far; an infinite mass
# makes every pair beyond the cutoff NaN (inf times 0)
@pytest.mark.parametrize("what", ["position", "mass"])
def test_nonfinite_j_reaches_every_i(pg, orc, what):
    n, r_cut = 16500, 0.1
    x, m = gen.plummer(n, 17)
    xj, mj = x.copy(), m.copy()
    far = int(np.argmax(np.linalg.norm(x, axis=1)))
    if what == "position":
        xj[far] = np.nan
    else:
        mj[far] = np.inf
    v, _, _ = table(orc, r_cut)
    a, _ = run(pg, x, xj, mj, v, r_cut, False)
    rest = np.arange(n) != far
    assert np.isnan(a[rest]).any(axis=1).all()


def test_nonfinite_i_stays_its_own(pg, orc):
    n, r_cut = 16500, 0.1
    x, m = gen.plummer(n, 18)
    xi = x.copy()
    xi[123] = np.nan
    v, G0, G1 = table(orc, r_cut)
    a, _ = run(pg, xi, x, m, v, r_cut, False)
    assert np.isnan(a[123]).all()
    idx = gen.sample_indices(n, 800, 5)
    check(orc, a, x, x, m, r_cut, G0, G1, idx[idx != 123], False)


@pytest.mark.parametrize("n, r_cut", [(16384, 0.1), (20011, 0.2), (16400, 60.0)])
def test_gradients(pg, orc, n, r_cut):
    torch = pytest.importorskip("torch")
    from paper_1203_4037_gb300 import autograd as AG
    x, m = gen.plummer(n, 41)
    w = gen.unit_vectors(n, 42)
    v, _, _ = table(orc, r_cut)
    xt, mt, vt = (torch.tensor(t, device="cuda", requires_grad=True) for t in (x, m, v))
    a = AG.table_force(xt, mt, vt, r_cut, E, F)
    dx, dm, dv = torch.autograd.grad(a, (xt, mt, vt), torch.tensor(w, device="cuda"))
    idx = gen.sample_indices(n, 64, 9)
    ox, om = orc.grad_table_at(x, m, w, E, F, r_cut, v, idx)
    ov = orc.grad_table_v(x, m, w, E, F, r_cut, v)

    def rel(p, q):
        return np.linalg.norm(p - q) / np.linalg.norm(q)

    assert rel(dx.cpu().numpy()[idx], ox) <= 1e-4
    assert rel(dm.cpu().numpy()[idx], om) <= 1e-4
    assert rel(dv.cpu().numpy(), ov) <= 1e-4


# lengths scaled by a power of two scale every result exactly: at 2^-70 the
# square of r_cut is an FP32 denormal, at 2^70 beyond FP32
@pytest.mark.parametrize("k", [-70, 70])
def test_unit_of_length(pg, orc, k):
    torch = pytest.importorskip("torch")
    from paper_1203_4037_gb300 import autograd as AG
    n, r_cut, u = 20011, 0.1, 2.0 ** k
    x, m = gen.plummer(n, 29)
    w = torch.tensor(gen.unit_vectors(n, 30), device="cuda")
    v, _, _ = table(orc, r_cut)

    def grads(s):
        xt, mt, vt = (torch.tensor(t, device="cuda", requires_grad=True) for t in (x * s, m, v))
        a = AG.table_force(xt, mt, vt, r_cut * s, E, F)
        return (t.cpu().numpy() for t in torch.autograd.grad(a, (xt, mt), w))

    assert np.array_equal(run(pg, x * u, x * u, m, v, r_cut * u, True)[0], run(pg, x, x, m, v, r_cut, True)[0] * u)
    (dx, dm), (dxu, dmu) = grads(1.0), grads(u)
    assert np.array_equal(dxu, dx) and np.array_equal(dmu, dm * u)


# a shift that every coordinate takes exactly changes no bit, also where
# FP32 coordinates from the caller's origin would not tell the particles apart
@pytest.mark.parametrize("shift", [2.0 ** 14, 2.0 ** 26])
def test_far_from_the_origin(pg, orc, shift):
    n, r_cut = 20011, 0.1
    x, m = gen.plummer(n, 31)
    x = np.round(x * 2.0 ** 20) / 2.0 ** 20
    v, _, _ = table(orc, r_cut)
    assert np.array_equal(run(pg, x + shift, x + shift, m, v, r_cut, True)[0], run(pg, x, x, m, v, r_cut, True)[0])


# K u of a pair with a non-finite loss weight is non-finite near or far (0
# times it), on both sides of the switch to sorted tiles (16384)
@pytest.mark.parametrize("n", [16000, 16500])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_nonfinite_weight_reaches_every_gradient(pg, orc, n, bad):
    torch = pytest.importorskip("torch")
    from paper_1203_4037_gb300 import autograd as AG
    x, m = gen.plummer(n, 43)
    w = gen.unit_vectors(n, 44)
    far = int(np.argmax(np.linalg.norm(x, axis=1)))
    w[far, 1] = bad
    v, _, _ = table(orc, 0.1)
    xt, mt = (torch.tensor(t, device="cuda", requires_grad=True) for t in (x, m))
    a = AG.table_force(xt, mt, torch.tensor(v, device="cuda"), 0.1, E, F)
    dx, dm = torch.autograd.grad(a, (xt, mt), torch.tensor(w, device="cuda"))
    assert not torch.isfinite(dx).any() and not torch.isfinite(dm).any()


def test_without_room_for_the_near_records(pg, orc):
    # the FP32 j records (64 MiB) cannot be had: the all-pairs kernel runs alone
    torch = pytest.importorskip("torch")
    n, nj, r_cut = 16384, 1 << 22, 0.1
    x, _ = gen.plummer(n, 51)
    xj, mj = gen.plummer(nj, 52)
    v, _, _ = table(orc, r_cut)
    want = run(pg, x, xj, mj, v, r_cut, False)[0]
    with pg.Context(0) as c:
        c.set_mode(pg.PG_TABLE)
        c.set_table_values(v, r_cut, E, F)
        c.set_allpairs_path(pg.PG_PATH_TILED)
        c.set_j(xj, mj)
        c.set_i(x)
        torch.cuda.empty_cache()
        keep = torch.empty(torch.cuda.mem_get_info()[0] - (48 << 20), dtype=torch.uint8, device="cuda")
        try:
            c.run()
            got = c.get_force(n)[0]
        finally:
            del keep
            torch.cuda.empty_cache()
    err = np.linalg.norm(got - want, axis=1)
    assert np.max(err) <= 1e-5 * np.max(np.linalg.norm(want, axis=1))


def test_a_small_cutoff_leaves_pairs_out(pg, orc):
    # the near-pair kernels do the work: a third of the time and less of the
    # same set with every pair near (forward 360 against 1210 us a call,
    # gradients 0.55 against 63 ms)
    torch = pytest.importorskip("torch")
    n = 40000
    x, m = gen.plummer(n, 61)
    w = torch.tensor(gen.unit_vectors(n, 62), device="cuda")
    dx, dm = torch.empty_like(w), torch.empty(n, dtype=torch.float64, device="cuda")
    ms = {}
    for r_cut in (0.1, 60.0):
        with pg.Context(0) as c:
            c.set_mode(pg.PG_TABLE)
            c.set_table_values(table(orc, r_cut)[0], r_cut, E, F)
            c.set_self(True)
            c.set_timing(True)
            c.set_j(x, m)
            c.set_i(x)
            for _ in range(3):
                c.run()
                c.backward_dev(w, dx, dm)
            t_back = c.kernel_time()
            c.run()
            ms[r_cut] = (c.kernel_time(), t_back)
    assert ms[0.1][0] < 0.6 * ms[60.0][0] and ms[0.1][1] < 0.6 * ms[60.0][1]
