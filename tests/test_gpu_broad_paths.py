"""Candidate vesicle pairs by the all-pairs test and by the Morton grid on the same
scenes, against the oracle's all-pairs box test: the same pairs and shifts in the
same order.  Free, periodic and mixed axes, few cells per axis and the cap of 255,
d_m > 0, odd and even numbers of digit passes of the pair sort, vesicles of an
order that is left out, overflowing lists."""
import math

import numpy as np
import pytest
import torch

from paper_1812_04719_gb300 import scenegen as G
from paper_1812_04719_gb300 import stiv as S
from tests.gpu_run import gpu_pairs_rows, run_gpu_on, verts_list
from tests.oracle_pool import oracle_vertices

pytestmark = pytest.mark.gpu

GRID, ALL_PAIRS = 0, 8192


def spheres(n, L, radii, seed, side=10.0, clusters=0, d_m=0.0):
    """n spheres of order 1 at random places of a box (free axes: of length side;
    with clusters, in that many clouds of extent 4 that far apart), each moved by
    a small step."""
    rng = np.random.default_rng(seed)
    L = np.asarray(L, dtype=np.float64)
    c = rng.uniform(0, 1, size=(n, 3)) * np.where(L > 0, L, side)
    if clusters:
        c = rng.uniform(0, 1, size=(clusters, 3))[rng.integers(0, clusters, n)] * side + rng.uniform(0, 4, size=(n, 3))
    r = np.exp(rng.uniform(math.log(radii[0]), math.log(radii[1]), size=n))
    step = rng.normal(size=(n, 3)) * 0.2 * radii[0]
    coefs = [np.stack([G.ellipsoid_coef(1, c[k], r[k] * np.eye(3)), G.ellipsoid_coef(1, c[k] + step[k], r[k] * np.eye(3))])
             for k in range(n)]
    sc = G._pack(f"spheres {n} {seed} {d_m}", [1] * n, coefs, L, c)
    sc.d_m = d_m
    return sc


SCENES = {
    "two_free": lambda: spheres(2, (0, 0, 0), (3.0, 4.0), 1),
    "one_cell": lambda: spheres(40, (30, 30, 30), (4.0, 5.0), 2),
    "two_passes": lambda: spheres(20, (20, 20, 20), (1.0, 3.0), 12),
    "few_cells": lambda: spheres(300, (30, 36, 42), (2.0, 4.0), 3),
    "mixed_axes": lambda: spheres(300, (30, 0, 26), (1.0, 3.0), 4, side=40.0),
    "one_periodic_axis": lambda: spheres(200, (0, 0, 18), (0.5, 2.0), 5),
    "free": lambda: spheres(1000, (0, 0, 0), (0.1, 0.6), 6),
    "cell_cap": lambda: spheres(600, (0, 0, 0), (0.3, 0.8), 7, side=4000.0, clusters=6),
    "many_cells": lambda: spheres(1500, (60, 60, 60), (0.2, 0.4), 8),
    "d_m": lambda: spheres(300, (30, 30, 30), (1.0, 2.0), 9, d_m=0.3),
    "one_large": lambda: spheres(500, (0, 0, 0), (0.05, 6.0), 10),
}


def engine(sc, limit, **kw):
    eng = S.Stiv.for_scene(sc, **kw)
    S.stiv_set_all_pairs_limit(eng.h, limit)
    return eng


@pytest.mark.parametrize("name", sorted(SCENES))
def test_both_paths_match_the_oracle(orc, name):
    sc = SCENES[name]()
    X = oracle_vertices(sc)
    boxes = np.stack([orc.vesicle_box(x, sc.d_m) for x in verts_list(sc, X)])
    pairs = orc.candidate_pairs(boxes, sc.L)
    assert len(pairs) > 0
    for limit in (GRID, ALL_PAIRS, sc.n, sc.n - 1):
        eng = engine(sc, limit, pair_cap=len(pairs) + 8, contact_cap=1 << 18)
        assert np.array_equal(gpu_pairs_rows(run_gpu_on(sc, X, grad=False, eng=eng)), pairs), limit


def test_grid_by_default_in_free_space(orc):
    sc = spheres(8193, (0, 0, 0), (0.05, 0.3), 11, side=20.0)
    X = oracle_vertices(sc)
    boxes = np.stack([orc.vesicle_box(x, 0.0) for x in verts_list(sc, X)])
    pairs = orc.candidate_pairs(boxes, sc.L)
    g = run_gpu_on(sc, X, grad=False, eng=S.Stiv.for_scene(sc, pair_cap=1 << 17, contact_cap=1 << 18))
    assert len(pairs) > 1000 and np.array_equal(gpu_pairs_rows(g), pairs)


@pytest.mark.parametrize("limit", [GRID, ALL_PAIRS])
@pytest.mark.parametrize("bad", [0, -3, 2, 1000])
def test_bad_order_is_left_out(limit, bad):
    sc = SCENES["mixed_axes"]()
    X = oracle_vertices(sc)
    want = gpu_pairs_rows(run_gpu_on(sc, X, grad=False, eng=engine(sc, ALL_PAIRS, pair_cap=1 << 13, contact_cap=1 << 18)))
    k = int(want[len(want) // 2, 0])
    eng = engine(sc, limit, pair_cap=1 << 13, contact_cap=1 << 18)
    ds = S.DeviceScene.from_scene(sc)
    ds.verts.copy_(torch.from_numpy(X))
    ds.p[k] = bad
    with pytest.raises(S.StivError) as e:
        eng.step(ds, grad=False, upsample=False)
    assert e.value.status == S.STIV_ERR_INPUT
    counts = eng.buf.counts.cpu().numpy()
    assert counts[S.C_STATUS] == S.F_BAD_ORDER
    b, n = eng.buf, int(counts[S.C_PAIRS])
    got = gpu_pairs_rows({q: x[:n].cpu().numpy() for q, x in (("i", b.ci), ("j", b.cj), ("shift", b.cs))})
    assert np.array_equal(got, want[(want[:, 0] != k) & (want[:, 1] != k)])


@pytest.mark.parametrize("limit", [GRID, ALL_PAIRS])
@pytest.mark.parametrize("precision", [S.STIV_FP64, S.STIV_MIXED])
def test_boxes_that_are_not_finite_are_left_out(limit, precision):
    """Vesicles that reach from -inf to inf on every axis or on one, or that are NaN
    on one, beside one of an order that is left out: flagged, in no pair, and the
    other pairs as without them."""
    sc = SCENES["free"]()
    X = oracle_vertices(sc)
    kw = dict(precision=precision, pair_cap=1 << 15, contact_cap=1 << 19)
    want = gpu_pairs_rows(run_gpu_on(sc, X, precision=precision, grad=False, eng=engine(sc, ALL_PAIRS, **kw)))
    out = [3, 40, 41, 500, 501, 999]     # infinite on all axes, on y, on z to one side, NaN on y, on x, bad order
    X = X.copy().reshape(sc.n, 2, 3, -1)
    X[3, 0, :, 5], X[3, 1, :, 5] = -np.inf, np.inf
    X[40, 0, 1, 5], X[40, 1, 1, 5] = -np.inf, np.inf
    X[41, 0, 2, 5] = -np.inf
    X[500, :, 1], X[501, :, 0] = np.nan, np.nan
    eng = engine(sc, limit, **kw)
    ds = S.DeviceScene.from_scene(sc, precision=precision)
    ds.verts.copy_(torch.from_numpy(X.ravel()))
    ds.p[999] = 1000
    with pytest.raises(S.StivError) as e:
        eng.step(ds, grad=False, upsample=False)
    assert e.value.status == S.STIV_ERR_INPUT
    counts = eng.buf.counts.cpu().numpy()
    assert counts[S.C_STATUS] == S.F_NONFINITE | S.F_BAD_ORDER
    b, n = eng.buf, int(counts[S.C_PAIRS])
    got = gpu_pairs_rows({q: x[:n].cpu().numpy() for q, x in (("i", b.ci), ("j", b.cj), ("shift", b.cs))})
    assert np.array_equal(got, want[~np.isin(want[:, 0], out) & ~np.isin(want[:, 1], out)])


@pytest.mark.parametrize("boxes_off", [-700, 3, 700])
def test_suspension_far_from_the_origin(orc, boxes_off):
    """Periodic coordinates that are never wrapped, whole boxes away."""
    sc = spheres(300, (32, 32, 0), (1.0, 3.0), 13, side=30.0)
    X = oracle_vertices(sc).reshape(sc.n, 2, 3, -1).copy()
    X[:, :, :2] += boxes_off * 32.0
    X = X.ravel()
    pairs = orc.candidate_pairs(np.stack([orc.vesicle_box(x, 0.0) for x in verts_list(sc, X)]), sc.L)
    assert len(pairs) > 300
    for limit in (GRID, ALL_PAIRS):
        g = run_gpu_on(sc, X, grad=False, eng=engine(sc, limit, pair_cap=1 << 13, contact_cap=1 << 18))
        assert np.array_equal(gpu_pairs_rows(g), pairs), limit


@pytest.mark.parametrize("what", ["spread", "large", "huge"])
def test_boxes_beyond_the_records_are_flagged(what):
    """The grid's records hold some 1000 unwrapped cells per axis.  Vesicles spread
    over more, and boxes that cover more (their cells counted past 2^31), are
    flagged; the next good call is right."""
    sc = spheres(300, (60, 60, 60), (0.2, 0.4), 14)
    X0 = oracle_vertices(sc)
    X = X0.reshape(sc.n, 2, 3, -1).copy()
    if what == "spread":
        X[::2] += 1000 * 60.0
    else:
        X[5:40, 1] += 1e6 if what == "large" else 1e200
    eng = engine(sc, GRID, pair_cap=1 << 12, contact_cap=1 << 16)
    ds = S.DeviceScene.from_scene(sc)
    ds.verts.copy_(torch.from_numpy(X.ravel()))
    b = eng._buffers(False)
    st = torch.cuda.current_stream().cuda_stream
    S.stiv_detect(eng.h, st, ds.n, ds.p_max, S._ptr(ds.p), S._ptr(ds.vert_off), S._ptr(ds.verts), b.pairs_struct(),
                  b.contacts_struct(), S._ptr(b.counts))
    counts = S.stiv_sync_counts(st, S._ptr(b.counts))[1]
    assert counts[S.C_STATUS] & S.F_BOX_TOO_SMALL
    want = run_gpu_on(sc, X0, grad=False, eng=engine(sc, ALL_PAIRS, pair_cap=1 << 12, contact_cap=1 << 16))
    got = run_gpu_on(sc, X0, grad=False, eng=eng)
    assert got["counts"][S.C_STATUS] == 0 and np.array_equal(gpu_pairs_rows(got), gpu_pairs_rows(want))


@pytest.mark.parametrize("limit", [GRID, ALL_PAIRS])
def test_overflowing_lists_grow(limit):
    sc = SCENES["few_cells"]()
    X = oracle_vertices(sc)
    want = gpu_pairs_rows(run_gpu_on(sc, X, grad=False, eng=engine(sc, ALL_PAIRS, pair_cap=1 << 14, contact_cap=1 << 18)))
    eng = engine(sc, limit, pair_cap=2, contact_cap=8)
    ds = S.DeviceScene.from_scene(sc)
    ds.verts.copy_(torch.from_numpy(X))
    b = eng._buffers(False)
    st = torch.cuda.current_stream().cuda_stream
    S.stiv_detect(eng.h, st, ds.n, ds.p_max, S._ptr(ds.p), S._ptr(ds.vert_off), S._ptr(ds.verts), b.pairs_struct(),
                  b.contacts_struct(), S._ptr(b.counts))
    rc, counts = S.stiv_sync_counts(st, S._ptr(b.counts))
    assert rc == S.STIV_ERR_CAPACITY and counts[S.C_STATUS] & (S.F_PAIRS_OVERFLOW | S.F_WORK_OVERFLOW)
    assert np.array_equal(gpu_pairs_rows(run_gpu_on(sc, X, grad=False, eng=eng)), want)


def test_limit_out_of_range():
    eng = S.Stiv()
    for bad in (-1, 8193):
        with pytest.raises(S.StivError):
            S.stiv_set_all_pairs_limit(eng.h, bad)
