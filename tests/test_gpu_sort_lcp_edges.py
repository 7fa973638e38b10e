"""Sizes at which the radix sort and the row-side sums of the LCP assembly can go
wrong: tile edges, key widths with odd and even numbers of digit passes and
sorting in place; rows whose points fill several sorting chunks."""
import numpy as np
import pytest

from paper_1812_04719_gb300 import scenegen as G
from paper_1812_04719_gb300 import stiv as S

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 255, 2047, 2048, 2049, 100_003, 1_300_000])
@pytest.mark.parametrize("bits", [1, 8, 9, 24, 27, 64])
@pytest.mark.parametrize("in_place", [False, True])
def test_sort_edges(n, bits, in_place):
    rng = np.random.default_rng(n + bits)
    k = rng.integers(0, 1 << 63, size=n, dtype=np.uint64) | (rng.integers(0, 2, size=n, dtype=np.uint64) << np.uint64(63))
    k[rng.integers(0, n, size=n // 4)] = k[0]          # equal keys: stability
    keys = torch.from_numpy(k.view(np.int64).copy()).cuda()
    vals = torch.arange(n, dtype=torch.int32, device="cuda")
    ko, vo = (keys, vals) if in_place else (torch.empty_like(keys), torch.empty_like(vals))
    nb = S.stiv_sort_scratch_bytes(n)
    scratch = torch.empty(nb, dtype=torch.uint8, device="cuda")
    S.stiv_sort_pairs(torch.cuda.current_stream().cuda_stream, n, bits, keys.data_ptr(), vals.data_ptr(),
                      ko.data_ptr(), vo.data_ptr(), scratch.data_ptr(), nb)
    order = np.argsort(k & np.uint64((1 << bits) - 1), kind="stable")
    assert np.array_equal(vo.cpu().numpy(), order.astype(np.int32))
    assert np.array_equal(ko.cpu().numpy().view(np.uint64), k[order])
    if not in_place:
        assert np.array_equal(keys.cpu().numpy().view(np.uint64), k)


@pytest.mark.parametrize("p,gap", [(8, 0.05), (12, -0.5), (24, -0.8)])
def test_one_row_sums(p, gap):
    """B of a single interpenetrating pair, |J|^2 of the rows summed per vertex.
    The sums hold up to 10^4 terms: 10^4 x 2^-53 relative."""
    sc = G.two_vesicles(p=p, seed=1, gap=gap, approach=0.3)
    eng = S.Stiv.for_scene(sc, pair_cap=16, contact_cap=1 << 16)
    ds = S.DeviceScene.from_scene(sc)
    r = eng.step(ds, grad=True)
    g, ves, vid = (r[k].cpu().numpy() for k in ("grad", "gves", "gvid"))
    J = np.zeros((2, G.nverts(2 * p), 3))
    np.add.at(J, (ves.ravel(), vid.ravel()), g.reshape(-1, 3))
    m = np.array([0.75, 1.5])
    t = np.array([1e-3, 2e-3])
    want = sum(m[v] * (J[v] ** 2).sum() + t[v] * (J[v].sum(axis=0) ** 2).sum() for v in range(2))
    a = S.ContactLCP().assemble(eng, ds, torch.as_tensor(m, device="cuda"), torch.as_tensor(t, device="cuda"))
    assert a["n"] == 1 and a["nnz"] == 1
    if gap < 0:
        assert len(ves) > 600       # over 1024 points on a side: several chunks
    assert abs(float(a["val"][0]) - want) <= 1e-12 * want
    b = S.ContactLCP().assemble(eng, ds, torch.as_tensor(m, device="cuda"), torch.as_tensor(t, device="cuda"))
    assert float(a["val"][0]) == float(b["val"][0])


@pytest.mark.parametrize("p,gap", [(8, 0.05), (16, -0.9), (32, -0.9)])
def test_long_contact_segments(orc, p, gap):
    """The ordering of one pair's contacts, of a segment that fits the sorting
    CTA's shared memory and of longer ones (2048 entries, merged): the oracle's list
    on the same vertices."""
    from tests.gpu_run import run_gpu_on, verts_list
    from tests.oracle_pool import oracle_vertices
    sc = G.two_vesicles(p=p, seed=1, gap=gap, approach=0.4)
    X = oracle_vertices(sc)
    g = run_gpu_on(sc, X, pair_cap=16, contact_cap=1 << 17)
    c = orc.contacts(sc.P, verts_list(sc, X), np.zeros((1, 5), np.int32) + np.array([[0, 1, 0, 0, 0]], np.int32), sc.L,
                     sc.eps * sc.dt, grad=False)
    if p == 32:
        assert len(c["pair"]) > 4096
    for k in ("pair", "type", "a", "b"):
        assert np.array_equal(g[k], c[k]), k
    assert np.array_equal(g["tau"].view(np.int64), np.ascontiguousarray(c["tau"]).view(np.int64))
