"""LCP rows of more contacts than one CTA takes at once: pairs that go deep into each
other beside short rows, against J M J^T of the summed gradient rows in numpy."""
import numpy as np
import pytest

from paper_1812_04719_gb300 import scenegen as G
from paper_1812_04719_gb300 import stiv as S

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def scene(p, approach):
    """Two vesicles that run into a third from both sides, and a far pair that meets
    slightly."""
    a = G.two_vesicles(p=p, seed=4, gap=0.02, approach=approach)
    b = G.two_vesicles(p=6, seed=2)
    c1, c2 = a.coef_of(0), a.coef_of(1)
    far = [b.coef_of(0).copy(), b.coef_of(1).copy()]
    for c in far:
        c[:, :, 0] += 40.0 * np.sqrt(4 * np.pi)
    return G._pack(f"long rows {p}", [p, p, p, 6, 6], [c1, c2, -c2] + far, np.zeros(3), np.zeros((5, 3)))


@pytest.mark.parametrize("p,approach,aligned", [(12, 1.5, True), (16, 1.5, True), (16, 1.5, False), (24, 2.0, True)])
def test_long_rows(p, approach, aligned):
    """Sums of up to 10^4 terms: 10^4 x 2^-53 relative to the entries' scale."""
    sc = scene(p, approach)
    eng = S.Stiv.for_scene(sc, pair_cap=16, contact_cap=1 << 18)
    ds = S.DeviceScene.from_scene(sc)
    r = eng.step(ds, grad=True)
    pair, g, ves, vid = (r[k].cpu().numpy() for k in ("pair", "grad", "gves", "gvid"))
    rows, row = np.unique(pair, return_inverse=True)
    count = np.bincount(row)
    assert count.max() > 2048 and count.min() < 2048 and len(rows) >= 3
    J = np.zeros((len(rows), sc.n, G.nverts(2 * p), 3))
    np.add.at(J, (np.repeat(row, 4), ves.ravel(), vid.ravel()), g.reshape(-1, 3))
    m, t = np.linspace(0.5, 1.5, sc.n), np.linspace(1e-3, 2e-3, sc.n)
    B = np.einsum("v,rvkc,svkc->rs", m, J, J) + np.einsum("v,rvc,svc->rs", t, J.sum(axis=2), J.sum(axis=2))
    if not aligned:   # the ids at addresses that allow no 16-byte loads
        b = eng.buf
        for k in ("gves", "gvid"):
            x = torch.zeros(b.gves.numel() + 1, dtype=torch.int32, device="cuda")[1:].view_as(b.gves)
            x.copy_(getattr(b, k))
            setattr(b, k, x)
    lcp = S.ContactLCP()
    got = []
    for _ in range(2):
        a = lcp.assemble(eng, ds, torch.as_tensor(m, device="cuda"), torch.as_tensor(t, device="cuda"))
        assert a["n"] == len(rows) and np.array_equal(a["row_pair"].cpu().numpy(), rows)
        ptr, col, val = (a[k].cpu().numpy() for k in ("row_ptr", "col", "val"))
        D = np.zeros_like(B)
        D[np.repeat(np.arange(len(rows)), np.diff(ptr)), col] = val
        got.append(D)
    scale = np.sqrt(np.outer(np.diag(B), np.diag(B)))
    assert np.all(np.abs(got[0] - B) <= 1e-12 * scale)
    assert np.array_equal(got[0], got[1]) and np.array_equal(got[0], got[0].T)
