"""The contact LCP at the largest orders, where a row's vertex table and the
kernel's own arrays together pass 48 KB of shared memory (p = 32)."""
import numpy as np
import pytest

from paper_1812_04719_gb300 import scenegen as G
from paper_1812_04719_gb300 import stiv as S

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,other", [(31, 31), (32, 32), (32, 5)])
def test_lcp_one_row(p, other):
    """B of one interpenetrating pair, |J|^2 of the rows summed per vertex, and
    its LCP.  Sums of up to 10^4 terms: 10^4 x 2^-53 relative."""
    sc = G.two_vesicles(p=p, seed=1, gap=-0.5, approach=0.3)
    if other != p:                      # the second vesicle of a small order
        q = G.two_vesicles(p=other, seed=1, gap=-0.5, approach=0.3)
        n1 = 6 * (p + 1) ** 2
        sc.p = np.array([p, other], dtype=sc.p.dtype)
        sc.coef = np.concatenate([sc.coef[:n1], q.coef[6 * (other + 1) ** 2:]])
        sc.coef_off = np.array([0, n1], dtype=sc.coef_off.dtype)
    eng = S.Stiv.for_scene(sc, pair_cap=16, contact_cap=1 << 17)
    ds = S.DeviceScene.from_scene(sc)
    r = eng.step(ds, grad=True)
    g, ves, vid = (r[k].cpu().numpy() for k in ("grad", "gves", "gvid"))
    assert len(ves) > 100
    J = np.zeros((2, G.nverts(2 * p), 3))
    np.add.at(J, (ves.ravel(), vid.ravel()), g.reshape(-1, 3))
    m, t = np.array([0.75, 1.5]), np.array([1e-3, 2e-3])
    want = sum(m[v] * (J[v] ** 2).sum() + t[v] * (J[v].sum(axis=0) ** 2).sum() for v in range(2))
    lcp = S.ContactLCP()
    a = lcp.assemble(eng, ds, torch.as_tensor(m, device="cuda"), torch.as_tensor(t, device="cuda"))
    assert a["n"] == 1 and a["nnz"] == 1
    assert abs(float(a["val"][0]) - want) <= 1e-12 * want
    V = float(r["V_pair"][int(a["row_pair"][0])])
    assert abs(float(lcp.solve(eng)["lam"][0]) - V / want) <= 1e-9 * V / want
