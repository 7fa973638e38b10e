"""Tensor-core synthesis and adjoint (STIV_MIXED) at the edges of their tiles: a
vertex and a coefficient gradient are sums in a fixed order over their own
column, so they are the same bits in a batch whose column tiles go in pairs, in
one whose tiles go singly, and alone; and the integer-pipe rounding of the
operands to FP32 keeps zeros, FP32-subnormal and large values within the FP64
synthesis's bound."""
import numpy as np
import pytest
import torch

from paper_1812_04719_gb300 import scenegen as G
from paper_1812_04719_gb300 import stiv as S

pytestmark = pytest.mark.gpu


def scene(ps, rng):
    coefs = [rng.standard_normal((2, 3, (p + 1) ** 2)) for p in ps]
    return G._pack("tiles", ps, coefs, (0.0, 0.0, 0.0), np.zeros((len(ps), 3)))


def both(sc, gX, precision=S.STIV_MIXED):
    """Vertices, and the coefficient gradient of gX (written over NaN)."""
    eng = S.Stiv(precision=precision)
    ds = S.DeviceScene.from_scene(sc, precision=precision)
    eng.upsample(ds)
    g = torch.as_tensor(gX, device="cuda")
    out = torch.full_like(ds.coef, float("nan"))
    st = torch.cuda.current_stream().cuda_stream
    S.stiv_grad_to_coef(eng.h, st, ds.n, ds.p_max, ds.p.data_ptr(), ds.coef_off.data_ptr(), ds.vert_off.data_ptr(),
                        g.data_ptr(), out.data_ptr())
    torch.cuda.synchronize()
    res = ds.verts.cpu().numpy(), out.cpu().numpy()
    eng.close()
    return res


@pytest.mark.parametrize("ps", [[32] * 205 + [3] * 7 + [7] * 30,       # synthesis tiles in pairs, an odd last one
                                [1] * 5 + [2] * 26001,                 # adjoint tiles in pairs
                                [16] * 22 + [5, 11]], ids=["synthesis_pairs", "adjoint_pairs", "single"])
def test_tiles_do_not_change_bits(ps):
    rng = np.random.default_rng(len(ps))
    ps = list(rng.permutation(ps))
    sc = scene(ps, rng)
    gX = rng.standard_normal(sc.n_vert_values())
    X, q = both(sc, gX)
    vo, vs = sc.vert_off(), sc.vert_sizes()
    # 1, 21 and 22 vesicles: a column tile of 128 holds 21 of 6 columns, 42 of 3
    for pick in ([0], list(range(len(ps) - 21, len(ps))), list(range(3, 25)) if len(ps) > 24 else [1, 2]):
        sub = G._pack("sub", [ps[v] for v in pick], [sc.coef_of(v) for v in pick], (0.0, 0.0, 0.0),
                      np.zeros((len(pick), 3)))
        xs, qs = both(sub, np.concatenate([gX[vo[v]:vo[v] + vs[v]] for v in pick]))
        assert np.array_equal(xs.view(np.int32),
                              np.concatenate([X[vo[v]:vo[v] + vs[v]] for v in pick]).view(np.int32))
        assert np.array_equal(qs.view(np.int64),
                              np.concatenate([q[sc.coef_off[v]:sc.coef_off[v] + sc.coef_of(v).size]
                                              for v in pick]).view(np.int64))
    for v in (0, len(ps) - 1):                       # X0 is a constant of the step
        n = sc.coef_of(v).size // 2
        assert np.all(q[sc.coef_off[v]:sc.coef_off[v] + n] == 0.0)


@pytest.mark.parametrize("scale", [0.0, 1e-320, 1e-42, 2.0 ** -126, 1.0, 1e30])
def test_operand_rounding(scale):
    """|X - X64| <= 2^-23 |X| + 2^-19 sum |a_q| Ymax as for ordinary values,
    plus FP32's smallest normal value per term where subnormals may be lost."""
    rng = np.random.default_rng(5)
    p = 6
    sc = scene([p] * 3, rng)
    sc.coef *= scale
    sc.coef[::7] = -0.0
    sc.coef[1::7] = np.where(rng.random(sc.coef[1::7].size) < 0.5, 1.0, -1.0) * scale * (1 + 2.0 ** -24)  # ties
    gX = np.zeros(sc.n_vert_values())
    X, _ = both(sc, gX)
    X64, _ = both(sc, gX, S.STIV_FP64)
    nv = sc.vert_sizes()[0] // 6
    a1 = np.abs(sc.coef.reshape(-1, (p + 1) ** 2)[:, 1:]).sum(axis=1)[:, None]
    X, X64 = X.astype(np.float64).reshape(-1, nv), X64.reshape(-1, nv)
    ymax = np.sqrt((2 * p + 1) / (2 * np.pi))
    bound = 2.0 ** -23 * np.abs(X64) + 2.0 ** -19 * a1 * ymax + 2.0 ** -126 * 3 * (p + 1) ** 2 * ymax
    assert np.all(np.abs(X - X64) <= bound)
